// kernels.cuh -- device code of the random-phase Trotter path (sm_103a).
//
//   init_kernel   : the paper's entangled random-phase state (or its product
//                   state), phases from an in-kernel Philox4x32-10, fused
//                   P(0)/norm reduction.
//   coef_kernel   : FP64 generation of every flip-flop gate's three-shear
//                   coefficients (tan theta/2, sin theta) for dt/2 and dt, and
//                   the FP32 pair closest to a rotation.
//   diag_kernel   : FP64 -> 64-bit fixed-point turn tables of e^{-i tau a_ij/4 s s}.
//   sweep_kernel  : one pass over the whole state in shared-memory tiles of 2^K
//                   amplitudes: applies the pass's gates, the diagonal phase and
//                   the polarization reduction, then writes the tile back.
//   sweep2_kernel : the same pass with register-blocked phases (complex64).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace spinrp {

template <typename R> struct CT;
template <> struct CT<float> { using T = float2; };
template <> struct CT<double> { using T = double2; };

struct LayoutArg {
  uint8_t logical_of[kMaxM];  // physical bit position -> logical spin
};

// Sweeps follow each other with programmatic dependences: a sweep's blocks may
// be resident, with the pass's program staged (it does not depend on the sweep
// before), while that sweep still runs; grid_wait() returns once every earlier
// kernel has finished and its writes are visible, grid_go() lets the next
// sweep's blocks in once all of this one's have called it (see launch_sweep).
// A sweep calls it after its wait, so that one sweep at most waits beside the one
// that runs: called before, the sweeps after the next came in too, and SMs filled
// with waiting blocks got two blocks of one sweep while others had none (128-block
// sweeps, us per step: 19-spin complex128 star 1219 -> 689, 19-spin complex64
// chain 21.1 -> 15.9).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint64_t deposit_bits(uint64_t v, const uint8_t *pos, int n) {
  uint64_t r = 0;
  for (int k = 0; k < n; ++k) r |= ((v >> k) & 1ull) << pos[k];
  return r;
}

// Insert a zero bit at position b of x.
__device__ __forceinline__ uint32_t insert_zero(uint32_t x, int b) {
  return ((x >> b) << (b + 1)) | (x & ((1u << b) - 1u));
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): 10 rounds of two 32x32
// multiplies (multipliers 0xD2511F53, 0xCD9E8D57) mixed with the counter and a
// key bumped by the Weyl constants 0x9E3779B9, 0xBB67AE85.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// e^{2 pi i theta / 2^64} for a 64-bit fixed-point turn count theta.
__device__ __forceinline__ double2 cis_turns(uint64_t theta, double) {
  const double turns = (double)(int64_t)theta * 5.421010862427522e-20;  // 2^-64
  double s, c;
  sincospi(2.0 * turns, &s, &c);
  return make_double2(c, s);
}
// FP32 version: split off the nearest quarter turn exactly in integers, take
// sin/cos of the remainder (|r| <= 1/8 turn, so float keeps ~2^-27 turn
// absolute precision) and rotate by the quarter turns.
__device__ __forceinline__ float2 cis_turns(uint64_t theta, float) {
  const int64_t h = (int64_t)(int32_t)(uint32_t)(theta >> 32);  // turns * 2^32, signed
  const int64_t k = (h + (1ll << 29)) >> 30;                     // nearest quarter turn
  const int32_t r = (int32_t)(h - (k << 30));                    // |r| <= 2^29
  float s, c;
  sincospif((float)r * 4.656612873077393e-10f, &s, &c);          // angle = pi * r * 2^-31
  switch ((int)(k & 3)) {
    case 0: return make_float2(c, s);
    case 1: return make_float2(-s, c);
    case 2: return make_float2(-c, -s);
    default: return make_float2(s, -c);
  }
}

template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
  C r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// Deterministic grid reduction of (N_up, N_dn) for the job of this block row:
// block partials in FP64, the last block to finish sums them in block order,
// appends (P, norm) to the job's series at its step counter (slot 0 when
// `reset`) and advances the counter.
__device__ void reduce_finalize(double up, double dn, const JobPtrs &jp, bool reset) {
  double2 *partials = jp.partials;
  unsigned *ticket = jp.ticket;
  __shared__ double s_up[32], s_dn[32];
  __shared__ int s_last;
  for (int o = 16; o; o >>= 1) {
    up += __shfl_xor_sync(0xffffffffu, up, o);
    dn += __shfl_xor_sync(0xffffffffu, dn, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane == 0) s_up[warp] = up, s_dn[warp] = dn;
  __syncthreads();
  if (threadIdx.x == 0) {
    double u = 0.0, d = 0.0;
    for (int w = 0; w < nw; ++w) u += s_up[w], d += s_dn[w];
    partials[blockIdx.x] = make_double2(u, d);
    __threadfence();
    const unsigned t = atomicAdd(ticket, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double u = 0.0, d = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    const double2 p = __ldcg(&partials[b]);
    u += p.x, d += p.y;
  }
  for (int o = 16; o; o >>= 1) {
    u += __shfl_xor_sync(0xffffffffu, u, o);
    d += __shfl_xor_sync(0xffffffffu, d, o);
  }
  __syncthreads();
  if (lane == 0) s_up[warp] = u, s_dn[warp] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double U = 0.0, D = 0.0;
    for (int w = 0; w < nw; ++w) U += s_up[w], D += s_dn[w];
    const int64_t slot = reset ? 0 : *jp.step;
    jp.series[2 * slot] = (U - D) / (U + D);
    jp.series[2 * slot + 1] = U + D;
    *jp.step = slot + 1;
    *ticket = 0u;
  }
}

// ---------------------------------------------------------------------------
// All-site readout (P_{q1}(t) for every spin q).  A reducing sweep leaves per
// block, per tile bit, the weight with that bit up (and the block's norm);
// write_site_partials turns them into per-spin columns and
// sites_finalize_kernel sums the columns over blocks in a fixed order.
// ---------------------------------------------------------------------------
constexpr int kSiteSlots = kMaxK + 1;  // tile bits 0..kMaxK-1, slot kMaxK = norm
constexpr int kMaxWarps = 16;

// Warp-sum v (in the thread's precision) and park it at s_w[warp][slot]; tid:
// the thread's index in the group that owns the tile.
template <typename R>
__device__ __forceinline__ void warp_site_sum(R v, int slot, double *s_w, int tid) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) s_w[(tid >> 5) * kSiteSlots + slot] = (double)v;
}

// After a barrier that follows every warp_site_sum: sums over the warps of the
// tile's nt threads in order, written as tile blk's row (of nblk) of the (M + 1)
// columns.
__device__ __forceinline__ void write_site_partials(const PassDesc &d, int M, uint64_t base, const double *s_w,
                                                    double *psites, int tid, int nt, size_t blk, size_t nblk) {
  const int nw = (nt + 31) >> 5, K = d.K;
  for (int i = tid; i <= M; i += nt) {
    // a tile bit's weight, or the tile's for an outer spin and the norm (one
    // FP64 sum a thread: they run at 1/64 of the FP32 rate)
    const int from = i < K ? i : kMaxK;
    double v = 0.0;
    for (int w = 0; w < nw; ++w) v += s_w[w * kSiteSlots + from];
    int col = 0;
    if (i < K) {
      col = 1 + d.tile_spin[i];
    } else if (i < M) {
      const int o = i - K;
      if (!((base >> d.outer_pos[o]) & 1ull)) v = 0.0;
      col = 1 + d.outer_spin[o];
    }
    psites[col * nblk + blk] = v;
  }
}

// Whole-state scan (after init or load): per block, the norm and the weight
// with each spin up, as the same (M + 1) columns.
template <typename R>
__global__ void __launch_bounds__(256)
state_sites_kernel(const JobPtrs *__restrict__ jobs, int M, LayoutArg lay) {
  const JobPtrs jp = jobs[blockIdx.y];
  const typename CT<R>::T *__restrict__ psi = static_cast<const typename CT<R>::T *>(jp.psi);
  const uint64_t N = 1ull << M;
  R up[kMaxM], norm = 0;
#pragma unroll
  for (int p = 0; p < kMaxM; ++p) up[p] = 0;
  for (uint64_t y = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; y < N;
       y += (uint64_t)gridDim.x * blockDim.x) {
    const typename CT<R>::T v = psi[y];
    const R pr = v.x * v.x + v.y * v.y;
    norm += pr;
#pragma unroll
    for (int p = 0; p < kMaxM; ++p)
      if (p < M && ((y >> p) & 1ull)) up[p] += pr;
  }
  __shared__ double s_w[kMaxWarps * (kMaxM + 1)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int p = 0; p <= kMaxM; ++p) {
    R v = p < kMaxM ? up[p] : norm;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_w[warp * (kMaxM + 1) + p] = (double)v;
  }
  __syncthreads();
  const size_t nblk = gridDim.x, blk = blockIdx.x;
  for (int i = threadIdx.x; i <= M; i += blockDim.x) {
    const int slot = i < M ? i : kMaxM;
    double v = 0.0;
    for (int w = 0; w < nw; ++w) v += s_w[w * (kMaxM + 1) + slot];
    const int col = i < M ? 1 + lay.logical_of[i] : 0;
    jp.psites[col * nblk + blk] = v;
  }
}

// P of every spin for the entry the preceding reduction recorded (slot
// *step - 1): block q sums columns 0 and 1 + q over the nblk block rows in a
// fixed order, P_q = (2 N_up - N) / N; NaN, as P and the norm, when err (if any)
// says that a wait of the pipelined sweep gave up, which leaves columns unwritten.
__global__ void __launch_bounds__(256)
sites_finalize_kernel(const JobPtrs *__restrict__ jobs, int M, int nblk, const int *err) {
  const JobPtrs jp = jobs[blockIdx.y];
  const int q = blockIdx.x;
  const double *__restrict__ c0 = jp.psites;
  const double *__restrict__ cq = jp.psites + (size_t)(1 + q) * nblk;
  double n = 0.0, u = 0.0;
  for (int r = threadIdx.x; r < nblk; r += blockDim.x) n += c0[r], u += cq[r];
  __shared__ double sn[256], su[256];
  sn[threadIdx.x] = n;
  su[threadIdx.x] = u;
  __syncthreads();
  for (int h = 128; h; h >>= 1) {
    if (threadIdx.x < h) sn[threadIdx.x] += sn[threadIdx.x + h], su[threadIdx.x] += su[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int64_t slot = *jp.step - 1;
    const bool bad = err && *err != 0;
    jp.site_series[slot * M + q] = bad ? __longlong_as_double(0x7ff8000000000000ll) : (2.0 * su[0] - sn[0]) / sn[0];
  }
}

// ---------------------------------------------------------------------------
// Random-phase initial state.
// ---------------------------------------------------------------------------
// kind INIT_ENTANGLED: an independent phase per basis state of spins 2..M.
// kind INIT_PRODUCT: the paper's product state, spin 1 up and every other spin
// l in (|down> + e^{-i phi_l}|up>)/sqrt 2, phi_l = 2 pi u_l with u_l the top 53
// bits of Philox4x32-10(counter = (l-1, 0, 0, 1), key) times 2^-53; the
// amplitude's phase -sum phi_l over the up spins is summed exactly as 64-bit
// fixed-point turns.
enum InitKind { INIT_ENTANGLED = 0, INIT_PRODUCT = 1 };

// amp_d: 2^{-(M-1)/2}, p0: the physical position of spin 1 (both from the
// host: a double exp2 in every thread cost 15 us by itself, FP64 runs at 1/64
// of the FP32 rate).
// orient: logical mask of the first-colour spins of an oriented state (0 for
// a plain one): amplitudes with an odd number of them up are stored (Im, Re).
template <typename R>
__global__ void __launch_bounds__(256)
init_kernel(const JobPtrs *__restrict__ jobs, int M, const __grid_constant__ LayoutArg lay, double amp_d, int p0,
            uint64_t seed0, const uint64_t *__restrict__ seeds, int kind, uint64_t orient) {
  using C = typename CT<R>::T;
  const JobPtrs jp = jobs[blockIdx.y];
  C *__restrict__ psi = static_cast<C *>(jp.psi);
  const uint64_t seed = seeds ? seeds[blockIdx.y] : seed0;
  const R amp = (R)amp_d;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  // product state: turns u_l * 2^64 of each physical bit position (0 for spin 1)
  __shared__ uint64_t s_turns[kMaxM];
  if (kind == INIT_PRODUCT) {
    for (int p = threadIdx.x; p < M; p += blockDim.x) {
      const int q = lay.logical_of[p];
      uint64_t t = 0;
      if (q > 0) {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)q, 0u, 0u, 1u), key);
        t = ((((uint64_t)w.x << 32) | w.y) >> 11) << 11;
      }
      s_turns[p] = t;
    }
    __syncthreads();
  }
  // Index z runs over the 2^(M-1) basis states with spin 1 up, physical bits
  // without spin 1's position p0; its partner with spin 1 down is zero and
  // written beside it.  Bits 0..7 of z come from the thread, the next eb from a
  // loop, the rest from the chunk the block takes, and z's logical index (and
  // product phase) is a sum over its bits, so each group of bits is summed once
  // where it changes.  Bound by Philox and sincos (about 130 instructions a
  // state) next to the store: mapping the bits one by one for every amplitude
  // took twelve times the store's time (complex64, 2^26 amplitudes: 948 us before,
  // 241 us so, 79 us for the store alone; 2^20: 29 us before, 16 us so).
  const int n = M - 1, eb = min(4, max(0, n - 18)), lane = threadIdx.x & 31;
  auto phys = [&](int k) { return k < p0 ? k : k + 1; };  // physical position of bit k of z
  uint64_t x_thr = 1, th_thr = 0;
  for (int k = 0; k < 8 && k < n; ++k)
    if ((threadIdx.x >> k) & 1) {
      x_thr |= 1ull << lay.logical_of[phys(k)];
      if (kind == INIT_PRODUCT) th_thr -= s_turns[phys(k)];
    }
  // the loop's bits: one mask (and product phase) each
  uint64_t x_e[4], th_e[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    x_e[k] = k < eb ? 1ull << lay.logical_of[phys(8 + k)] : 0ull;
    th_e[k] = kind == INIT_PRODUCT && k < eb ? s_turns[phys(8 + k)] : 0ull;
  }
  const uint64_t chunks = n > 8 + eb ? 1ull << (n - 8 - eb) : 1ull, low = (1ull << p0) - 1ull;
  double up = 0;
  for (uint64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
    // the chunk's bits: lane k has bit 8 + eb + k (fewer than 32)
    const int kc = 8 + eb + lane;
    const bool on = kc < n && ((c >> lane) & 1ull);
    const uint64_t xb = on ? 1ull << lay.logical_of[phys(kc)] : 0ull;
    uint64_t th_c = th_thr;
    if (kind == INIT_PRODUCT) {
      uint64_t t = on ? s_turns[phys(kc)] : 0ull;
      for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      th_c -= t;
    }
    const uint64_t x_c = x_thr | __reduce_or_sync(0xffffffffu, (uint32_t)xb) |
                         (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(xb >> 32)) << 32;
    R part = 0;
#pragma unroll 2
    for (int e = 0; e < (1 << eb); ++e) {
      const uint64_t z = (((c << eb) | (uint64_t)e) << 8) | threadIdx.x;
      if (z >= 1ull << n) break;
      uint64_t x = x_c, th = th_c;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((e >> k) & 1) x |= x_e[k], th -= th_e[k];
      C v;
      if (kind == INIT_PRODUCT) {
        const C t = cis_turns(th, (R)0);
        v.x = amp * t.x, v.y = amp * t.y;
      } else {
        const uint64_t r = x >> 1;
        const uint4 w = philox4x32_10(make_uint4((uint32_t)r, (uint32_t)(r >> 32), 0u, 0u), key);
        const uint64_t bits = ((uint64_t)w.x << 32) | w.y;
        C t;
        if (sizeof(R) == 8) {
          // u = top 53 bits * 2^-53 exactly as defined; angle 2 pi u
          double s, cc;
          sincospi(2.0 * ((double)(bits >> 11) * 1.1102230246251565e-16), &s, &cc);
          t.x = (R)cc, t.y = (R)s;
        } else {
          const float2 f = cis_turns(bits, 0.0f);
          t.x = (R)f.x, t.y = (R)f.y;
        }
        v.x = amp * t.x, v.y = amp * t.y;
      }
      part += v.x * v.x + v.y * v.y;
      if (__popcll(x & orient) & 1) {
        const R t = v.x;
        v.x = v.y, v.y = t;
      }
      const uint64_t y = ((z & ~low) << 1) | (z & low);
      C zero;
      zero.x = 0, zero.y = 0;
      psi[y] = zero;
      psi[y | (low + 1ull)] = v;
    }
    up += (double)part;
  }
  reduce_finalize(up, 0.0, jp, true);
}

// ---------------------------------------------------------------------------
// Per-evolve FP64 tables.
// ---------------------------------------------------------------------------
__global__ void coef_kernel(const JobPtrs *__restrict__ jobs, int nb, double dt) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= 2 * nb) return;
  const double *__restrict__ bvals = jobs[blockIdx.y].bvals;
  GateCoef *__restrict__ out = const_cast<GateCoef *>(jobs[blockIdx.y].coefs);
  const double tau = (k & 1) ? dt : 0.5 * dt;
  const double th = 0.5 * bvals[k >> 1] * tau;  // exp(-i tau b (SxSx+SySy)) = cos th - i sin th sigma_x
  const double s = sin(th);
  GateCoef g;
  g.s = s;
  g.t = tan(0.5 * th);
  // FP32 shear pair: among +-2 ulps of the rounded values, the one closest to a
  // rotation, |s (1 + t^2) - 2 t| (zero exactly when s = sin 2 atan t)
  const float t0 = (float)g.t, s1 = (float)s;
  float bt = t0, bs2 = s1;
  double best2 = fabs((double)s1 * (1.0 + (double)t0 * t0) - 2.0 * (double)t0);
  for (int dtt = -2; dtt <= 2; ++dtt)
    for (int ds = -2; ds <= 2; ++ds) {
      const float tf = (t0 == 0.0f) ? t0 : __int_as_float(__float_as_int(t0) + dtt);
      const float sf = (s1 == 0.0f) ? s1 : __int_as_float(__float_as_int(s1) + ds);
      const double def = fabs((double)sf * (1.0 + (double)tf * tf) - 2.0 * (double)tf);
      if (def < best2) best2 = def, bt = tf, bs2 = sf;
    }
  g.tf = bt;
  g.sft = bs2;
  out[k] = g;
}

// Per job: the register-blocked program's ops with their FP32 gate
// coefficients looked up once per dt (the sweep kernels copy them as is).
__global__ void resolve_ops_kernel(const JobPtrs *__restrict__ jobs, const ROp *__restrict__ rops,
                                   int nrops) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nrops) return;
  const JobPtrs &jp = jobs[blockIdx.y];
  const ROp r = rops[i];
  ROpRes o;
  o.kind = r.kind, o.combo = r.combo, o.arg = r.arg, o.pad = 0;
  o.tab = r.kind == OP_GATE ? 0u : (uint32_t)r.coef;  // a diagonal op's table, a round's gates
  o.t = 0.f, o.s = 0.f;
  if (r.kind == OP_GATE) {
    const GateCoef g = jp.coefs[r.coef];
    o.t = g.tf, o.s = g.sft;
  }
  jp.sops[i] = o;
}

// q[v][p][p'] (physical positions): turns of the pair phase -tau_v a_ij / 4 (the
// phase of e^{-i tau a_ij s_i s_j} for s_i s_j = +1/4), as 64-bit fixed point.
// tau_0 = dt/2, tau_1 = dt.
__global__ void diag_kernel(const JobPtrs *__restrict__ jobs, LayoutArg lay, int M, double dt) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= 2 * M * M) return;
  const double *__restrict__ a = jobs[blockIdx.y].a;
  uint64_t *__restrict__ q = const_cast<uint64_t *>(jobs[blockIdx.y].qdiag);
  const int v = k / (M * M), p = (k / M) % M, p2 = k % M;
  uint64_t val = 0;
  if (p != p2) {
    const int i = lay.logical_of[p], j = lay.logical_of[p2];
    const double aij = a[(i < j ? i : j) * M + (i < j ? j : i)];
    const double tau = v ? dt : 0.5 * dt;
    const double t = -tau * aij * 0.039788735772973836;  // 1/(8 pi)
    const double f = t - rint(t);                          // [-1/2, 1/2] turns
    val = ((uint64_t)llrint(f * 9.223372036854775808e18)) << 1;
  }
  q[k] = val;
}

// A job's diagonal tables (see DiagTab), from the pair phases of diag_kernel:
// one thread per entry, the sums exact modulo 2^64.
__global__ void diag_tab_kernel(const JobPtrs *__restrict__ jobs, const __grid_constant__ DiagTab t, int M) {
  const JobPtrs &jp = jobs[blockIdx.y];
  const int nr = 1 << t.rb, nt = 1 << t.L;
  const int e = blockIdx.x * blockDim.x + threadIdx.x, v = e >= t.words, i = e - v * t.words;
  if (e >= 2 * t.words) return;
  const uint64_t *__restrict__ q = jp.qdiag + (size_t)v * M * M;
  // the pair phases among n tile bits from bit b0, signs from the bits of x
  auto pairs = [&](int b0, int n, int x) {
    uint64_t s = 0;
    for (int a = 0; a < n; ++a)
      for (int b = a + 1; b < n; ++b) {
        const uint64_t y = q[t.pos[b0 + a] * M + t.pos[b0 + b]];
        s += (((x >> a) ^ (x >> b)) & 1) ? (0ull - y) : y;
      }
    return s;
  };
  uint64_t r = 0;
  if (i < nr) {
    r = pairs(t.L, t.rb, i);
  } else if (i < nr + nt) {
    r = pairs(0, t.L, i - nr);
  } else {
    const int k = ((i - nr) >> t.L) - 1, x = (i - nr) & (nt - 1);
    for (int b = 0; b < t.L; ++b) {
      const uint64_t y = q[t.pos[t.L + k] * M + t.pos[b]];
      r += ((x >> b) & 1) ? y : (0ull - y);
    }
  }
  jp.dtab[e] = r;
}

// ---------------------------------------------------------------------------
// One sweep.  Each block owns one tile: it loads the tile's 2^K amplitudes
// into shared memory, applies the pass's ops in order and stores the tile.
// ---------------------------------------------------------------------------
// A gate as two real plane rotations: exp(-i theta sigma_x) maps
// (Re a, Im b) and (Re b, Im a) each by [[c, s], [-s, c]], c = cos theta,
// s = sin theta, and each rotation is three shears x += t y, y -= s x,
// x += t y with t = tan(theta/2): three FMAs per plane.  A shear has
// determinant one whatever t and s are rounded to, so rounding leaves no
// uniform gain or loss of norm.
__device__ __forceinline__ void shear_plane(float &x, float &y, float t, float s) {
  const float v = fmaf(t, y, x);
  y = fmaf(-s, v, y);
  x = fmaf(t, y, v);
}
__device__ __forceinline__ void shear_plane(double &x, double &y, double t, double s) {
  const double v = fma(t, y, x);
  y = fma(-s, v, y);
  x = fma(t, y, v);
}

// The plain sweep: tiles below ten spins, and the complex128 all-site readout.
// A gate takes the tile's pairs from shared memory, real and imaginary parts
// apart, one thread a plane (half the FP64 chain, and twice the warps, of a
// thread a pair), with the pass's ops and coefficients staged there first.  A
// 14-spin complex128 sweep is bound by its gates' latency: 0.75 us a gate with
// op and coefficients read from global memory at each gate and both planes in
// one thread, 0.45 us so (the 26-gate sweep 23 -> 18 us with its launch, the
// 400-step job 15.0 -> 10.3 ms with the sweeps chained too).
// Two blocks of 512 threads share an SM, so 64 registers: the readout keeps five
// sums for the bits a thread walks, not one for every tile bit, which took 86 and
// an SM a block at a time (20-spin complex128 all-site chain 246 -> 208 us a step).
constexpr int kMaxPlainOps = 192;  // every pair of 14 tile bits twice, and the element-wise ops
static_assert(kMaxK * (kMaxK - 1) + 4 <= kMaxPlainOps, "ops of a pass");

template <typename R, bool SITES>
__global__ void __launch_bounds__(512, 2)
sweep_kernel(const JobPtrs *__restrict__ jobs, const PassDesc *__restrict__ pdesc,
             const Op *__restrict__ ops, int M) {
  using C = typename CT<R>::T;
  struct SOp {
    uint8_t kind, u, v, arg;
    R t, s;
  };
  const JobPtrs jp = jobs[blockIdx.y];
  C *__restrict__ psi = static_cast<C *>(jp.psi);
  const uint64_t *__restrict__ qdiag = jp.qdiag;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PassDesc d;
  __shared__ uint64_t sH[kMaxK];
  __shared__ uint64_t sQ[kMaxK * kMaxK];
  __shared__ uint64_t sOut;
  __shared__ double s_w[SITES ? kMaxWarps * kSiteSlots : 1];
  __shared__ SOp s_ops[kMaxPlainOps];
  {
    const int nwords = (int)(sizeof(PassDesc) / 4);
    for (int w = threadIdx.x; w < nwords; w += blockDim.x)
      reinterpret_cast<int *>(&d)[w] = reinterpret_cast<const int *>(pdesc)[w];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < d.nops; k += blockDim.x) {
    const Op op = ops[d.op0 + k];
    SOp o{op.kind, op.u, op.v, op.arg, 0, 0};
    if (op.kind == OP_GATE) {
      const GateCoef g = jp.coefs[op.coef];
      o.t = sizeof(R) == 8 ? (R)g.t : (R)g.tf;
      o.s = sizeof(R) == 8 ? (R)g.s : (R)g.sft;
    }
    s_ops[k] = o;
  }
  const int K = d.K;
  const int nt = blockDim.x, tid = threadIdx.x;
  const int lognt = 31 - __clz(nt);
  const int L = lognt < K ? lognt : K;  // tile bits taken from the thread index
  const uint32_t T = 1u << K;
  R *const re = reinterpret_cast<R *>(smem_raw), *const im = re + T;
  const uint64_t base = deposit_bits(blockIdx.x, d.outer_pos, M - K);
  const uint64_t off_lo = deposit_bits(tid, d.tile_pos, L);
  auto offset = [&](uint32_t t) -> uint64_t {
    uint64_t o = off_lo;
    for (int q = L; q < K; ++q) o |= (uint64_t)((t >> q) & 1u) << d.tile_pos[q];
    return o;
  };
  grid_wait();
  grid_go();
  for (uint32_t t = tid; t < T; t += nt) {
    const C a = psi[base + offset(t)];
    re[t] = a.x, im[t] = a.y;
  }
  __syncthreads();

  R up = 0, dn = 0;
  for (int k = 0; k < d.nops; ++k) {
    const SOp op = s_ops[k];
    if (op.kind == OP_GATE) {
      const int lo = op.u < op.v ? op.u : op.v, hi = op.u < op.v ? op.v : op.u;
      const uint32_t bu = 1u << op.u, bv = 1u << op.v;
      // task w: pair w mod T/4 and the plane (re a, im b) or (re b, im a)
      for (uint32_t w = tid; w < (T >> 1); w += nt) {
        const bool second = w >= (T >> 2);
        const uint32_t t0 = insert_zero(insert_zero(second ? w - (T >> 2) : w, lo), hi);
        R *const px = re + (t0 | (second ? bv : bu)), *const py = im + (t0 | (second ? bu : bv));
        R x = *px, y = *py;
        shear_plane(x, y, op.t, op.s);
        *px = x, *py = y;
      }
      __syncthreads();
    } else if (op.kind == OP_DIAG) {
      // Theta(x) = sum_{p<p'} q_pp' sigma_p sigma_p' (mod 2^64), split into
      // outer-outer, outer-tile and tile-tile parts.
      const uint64_t *q = qdiag + (size_t)op.arg * M * M;
      const int nout = M - K;
      if (tid < K) {
        const int p = d.tile_pos[tid];
        uint64_t h = 0;
        for (int o = 0; o < nout; ++o) {
          const int po = d.outer_pos[o];
          const uint64_t v = q[p * M + po];
          h += ((base >> po) & 1ull) ? v : (0ull - v);
        }
        sH[tid] = h;
      } else if (tid == K) {
        uint64_t s = 0;
        for (int o = 0; o < nout; ++o)
          for (int o2 = o + 1; o2 < nout; ++o2) {
            const int p = d.outer_pos[o], p2 = d.outer_pos[o2];
            const uint64_t v = q[p * M + p2];
            s += (((base >> p) ^ (base >> p2)) & 1ull) ? (0ull - v) : v;
          }
        sOut = s;
      }
      for (int w = tid; w < K * K; w += nt) {
        const int a = w / K, b = w % K;
        sQ[w] = q[d.tile_pos[a] * M + d.tile_pos[b]];
      }
      __syncthreads();
      // per-thread part: tile bits 0..L-1 come from tid
      uint64_t thr = sOut;
      for (int a = 0; a < L; ++a) {
        const uint64_t ba = (tid >> a) & 1u;
        thr += ba ? sH[a] : (0ull - sH[a]);
        for (int b = a + 1; b < L; ++b)
          thr += (ba ^ ((tid >> b) & 1u)) ? (0ull - sQ[a * K + b]) : sQ[a * K + b];
      }
      for (uint32_t t = tid; t < T; t += nt) {
        uint64_t th = thr;
        for (int a = L; a < K; ++a) {
          const uint32_t ba = (t >> a) & 1u;
          uint64_t f = sH[a];
          for (int b = 0; b < L; ++b)
            f += ((tid >> b) & 1u) ? sQ[b * K + a] : (0ull - sQ[b * K + a]);
          th += ba ? f : (0ull - f);
          for (int b = a + 1; b < K; ++b)
            th += (ba ^ ((t >> b) & 1u)) ? (0ull - sQ[a * K + b]) : sQ[a * K + b];
        }
        C a;
        a.x = re[t], a.y = im[t];
        a = cmul(a, cis_turns(th, (R)0));
        re[t] = a.x, im[t] = a.y;
      }
      __syncthreads();
    } else if (op.kind == OP_REDUCE) {
      // weights by the tile bits a thread walks, L and up (L is nine, or K - 1 or K below that)
      R tsum = 0, uhi[kMaxK - 9];
#pragma unroll
      for (int e = 0; e < kMaxK - 9; ++e) uhi[e] = 0;
      for (uint32_t t = tid; t < T; t += nt) {
        const R pr = re[t] * re[t] + im[t] * im[t];
        const uint64_t bit = d.site_tile >= 0 ? ((t >> d.site_tile) & 1u)
                                              : ((base >> d.site_pos) & 1ull);
        if (bit) up += pr;
        else dn += pr;
        if constexpr (SITES) {
          tsum += pr;
#pragma unroll
          for (int e = 0; e < kMaxK - 9; ++e)
            if ((t >> (L + e)) & 1u) uhi[e] += pr;
        }
      }
      if constexpr (SITES) {
        // tile bits below L come from the thread index: the thread's whole sum
#pragma unroll
        for (int q = 0; q < kMaxK; ++q)
          warp_site_sum<R>(q < L ? (((tid >> q) & 1) ? tsum : (R)0) : q == L ? uhi[0] : q > 9 ? uhi[q - 9] : (R)0,
                           q, s_w, tid);
        warp_site_sum<R>(tsum, kMaxK, s_w, tid);
      }
      __syncthreads();  // later ops overwrite the tile
    }
  }
  // output tile bit q holds the spin that input tile bit perm[q] held
  for (uint32_t t = tid; t < T; t += nt) {
    uint32_t ti = t;
    if (d.relabel) {
      ti = 0;
      for (int q = 0; q < K; ++q) ti |= ((t >> q) & 1u) << d.perm[q];
    }
    C a;
    a.x = re[ti], a.y = im[ti];
    psi[base + offset(t)] = a;
  }
  if constexpr (SITES)
    if (d.has_reduce) write_site_partials(d, M, base, s_w, jp.psites, tid, nt, blockIdx.x, gridDim.x);
  if (d.has_reduce) reduce_finalize((double)up, (double)dn, jp, false);
}

// Gather amplitudes at LOGICAL indices into a staging buffer (FP64 pairs); the
// physical index is formed here (loading and reading 2^18 amplitudes: 4.5 ms
// with a host loop over the bits of every index, 0.4 ms so).  orient: physical positions of the first-colour
// spins of an oriented state (0 for a plain one); those amplitudes stored
// (Im, Re) are read back as (Re, Im).
__device__ __forceinline__ uint64_t to_physical(uint64_t x, int M, const LayoutArg &lay) {
  uint64_t y = 0;
  for (int p = 0; p < M; ++p) y |= ((x >> lay.logical_of[p]) & 1ull) << p;
  return y;
}

template <typename R>
__global__ void gather_kernel(const typename CT<R>::T *__restrict__ psi, const int64_t *__restrict__ idx, int64_t n,
                              double2 *out, int M, const __grid_constant__ LayoutArg lay, uint64_t orient) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t y = to_physical((uint64_t)idx[k], M, lay);
    const typename CT<R>::T v = psi[y];
    const bool sw = __popcll(y & orient) & 1;
    out[k] = sw ? make_double2((double)v.y, (double)v.x) : make_double2((double)v.x, (double)v.y);
  }
}

// Scatter the amplitudes of logical indices first .. first + n - 1.
template <typename R>
__global__ void scatter_kernel(typename CT<R>::T *__restrict__ psi, uint64_t first, int64_t n,
                               const double2 *__restrict__ in, int M, const __grid_constant__ LayoutArg lay,
                               uint64_t orient) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t y = to_physical(first + (uint64_t)k, M, lay);
    typename CT<R>::T v;
    const bool sw = __popcll(y & orient) & 1;
    v.x = (R)(sw ? in[k].y : in[k].x);
    v.y = (R)(sw ? in[k].x : in[k].y);
    psi[y] = v;
  }
}

// Polarization/norm of the whole state (after a load).
template <typename R>
__global__ void __launch_bounds__(256)
observe_kernel(const JobPtrs *__restrict__ jobs, int M, int site_pos) {
  const JobPtrs jp = jobs[blockIdx.y];
  const typename CT<R>::T *__restrict__ psi = static_cast<const typename CT<R>::T *>(jp.psi);
  const uint64_t N = 1ull << M;
  double up = 0, dn = 0;
  for (uint64_t y = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; y < N;
       y += (uint64_t)gridDim.x * blockDim.x) {
    const typename CT<R>::T v = psi[y];
    const double pr = (double)v.x * v.x + (double)v.y * v.y;
    if ((y >> site_pos) & 1ull) up += pr;
    else dn += pr;
  }
  reduce_finalize(up, dn, jp, true);
}

// ===========================================================================
// Register-blocked sweep (complex64).  The tile lives in shared memory with
// an XOR swizzle; global<->shared copies are 16-byte cp.async loads and
// 16-byte stores; between them the pass runs as a sequence of phases, each a
// register-resident 32-amplitude subcube per thread (see PhaseDesc).
// ===========================================================================
namespace sw2 {

// Shared-memory slot of tile index t: the low four bits are XORed with bits
// 4-7, 8-11 and 12-15.  Linear over XOR, so slot(a ^ b) = slot(a) ^ slot(b);
// lanes that differ in four tile bits of distinct residues mod 4 hit 16
// distinct 8-byte bank pairs.
__device__ __forceinline__ uint32_t slot(uint32_t t) {
  return t ^ (((t >> 4) ^ (t >> 8) ^ (t >> 12)) & 15u);
}

// Packed FP32x2 arithmetic on 64-bit registers (two lanes per instruction,
// sm_100 and later).  A pack holds (low lane, high lane) = (bit clear, bit set).
typedef unsigned long long u64;
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 pack2(float lo, float hi) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(u64 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// A thread's 2^RB amplitudes in a phase are NP = 2^(RB-1) packs: RE[j] =
// (re with register bit 0 clear, re with it set), IM[j] likewise, j = register
// bits 1..RB-1.  Register bit 0 (the "pack bit") is chosen by the host as the
// bit with the fewest gates in the phase.

// In-place x += a * b on packed FP32x2 (the accumulator keeps its register,
// so a gate leaves every pack where it found it).
__device__ __forceinline__ void fma2_acc(u64 &x, u64 a, u64 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(x) : "l"(a), "l"(b));
}

// Three in-place shears on the plane (high lane of P, low lane of Q) or
// (low lane of P, high lane of Q): X += t Y, Y += n X, X += t Y.
__device__ __forceinline__ void shear_hi_lo(u64 &P, u64 &Q, float t, float n) {
  asm("{\n\t.reg .f32 pl, ph, ql, qh;\n\t"
      "mov.b64 {pl, ph}, %0;\n\tmov.b64 {ql, qh}, %1;\n\t"
      "fma.rn.f32 ph, %2, ql, ph;\n\tfma.rn.f32 ql, %3, ph, ql;\n\tfma.rn.f32 ph, %2, ql, ph;\n\t"
      "mov.b64 %0, {pl, ph};\n\tmov.b64 %1, {ql, qh};\n\t}"
      : "+l"(P), "+l"(Q) : "f"(t), "f"(n));
}
__device__ __forceinline__ void shear_lo_hi(u64 &P, u64 &Q, float t, float n) {
  asm("{\n\t.reg .f32 pl, ph, ql, qh;\n\t"
      "mov.b64 {pl, ph}, %0;\n\tmov.b64 {ql, qh}, %1;\n\t"
      "fma.rn.f32 pl, %2, qh, pl;\n\tfma.rn.f32 qh, %3, pl, qh;\n\tfma.rn.f32 pl, %2, qh, pl;\n\t"
      "mov.b64 %0, {pl, ph};\n\tmov.b64 %1, {ql, qh};\n\t}"
      : "+l"(P), "+l"(Q) : "f"(t), "f"(n));
}

// Gate on register bits (JU + 1, JV + 1): two amplitude pairs per packed
// instruction, same three-shear update as shear_plane, in place.
template <int NP, int JU, int JV>
__device__ __forceinline__ void gate_packed(u64 (&RE)[NP], u64 (&IM)[NP], float t, float s) {
  const u64 t2 = pack2(t, t), n2 = pack2(-s, -s);
  // plane (Re a, Im b) = (RE[j], IM[k]); plane (Re b, Im a) = (RE[k], IM[j]);
  // each shear step over every plane of the gate before the next (independent
  // instructions back to back)
#pragma unroll
  for (int j = 0; j < NP; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0) {
      const int k = j ^ (1 << JU) ^ (1 << JV);
      fma2_acc(RE[j], t2, IM[k]);
      fma2_acc(RE[k], t2, IM[j]);
    }
#pragma unroll
  for (int j = 0; j < NP; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0) {
      const int k = j ^ (1 << JU) ^ (1 << JV);
      fma2_acc(IM[k], n2, RE[j]);
      fma2_acc(IM[j], n2, RE[k]);
    }
#pragma unroll
  for (int j = 0; j < NP; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0) {
      const int k = j ^ (1 << JU) ^ (1 << JV);
      fma2_acc(RE[j], t2, IM[k]);
      fma2_acc(RE[k], t2, IM[j]);
    }
}

// Gate on the pack bit and register bit JV + 1: the pair is the high lane of
// pack j (JV clear) and the low lane of pack j + 2^JV; scalar arithmetic.
template <int NP, int JV>
__device__ __forceinline__ void gate_packbit(u64 (&RE)[NP], u64 (&IM)[NP], float t, float s) {
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    if (((j >> JV) & 1) == 0) {
      const int k = j | (1 << JV);
      // a = high lanes of pack j, b = low lanes of pack k:
      // plane (Re a, Im b) = (RE[j].hi, IM[k].lo); plane (Re b, Im a) = (RE[k].lo, IM[j].hi)
      shear_hi_lo(RE[j], IM[k], t, -s);
      shear_lo_hi(RE[k], IM[j], t, -s);
    }
  }
}

// Gate on the register bits (ku, kv) of combo C = index of the pair ku < kv in
// lexicographic order; the first RB - 1 pairs have the pack bit (ku = 0).
template <int NP, int C>
__device__ __forceinline__ void gate_of(u64 (&RE)[NP], u64 (&IM)[NP], float t, float s) {
  constexpr int RB = NP == 16 ? 5 : 6;
  static_assert(NP == 1 << (RB - 1), "five or six register bits");
  if constexpr (C < RB - 1) {
    gate_packbit<NP, C>(RE, IM, t, s);
  } else {
    constexpr int D = C - (RB - 1);  // among the pairs of bits 1..RB-1
    constexpr int U = D < RB - 2 ? 0 : D < 2 * RB - 5 ? 1 : D < 3 * RB - 9 ? 2 : 3;
    constexpr int V = D - (U * (2 * (RB - 1) - U - 1)) / 2 + U + 1;
    static_assert(U < V && V < RB - 1, "a pair of register bits");
    gate_packed<NP, U, V>(RE, IM, t, s);
  }
}

// The gate of a pair by a jump (sparse passes of the pipelined sweep).
__device__ __forceinline__ void gate_combo(u64 (&RE)[32], u64 (&IM)[32], int combo, float t, float s) {
  switch (combo) {
    case 0: gate_of<32, 0>(RE, IM, t, s); break;
    case 1: gate_of<32, 1>(RE, IM, t, s); break;
    case 2: gate_of<32, 2>(RE, IM, t, s); break;
    case 3: gate_of<32, 3>(RE, IM, t, s); break;
    case 4: gate_of<32, 4>(RE, IM, t, s); break;
    case 5: gate_of<32, 5>(RE, IM, t, s); break;
    case 6: gate_of<32, 6>(RE, IM, t, s); break;
    case 7: gate_of<32, 7>(RE, IM, t, s); break;
    case 8: gate_of<32, 8>(RE, IM, t, s); break;
    case 9: gate_of<32, 9>(RE, IM, t, s); break;
    case 10: gate_of<32, 10>(RE, IM, t, s); break;
    case 11: gate_of<32, 11>(RE, IM, t, s); break;
    case 12: gate_of<32, 12>(RE, IM, t, s); break;
    case 13: gate_of<32, 13>(RE, IM, t, s); break;
    default: gate_of<32, 14>(RE, IM, t, s); break;
  }
}

// One round of a phase's gates: the pairs of `mask` in ascending order of C,
// coefficients from consecutive ops.  Straight code with a test before each
// pair: gates that run follow each other in the instruction stream, and the
// next gate's coefficients load while this one computes.  A jump per gate (a
// switch on the pair) took about 280 cycles a gate for a lone warp, most of it
// the jump and the instruction fetch after it; a walk takes about 320 cycles and
// 57 a gate (clock64 around it in resident_kernel, five register bits: 519 cycles
// for 3.6 gates on the 10-spin ladder, 649 for 5.7 on the 12-spin star; a six-gate
// phase of a 2^12 tile 2850 -> 1890).  One walk direction only: with a second,
// descending copy the sweep's code outgrew the instruction cache (stalls on
// instructions 1.7 per issue against 0.3, 15 % slower on ladders); the phase
// planner orders the register bits so that one ascending walk takes nearly every
// phase.
template <int NP, int C = 0>
__device__ __forceinline__ void run_round(u64 (&RE)[NP], u64 (&IM)[NP], uint32_t mask, const ROpRes *op, float2 ts) {
  constexpr int RB = NP == 16 ? 5 : 6, NC = RB * (RB - 1) / 2;
  if ((mask >> C) & 1u) {
    const float2 now = ts;
    ++op;
    ts = make_float2(op->t, op->s);
    gate_of<NP, C>(RE, IM, now.x, now.y);
  }
  if constexpr (C + 1 < NC) run_round<NP, C + 1>(RE, IM, mask, op, ts);
}

// lowest set bit of a compile-time g in 1..31 (Gray-code walk)
__host__ __device__ constexpr int ctz5(int g) {
  return (g & 1) ? 0 : (g & 2) ? 1 : (g & 4) ? 2 : (g & 8) ? 3 : 4;
}
// same for g in 1..63; gray(g) = g ^ (g >> 1) differs from gray(g - 1) in bit
// ctz6(g), which gray(g) has set when gray_up(g)
__host__ __device__ constexpr int ctz6(int g) { return (g & 31) ? ctz5(g & 31) : 5; }
__host__ __device__ constexpr bool gray_up(int g) { return (((g ^ (g >> 1)) >> ctz6(g)) & 1) != 0; }

// 8-byte asynchronous global->shared copy (one amplitude): the swizzle may
// move an amplitude pair to an odd slot, so 16-byte copies would misalign.
__device__ __forceinline__ void cp_async8(uint32_t smem_addr, const void *gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t smem_addr, const void *gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}


// Barrier of the threads a tile's phases run on (the whole block).
struct SyncBlock {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// Origin of tile `blk` of a pass: lane k places bit k of the tile index at
// outer_pos[k] (M - K < 32 outer bits), a warp OR-reduction assembles the
// offset.  Called by whole warps.
__device__ __forceinline__ uint64_t tile_origin(unsigned blk, const PassDesc &d, int M) {
  const int lane = threadIdx.x & 31;
  const uint64_t c = lane < M - d.K ? (uint64_t)((blk >> lane) & 1u) << d.outer_pos[lane] : 0ull;
  const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)c);
  const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(c >> 32));
  return ((uint64_t)hi << 32) | lo;
}

// Global -> shared copy of a tile by the 2^lognt threads tid of its group
// (8-byte async copies; 16 consecutive threads read one 128-byte run).
// Input amplitude a = tid + nt * e: tile bits 0..lognt-1 from tid, the RB high
// bits from e, e walked in Gray-code order in runs of eight: each copy moves
// the source by +-2^tile_pos (a compile-time sign) and the destination slot by
// one XOR (the slot is XOR-linear); each run starts afresh from the thread's
// origin, so the address chains stay short.
template <int RB>
__device__ __forceinline__ void load_tile(const float2 *psi, uint64_t base, const PassDesc &d, int tid,
                                          int lognt, uint32_t sbase) {
  constexpr int NA = 1 << RB;
  uint64_t off_amp_lo = 0;
  for (int k = 0; k < lognt; ++k)
    if ((tid >> k) & 1) off_amp_lo |= 1ull << d.tile_pos[k];
  int64_t dg[RB];
  uint32_t ds[RB];
#pragma unroll
  for (int k = 0; k < RB; ++k) {
    dg[k] = (int64_t)8 << d.tile_pos[lognt + k];
    ds[k] = slot(1u << (lognt + k)) << 3;
  }
  const char *src0 = reinterpret_cast<const char *>(psi + base + off_amp_lo);
  const uint32_t sb0 = slot((uint32_t)tid) << 3;
  const char *src = src0;
  uint32_t sb = sb0;
#pragma unroll
  for (int g = 0; g < NA; ++g) {
    if ((g & 7) == 0) {
      src = src0, sb = sb0;
#pragma unroll
      for (int k = 0; k < RB; ++k)
        if (((g ^ (g >> 1)) >> k) & 1) src += dg[k], sb ^= ds[k];
    } else {
      const int k = ctz6(g);
      src += gray_up(g) ? dg[k] : -dg[k];
      sb ^= ds[k];
    }
    cp_async8(sbase + sb, src);
  }
}

// L2 prefetch of the tile at origin base2: one 128-byte run (tile bits 0..3,
// the low physical bits) per request; run r = tid + nt * i (tile bits 4.. of
// its first amplitude): bits from tid once, then the RB - 4 high bits per run.
template <int RB>
__device__ __forceinline__ void prefetch_tile(const float2 *psi, uint64_t base2, const PassDesc &d, int tid,
                                              int lognt) {
  uint64_t ot = base2;
  for (int b = 0; b < lognt; ++b)
    if ((tid >> b) & 1) ot |= 1ull << d.tile_pos[4 + b];
#pragma unroll
  for (int i = 0; i < (1 << (RB - 4)); ++i) {
    uint64_t off = ot;
#pragma unroll
    for (int b = 0; b < RB - 4; ++b)
      if ((i >> b) & 1) off |= 1ull << d.tile_pos[4 + lognt + b];
    asm volatile("prefetch.global.L2 [%0];" ::"l"(psi + off));
  }
}

// Tile index of this thread's subcube origin in phase ph (register bits clear).
__device__ __forceinline__ uint32_t thread_origin(const PhaseDesc &ph, int tid, int lognt) {
  uint32_t t0 = 0;
  for (int k = 0; k < 5; ++k) t0 |= ((uint32_t)(tid >> k) & 1u) << ph.lanes[k];
  for (int k = 0; k < lognt - 5; ++k) t0 |= ((uint32_t)(tid >> (5 + k)) & 1u) << ph.warps[k];
  return t0;
}

// For each variant v of the pass's diagonal ops: fields of the outer spins on a
// tile's bits, sH[v kFieldStride + t] = sum_o sigma_o q_to, and their own part of
// Theta at t = K (exact modulo 2^64), by the 2^lognt threads tid of the group:
// eight lanes share each entry, so the loads of a row are in flight together.
// The group's next barrier publishes them.
__device__ __forceinline__ void diag_fields(const PassDesc &d, uint64_t base, int tid, int lognt, int M,
                                            const uint64_t *__restrict__ qdiag, uint64_t *sH) {
  const int K = d.K, nout = M - K, part = tid & 7;
#pragma unroll 1
  for (int var = 0; var < 2; ++var) {
    if (!((d.diag >> var) & 1)) continue;
    const uint64_t *__restrict__ q = qdiag + (size_t)var * M * M;
    for (int t0 = 0; t0 <= K; t0 += 1 << (lognt - 3)) {
      const int t = t0 + (tid >> 3);
      uint64_t v = 0;
      if (t < K) {
        const int row = d.tile_pos[t] * M;
        for (int o = part; o < nout; o += 8) {
          const int po = d.outer_pos[o];
          const uint64_t x = q[row + po];
          v += ((base >> po) & 1ull) ? x : (0ull - x);
        }
      } else if (t == K) {
        for (int o = part; o < nout; o += 8) {
          const int pa = d.outer_pos[o];
          uint64_t r = 0;
          for (int o2 = o + 1; o2 < nout; ++o2) {
            const int pb = d.outer_pos[o2];
            const uint64_t x = q[pa * M + pb];
            r += ((base >> pb) & 1ull) ? x : (0ull - x);
          }
          v += ((base >> pa) & 1ull) ? r : (0ull - r);
        }
      }
#pragma unroll
      for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (part == 0 && t <= K) sH[var * kFieldStride + t] = v;
    }
  }
}

// e^{i theta} of two angles given as turns x 2^32 plus an eighth of a turn:
// (re, im) packed.  The top two bits are the quarter turn, the others minus the
// eighth the remainder y x pi/4, |y| <= 1, whose sine and cosine are minimax
// polynomials in y^2 (Remez exchange; pi/4 split in two floats, the cosine's
// leading coefficient rounded before the others were fitted, so that neither
// the angle's scale nor the modulus is biased).  Errors against 64 bits over
// all remainders: rms 1.44e-8 (sine) and 1.87e-8 (cosine), where correctly
// rounded values have 1.42e-8 and 1.81e-8.
__device__ __forceinline__ void cis_eighths(uint32_t a0, uint32_t a1, u64 &re, u64 &im) {
  const float f0 = (float)((int)(a0 & 0x3fffffffu) - 0x20000000);
  const float f1 = (float)((int)(a1 & 0x3fffffffu) - 0x20000000);
  const float k = 1.862645149230957e-09f;  // 2^-29
  const u64 y = mul2(pack2(f0, f1), pack2(k, k)), z = mul2(y, y);
  auto c2 = [](float v) { return pack2(v, v); };
  u64 p = fma2(c2(-3.58774269e-05f), z, c2(0.00248987228f));
  p = fma2(p, z, c2(-0.0807453692f));
  p = fma2(p, z, c2(-3.26817364e-08f));
  const float2 s = unpack2(fma2(y, c2(0.785398185f), mul2(p, y)));
  u64 q = fma2(c2(3.50271148e-06f), z, c2(-0.000325882982f));
  q = fma2(q, z, c2(0.0158542898f));
  q = fma2(q, z, c2(-0.308425128f));
  const float2 c = unpack2(fma2(q, z, c2(1.0f)));
  // quarter turns 0..3: (c, s), (-s, c), (-c, -s), (s, -c)
  const bool w0 = (a0 & 0x40000000u) != 0, w1 = (a1 & 0x40000000u) != 0;
  const uint32_t r0 = __float_as_uint(w0 ? s.x : c.x) ^ ((a0 ^ (a0 << 1)) & 0x80000000u);
  const uint32_t r1 = __float_as_uint(w1 ? s.y : c.y) ^ ((a1 ^ (a1 << 1)) & 0x80000000u);
  const uint32_t i0 = __float_as_uint(w0 ? c.x : s.x) ^ (a0 & 0x80000000u);
  const uint32_t i1 = __float_as_uint(w1 ? c.y : s.y) ^ (a1 & 0x80000000u);
  re = pack2(__uint_as_float(r0), __uint_as_float(r1));
  im = pack2(__uint_as_float(i0), __uint_as_float(i1));
}

// The diagonal op e^{-i tau D} on a tile in shared memory, by the 2^lognt
// threads tid of the group: thread tid takes the amplitudes t = tid + 2^lognt e,
// e = 0..2^RB - 1.  Theta(t) is the table's thread part, plus the fields on the
// thread's bits, plus sum_k sigma_k g_k + (register part e) over the RB high
// tile bits, g_k the field of the thread's bits and of the outer spins on bit
// k: two 64-bit additions an amplitude (exact), the register part one
// broadcast load for two.  A loop over eight amplitudes at a time, out of
// line: bound by latency and, when unrolled over all 2^RB, by instruction
// fetch (its code runs once a tile and no longer fits the instruction cache
// next to the gates; applied inside a phase's registers it also spilled, 0.73
// of the speed on ladders that never run it).  One tile of 2^12, a warp per
// scheduler: about 10^4 cycles untabulated and unrolled, 4300 so.
// ORIENT: amplitudes of odd orientation are stored (Im, Re) and take the
// conjugate phase (the stored word is i conj(psi), and i conj(psi e^{ia}) =
// i conj(psi) e^{-ia}).
template <int RB, bool ORIENT>
__device__ __noinline__ void diag_tile(float2 *tile2, const uint64_t *__restrict__ tab, const uint64_t *sH, int K,
                                       int tid, int lognt, uint32_t black, uint32_t outer_par) {
  const uint64_t *__restrict__ tthr = tab + (1 << RB) + tid;
  uint64_t g[RB], base = sH[K] + tthr[0] + (1ull << 61);
#pragma unroll
  for (int k = 0; k < RB; ++k) g[k] = sH[lognt + k] + tthr[(size_t)(k + 1) << lognt];
#pragma unroll
  for (int b = 0; b < kMaxK - 5; ++b)
    if (b < lognt) {
      const uint64_t h = sH[b];
      base += ((tid >> b) & 1) ? h : (0ull - h);
    }
  uint32_t ds[RB];
#pragma unroll
  for (int k = 0; k < RB; ++k) base -= g[k], g[k] += g[k], ds[k] = slot(1u << (lognt + k)) << 3;
  char *const tb = reinterpret_cast<char *>(tile2);
  const uint32_t o0 = slot((uint32_t)tid) << 3;
#pragma unroll 1
  for (int hi = 0; hi < (1 << (RB - 3)); ++hi) {
    uint64_t lin = base;
    uint32_t o = o0;
#pragma unroll
    for (int k = 3; k < RB; ++k)
      if ((hi >> (k - 3)) & 1) lin += g[k], o ^= ds[k];
    const ulonglong2 *__restrict__ treg = reinterpret_cast<const ulonglong2 *>(tab) + 4 * hi;
    float2 v[8];
    uint32_t oe[8];
    u64 c[4], sn[4];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      oe[e] = o ^ ((e & 1) ? ds[0] : 0) ^ ((e & 2) ? ds[1] : 0) ^ ((e & 4) ? ds[2] : 0);
      v[e] = *reinterpret_cast<const float2 *>(tb + oe[e]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // amplitudes e = 8 hi + 2 i and the next one
      const uint64_t l = lin + ((i & 1) ? g[1] : 0) + ((i & 2) ? g[2] : 0);
      const ulonglong2 t = treg[i];
      cis_eighths((uint32_t)((l + t.x) >> 32), (uint32_t)((l + g[0] + t.y) >> 32), c[i], sn[i]);
      if constexpr (ORIENT) {
        const uint32_t e = 8u * hi + 2u * i, ta = (uint32_t)tid | (e << lognt);
        const uint32_t pa = (__popc(ta & black) ^ outer_par) & 1u, pb = pa ^ ((black >> lognt) & 1u);
        sn[i] ^= ((u64)pa << 31) | ((u64)pb << 63);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 cc = unpack2(c[i]), ss = unpack2(sn[i]);
      *reinterpret_cast<float2 *>(tb + oe[2 * i]) = cmul(v[2 * i], make_float2(cc.x, ss.x));
      *reinterpret_cast<float2 *>(tb + oe[2 * i + 1]) = cmul(v[2 * i + 1], make_float2(cc.y, ss.y));
    }
  }
}

// Register-blocked phases of an oriented program (see Orientation): the
// thread's 2^RB amplitudes are NA words P[j], j = register bits (the first NB
// = ph.nb of them of the first colour), each the stored (Re, Im) or (Im, Re)
// pair as is.  A gate on register bits (JU < NB <= JV) updates the pairs (j, k = j ^
// 2^JU ^ 2^JV), j with bit JU set, by P[j] += T P[k]; P[k] += S P[j]; P[j] +=
// T P[k] (packed FP32x2), with T = (t, -t), S = (-s, s) when amplitude j is
// stored (Re, Im) and both negated when it is stored (Im, Re): the three
// shears of shear_plane, the second plane's written y-first (y -= t x,
// x += s y, y -= t x, the same rotation).  Orientation of j = parity of its
// first-colour register bits (compile time) XOR the thread's (folded into T, S).
// parity of the low nb bits of j (folded to a constant for a constant j)
__device__ __forceinline__ bool par_low(int j, int nb) { return (__popc((unsigned)j & ((1u << nb) - 1u)) & 1) != 0; }

template <int NA, int NB, int JU, int JV>
__device__ __forceinline__ void gate_oriented(u64 (&P)[NA], u64 T, u64 S) {
  constexpr u64 kNeg = 0x8000000080000000ull;
  const u64 Tn = T ^ kNeg, Sn = S ^ kNeg;
#pragma unroll
  for (int j = 0; j < NA; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0)
      fma2_acc(P[j], par_low(j, NB) ? Tn : T, P[j ^ (1 << JU) ^ (1 << JV)]);
#pragma unroll
  for (int j = 0; j < NA; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0)
      fma2_acc(P[j ^ (1 << JU) ^ (1 << JV)], par_low(j, NB) ? Sn : S, P[j]);
#pragma unroll
  for (int j = 0; j < NA; ++j)
    if (((j >> JU) & 1) == 1 && ((j >> JV) & 1) == 0)
      fma2_acc(P[j], par_low(j, NB) ? Tn : T, P[j ^ (1 << JU) ^ (1 << JV)]);
}

// Gate on register bits (ku, kv) of a phase with nb first-colour register
// bits: key = 64 nb + 8 ku + kv.
__device__ __forceinline__ void gate_combo_oriented(u64 (&P)[64], int key, u64 T, u64 S) {
  switch (key) {
    case 130: gate_oriented<64, 2, 0, 2>(P, T, S); break;
    case 131: gate_oriented<64, 2, 0, 3>(P, T, S); break;
    case 132: gate_oriented<64, 2, 0, 4>(P, T, S); break;
    case 133: gate_oriented<64, 2, 0, 5>(P, T, S); break;
    case 138: gate_oriented<64, 2, 1, 2>(P, T, S); break;
    case 139: gate_oriented<64, 2, 1, 3>(P, T, S); break;
    case 140: gate_oriented<64, 2, 1, 4>(P, T, S); break;
    case 141: gate_oriented<64, 2, 1, 5>(P, T, S); break;
    case 195: gate_oriented<64, 3, 0, 3>(P, T, S); break;
    case 196: gate_oriented<64, 3, 0, 4>(P, T, S); break;
    case 197: gate_oriented<64, 3, 0, 5>(P, T, S); break;
    case 203: gate_oriented<64, 3, 1, 3>(P, T, S); break;
    case 204: gate_oriented<64, 3, 1, 4>(P, T, S); break;
    case 205: gate_oriented<64, 3, 1, 5>(P, T, S); break;
    case 211: gate_oriented<64, 3, 2, 3>(P, T, S); break;
    case 212: gate_oriented<64, 3, 2, 4>(P, T, S); break;
    case 213: gate_oriented<64, 3, 2, 5>(P, T, S); break;
    case 260: gate_oriented<64, 4, 0, 4>(P, T, S); break;
    case 261: gate_oriented<64, 4, 0, 5>(P, T, S); break;
    case 268: gate_oriented<64, 4, 1, 4>(P, T, S); break;
    case 269: gate_oriented<64, 4, 1, 5>(P, T, S); break;
    case 276: gate_oriented<64, 4, 2, 4>(P, T, S); break;
    case 277: gate_oriented<64, 4, 2, 5>(P, T, S); break;
    case 284: gate_oriented<64, 4, 3, 4>(P, T, S); break;
    case 285: gate_oriented<64, 4, 3, 5>(P, T, S); break;
    default: break;
  }
}
__device__ __forceinline__ void gate_combo_oriented(u64 (&P)[32], int key, u64 T, u64 S) {
  switch (key) {
    case 130: gate_oriented<32, 2, 0, 2>(P, T, S); break;
    case 131: gate_oriented<32, 2, 0, 3>(P, T, S); break;
    case 132: gate_oriented<32, 2, 0, 4>(P, T, S); break;
    case 138: gate_oriented<32, 2, 1, 2>(P, T, S); break;
    case 139: gate_oriented<32, 2, 1, 3>(P, T, S); break;
    case 140: gate_oriented<32, 2, 1, 4>(P, T, S); break;
    case 195: gate_oriented<32, 3, 0, 3>(P, T, S); break;
    case 196: gate_oriented<32, 3, 0, 4>(P, T, S); break;
    case 203: gate_oriented<32, 3, 1, 3>(P, T, S); break;
    case 204: gate_oriented<32, 3, 1, 4>(P, T, S); break;
    case 211: gate_oriented<32, 3, 2, 3>(P, T, S); break;
    case 212: gate_oriented<32, 3, 2, 4>(P, T, S); break;
    default: break;
  }
}

template <int RB, bool SITES>
__device__ __forceinline__ void oriented_phase(float2 *tile2, const PassDesc &d, const PhaseDesc &ph,
                                               const ROpRes *ops, uint64_t base, int tid, int lognt,
                                               float &up, float &dn, double *s_w, uint32_t s0,
                                               const uint32_t (&sm)[RB], uint32_t outer_par) {
  constexpr int NA = 1 << RB;
  const uint32_t t0 = thread_origin(ph, tid, lognt);
  const int key0 = 64 * ph.nb;
  // the thread's orientation: its fixed tile bits and the tile's outer bits
  const uint32_t tp = (__popc(t0 & d.black_tile) & 1u) ^ outer_par;
  const u64 flip = tp ? 0x8000000080000000ull : 0ull;
  u64 P[NA];
  const char *tb = reinterpret_cast<const char *>(tile2);
  uint32_t mb[RB];
#pragma unroll
  for (int k = 0; k < RB; ++k) mb[k] = sm[k] << 3;
  const uint32_t ob = s0 << 3;
  {
    uint32_t o = ob;
#pragma unroll
    for (int g = 0; g < NA; ++g) {
      const int j = g ^ (g >> 1);
      if ((g & 7) == 0) {
        o = ob;
#pragma unroll
        for (int k = 0; k < RB; ++k)
          if ((j >> k) & 1) o ^= mb[k];
      } else {
        o ^= mb[ctz6(g)];
      }
      P[j] = *reinterpret_cast<const u64 *>(tb + o);
    }
  }
  ROpRes cur = ops[0];
  for (int k = 0; k < ph.nops; ++k) {
    const ROpRes nxt = ops[k + 1 < ph.nops ? k + 1 : k];  // prefetch
    if (cur.kind == OP_GATE) {
      const u64 T = pack2(cur.t, -cur.t) ^ flip, S = pack2(-cur.s, cur.s) ^ flip;
      gate_combo_oriented(P, key0 + cur.combo, T, S);
    } else if (cur.kind == OP_REDUCE) {
      int kr = -1;
#pragma unroll
      for (int q = 0; q < RB; ++q)
        if (ph.rb[q] == d.site_tile) kr = q;
      const uint32_t fixed_bit = d.site_tile < 0 ? (uint32_t)((base >> d.site_pos) & 1ull)
                                                 : (t0 >> d.site_tile) & 1u;
      float tsum = 0.f, ureg[RB];
#pragma unroll
      for (int q = 0; q < RB; ++q) ureg[q] = 0.f;
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        const float2 v = unpack2(P[j]);
        const float pr = fmaf(v.x, v.x, v.y * v.y);
        const uint32_t bit = kr >= 0 ? ((uint32_t)(j >> kr) & 1u) : fixed_bit;
        if (bit) up += pr;
        else dn += pr;
        if constexpr (SITES) {
          tsum += pr;
#pragma unroll
          for (int q = 0; q < RB; ++q)
            if ((j >> q) & 1) ureg[q] += pr;
        }
      }
      if constexpr (SITES) {
#pragma unroll
        for (int q = 0; q < kMaxK; ++q) {
          float v = ((t0 >> q) & 1u) ? tsum : 0.f;
#pragma unroll
          for (int k2 = 0; k2 < RB; ++k2)
            if (ph.rb[k2] == q) v = ureg[k2];
          warp_site_sum<float>(v, q, s_w, tid);
        }
        warp_site_sum<float>(tsum, kMaxK, s_w, tid);
      }
    }
    cur = nxt;
  }
  {
    char *tw = reinterpret_cast<char *>(tile2);
    uint32_t o = ob;
#pragma unroll
    for (int g = 0; g < NA; ++g) {
      const int j = g ^ (g >> 1);
      if ((g & 7) == 0) {
        o = ob;
#pragma unroll
        for (int k = 0; k < RB; ++k)
          if ((j >> k) & 1) o ^= mb[k];
      } else {
        o ^= mb[ctz6(g)];
      }
      *reinterpret_cast<u64 *>(tw + o) = P[j];
    }
  }
}

// A thread's first-phase subcube straight from the state (direct passes): tile
// bits 0 and 1 are register bits 1 and 2, so each 32-byte load brings four
// neighbouring amplitudes, and the next tile bits are lane bits where the
// planner could leave them, so a warp's loads fill 128-byte lines.  Against a
// copy through shared memory this saves a tile's write there and a read, and
// the copy's address arithmetic for every amplitude (400-step 14-spin ladder
// 7.44 -> 7.15 ms, 40-step 18-spin one 6.3 -> 6.0; not used by the pipelined
// sweep, whose compute groups would wait on their own loads and stores:
// measured 8 to 20 % slower there).  Quads are walked in
// Gray-code order over register bits 0 and 3..RB-1.
__device__ __forceinline__ uint64_t direct_offset(uint64_t base, const uint8_t *thr, int tid, int lognt) {
  uint64_t off = base;
#pragma unroll
  for (int b = 0; b < kMaxK - 5; ++b)
    if (b < lognt && ((tid >> b) & 1)) off |= 1ull << thr[b];
  return off;
}
// register index (quad's first amplitude) of Gray-code step g
__host__ __device__ constexpr int quad_index(int g) { return ((g ^ (g >> 1)) & 1) | (((g ^ (g >> 1)) >> 1) << 3); }

template <int RB>
__device__ __forceinline__ void load_direct(const float2 *psi, uint64_t base, const PassDesc &d, int tid, int lognt,
                                            u64 (&RE)[1 << (RB - 1)], u64 (&IM)[1 << (RB - 1)]) {
  const char *src = reinterpret_cast<const char *>(psi + direct_offset(base, d.in_thr, tid, lognt));
  int64_t dg[RB - 2];
#pragma unroll
  for (int k = 0; k < RB - 2; ++k) dg[k] = (int64_t)8 << d.in_reg[k ? k + 2 : 0];
  u64 A[1 << RB];
#pragma unroll
  for (int g = 0; g < (1 << (RB - 2)); ++g) {
    if (g) src += gray_up(g) ? dg[ctz5(g)] : -dg[ctz5(g)];
    const int i = quad_index(g);
    asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(A[i]), "=l"(A[i | 2]), "=l"(A[i | 4]), "=l"(A[i | 6])
                 : "l"(src)
                 : "memory");
  }
#pragma unroll
  for (int j = 0; j < (1 << (RB - 1)); ++j) {
    const float2 a = unpack2(A[2 * j]), b = unpack2(A[2 * j + 1]);
    RE[j] = pack2(a.x, b.x);
    IM[j] = pack2(a.y, b.y);
  }
}

// The last phase's subcubes straight to the state, output tile bits 0 and 1
// being register bits 1 and 2.
template <int RB>
__device__ __forceinline__ void store_direct(float2 *psi, uint64_t base, const PassDesc &d, int tid, int lognt,
                                             const u64 (&RE)[1 << (RB - 1)], const u64 (&IM)[1 << (RB - 1)]) {
  char *dst = reinterpret_cast<char *>(psi + direct_offset(base, d.out_thr, tid, lognt));
  int64_t dg[RB - 2];
#pragma unroll
  for (int k = 0; k < RB - 2; ++k) dg[k] = (int64_t)8 << d.out_reg[k ? k + 2 : 0];
#pragma unroll
  for (int g = 0; g < (1 << (RB - 2)); ++g) {
    if (g) dst += gray_up(g) ? dg[ctz5(g)] : -dg[ctz5(g)];
    const int i = quad_index(g), j = i >> 1;
    u64 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 r = unpack2(RE[j | q]), m = unpack2(IM[j | q]);
      v[q] = (i & 1) ? pack2(r.y, m.y) : pack2(r.x, m.x);
    }
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(v[0]), "l"(v[1]), "l"(v[2]), "l"(v[3])
                 : "memory");
  }
}

// All-site readout of a phase: every tile bit's weight over the warp into
// s_w[warp][bit] and the whole weight into slot kMaxK, from the thread's sums
// acc (by register bits 1, 2, RB - 1 and the pack bit, in the lanes) and ext (by
// the register bits between).  The register bits' sums are reduced together,
// half of them exchanged at each step (9 shuffles for all), the lane bits'
// build up along one butterfly (15), a warp bit's is the warp's whole sum or
// nothing.  (A butterfly for each tile bit, 75 shuffles, its values picked from
// the registers at run time, cost 30 us of an 84 us sweep of 2^23 amplitudes.)
template <int RB>
__device__ __forceinline__ void site_sums(const u64 (&acc)[8], const u64 (&ext)[2], const PhaseDesc &ph, int tid,
                                          int lognt, double *s_w) {
  const int lane = tid & 31, warp = tid >> 5;
  double *const row = s_w + warp * kSiteSlots;
  float v[8], T = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 x = unpack2(acc[i]);
    const float y = x.x + x.y;
    T += y, v[0] += x.y;
    if (i & 1) v[1] += y;
    if (i & 2) v[2] += y;
    if (i & 4) v[RB - 1] += y;
  }
  const float2 e0 = unpack2(ext[0]), e1 = unpack2(ext[1]);
  v[3] = e0.x + e0.y;
  if (RB == 6) v[4] = e1.x + e1.y;
  // lane l keeps sum l >> 2
#pragma unroll
  for (int h = 4, o = 16; h; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const float got = __shfl_xor_sync(0xffffffffu, up ? v[k] : v[k + h], o);
      v[k] = (up ? v[k + h] : v[k]) + got;
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  float U[5];
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    const float p = __shfl_xor_sync(0xffffffffu, T, 1 << b);
#pragma unroll
    for (int i = 0; i < b; ++i) U[i] += __shfl_xor_sync(0xffffffffu, U[i], 1 << b);
    U[b] = ((lane >> b) & 1) ? T : p;
    T += p;
  }
  // one conversion and one store for the warp: lanes 4 k hold register bit k,
  // lanes 4 b + 1 lane bit b (b = 5: the whole), lanes 4 b + 2 warp bit b
  const int i = lane >> 2, kind = lane & 3;
  float x = v[0];
  int bit = i < RB ? ph.rb[i] : -1;
  if (kind == 1) {
    x = i == 0 ? U[0] : i == 1 ? U[1] : i == 2 ? U[2] : i == 3 ? U[3] : i == 4 ? U[4] : T;
    bit = i < 5 ? ph.lanes[i] : i == 5 ? kMaxK : -1;
  } else if (kind == 2) {
    x = ((warp >> i) & 1) ? T : 0.f;
    bit = i < lognt - 5 ? ph.warps[i] : -1;
  }
  if (kind < 3 && bit >= 0) row[bit] = (double)x;
}

// The pass's phases on one tile in shared memory, run by the 2^lognt threads
// tid of its group; `sync` is the group's barrier, sH the outer spins' fields
// when the pass has a diagonal op (diag_fields), dtab its tables and s_w the
// all-site scratch (SITES only).  ORIENT: the program and the state are oriented (see Orientation).
// ENDS kDirect: RE/IM hold the first phase's subcubes (load_direct) and the last
// phase goes to the state psi; kInPlace: the tile is in tile2 before and after.
// WALK: rounds as walks over the register-bit pairs, else a jump to each gate
// (the same gates in the same order).  DIAG: the pass may have a diagonal op.
enum { kInPlace = 0, kDirect = 1 };
template <int RB, bool SITES, bool ORIENT, int ENDS, bool WALK = true, bool DIAG = true, typename Sync>
__device__ __forceinline__ void run_phases(float2 *tile2, const PassDesc &d, const PhaseDesc *s_ph,
                                           const ROpRes *s_op, uint64_t base, int tid, int lognt,
                                           const uint64_t *__restrict__ dtab, float &up, float &dn,
                                           const uint64_t *sH, double *s_w, Sync sync,
                                           u64 (&RE)[1 << (RB - 1)], u64 (&IM)[1 << (RB - 1)], float2 *psi) {
  constexpr int NP = 1 << (RB - 1);
  const uint32_t outer_par = ORIENT ? (uint32_t)(__popcll(base & d.black_outer) & 1) : 0u;
  // masks of the thread-index bits, two to a word
  uint32_t tm[5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
    tm[i] = (((tid >> (2 * i)) & 1) ? 0xffffu : 0u) | (((tid >> (2 * i + 1)) & 1) ? 0xffff0000u : 0u);
  int st = 0;  // step of the pass
  for (int p = 0; p < d.nphases; ++p) {
    const PhaseDesc &ph = s_ph[p];
    // slot of this thread's subcube origin (host-precomputed slot of each
    // thread-index bit) and of the register bits, from two 16-byte words (bit
    // by bit these loads took 430 cycles a phase)
    const uint4 w0 = reinterpret_cast<const uint4 *>(&ph)[0], w1 = reinterpret_cast<const uint4 *>(&ph)[1];
    const uint32_t sx = (w0.x & tm[0]) ^ (w0.y & tm[1]) ^ (w0.z & tm[2]) ^ (w0.w & tm[3]) ^ (w1.x & tm[4]);
    const uint32_t s0 = (sx ^ (sx >> 16)) & 0xffffu;
    uint32_t sm[RB];
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const uint32_t v = k < 2 ? w1.y : k < 4 ? w1.z : w1.w;
      sm[k] = (k & 1) ? v >> 16 : v & 0xffffu;
    }
    const int o0 = ph.op0 - d.rop0;
    // the phase's first step, and the coefficients of its first gate if it is a round
    uint32_t step = ORIENT ? 0u : d.steps[st];
    if (DIAG && (ORIENT ? ph.nops == 1 && s_op[o0].kind == OP_DIAG : (step & kStepDiag) != 0)) {
      diag_tile<RB, ORIENT>(tile2, dtab + s_op[o0].tab, sH + s_op[o0].arg * kFieldStride, d.K, tid, lognt,
                            d.black_tile, outer_par);
      sync();
      ++st;
      continue;
    }
    float2 ts = make_float2(0.f, 0.f);
    if constexpr (WALK && !ORIENT) ts = make_float2(s_op[o0 + 1].t, s_op[o0 + 1].s);
    if constexpr (ORIENT) {
      oriented_phase<RB, SITES>(tile2, d, ph, s_op + o0, base, tid, lognt, up, dn, s_w, s0, sm, outer_par);
      sync();
      continue;
    }
    // load the subcube as NP packs, walking the packs in Gray-code order so
    // each step changes one register bit (one XOR on the byte offset)
    const char *tb = reinterpret_cast<const char *>(tile2);
    uint32_t mb[RB];
#pragma unroll
    for (int k = 0; k < RB; ++k) mb[k] = sm[k] << 3;
    const uint32_t ob = s0 << 3;
    if (ENDS != kDirect || p > 0) {
      uint32_t o = ob;
#pragma unroll
      for (int g = 0; g < NP; ++g) {
        const int j = g ^ (g >> 1);
        if ((g & 7) == 0) {
          o = ob;
#pragma unroll
          for (int k = 0; k < RB - 1; ++k)
            if ((j >> k) & 1) o ^= mb[1 + k];
        } else {
          o ^= mb[1 + ctz5(g)];
        }
        const uint32_t o1 = o ^ mb[0];
        const float2 v0 = *reinterpret_cast<const float2 *>(tb + o);
        const float2 v1 = *reinterpret_cast<const float2 *>(tb + o1);
        RE[j] = pack2(v0.x, v1.x);
        IM[j] = pack2(v0.y, v1.y);
      }
    }
    for (int k = o0;;) {  // op of the step
      if ((step & kStepReduce) == 0) {
        const int n = (int)(step >> 16) & 0xff;
        if constexpr (WALK) {
          run_round<NP>(RE, IM, step & 0x7fffu, s_op + k + 1, ts);
        } else {
          static_assert(WALK || ORIENT || RB == 6, "a jump to each gate: six register bits");
          for (int i = 1; i <= n; ++i) {
            const ROpRes cur = s_op[k + i];
            gate_combo(RE, IM, cur.combo, cur.t, cur.s);
          }
        }
        k += 1 + n;
      } else {
        // weights by register bits 1, 2 and RB - 1 (and the pack bit, the lanes),
        // one of which the readout spin is if it is a register bit at all (with
        // the spin's register bit found at run time and every pack tested for
        // it, this took 1300 cycles of a lone warp)
        u64 acc[8], ext[2] = {0ull, 0ull};
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0ull;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          u64 &a = acc[(j & 3) | ((j >> (RB - 2)) << 2)];
          const u64 pr = fma2(RE[j], RE[j], mul2(IM[j], IM[j]));
          a = add2(a, pr);
          if constexpr (SITES) {  // and by the register bits between
            if ((j >> 2) & 1) ext[0] = add2(ext[0], pr);
            if (RB == 6 && ((j >> 3) & 1)) ext[1] = add2(ext[1], pr);
          }
        }
        const int L = d.site_label;
        const uint32_t bit = d.site_thr >= 0 ? (uint32_t)(tid >> d.site_thr) & 1u
                                             : (uint32_t)((base >> d.site_pos) & 1ull);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 v = unpack2(acc[i]);
          const bool hi = L == 1 ? (i & 1) != 0 : L == 2 ? (i & 2) != 0 : L > 2 ? (i & 4) != 0 : bit != 0;
          up += L == 0 ? v.y : hi ? v.x + v.y : 0.f;
          dn += L == 0 ? v.x : hi ? 0.f : v.x + v.y;
        }
        if constexpr (SITES) site_sums<RB>(acc, ext, ph, tid, lognt, s_w);
        ++k;
      }
      ++st;
      if (step & kStepEnd) break;
      step = d.steps[st];
      if constexpr (WALK) ts = make_float2(s_op[k + 1].t, s_op[k + 1].s);
    }
    if (ENDS == kDirect && p == d.nphases - 1) {
      // one phase only: every load of the tile before its relabelled stores
      if (p == 0) sync();
      store_direct<RB>(psi, base, d, tid, lognt, RE, IM);
    } else {
      char *tw = reinterpret_cast<char *>(tile2);
      uint32_t o = ob;
#pragma unroll
      for (int g = 0; g < NP; ++g) {
        const int j = g ^ (g >> 1);
        if ((g & 7) == 0) {
          o = ob;
#pragma unroll
          for (int k = 0; k < RB - 1; ++k)
            if ((j >> k) & 1) o ^= mb[1 + k];
        } else {
          o ^= mb[1 + ctz5(g)];
        }
        const uint32_t o1 = o ^ mb[0];
        const float2 r = unpack2(RE[j]), i = unpack2(IM[j]);
        *reinterpret_cast<float2 *>(tw + o) = make_float2(r.x, i.x);
        *reinterpret_cast<float2 *>(tw + o1) = make_float2(r.y, i.y);
      }
    }
    sync();
  }
}

// Shared -> global store of a tile, output tile bits relabelled by perm.
// Output chunk ch = tid + nt * e of two amplitudes covers output tile index
// 2 ch: bits 1..lognt from tid, the RB - 1 high ones from e (Gray order
// again).  The amplitude there is input tile index sum of bits perm[q], so its
// slot is an XOR of per-bit slots; the chunk's second amplitude is output bit
// 0 = input bit perm[0].
template <int RB>
__device__ __forceinline__ void store_tile(float2 *psi, uint64_t base, const PassDesc &d, int tid, int lognt,
                                           const float2 *tile2) {
  constexpr int NP = 1 << (RB - 1);
  uint64_t off_lo = 0;
  uint32_t pin_lo = 0;
  for (int k = 0; k < lognt; ++k)
    if ((tid >> k) & 1) {
      const int q = d.store_bit[k];
      off_lo |= 1ull << d.tile_pos[q], pin_lo |= 1u << d.perm[q];
    }
  int64_t dh[RB - 1];
  uint32_t dsl[RB - 1];
#pragma unroll
  for (int k = 0; k < RB - 1; ++k) {
    const int q = d.store_bit[lognt + k];
    dh[k] = (int64_t)8 << d.tile_pos[q];
    dsl[k] = slot(1u << d.perm[q]) << 3;
  }
  const char *tb = reinterpret_cast<const char *>(tile2);
  const uint32_t sl1 = slot(1u << d.perm[0]) << 3;
  const uint32_t so0 = slot(pin_lo) << 3;
  char *const dst0 = reinterpret_cast<char *>(psi + base + off_lo);
  uint32_t so = so0;
  char *dst = dst0;
#pragma unroll
  for (int g = 0; g < NP; ++g) {
    if ((g & 7) == 0) {
      so = so0, dst = dst0;
#pragma unroll
      for (int k = 0; k < RB - 1; ++k)
        if (((g ^ (g >> 1)) >> k) & 1) dst += dh[k], so ^= dsl[k];
    } else {
      const int k = ctz5(g);
      dst += gray_up(g) ? dh[k] : -dh[k];
      so ^= dsl[k];
    }
    const float2 v0 = *reinterpret_cast<const float2 *>(tb + so);
    const float2 v1 = *reinterpret_cast<const float2 *>(tb + (so ^ sl1));
    *reinterpret_cast<float4 *>(dst) = make_float4(v0.x, v0.y, v1.x, v1.y);
  }
}

}  // namespace sw2

// Register-blocked sweep with RB register bits (2^RB amplitudes per thread,
// 2^(K-RB) threads per tile), one tile per block.  ORIENT: an oriented
// program on an oriented state (see Orientation).  DIRECT: a direct pass, whose
// first and last phase move the tile between registers and the state.
template <int RB, bool SITES, bool ORIENT, bool DIRECT>
__global__ void __launch_bounds__(RB == 5 ? 512 : 256)
sweep2_kernel(const JobPtrs *__restrict__ jobs, float2 *psi1, const ROpRes *sops1,
              const __grid_constant__ PassDesc d, const PhaseDesc *__restrict__ phases, int M,
              unsigned ahead, bool chained) {
  // one job (gridDim.y == 1): its amplitude and op arrays come with the launch
  // so the tile copies can start at once; the rest of the job's pointers
  // (and everything for a batch) from the job table
  const bool one = gridDim.y == 1;
  const JobPtrs jp = jobs[blockIdx.y];
  float2 *__restrict__ psi = one ? psi1 : static_cast<float2 *>(jp.psi);
  extern __shared__ __align__(16) float2 tile2[];
  __shared__ uint64_t sH[2 * kFieldStride];
  __shared__ __align__(16) PhaseDesc s_ph[kMaxPassPhases];
  __shared__ __align__(16) ROpRes s_op[kMaxPassOps + 2];  // coefficients are read ahead
  __shared__ double s_w[SITES ? kMaxWarps * kSiteSlots : 1];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lognt = d.K - RB;
  const uint64_t base = sw2::tile_origin(blockIdx.x, d, M);
  // the pass's program (coefficients already resolved for this dt) and, when
  // chained, the outer fields while the sweep before this one finishes, then
  // the tile, then the L2 prefetch of the tile of block blockIdx.x + ahead
  // (ahead = blocks resident at once): DRAM keeps streaming while tiles
  // compute, and that block's loads find its tile in L2
  {
    const char *pw = reinterpret_cast<const char *>(phases + d.phase0);
    const uint32_t a_ph = (uint32_t)__cvta_generic_to_shared(s_ph);
    const int nw = d.nphases * (int)(sizeof(PhaseDesc) / 16);
    for (int i = tid; i < nw; i += nt) sw2::cp_async16(a_ph + 16u * i, pw + 16 * i);
    const ROpRes *so = (one ? sops1 : jp.sops) + d.rop0;
    const uint32_t a_op = (uint32_t)__cvta_generic_to_shared(s_op);
    for (int i = tid; i < d.nrops; i += nt) sw2::cp_async16(a_op + 16u * i, so + i);
  }
  if (chained && d.diag) sw2::diag_fields(d, base, tid, lognt, M, jp.qdiag, sH);
  grid_wait();
  grid_go();
  sw2::u64 RE[1 << (RB - 1)], IM[1 << (RB - 1)];
  if constexpr (DIRECT) sw2::load_direct<RB>(psi, base, d, tid, lognt, RE, IM);
  else sw2::load_tile<RB>(psi, base, d, tid, lognt, (uint32_t)__cvta_generic_to_shared(tile2));
  if (ahead && blockIdx.x + ahead < gridDim.x)
    sw2::prefetch_tile<RB>(psi, sw2::tile_origin(blockIdx.x + ahead, d, M), d, tid, lognt);
  if (!chained && d.diag) sw2::diag_fields(d, base, tid, lognt, M, jp.qdiag, sH);
  sw2::cp_async_wait_all();
  __syncthreads();

  float up = 0.f, dn = 0.f;
  sw2::run_phases<RB, SITES, ORIENT, DIRECT ? sw2::kDirect : sw2::kInPlace>(
      tile2, d, s_ph, s_op, base, tid, lognt, jp.dtab, up, dn, sH, s_w, sw2::SyncBlock{}, RE, IM, psi);
  if constexpr (!DIRECT) sw2::store_tile<RB>(psi, base, d, tid, lognt, tile2);
  if constexpr (SITES)
    if (d.has_reduce) write_site_partials(d, M, base, s_w, jp.psites, tid, nt, blockIdx.x, gridDim.x);
  if (d.has_reduce) reduce_finalize((double)up, (double)dn, jp, false);
}

// ===========================================================================
// Whole states resident in shared memory.  When one tile holds the whole
// state (K = M, one segment), every Trotter step is one pass over that tile,
// so a block can keep the state in shared memory for all the steps of an
// evolve call: one global load at the start, one store at the end, and the
// P / norm readout after every step reduced inside the block.
// ===========================================================================
// The four passes of a one-tile plan: the first, steady and last step of an
// evolve call of two or more steps, and the step of a one-step call.
struct ResidentPasses {
  PassDesc first, mid, last, only;
};

// One block per job (blockIdx.y); 2^(M-RB) threads.  Dynamic shared memory:
// the state (8 B x 2^M), then the plan's phase program (nph PhaseDesc) and its
// resolved ops (nrops ROpRes).  ORIENT: oriented program and state.
template <int RB, bool ORIENT>
__global__ void __launch_bounds__(256)
resident_kernel(const JobPtrs *__restrict__ jobs, const __grid_constant__ ResidentPasses rp,
                const PhaseDesc *__restrict__ phases, int nph, int nrops, int M, int64_t steps) {
  const JobPtrs jp = jobs[blockIdx.y];
  float2 *__restrict__ psi = static_cast<float2 *>(jp.psi);
  extern __shared__ __align__(16) float2 tile2[];
  PhaseDesc *s_ph = reinterpret_cast<PhaseDesc *>(tile2 + (size_t(1) << M));
  ROpRes *s_op = reinterpret_cast<ROpRes *>(s_ph + nph);
  __shared__ uint64_t sH[2 * kFieldStride];
  __shared__ double s_up[8], s_dn[8];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lognt = M - RB;
  // the state (tile bits = physical bits: base 0, no relabelling), then the program
  sw2::load_tile<RB>(psi, 0, rp.first, tid, lognt, (uint32_t)__cvta_generic_to_shared(tile2));
  {
    const char *pw = reinterpret_cast<const char *>(phases);
    const uint32_t a_ph = (uint32_t)__cvta_generic_to_shared(s_ph);
    const int nw = nph * (int)(sizeof(PhaseDesc) / 16);
    for (int i = tid; i < nw; i += nt) sw2::cp_async16(a_ph + 16u * i, pw + 16 * i);
    const uint32_t a_op = (uint32_t)__cvta_generic_to_shared(s_op);
    for (int i = tid; i < nrops; i += nt) sw2::cp_async16(a_op + 16u * i, jp.sops + i);
  }
  for (int i = tid; i < 2 * kFieldStride; i += nt) sH[i] = 0;  // no outer spins: no fields
  sw2::cp_async_wait_all();
  __syncthreads();
  const int64_t slot0 = *jp.step;
  const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  for (int64_t k = 0; k < steps; ++k) {
    const PassDesc &d = steps == 1 ? rp.only : k == 0 ? rp.first : k == steps - 1 ? rp.last : rp.mid;
    float up = 0.f, dn = 0.f;
    sw2::u64 RE[1 << (RB - 1)], IM[1 << (RB - 1)];
    sw2::run_phases<RB, false, ORIENT, sw2::kInPlace>(tile2, d, s_ph + d.phase0, s_op + d.rop0, 0ull, tid, lognt,
                                                      jp.dtab, up, dn, sH, nullptr, sw2::SyncBlock{}, RE, IM, nullptr);
    // this step's N_up / N_dn: FP64 sums over the block in a fixed order
    double u = up, w = dn;
    for (int o = 16; o; o >>= 1) {
      u += __shfl_xor_sync(0xffffffffu, u, o);
      w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    if (lane == 0) s_up[warp] = u, s_dn[warp] = w;
    __syncthreads();
    if (tid == 0) {
      double U = 0.0, D = 0.0;
      for (int i = 0; i < nw; ++i) U += s_up[i], D += s_dn[i];
      jp.series[2 * (slot0 + k)] = (U - D) / (U + D);
      jp.series[2 * (slot0 + k) + 1] = U + D;
    }
    __syncthreads();
  }
  sw2::store_tile<RB>(psi, 0, rp.first, tid, lognt, tile2);
  if (tid == 0) *jp.step = slot0 + steps;
}

}  // namespace spinrp
