// planner.cpp -- cuts the forward half step of the Trotter product into
// shared-memory tile sweeps.
//
// The forward half step applies the flip-flop bonds in canonical order
// g_0, g_1, ..., g_{B-1}.  Two gates on disjoint spin pairs commute exactly, so
// any order that keeps, for every spin, the sequence of gates touching it is
// the same operator.  The planner exploits this freedom (and nothing else): it
// greedily grows a set Q of K spins and takes every gate that becomes
// applicable using spins of Q only; that set of gates is one segment (one
// device sweep over 2^(M-K) tiles of 2^K amplitudes).  It repeats until every
// gate is placed.  The reverse half step reuses the segments backwards.
//
// Coalescing: every tile must contain the c lowest physical bits, so that a
// tile is made of contiguous runs of 2^c amplitudes.  Consecutive segments k,
// k+1 therefore share c spins X_k ("exit set" of k): sweep k writes its tile
// back with X_k moved into the low bits (an in-place relabelling of bit
// positions inside the tile), and segment k+1 is grown starting from X_k.
// On the way back (reverse half step) each sweep undoes its relabelling, so
// the layout at every step boundary is the same (pos).
#include <algorithm>
#include <array>
#include <limits>
#include <queue>

#include "internal.h"

namespace spinrp {

namespace {

struct Frontier {
  const std::vector<std::pair<int, int>> *bonds;
  const std::vector<std::vector<int>> *chain;  // per spin: bonds touching it, in order
  std::vector<int> ptr;                        // per spin: next undone position in its chain
  int ndone = 0;

  bool ready(int b) const {
    const auto &bd = (*bonds)[b];
    const auto &ci = (*chain)[bd.first], &cj = (*chain)[bd.second];
    return ptr[bd.first] < (int)ci.size() && ci[ptr[bd.first]] == b &&
           ptr[bd.second] < (int)cj.size() && cj[ptr[bd.second]] == b;
  }
  int head(int q) const {
    const auto &c = (*chain)[q];
    return ptr[q] < (int)c.size() ? c[ptr[q]] : -1;
  }
  int pending(int q) const { return (int)(*chain)[q].size() - ptr[q]; }
  // Apply every gate reachable inside spin set Q (bit mask), smallest bond
  // index first; appends the applied bonds to out (if non-null).
  int closure(uint64_t Q, std::vector<int> *out) {
    std::priority_queue<int, std::vector<int>, std::greater<int>> pq;
    const int M = (int)ptr.size();
    for (int q = 0; q < M; ++q) {
      if (!((Q >> q) & 1)) continue;
      int b = head(q);
      if (b < 0) continue;
      const auto &bd = (*bonds)[b];
      if (((Q >> bd.first) & 1) && ((Q >> bd.second) & 1) && ready(b)) pq.push(b);
    }
    int applied = 0, last = -1;
    while (!pq.empty()) {
      int b = pq.top();
      pq.pop();
      if (b == last || !ready(b)) continue;  // pushed once per endpoint
      last = b;
      const auto &bd = (*bonds)[b];
      ++ptr[bd.first];
      ++ptr[bd.second];
      ++applied;
      ++ndone;
      if (out) out->push_back(b);
      for (int q : {bd.first, bd.second}) {
        int nb = head(q);
        if (nb < 0) continue;
        const auto &nbd = (*bonds)[nb];
        if (((Q >> nbd.first) & 1) && ((Q >> nbd.second) & 1) && ready(nb)) pq.push(nb);
      }
    }
    return applied;
  }
};

}  // namespace

bool build_plan(int M, const std::vector<std::pair<int, int>> &bonds, int K, int c, Plan *plan,
                std::string *err) {
  if (M < 1 || M > kMaxM || K < 1) {
    *err = "plan: bad size";
    return false;
  }
  const int B = (int)bonds.size();
  plan->M = M;
  plan->seg.clear();
  plan->segQ.clear();
  plan->exitX.clear();
  plan->pos.assign(M, -1);
  if (K >= M) {
    // one tile holds the whole state: one segment, canonical order, identity layout
    plan->K = M;
    plan->c = M;
    std::vector<PlanGate> g;
    for (int b = 0; b < B; ++b) g.push_back({b, bonds[b].first, bonds[b].second});
    plan->seg.push_back(g);
    std::vector<int> all(M);
    for (int q = 0; q < M; ++q) all[q] = q, plan->pos[q] = q;
    plan->segQ.push_back(all);
    return true;
  }
  c = std::max(0, std::min(c, K - 2));
  plan->K = K;
  plan->c = c;

  std::vector<std::vector<int>> chain(M);
  for (int b = 0; b < B; ++b) {
    chain[bonds[b].first].push_back(b);
    chain[bonds[b].second].push_back(b);
  }
  Frontier fr;
  fr.bonds = &bonds;
  fr.chain = &chain;
  fr.ptr.assign(M, 0);

  std::vector<int> order;  // spins in order of first use (physical layout)
  uint64_t placed = 0;
  auto place = [&](int q) {
    if (!((placed >> q) & 1)) order.push_back(q), placed |= 1ull << q;
  };

  uint64_t entry = 0;  // spins the next segment must contain (previous exit set)
  int guard = 0;
  while (fr.ndone < B || plan->seg.empty()) {
    if (++guard > 4 * B + 8) {
      *err = "plan: no progress (tile too narrow)";
      return false;
    }
    uint64_t Q = entry;
    std::vector<int> added;
    while (__builtin_popcountll(Q) < K) {
      Frontier base_trial = fr;
      const long base = base_trial.closure(Q, nullptr);
      int best = -1;
      long best_gain = -1, best_adj = -1, best_first = std::numeric_limits<long>::min();
      for (int q = 0; q < M; ++q) {
        if ((Q >> q) & 1) continue;
        Frontier trial = fr;
        const long gain = trial.closure(Q | (1ull << q), nullptr);
        long adj = 0, first = B;
        for (int k = fr.ptr[q]; k < (int)chain[q].size(); ++k) {
          const int b = chain[q][k];
          const int other = bonds[b].first == q ? bonds[b].second : bonds[b].first;
          if ((Q >> other) & 1) ++adj;
          first = std::min<long>(first, b);
        }
        const bool better = best < 0 || gain > best_gain || (gain == best_gain && adj > best_adj) ||
                            (gain == best_gain && adj == best_adj && -first > best_first);
        if (better) best = q, best_gain = gain, best_adj = adj, best_first = -first;
      }
      if (best < 0) break;
      if (best_gain <= base) {
        // no single spin adds a gate: take the spins of the earliest gate that
        // is ready after the closure of Q and fits (the smallest undone gate is
        // always ready, so with K >= c + 2 this always makes progress)
        Frontier after = fr;
        after.closure(Q, nullptr);
        const int room = K - __builtin_popcountll(Q);
        int pick = -1;
        for (int b = 0; b < B && pick < 0; ++b) {
          if (!after.ready(b)) continue;
          const int need = !((Q >> bonds[b].first) & 1) + !((Q >> bonds[b].second) & 1);
          if (need > 0 && need <= room) pick = b;
        }
        if (pick < 0) break;
        for (int q : {bonds[pick].first, bonds[pick].second})
          if (!((Q >> q) & 1)) Q |= 1ull << q, added.push_back(q);
        continue;
      }
      Q |= 1ull << best;
      added.push_back(best);
    }
    // a tile always spans exactly K spins: pad with unused ones
    for (int q = 0; q < M && __builtin_popcountll(Q) < K; ++q)
      if (!((Q >> q) & 1)) Q |= 1ull << q, added.push_back(q);
    std::vector<int> applied;
    fr.closure(Q, &applied);
    if (applied.empty() && fr.ndone < B) {
      *err = "plan: a segment placed no gate (tile too narrow)";
      return false;
    }
    std::vector<PlanGate> g;
    for (int b : applied) g.push_back({b, bonds[b].first, bonds[b].second});
    plan->seg.push_back(g);
    std::vector<int> qs;
    for (int q = 0; q < M; ++q)
      if ((Q >> q) & 1) qs.push_back(q);
    plan->segQ.push_back(qs);
    // exit set: the c spins of Q whose next pending gate comes earliest, in that
    // order (the next segment starts with the first ones, and its reverse ends
    // with them: direct passes hold low bits 0 and 1 in those phases)
    std::vector<std::pair<long, int>> cand;
    for (int q : qs) {
      const int h = fr.head(q);
      cand.push_back({h < 0 ? (long)B + 1000 - fr.pending(q) : (long)h, q});
    }
    std::sort(cand.begin(), cand.end());
    std::vector<int> X;
    for (int k = 0; k < c; ++k) X.push_back(cand[k].second);  // the earliest first: low bits 0, 1, ...
    plan->exitX.push_back(X);
    entry = 0;
    for (int q : X) entry |= 1ull << q;
    for (int q : added) place(q);
  }
  const int s = (int)plan->seg.size();
  // layout at step boundaries: the first exit set in the low bits (for a
  // single segment: the first c spins of its tile), then spins in order of use
  std::vector<int> low = s >= 2 ? plan->exitX[0]
                                : std::vector<int>(plan->segQ[0].begin(), plan->segQ[0].begin() + c);
  std::vector<int> final_order = low;
  uint64_t in_low = 0;
  for (int q : low) in_low |= 1ull << q;
  for (int q : order)
    if (!((in_low >> q) & 1)) final_order.push_back(q);
  for (int q = 0; q < M; ++q)
    if (!((placed >> q) & 1) && !((in_low >> q) & 1)) final_order.push_back(q);
  for (int p = 0; p < M; ++p) plan->pos[final_order[p]] = p;
  plan->exitX.resize(std::max(0, s - 1));
  return true;
}


// ---------------------------------------------------------------------------
// Phases of the register-blocked sweep: the gates of a pass (on its K tile
// bits) are applied in phases, each holding RB tile bits in registers.  A
// phase applies every gate both of whose bits it holds as soon as all earlier
// gates on those bits are done (so each bit keeps its gate sequence and the
// operator is unchanged).  Fewer phases mean fewer shared-memory round trips;
// a beam search over the register sets looks further ahead than the greedy
// segment planner.
// ---------------------------------------------------------------------------
namespace {

typedef std::array<uint8_t, kMaxK> BitPtr;  // per tile bit: gates of its chain done

struct PhaseState {
  BitPtr ptr;
  int done = 0;
  int pre = 0;               // gates before the fence done
  int parent = -1;           // index into the previous beam level
  uint32_t set = 0;          // register set that produced this state
  int penalty = 0;           // among states of as many gates done, the least first
};

// The bits' gate chains in one array, each ended by -1, for the closures of the
// beam search (a few thousand per phase): only what a set reaches, not in which
// order, so the gates of a bit are taken as far as they go.
struct Chains {
  std::vector<int> flat, ends;  // chain of bit q from flat[off[q]]; sum of a gate's two bits
  std::array<int, kMaxK> off{};
  Chains(const std::vector<std::pair<int, int>> &g, const std::vector<std::vector<int>> &chain) {
    for (int q = 0; q < (int)chain.size(); ++q) {
      off[q] = (int)flat.size();
      flat.insert(flat.end(), chain[q].begin(), chain[q].end());
      flat.push_back(-1);
    }
    for (const auto &e : g) ends.push_back(e.first + e.second);
  }
  // what phase_closure does, without the list of gates
  int closure(BitPtr &ptr, uint32_t R, int fence, int *pre) const {
    int applied = 0;
    for (bool progress = true; progress;) {
      progress = false;
      for (uint32_t m = R; m; m &= m - 1u) {
        const int q = __builtin_ctz(m);
        for (;;) {
          const int b = flat[off[q] + ptr[q]];
          if (b < 0 || (b >= fence && *pre != fence)) break;
          const int o = ends[b] - q;
          if (!((R >> o) & 1u) || flat[off[o] + ptr[o]] != b) break;
          ++ptr[q], ++ptr[o], ++applied;
          if (b < fence) ++*pre;
          progress = true;
        }
      }
    }
    return applied;
  }
};

// Apply every gate reachable inside bit set R (smallest index first); gates
// from `fence` on only once every gate before it is done (*pre counts those).
int phase_closure(const std::vector<std::pair<int, int>> &g, const std::vector<std::vector<int>> &chain,
                  BitPtr &ptr, uint32_t R, int fence, int *pre, std::vector<int> *out) {
  auto ready = [&](int b) {
    const int u = g[b].first, v = g[b].second;
    return (b < fence || *pre == fence) && ptr[u] < chain[u].size() && chain[u][ptr[u]] == b &&
           ptr[v] < chain[v].size() && chain[v][ptr[v]] == b;
  };
  int applied = 0;
  for (bool progress = true; progress;) {
    progress = false;
    int best = -1;
    for (int q = 0; q < (int)chain.size(); ++q) {
      if (!((R >> q) & 1) || ptr[q] >= chain[q].size()) continue;
      const int b = chain[q][ptr[q]];
      if (((R >> g[b].first) & 1) && ((R >> g[b].second) & 1) && ready(b) && (best < 0 || b < best)) best = b;
    }
    if (best >= 0) {
      ++ptr[g[best].first];
      ++ptr[g[best].second];
      ++applied;
      if (best < fence) ++*pre;
      if (out) out->push_back(best);
      progress = true;
    }
  }
  return applied;
}

}  // namespace

// Every combination of `take` out of the n items (indices), in lexicographic
// order, passed to f as a bit mask over items[].
template <typename F>
static void for_each_subset(const std::vector<int> &items, int take, F f) {
  const int n = (int)items.size();
  if (take > n || take < 0) return;
  std::vector<int> pick(take);
  for (int i = 0; i < take; ++i) pick[i] = i;
  while (true) {
    uint32_t R = 0;
    for (int i : pick) R |= 1u << items[i];
    f(R);
    int i = take - 1;
    while (i >= 0 && pick[i] == n - take + i) --i;
    if (i < 0) break;
    ++pick[i];
    for (int j = i + 1; j < take; ++j) pick[j] = pick[j - 1] + 1;
  }
}

bool plan_phases(int K, const std::vector<std::pair<int, int>> &gates, int RB, int beam, int fence,
                 std::vector<uint32_t> *sets, std::vector<std::vector<int>> *applied, uint32_t black,
                 uint32_t nb_allowed, const PhaseEnds &ends) {
  sets->clear();
  applied->clear();
  const int n = (int)gates.size();
  if (n == 0) return true;
  std::vector<std::vector<int>> chain(K);
  for (int b = 0; b < n; ++b) {
    if (gates[b].first < 0 || gates[b].first >= K || gates[b].second < 0 || gates[b].second >= K ||
        gates[b].first == gates[b].second)
      return false;
    chain[gates[b].first].push_back(b);
    chain[gates[b].second].push_back(b);
  }
  const Chains chains(gates, chain);
  std::vector<std::vector<PhaseState>> levels(1);
  if (fence < 0 || fence > n) fence = n;
  BitPtr zero;
  zero.fill(0);
  levels[0].push_back(PhaseState{zero, 0, 0, -1, 0});
  // a set of RB bits from R: idle bits added, the last set's first, the ones
  // to avoid last
  const uint32_t all = (1u << K) - 1u;
  auto pad = [&](uint32_t R, uint32_t avoid) {
    for (uint32_t pool : {ends.last, all & ~avoid, all})
      for (int q = 0; q < K && __builtin_popcount(R) < RB; ++q)
        if ((pool >> q) & 1u) R |= 1u << q;
    return R;
  };
  auto penalty = [&](const PhaseState &s, int depth) {
    int p = depth == 0 ? __builtin_popcount(s.set & ends.avoid_first) : 0;
    if (s.done == n) p += (s.set & ends.last) == ends.last ? __builtin_popcount(s.set & ends.avoid_last) : 8;
    return p;
  };
  for (int depth = 0; depth < 4 * n + 4; ++depth) {
    const std::vector<PhaseState> &cur = levels.back();
    // the `beam` best distinct states (most gates done, then least penalty, then
    // the first found), in that order
    std::vector<PhaseState> kept;
    auto before = [](const PhaseState &a, const PhaseState &b) {
      return a.done != b.done ? a.done > b.done : a.penalty < b.penalty;
    };
    auto keep = [&](const PhaseState &ch) {
      if ((int)kept.size() >= beam && !before(ch, kept.back())) return;
      for (size_t k = 0; k < kept.size(); ++k)
        if (kept[k].ptr == ch.ptr) {
          if (!before(ch, kept[k])) return;
          kept.erase(kept.begin() + k);
          break;
        }
      kept.insert(std::upper_bound(kept.begin(), kept.end(), ch, before), ch);
      if ((int)kept.size() > beam) kept.pop_back();
    };
    for (int si = 0; si < (int)cur.size(); ++si) {
      const PhaseState &st = cur[si];
      // bits with gates still to do; a useful set holds RB of them (all of
      // them when fewer remain), padded with idle bits
      std::vector<int> live;
      for (int q = 0; q < K; ++q)
        if (st.ptr[q] < chain[q].size()) live.push_back(q);
      // the gates that can come next: most sets hold none of them
      std::vector<uint32_t> ready;
      for (int q : live) {
        const int b = chain[q][st.ptr[q]], o = chains.ends[b] - q;
        if (q < o && chains.flat[chains.off[o] + st.ptr[o]] == b && (b < fence || st.pre == fence))
          ready.push_back(1u << q | 1u << o);
      }
      auto try_set = [&](uint32_t R) {
        if (std::none_of(ready.begin(), ready.end(), [&](uint32_t m) { return (m & ~R) == 0u; })) return;
        PhaseState ch{st.ptr, st.done, st.pre, si, R};
        ch.done += chains.closure(ch.ptr, R, fence, &ch.pre);
        ch.penalty = penalty(ch, depth);
        keep(ch);
      };
      if (nb_allowed == 0) {
        // the first set holds ends.first; a set that may be the last one is
        // also tried with ends.last
        const uint32_t must = depth == 0 ? ends.first : 0u;
        const uint32_t avoid = (depth == 0 ? ends.avoid_first : 0u) | ends.avoid_last;
        for (uint32_t base : {must, must | ends.last}) {
          const int room = RB - __builtin_popcount(base);
          if (room < 0) continue;
          std::vector<int> pick;
          for (int q : live)
            if (!((base >> q) & 1u)) pick.push_back(q);
          for_each_subset(pick, std::min<int>(room, (int)pick.size()),
                          [&](uint32_t R) { try_set(pad(base | R, avoid)); });
          if (ends.last == 0 || (must | ends.last) == must) break;
        }
      } else {
        // for each allowed count nb: nb live bits of the colour `black` and
        // RB - nb of the other (fewer when fewer are live), each side padded
        // with idle bits of its colour
        std::vector<int> lb, lw;
        for (int q : live) (((black >> q) & 1u) ? lb : lw).push_back(q);
        for (int nb = 0; nb <= RB; ++nb) {
          if (!((nb_allowed >> nb) & 1u)) continue;
          const int tb = std::min<int>(nb, (int)lb.size()), tw = std::min<int>(RB - nb, (int)lw.size());
          for_each_subset(lb, tb, [&](uint32_t Rb) {
            for (int q = 0; q < K && __builtin_popcount(Rb) < nb; ++q)
              if ((black >> q) & 1u) Rb |= 1u << q;
            if (__builtin_popcount(Rb) != nb) return;
            for_each_subset(lw, tw, [&](uint32_t Rw) {
              for (int q = 0; q < K && __builtin_popcount(Rw) < RB - nb; ++q)
                if (!((black >> q) & 1u)) Rw |= 1u << q;
              if (__builtin_popcount(Rw) != RB - nb) return;
              try_set(Rb | Rw);
            });
          });
        }
      }
    }
    if (kept.empty()) return false;
    levels.push_back(std::move(kept));
    if (levels.back().front().done == n) {
      // walk back the sets of the first finished state, then replay them
      std::vector<uint32_t> path;
      for (int lv = (int)levels.size() - 1, si = 0; lv > 0; --lv) {
        path.push_back(levels[lv][si].set);
        si = levels[lv][si].parent;
      }
      std::reverse(path.begin(), path.end());
      BitPtr ptr = zero;
      int pre = 0;
      for (uint32_t R : path) {
        std::vector<int> out;
        phase_closure(gates, chain, ptr, R, fence, &pre, &out);
        sets->push_back(R);
        applied->push_back(out);
      }
      if ((sets->back() & ends.last) != ends.last) {
        sets->push_back(pad(ends.last, ends.avoid_last));
        applied->push_back({});
      }
      return true;
    }
  }
  return false;
}

// ---------------------------------------------------------------------------
// Rounds of a phase (see PhaseRound).
// ---------------------------------------------------------------------------
namespace {

// A phase's gates by register bit.
struct RoundGates {
  int RB, n;
  std::vector<int> pos;     // the register bits, ascending tile bits
  std::vector<int> ku, kv;  // a gate's two bits, as indices into pos
  std::array<std::vector<int>, kMaxRegBits> chain;  // a bit's gates in order, then n
  RoundGates(const std::vector<std::pair<int, int>> &gates, const std::vector<int> &rb)
      : RB((int)rb.size()), n((int)gates.size()), pos(rb) {
    std::sort(pos.begin(), pos.end());
    auto at = [&](int q) { return (int)(std::find(pos.begin(), pos.end(), q) - pos.begin()); };
    for (int g = 0; g < n; ++g) {
      ku.push_back(at(gates[g].first)), kv.push_back(at(gates[g].second));
      chain[ku[g]].push_back(g), chain[kv[g]].push_back(g);
    }
    for (int k = 0; k < RB; ++k) chain[k].push_back(n);
  }
  // Rounds of the gates before `split`, then of the others, with the bits in the
  // order `order` (indices into pos): their number, or `most` if that many or
  // more; written when out is non-null, an empty one between them for split >= 0.
  int rounds(const std::vector<int> &order, int split, int most, std::vector<PhaseRound> *out) const {
    std::array<int, kMaxRegBits> ptr{};
    std::vector<int> combo;
    if (out) {
      std::array<int, kMaxRegBits> idx{};
      for (int k = 0; k < RB; ++k) idx[order[k]] = k;
      for (int g = 0; g < n; ++g) {
        const int u = std::min(idx[ku[g]], idx[kv[g]]), v = std::max(idx[ku[g]], idx[kv[g]]);
        combo.push_back(u * (2 * RB - u - 1) / 2 + v - u - 1);
      }
    }
    int r = 0, done = 0;
    for (int part = 0; part < 2; ++part) {
      const int to = part ? n : std::max(split, 0);
      while (done < to) {
        if (r >= most) return most;
        PhaseRound rd;
        for (int u = 0; u < RB; ++u)
          for (int v = u + 1; v < RB; ++v) {
            const int a = order[u], b = order[v], g = chain[a][ptr[a]];
            if (g >= to || g != chain[b][ptr[b]]) continue;
            ++ptr[a], ++ptr[b], ++done;
            if (out) rd.gates.push_back(g);
          }
        ++r;
        if (out) rd.combo = combo, out->push_back(rd);
      }
      if (out && split >= 0 && part == 0) out->push_back(PhaseRound{});
    }
    return std::min(r, most);
  }
};

}  // namespace

void plan_rounds(const std::vector<std::pair<int, int>> &gates, int RB, int split, int fix1, int fix2,
                 int fix_last, std::vector<int> *rb, std::vector<PhaseRound> *rounds) {
  const RoundGates rg(gates, *rb);
  std::vector<int> order(RB), best_order;
  for (int k = 0; k < RB; ++k) order[k] = k;
  // a gate on the pack bit costs a gate more, a round about two (its tests)
  int best = std::numeric_limits<int>::max();
  do {
    if ((fix1 >= 0 && rg.pos[order[1]] != fix1) || (fix2 >= 0 && rg.pos[order[2]] != fix2) ||
        (fix_last >= 0 && rg.pos[order[RB - 1]] != fix_last))
      continue;
    const int pack = (int)rg.chain[order[0]].size() - 1;
    if (pack >= best) continue;
    const int most = best == std::numeric_limits<int>::max() ? best : (best - pack + 1) / 2;
    const int r = rg.rounds(order, split, most, nullptr);
    if (r < most) best = pack + 2 * r, best_order = order;
  } while (std::next_permutation(order.begin(), order.end()));
  for (int k = 0; k < RB; ++k) (*rb)[k] = rg.pos[best_order[k]];
  rounds->clear();
  rg.rounds(best_order, split, std::numeric_limits<int>::max(), rounds);
}

}  // namespace spinrp
