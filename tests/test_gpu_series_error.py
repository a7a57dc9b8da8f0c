"""GPU: every series of a state reports the pipelined sweeps' error word.

The word is set from the host between two calls (no sweep runs with it set) in
the state's work buffer, 128 bytes into the 256-byte area that holds the series
counter at byte 64 and nothing else."""
import numpy as np
import pytest

from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_series_report_the_error_word():
    import torch

    st = spinrp.State(spinrp.System(W.chain(23, 0.9), W.XY), "c64", series_cap=8).set_sites(True)
    assert st.pipeline()
    st.init_random_phase(5).evolve(0.05, 3)
    readers = (lambda: st.polarization(1), lambda: st.polarization(7), st.norm_series, st.site_series)
    good = [r() for r in readers]
    assert all(np.all(np.isfinite(x)) for x in good)
    words = st._bufs[1][: 1 << 20].view(torch.int32).view(-1, 64)
    area = torch.zeros(64, dtype=torch.int32, device="cuda")
    area[16] = 4  # entries recorded
    at = torch.nonzero((words == area).all(dim=1)).flatten().tolist()
    assert len(at) == 1
    words[at[0], 32] = 1
    for r in readers:
        with pytest.raises(spinrp.SpinrpError) as e:
            r()
        assert e.value.code == spinrp.ETIMEOUT
    words[at[0], 32] = 0
    for r, x in zip(readers, good):
        assert np.array_equal(r(), x)
    st.close()
