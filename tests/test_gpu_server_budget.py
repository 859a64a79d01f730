"""A query server whose budget holds a job's sparse operands but not its row-split ones still answers it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("short", [0, 1, 4 << 20, 14 << 20])
def test_m7_within_a_tight_budget(short):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    ms, ns = np.full(5, 7, dtype=np.int32), np.array([3, 20, 26, 57, 200], dtype=np.int64)
    want = [rd.gamma_R(7, int(n)) for n in ns]
    with rd.Server(hbm_budget_bytes=8 << 30, kmax=64) as sv:
        sv.wait(sv.submit(ms, ns))
        peak = sv.stats()["bytes_peak"]
    with rd.Server(hbm_budget_bytes=peak - short, kmax=64) as sv:
        g, st, _ = sv.wait(sv.submit(ms, ns))
        used = sv.stats()["bytes_peak"]
    assert np.all(st == rd.RD_OK) and list(g) == want and used <= peak - short
