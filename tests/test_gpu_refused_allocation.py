"""A device allocation that is refused is reported by the call that asked for it, and by no later one."""
import pytest

pytestmark = pytest.mark.gpu


def test_calls_after_a_refused_allocation(orc):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    want = orc.power_until_periodic(5, kmax=48)["gamma"][20]
    rd.gamma_R_clear()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(rd.RdError) as e:
            rd.gamma_R(9, 20)  # 3.4 GB in its smallest form
        assert e.value.status == rd.RD_ERR_NOMEM
        assert rd.gamma_R(5, 20) == want
        with rd.Server(hbm_budget_bytes=64 << 30, kmax=64) as sv:  # more than there is
            _, st, _ = sv.wait(sv.submit([9], [20]))
            assert list(st) == [rd.RD_ERR_NOMEM]
            g, st, _ = sv.wait(sv.submit([5], [20]))
            assert (list(g), list(st)) == ([want], [rd.RD_OK])
    finally:
        del filler
        torch.cuda.empty_cache()
        rd.gamma_R_clear()
