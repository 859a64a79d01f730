"""rd_gamma_R's first query of an m with little free device memory: the search with 6 ring slots wherever it fits, the
low-memory form (3 slots, the intermediate in column chunks) below that, RD_ERR_NOMEM where neither does."""
import threading

import pytest

from conftest import oracle_first_repeat

pytestmark = pytest.mark.gpu

GB = 1 << 30


@pytest.fixture(scope="module")
def rd():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    return rd


def used_by_first_query(rd, m, n, leave):
    """gamma_R(m, n) from an empty cache with `leave` bytes of device memory free; the most that it held meanwhile."""
    import torch

    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - leave, dtype=torch.uint8, device="cuda") if free > leave else None
    before, low, stop = torch.cuda.mem_get_info()[0], [1 << 62], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])

    rd.gamma_R_clear()
    t = threading.Thread(target=watch)
    t.start()
    try:
        got = rd.gamma_R(m, n)
    finally:
        stop.set()
        t.join()
        del filler
        torch.cuda.empty_cache()
    return got, before - low[0]


def test_the_search_with_six_slots_wherever_it_fits(rd):
    """m = 9, 0.96 GB per power: 7.0 GB with 6 slots and the whole intermediate, 3.4 GB in the low-memory form."""
    o = oracle_first_repeat(9)
    for leave, least, most in ((9 * GB, 6 * GB, 8 * GB), (8 * GB, 6 * GB, 8 * GB), (6 * GB, 2 * GB, 4 * GB)):
        got, used = used_by_first_query(rd, 9, 20, leave)
        assert got == o["gamma"][20]
        assert least < used < most, (leave, used)


def test_no_form_fits(rd):
    for m, leave in ((9, 2 * GB), (12, 1 << 62)):
        with pytest.raises(rd.RdError) as e:
            used_by_first_query(rd, m, 20, leave)
        assert e.value.status == rd.RD_ERR_NOMEM
