"""The block-sparse product on random operands around the line between its two kernels (operands of up to 4096 rows and
columns: the last 2048-column slab mostly empty, few CTAs, R = 8), against the oracle, and the time on the side of the
line where random operands are best left to the CTA per block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF = 0x3FFF


@pytest.fixture(scope="module")
def rd():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    return rd


def operands(M, K, N, finite, seed):
    r = np.random.default_rng(seed)
    a = np.where(r.random((M, K)) < finite, r.integers(0, 40, (M, K)), INF).astype(np.int16)
    b = np.where(r.random((K, N)) < 0.9, r.integers(0, 0x2000, (K, N)), INF).astype(np.int16)
    return a, b


def upload(h):
    import torch

    t = torch.full((h.shape[0], (h.shape[1] + 7) // 8 * 8), -3, dtype=torch.int16)
    t[:, :h.shape[1]] = torch.from_numpy(h)
    return t.cuda()


# either side of 0.65 of one slab (1331 columns) and of two (2662), and of 3.5 CTAs per SM (532 on 152 SMs)
@pytest.mark.parametrize("R", [1, 2, 4, 8])
@pytest.mark.parametrize("M,K,N", [(1200, 50, 1331), (1200, 50, 1332), (1200, 60, 2662), (1200, 60, 2664),
                                   (532, 64, 2048), (533, 64, 2048), (1064, 33, 1999), (1066, 33, 1999),
                                   (2200, 40, 1900), (4096, 20, 4096)])
def test_sparse_product_around_the_line(rd, orc, M, K, N, R):
    import torch

    a, b = operands(M, K, N, 0.2, M + N)
    C = torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")
    low = torch.zeros(1, dtype=torch.int32, device="cuda")
    rd.sparse_minplus(rd.sparse_plan(upload(a), M, K, R=R), upload(b), C, N=N, min_out=low)
    got, want = C.cpu().numpy(), orc.minplus_i16(a, b)
    assert np.array_equal(got[:, :N].astype(np.int32), want)
    assert (got[:, N:] == -7).all() and int(low) == int(want.min())


def test_random_operands_with_full_slabs_are_not_slower_than_a_longer_product(rd):
    """4096 columns and 4104 take the same number of 2048-column slabs but for one nearly empty third: the product of
    4096 must not take longer.  (With a warp per block it took 1.3 times as long.)"""
    import torch

    M, K, ms = 4000, 4000, {}
    a, b = operands(M, K, 4104, 0.02, 3)
    plan, B = rd.sparse_plan(upload(a), M, K, R=2), upload(b)
    C = torch.empty((M, 4104), dtype=torch.int16, device="cuda")
    for N in (4096, 4104):
        best = 1e9
        for _ in range(6):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            for _ in range(20):
                rd.sparse_minplus(plan, B, C, N=N)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        ms[N] = best
    assert ms[4096] <= ms[4104], ms
