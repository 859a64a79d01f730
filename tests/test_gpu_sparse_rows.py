"""The warp-per-block kernel of the block-sparse product (operands of at most 4096 rows and columns) against the
oracle, bit for bit: edges of its 256-column slabs, of its 32-entry chunks and of the blocks per CTA."""
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


@pytest.mark.parametrize("R", [1, 2, 4, 8])
@pytest.mark.parametrize("M,K,N,finite", [(1, 1, 1, 1.0), (3, 40, 8, 0.9), (33, 31, 255, 0.5), (70, 65, 256, 1.0),
                                          (129, 300, 257, 0.3), (500, 97, 1030, 0.02), (4096, 64, 40, 0.2),
                                          (20, 128, 4096, 0.4), (4097, 40, 48, 0.3)])
def test_sparse_product(rd, orc, M, K, N, finite, R):
    import torch

    r = np.random.default_rng(M * 7 + K * 3 + N)
    a = np.where(r.random((M, K)) < finite, r.integers(0, 40, (M, K)), INF).astype(np.int16)
    b = np.where(r.random((K, N)) < 0.9, r.integers(0, 0x2000, (K, N)), INF).astype(np.int16)

    def upload(h):
        t = torch.full((h.shape[0], (h.shape[1] + 7) // 8 * 8), -3, dtype=torch.int16)
        t[:, :h.shape[1]] = torch.from_numpy(h)
        return t.cuda()

    A, B = upload(a), upload(b)
    C = torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")
    low = torch.zeros(1, dtype=torch.int32, device="cuda")
    rd.sparse_minplus(rd.sparse_plan(A, M, K, R=R), B, C, N=N, min_out=low)
    got, want = C.cpu().numpy(), orc.minplus_i16(a, b)
    assert np.array_equal(got[:, :N].astype(np.int32), want)
    assert (got[:, N:] == -7).all() and int(low) == int(want.min())
