"""rd_tune_gemm against the shape that a product runs without an entry, which may split K in 3, 5, 6 or 7 (no entry of
the table says that): tuning never makes the product slower."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rd():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    return rd


@pytest.fixture(autouse=True)
def empty_table(rd):
    rd.tune_set([])
    yield
    rd.tune_set([])


def microseconds(f):
    import torch

    best = 1e9
    for _ in range(8):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        for _ in range(50):
            f()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 20)
    return best


@pytest.mark.parametrize("M,N,K", [(800, 800, 800), (300, 300, 300), (200, 300, 600), (1000, 1187, 633)])
def test_tuning_does_not_make_a_product_slower(rd, orc, M, N, K):
    """The sizes' own shapes split K in 5 or 7, and their products stay on the DPX units; an entry for the size class that
    was there before (a slow one) goes where none is needed."""
    import torch
    from paper_2409_17658_gb300 import inputs

    a, b = inputs.matrix(M, K, seed=3, dist="wide"), inputs.matrix(K, N, seed=4, dist="wide")

    def upload(h):
        t = torch.full((h.shape[0], (h.shape[1] + 7) // 8 * 8), -3, dtype=torch.int16)
        t[:, :h.shape[1]] = torch.from_numpy(h)
        return t.cuda()

    A, B = upload(a), upload(b)
    C = torch.empty((M, (N + 7) // 8 * 8), dtype=torch.int16, device="cuda")
    product = lambda: rd.minplus_gemm(A, B, C, M, N, K)
    product()
    own = microseconds(product)
    key, aux = rd.tune_bucket(max(M, N)), rd.tune_bucket(K)
    other = dict(mode="sparse_r", key=1, aux=0, p=[1, 0, 0, 0], ms=-1.0)
    rd.tune_set([dict(mode="gemm_splitk", key=key, aux=aux, p=[1, 0, 0, 0], ms=-1.0), other])
    e = rd.tune_gemm(A, B, C, M, N, K, reps=20)
    kept = rd.tune_lookup(rd.RD_TUNE_GEMM_SPLITK, key, aux)
    assert kept is None or kept == e
    assert rd.tune_lookup(rd.RD_TUNE_SPARSE_R, 1, 0) == other and len(rd.tune_table()) == (1 if kept is None else 2)
    tuned = microseconds(product)
    print(M, N, K, own, tuned, e, kept)
    assert tuned <= 1.06 * own, (own, tuned, e)
    rd.tune_set([e])  # what it returns can be set
    assert np.array_equal(C.cpu().numpy()[:, :N].astype(np.int32), orc.minplus_i16(a, b))
