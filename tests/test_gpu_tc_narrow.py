"""The tensor-core product in its narrow form (tiles of 256 columns) and at ragged edges, against the oracle and, entry by
entry, against the stream-K product (DPX units only): N cut inside a 16-byte chunk of B, several tiles per pair of
CTAs, the early look (K >= 2497), views with wide strides, results of fewer than 8 columns, a captured product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF = 0x3FFF
SHAPES = [(1000, 1001, 2600), (1500, 1300, 1200), (40000, 250, 600), (39212, 249, 2600), (5000, 703, 2600)]


@pytest.fixture(scope="module")
def rd():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2409_17658_gb300 import build

    build.build()
    import paper_2409_17658_gb300 as rd

    return rd


def operands(kind, M, N, K, seed):
    r = np.random.default_rng(seed)

    def draw(rows, cols):
        return np.where(r.random((rows, cols)) < 0.5, INF, r.integers(0, 33, (rows, cols))).astype(np.int16)

    a, b = draw(M, K), draw(K, N)
    if kind == "halves":  # the lower half's tiles are left, by the early look or at their end
        a[M // 2:] = np.where(a[M // 2:] == INF, INF, a[M // 2:] + 0x1000)
    return a, b


def upload(h, junk=-3):
    import torch

    t = torch.full((h.shape[0], (h.shape[1] + 7) // 8 * 8), junk, dtype=torch.int16)
    t[:, :h.shape[1]] = torch.from_numpy(h)
    return t.cuda()


def result(M, N):
    import torch

    return torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")


def assert_entries(orc, a, b, C):
    M, N = a.shape[0], b.shape[1]
    r = np.random.default_rng(1)
    ri = np.concatenate([r.integers(0, M, 4000), np.full(N, M - 1), r.integers(0, M, 2000)])
    cj = np.concatenate([r.integers(0, N, 4000), np.arange(N), np.full(2000, N - 1)])
    got = C.cpu().numpy()
    assert np.array_equal(got[ri, cj].astype(np.int32), orc.minplus_i16_entries(a, b, ri, cj))
    assert (got[:, N:] == -7).all()


@pytest.mark.parametrize("kind", ["u32", "halves"])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_narrow_tiles(rd, orc, M, N, K, kind):
    import torch

    a, b = operands(kind, M, N, K, M + N)
    A, B, C, D = upload(a), upload(b, -5), result(M, N), result(M, N)
    low = torch.zeros(1, dtype=torch.int32, device="cuda")
    rd.minplus_gemm(A, B, C, M, N, K, min_out=low)
    assert_entries(orc, a, b, C)
    rd.minplus_gemm_streamk(A, B, D, rd.minplus_gemm_streamk_workspace(M, N, K), M, N, K)
    assert torch.equal(C, D) and int(low) == int(C[:, :N].min())


@pytest.mark.parametrize("kind", ["u32", "halves"])
def test_captured_product_against_the_oracle(rd, orc, kind):
    import torch

    M, N, K = 1500, 1300, 1200
    a, b = operands(kind, M, N, K, 9)
    A, B, C = upload(a), upload(b), result(M, N)
    rd.minplus_gemm(A, B, C, M, N, K)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        rd.minplus_gemm(A, B, C, M, N, K, stream=stream)
    C[:, :N] = 0
    graph.replay()
    torch.cuda.synchronize()
    assert_entries(orc, a, b, C)


def test_views_with_wide_strides(rd, orc):
    """Operands and result are windows of wide parents: row strides of 4096, 8192 and 2048 entries."""
    import torch

    M, N, K = 1300, 1001, 1100
    a, b = operands("u32", M, N, K, 12)
    pa = torch.full((M, 4096), 1, dtype=torch.int16, device="cuda")
    pb = torch.full((K, 8192), 1, dtype=torch.int16, device="cuda")
    pc = torch.full((M, 2048), -7, dtype=torch.int16, device="cuda")
    pa[:, 1024:1024 + K] = torch.from_numpy(a).cuda()
    pb[:, 808:808 + N] = torch.from_numpy(b).cuda()
    rd.minplus_gemm(pa[:, 1024:], pb[:, 808:], pc[:, 520:], M, N, K)
    got = pc[:, 520:520 + (N + 7) // 8 * 8].contiguous()
    assert_entries(orc, a, b, got)
    pc[:, 520:520 + N] = -7
    assert bool((pc == -7).all())


def test_batch_of_very_narrow_results(rd, orc):
    """Fewer than 8 columns, beside a product that takes the batch to the tensor cores."""
    shapes = [(5, 3, 64), (300, 7, 200), (1, 1, 640), (2, 1, 2561), (700, 8, 1000), (900, 903, 2561)]
    host = [operands("u32", *s, 20 + i) for i, s in enumerate(shapes)]
    problems = [(upload(a), upload(b, -5), result(s[0], s[1]), *s, None) for (a, b), s in zip(host, shapes)]
    rd.minplus_gemm_batched(problems)
    for (a, b), p in zip(host, problems):
        got, N = p[2].cpu().numpy(), b.shape[1]
        assert np.array_equal(got[:, :N].astype(np.int32), orc.minplus_i16(a, b)) and (got[:, N:] == -7).all()
