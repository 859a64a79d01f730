"""The tensor-core tile of the dense (min,+) product against the oracle, bit for bit (integer work: no tolerance).

The batched entry point tries it for every K >= 64, so small shapes reach it.  Shapes sit at the edges of its tiles
(256 rows and 512 columns per pair of CTAs, halves of 128 and 256), its 64-term stages and its early look (from
40 stages on); the values decide whether an output is decided, computed term by term, or left to the DPX tile.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF = 0x3FFF
SHAPES = [(1, 8, 64), (2, 9, 65), (128, 256, 64), (129, 257, 127), (256, 512, 128), (257, 513, 129), (127, 255, 192),
          (255, 511, 191), (300, 521, 1023), (260, 515, 1024), (130, 1025, 1600), (140, 601, 2496), (257, 513, 2561)]


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

    def draw(rows, cols, top, inf):
        return np.where(r.random((rows, cols)) < inf, INF, r.integers(0, top, (rows, cols))).astype(np.int16)

    if kind == "small":     # every output decided
        return draw(M, K, 4, 0.1), draw(K, N, 4, 0.1)
    if kind == "u32":       # at small K some outputs undecided
        return draw(M, K, 33, 0.5), draw(K, N, 33, 0.5)
    if kind == "wide":      # not tried
        return draw(M, K, 0x2000, 0.5), draw(K, N, 0x2000, 0.5)
    if kind == "holes":     # rows without a finite entry: undecided everywhere along them
        a, b = draw(M, K, 4, 0.1), draw(K, N, 4, 0.1)
        a[::5] = INF
        return a, b
    a, b = draw(M, K, 4, 0.1), draw(K, N, 4, 0.1)  # "halves": worth trying, then large over half of the terms' rows
    a[M // 2:] = np.where(a[M // 2:] == INF, INF, a[M // 2:] + 0x1000)
    return a, b


def upload(host, junk):
    import torch

    rows, cols = host.shape
    t = torch.full((rows, (cols + 7) // 8 * 8), junk, dtype=torch.int16)
    t[:, :cols] = torch.from_numpy(host)
    return t.cuda()


@pytest.mark.parametrize("kind", ["small", "u32", "wide", "holes", "halves"])
def test_batched_products_on_the_tensor_cores(rd, orc, kind):
    import torch

    problems, want = [], []
    for i, (M, N, K) in enumerate(SHAPES):
        a, b = operands(kind, M, N, K, 100 + i)
        C = torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")
        # the padding is never part of the result, whatever it holds
        problems.append((upload(a, -3), upload(b, -5), C, M, N, K, torch.zeros(1, dtype=torch.int32, device="cuda")))
        want.append(orc.minplus_i16(a, b))
    for _ in range(2):  # the same buffers again: marks of the first call are gone
        rd.minplus_gemm_batched(problems)
    for (_, _, C, M, N, K, low), w in zip(problems, want):
        got = C.cpu().numpy()
        assert np.array_equal(got[:, :N].astype(np.int32), w), (kind, M, N, K)
        assert (got[:, N:] == -7).all() and int(low) == int(w.min()), (kind, M, N, K)


@pytest.mark.parametrize("kind", ["u32", "wide", "halves"])
def test_one_product_on_the_tensor_cores(rd, orc, kind):
    """A product large enough for rd_minplus_gemm to try them, ragged in every dimension; sampled entries."""
    import torch

    M, N, K = 2100, 2301, 2130
    a, b = operands(kind, M, N, K, 7)
    C = torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")
    low = torch.zeros(1, dtype=torch.int32, device="cuda")
    rd.minplus_gemm(upload(a, -3), upload(b, -5), C, M, N, K, min_out=low)
    got = C.cpu().numpy()
    r = np.random.default_rng(1)
    ri = np.concatenate([r.integers(0, M, 3000), np.full(N, M - 1)])
    cj = np.concatenate([r.integers(0, N, 3000), np.arange(N)])
    assert np.array_equal(got[ri, cj].astype(np.int32), orc.minplus_i16_entries(a, b, ri, cj))
    assert (got[:, N:] == -7).all() and int(low) == int(got[:, :N].min())


def test_entries_outside_the_range_keep_their_result(rd):
    """Entries with bit 14 or 15 set (outside the documented range) take the DPX tile, whose sums wrap at 16 bits."""
    import torch

    M, N, K = 200, 300, 256
    a, b = operands("small", M, N, K, 3)
    a[150, 17], b[40, 299] = -9, 0x4001
    A, B = upload(a, INF), upload(b, INF)
    C = torch.empty((M, 304), dtype=torch.int16, device="cuda")
    rd.minplus_gemm_batched([(A, B, C, M, N, K, None)])
    with np.errstate(over="ignore"):
        s = np.minimum(INF, np.array([(a[i][:, None] + b).min(0) for i in range(M)], dtype=np.int16)).astype(np.int32)
    assert np.array_equal(C.cpu().numpy()[:, :N].astype(np.int32), s)


@pytest.mark.parametrize("dist", ["u32", "wide"])
@pytest.mark.parametrize("K", [33, 64, 65, 100, 129, 161, 193, 225, 257])
def test_small_products_split_k_in_any_number_of_slices(rd, orc, K, dist):
    """Few output tiles: K is cut into 2 .. 8 slices of whole k-tiles, not only powers of two, and the slices' rows of
    the tile into uneven shares."""
    import torch

    for i, (M, N) in enumerate([(2, 8), (97, 130), (128, 128), (129, 257), (300, 201)]):
        a, b = operands(dist, M, N, K, 40 + i)
        C = torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")
        low = torch.zeros(1, dtype=torch.int32, device="cuda")
        rd.minplus_gemm(upload(a, -3), upload(b, -5), C, M, N, K, min_out=low)
        w, got = orc.minplus_i16(a, b), C.cpu().numpy()
        assert np.array_equal(got[:, :N].astype(np.int32), w), (M, N, K)
        assert (got[:, N:] == -7).all() and int(low) == int(w.min()), (M, N, K)


@pytest.mark.parametrize("kind", ["u32", "wide", "halves"])
def test_captured_product_replays(rd, kind):
    """Both launches of a product in a CUDA graph, replayed over a result of other values."""
    import torch

    M, N, K = 1500, 1300, 1200
    a, b = operands(kind, M, N, K, 9)
    A, B = upload(a, INF), upload(b, INF)
    want, C = (torch.full((M, 1304), -7, dtype=torch.int16, device="cuda") for _ in range(2))
    low = torch.zeros(1, dtype=torch.int32, device="cuda")
    rd.minplus_gemm(A, B, want, M, N, K)
    torch.cuda.synchronize()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        rd.minplus_gemm(A, B, C, M, N, K, min_out=low, stream=stream)
    for _ in range(3):
        C.fill_(0)
        C[:, N:] = -7
        graph.replay()
    assert torch.equal(C, want) and int(low) == int(want[:, :N].min())
