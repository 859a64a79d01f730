"""Cases of the tensor-core tile that need the checked build of the library (librd_checked.so, -DRD_CHECKED): a wait
that runs out, and which path computed a product.

Not collected by a plain `pytest tests` (the file name does not start with test_): test_gpu_tc_checked.py runs it in a
child process.
"""
import ctypes
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

INF = 0x3FFF


@pytest.fixture(scope="module")
def rd():
    lib = os.environ.get("RD_CHECKED_LIB")
    if not lib:
        pytest.fail("run by test_gpu_tc_checked.py under the checked build")
    import paper_2409_17658_gb300 as rd

    prev = rd.use_library(lib)
    yield rd
    rd.use_library_handle(prev)


def check(rd, wait_rounds=1 << 18, hold_at=-1, hold_us=0, deaf=0):
    """Applies settings (by default: the ordinary ones); returns the counts since the last call."""
    settings = (ctypes.c_uint32 * 4)(wait_rounds, hold_at & 0xFFFFFFFF, hold_us, deaf)
    counts = (ctypes.c_uint32 * 5)()
    assert rd._lib().rd_tc_check(settings, counts) == rd.RD_OK
    return dict(zip(("decided", "fixed", "left", "lost", "early"), counts))


@pytest.fixture(autouse=True)
def ordinary_settings(rd):
    check(rd)
    yield
    check(rd)


def draw(rows, cols, top, inf, seed):
    r = np.random.default_rng(seed)
    return np.where(r.random((rows, cols)) < inf, INF, r.integers(0, top, (rows, cols))).astype(np.int16)


def upload(host):
    import torch

    t = torch.full((host.shape[0], (host.shape[1] + 7) // 8 * 8), -3, dtype=torch.int16)
    t[:, :host.shape[1]] = torch.from_numpy(host)
    return t.cuda()


def result(M, N):
    import torch

    return torch.full((M, (N + 7) // 8 * 8), -7, dtype=torch.int16, device="cuda")


def assert_product(orc, a, b, C, seed=1):
    """Sampled entries, and the last row and column, against the oracle."""
    M, N = a.shape[0], b.shape[1]
    r = np.random.default_rng(seed)
    ri = np.concatenate([r.integers(0, M, 20000), np.full(N, M - 1), np.arange(M)])
    cj = np.concatenate([r.integers(0, N, 20000), np.arange(N), np.full(M, N - 1)])
    got = C.cpu().numpy()
    assert np.array_equal(got[ri, cj].astype(np.int32), orc.minplus_i16_entries(a, b, ri, cj))
    assert (got[:, N:] == -7).all()


def parts(M, N):
    return -(-M // 128) * -(-N // 256)


# (M, N, K) and the stage of a tile: tiles of 256 columns, three for the pair that is held; tiles of 512, two; the same
# with an early look behind that stage
LOST = [(256 * 76 * 2 + 300, 250, 600, 5), (256 * 30, 2500, 700, 5), (256 * 30, 2500, 2600, 2)]


@pytest.mark.parametrize("tile", [0, 1])
@pytest.mark.parametrize("M,N,K,stage", LOST)
def test_a_wait_that_runs_out_leaves_the_rest_of_the_pair(rd, orc, M, N, K, stage, tile):
    """The held pair's MMA warp comes back after every other thread has given up; its tiles from that one on are the
    DPX launch's, the others' are not, and the next product finds nothing changed."""
    a, b = draw(M, K, 4, 0.1, 1), draw(K, N, 4, 0.1, 2)
    A, B, C = upload(a), upload(b), result(M, N)
    check(rd, wait_rounds=256, hold_at=tile * -(-K // 64) + stage, hold_us=100_000)
    rd.minplus_gemm(A, B, C, M, N, K)
    seen = check(rd)
    assert seen["lost"] == 1 and seen["left"] >= 2 and seen["decided"] + seen["left"] == parts(M, N), seen
    assert_product(orc, a, b, C)
    C.fill_(-7)
    rd.minplus_gemm(A, B, C, M, N, K)
    seen = check(rd)
    assert seen == dict(decided=parts(M, N), fixed=seen["fixed"], left=0, lost=0, early=0), seen
    assert_product(orc, a, b, C)


def test_a_wait_that_runs_out_in_a_batch(rd, orc):
    shapes = [(256 * 20, 2000, 640), (3000, 3001, 600), (700, 520, 200)]
    host = [(draw(M, K, 4, 0.1, i), draw(K, N, 4, 0.1, 9 + i)) for i, (M, N, K) in enumerate(shapes)]
    problems = [(upload(a), upload(b), result(M, N), M, N, K, None) for (a, b), (M, N, K) in zip(host, shapes)]
    check(rd, wait_rounds=256, hold_at=3, hold_us=100_000)
    rd.minplus_gemm_batched(problems)
    seen = check(rd)
    total = sum(parts(M, N) for M, N, _ in shapes)
    assert seen["lost"] == 1 and seen["left"] >= 2 and seen["decided"] + seen["left"] == total, seen
    for (a, b), p in zip(host, problems):
        assert_product(orc, a, b, p[2])


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("deaf", [1, 2, 3])
def test_both_ctas_of_a_pair_go_by_one_answer(rd, orc, deaf, batched):
    """One CTA of every pair finds nothing in its half of the sample, the other everything: both take the tensor cores
    (their counts together still say so).  Neither finds anything: both leave every part."""
    M, N, K = 2000, 1801, 1000
    a, b = draw(M, K, 4, 0.1, 5), draw(K, N, 4, 0.1, 6)
    A, B, C = upload(a), upload(b), result(M, N)
    check(rd, deaf=deaf)
    if batched:  # two products: the question is asked anew for each
        C2 = result(M, N)
        rd.minplus_gemm_batched([(A, B, C, M, N, K, None), (A, B, C2, M, N, K, None)])
    else:
        rd.minplus_gemm(A, B, C, M, N, K)
    seen, n = check(rd), parts(M, N) * (2 if batched else 1)
    assert (seen["decided"], seen["lost"]) == (0 if deaf == 3 else n, 0), seen
    assert_product(orc, a, b, C)
    if batched:
        assert_product(orc, a, b, C2)


@pytest.mark.parametrize("M,N,K", [(1300, 1000, 1100), (2000, 1801, 1000)])
def test_operands_and_result_in_interleaved_rows(rd, orc, M, N, K):
    """A, B and C side by side in the rows of one parent (row strides far above their widths)."""
    import torch

    ld = 2048
    parent = torch.full((max(M, K), 3 * ld), -7, dtype=torch.int16)
    a, b = draw(M, K, 33, 0.5, 7), draw(K, N, 33, 0.5, 8)
    parent[:M, :K], parent[:K, ld:ld + N] = torch.from_numpy(a), torch.from_numpy(b)
    parent = parent.cuda()
    before, C = parent.clone(), parent[:M, 2 * ld:]
    rd.minplus_gemm(parent[:M, :ld], parent[:K, ld:2 * ld], C, M, N, K)
    seen = check(rd)
    assert seen["decided"] == parts(M, N) and seen["left"] == 0, seen
    assert_product(orc, a, b, C)
    C[:, :N] = -7
    assert torch.equal(parent, before)


def structured(kind, n, seed):
    """Operands uniform in [0, 32] with infinity at probability 1/2, and infinite by a pattern."""
    a, b = draw(n, n, 33, 0.5, seed), draw(n, n, 33, 0.5, seed + 1)
    if kind == "blocks":  # two diagonal blocks
        for x in (a, b):
            x[: n // 2, n // 2:] = x[n // 2:, : n // 2] = INF
    elif kind == "triangle":
        for x in (a, b):
            x[np.tril_indices(n, -1)] = INF
    elif kind == "columns":
        b[:, ::2] = INF
    elif kind == "odd rows":
        a[1::2] = INF
    elif kind == "half the rows":
        a[: n // 2] = INF
    elif kind == "apart":  # small entries of A meet large ones of B
        a[:, : n // 2] = np.where(a[:, : n // 2] == INF, INF, a[:, : n // 2] + 0x800)
        b[n // 2:] = np.where(b[n // 2:] == INF, INF, b[n // 2:] + 0x800)
    return a, b


@pytest.mark.parametrize("n", [1024, 1500])
@pytest.mark.parametrize("kind", ["even", "blocks", "triangle", "columns", "odd rows", "half the rows", "apart"])
def test_the_sample_sees_what_stays_undecided(rd, orc, kind, n):
    """Sizes where the DPX launch gains nothing from the tiles that the tensor cores decide: none is tried unless the
    hits are spread over the whole product."""
    a, b = structured(kind, n, 11)
    C = result(n, n)
    rd.minplus_gemm(upload(a), upload(b), C, n, n, n)
    seen = check(rd)
    want = (parts(n, n), 0) if kind == "even" else (0, parts(n, n))
    assert (seen["decided"], seen["left"]) == want, seen
    assert_product(orc, a, b, C)


def test_large_products_are_decided_in_part(rd, orc):
    """2048^3 with the upper half of A's rows infinite: the lower half's parts on the tensor cores, the others not."""
    n = 2048
    a, b = structured("half the rows", n, 21)
    C = result(n, n)
    rd.minplus_gemm(upload(a), upload(b), C, n, n, n)
    seen = check(rd)
    assert (seen["decided"], seen["left"]) == (parts(n, n) // 2, parts(n, n) // 2), seen
    assert_product(orc, a, b, C)


def test_outputs_computed_term_by_term(rd, orc):
    """A few rows' worth of single outputs without a small pair: computed beside the decided ones, not left."""
    n = 1100
    a, b = draw(n, n, 33, 0.5, 31), draw(n, n, 33, 0.5, 32)
    a[700] = np.where(np.arange(n) % 64 == 0, a[700], INF)  # 17 terms: part of the row stays undecided
    b[:, 40:1000] = np.where(b[:, 40:1000] == INF, INF, b[:, 40:1000] % 4)
    b[:, :8] = np.where(np.arange(n)[:, None] % 60 == 0, b[:, :8], INF)
    C = result(n, n)
    rd.minplus_gemm(upload(a), upload(b), C, n, n, n)
    seen = check(rd)
    assert seen["decided"] + seen["left"] == parts(n, n) and seen["decided"] > 0, seen
    assert_product(orc, a, b, C)


@pytest.mark.parametrize("count,n,tried", [(1, 100, False), (64, 100, False), (128, 64, False), (100, 128, False),
                                           (1, 200, True), (16, 500, True), (128, 256, True)])
def test_small_batches_stay_on_dpx(rd, orc, count, n, tried):
    """The tensor cores are tried where the modeled schedules say so, for the batch as a whole."""
    host = [(draw(n, n, 4, 0.1, 40 + i), draw(n, n, 4, 0.1, 90 + i)) for i in range(3)]
    dev = [(upload(a), upload(b)) for a, b in host]
    outs = [result(n, n) for _ in range(count)]
    rd.minplus_gemm_batched([(*dev[i % 3], C, n, n, n, None) for i, C in enumerate(outs)])
    seen = check(rd)
    assert (seen["decided"], seen["left"]) == (count * parts(n, n) if tried else 0, 0), seen
    want = [orc.minplus_i16(a, b) for a, b in host]
    for i, C in enumerate(outs):
        got = C.cpu().numpy()
        assert np.array_equal(got[:, :n].astype(np.int32), want[i % 3]) and (got[:, n:] == -7).all()


# both tile widths: 256 columns (the first four, two of them with several tiles per pair of CTAs) and 512; N cuts a
# 16-byte chunk of B
WIDTHS = [(1000, 1001, 2600), (1500, 1300, 1200), (40000, 250, 600), (39212, 249, 2600), (2100, 2301, 2130),
          (4000, 4001, 2600)]


@pytest.mark.parametrize("M,N,K", WIDTHS)
def test_every_part_is_decided_on_the_tensor_cores(rd, orc, M, N, K):
    a, b = draw(M, K, 33, 0.5, 51), draw(K, N, 33, 0.5, 52)
    C = result(M, N)
    rd.minplus_gemm(upload(a), upload(b), C, M, N, K)
    seen = check(rd)
    assert seen == dict(decided=parts(M, N), fixed=seen["fixed"], left=0, lost=0, early=0), seen
    assert_product(orc, a, b, C)


@pytest.mark.parametrize("M,N,K", [(39212, 249, 2600), (4000, 4001, 2600)])
def test_the_early_look_turns_tiles_away(rd, orc, M, N, K):
    """A's lower half holds large entries: its tiles are left an eighth of the way, the upper half's are decided, and the
    tile across the middle at its end or by the look."""
    a, b = draw(M, K, 33, 0.5, 53), draw(K, N, 33, 0.5, 54)
    a[M // 2:] = np.where(a[M // 2:] == INF, INF, a[M // 2:] + 0x1000)
    C = result(M, N)
    rd.minplus_gemm(upload(a), upload(b), C, M, N, K)
    seen, columns = check(rd), -(-N // 256)
    tiles = (-(-M // 256) - (M // 2 + 255) // 256) * (1 if N <= 256 else -(-N // 512))  # whole rows of tiles below it
    assert seen["early"] >= tiles and seen["lost"] == 0, (seen, tiles)
    assert seen["decided"] >= M // 2 // 256 * 2 * columns and seen["decided"] + seen["left"] == parts(M, N), seen
    assert_product(orc, a, b, C)
