"""The workloads whose time is measured, through the package's public entry points.

Kinds of case ("kind"):
  gemm    one dense (min,+) product C = A (x) B (rd_minplus_gemm);
  gemv    one row vector times a matrix (rd_minplus_gemv);
  batch   many uneven dense products in one call (rd_minplus_gemm_batched);
  split   one power step A(G) (x) B through the row-split plan (rd_split_minplus);
  sparse  the same product through the block-sparse form of A (rd_sparse_minplus);
  gamma   gamma_R queries of one m from an empty cache (rd_gamma_R): states, A(G), the plan and the
          whole period search;
  server  a fresh query server answering one batch of (m, n) queries (rd_server_*).

Entries of dense operands: "u32" is uniform in [0, 32] with infinity at probability 1/2 (the synthetic
workload of bench.py); "wide" is uniform over the whole finite range [0, 0x1FFF] with infinity at
probability 1/2.  The right operand of a power step is a normalised power: all finite, a few multiples
of m wide.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2409_17658_gb300 as rd
from paper_2409_17658_gb300 import inputs

INF = rd.RD_INF
EXACT_MOST = 10 ** 11  # add-mins that exact() computes

# C_m, the number of correct words (Table 1 of the paper), m = 1..10
STATES = {1: 4, 2: 11, 3: 33, 4: 97, 5: 287, 6: 848, 7: 2507, 8: 7411, 9: 21909, 10: 64769}
# arcs of A(G): the finite entries that a product combines with each column
ARCS = {1: 7, 2: 33, 3: 167, 4: 836, 5: 4195, 6: 21043, 7: 105566, 8: 529584, 9: 2656733, 10: 13327868}


def listed() -> list[dict]:
    return [
        dict(name="gemm_97x130x161", kind="gemm", M=97, N=130, K=161, dist="u32"),
        dict(name="gemm_1024", kind="gemm", M=1024, N=1024, K=1024, dist="u32"),
        dict(name="gemm_2507x3001x1999", kind="gemm", M=2507, N=3001, K=1999, dist="u32"),
        dict(name="gemm_4096_wide", kind="gemm", M=4096, N=4096, K=4096, dist="wide"),
        dict(name="gemm_16384", kind="gemm", M=16384, N=16384, K=16384, dist="u32"),
        dict(name="gemv_16384", kind="gemv", N=16384, K=16384, dist="u32"),
        dict(name="batch_64", kind="batch", count=64, lo=128, hi=8192, sizes=4, dist="u32"),
        dict(name="split_m8", kind="split", m=8),
        dict(name="split_m10", kind="split", m=10),
        dict(name="sparse_m9", kind="sparse", m=9, R=2),
        dict(name="gamma_m9", kind="gamma", m=9, queries=16),
        dict(name="server_m2_8", kind="server", lo=2, hi=8, queries=256),
    ]


def _log_uniform(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["gemm", "gemm", "gemm", "gemv", "batch", "split", "split", "sparse", "gamma", "server"])
    if kind == "gemm":
        dist = rng.choice(["u32", "u32", "wide"])
        return dict(kind="gemm", M=_log_uniform(rng, 64, 12288), N=_log_uniform(rng, 64, 12288),
                    K=_log_uniform(rng, 64, 12288), dist=dist)
    if kind == "gemv":
        return dict(kind="gemv", N=_log_uniform(rng, 256, 32768), K=_log_uniform(rng, 256, 32768), dist="u32")
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(8, 64), lo=128, hi=_log_uniform(rng, 512, 8192),
                    sizes=rng.randint(1, 10 ** 6), dist="u32")
    if kind == "split":
        return dict(kind="split", m=rng.randint(5, 10), values=rng.randint(2, 4))
    if kind == "sparse":
        return dict(kind="sparse", m=rng.randint(5, 9), R=rng.choice([1, 2, 4]))
    if kind == "gamma":
        return dict(kind="gamma", m=rng.randint(2, 9), queries=rng.randint(1, 64))
    lo = rng.randint(2, 6)
    return dict(kind="server", lo=lo, hi=rng.randint(lo, 9), queries=rng.randint(8, 3000))


def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _matrix(rows: int, cols: int, dist: str, g) -> torch.Tensor:
    """rows x cols entries in rows of padded_dim(cols); the padding holds infinity."""
    top = 33 if dist == "u32" else rd.RD_MAX_FINITE + 1
    out = torch.randint(0, top, (rows, rd.padded_dim(cols)), generator=g, device="cuda", dtype=torch.int16)
    for r in range(0, rows, 4096):  # in parts: the draws are larger than the matrix
        part = out[r:r + 4096]
        part[torch.rand(part.shape, generator=g, device="cuda") < 0.5] = INF
    out[:, cols:] = INF
    return out


def _power_like(n: int, m: int, values: int, g) -> torch.Tensor:
    return torch.randint(0, values * m + 1, (n, rd.padded_dim(n)), generator=g, device="cuda", dtype=torch.int16)


def _batch_sizes(case: dict) -> list[int]:
    return inputs.log_uniform_sizes(case["count"], case["lo"], case["hi"], case["sizes"])


def prepare(case: dict, seed: int) -> dict:
    kind, g = case["kind"], _generator(seed)
    state = dict(case=case)
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        state.update(A=_matrix(M, K, case["dist"], g), B=_matrix(K, N, case["dist"], g),
                     C=torch.empty((M, rd.padded_dim(N)), dtype=torch.int16, device="cuda"))
    elif kind == "gemv":
        N, K = case["N"], case["K"]
        state.update(x=_matrix(1, K, case["dist"], g)[0, :K], B=_matrix(K, N, case["dist"], g),
                     y=torch.empty(rd.padded_dim(N), dtype=torch.int16, device="cuda"))
    elif kind == "batch":
        state["problems"] = [
            (_matrix(n, n, case["dist"], g), _matrix(n, n, case["dist"], g),
             torch.empty((n, rd.padded_dim(n)), dtype=torch.int16, device="cuda"), n, n, n, None)
            for n in _batch_sizes(case)]
    elif kind == "split":
        m = case["m"]
        n = rd.state_count(m)
        state.update(n=n, plan=rd.split_plan(m), B=_power_like(n, m, case.get("values", 3), g),
                     C=torch.empty((n, rd.padded_dim(n)), dtype=torch.int16, device="cuda"))
    elif kind == "sparse":
        m = case["m"]
        A, n = rd.transfer_matrix(m)
        state.update(n=n, plan=rd.sparse_plan(A, n, n, R=case["R"]), B=_power_like(n, m, 3, g),
                     C=torch.empty((n, rd.padded_dim(n)), dtype=torch.int16, device="cuda"))
    elif kind == "gamma":
        state["ns"] = [int(v) for v in np.random.default_rng(seed).integers(3, 1001, case["queries"])]
    elif kind == "server":
        r = np.random.default_rng(seed)
        state["ms"] = r.integers(case["lo"], case["hi"] + 1, case["queries"]).astype(np.int32)
        state["ns"] = r.integers(3, 201, case["queries"]).astype(np.int64)
    return state


def run(state: dict):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        rd.minplus_gemm(state["A"], state["B"], state["C"], M, N, K)
        return state["C"][:, :N]
    if kind == "gemv":
        rd.minplus_gemv(state["x"], state["B"], state["y"], case["N"], case["K"])
        return state["y"][:case["N"]]
    if kind == "batch":
        rd.minplus_gemm_batched(state["problems"])
        return [p[2][:, :p[4]] for p in state["problems"]]
    if kind == "split":
        rd.split_minplus(state["plan"], state["B"], state["C"])
        return state["C"][:, :state["n"]]
    if kind == "sparse":
        rd.sparse_minplus(state["plan"], state["B"], state["C"], N=state["n"])
        return state["C"][:, :state["n"]]
    if kind == "gamma":
        rd.gamma_R_clear()
        return np.array([rd.gamma_R(case["m"], n) for n in state["ns"]], dtype=np.int64)
    with rd.Server(hbm_budget_bytes=64 << 30) as server:
        gamma, status, _ = server.wait(server.submit(state["ms"], state["ns"]))
    return dict(gamma=gamma, status=status)


def work(case: dict) -> dict:
    """Bytes: operands read once, results written once.  Operations: an add and a min per combined pair
    (dense: every pair; A(G): its arcs times the columns; a search: one such product and one pass over the
    power for each power up to the first repeat, about 2 m + 8 of them)."""
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=2 * (M * K + K * N + M * N), flops=2 * M * N * K)
    if kind == "gemv":
        N, K = case["N"], case["K"]
        return dict(bytes=2 * (K + K * N + N), flops=2 * N * K)
    if kind == "batch":
        sizes = _batch_sizes(case)
        return dict(bytes=sum(6 * n * n for n in sizes), flops=sum(2 * n ** 3 for n in sizes))
    if kind in ("split", "sparse"):
        n = STATES[case["m"]]
        return dict(bytes=4 * n * n, flops=2 * ARCS[case["m"]] * n)
    ms = [case["m"]] if kind == "gamma" else range(case["lo"], case["hi"] + 1)
    steps = {m: 2 * m + 8 for m in ms}
    return dict(bytes=sum(4 * STATES[m] ** 2 * steps[m] for m in ms),
                flops=sum(2 * ARCS[m] * STATES[m] * steps[m] for m in ms))


def _exact_product(A: torch.Tensor, B: torch.Tensor) -> torch.Tensor:
    """min_t A[i][t] + B[t][j] in 64 bits; infinity where no term is finite."""
    big = 1 << 40
    A = torch.where(A == INF, big, A.to(torch.int64))
    B = torch.where(B == INF, big, B.to(torch.int64)).t().contiguous()
    out = torch.empty((A.shape[0], B.shape[0]), dtype=torch.int64, device=A.device)
    rows = max(1, (1 << 28) // max(1, B.numel()))
    for r in range(0, A.shape[0], rows):
        out[r:r + rows] = (A[r:r + rows, None, :] + B[None]).amin(2)
    return torch.where(out >= big, INF, out)


def _transfer(m: int) -> torch.Tensor:
    """A(G) from the word and row rules of Sec. 4.A (words in lexicographic order, a = 0 .. d = 3)."""
    words = [w for w in np.ndindex(*([4] * m))
             if not any(p in ((0, 3), (3, 0), (0, 1), (1, 0), (1, 1)) for p in zip(w, w[1:]))]
    W = np.array(words, dtype=np.int64)
    n = len(W)
    label = 2 * (W == 0).sum(1) + (W == 1).sum(1)
    near_a = np.zeros((n, m), dtype=bool)
    near_a[:, 1:] |= W[:, :-1] == 0
    near_a[:, :-1] |= W[:, 1:] == 0
    # rows: the letter of q_i; columns: p_i = a, b, c beside an a, d, c beside none
    admits = np.array([[1, 0, 1, 0, 1], [0, 0, 1, 1, 0], [1, 1, 1, 1, 0], [1, 0, 0, 0, 0]], dtype=bool)
    kind = np.where((W == 2) & ~near_a, 4, W)
    ok = np.ones((n, n), dtype=bool)
    for i in range(m):
        ok &= admits[W[:, i]][:, kind[:, i]]
    return torch.from_numpy(np.where(ok, label[None, :], INF)).cuda()


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind in ("gamma", "server"):
        return None
    if kind in ("split", "sparse"):
        if STATES[case["m"]] ** 3 > EXACT_MOST:
            return None
        n = STATES[case["m"]]
        return _exact_product(_transfer(case["m"]), prepare(case, seed)["B"][:, :n])
    if kind == "gemv":
        if case["N"] * case["K"] > EXACT_MOST:
            return None
        s = prepare(case, seed)
        return _exact_product(s["x"][None], s["B"][:, :case["N"]])[0]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        if M * N * K > EXACT_MOST:
            return None
        s = prepare(case, seed)
        return _exact_product(s["A"][:, :K], s["B"][:, :N])
    return [_exact_product(A[:, :K], B[:, :N]) if M * N * K <= EXACT_MOST // 64 else None
            for A, B, _, M, N, K, _ in prepare(case, seed)["problems"]]
