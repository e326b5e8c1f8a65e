"""The work that a user of this library has it do, as cases that can be timed.

A case is a dict of plain values; its "kind" says which public entry points a
pass calls:

  update        one rank-k update of a factor (a new observation block comes in)
  pair          update by V, then downdate by 0.9 V: a block comes in and most
                of an earlier one leaves, as two calls
  mixed         the same in one call with a sign per vector
  solve         two triangular substitutions with the factor for nrhs
                right-hand sides
  modify_solve  modify the factor and solve with the modified one in one call
                (recursive least squares, an active-set or a filtering step)
  batch         many factors of uneven order in one planned execution, some
                updated and some downdated, then the opposite modifications
  serve         requests on resident factors through the server: submitted in
                a burst with V in page-locked host memory, drained, and the
                factors read back

Orders, vector counts and types are those of the library's own benchmark and
tests: the rank-1 pair at n = 512, the paper's n = 5000 with k = 16 and 1,
n = 32768 with k in {1, 4, 16, 64}, 512 factors with n in [64, 4096], a served
mix with n in [256, 8192] and k in [1, 32], both storage types.  Storage is the
C ABI's: an (n, ld) tensor whose row j is column j of the upper factor, V a
(k, n) tensor whose row p is vector p.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1011_1173_gb300 import chm

F64, F32 = "f64", "f32"
KEEP = 0.9  # a downdate removes this multiple of a block that was added before


def listed():
    return [
        # the smallest call in use: one vector, a factor that one SM's neighbours hold; latency and launches
        {"name": "pair_f64_n512_k1", "kind": "pair", "dtype": F64, "n": 512, "ld": 512, "k": 1},
        # an ordinary model-sized factor, ragged order and padded columns, a few vectors of both signs in one call
        {"name": "mixed_f32_n1001_k6", "kind": "mixed", "dtype": F32, "n": 1001, "ld": 1003, "k": 6},
        # the paper's headline shape: sixteen vectors into a factor of order 5000, and out again
        {"name": "pair_f64_n5000_k16", "kind": "pair", "dtype": F64, "n": 5000, "ld": 5000, "k": 16},
        # its rank-1 path
        {"name": "pair_f64_n5000_k1", "kind": "pair", "dtype": F64, "n": 5000, "ld": 5000, "k": 1},
        # the large single factor, the memory-bound end: one vector, float storage
        {"name": "pair_f32_n32768_k1", "kind": "pair", "dtype": F32, "n": 32768, "ld": 32768, "k": 1},
        # the large single factor with a block of vectors, float storage
        {"name": "mixed_f32_n32768_k16", "kind": "mixed", "dtype": F32, "n": 32768, "ld": 32768, "k": 16},
        # and in double: the largest call
        {"name": "update_f64_n32768_k16", "kind": "update", "dtype": F64, "n": 32768, "ld": 32768, "k": 16},
        # what a maintained factor is for: a block of right-hand sides against it
        {"name": "solve_f64_n5000_nrhs16", "kind": "solve", "dtype": F64, "n": 5000, "ld": 5000, "nrhs": 16},
        # one step of a recursive estimator: one vector in, one system solved
        {"name": "modify_solve_f64_n2000_k1", "kind": "modify_solve", "dtype": F64, "n": 2000, "ld": 2000, "k": 1, "nrhs": 1},
        # the batched workload: 512 independent factors of uneven order
        {"name": "batch_f64_512", "kind": "batch", "dtype": F64, "count": 512, "n_lo": 64, "n_hi": 4096, "sizes": 3},
        # the same kind of work in float storage with fewer, smaller factors
        {"name": "batch_f32_96", "kind": "batch", "dtype": F32, "count": 96, "n_lo": 64, "n_hi": 2048, "sizes": 5},
        # serving: a burst of requests on resident factors, popular ones more often
        {"name": "serve_f32_48", "kind": "serve", "dtype": F32, "count": 48, "n_lo": 256, "n_hi": 8192, "requests": 160, "sizes": 7},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["update", "pair", "pair", "mixed", "mixed", "solve", "modify_solve", "batch", "serve"])
    dtype = rng.choice([F64, F32])
    if kind == "batch":
        return {"kind": kind, "dtype": dtype, "count": _log_int(rng, 8, 400), "n_lo": 64,
                "n_hi": _log_int(rng, 256, 4096), "sizes": rng.randrange(1 << 20)}
    if kind == "serve":
        count = _log_int(rng, 8, 48)
        return {"kind": kind, "dtype": dtype, "count": count, "n_lo": 256, "n_hi": _log_int(rng, 1024, 6000),
                "requests": _log_int(rng, count, 160), "sizes": rng.randrange(1 << 20)}
    n = _log_int(rng, 64, 32768)
    pad = rng.choice([0, 0, 0, 1, 2, 5])
    if kind == "solve":
        nrhs = _log_int(rng, 1, 64)
        n = min(n, 32768 * 8 // nrhs)  # at most the largest listed case's time
        return {"kind": kind, "dtype": dtype, "n": n, "ld": n + pad, "nrhs": nrhs}
    k = _log_int(rng, 2 if kind == "mixed" else 1, 64)
    most = 16 * 32768 ** 2 * (0.45 if kind == "pair" else 0.9)  # of k n^2
    if k * n * n > most:
        n = int(math.sqrt(most / k))
    c = {"kind": kind, "dtype": dtype, "n": n, "ld": n + pad, "k": k}
    if kind == "modify_solve":
        c["nrhs"] = _log_int(rng, 1, 8)
    return c


def _dtype(case):
    return torch.float64 if case["dtype"] == F64 else torch.float32


def _gen(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _spd_factor(n, ld, dtype, g):
    """Factor of B^T B / n + I, B ~ N(0, 1)."""
    B = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")
    A = (B.T @ B).div_(n)
    A.diagonal().add_(1.0)
    out = torch.zeros((n, ld), dtype=dtype, device="cuda")
    out[:, :n].copy_(torch.linalg.cholesky(A))
    return out


def _random_factor(out, n, g):
    """A factor drawn as one: diagonal 1 + U[0, 1), N(0, 1/n) above it."""
    R = out[:, :n]
    R.copy_(torch.randn((n, n), generator=g, dtype=out.dtype, device="cuda").mul_(n ** -0.5).tril_(-1))
    R.diagonal().copy_(1.0 + torch.rand((n,), generator=g, dtype=out.dtype, device="cuda"))
    return out


def _factor(case, g):
    n, ld, dtype = case["n"], case["ld"], _dtype(case)
    if n <= 5000:
        return _spd_factor(n, ld, dtype, g)
    return _random_factor(torch.zeros((n, ld), dtype=dtype, device="cuda"), n, g)


def _block(k, n, dtype, g, scale=1.0):
    """Vectors of an update: N(0, scale^2 / n)."""
    return torch.randn((k, n), generator=g, dtype=dtype, device="cuda").mul_(scale * n ** -0.5)


def _single_inputs(case, seed):
    g = _gen(seed, "cuda")
    s = {"L": _factor(case, g)}
    n, k, dtype = case["n"], case.get("k", 0), _dtype(case)
    if case["kind"] == "mixed":
        up = (k + 1) // 2
        V = _block(up, n, dtype, g)
        s["V"] = torch.cat([V, V[:k - up] * KEEP]).contiguous()
        s["sigma"] = [1] * up + [-1] * (k - up)
    elif k:
        s["V"] = _block(k, n, dtype, g)
        if case["kind"] == "pair":
            s["W"] = s["V"] * KEEP
    if "nrhs" in case:
        s["B"] = torch.randn((case["nrhs"], n), generator=g, dtype=dtype, device="cuda")
    return s


def _orders(case):
    """Orders, vector counts and signs of a batch; they are the case's, not the seed's."""
    r = random.Random(case["sizes"])
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    ns = [int(math.exp(r.uniform(lo, hi))) for _ in range(case["count"])]
    ks = [r.choice([1, 4, 16]) for _ in ns]
    signs = [r.choice([1, -1]) for _ in ns]
    return ns, ks, signs


def _requests(case):
    """Orders of the resident factors and the (factor, k, sign) of each request: factors by
    Zipf(1.1), k uniform on [1, 32], 70 % updates; a downdate takes KEEP times the factor's
    latest update that has not left yet, and is an update where there is none."""
    r = random.Random(case["sizes"])
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    ns = [int(math.exp(r.uniform(lo, hi))) for _ in range(case["count"])]
    weight = [1.0 / (i + 1) ** 1.1 for i in range(len(ns))]
    r.shuffle(weight)
    added = [[] for _ in ns]
    asked = []
    for i in range(case["requests"]):
        f = r.choices(range(len(ns)), weight)[0]
        if r.random() < 0.3 and added[f]:
            j = added[f].pop()
            asked.append((f, asked[j][1], -1, j))
        else:
            added[f].append(i)
            asked.append((f, r.randint(1, 32), 1, None))
    return ns, asked


def _many_factors(ns, dtype, g):
    """Square factors in one allocation; returns it and a view per factor."""
    flat = torch.zeros(sum(n * n for n in ns), dtype=dtype, device="cuda")
    views, at = [], 0
    for n in ns:
        views.append(_random_factor(flat[at:at + n * n].view(n, n), n, g))
        at += n * n
    return flat, views


def _batch_inputs(case, seed):
    ns, ks, signs = _orders(case)
    dtype, g = _dtype(case), _gen(seed, "cuda")
    flat, Ls = _many_factors(ns, dtype, g)
    # a block that is taken out first is a small one, which every such factor can spare
    Vs = [_block(k, n, dtype, g, 1.0 if s > 0 else 0.3) for n, k, s in zip(ns, ks, signs)]
    Ws = [V * (KEEP if s > 0 else 1 / KEEP) for V, s in zip(Vs, signs)]
    return {"flat": flat, "Ls": Ls, "Vs": Vs, "Ws": Ws}


def _serve_inputs(case, seed):
    ns, asked = _requests(case)
    dtype, g = _dtype(case), _gen(seed, "cuda")
    flat, Ls = _many_factors(ns, dtype, g)
    Vs = []
    for f, k, sign, of in asked:
        Vs.append(_block(k, ns[f], dtype, g) if of is None else Vs[of] * KEEP)
    return flat, Ls, Vs


def prepare(case, seed):
    kind, dtype = case["kind"], _dtype(case)
    code = chm.CHM_F64 if case["dtype"] == F64 else chm.CHM_F32_MIXED
    if kind == "batch":
        ns, ks, signs = _orders(case)
        s = _batch_inputs(case, seed)
        s["there"] = chm.BatchPlan(ns, ns, ks, signs, code)
        s["back"] = chm.BatchPlan(ns, ns, ks, [-x for x in signs], code)
    elif kind == "serve":
        ns, asked = _requests(case)
        flat, Ls, Vs = _serve_inputs(case, seed)
        torch.cuda.synchronize()
        s = {"out": flat, "views": Ls, "server": chm.Server(24 << 30, code)}
        s["fids"] = [s["server"].add_factor(L) for L in Ls]
        s["asked"] = [(s["fids"][f], V.cpu().pin_memory(), sign) for (f, k, sign, of), V in zip(asked, Vs)]
    else:
        s = _single_inputs(case, seed)
        if "B" in s:
            s["X"] = torch.empty_like(s["B"])
    s["kind"] = kind
    return s


def run(s):
    kind = s["kind"]
    if kind == "pair":
        chm.check(chm.update(s["L"], s["V"]))
        chm.check(chm.downdate(s["L"], s["W"]))
        return s["L"]
    if kind == "update":
        chm.check(chm.update(s["L"], s["V"]))
        return s["L"]
    if kind == "mixed":
        chm.check(chm.modify(s["L"], s["V"], s["sigma"]))
        return s["L"]
    if kind == "solve":
        s["X"].copy_(s["B"])
        chm.check(chm.solve(s["L"], s["X"]))
        return s["X"]
    if kind == "modify_solve":
        s["X"].copy_(s["B"])
        chm.check(chm.modify_solve(s["L"], s["V"], s["X"]))
        return {"L": s["L"], "X": s["X"]}
    if kind == "batch":
        chm.check(s["there"].execute(s["Ls"], s["Vs"]))
        chm.check(s["back"].execute(s["Ls"], s["Ws"]))
        return s["flat"]
    server = s["server"]
    for fid, V, sign in s["asked"]:
        server.submit(fid, V, sign)
    chm.check(server.drain())
    for _, status, _ in server.poll():
        chm.check(status)
    for fid, view in zip(s["fids"], s["views"]):
        chm.check(server.get_factor(fid, view))
    return s["out"]


def _modify_work(n, k, elt):
    """One modification: the triangle read and written and V read; the rotations' four flops per
    element and vector, and Compute."""
    return elt * (n * (n + 1) + n * k), k * (2 * n * (n - 1) + 6 * n)


def work(case):
    elt = 8 if case["dtype"] == F64 else 4
    kind = case["kind"]
    if kind == "batch":
        ns, ks, _ = _orders(case)
        parts = [_modify_work(n, k, elt) for n, k in zip(ns, ks)] * 2
    elif kind == "serve":
        ns, asked = _requests(case)
        parts = [_modify_work(ns[f], k, elt) for f, k, _, _ in asked] + [(2 * elt * n * n, 0) for n in ns]
    elif kind == "solve":
        n, nrhs = case["n"], case["nrhs"]
        parts = [(elt * (n * (n + 1) // 2 + 2 * n * nrhs), 2 * n * n * nrhs)]
    else:
        n, k = case["n"], case["k"]
        parts = [_modify_work(n, k, elt)] * (2 if kind == "pair" else 1)
        if kind == "modify_solve":
            parts.append((2 * elt * n * case["nrhs"], 2 * n * n * case["nrhs"]))
    return {"bytes": float(sum(b for b, _ in parts)), "flops": float(sum(f for _, f in parts))}


def _exact_modify(L, n, V, sigma, step=256):
    """The lower factor of L L^T + V^T diag(sigma) V over L's leading n columns, in place, by
    blocks: with Z = V^T less what the finished columns explain and H = Sigma + P^T P of the
    finished rows P of L^{-1} V^T, the rest of the matrix is that of L plus Z H^{-1} Z^T."""
    Z = V.T.contiguous()
    H = torch.diag(torch.tensor([float(x) for x in sigma], dtype=L.dtype, device=L.device))
    for a in range(0, n, step):
        b = min(n, a + step)
        D, R = L[a:b, a:b].clone(), L[b:n, a:b].clone()
        MZ = torch.linalg.solve(H, Z[a:b].T)
        new = torch.linalg.cholesky(D @ D.T + Z[a:b] @ MZ)
        P = torch.linalg.solve_triangular(D, Z[a:b], upper=False)
        L[a:b, a:b] = new
        if b < n:
            L[b:n, a:b] = torch.linalg.solve_triangular(new, (R @ D.T + Z[b:] @ MZ).T, upper=False).T
            Z[b:] -= R @ P
        H += P.T @ P
    return L


def _exact_solve(L, n, B):
    Y = torch.linalg.solve_triangular(L[:, :n], B.T, upper=False)
    return torch.linalg.solve_triangular(L[:, :n].T, Y, upper=True).T.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        s = _batch_inputs(case, seed)
        _, ks, signs = _orders(case)
        flat, at = s["flat"].double(), 0
        for L, V, W, k, sign in zip(s["Ls"], s["Vs"], s["Ws"], ks, signs):
            n = L.shape[0]
            _exact_modify(flat[at:at + n * n].view(n, n), n, torch.cat([V, W]).double(), [sign] * k + [-sign] * k)
            at += n * n
        return flat
    if kind == "serve":
        ns, asked = _requests(case)
        flat, Ls, Vs = _serve_inputs(case, seed)
        flat, at = flat.double(), 0
        for f, n in enumerate(ns):
            mine = [(V, sign) for (g, _, sign, _), V in zip(asked, Vs) if g == f]
            if mine:
                V = torch.cat([V for V, _ in mine]).double()
                _exact_modify(flat[at:at + n * n].view(n, n), n, V, [s for V, s in mine for _ in range(V.shape[0])])
            at += n * n
        return flat
    s = _single_inputs(case, seed)
    n = case["n"]
    L = s["L"].double()
    if kind == "solve":
        return _exact_solve(L, n, s["B"].double())
    V, sigma = s["V"].double(), s.get("sigma", [1] * case["k"])
    if kind == "pair":
        V, sigma = torch.cat([V, s["W"].double()]), [1] * case["k"] + [-1] * case["k"]
    _exact_modify(L, n, V, sigma)
    if kind == "modify_solve":
        return {"L": L, "X": _exact_solve(L, n, s["B"].double())}
    return L
