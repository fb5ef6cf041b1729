"""The work that users of tile_chol have it do, as cases that can be timed and compared.

A Gaussian-process / geostatistics program generates a Matern covariance matrix, optionally maps
its tiles to precisions, factors it, solves with the factor and evaluates the log-likelihood; it
does so for one small problem many times (an optimiser over theta), for one large problem, for
many problems of uneven size at once, or for a matrix held in host memory.  Every case goes
through the public entry points of ``tile_chol`` with seeded synthetic points.

A case is a dict with a ``kind`` (see ``_KINDS``) and plain sizes and options.  Matrices that a
case takes as input are evaluated with torch, so that the input does not depend on the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_09819_gb300 import tile_chol as tc

_DEV = "cuda:0"
_F64 = torch.float64


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # smallest whole call: one theta of an optimiser's loop on a small ragged problem
        {"name": "likelihood_n700", "kind": "likelihood", "n": 700, "tile": 128, "mode": 2, "nu": 0.5,
         "range": 0.1, "refine": 2},
        # the library's default engine (FP64 pipe) on the small plain-FP64 workload
        {"name": "factor_dfma_n2048", "kind": "factor", "n": 2048, "tile": 256, "mode": 0, "nu": 0.5, "range": 0.1},
        # an ordinary order that is no multiple of its tile, FP64 on the tensor cores
        {"name": "factor_fp64_n10000", "kind": "factor", "n": 10000, "tile": 512, "mode": 2, "nu": 0.5, "range": 0.05},
        # the FP64 workload's tile and theta at half its order: the largest FP64 factorization here
        {"name": "factor_fp64_n32768", "kind": "factor", "n": 32768, "tile": 1024, "mode": 2, "nu": 0.5,
         "range": 0.05},
        # the four-precision workload's tile, theta and accuracy level at a quarter of its order
        {"name": "factor_mixed_n32768", "kind": "mixed", "n": 32768, "tile": 2048, "mode": 2, "nu": 1.5,
         "range": 0.03, "eps": 1e-9, "band": 2, "precs": 4},
        # refined single right-hand side and Eq. 1: what follows every large factorization
        {"name": "solve_refined_n32768", "kind": "solve", "n": 32768, "tile": 1024, "mode": 2, "nu": 0.5,
         "range": 0.05, "nrhs": 1, "refine": 2},
        # kriging weights of many prediction sites: a block of right-hand sides
        {"name": "solve_rhs64_n8192", "kind": "solve", "n": 8192, "tile": 512, "mode": 2, "nu": 0.5,
         "range": 0.05, "nrhs": 64, "refine": 1},
        # the covariance of a large problem (nu = 3/2), once per theta
        {"name": "generate_n32768", "kind": "generate", "n": 32768, "tile": 1024, "nu": 1.5, "range": 0.03},
        # a smoothness that has no closed form (an optimiser over nu)
        {"name": "generate_anynu_n4500", "kind": "generate", "n": 4500, "tile": 512, "nu": 0.8, "range": 0.07},
        # the precision map of a matrix that is on the device already
        {"name": "map_n32768", "kind": "map", "n": 32768, "tile": 2048, "nu": 1.5, "range": 0.03, "eps": 1e-9,
         "band": 2, "precs": 4},
        # many uneven problems at once: maps, factorizations, refined 16-column solves, likelihoods
        {"name": "batched_96", "kind": "batched", "count": 96, "lo": 64, "hi": 4096, "tile": 128, "mode": 2,
         "nrhs": 16, "eps": 1e-7},
        # a matrix in page-locked host memory with a device cache of 0.44 of it, and one solve
        {"name": "ooc_n16384", "kind": "ooc", "n": 16384, "tile": 1024, "mode": 2, "nu": 0.5, "range": 0.02,
         "cap": 0.44},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _theta(rng):
    return rng.choice([0.5, 1.5, 2.5]), round(rng.uniform(0.02, 0.1), 4)


def _tile(rng, n, tiles, most=64):
    """A tile size that leaves at least two and at most `most` tile rows."""
    fit = [b for b in tiles if 2 * b <= n <= most * b]
    return rng.choice(fit) if fit else tiles[0]


def draw(rng):
    kind = rng.choice(["likelihood", "factor", "factor", "mixed", "solve", "solve", "generate", "map", "batched", "ooc"])
    nu, rg = _theta(rng)
    if kind == "likelihood":
        mode = rng.choice([0, 2])
        n = _log_int(rng, 64, 4096)
        b = _tile(rng, n, [128, 256, 512] if mode else [64, 128, 256])
        return {"kind": kind, "n": n, "tile": b, "mode": mode, "nu": nu, "range": rg, "refine": rng.choice([1, 2])}
    if kind == "factor":
        mode = rng.choice([0, 1, 2, 2])
        n = _log_int(rng, 300, 10000 if mode == 0 else 30000)
        b = _tile(rng, n, [128, 256, 512, 1024, 2048])
        return {"kind": kind, "n": n, "tile": b, "mode": mode, "nu": nu, "range": rg}
    if kind == "mixed":
        n = _log_int(rng, 2000, 30000)
        b = _tile(rng, n, [256, 512, 1024, 2048])
        return {"kind": kind, "n": n, "tile": b, "mode": rng.choice([1, 2]), "nu": nu, "range": rg,
                "eps": 10.0 ** -rng.randint(7, 10), "band": rng.choice([0, 1, 2]), "precs": rng.choice([2, 3, 4])}
    if kind == "solve":
        n = _log_int(rng, 500, 30000)
        b = _tile(rng, n, [128, 256, 512, 1024, 2048])
        most = max(1, min(64, int(16 * (32768 / n) ** 2)))
        return {"kind": kind, "n": n, "tile": b, "mode": 2, "nu": nu, "range": rg,
                "nrhs": rng.choice([1, _log_int(rng, 1, most)]), "refine": rng.choice([0, 1, 2])}
    if kind == "generate":
        general = rng.random() < 0.4
        n = _log_int(rng, 500, 5000 if general else 32000)
        b = _tile(rng, n, [128, 256, 512, 1024, 2048])
        return {"kind": kind, "n": n, "tile": b, "nu": round(rng.uniform(0.3, 3.0), 3) if general else nu, "range": rg}
    if kind == "map":
        n = _log_int(rng, 1000, 32000)
        b = _tile(rng, n, [128, 256, 512, 1024, 2048])
        return {"kind": kind, "n": n, "tile": b, "nu": nu, "range": rg, "eps": 10.0 ** -rng.randint(6, 10),
                "band": rng.choice([0, 1, 2]), "precs": rng.choice([2, 3, 4])}
    if kind == "batched":
        return {"kind": kind, "count": _log_int(rng, 4, 96), "lo": 64, "hi": _log_int(rng, 512, 4096),
                "tile": rng.choice([128, 256]), "mode": rng.choice([0, 2, 2]), "nrhs": rng.choice([1, 4, 16]),
                "eps": 10.0 ** -rng.randint(6, 8)}
    n = _log_int(rng, 4096, 16384)
    b = 512 if n < 8192 else 1024
    return {"kind": kind, "n": n, "tile": b, "mode": rng.choice([1, 2]), "nu": nu, "range": rg,
            "cap": round(rng.uniform(0.44, 0.8), 3)}


# ------------------------------------------------------------------------------- the inputs
_NUGGET = 1e-4


def _points(n, seed):
    """n uniform points of the unit square along a Z-order curve (16 bits per axis)."""
    p = np.random.Generator(np.random.PCG64(seed)).random((n, 2))
    q = np.minimum(np.floor(p * 65536.0), 65535).astype(np.uint64)
    key = np.zeros(n, dtype=np.uint64)
    for bit in range(16):
        one, at = np.uint64(1), np.uint64(bit)
        key |= ((q[:, 0] >> at) & one) << np.uint64(2 * bit)
        key |= ((q[:, 1] >> at) & one) << np.uint64(2 * bit + 1)
    return torch.from_numpy(np.ascontiguousarray(p[np.argsort(key, kind="stable")])).to(_DEV)


def _correlation(x, nu):
    """Matern correlation at x = distance / range in 64 bits."""
    if nu == 0.5:
        return torch.exp(-x)
    if nu == 1.5:
        return (1.0 + x) * torch.exp(-x)
    if nu == 2.5:
        return (1.0 + x + x * x / 3.0) * torch.exp(-x)
    # K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt: the trapezoid rule with step 1/8 is exact
    # to rounding for this analytic, doubly exponentially falling integrand
    xs = torch.clamp(x, min=1e-12)
    acc = 0.5 * torch.exp(-xs)
    for k in range(1, 300):
        t = k / 8.0
        acc += torch.exp(math.log(math.cosh(nu * t)) - xs * math.cosh(t))
    val = torch.exp(nu * torch.log(xs)) * acc / 8.0 * (2.0 ** (1.0 - nu) / math.gamma(nu))
    return torch.where(x > 0, val, torch.ones_like(val))


def _cov(rows, cols, nu, rg):
    d = rows[:, None, :] - cols[None, :, :]
    return _correlation(torch.sqrt(d[..., 0] ** 2 + d[..., 1] ** 2) / rg, nu)


def _tiles(pts, b, nu, rg):
    """The packed lower tiles of the covariance (column-major tiles, identity padding)."""
    n = pts.shape[0]
    nt = -(-n // b)
    out = torch.zeros(nt * (nt + 1) // 2 * b * b, dtype=_F64, device=_DEV)
    for i in range(nt):
        nv = min(n, (i + 1) * b) - i * b
        at = i * (i + 1) // 2 * b * b
        block = out[at:at + (i + 1) * b * b].view((i + 1) * b, b)     # [column, row]
        for c in range(0, i * b + nv, 4096):
            e = min(c + 4096, i * b + nv)
            block[c:e, :nv] = _cov(pts[c:e], pts[i * b:i * b + nv], nu, rg)
        diag = torch.arange(b, device=_DEV)
        block[i * b + diag[:nv], diag[:nv]] += _NUGGET
        block[i * b + diag[nv:], diag[nv:]] = 1.0
    return out


def _dense(pts, nu, rg):
    n = pts.shape[0]
    A = torch.empty(n, n, dtype=_F64, device=_DEV)
    for c in range(0, n, 2048):
        A[c:c + 2048] = _cov(pts[c:c + 2048], pts, nu, rg)
    A.diagonal().add_(_NUGGET)
    return A


def _pack_factor(L, b):
    """Dense lower factor into packed tiles, zeros above the diagonal and in the padding."""
    n = L.shape[0]
    nt = -(-n // b)
    out = torch.zeros(nt * (nt + 1) // 2 * b * b, dtype=_F64, device=_DEV)
    for i in range(nt):
        nv = min(n, (i + 1) * b) - i * b
        at = i * (i + 1) // 2 * b * b
        block = out[at:at + (i + 1) * b * b].view((i + 1) * b, b)
        block[:i * b + nv, :nv] = L[i * b:i * b + nv, :i * b + nv].T
    return out


def _rhs(n, nrhs, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(nrhs, n, dtype=_F64, generator=g).to(_DEV)     # column-major n x nrhs


def _handle(case, **more):
    return tc.Handle(0, fp64_mode=case["mode"], **more)


def _batch(case):
    """Orders (log-uniform) and thetas of a batch; its points and right-hand sides come from the seed."""
    rng = np.random.Generator(np.random.PCG64(case["count"]))
    ns = [int(round(case["lo"] * (case["hi"] / case["lo"]) ** u)) for u in rng.random(case["count"])]
    ranges = [float(v) for v in rng.uniform(0.02, 0.2, case["count"])]
    nus = [float(v) for v in rng.choice([0.5, 1.5, 2.5], case["count"])]
    return ns, ranges, nus


# ------------------------------------------------------------------------------- likelihood
def _prepare_likelihood(c, seed):
    n, b = c["n"], c["tile"]
    return {"H": _handle(c), "pts": _points(n, seed), "y": _rhs(n, 1, seed)[0], "x": torch.empty(n, dtype=_F64, device=_DEV),
            "A": torch.empty(tc.tile_count(n, b) * b * b, dtype=_F64, device=_DEV)}


def _run_likelihood(s):
    c, h, n = s["case"], s["H"].h, s["case"]["n"]
    tc.tc_matern_tiles(h, n, c["tile"], s["pts"], 1.0, c["range"], c["nu"], _NUGGET, s["A"])
    tc.tile_chol_factor(h, n, c["tile"], s["A"])
    tc.tile_chol_solve(h, 1, s["y"], n, s["x"], n, c["refine"], 1e-14)
    return [s["A"], s["x"], tc.tile_chol_loglik_solved(h, s["y"], s["x"]), tc.tile_chol_logdet(h)]


def _exact_likelihood(c, seed):
    pts, y = _points(c["n"], seed), _rhs(c["n"], 1, seed)[0]
    L = torch.linalg.cholesky(_dense(pts, c["nu"], c["range"]))
    x = torch.cholesky_solve(y[:, None], L)[:, 0]
    logdet = 2.0 * float(L.diagonal().log().sum())
    ll = -0.5 * c["n"] * math.log(2.0 * math.pi) - 0.5 * logdet - 0.5 * float(y @ x)
    return [_tiles(pts, c["tile"], c["nu"], c["range"]), x, ll, logdet]


# ------------------------------------------------------------------------------- factor
def _prepare_factor(c, seed):
    A = _tiles(_points(c["n"], seed), c["tile"], c["nu"], c["range"])
    return {"H": _handle(c), "A": A, "L": torch.empty_like(A)}


def _run_factor(s):
    c, h = s["case"], s["H"].h
    tc.tile_chol_factor(h, c["n"], c["tile"], s["A"])
    tc.tile_chol_get_factor(h, s["L"])
    return [s["L"], tc.tile_chol_logdet(h)]


def _exact_factor(c, seed):
    L = torch.linalg.cholesky(_dense(_points(c["n"], seed), c["nu"], c["range"]))
    return [_pack_factor(L, c["tile"]), 2.0 * float(L.diagonal().log().sum())]


# ------------------------------------------------------------------------------- mixed
def _prepare_mixed(c, seed):
    s = _prepare_factor(c, seed)
    s["map"] = np.zeros(tc.ntiles(c["n"], c["tile"]) ** 2, dtype=np.uint8)
    return s


def _run_mixed(s):
    c, h = s["case"], s["H"].h
    tc.tile_chol_factor_mapped(h, c["n"], c["tile"], s["A"], c["eps"], c["band"], c["precs"], s["map"])
    tc.tile_chol_get_factor(h, s["L"])
    return [s["L"], tc.tile_chol_logdet(h), s["map"]]


def _exact_mixed(c, seed):
    return _exact_factor(c, seed) + [None]


# ------------------------------------------------------------------------------- solve
def _prepare_solve(c, seed):
    n, b = c["n"], c["tile"]
    A = _tiles(_points(n, seed), b, c["nu"], c["range"])
    B = _rhs(n, c["nrhs"], seed)
    H = _handle(c)
    torch.cuda.synchronize()
    tc.tile_chol_factor(H.h, n, b, A)
    return {"H": H, "A": A, "B": B, "X": torch.empty_like(B)}


def _run_solve(s):
    c, h, n = s["case"], s["H"].h, s["case"]["n"]
    tc.tile_chol_solve(h, c["nrhs"], s["B"], n, s["X"], n, c["refine"], 1e-15)
    if c["nrhs"] > 1:
        return [s["X"]]
    return [s["X"], tc.tile_chol_loglik_solved(h, s["B"], s["X"])]


def _exact_solve(c, seed):
    n = c["n"]
    L = torch.linalg.cholesky(_dense(_points(n, seed), c["nu"], c["range"]))
    B = _rhs(n, c["nrhs"], seed)
    X = torch.cholesky_solve(B.T.contiguous(), L).T.contiguous()
    if c["nrhs"] > 1:
        return [X]
    logdet = 2.0 * float(L.diagonal().log().sum())
    return [X, -0.5 * n * math.log(2.0 * math.pi) - 0.5 * logdet - 0.5 * float(B[0] @ X[0])]


# ------------------------------------------------------------------------------- generate
def _prepare_generate(c, seed):
    n, b = c["n"], c["tile"]
    return {"H": tc.Handle(0), "pts": _points(n, seed),
            "A": torch.empty(tc.tile_count(n, b) * b * b, dtype=_F64, device=_DEV)}


def _run_generate(s):
    c = s["case"]
    tc.tc_matern_tiles(s["H"].h, c["n"], c["tile"], s["pts"], 1.0, c["range"], c["nu"], _NUGGET, s["A"])
    return s["A"]


def _exact_generate(c, seed):
    return _tiles(_points(c["n"], seed), c["tile"], c["nu"], c["range"])


# ------------------------------------------------------------------------------- map
def _prepare_map(c, seed):
    nt = tc.ntiles(c["n"], c["tile"])
    return {"H": tc.Handle(0), "A": _tiles(_points(c["n"], seed), c["tile"], c["nu"], c["range"]),
            "map": np.zeros(nt * nt, dtype=np.uint8), "norms": np.zeros(nt * nt + 1)}


def _run_map(s):
    c = s["case"]
    tc.tile_chol_precision_map(s["H"].h, c["n"], c["tile"], s["A"], c["eps"], c["band"], c["precs"], s["map"], s["norms"])
    return [s["map"], s["norms"]]


def _exact_map(c, seed):
    n, b = c["n"], c["tile"]
    nt = tc.ntiles(n, b)
    A = _dense(_points(n, seed), c["nu"], c["range"])
    norms = torch.zeros(nt * nt + 1, dtype=_F64)
    for i in range(nt):
        for j in range(i + 1):
            norms[i * nt + j] = float(torch.linalg.vector_norm(A[i * b:(i + 1) * b, j * b:(j + 1) * b]))
    norms[nt * nt] = float(torch.linalg.vector_norm(A))
    return [None, norms.numpy()]


# ------------------------------------------------------------------------------- batched
def _prepare_batched(c, seed):
    ns, ranges, nus = _batch(c)
    b, nrhs = c["tile"], c["nrhs"]
    sizes = [tc.ntiles(n, b) ** 2 for n in ns]
    flat = torch.zeros(sum(sizes), dtype=torch.uint8, device=_DEV)
    A = [_tiles(_points(n, seed + 1 + i), b, nus[i], ranges[i]) for i, n in enumerate(ns)]
    B = [_rhs(n, nrhs, seed + 1 + i) for i, n in enumerate(ns)]
    Xflat = torch.empty(nrhs * sum(ns), dtype=_F64, device=_DEV)
    X = [x.view(nrhs, n) for x, n in zip(torch.split(Xflat, [nrhs * n for n in ns]), ns)]
    return {"H": _handle(c), "ns": ns, "flat": flat, "maps": list(torch.split(flat, sizes)), "A": A, "B": B,
            "Y": [x[0].contiguous() for x in B], "X": X, "Xflat": Xflat}


def _run_batched(s):
    c, h, b = s["case"], s["H"].h, s["case"]["tile"]
    for n, A, m in zip(s["ns"], s["A"], s["maps"]):
        tc.tile_chol_precision_map_noalloc(n, b, A, c["eps"], 0, 4, m)
    s["flat"][s["flat"] == tc.TC_FP32] = tc.TC_FP64       # FP64 diagonal, FP16 / FP8 off it, else FP64
    _, _, logdets = tc.tile_chol_factor_batched(h, s["ns"], b, s["A"], s["maps"])
    tc.tile_chol_solve_batched(h, c["nrhs"], s["B"], s["X"], 10, 1e-13)
    ll = tc.tile_chol_loglik_batched(h, s["Y"])
    return [s["Xflat"], np.array(logdets), np.array(ll), s["flat"]]


def _exact_batched(c, seed):
    ns, ranges, nus = _batch(c)
    X, logdets, ll = [], [], []
    for i, n in enumerate(ns):
        L = torch.linalg.cholesky(_dense(_points(n, seed + 1 + i), nus[i], ranges[i]))
        B = _rhs(n, c["nrhs"], seed + 1 + i)
        x = torch.cholesky_solve(B.T.contiguous(), L).T.contiguous()
        X.append(x.reshape(-1))
        logdets.append(2.0 * float(L.diagonal().log().sum()))
        ll.append(-0.5 * n * math.log(2.0 * math.pi) - 0.5 * logdets[-1] - 0.5 * float(B[0] @ x[0]))
    return [torch.cat(X), np.array(logdets), np.array(ll), None]


# ------------------------------------------------------------------------------- out of core
def _prepare_ooc(c, seed):
    n, b = c["n"], c["tile"]
    A = _tiles(_points(n, seed), b, c["nu"], c["range"])
    host = torch.empty(A.shape, dtype=_F64, pin_memory=True)
    y = _rhs(n, 1, seed)[0].cpu().pin_memory()
    return {"H": _handle(c, device_cap_bytes=int(c["cap"] * A.numel() * 8)), "A": A, "host": host, "y": y,
            "x": torch.empty_like(y).pin_memory()}


def _run_ooc(s):
    c, h, n = s["case"], s["H"].h, s["case"]["n"]
    s["host"].copy_(s["A"])                               # the factorization overwrites its matrix
    tc.tile_chol_factor_ooc(h, n, c["tile"], s["host"])
    tc.tile_chol_solve(h, 1, s["y"], n, s["x"], n)
    return [s["host"], s["x"], tc.tile_chol_logdet(h)]


def _exact_ooc(c, seed):
    n = c["n"]
    L = torch.linalg.cholesky(_dense(_points(n, seed), c["nu"], c["range"]))
    x = torch.cholesky_solve(_rhs(n, 1, seed)[0][:, None], L)[:, 0]
    return [None, x, 2.0 * float(L.diagonal().log().sum())]  # what lies above the diagonal is not specified


# ------------------------------------------------------------------------------- work
def _matrix_bytes(n):
    return 4.0 * n * (n + 1)                               # the lower triangle, 8 bytes an element


def _work(c):
    kind = c["kind"]
    if kind == "batched":
        ns, _, _ = _batch(c)
        return {"bytes": sum(2 * _matrix_bytes(n) + 16.0 * n * c["nrhs"] for n in ns),
                "flops": sum(n ** 3 / 3.0 + 4.0 * n * n * c["nrhs"] for n in ns)}
    n = c["n"]
    A, elements = _matrix_bytes(n), n * (n + 1) / 2.0
    if kind == "likelihood":
        return {"bytes": 2 * A + 32.0 * n, "flops": n ** 3 / 3.0 + 4.0 * n * n + 10 * elements}
    if kind in ("factor", "mixed", "ooc"):
        return {"bytes": 2 * A, "flops": n ** 3 / 3.0 + (2.0 * n * n if kind == "ooc" else 0.0)}
    if kind == "solve":                                    # two sweeps; refined: a residual too
        refined = 1 if c["refine"] else 0
        return {"bytes": (1 + refined) * A + 16.0 * n * c["nrhs"], "flops": (2 + 2 * refined) * float(n) * n * c["nrhs"]}
    if kind == "generate":
        return {"bytes": A + 16.0 * n, "flops": (10 if c["nu"] in (0.5, 1.5, 2.5) else 100) * elements}
    return {"bytes": A, "flops": 2 * elements}             # map


# ------------------------------------------------------------------------------- entry points
_KINDS = {
    "likelihood": (_prepare_likelihood, _run_likelihood, _exact_likelihood),
    "factor": (_prepare_factor, _run_factor, _exact_factor),
    "mixed": (_prepare_mixed, _run_mixed, _exact_mixed),
    "solve": (_prepare_solve, _run_solve, _exact_solve),
    "generate": (_prepare_generate, _run_generate, _exact_generate),
    "map": (_prepare_map, _run_map, _exact_map),
    "batched": (_prepare_batched, _run_batched, _exact_batched),
    "ooc": (_prepare_ooc, _run_ooc, _exact_ooc),
}


def prepare(case, seed):
    state = _KINDS[case["kind"]][0](case, seed)
    state["case"] = case
    torch.cuda.synchronize()                               # the handle works on a stream of its own
    return state


def run(state):
    return _KINDS[state["case"]["kind"]][1](state)


def exact(case, seed):
    return _KINDS[case["kind"]][2](case, seed)


def work(case):
    return _work(case)
