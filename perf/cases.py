"""Performance cases of the library: what its users have it do, through its public entry points.

Four kinds of work:

* ``prob``: one probability on a resident factor (``tlrmvn_prob`` with host arrays,
  ``tlrmvn_prob_device`` with device arrays), in each precision, for normal and
  Student-t problems, one- and two-sided limits, from 256 to 65,536 variables;
* ``batch``: many small problems of uneven size replayed through one plan
  (``BatchPlan.run``), as a likelihood optimiser does;
* ``server``: a burst of requests on resident factors (``Server``);
* ``factor``: the tile-low-rank Cholesky factor of a covariance kernel on 2-D
  locations (``tlrmvn_factor_kernel``), kept as its exported checkpoint.

The probabilities run on factors loaded with ``tlrmvn_factor_import``, the library's
checkpoint format, whose arrays are drawn here from the seed, so that the same numbers
can be worked out in 64 bits without the library.  Their shape is that of the spatial
factors the library builds: dense lower-triangular diagonal tiles (the Cholesky factor
of an exponential kernel on a patch of a jittered grid, shrunk by what the earlier
tiles explain) and off-diagonal ranks that fall with the distance of two tiles, from
``near`` for neighbours (44 to 64 measured on the library's own factors, by tolerance
and rank cap) to ``far`` (1 to 3).  Such a factor belongs to a covariance L L^T like any other.

Numbers of the float64 and float32 paths are handed on in the type that they were
computed in; those of the paths with 16-bit products in 16 bits, together in one array.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2003_11183_gb300 as tl

PRECISION = {"fp64": tl.FP64, "fp32": tl.FP32, "bf16": tl.BF16_SHIFT, "fp16": tl.FP16_SHIFT}
RESULT = {"fp64": np.float64, "fp32": np.float32, "bf16": np.float16, "fp16": np.float16}
MASK64 = (1 << 64) - 1
EXACT_VARIABLES = 30000  # variables that the 64-bit reference walks in about 15 seconds
FLOPS_SPECIAL = 60  # flops of one Phi, one Phi^-1 and one log by their shortest polynomials


# ---- the cases ---------------------------------------------------------------------------------

def _prob(name, call, precision, n, m, shifts, points, limits="uniform", nu=math.inf, near=46, far=2, beta=0.1,
          periodize=True, own_shifts=False):
    return {"name": name, "kind": "prob", "call": call, "precision": precision, "n": n, "m": m, "shifts": shifts,
            "points": points, "limits": limits, "nu": nu, "near": near, "far": far, "beta": beta,
            "periodize": periodize, "own_shifts": own_shifts}


def listed():
    return [
        # the smallest problem users check their set-up with: 256 sites, float64, host arrays
        _prob("prob_n256_fp64_host", "host", "fp64", 256, 64, 20, 500),
        # a served request on a small resident factor in the default precision: launches and latency
        _prob("prob_n1024_fp32_host", "host", "fp32", 1024, 128, 10, 1000),
        # a served Student-t request (the degrees of freedom of the paper's wind data)
        _prob("prob_n4096_t7_fp32_host", "host", "fp32", 4096, 256, 10, 1000, nu=7.0),
        # the largest served request on the tensor-core path: few samples, many variables
        _prob("prob_n16384_bf16_host", "host", "bf16", 16384, 256, 10, 1000),
        # intervals (two-sided limits), a ragged site count and sample count, the plain lattice, fp16 products
        _prob("prob_n3900_t3_two_sided_fp16", "device", "fp16", 3900, 512, 8, 1301, limits="two_sided", nu=3.0, near=64,
              far=1, periodize=False),
        # an accurate estimate at 16,384 sites in the default precision
        _prob("prob_n16384_fp32", "device", "fp32", 16384, 256, 20, 5000, near=46, far=3, beta=0.3),
        # the headline problem: 65,536 sites, Student-t, the caller's own shifts (as replicas pass them)
        _prob("prob_n65536_t7_bf16", "device", "bf16", 65536, 512, 20, 5000, limits="normal", nu=7.0, near=64, far=1,
              own_shifts=True),
        # the convergence study's float64 runs: high limits, tiles of sqrt(n)
        _prob("prob_n4096_study_fp64", "device", "fp64", 4096, 64, 20, 1000, limits="high", near=40, far=2, beta=0.3),
        # 64 problems of uneven size with new limits, the optimiser's inner step in the default precision
        {"name": "batch_64_fp32", "kind": "batch", "precision": "fp32", "count": 64, "n_min": 256, "n_max": 4096,
         "m": 128, "shifts": 10, "points": 2000, "near": 46, "far": 2, "beta": 0.15, "t_share": 0.25},
        # 20 requests that arrive at once on four resident factors, normal and Student-t, float32 and bf16
        {"name": "server_burst_20", "kind": "server", "requests": 20, "lanes": 4, "n0": 512, "n1": 1024, "n2": 2048,
         "n3": 4096, "m": 128, "shifts": 10, "points": 1000, "near": 46, "far": 2, "beta": 0.1},
        # the covariance of one likelihood evaluation: a small factor, reordered iteratively
        {"name": "factor_n1024_iterative", "kind": "factor", "n": 1024, "m": 128, "kernel": "exp", "beta": 0.1,
         "ell": 0.1, "tol": 1e-5, "max_rank": 0, "reorder": 2, "schur": 0},
        # a factor made to be served: block reordering
        {"name": "factor_n4096_block", "kind": "factor", "n": 4096, "m": 256, "kernel": "matern", "beta": 0.1,
         "ell": 0.1, "tol": 1e-5, "max_rank": 0, "reorder": 1, "schur": 0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["prob", "batch", "server", "factor"], [10, 3, 1, 3])[0]
    beta = round(math.exp(rng.uniform(math.log(0.05), math.log(0.3))), 3)
    if kind == "prob":
        precision = rng.choice(["fp64", "fp32", "fp32", "bf16", "bf16", "fp16"])
        n_max, work_max = {"fp64": (8192, 8e7), "fp32": (32768, 1.6e9), "bf16": (65536, 6.5e9),
                           "fp16": (65536, 6.5e9)}[precision]
        n = _log_int(rng, 256, n_max)
        m = min(n, rng.choice([64, 128, 256, 512, _log_int(rng, 48, 512)]))
        m = max(m, n // 128)
        shifts = rng.choice([4, 8, 10, 20])
        points = _log_int(rng, 100, 5000)
        points = max(16, min(points, int(work_max / n / shifts)))
        return {"kind": "prob", "call": rng.choice(["host", "device"]), "precision": precision, "n": n, "m": m,
                "shifts": shifts, "points": points, "limits": rng.choice(["uniform", "uniform", "normal", "high",
                                                                          "two_sided"]),
                "nu": rng.choice([math.inf, math.inf, 3.0, 7.0, round(rng.uniform(2.5, 30.0), 2)]),
                "near": rng.randint(20, 64), "far": rng.randint(1, 3), "beta": beta,
                "periodize": rng.random() < 0.85, "own_shifts": rng.random() < 0.3}
    if kind == "batch":
        n_max = _log_int(rng, 700, 4096)
        return {"kind": "batch", "precision": rng.choice(["fp32", "bf16"]), "count": _log_int(rng, 6, 64),
                "n_min": _log_int(rng, 100, 400), "n_max": n_max, "m": rng.choice([64, 100, 128]),
                "shifts": 10, "points": _log_int(rng, 150, 2000), "near": rng.randint(20, 48),
                "far": rng.randint(1, 3), "beta": beta, "t_share": rng.choice([0.0, 0.25, 1.0])}
    if kind == "server":
        return {"kind": "server", "requests": rng.randint(8, 24), "lanes": rng.choice([2, 4, 6]),
                "n0": _log_int(rng, 300, 8192), "n1": _log_int(rng, 300, 8192), "n2": _log_int(rng, 300, 8192),
                "n3": _log_int(rng, 300, 8192), "m": rng.choice([128, 256]), "shifts": 10,
                "points": _log_int(rng, 200, 1500), "near": rng.randint(20, 48), "far": rng.randint(1, 3), "beta": beta}
    n = _log_int(rng, 300, 4096)
    return {"kind": "factor", "n": n, "m": min(n, rng.choice([64, 128, 256, max(32, int(math.sqrt(n)))])),
            "kernel": rng.choice(["exp", "matern", "both"]), "beta": beta, "ell": round(rng.uniform(0.05, 0.2), 3),
            "tol": rng.choice([1e-4, 1e-5, 1e-6]), "max_rank": rng.choice([0, 0, 64]),
            "reorder": rng.choice([0, 1, 2]), "schur": rng.choice([0, 0, 1])}


# ---- inputs --------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _ranks(order, m, near, far):
    """Ranks of the off-diagonal tiles: position i holds the tile at grid cell order[i]; ranks fall with the
    distance of two cells as on the library's own spatial factors."""
    r = len(order)
    g = int(math.ceil(math.sqrt(r)))
    xy = np.stack([np.asarray(order) // g, np.asarray(order) % g], 1).astype(np.float64)
    d = np.sqrt(((xy[:, None] - xy[None]) ** 2).sum(-1))
    k = np.rint(far + (near - far) * np.maximum(d, 1.0) ** -3.6).astype(np.int64)
    return np.tril(np.minimum(k, m), -1)


def _structure(n, m, near, far, rng):
    """(tile offsets, rank table): all tiles of m variables but one, which may be shorter and sits anywhere."""
    r = -(-n // m)
    order = rng.permutation(r)
    sizes = np.full(r, m, dtype=np.int64)
    sizes[int(rng.integers(r))] = n - (r - 1) * m
    return np.concatenate([[0], np.cumsum(sizes)]), _ranks(order, m, near, far)


def _factor_arrays(n, m, near, far, beta, seed):
    """A factor's arrays in float64 on the host: tile offsets, permutation, ranks, diagonal tiles, and per row
    tile i its U columns (for tiles j = 0..i-1 in order) and their V columns."""
    rng = np.random.default_rng(seed)
    off, rank = _structure(n, m, near, far, rng)
    r = len(off) - 1
    dev = _device()
    # Diagonal tiles: the field of an exponential kernel on a patch of a jittered grid of spacing 1/sqrt(n), in
    # random order, given the earlier tiles: less variance and a shorter range, the same local roughness.
    explained = 0.4 * (1.0 - np.exp(-8.0 * np.arange(r) / max(r, 8)))  # of the variance, by the earlier tiles
    g = int(math.ceil(math.sqrt(m)))
    cell = np.arange(m)
    pts = np.empty((r, m, 2))
    for i in range(r):
        c = rng.permutation(cell)
        pts[i, :, 0] = c // g
        pts[i, :, 1] = c % g
    pts += 0.8 * rng.random((r, m, 2))
    x = torch.as_tensor(pts / math.sqrt(n), device=dev)
    left = torch.as_tensor(1.0 - explained, device=dev)[:, None, None]
    cov = left * torch.exp(-torch.cdist(x, x, compute_mode="donot_use_mm_for_euclid_dist") / (beta * left))
    cov += 1e-8 * torch.eye(m, dtype=torch.float64, device=dev)
    B = torch.linalg.cholesky(cov).cpu().numpy()
    # Off-diagonal tiles: what the earlier tiles explain, smooth over the tile (waves about as long as it is).
    U, V = [], []
    for i in range(r):
        mi, k = int(off[i + 1] - off[i]), int(rank[i].sum())
        if not k:
            U.append(np.zeros((mi, 0)))
            V.append([])
            continue
        js = np.repeat(np.arange(r), rank[i])
        comp = np.concatenate([np.arange(x) for x in rank[i] if x])
        size = np.exp(-0.3 * comp) * np.sqrt(rank[i][js])
        size *= math.sqrt(explained[i] / float((size ** 2).sum()))
        # |u| = |v|, as the compression leaves them: V^T y has a unit variance times |v|
        s = (size * math.sqrt(mi)) ** 0.5
        wave = rng.standard_normal((2, k)) * (1.0 + comp / 16.0) * (2.0 / g)
        U.append(math.sqrt(2.0) * np.cos(pts[i, :mi] @ wave + rng.uniform(0.0, 2.0 * math.pi, k)) * (size / s))
        v, o = [], 0
        for j in range(i):
            q = int(rank[i, j])
            mj = int(off[j + 1] - off[j])
            v.append(rng.standard_normal((mj, q)) / math.sqrt(mj) * s[o:o + q])
            o += q
        V.append(v)
    return off, rng.permutation(n), rank, B, U, V


def _load(arrays, m):
    off, perm, rank, B, U, V = arrays
    r = len(off) - 1
    Ud, Vd = {}, {}
    for i in range(r):
        o = 0
        for j in range(i):
            k = int(rank[i, j])
            if k:
                Ud[(i, j)] = U[i][:, o:o + k]
                Vd[(i, j)] = V[i][j]
                o += k
    tiles = [B[i, :off[i + 1] - off[i], :off[i + 1] - off[i]] for i in range(r)]
    return tl.tlrmvn_factor_import(tl.build_export(int(off[-1]), m, off, perm, tiles, Ud, Vd))


def _limits(kind, n, rng):
    a = np.full(n, -np.inf)
    if kind == "uniform":
        return a, rng.uniform(0.0, 1.0, n)
    if kind == "normal":
        return a, rng.normal(1.0, 0.5, n)
    if kind == "high":
        return a, rng.normal(5.5, 1.25, n)
    return rng.uniform(-3.0, -1.5, n), rng.uniform(0.5, 2.0, n)


def _shift_table(seed, m_shifts, coords):
    rng = np.random.default_rng(seed)
    return rng.integers(0, MASK64, size=(m_shifts, coords), dtype=np.uint64, endpoint=True)


def _prob_inputs(case, seed):
    arrays = _factor_arrays(case["n"], case["m"], case["near"], case["far"], case["beta"], 7919 * seed + 1)
    rng = np.random.default_rng(7919 * seed + 2)
    a, b = _limits(case["limits"], case["n"], rng)
    shifts = _shift_table(7919 * seed + 3, case["shifts"], case["n"] + 1) if case["own_shifts"] else None
    return arrays, a, b, shifts


def _batch_problems(case, seed):
    rng = np.random.default_rng(7919 * seed + 4)
    out = []
    for p in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        nu = 7.0 if rng.random() < case["t_share"] else math.inf
        out.append((n, nu, 7919 * seed + 100 + p))
    return out


def _server_requests(case, seed):
    """(factor, nu, precision, limits' seed, shifts' seed) of every request."""
    return [(q % 4, [math.inf, 7.0, 3.0][q % 3], ["fp32", "bf16"][(q // 2) % 2], 7919 * seed + 300 + q,
             (7919 * seed + 600 + q) & MASK64) for q in range(case["requests"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "prob":
        arrays, a, b, shifts = _prob_inputs(case, seed)
        state = {"case": case, "F": _load(arrays, case["m"]), "shifts": shifts, "seed": 7919 * seed + 5}
        if case["call"] == "host":
            state |= {"a": a, "b": b}
        else:
            dev = torch.device("cuda")
            state |= {"a": torch.as_tensor(a, device=dev), "b": torch.as_tensor(b, device=dev),
                      "out": torch.zeros(2, dtype=torch.float64, device=dev),
                      "samples": torch.zeros(case["shifts"] * case["points"], dtype=torch.float64, device=dev)}
        return state
    if kind == "batch":
        factors, nus, al, bl = [], [], [], []
        for n, nu, s in _batch_problems(case, seed):
            m = min(case["m"], n)
            factors.append(_load(_factor_arrays(n, m, case["near"], case["far"], case["beta"], s), m))
            a, b = _limits("uniform", n, np.random.default_rng(s + 50000))
            nus.append(nu)
            al.append(a)
            bl.append(b)
        plan = tl.BatchPlan(factors, nus, case["shifts"], case["points"], seed=7919 * seed + 5,
                            precision=PRECISION[case["precision"]])
        return {"case": case, "plan": plan, "a": al, "b": bl}
    if kind == "server":
        factors = []
        for f in range(4):
            n = case["n%d" % f]
            m = min(case["m"], n)
            factors.append(_load(_factor_arrays(n, m, case["near"], case["far"], case["beta"], 7919 * seed + 10 + f), m))
        reqs = []
        for f, nu, precision, ls, ss in _server_requests(case, seed):
            a, b = _limits("uniform", case["n%d" % f], np.random.default_rng(ls))
            reqs.append((f, a, b, nu, precision, ss))
        return {"case": case, "factors": factors, "server": tl.Server(factors, lanes=case["lanes"]), "requests": reqs}
    n = case["n"]
    rng = np.random.default_rng(7919 * seed + 6)
    g = int(math.ceil(math.sqrt(n)))
    c = np.arange(g * g)[:n]
    xy = (np.stack([c // g, c % g], 1) + 0.8 * rng.random((n, 2))) / g
    a, b = _limits("uniform", n, rng)
    kernel, params = {"exp": (tl.KERNEL_EXP, (case["beta"],)), "matern": (tl.KERNEL_MATERN15, (case["ell"],)),
                      "both": (tl.KERNEL_EXP_MATERN15, (case["beta"], case["ell"]))}[case["kernel"]]
    return {"case": case, "xy": xy, "a": a, "b": b, "kernel": kernel, "params": params}


# ---- one pass -------------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "prob":
        T = RESULT[case["precision"]]
        if case["call"] == "host":
            lp, er, per_shift, _ = tl.tlrmvn_prob(state["F"], state["a"], state["b"], case["nu"],
                                                  PRECISION[case["precision"]], case["shifts"], case["points"],
                                                  shifts=state["shifts"], seed=state["seed"],
                                                  periodize=case["periodize"], per_shift=True)
            return {"logs": np.concatenate([[lp, er], per_shift]).astype(T)}
        tl.tlrmvn_prob_device(state["F"], state["a"], state["b"], state["out"], case["nu"],
                              PRECISION[case["precision"]], case["shifts"], case["points"], shifts=state["shifts"],
                              seed=state["seed"], periodize=case["periodize"], per_sample=state["samples"])
        t = {np.float64: torch.float64, np.float32: torch.float32, np.float16: torch.float16}[T]
        return {"logs": torch.cat([state["out"], state["samples"]]).to(t)}
    if kind == "batch":
        T = RESULT[case["precision"]]
        lp, er = state["plan"].run(state["a"], state["b"])
        got = np.stack([lp, er], 1).astype(T)
        return {"estimates": list(got) if T is np.float32 else got}
    if kind == "server":
        srv = state["server"]
        ids = [srv.submit(f, a, b, nu, PRECISION[precision], case["shifts"], case["points"], seed=ss)
               for f, a, b, nu, precision, ss in state["requests"]]
        got = [srv.wait(i)[:2] for i in ids]
        return {p: np.array([e for e, q in zip(got, state["requests"]) if q[4] == p]).astype(RESULT[p])
                for p in ("fp32", "bf16")}
    F = tl.tlrmvn_factor_kernel(state["xy"], state["kernel"], state["params"], 1e-8, state["a"], state["b"], case["m"],
                                case["tol"], case["max_rank"], case["reorder"], schur=case["schur"])
    buf = tl.tlrmvn_factor_export(F)
    F.close()
    n, r, m, _ = (int(x) for x in np.frombuffer(buf, np.int64, 4, 8))
    o = 40 + 8 * (r + 1)
    perm = np.frombuffer(buf, np.int64, n, o)
    o += 8 * n
    rank = np.frombuffer(buf, np.int32, r * r, o)
    o += 4 * r * r
    B = np.frombuffer(buf, np.float64, r * m * m, o)
    o += 8 * r * m * m
    # U and V of the off-diagonal tiles, in an array whose length does not depend on the ranks found (some 100 for
    # the neighbours of a tile and a quarter of that for the others are never reached)
    pairs = r * (r - 1) // 2
    near = min(pairs, 4 * r)
    uv = np.frombuffer(buf, np.float64, (len(buf) - o) // 8, o)
    out = np.zeros(max(uv.size, 2 * m * (near * min(m, 100) + (pairs - near) * min(m, 25))))
    out[:uv.size] = uv
    return {"perm": perm, "rank": rank, "B": B, "UV": out}


# ---- what a pass cannot do without -------------------------------------------------------------------

def _prob_work(n, m, near, far, shifts, points, es, seed=1):
    off, rank = _structure(n, m, near, far, np.random.default_rng(seed))
    sizes = np.diff(off)
    S = shifts * points
    uv = float((rank * (sizes[:, None] + sizes[None, :])).sum())  # entries of all U and V
    flops = S * (float((sizes * (sizes - 1)).sum()) + 2.0 * uv + FLOPS_SPECIAL * n)
    nbytes = es * (float((sizes * (sizes + 1) // 2).sum()) + uv) + 16.0 * n + 8.0 * shifts * (n + 1)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "prob":
        es = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}[case["precision"]]
        nbytes, flops = _prob_work(case["n"], case["m"], case["near"], case["far"], case["shifts"], case["points"], es)
        return {"bytes": nbytes + 8.0 * case["shifts"] * case["points"], "flops": flops}
    if kind in ("batch", "server"):
        if kind == "batch":
            problems = [(n, {"fp32": 4, "bf16": 2}[case["precision"]]) for n, _, _ in _batch_problems(case, 1)]
        else:
            problems = [(case["n%d" % f], {"fp32": 4, "bf16": 2}[p]) for f, _, p, _, _ in _server_requests(case, 1)]
        got = [_prob_work(n, min(case["m"], n), case["near"], case["far"], case["shifts"], case["points"], es)
               for n, es in problems]
        return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}
    # the factor: Cholesky of the diagonal tiles, and per off-diagonal tile the covariance, the product with the
    # inverse of a triangular tile and the compression to a rank of about 8
    n, m = case["n"], case["m"]
    r = -(-n // m)
    tiles = r * (r - 1) / 2
    conditioning = {0: 0, 1: r, 2: tiles + r}[case["reorder"]]
    flops = (r + conditioning) * m ** 3 / 3 + tiles * (m ** 3 + 20.0 * m * m + 2.0 * 8 * m * m)
    return {"bytes": 16.0 * n + 8.0 * (r * m * m / 2 + tiles * 16 * m), "flops": flops}


# ---- the same in 64 bits -------------------------------------------------------------------------------

def _primes(count):
    top = max(32, int(count * (math.log(count + 2) + math.log(math.log(count + 3)) + 1)))
    sieve = np.ones(top, dtype=bool)
    sieve[:2] = False
    for p in range(2, int(math.isqrt(top)) + 1):
        if sieve[p]:
            sieve[p * p::p] = False
    return np.flatnonzero(sieve)[:count]


def _generators(count):
    """floor(frac(sqrt(p)) 2^64) of the first primes."""
    out = np.empty(count, dtype=np.uint64)
    for i, p in enumerate(_primes(count)):
        out[i] = math.isqrt(int(p) << 128) & MASK64
    return out


def _splitmix(seed, count):
    with np.errstate(over="ignore"):
        z = np.uint64(seed & MASK64) + (np.arange(1, count + 1, dtype=np.uint64)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _lattice(Q, D, k, periodize):
    """(w, 1 - w) of lattice points k (int64) for one coordinate: generator Q, shifts D (int64, one per sample)."""
    x = k * Q + D
    if periodize:
        num = 2 * ((x >> 11) & ((1 << 53) - 1)) + 1 - (1 << 53)
        num = num.abs()
    else:
        num = 2 * ((x >> 12) & ((1 << 52) - 1)) + 1
    return num.double() * 2.0 ** -53, ((1 << 53) - num).double() * 2.0 ** -53


def _chi_scale(w, wc, nu):
    """chi_nu^-1(w) / sqrt(nu) by Newton's method on the regularised incomplete gamma function."""
    a = torch.full_like(w, 0.5 * nu)
    z = torch.special.ndtri(torch.minimum(w, wc))
    z = torch.where(w <= wc, z, -z)
    t = 2.0 / (9.0 * nu)
    x = torch.clamp(0.5 * nu * (1.0 - t + z * math.sqrt(t)) ** 3, min=1e-300)
    small = torch.exp((torch.log(w) + torch.special.gammaln(a + 1.0)) / a)  # the leading term near 0
    x = torch.where(x < 0.1 * small, small, x)
    for _ in range(60):
        f = torch.where(w < 0.5, torch.special.gammainc(a, x) - w, wc - torch.special.gammaincc(a, x))
        pdf = torch.exp((a - 1.0) * torch.log(x) - x - torch.special.gammaln(a))
        step = f / pdf
        new = torch.where(x - step > 0.0, x - step, 0.5 * x)
        done = bool(((new - x).abs() <= 1e-15 * x).all())
        x = new
        if done:
            break
    return torch.sqrt(2.0 * x / nu)


def _ndtr(x):
    """Phi(x), accurate in the lower tail."""
    return 0.5 * torch.erfc(-math.sqrt(0.5) * x)


def _log_ndtri(lu):
    """Phi^-1(exp(lu)) for lu far below 0, by Newton's method on log Phi."""
    lu = torch.clamp(lu, max=-2.0)
    z = -torch.sqrt(-2.0 * lu)
    for _ in range(12):
        lp = torch.special.log_ndtr(z)
        z = z - (lp - lu) * torch.exp(lp + 0.5 * z * z) * math.sqrt(2.0 * math.pi)
    return z


def _estimate(logs, shifts):
    ell = torch.logsumexp(logs.reshape(shifts, -1), 1) - math.log(logs.numel() // shifts)
    lp = torch.logsumexp(ell, 0) - math.log(shifts)
    e = torch.exp(ell - lp)
    err = e.std(unbiased=True) / math.sqrt(shifts) if shifts > 1 else torch.tensor(math.nan)
    return ell, float(lp), float(err)


def _integrand(arrays, a, b, nu, table, points, periodize):
    """Log integrand of every sample (shift-major) of the separation-of-variables estimate on the factor."""
    off, perm, rank, B, U, V = arrays
    dev = _device()
    n, r, shifts = int(off[-1]), len(off) - 1, table.shape[0]
    S = shifts * points
    Q = _generators(n + 1).view(np.int64)
    D = torch.as_tensor(table.view(np.int64).T.copy(), device=dev)  # (n + 1, shifts)
    k = torch.arange(1, points + 1, dtype=torch.int64, device=dev).repeat(shifts)
    own = torch.arange(shifts, device=dev).repeat_interleave(points)
    rs = 1.0
    if math.isfinite(nu):
        rs = _chi_scale(*_lattice(int(Q[n]), D[n][own], k, periodize), nu)
    ap, bp = a[perm], b[perm]
    one_sided = bool(np.all(np.isneginf(ap)))
    logs = torch.zeros(S, dtype=torch.float64, device=dev)
    start = np.concatenate([[0], np.cumsum(rank.sum(1))])  # first row of each tile's projections
    W = torch.zeros(int(start[-1]), S, dtype=torch.float64, device=dev)
    Qd = torch.as_tensor(Q, device=dev)[:, None]
    for i in range(r):
        t0, mi = int(off[i]), int(off[i + 1] - off[i])
        Bi = torch.as_tensor(B[i, :mi, :mi], device=dev)
        shift = torch.as_tensor(U[i], device=dev) @ W[int(start[i]):int(start[i + 1])]
        Y = torch.zeros(mi, S, dtype=torch.float64, device=dev)
        diag = np.diag(B[i])
        for q0 in range(0, mi, 64):
            q1 = min(q0 + 64, mi)
            if q0:
                shift[q0:q1] += Bi[q0:q1, :q0] @ Y[:q0]
            w, wc = _lattice(Qd[t0 + q0:t0 + q1], D[t0 + q0:t0 + q1][:, own], k, periodize)
            if one_sided:
                bts = torch.empty_like(w)
            for v in range(q0, q1):
                s = torch.addmv(shift[v], Y[q0:v].T, Bi[v, q0:v]) if v > q0 else shift[v]
                bt = (float(bp[t0 + v]) * rs - s) / float(diag[v])
                if one_sided:
                    # u = w Phi(bt) and its complement, from the smaller of Phi(bt) and Phi(-bt)
                    bts[v - q0] = bt
                    h = _ndtr(-bt.abs())
                    neg = bt < 0.0
                    e, ec = torch.where(neg, h, 1.0 - h), torch.where(neg, 1.0 - h, h)
                    u, uc = w[v - q0] * e, torch.addcmul(ec, wc[v - q0], e)
                    sign, hi, ld = 1.0, bt, None
                else:  # an interval: reflected so that it starts in the lower half
                    at = (float(ap[t0 + v]) * rs - s) / float(diag[v])
                    up = at > 0.0
                    lo, hi = torch.where(up, -bt, at), torch.where(up, -at, bt)
                    ww, wwc = torch.where(up, wc[v - q0], w[v - q0]), torch.where(up, w[v - q0], wc[v - q0])
                    sign = torch.where(up, -1.0, 1.0)
                    d, e, ec = _ndtr(lo), _ndtr(hi), _ndtr(-hi)
                    diff = torch.where(hi <= 0.0, e - d, 1.0 - ec - d)
                    ld = torch.log(diff)
                    u, uc = d + ww * diff, ec + wwc * diff
                z = torch.special.ndtri(torch.minimum(u, uc))
                if float(hi.min()) < -30.0:  # Phi near or below the smallest float: the same in logs
                    deep = hi < -30.0
                    lb = torch.special.log_ndtr(hi)
                    if one_sided:
                        lu = torch.log(w[v - q0]) + lb
                    else:
                        dl = torch.special.log_ndtr(lo) - lb
                        ld = torch.where(deep, lb + torch.log(-torch.expm1(dl)), ld)
                        lu = lb + torch.log(ww + wwc * torch.exp(dl))
                    z = torch.where(deep, _log_ndtri(lu), z)
                    u, uc = torch.where(deep, 0.0, u), torch.where(deep, 1.0, uc)
                if ld is not None:
                    logs += ld
                Y[v] = sign * torch.where(u <= uc, z, -z)
            if one_sided:
                logs += torch.where(bts <= 0.0, torch.special.log_ndtr(bts),
                                    torch.log1p(-_ndtr(-bts))).sum(0)
        for t in range(i + 1, r):
            kk = int(rank[t, i])
            if kk:
                o = int(start[t] + rank[t, :i].sum())
                W[o:o + kk] = torch.as_tensor(V[t][i], device=dev).T @ Y
    return logs


def _seed_table(seed, shifts, n):
    return _splitmix(seed, shifts * (n + 1)).reshape(shifts, n + 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "prob":
        n, S = case["n"], case["shifts"] * case["points"]
        if n * S > 2e9 or n > 32768:
            return None  # over 20 seconds
        arrays, a, b, table = _prob_inputs(case, seed)
        if table is None:
            table = _seed_table(7919 * seed + 5, case["shifts"], n)
        logs = _integrand(arrays, a, b, case["nu"], table, case["points"], case["periodize"])
        ell, lp, er = _estimate(logs, case["shifts"])
        if case["call"] == "host":
            return {"logs": np.concatenate([[lp, er], ell.cpu().numpy()])}
        return {"logs": np.concatenate([[lp, er], logs.cpu().numpy()])}
    if kind == "batch":
        out, left = [], EXACT_VARIABLES
        for p, (n, nu, s) in enumerate(_batch_problems(case, seed)):
            left -= n
            if left < 0:
                out.append(None)  # over 20 seconds with the others
                continue
            arrays = _factor_arrays(n, min(case["m"], n), case["near"], case["far"], case["beta"], s)
            a, b = _limits("uniform", n, np.random.default_rng(s + 50000))
            table = _seed_table(7919 * seed + 5 + p, case["shifts"], n)
            logs = _integrand(arrays, a, b, nu, table, case["points"], True)
            out.append(np.array(_estimate(logs, case["shifts"])[1:]))
        if case["precision"] == "bf16":
            return {"estimates": np.array(out)} if left >= 0 else None
        return {"estimates": out}
    if kind == "server":
        reqs = _server_requests(case, seed)
        if sum(case["n%d" % f] for f, *_ in reqs) > 1.3 * EXACT_VARIABLES:
            return None  # over 20 seconds
        arrays = [_factor_arrays(case["n%d" % f], min(case["m"], case["n%d" % f]), case["near"], case["far"],
                                 case["beta"], 7919 * seed + 10 + f) for f in range(4)]
        out = {"fp32": [], "bf16": []}
        for f, nu, precision, ls, ss in reqs:
            n = case["n%d" % f]
            a, b = _limits("uniform", n, np.random.default_rng(ls))
            logs = _integrand(arrays[f], a, b, nu, _seed_table(ss, case["shifts"], n), case["points"], True)
            out[precision].append(_estimate(logs, case["shifts"])[1:])
        return {p: np.array(v) for p, v in out.items()}
    return None  # a truncated, reordered factor is defined by the steps that make it
