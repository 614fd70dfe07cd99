"""The work that users of this framework have it do, as cases that can be timed.

A case is a dict: a "kind" (which entry points a pass calls), the matrix
family with its sizes, and the options of the call.  Matrices are built on
the GPU with plain torch; x* ~ U[-1, 1] comes from the seed and b = A x*.  A
pass returns the solution and, where the method chooses them, the class of
eps1, the 2BFS pseudo-diameter and the decay rate v.  Iteration counts and
clock marks of the result record are not among the outputs: the count moves
by one or two with the order of the sums, and the marks are times.
"""
import math

import numpy as np
import torch

from paper_2412_08059_gb300 import mpcg

DEV = "cuda"


# ---------------------------------------------------------------------------------------
# Matrices (CSR: int32 row_ptr and col, float64 val, columns sorted, diagonal stored)
# ---------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _grid(nx, ny, nz, cy, cz, sigma):
    """Dirichlet Laplacian of an nx x ny x nz grid (nz = 1: 5-point), x fastest,
    coefficients (1, cy, cz), plus sigma I."""
    n, pl = nx * ny * nz, nx * ny
    i = torch.arange(n, device=DEV)
    x, y, z = i % nx, (i // nx) % ny, i // pl
    deep = nz > 1
    diag = 2.0 + 2.0 * cy + (2.0 * cz if deep else 0.0) + sigma
    ones = torch.ones_like(x, dtype=torch.bool)
    legs = [(-nx, -cy, y > 0), (-1, -1.0, x > 0), (0, diag, ones), (1, -1.0, x < nx - 1), (nx, -cy, y < ny - 1)]
    if deep:
        legs = [(-pl, -cz, z > 0)] + legs + [(pl, -cz, z < nz - 1)]
    mask = torch.stack([m for _, _, m in legs], 1)
    cols = torch.stack([i + o for o, _, _ in legs], 1)
    vals = torch.tensor([v for _, v, _ in legs], dtype=torch.float64, device=DEV).expand(n, len(legs))
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(mask.sum(1), 0)
    return rp, cols[mask], vals[mask]


def _row_sums(rp, v):
    return torch.segment_reduce(v, "sum", offsets=rp)


def _from_pairs(n, lo, hi, value, diagonal):
    """Symmetric CSR from undirected edges lo < hi without duplicates; diagonal(sum_j |a_ij|)."""
    i = torch.arange(n, device=DEV)
    r, c = torch.cat([lo, hi, i]), torch.cat([hi, lo, i])
    v = torch.cat([value, value, torch.zeros(n, dtype=torch.float64, device=DEV)])
    key, order = torch.sort(r * n + c)
    v = v[order]
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    c = key % n
    v[(key // n) == c] = diagonal(_row_sums(rp, v.abs()))
    return rp, c, v


def _dominant(mu):
    return lambda s: torch.where(s > 0, mu * s, torch.ones_like(s))


def _values(count, g):
    """Magnitudes U(0, 3) or U(7, 10) with equal chance, signs with equal chance."""
    u = torch.rand(4, count, generator=g, device=DEV, dtype=torch.float64)
    mag = torch.where(u[0] > 0.5, 3.0 * u[2], 7.0 + 3.0 * u[3])
    return torch.where(u[1] > 0.5, mag, -mag)


def _distinct(n, a, b):
    keep = a != b
    a, b = a[keep], b[keep]
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    return key // n, key % n


def _matrix(m, seed):
    g = _gen(7919 * seed + 11)
    f, n = m["family"], size_of(m)[0]
    if f == "lap2d":
        return _grid(m["nx"], m["ny"], 1, 1.0, 0.0, m.get("sigma", 0.0))
    if f == "lap3d":
        return _grid(m["nx"], m["ny"], m["nz"], 1.0, m.get("eps", 1.0), m.get("sigma", 0.0))
    if f == "regular":  # configuration model, self-loops and double edges removed
        stubs = torch.arange(n, device=DEV).repeat_interleave(m["degree"])
        stubs = stubs[torch.randperm(stubs.numel(), generator=g, device=DEV)]
        half = stubs.numel() // 2
        lo, hi = _distinct(n, stubs[:half], stubs[half:2 * half])
        return _from_pairs(n, lo, hi, -torch.ones(lo.numel(), dtype=torch.float64, device=DEV),
                           lambda s: s + m["shift"])
    if f == "tree":  # random tree on a random order of the vertices, plus c n random edges
        k = torch.arange(1, n, device=DEV)
        u = torch.rand(n - 1, generator=g, device=DEV, dtype=torch.float64)
        parent = torch.minimum((u * k).long(), k - 1)
        perm = torch.randperm(n, generator=g, device=DEV)
        extra = torch.randint(0, n, (2, int(m["c"] * n)), generator=g, device=DEV)
        lo, hi = _distinct(n, torch.cat([perm[k], extra[0]]), torch.cat([perm[parent], extra[1]]))
        return _from_pairs(n, lo, hi, _values(lo.numel(), g), _dominant(m["mu"]))
    if f == "banded":  # every pair within the band with probability p
        lo, hi = [], []
        for off in range(1, (m["band"] - 1) // 2 + 1):
            i = torch.arange(n - off, device=DEV)
            i = i[torch.rand(n - off, generator=g, device=DEV) < m["p"]]
            lo.append(i)
            hi.append(i + off)
        lo, hi = torch.cat(lo), torch.cat(hi)
        return _from_pairs(n, lo, hi, _values(lo.numel(), g), _dominant(m["mu"]))
    raise KeyError(f)


def size_of(m):
    """(rows, stored entries) of a matrix, the entries close to the drawn number for random graphs."""
    f = m["family"]
    if f == "lap2d":
        nx, ny = m["nx"], m["ny"]
        return nx * ny, 5 * nx * ny - 2 * (nx + ny)
    if f == "lap3d":
        nx, ny, nz = m["nx"], m["ny"], m["nz"]
        return nx * ny * nz, 7 * nx * ny * nz - 2 * (nx * ny + ny * nz + nx * nz)
    n = m["n"]
    if f == "regular":
        return n, n * (m["degree"] + 1)
    if f == "tree":
        return n, 3 * n + 2 * int(m["c"] * n)
    return n, n + int(n * (m["band"] - 1) * m["p"])


def _star(n, seed):
    return 2.0 * torch.rand(n, generator=_gen(seed), device=DEV, dtype=torch.float64) - 1.0


def _system(m, seed):
    """(device matrix, b, x*) with b = A x*."""
    rp, col, val = _matrix(m, seed)
    xs = _star(rp.numel() - 1, seed)
    b = _row_sums(rp, val * xs[col])
    return mpcg.DeviceCSR(rp, col, val, DEV), b, xs


# ---------------------------------------------------------------------------------------
# Several systems: sizes log-uniform over a range, the four grid families in turn
# ---------------------------------------------------------------------------------------
def _mix(count, n_lo, n_hi, pick):
    r = np.random.default_rng(pick)
    out = []
    for k in range(count):
        n = math.exp(r.uniform(math.log(n_lo), math.log(n_hi)))
        if k % 4 == 0:
            s = max(2, round(math.sqrt(min(n, 2.6e5))))
            out.append({"family": "lap2d", "nx": s, "ny": s + int(r.integers(0, 3))})
        else:
            s = max(2, round(n ** (1.0 / 3.0)))
            out.append({"family": "lap3d", "nx": s, "ny": s, "nz": s,
                        "eps": (1.0, 1.0, float(r.choice([1e-2, 1e-3])), 1.0)[k % 4],
                        "sigma": (0.0, 0.0, 0.0, float(r.choice([1e-4, 1e-2, 1.0])))[k % 4]})
    return out


def _slices(mats):
    """Offsets of the systems' vectors in one buffer (256-byte steps) and its length."""
    at, off = [], 0
    for m in mats:
        at.append(off)
        off += (size_of(m)[0] + 31) // 32 * 32
    return at, off


def _sample_rows(count):
    """A labelled sample like those of the evaluation protocol: features (n, m, l~, v) spread
    over the families' ranges and classes of eps1 = 1e-2 .. 1e-7."""
    r = np.random.default_rng(5)
    n = np.exp(r.uniform(math.log(1e3), math.log(2e6), count)).round()
    feat = np.stack([n, (n * r.uniform(3.0, 9.0, count)).round(),
                     np.exp(r.uniform(math.log(5.0), math.log(5e3), count)).round(),
                     r.uniform(0.3, 0.99, count)], 1)
    return feat, r.choice(np.array([2, 3, 4, 5, 6, 7], np.int8), count, p=[.05, .05, .1, .2, .3, .3])


def _sample(count):
    return mpcg.DeviceSample(*_sample_rows(count), device=DEV)


# ---------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # one small system, eps1 given: the plain method on the 64 x 64 Poisson matrix
        {"name": "solve_poisson64", "kind": "solve", "family": "lap2d", "nx": 64, "ny": 64, "mode": "eps1", "eps1": 1e-4, "eps2": 1e-10},
        # one sparse matrix of the random family of the evaluation protocol, eps1 chosen
        {"name": "solve_tree_auto", "kind": "solve", "family": "tree", "n": 3001, "c": 0.5, "mu": 1.1, "mode": "auto", "sample": 1260, "eps2": 1e-10},
        # an ordinary system, odd sizes, eps1 chosen
        {"name": "solve_2d_auto", "kind": "solve", "family": "lap2d", "nx": 301, "ny": 203, "sigma": 1e-2, "mode": "auto", "sample": 256, "eps2": 1e-10},
        # an ordinary system in double precision only: the baseline every user compares with
        {"name": "solve_3d_fp64", "kind": "solve", "family": "lap3d", "nx": 61, "ny": 53, "nz": 47, "eps": 1e-2, "mode": "fp64", "eps2": 1e-10},
        # the headline size of the benchmark
        {"name": "solve_128_auto", "kind": "solve", "family": "lap3d", "nx": 128, "ny": 128, "nz": 128, "mode": "auto", "sample": 256, "eps2": 1e-10},
        # a large graph of small diameter, columns far from the diagonal
        {"name": "solve_regular_auto", "kind": "solve", "family": "regular", "n": 1 << 20, "degree": 8, "shift": 1e-3, "mode": "auto", "sample": 256, "eps2": 1e-10},
        # Jacobi preconditioning on a matrix with an uneven diagonal
        {"name": "solve_banded_pcg", "kind": "solve", "family": "banded", "n": 1 << 20, "band": 15, "p": 0.6, "mu": 1.1, "mode": "eps1", "eps1": 1e-5, "eps2": 1e-10, "precond": 1},
        # the features of a thin grid: thousands of narrow levels
        {"name": "features_thin", "kind": "features", "family": "lap2d", "nx": 4096, "ny": 64},
        # many systems in one call, eps1 chosen for each
        {"name": "batch_auto", "kind": "batch", "count": 192, "n_lo": 1e3, "n_hi": 2.6e5, "pick": 11, "mode": "auto", "sample": 256, "eps2": 1e-10},
        # the same in double precision only
        {"name": "batch_fp64", "kind": "batch", "count": 192, "n_lo": 1e3, "n_hi": 2.6e5, "pick": 12, "mode": "fp64", "eps2": 1e-10},
        # a burst of requests at the server, admitted as slots free up
        {"name": "serve_burst", "kind": "serve", "count": 32, "slots": 24, "n_lo": 1e3, "n_hi": 8e5, "pick": 21, "mode": "auto", "sample": 256, "iters": 40},
        # classification of a test set, with the neighbours that the localization measure counts
        {"name": "knn_testset", "kind": "knn", "count": 4800, "sample": 1260, "k": 5, "weighted": 1, "neighbours": 1},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["features", "batch", "batch", "serve", "knn"])
    if kind == "solve":
        f = rng.choice(["lap2d", "lap2d", "lap3d", "lap3d", "lap3d", "tree", "regular", "banded"])
        c = {"kind": "solve", "family": f}
        if f == "lap2d":
            s = math.sqrt(_log(rng, 1e3, 1.2e5))
            t = rng.uniform(0.6, 1.6)
            c.update(nx=max(8, round(s * t)), ny=max(8, round(s / t)), sigma=rng.choice([0.0, 1e-3, 1e-2]))
        elif f == "lap3d":
            s = _log(rng, 1e3, 1.9e6) ** (1.0 / 3.0)
            c.update(nx=max(4, round(s * rng.uniform(0.8, 1.0))), ny=max(4, round(s)), nz=max(4, round(s * rng.uniform(0.8, 1.0))))
            c.update(rng.choice([{"sigma": 0.0}, {"sigma": 1e-4}, {"sigma": 1e-2}, {"sigma": 1.0}, {"eps": 1e-2}, {"eps": 1e-3}]))
        elif f == "tree":
            c.update(n=round(_log(rng, 301, 2e5)), c=rng.choice([0.0, 0.25, 0.5, 1.0]), mu=rng.choice([1.1, 3.0]))
        elif f == "regular":
            c.update(n=round(_log(rng, 5e3, 1e6)), degree=rng.choice([6, 8]), shift=1e-3)
        else:
            c.update(n=round(_log(rng, 301, 1e6)), band=rng.choice([3, 7, 15, 29]), p=rng.choice([0.3, 0.6, 0.9]), mu=1.1)
        c["eps2"] = rng.choice([1e-8, 1e-10, 1e-10])
        c["mode"] = rng.choice(["auto", "auto", "eps1", "fp64"])
        if c["mode"] == "auto":
            c["sample"] = rng.choice([36, 256, 1260])
        elif c["mode"] == "eps1":
            c["eps1"] = rng.choice([1e-3, 1e-4, 1e-5, 1e-6])
        if f == "banded" and rng.random() < 0.5:
            c["precond"] = 1
        return c
    if kind == "features":
        short = round(_log(rng, 16, 256))
        long = round(_log(rng, 256, 4096))
        nx, ny = (long, short) if rng.random() < 0.5 else (short, long)
        return {"kind": "features", "family": "lap2d", "nx": nx, "ny": ny}
    if kind in ("batch", "serve"):
        c = {"kind": kind, "count": round(_log(rng, 8, 160 if kind == "batch" else 32)), "n_lo": 1e3,
             "n_hi": float(round(_log(rng, 3e4, 2.6e5 if kind == "batch" else 8e5))), "pick": rng.randrange(1 << 20),
             "mode": rng.choice(["auto", "fp64"])}
        if c["mode"] == "auto":
            c["sample"] = 256
        if kind == "batch":
            c.update(eps2=1e-10, team_rows=rng.choice([8192, 16384, 32768]))
        else:
            c.update(slots=rng.choice([8, 24, 64]), iters=40)
        return c
    return {"kind": "knn", "count": round(_log(rng, 64, 4800)), "sample": round(_log(rng, 36, 1260)), "k": rng.choice([1, 5, 10, 15, 20]),
            "weighted": rng.choice([0, 1, 1]), "neighbours": rng.choice([0, 1])}


# ---------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------
def _options(c):
    kw = {"eps2": c["eps2"]} if "eps2" in c else {}
    if c["mode"] == "eps1":
        kw["eps1"] = c["eps1"]
    if c["mode"] == "fp64":
        kw["fp64_only"] = 1
    for k in ("precond", "team_rows"):
        if k in c:
            kw[k] = c[k]
    return mpcg.options(**kw)


def _record(res, count, mode):
    """Views of the records' status and, where eps1 is chosen, its class, l~ and v."""
    ints = res.view(torch.int32).view(count, -1)
    out = {"status": ints[:, 0]}
    if mode == "auto":
        reals = res.view(torch.float64).view(count, -1)
        out.update(cls=ints[:, 3], pdiam=reals[:, 5], v=reals[:, 6])
    return out


def prepare(case, seed):
    kind = case["kind"]
    S = _sample(case["sample"]) if "sample" in case else None
    if kind == "knn":
        g = _gen(seed)
        u = torch.rand(case["count"], 4, generator=g, device=DEV, dtype=torch.float64)
        n = torch.exp(u[:, 0] * math.log(2e3) + math.log(1e3)).round()
        chi = torch.stack([n, (n * (3.0 + 6.0 * u[:, 1])).round(), torch.exp(u[:, 2] * math.log(1e3) + math.log(5.0)).round(), 0.3 + 0.69 * u[:, 3]], 1)
        return {"kind": kind, "chi": chi.contiguous(), "S": S, "case": case}
    if kind in ("solve", "features"):
        A, b, _ = _system(case, seed)
        s = {"kind": kind, "A": A, "b": b, "S": S}
        if kind == "features":
            s["ws"] = mpcg.workspace(A.n, A.nnz)
            return s
        s["o"] = _options(case)
        s["ws"] = mpcg.workspace(A.n, A.nnz, opts=s["o"])
        s["x"] = torch.empty(A.n, dtype=torch.float64, device=DEV)
        s["res"] = mpcg.result_buffer(1, DEV)
        s["out"] = {"x": s["x"], **_record(s["res"], 1, case["mode"])}
        return s
    mats = _mix(case["count"], case["n_lo"], case["n_hi"], case["pick"])
    at, total = _slices(mats)
    x = torch.zeros(total, dtype=torch.float64, device=DEV)
    sys = [_system(m, 1000 * (seed % 100000) + i) for i, m in enumerate(mats)]
    s = {"kind": kind, "A": [a for a, _, _ in sys], "b": [b for _, b, _ in sys], "S": S, "o": _options(case),
         "x": [x[o:o + a.n] for o, (a, _, _) in zip(at, sys)], "res": mpcg.result_buffer(len(mats), DEV)}
    s["out"] = {"x": x, **_record(s["res"], len(mats), case["mode"])}
    if kind == "batch":
        s["ws"] = torch.empty(mpcg.batch_workspace_bytes(s["A"]), dtype=torch.uint8, device=DEV)
        return s
    need = sorted((mpcg.workspace_bytes(a.n, a.nnz) + 256 for a in s["A"]), reverse=True)
    s["server"] = mpcg.Server(case["slots"], sum(need[:max(4, case["slots"] // 2)]), s["o"], S, DEV)
    one = s["res"].numel() // len(mats)
    s["recs"] = [s["res"][i * one:(i + 1) * one] for i in range(len(mats))]
    s["eps2"] = [(1e-8, 1e-10)[i % 2] for i in range(len(mats))]
    s["iters"] = case["iters"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "solve":
        mpcg.solve_async(s["A"], s["b"], s["x"], s["o"], s["ws"], s["res"], s["S"])
        return s["out"]
    if kind == "features":
        f = mpcg.features(s["A"], s["b"], ws=s["ws"])
        return {"pdiam": int(f["pdiam"]), "v": f["v"], "status": f["status"]}
    if kind == "batch":
        mpcg.solve_batch_async(s["A"], s["b"], s["x"], s["o"], s["ws"], s["res"], s["S"])
        return s["out"]
    if kind == "serve":  # every request waits at the door; the host looks at the phases after each step
        srv, live, nxt = s["server"], {}, 0
        while nxt < len(s["A"]) or live:
            while nxt < len(s["A"]):
                slot = srv.admit(s["A"][nxt], s["b"][nxt], s["x"][nxt], s["eps2"][nxt], s["recs"][nxt])
                if slot is None:
                    break
                live[slot] = nxt
                nxt += 1
            srv.step(s["iters"])
            torch.cuda.current_stream().synchronize()
            phase = srv.phase.tolist()
            for slot in [k for k in live if phase[k] == mpcg.PHASE_DONE]:
                srv.retire(slot)
                del live[slot]
        return s["out"]
    c = s["case"]
    r = mpcg.knn_batch(s["chi"], s["S"], neighbours=bool(c["neighbours"]), knn_k=c["k"], weighted=c["weighted"])
    return {"cls": r[0], "nbr": r[1]} if c["neighbours"] else {"cls": r}


# ---------------------------------------------------------------------------------------
# Work, tolerance, exact results
# ---------------------------------------------------------------------------------------
def _iterations(m, eps2):
    """Double-precision CG iterations to eps2, roughly: 0.22 sqrt(kappa) ln(2 / eps2)
    with the closed-form condition number of the grids, and of the dominant diagonal
    (1 + 1 / mu) / (1 - 1 / mu) of the other families."""
    f = m["family"]
    if f in ("lap2d", "lap3d"):
        sides = [(m["nx"], 1.0), (m["ny"], 1.0)] + ([(m["nz"], m.get("eps", 1.0))] if f == "lap3d" else [])
        sigma = m.get("sigma", 0.0)
        top = sigma + sum(2.0 * c * (1.0 + math.cos(math.pi / (s + 1))) for s, c in sides)
        low = sigma + sum(2.0 * c * (1.0 - math.cos(math.pi / (s + 1))) for s, c in sides)
        kappa = top / low
    elif f == "regular":
        kappa = 16.0
    else:
        kappa = (1.0 + 1.0 / m["mu"]) / (1.0 - 1.0 / m["mu"]) * 4.0
    return 2.0 + 0.22 * math.sqrt(kappa) * math.log(2.0 / eps2)


def work(case):
    if case["kind"] == "knn":
        q, n = case["count"], case["sample"]
        return {"bytes": 32.0 * q + 33.0 * n + 4.0 * q * (1 + case["neighbours"] * case["k"]), "flops": 12.0 * q * n}
    if case["kind"] == "features":
        n, m = size_of(case)
        return {"bytes": 12.0 * m + 12.0 * n, "flops": 10 * 2.0 * (m + 5.0 * n)}
    if case["kind"] == "solve":
        todo = [(case, case["eps2"])]
    else:
        todo = [(m, case.get("eps2", (1e-8, 1e-10)[i % 2]))
                for i, m in enumerate(_mix(case["count"], case["n_lo"], case["n_hi"], case["pick"]))]
    total = {"bytes": 0.0, "flops": 0.0}
    for m, eps2 in todo:
        n, z = size_of(m)
        total["bytes"] += 12.0 * z + 4.0 * n + 16.0 * n  # the matrix and b read, x written
        total["flops"] += 2.0 * (z + 5.0 * n) * _iterations(m, eps2)
    return total


def tolerance(case):
    """Two correct solves may stop an iteration apart, and then their x differ by about as much as
    each differs from x*: measured up to 1.8e-7 at eps2 = 1e-10 and 1.1e-5 at 1e-8 (relative
    2-norm; with the sums in another order and the same count, below 1e-10)."""
    if case["kind"] == "knn":
        return "exact"  # whole numbers
    if case["kind"] == "features":
        return {"rel": 1e-6}  # v, from single-precision iterations with double-accurate norms
    loose = case["kind"] == "serve" or case.get("eps2") == 1e-8
    return {"rel": 4e-5 if loose else 1e-6}


def exact(case, seed):
    """The x that b was made from: A x = b holds for it to the rounding of b.  Whole numbers and
    v (a ratio of single-precision residuals) have no 64-bit value of their own."""
    if case["kind"] in ("knn", "features"):
        return None
    none = {"status": None}
    if case["mode"] == "auto":
        none.update(cls=None, pdiam=None, v=None)
    if case["kind"] == "solve":
        return {"x": _star(size_of(case)[0], seed), **none}
    mats = _mix(case["count"], case["n_lo"], case["n_hi"], case["pick"])
    at, total = _slices(mats)
    x = torch.zeros(total, dtype=torch.float64, device=DEV)
    for i, (o, m) in enumerate(zip(at, mats)):
        n = size_of(m)[0]
        x[o:o + n] = _star(n, 1000 * (seed % 100000) + i)
    return {"x": x, **none}
