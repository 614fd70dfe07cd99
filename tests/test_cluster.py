"""The cluster kernel (small systems) against the grid-wide kernels.

An explicit grid size keeps the grid-wide kernels, so the same call runs both
ways.  Sizes at the edges: one row, a ragged last slice, fewer slices than
blocks, one slice more than fills a block's 16 warps, every instance (rows
per thread), the largest size, and one past it (both calls then take the
grid), and matrices with scattered columns, which take it too.  The two ways sum the inner products in another order, so counts may
differ by 2 % (at least 1), x within the parity bar of 1e-6; l~, the class
and the status are equal."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_08059_gb300 import build, mpcg
    build.build()
    mpcg.load()
    return mpcg


def _grid(n):
    """A 2-D grid of n = nx * ny rows with the most square nx that divides n."""
    nx = next(k for k in range(int(n ** 0.5), 0, -1) if n % k == 0)
    return synth.laplacian_2d(n // nx, nx, sigma=1e-2)


def _two(n):
    """Two components (the per-component 2BFS)."""
    A, B = _grid(n), _grid(n // 2)
    return synth.CSR(np.concatenate([A.row_ptr, A.nnz + B.row_ptr[1:]]).astype(np.int32),
                     np.concatenate([A.col, A.n + B.col]).astype(np.int32),
                     np.concatenate([A.val, B.val]))


def _hubs(n, hubs, far=0):
    """Every vertex joined to one of the first `hubs` vertices, which form a chain; vertices past
    the hubs also to `far` others."""
    i = np.arange(hubs, n)
    c = np.arange(hubs - 1)
    a = [np.stack([i % hubs, i]), np.stack([c, c + 1])]
    for k in range(far):
        j = i + 37 * (k + 1)
        a.append(np.stack([i[j < n], j[j < n]]))
    e = np.unique(np.concatenate(a, 1), axis=1)
    deg = np.bincount(e[0], minlength=n) + np.bincount(e[1], minlength=n)
    off = -0.5 - np.random.default_rng(n).random(e.shape[1])
    return synth.from_edges(n, e[0], e[1], off, 2.0 * deg + 1.0)


CASES = {f"grid{n}": (lambda n=n: _grid(n)) for n in
         (1, 31, 33, 480, 512, 513, 8192, 8224, 16384, 16400, 32768, 39990, 40200)}
CASES.update({
    "star_1001": lambda: synth.star(1001, 1.1),          # one row past the width cap
    # long rows: one or two of a slice (summed by the warp), more (by their lanes, behind the
    # slices' entries or, without room there, from the CSR), and more entries than a count holds
    "star_12000": lambda: synth.star(12000, 3.0),
    "star_40000": lambda: synth.star(40000, 3.0),
    "hubs_2_4000": lambda: _hubs(4000, 2),
    "hubs_5_4000": lambda: _hubs(4000, 5, 1),
    "hubs_16_9000": lambda: _hubs(9000, 16),
    "hubs_70_9000": lambda: _hubs(9000, 70, 2),
    "hubs_400_30000": lambda: _hubs(30000, 400),
    "rtree_5000": lambda: synth.random_tree_plus(5000, 0.5, 1.1, seed=3),
    # whole copies of the gathered vector up to 4,096 rows, where columns are far away
    "rreg_300": lambda: synth.random_regular_laplacian(300, 6, 1e-2, seed=4),
    "rreg_4096": lambda: synth.random_regular_laplacian(4096, 8, 1e-3, seed=4),
    "rreg_4097": lambda: synth.random_regular_laplacian(4097, 8, 1e-3, seed=4),
    "rtree_3001": lambda: synth.random_tree_plus(3001, 0.5, 1.1, seed=8),
    "rreg_20000": lambda: synth.random_regular_laplacian(20000, 8, 1e-3, seed=4),  # columns far away
    "band_9000_b29": lambda: synth.banded(9000, 29, 0.6, 1.1, seed=7),
    "two_3000": lambda: _two(2000),
})
MODES = {"eps1": dict(eps1=1e-5), "auto": dict(), "fp64": dict(fp64_only=1)}


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("name", sorted(CASES))
def test_cluster_against_grid(mp, name, mode):
    A = CASES[name]()
    _, b = synth.rhs(A, seed=5)
    feat, cls = synth.random_sample(300, seed=2)
    S = mp.DeviceSample(feat, cls) if mode == "auto" else None
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    xc, rc = mp.solve(dA, db, S, **MODES[mode])
    xg, rg = mp.solve(dA, db, S, grid_blocks=4096, **MODES[mode])
    assert (rc["status"], rc["pdiam"], rc["cls"]) == (rg["status"], rg["pdiam"], rg["cls"]), (rc, rg)
    for k in ("n1", "n2"):
        assert abs(rc[k] - rg[k]) <= max(1, 0.02 * rg[k]), (k, rc[k], rg[k])
    assert rc["true_rel_resid"] <= 1e-10
    assert abs(rc["v"] - rg["v"]) <= 1e-9
    assert torch.linalg.vector_norm(xc - xg) <= 1e-6 * torch.linalg.vector_norm(xg)
    x2, r2 = mp.solve(dA, db, S, **MODES[mode])
    assert torch.equal(xc, x2)  # the sums have a fixed order


ROUTES = {  # past 4,096 rows: whether the cluster kernel runs the system
    "rreg_4097": (lambda: synth.random_regular_laplacian(4097, 8, 1e-3, seed=4), True),
    "rreg_12000": (lambda: synth.random_regular_laplacian(12000, 8, 1e-3, seed=4), False),
    "rreg_20000": (lambda: synth.random_regular_laplacian(20000, 8, 1e-3, seed=4), False),
    "rtree_9000": (lambda: synth.random_tree_plus(9000, 0.5, 3.0, seed=8), True),
    "rtree_36000": (lambda: synth.random_tree_plus(36000, 0.5, 3.0, seed=8), False),
    "grid_2000x15": (lambda: synth.laplacian_2d(2000, 15, sigma=1e-2), True),  # neighbours two blocks away
    "cube_30": (lambda: synth.laplacian_3d(30, sigma=1e-2), True),
}


@pytest.mark.parametrize("mode", ["eps1", "fp64", "auto"])
@pytest.mark.parametrize("name", sorted(ROUTES))
def test_scattered_columns_take_the_grid(mp, name, mode):
    """A matrix whose gathers are scattered over the cluster's blocks runs in the
    grid-wide kernels, which are then faster: x is theirs to the last bit (a call
    that asks for a grid as large as the device takes), where the cluster's sums
    have another order.  (Algorithm II has another grid then, so x is compared
    with the bars of the two ways.)"""
    make, cluster = ROUTES[name]
    A = make()
    _, b = synth.rhs(A, seed=5)
    feat, cls = synth.random_sample(300, seed=2)
    S = mp.DeviceSample(feat, cls) if mode == "auto" else None
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    x, r = mp.solve(dA, db, S, **MODES[mode])
    xg, rg = mp.solve(dA, db, S, grid_blocks=4096, **MODES[mode])
    assert r["status"] == rg["status"] and (r["cls"], r["pdiam"]) == (rg["cls"], rg["pdiam"])
    assert torch.linalg.vector_norm(x - xg) <= 1e-6 * torch.linalg.vector_norm(xg)
    if mode != "auto":
        assert torch.equal(x, xg) != cluster
    zero = torch.zeros_like(db)
    x, r = mp.solve(dA, zero, S, **MODES[mode])
    assert r["status"] == mp.OK and not x.any()


@pytest.mark.parametrize("mode", sorted(MODES))
def test_cluster_statuses(mp, mode):
    """b = 0, NaN in b, an indefinite matrix, a cap, a cancel word set, a broken CSR;
    in Algorithm II (the 2BFS cluster beside CG) also a label that is no class.
    Both ways end alike, and a call after them is right."""
    A = _grid(3000)
    _, b = synth.rhs(A, seed=5)
    feat, cls = synth.random_sample(300, seed=2)
    S = mp.DeviceSample(feat, cls) if mode == "auto" else None
    kw = dict(MODES[mode])
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    want, _ = mp.solve(dA, db, S, **kw)

    def both(A_, b_, S_=S, **more):
        r = mp.solve(A_, b_, S_, **kw, **more)[1]
        g = mp.solve(A_, b_, S_, grid_blocks=4096, **kw, **more)[1]
        assert r["status"] == g["status"], (r, g)
        return r, g

    x, r = mp.solve(dA, torch.zeros_like(db), S, **kw)
    assert r["status"] == mp.OK and not x.any()
    bad = db.clone()
    bad[1234] = float("nan")
    assert both(dA, bad)[0]["status"] == mp.ERR_NAN
    # d^T A d < 0 at the first iteration: in Algorithm II a breakdown in the k0 phase
    assert both(mp.DeviceCSR(dA.row_ptr, dA.col, -dA.val), db)[0]["status"] == mp.ERR_BREAKDOWN
    r, g = both(dA, db, max_it_fp64=3, max_it_fp32=2)
    assert r["status"] == mp.ERR_NOT_CONVERGED and r["n2"] == g["n2"] == 3 and r["n1"] == g["n1"]
    assert abs(r["true_rel_resid"] - g["true_rel_resid"]) <= 1e-6 * g["true_rel_resid"]
    word = torch.ones(1, dtype=torch.int32, pin_memory=True)
    assert both(dA, db, cancel=word.data_ptr())[0]["status"] == mp.ERR_CANCELLED
    col = dA.col.clone()
    col[0] = A.n
    assert both(mp.DeviceCSR(dA.row_ptr, col, dA.val), db)[0]["status"] == mp.ERR_INVALID_ARG
    if mode == "auto":
        for label in (-1, 16, 77):
            assert both(dA, db, mp.DeviceSample(feat, np.full_like(cls, label)))[0]["status"] == mp.ERR_INVALID_ARG
        mixed = cls.copy()
        mixed[::2] = 16  # valid classes are met before the vote finds the label
        assert both(dA, db, mp.DeviceSample(feat, mixed), knn_k=64)[0]["status"] == mp.ERR_INVALID_ARG
    assert torch.equal(mp.solve(dA, db, S, **kw)[0], want)


def test_label_wait_that_runs_out(mp):
    """Every class of the sample is met long before the 2BFS of a long path ends: CG
    waits for the label until its time limit, and the call ends with the status."""
    A = synth.path(30000)
    _, b = synth.rhs(A, seed=5)
    feat, _ = synth.random_sample(60, seed=2)
    S = mp.DeviceSample(feat, np.full(60, 1, np.int8))
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    for kw in (dict(), dict(grid_blocks=4096)):
        assert mp.solve(dA, db, S, timeout_ms=2, **kw)[1]["status"] == mp.ERR_TIMEOUT
    x, r = mp.solve(dA, db, S)
    assert r["status"] >= 0 and r["pdiam"] == A.n - 1
