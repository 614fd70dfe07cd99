"""The one-block 2BFS of mpcg_pseudo_diameter and mpcg_features (GPU) against
the oracle: long thin graphs it finishes, graphs whose frontier grows past its
limits (the grid-wide search then does the work), the sizes at which its
limits change, disconnected graphs, rows past the sliced layout's cap, and
both column formats (columns further than 32,767 from their row)."""
import numpy as np
import pytest

import oracle
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


def _two(A, B):
    return synth.CSR(np.concatenate([A.row_ptr, A.nnz + B.row_ptr[1:]]).astype(np.int32),
                     np.concatenate([A.col, A.n + B.col]).astype(np.int32),
                     np.concatenate([A.val, B.val]))


def _lollipop(path, nx, ny):
    """A path into the corner of a grid and another path out of the opposite one."""
    a = np.arange(path - 1)
    g = np.arange(nx * ny).reshape(ny, nx) + path
    n = 2 * path + nx * ny
    i = np.concatenate([a, [path - 1], g[:, :-1].ravel(), g[:-1].ravel(), [g[-1, -1]], a + path + nx * ny])
    j = np.concatenate([a + 1, [g[0, 0]], g[:, 1:].ravel(), g[1:].ravel(), [path + nx * ny], a + path + nx * ny + 1])
    deg = np.bincount(i, minlength=n) + np.bincount(j, minlength=n)
    return synth.from_edges(n, i, j, -np.ones(i.size), deg + 0.1)


CASES = {
    "one": lambda: synth.laplacian_2d(1, 1),
    "path_3000": lambda: synth.path(3000),
    "thin_2000x40": lambda: synth.laplacian_2d(2000, 40),
    "thin_40x2000": lambda: synth.laplacian_2d(40, 2000),
    "square_128": lambda: synth.laplacian_2d(128, 128),        # n = 16384
    "square_130": lambda: synth.laplacian_2d(130, 130),        # past it
    "square_540": lambda: synth.laplacian_2d(540, 540),        # n = 291600
    "square_550": lambda: synth.laplacian_2d(550, 550),        # past the largest
    "cube_30": lambda: synth.laplacian_3d(30),                 # given up for the grid
    "star_5000": lambda: synth.star(5000, 1.1),                # a row past the width cap
    "rreg_40000": lambda: synth.random_regular_laplacian(40000, 8, 1e-3, seed=5),
    "band_20000": lambda: synth.banded(20000, 15, 0.6, 1.1, seed=7),
    "two_parts": lambda: _two(synth.laplacian_2d(300, 20), synth.laplacian_2d(50, 50)),
    "two_thin": lambda: _two(synth.laplacian_2d(20, 900), synth.laplacian_2d(20, 900)),
    "lone_first": lambda: _two(synth.laplacian_2d(1, 1), synth.laplacian_2d(30, 700)),  # vertex 0 by itself
    "lone_last": lambda: _two(synth.laplacian_2d(30, 700), synth.laplacian_2d(1, 1)),
    "forest": lambda: synth.banded(30000, 3, 0.9, 1.1, seed=3),
    # past the largest size, where the blocks search together: levels of one warp, also handed
    # back to the blocks for a wide middle part, and again to the warp
    "thin_20100x15": lambda: synth.laplacian_2d(20100, 15),
    "lollipop": lambda: _lollipop(2000, 600, 500),
    "no_edges": lambda: synth.banded(20000, 3, 0.0, 1.1, seed=3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_block_pdiam(mp, name):
    A = CASES[name]()
    dA = mp.DeviceCSR.from_host(A)
    want, t = oracle.pseudo_diameter(A, return_t=True)
    assert mp.pseudo_diameter(dA) == (want, t)
    _, b = synth.rhs(A, seed=3)
    db = torch.from_numpy(b).cuda()
    f = mp.features(dA, db)
    assert f["pdiam"] == want and f["status"] in (mp.OK, mp.WARN_EPS1_NOT_REACHED)
    # beside the iterations of a solve: the same search by the feature blocks
    feat, cls = synth.random_sample(60, seed=2)
    x, r = mp.solve(dA, db, mp.DeviceSample(feat, cls), max_it_fp64=1, max_true_restarts=0)
    assert r["pdiam"] == want
