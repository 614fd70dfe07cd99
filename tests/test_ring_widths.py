"""The SpMV of the grid-wide CG kernels at every row width it has a form for.

Widths 3..9 have unrolled forms for two adjacent slices and for one; other
widths and slices of unequal widths are summed in parts.  Two blocks give a
block many slices (pairs, an odd slice at the end, entries that cross into the
ring's next stage); 300 blocks, as many as the device takes, give it fewer
slices than warps.  Both column formats.  Against the oracle: counts within
2 % (at least 1), x within 1e-6."""
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


N = 4001  # 126 slices, the last one row


def _mixed():
    """Slice widths from 1 to past the layout's cap, changing from slice to slice."""
    rng = np.random.default_rng(3)
    ii, jj = [], []
    for s in range(0, N - 64, 32):
        w = int(rng.integers(0, 14))
        for r in range(32):
            if r % 3 == 0:
                ii += [s + r] * w
                jj += [s + r + 1 + k for k in range(w)]
    i, j = np.array(ii), np.array(jj)
    off = -np.ones(i.size)
    deg = np.bincount(i, minlength=N) + np.bincount(j, minlength=N)
    return synth.from_edges(N, i, j, off, deg + 0.5)


CASES = {f"band{2 * h + 1}": (lambda h=h: synth.banded(N, 2 * h + 1, 1.0, 1.1, seed=h)) for h in (1, 2, 3, 4, 5, 9)}
CASES.update({f"regular{d}": (lambda d=d: synth.random_regular_laplacian(N, d, 1e-2, seed=d)) for d in (3, 5, 7)})
CASES["mixed"] = _mixed
CASES["diagonal"] = lambda: synth.from_edges(N, np.zeros(0, int), np.zeros(0, int), np.zeros(0),
                                             np.linspace(1.0, 3.0, N))


@pytest.mark.parametrize("blocks", [2, 300])
@pytest.mark.parametrize("name", sorted(CASES))
def test_widths(mp, name, blocks):
    A = CASES[name]()
    _, b = synth.rhs(A, seed=2)
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    for kw in (dict(eps1=1e-4), dict(fp64_only=1)):
        if "eps1" in kw:
            xo, ro = oracle.solve(A, b, **kw)
        else:
            xo, it, st = oracle.cg64(A, b, 1e-10)
            ro = {"status": st, "n1": 0, "n2": it}
        got = []
        for variant in (0, 1):
            x, r = mp.solve(dA, db, grid_blocks=blocks, spmv_variant=variant, **kw)
            assert r["status"] == ro["status"]
            for k in ("n1", "n2"):
                assert abs(r[k] - ro[k]) <= max(1, int(0.02 * ro[k])), (k, r[k], ro[k])
            assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-6 * np.linalg.norm(xo)
            got.append(x)
        assert torch.equal(got[0], got[1])  # the column format does not change a bit
