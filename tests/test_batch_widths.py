"""Systems of one plan block get one or both of its launch blocks by their rows
and by their share of the batch's work: both sides of the line in rows, a batch
of one, and a batch in which one system outweighs many equal ones, against the
CPU oracle and (many equal systems) against each other.  Systems of larger teams
whose 2BFS frontiers outgrow the one-block search, beside others."""
import numpy as np
import pytest

import oracle
import synth

from test_batch import mp, parity, run_batch, sample_over  # noqa: F401  (mp: the fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BATCHES = {
    "one": [synth.laplacian_2d(90, 71)],
    "line": [synth.path(2048), synth.path(2049), synth.laplacian_2d(32, 64), synth.laplacian_2d(3, 683)],
    "outweighed": [synth.laplacian_2d(120, 130)] + [synth.banded(300, 7, 0.6, 1.1, seed=s) for s in range(40)],
    # frontiers past the one-block search's limit in teams of 4 blocks and more, and one below it
    "scattered": [synth.random_regular_laplacian(20000, 8, 1e-2, seed=3), synth.random_tree_plus(14000, 0.5, 3.0, seed=3),
                  synth.random_regular_laplacian(9000, 6, 1e-2, seed=5), synth.laplacian_3d(20, sigma=1e-2),
                  synth.random_regular_laplacian(2400, 6, 1e-2, seed=5), synth.path(700)],
    "shared": [synth.laplacian_2d(50, 43, sigma=1e-3)] * 400,
}


@pytest.mark.parametrize("name", list(BATCHES))
@pytest.mark.parametrize("mode", ["auto", "fp64"])
def test_one_or_both_launch_blocks(mp, name, mode):
    mats = BATCHES[name]
    bs = [synth.rhs(A, seed=80 + (0 if name == "shared" else i))[1] for i, A in enumerate(mats)]
    feat, cls = sample_over(mats)
    S = mp.DeviceSample(feat, cls) if mode == "auto" else None
    kw = {"fp64_only": 1} if mode == "fp64" else {}
    xs, rs = run_batch(mp, mats, bs, S, team_rows=2048 if name == "scattered" else 16384, **kw)
    for i in range(1 if name == "shared" else len(mats)):
        A, b, x, r = mats[i], bs[i], xs[i], rs[i]
        assert r["team_blocks"] == 1 or name == "scattered"
        if mode == "fp64":
            xo, ro = oracle.solve(A, b, eps1=1.0)  # any start: the bars below do not depend on it
            assert r["status"] == 0 and r["true_rel_resid"] <= 1e-10
            assert np.linalg.norm(x - xo) <= 1e-6 * np.linalg.norm(xo)
        else:
            xo, ro = oracle.solve(A, b, S=(feat, cls))
            assert r["pdiam"] == ro["pdiam"] and r["cls"] == ro["cls"]
            parity(r, ro, x, xo)
    if name == "shared":  # one block each at first, both where a team of two takes one
        for x, r in zip(xs, rs):
            assert r["status"] == 0 and r["cls"] == rs[0]["cls"]
            assert np.linalg.norm(x - xs[0]) <= 1e-9 * np.linalg.norm(xs[0])
