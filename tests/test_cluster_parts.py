"""The two clusters of a small Algorithm II solve.

CG may wait for the label, which only the 2BFS of the other cluster leads to,
and nothing orders the two clusters of a launch.  So the parts go by the order
in which they begin, not by their place in the grid (read from the source, on
the CPU), and solves of many threads, each on its own stream, all end with
what each gives alone (GPU)."""
import os
import re
import threading

import pytest

import synth

torch = pytest.importorskip("torch")

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_08059_gb300", "csrc",
                   "cluster.cu")


def test_no_part_goes_by_the_place_in_the_grid():
    src = open(SRC).read()
    src = src[src.index("void cl_bfs("):src.index("// Host")]
    assert not re.search(r"blockIdx\.x\s*([<>]|[=!]=)", src)
    assert "atomicAdd(&ctl->cl_begun, 1) == 0 ? kClPartBfs" in src


@pytest.mark.gpu
def test_many_streams():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_08059_gb300 import build, mpcg
    build.build()
    mpcg.load()
    feat, cls = synth.random_sample(300, seed=2)
    S = mpcg.DeviceSample(feat, cls)
    mats = [synth.laplacian_2d(40 + 7 * k, 30 + 3 * k, sigma=1e-2) for k in range(6)]
    mats += [synth.random_tree_plus(701, 0.5, 1.1, seed=3), synth.path(900)]
    dev = [(mpcg.DeviceCSR.from_host(A), torch.from_numpy(synth.rhs(A, seed=6)[1]).cuda()) for A in mats]
    want = [mpcg.solve(A, b, S) for A, b in dev]
    o = mpcg.options()
    got = [None] * len(dev)

    def work(k):
        A, b = dev[k]
        st = torch.cuda.Stream()
        ws, res = mpcg.workspace(A.n, A.nnz), mpcg.result_buffer(1)
        xs = [torch.empty_like(b) for _ in range(8)]
        st.wait_stream(torch.cuda.default_stream())
        for x in xs:
            mpcg.solve_async(A, b, x, o, ws, res, S, stream=st)
        st.synchronize()
        got[k] = xs, mpcg.read_results(res)[0]

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(dev))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (xw, rw), (xs, r) in zip(want, got):
        assert (r["status"], r["cls"], r["n1"], r["n2"], r["pdiam"]) == (rw["status"], rw["cls"], rw["n1"], rw["n2"], rw["pdiam"])
        assert all(torch.equal(x, xw) for x in xs)
