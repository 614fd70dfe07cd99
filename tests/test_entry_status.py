"""A solve that is cancelled while its kernels start.

A block that already waits polls the caller's cancel word and sets the status,
while others of the same launch may still be reading it at their entry.  The
threads of a block must then agree on whether to leave: a barrier waits for
the warps that stay for ever if others have left.

The first test reads the kernels' source (CPU): in a kernel with block
barriers the status is read by one thread.  The second sets the word at
many moments after the call was enqueued, on every route of a solve: each
call ends as finished or cancelled, and the next one is right."""
import os
import re
import time

import pytest

import synth

torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_08059_gb300", "csrc")
NO_BARRIER = {"k_fill", "k_spmv", "k_knn"}  # straight through, or one warp


def kernels():
    """(file, name, body) of every kernel."""
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\) )?(\w+)\(", src):
            at = src.find("{", m.end())
            if at < 0 or ";" in src[m.end():at]:  # a declaration, or words of a comment
                continue
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield f, m.group(1), src[at:end]


def test_one_thread_reads_the_status():
    seen = set()
    for f, name, body in kernels():
        seen.add(name)
        depth = 0
        for line in body.splitlines():
            # (deeper down, the bounded waits of one lane read it)
            if "volatile_status(" in line and depth <= 2 and name not in NO_BARRIER:
                assert re.search(r"lead0|threadIdx\.x == 0|tid == 0", line), (f, name, line.strip())
            if name in NO_BARRIER:
                assert "__syncthreads" not in line and "bar.sync" not in line, (f, name)
            depth += line.count("{") - line.count("}")
    assert {"k_cg32", "k_cg64", "k_stage1", "k_cluster", "k_pdiam", "k_pdiam_block", "k_bfs1"} | NO_BARRIER <= seen


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_08059_gb300 import build, mpcg
    build.build()
    mpcg.load()
    return mpcg


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["auto", "eps1", "fp64"])
@pytest.mark.parametrize("route", ["cluster", "grid", "steps"])
def test_cancel_while_starting(mp, route, mode):
    A = synth.laplacian_2d(60, 55, sigma=1e-2)
    _, b = synth.rhs(A, seed=4)
    feat, cls = synth.random_sample(300, seed=2)
    S = mp.DeviceSample(feat, cls) if mode == "auto" else None
    kw = {"auto": {}, "eps1": dict(eps1=1e-5), "fp64": dict(fp64_only=1)}[mode]
    # the cluster kernel; the persistent grid; the grid with the method's steps as launches
    kw.update({"cluster": {}, "grid": dict(grid_blocks=4096), "steps": dict(precond=1)}[route])
    dA, db = mp.DeviceCSR.from_host(A), torch.from_numpy(b).cuda()
    word = torch.zeros(1, dtype=torch.int32, pin_memory=True)
    o = mp.options(cancel=word.data_ptr(), **kw)
    ws, x, res = mp.workspace(A.n, A.nnz, opts=o), torch.empty_like(db), mp.result_buffer(1)
    want, _ = mp.solve(dA, db, S, **kw)
    ended = set()
    for k in range(60):
        word.numpy()[0] = 0
        torch.cuda.synchronize()
        mp.solve_async(dA, db, x, o, ws, res, S)
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 5e-6 * k:
            pass
        word.numpy()[0] = 1
        torch.cuda.synchronize()
        st = mp.read_results(res)[0]["status"]
        assert st in (mp.OK, mp.WARN_EPS1_NOT_REACHED, mp.WARN_TRUE_RESID_RESTARTED, mp.ERR_CANCELLED), (k, st)
        ended.add(st)
    assert mp.ERR_CANCELLED in ended
    word.numpy()[0] = 0
    mp.solve_async(dA, db, x, o, ws, res, S)
    torch.cuda.synchronize()
    assert torch.equal(x, want)
