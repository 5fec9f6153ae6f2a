"""Calls that keep device scratch with the context: several streams and
threads, against numpy."""
import threading

import numpy as np
import pytest

from synth import uniform_ksat, zipf_weighted

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2402_03640_gb300 as p
    from paper_2402_03640_gb300 import build
    build.build()
    p.load()
    return p


def costs(cnf, a):
    """Costs of a int8 [n][nb] (true where > 0)."""
    w = np.ones(cnf.m, np.int64) if cnf.weights is None else cnf.weights
    clause = np.repeat(np.arange(cnf.m), np.diff(cnf.off))
    out = np.empty(a.shape[1], np.int64)
    for b in range(a.shape[1]):
        true = (a[np.abs(cnf.lits) - 1, b] > 0) == (cnf.lits > 0)
        out[b] = w[np.bincount(clause[true], minlength=cnf.m) == 0].sum()
    return out


@pytest.fixture(scope="module")
def batches():
    """An instance past the direct kernel's range and two batches of different
    sizes with their costs."""
    import torch
    cnf = zipf_weighted(30011, 200003, seed=6)
    rng = np.random.default_rng(7)
    a = [rng.choice(np.array([-1, 1], np.int8), size=(cnf.n, nb)) for nb in (64, 130)]
    return cnf, [torch.from_numpy(x).cuda() for x in a], [costs(cnf, x) for x in a]


def test_evaluations_on_two_streams(pkg, batches):
    """Each call on another stream than the one before: a packed batch is not
    overwritten while the call before still reads it."""
    import torch
    cnf, dev, want = batches
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        torch.cuda.synchronize()
        got = []
        for r in range(40):
            s.set_stream(streams[r & 1])
            got.append(s.evaluate(dev[r & 1], "sparse"))
        torch.cuda.synchronize()
        for r, g in enumerate(got):
            assert np.array_equal(g.cpu().numpy(), want[r & 1]), r


def test_evaluations_from_two_threads(pkg, batches):
    import torch
    cnf, dev, want = batches
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        torch.cuda.synchronize()
        got = [[], []]

        def work(t):
            for _ in range(100):
                got[t].append(s.evaluate(dev[t], "sparse"))

        threads = [threading.Thread(target=work, args=(t,)) for t in (0, 1)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        for t in (0, 1):
            assert len(got[t]) == 100
            assert all(np.array_equal(g.cpu().numpy(), want[t]) for g in got[t])


def test_captured_evaluation_holds_no_allocation(pkg, batches):
    """A graph with a captured evaluation can have two instances at a time,
    and both give the batch's costs."""
    import ctypes

    import torch
    cnf, dev, want = batches
    st = torch.cuda.Stream()
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    raw = ctypes.c_void_p(st.cuda_stream)
    with pkg.Solver.from_cnf(cnf, restarts=1, stream=st) as s:
        out = torch.empty(dev[0].shape[1], dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        graph, execs = ctypes.c_void_p(), [ctypes.c_void_p(), ctypes.c_void_p()]
        assert rt.cudaStreamBeginCapture(raw, 1) == 0  # this thread's calls
        rc = s._lib.msat_evaluate(s._ctx, ctypes.c_void_p(dev[0].data_ptr()), dev[0].shape[1],
                                  ctypes.c_void_p(out.data_ptr()), 0)
        assert rt.cudaStreamEndCapture(raw, ctypes.byref(graph)) == 0 and rc == 0
        for e in execs:
            assert rt.cudaGraphInstantiate(ctypes.byref(e), graph, ctypes.c_ulonglong(0)) == 0
        for e in execs:
            out.fill_(-1)
            torch.cuda.synchronize()
            assert rt.cudaGraphLaunch(e, raw) == 0
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), want[0])
        for e in execs:
            rt.cudaGraphExecDestroy(e)
        rt.cudaGraphDestroy(graph)


def test_captured_evaluation_of_very_many_assignments(pkg):
    """Past one launch's range of the kernel without scratch."""
    import torch
    from synth import Cnf
    cnf = Cnf.from_clauses(3, [[1, 2], [-1, 3], [-2, -3]], weights=[5, 1 << 33, 7])
    nb = 65535 * 32 + 33
    rng = np.random.default_rng(8)
    a = rng.choice(np.array([-1, 1], np.int8), size=(3, nb))
    t = a > 0
    want = 5 * ~(t[0] | t[1]) + (1 << 33) * ~(~t[0] | t[2]) + 7 * ~(~t[1] | ~t[2])
    dev = torch.from_numpy(a).cuda()
    st = torch.cuda.Stream()
    with pkg.Solver.from_cnf(cnf, restarts=1, stream=st) as s:
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=st):
            out = s.evaluate(dev, "sparse")
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
        out = s.evaluate(dev, "sparse")
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)


def test_evaluation_past_a_launch_of_packed_groups(pkg):
    """More groups of 128 assignments than a launch takes."""
    import torch
    from synth import Cnf
    cnf = Cnf.from_clauses(2, [[1, 2], [-1], [1, -2]], weights=[5, 3, 1 << 33])
    nb = 65535 * 128 + 129
    a = torch.randint(0, 2, (2, nb), device="cuda", dtype=torch.int8) * 2 - 1
    t = a > 0
    want = 5 * (~(t[0] | t[1])).long() + 3 * t[0].long() + (1 << 33) * (~t[0] & t[1]).long()
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        assert torch.equal(s.evaluate(a, "sparse"), want)


def test_evaluation_without_scratch(pkg, batches):
    """Where the packed batch cannot be allocated, 128 assignments' worth of
    it, and where that cannot be had the kernel without scratch, give the same
    costs."""
    cnf, dev, want = batches
    group = 16 * cnf.n  # bytes of 128 packed assignments
    with pkg.Solver.from_cnf(cnf, restarts=2) as s:
        for limit in (0, group - 1, group, -1):
            assert s._lib.msat_selftest_scratch_limit(s._ctx, limit) == 0
            for a, w in zip(dev, want):
                assert np.array_equal(s.evaluate(a, "sparse").cpu().numpy(), w), limit
        s._lib.msat_selftest_scratch_limit(s._ctx, 0)
        x = s.x()
        assert np.array_equal(s.evaluate_x("sparse").cpu().numpy(), costs(cnf, np.where(x > 0, 1, -1)))


def test_growing_scratch_does_not_wait_for_the_stream(pkg, batches):
    """The first evaluation of a context and one with a larger batch return
    while earlier work of their stream still runs."""
    import torch
    cnf, dev, want = batches
    st = torch.cuda.Stream()
    for rep in range(2):  # the first round loads the kernels
        with pkg.Solver.from_cnf(cnf, restarts=1, stream=st) as s, torch.cuda.stream(st):
            torch.cuda.synchronize()
            torch.cuda._sleep(400_000_000)  # about 0.2 s
            busy = torch.cuda.Event()
            busy.record(st)
            got = [s.evaluate(a, "sparse") for a in dev]
            waited = busy.query()
            torch.cuda.synchronize()
            assert all(np.array_equal(g.cpu().numpy(), w) for g, w in zip(got, want))
    assert not waited


def test_scratch_is_reported(pkg, batches):
    """msat_info counts the packed batch among the device memory held."""
    cnf, dev, _ = batches
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        b0 = s.info()["device_bytes"]
        for a in dev:
            words = (a.shape[1] + 31) // 32
            words = (words + 3) // 4 * 4 if a.shape[1] > 64 else words
            s.evaluate(a, "sparse")
            assert s.info()["device_bytes"] == b0 + 4 * words * cnf.n


@pytest.mark.parametrize("how", ["stream", "thread"])
def test_best_beside_running_steps(pkg, how):
    """Reading the best assignments while steps of the context run on another
    stream, or are issued by another thread, leaves the trajectory as it is."""
    import torch
    cnf = uniform_ksat(3001, 12907, 3, seed=11)
    B, steps, lr = 64, 2001, 1e-2
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr) as s:
        s.step(steps, want_loss=False, per_pass=True)
        want = s.x()
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr) as s:
        s.best()  # loads the kernel
        calls = 0
        if how == "stream":
            a, b = torch.cuda.Stream(), torch.cuda.Stream()
            s.set_stream(a)
            s.step_async(steps, per_pass=True)
            s.set_stream(b)
            while not a.query():
                s.best()
                calls += 1
            s.set_stream(a)
        else:
            def work():
                for _ in range(steps):
                    s.step_async(1, final_eval=False, per_pass=True)
                s.step_async(0, per_pass=True)
            t = threading.Thread(target=work)
            t.start()
            while t.is_alive():
                s.best()
                calls += 1
            t.join()
        torch.cuda.synchronize()
        assert calls > 3
        assert np.array_equal(s.x(), want)


def test_best_without_scratch(pkg):
    """Where the transposed copy cannot be allocated the host transposes."""
    cnf = uniform_ksat(1501, 6000, 3, seed=6)
    with pkg.Solver.from_cnf(cnf, restarts=64, lr=1e-2) as s:
        s.step(3, per_pass=True)
        want = s.get_state()["best_assign"].T
        for limit in (0, cnf.n * 64 - 1, -1):
            s._lib.msat_selftest_scratch_limit(s._ctx, limit)
            assert np.array_equal(s.best()[0], want), limit


@pytest.mark.parametrize("call", ["msat_get_x", "msat_best", "msat_get_state"])
def test_a_refused_copy_leaves_the_array_alone(pkg, call):
    """A call that cannot copy (its stream is being captured) gives an error
    and has not written to the caller's array."""
    import ctypes

    import torch
    cnf = uniform_ksat(300000, 1000, 3, seed=5)
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    st = torch.cuda.Stream()
    raw = ctypes.c_void_p(st.cuda_stream)
    with pkg.Solver.from_cnf(cnf, restarts=4, stream=st) as s:
        a = np.full(4 * cnf.n * (1 if call == "msat_best" else 4), 0x5a, np.uint8)
        args = {"msat_get_x": (a.ctypes.data,), "msat_best": (a.ctypes.data, None),
                "msat_get_state": (a.ctypes.data, None, None, None, None, None, None)}[call]
        fn = getattr(s._lib, call)
        torch.cuda.synchronize()
        graph = ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(raw, 1) == 0  # this thread's calls
        rc = fn(s._ctx, *(None if v is None else ctypes.c_void_p(v) for v in args))
        rt.cudaStreamEndCapture(raw, ctypes.byref(graph))
        rt.cudaGetLastError()
        if graph.value:
            rt.cudaGraphDestroy(graph)
        assert rc != 0
        assert (a == 0x5a).all()
        assert s.x().shape[0] == cnf.n  # and the context goes on
