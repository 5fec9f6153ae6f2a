"""Calls that keep device scratch with the context: several streams and
threads, against numpy."""
import threading

import numpy as np
import pytest

from synth import zipf_weighted

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
