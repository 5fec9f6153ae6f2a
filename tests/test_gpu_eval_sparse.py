"""The clause-list evaluation of packed batches: exact costs at the edges of
its words, groups and weight bits, against numpy."""
import numpy as np
import pytest

from synth import Cnf, uniform_ksat, zipf_weighted

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


def _want(cnf, a):
    """Costs of a int8 [n][nb] (true where > 0)."""
    w = np.ones(cnf.m, np.int64) if cnf.weights is None else cnf.weights
    clause = np.repeat(np.arange(cnf.m), np.diff(cnf.off))
    cost = np.empty(a.shape[1], np.int64)
    for b in range(a.shape[1]):
        true = (a[np.abs(cnf.lits) - 1, b] > 0) == (cnf.lits > 0)
        cost[b] = w[np.bincount(clause[true], minlength=cnf.m) == 0].sum()
    return cost


def _instance(name):
    rng = np.random.default_rng(3)
    if name == "k3":
        return uniform_ksat(97, 417, 3, seed=1)
    if name == "k3_packed":  # one assignment is already past the direct kernel's range
        return uniform_ksat(9001, 400003, 3, seed=1)
    if name == "zipf":
        return zipf_weighted(150, 700, seed=2)
    if name == "zipf_packed":
        return zipf_weighted(30001, 300011, seed=2)
    count = 180000 if name == "wide_packed" else 190
    lens = np.concatenate([rng.integers(0, 12, size=count), [70, 33, 1]])
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    lits = ((rng.integers(0, 40, size=off[-1]) + 1) * rng.choice([-1, 1], size=off[-1])).astype(np.int32)
    w = rng.integers(1, 1 << 44, size=lens.size) if name.startswith("wide") else None
    return Cnf(40, off, lits, w)


SMALL = [(name, nb) for name in ("k3", "zipf", "mixed", "wide_weights") for nb in (1, 31, 32, 33, 64, 65, 129, 300)]
PACKED = [(name, nb) for name in ("wide_packed", "k3_packed", "zipf_packed") for nb in (1, 33, 64, 100, 130)]


@pytest.mark.parametrize("name,nb", SMALL + PACKED)
def test_packed_batch_costs(pkg, name, nb):
    import torch
    cnf = _instance(name)
    rng = np.random.default_rng(nb)
    a = rng.choice(np.array([-128, -1, 0, 1, 127], np.int8), size=(cnf.n, nb))  # any value > 0 is true
    want = _want(cnf, a)
    dev = torch.from_numpy(a).cuda()
    with pkg.Solver.from_cnf(cnf, restarts=4) as s:
        assert np.array_equal(s.evaluate(dev, "sparse").cpu().numpy(), want)
        assert np.array_equal(s.evaluate(dev[:, :1], "sparse").cpu().numpy(), want[:1])
        # the rounded x of the solver itself
        assert np.array_equal(s.evaluate_x("sparse").cpu().numpy(), _want(cnf, np.where(s.x() > 0, 1, -1)))


def test_captured_evaluation_outlives_the_buffer(pkg):
    """A captured evaluation replays correctly after a larger batch has
    replaced the context's own buffer, and needs no call before the capture."""
    import torch
    cnf = uniform_ksat(600, 90000, 3, seed=4)
    rng = np.random.default_rng(5)
    a = torch.from_numpy(rng.choice(np.array([-1, 1], np.int8), size=(cnf.n, 40))).cuda()
    big = torch.from_numpy(rng.choice(np.array([-1, 1], np.int8), size=(cnf.n, 500))).cuda()
    cap = torch.cuda.Stream()
    with pkg.Solver.from_cnf(cnf, restarts=1, stream=cap) as s:
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=cap):
            out = s.evaluate(a, "sparse")
        torch.cuda.synchronize()
        got = s.evaluate(big, "sparse")
        torch.cuda.synchronize()
        assert np.array_equal(got.cpu().numpy(), _want(cnf, big.cpu().numpy()))
        for _ in range(2):
            g.replay()
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), _want(cnf, a.cpu().numpy()))


@pytest.mark.parametrize("count", [1, 300, 30000, 330000])
@pytest.mark.parametrize("nb", [1, 33, 65, 130])
def test_long_clauses_are_read_by_the_warp(pkg, count, nb):
    """Clauses at the edges of 32 literals and of the warp's batches of 128,
    alone and among short and empty ones, for one to 32 clauses a warp."""
    import torch
    rng = np.random.default_rng(count + nb)
    n = 5000
    lens = rng.integers(0, 4, size=count)
    at = rng.choice(count, size=min(count, 40), replace=False)
    lens[at] = rng.choice([32, 33, 64, 65, 127, 128, 129, 160, 161, 4000], size=at.size)
    lens[at[0]] = 129
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    lits = ((rng.integers(0, n, size=off[-1]) + 1) * rng.choice([-1, 1], size=off[-1])).astype(np.int32)
    a = rng.choice(np.array([-1, 1], np.int8), size=(n, nb))
    # long clauses that one assignment leaves unsat, and some with one true literal
    for i, j in enumerate(at):
        lits[off[j]:off[j + 1]] = np.abs(lits[off[j]:off[j + 1]]) * -a[np.abs(lits[off[j]:off[j + 1]]) - 1, i % nb]
        if i % 3 == 1:
            k = off[j] + rng.integers(lens[j])
            lits[k] = -lits[k]
    for w in (None, rng.integers(1, 1 << 40, size=count)):
        cnf = Cnf(n, off, lits, w)
        with pkg.Solver.from_cnf(cnf, restarts=1) as s:
            got = s.evaluate(torch.from_numpy(a).cuda(), "sparse").cpu().numpy()
        assert np.array_equal(got, _want(cnf, a))
