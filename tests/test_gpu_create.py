"""Instances prepared on the device: the same results, bit for bit, as the
host path (taken by the same clauses with one literal written twice), against
the oracle, and the same errors."""
import numpy as np
import pytest

from synth import Cnf, uniform_ksat

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


def _distinct(rng, n, lens, hot=0, p_hot=0.0):
    """Clauses of distinct variables; variables below `hot` are drawn with
    probability p_hot, so that they have some hundred occurrences."""
    out = []
    for k in lens:
        v = set()
        while len(v) < k:
            v.add(int(rng.integers(hot)) if hot and rng.random() < p_hot else int(rng.integers(n)))
        out.append([(x + 1) * int(rng.choice([-1, 1])) for x in v])
    return out


def _mixed(seed):
    rng = np.random.default_rng(seed)
    n, m = 40000, 130000
    cl = _distinct(rng, n, rng.integers(0, 9, size=m), hot=60, p_hot=0.08)
    cl.append([int(v) + 1 for v in range(0, 64, 2)])  # 32 literals
    return Cnf.from_clauses(n, cl, weights=rng.integers(1, 1 << 30, size=len(cl)))


def _doubled(cnf):
    """The same clauses with the first literal of the last one written twice."""
    lits = np.concatenate([cnf.lits, cnf.lits[cnf.off[-2]:cnf.off[-2] + 1]])
    off = cnf.off.copy()
    off[-1] += 1
    return Cnf(cnf.n, off, lits.astype(np.int32), cnf.weights)


@pytest.mark.parametrize("maker,B", [("k3_small", 1), ("k3", 1), ("k3", 64), ("mixed", 2), ("mixed", 128)])
def test_device_and_host_preparation_agree(pkg, oracle, maker, B):
    """B=64 and 128 have the store's rows grouped by block."""
    import torch
    cnf = _mixed(4) if maker == "mixed" else uniform_ksat(*((60000, 258000) if maker == "k3" else (12000, 51600)), 3, seed=3)
    deg = np.bincount(np.abs(cnf.lits) - 1, minlength=cnf.n)
    assert maker != "mixed" or 33 < deg.max() <= 1024
    a = torch.randint(0, 2, (cnf.n, 5), device="cuda", dtype=torch.int8) * 2 - 1
    got = []
    for c in (cnf, _doubled(cnf)):
        with pkg.Solver.from_cnf(c, restarts=B, lr=1e-2) as s:
            loss, cost = s.step(5, per_pass=True)
            info = s.info()
            got.append((loss, cost, s.x(), *s.best(), s.evaluate(a, "sparse").cpu().numpy(), info))
    for u, v in zip(got[0][:-1], got[1][:-1]):
        assert np.array_equal(u, v)
    assert got[0][-1] == got[1][-1]
    if B <= 2:
        ref = oracle.solve(cnf, B, 1, 5, mode=oracle.MODE_F32, lr=1e-2)
        assert np.array_equal(got[0][2].astype(np.float64), ref["x_final"])
        assert np.array_equal(got[0][3], ref["best_assign"]) and np.array_equal(got[0][4], ref["best_cost"])


def test_large_malformed_instances_are_refused(pkg):
    from paper_2402_03640_gb300 import MsatError
    cnf = uniform_ksat(60000, 258000, 3, seed=3)
    for what in ("zero", "range", "offsets", "weight"):
        lits, off = cnf.lits.copy(), cnf.off.copy()
        w = np.ones(cnf.m, np.int64)
        if what == "zero":
            lits[1234] = 0
        elif what == "range":
            lits[5] = cnf.n + 1
        elif what == "offsets":
            off[100] = off[101] + 1
        else:
            w[77] = 0
        with pytest.raises(MsatError) as e:
            pkg.Solver(cnf.n, off, lits, w, restarts=1)
        want = {"zero": "position 1234", "range": "position 5", "offsets": "non-decreasing", "weight": "clause 77"}[what]
        assert want in str(e.value)


def test_best_assignments_of_large_batches(pkg):
    """The transposed best assignments equal the state's, before and after an
    odd number of steps."""
    cnf = uniform_ksat(1501, 6000, 3, seed=6)
    with pkg.Solver.from_cnf(cnf, restarts=64, lr=1e-2) as s:
        for k in (0, 1, 4):
            s.step(k, per_pass=True)
            x = s.x()
            assign, _ = s.best()
            assert np.array_equal(assign, s.get_state()["best_assign"].T)
            assert np.array_equal(s.x(), x)
            s.step(1, per_pass=True)
