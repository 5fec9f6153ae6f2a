"""The loss and cost of msat_forward on both of its routes (the clause pass's
last block up to 8 restarts, a reduction of its own above and where a thread
takes 8 restarts), and the clause-list evaluation on both sides of the direct
kernel's line, against numpy in 64 bits."""
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


def _want(cnf, x):
    w = np.ones(cnf.m) if cnf.weights is None else np.asarray(cnf.weights, np.float64)
    clause = np.repeat(np.arange(cnf.m), np.diff(cnf.off))
    lit = np.asarray(cnf.lits)
    loss, cost = [], []
    for b in range(x.shape[1]):
        xv = x[np.abs(lit) - 1, b].astype(np.float64)
        t = np.sign(lit) * np.tanh(xv)
        f = np.bincount(clause, weights=t, minlength=cnf.m)
        u = w * (np.bincount(clause[(xv > 0) == (lit > 0)], minlength=cnf.m) == 0)
        loss.append((u * f * f).sum() / max(u.sum(), 1.0))
        cost.append(int(u.sum()))
    return np.array(loss), np.array(cost)


@pytest.mark.parametrize("B,shape", [(1, {}), (2, {}), (4, {}), (8, {}), (8, {"fwd_vw": 8}), (8, {"fwd_vw": 1}), (16, {})])
@pytest.mark.parametrize("name", ["k3", "zipf", "k3_many"])
def test_forward_loss_and_cost(pkg, name, B, shape):
    import torch
    cnf = {"k3": lambda: uniform_ksat(301, 1291, 3, seed=2), "zipf": lambda: zipf_weighted(777, 3001, seed=3),
           "k3_many": lambda: uniform_ksat(60001, 258007, 3, seed=4)}[name]()
    x = np.random.default_rng(B).uniform(-1, 1, size=(cnf.n, B)).astype(np.float32)
    x[0, :] = 0.0
    loss, cost = _want(cnf, x)
    with pkg.Solver.from_cnf(cnf, restarts=B, **shape) as s:
        for _ in range(2):  # the counters are left as the next call needs them
            got, gc = s.forward(torch.from_numpy(x).cuda())
            assert np.array_equal(gc.cpu().numpy(), cost)
            # every term is >= 0: a term's relative error is twice that of f
            # (tanh 2 ulp, at most 19 additions of one sign) and a product's,
            # the sums before the two-word chain add a few tens of roundings
            assert np.abs(got.cpu().numpy().astype(np.float64) / loss - 1).max() < 96 * 2.0 ** -24


@pytest.mark.parametrize("m,nb", [(32768, 1), (32768, 32), (32768, 33), (32769, 1), (32769, 32), (16384, 64), (16385, 64)])
def test_evaluation_at_the_direct_line(pkg, m, nb):
    import torch
    cnf = uniform_ksat(3001, m, 3, seed=5)
    a = np.random.default_rng(nb).choice(np.array([-1, 1], np.int8), size=(cnf.n, nb))
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        assert np.array_equal(s.evaluate(torch.from_numpy(a).cuda(), "sparse").cpu().numpy(), _want(cnf, a)[1])
