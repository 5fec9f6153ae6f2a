"""Device memory of the serving engine against its budget."""
import ctypes

import numpy as np
import pytest

from synth import uniform_ksat

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # cudaMemPoolAttr


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


class _Pool:
    """Use of the stream-ordered pool that the engine's contexts come from."""

    def __init__(self):
        import torch
        torch.cuda.init()
        self.rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def get(self, attr):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, USED_HIGH, ctypes.byref(v)) == 0


def _best(pkg, cnf, steps, B):
    with pkg.Solver.from_cnf(cnf, restarts=B, seed_x=3, lr=1e-4) as s:
        s.step(steps)
        return s.best()[1]


@pytest.mark.parametrize("what,budget", [("k5", 8_600_000), ("k5", 16 << 20), ("k3", 16 << 20)])
def test_budget_holds_while_a_request_is_prepared(pkg, what, budget):
    """One request alone never holds more of the pool than the budget.  k5:
    uploaded offsets and literals are more than the context of one restart
    (8.8 MB against 8.5), so under the smaller budget the host prepares it."""
    import torch
    cnf = uniform_ksat(8000, 168000, 5, seed=1) if what == "k5" else uniform_ksat(60000, 258000, 3, seed=2)
    pool = _Pool()
    with pkg.Server(restarts=1, hbm_budget=budget, chunk=10) as srv:
        torch.cuda.synchronize()
        base = pool.get(USED_CURRENT)
        pool.reset_high()
        r = srv.wait(srv.submit(cnf, 20, seed_x=3), 300)
        high = pool.get(USED_HIGH)
    assert r["status"] == 0
    assert high - base <= budget
    assert np.array_equal(r["best_costs"], _best(pkg, cnf, 20, 1))
