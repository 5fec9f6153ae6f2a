"""The one-block-per-restart kernel at the edges of its slices, list layouts
and sums: bit-exact trajectories against the FP32-mode oracle, continued on
the per-pass kernels."""
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


def _mixed(seed, n, m, lo, hi, w_max=0):
    """Clauses of lo..hi literals (repeats and x-or-not-x clauses among them)."""
    rng = np.random.default_rng(seed)
    cl = [((rng.integers(0, n, size=k) + 1) * rng.choice([-1, 1], size=k)).tolist()
          for k in rng.integers(lo, hi + 1, size=m)]
    w = rng.integers(1, w_max, size=m) if w_max else None
    return Cnf.from_clauses(n, cl, weights=w)


CASES = {
    "one_clause": lambda: (uniform_ksat(3, 1, 3, seed=1), 1),
    "slice_less_one": lambda: (uniform_ksat(31, 31, 3, seed=2), 2),
    "slice_full": lambda: (uniform_ksat(32, 32, 3, seed=3), 2),
    "slice_plus_one": lambda: (uniform_ksat(33, 33, 3, seed=4), 4),
    "two_blocks_an_sm": lambda: (uniform_ksat(301, 1290, 3, seed=5), 256),
    "lists_in_l2": lambda: (uniform_ksat(2500, 10750, 3, seed=6), 2),
    "signs_apart": lambda: (uniform_ksat(5000, 21500, 3, seed=7), 1),
    "k5": lambda: (uniform_ksat(97, 2067, 5, seed=8), 4),
    "mixed": lambda: (_mixed(9, 61, 500, 0, 9), 2),
    "units_64bit_weights": lambda: (_mixed(10, 40, 300, 1, 4, w_max=1 << 40), 2),
    "long_weighted": lambda: (_mixed(11, 300, 400, 20, 90, w_max=50), 2),
    "many_leaves": lambda: (uniform_ksat(12, 9000, 3, seed=12), 1),
    "skewed": lambda: (zipf_weighted(900, 4100, seed=13), 4),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_solo_kernel_matches_oracle(pkg, oracle, name):
    cnf, B = CASES[name]()
    S, lr = 40, 2e-2
    ref = oracle.solve(cnf, B, 1, S + 3, mode=oracle.MODE_F32, lr=lr)
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr) as s:
        assert s.info()["small_kernel"] == 1
        # 33 steps cross a chunk of the Adam scalars; the cost after each call
        # is that of the final x
        _, c0 = s.step(0, want_loss=False)
        _, c1 = s.step(33, want_loss=False)
        _, c2 = s.step(7, want_loss=False)
        _, c3 = s.step(3, want_loss=False, per_pass=True)
        x = s.x()
        assign, best = s.best()
        assert s.info()["steps_done"] == S + 3
    assert np.array_equal(np.stack([c0, c1, c2, c3]), ref["cost_hist"][[0, 33, 40, 43]])
    assert np.array_equal(x.astype(np.float64), ref["x_final"])
    assert np.array_equal(best, ref["best_cost"]) and np.array_equal(assign, ref["best_assign"])


def test_solo_kernel_keeps_nan_in_its_restart(pkg):
    """A NaN in one restart's x stays in that variable: its clauses add
    nothing, as on the per-pass kernels."""
    cnf = uniform_ksat(60, 240, 3, seed=14)
    out = []
    for per_pass in (False, True):
        with pkg.Solver.from_cnf(cnf, restarts=2, lr=1e-2) as s:
            st = s.get_state()
            st["x"][7, 0] = np.nan
            st["x"][9, 1] = 0.0
            st["x"][11, 1] = -0.0
            s.set_state(st)
            _, cost = s.step(20, want_loss=False, per_pass=per_pass)
            out.append((cost, s.x(), s.best()[1]))
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("k", [3, 4, 5])
@pytest.mark.parametrize("B,shape", [(1, {}), (2, {}), (4, {}), (8, dict(fwd_vw=8)), (64, dict(fwd_vw=4)),
                                     (512, dict(fwd_vw=8))])
def test_clause_pass_of_fixed_lengths(pkg, oracle, k, B, shape):
    """The per-pass kernels on k-literal clauses for every width of the clause
    pass, with a variable of several chunks among the heavy ones."""
    cnf = uniform_ksat(60, 701, k, seed=15 + k)
    S, lr = 6, 2e-2
    ref = oracle.solve(cnf, B, 1, S, mode=oracle.MODE_F32, lr=lr)
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr, heavy_deg=8, **shape) as s:
        cost = [s.step(1, want_loss=False, per_pass=True)[1] for _ in range(S)]
        assert np.array_equal(np.stack(cost), ref["cost_hist"][1:])
        assert np.array_equal(s.x().astype(np.float64), ref["x_final"])


def test_heavy_variable_of_many_chunks(pkg, oracle):
    """A variable of more than 128 chunks of 1024 occurrences (several rounds
    of the chunk tree) and one of exactly 32 chunks."""
    rng = np.random.default_rng(16)
    m, n = 140001, 40
    a = np.where(np.arange(m) < 32 * 1024, 2, 3 + rng.integers(0, n - 3, size=m))
    lits = np.stack([np.full(m, 1), a, 3 + (a - 2 + rng.integers(0, n - 3, size=m)) % (n - 3)], 1)
    lits = lits * rng.choice([-1, 1], size=lits.shape)
    cnf = Cnf(n, np.arange(m + 1, dtype=np.int64) * 3, lits.reshape(-1).astype(np.int32))
    for B in (1, 8):
        ref = oracle.solve(cnf, B, 1, 3, mode=oracle.MODE_F32, lr=1e-2)
        with pkg.Solver.from_cnf(cnf, restarts=B, lr=1e-2) as s:
            assert s.info()["max_degree"] > 128 * 1024
            s.step(3, want_loss=False, want_cost=False, per_pass=True)
            assert np.array_equal(s.x().astype(np.float64), ref["x_final"])


@pytest.mark.parametrize("B", [1, 2, 8])
def test_nan_in_x_adds_nothing_on_the_per_pass_kernels(pkg, B):
    """A NaN in x: with stored w*f the clauses that hold it contribute nothing
    to the gradient of their other variables, which stay finite."""
    cnf = uniform_ksat(60, 240, 3, seed=14)
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=1e-2, f_mode="store") as s:
        st = s.get_state()
        st["x"][7, 0] = np.nan
        s.set_state(st)
        s.step(1, want_loss=False, per_pass=True)
        assert np.isfinite(np.delete(s.x(), 7, axis=0)).all()
