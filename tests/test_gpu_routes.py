"""Forms of the device preparation and of the step kernels, each with a look at
which route ran: the two preparations of one instance agree bit for bit (the
host's is asked for by the same clauses with one literal written twice), and
the small-instance kernel's step loop follows the oracle."""
import ctypes

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


def _prep(s):
    r = ctypes.c_int32(-1)
    assert s._lib.msat_selftest_preparation(s._ctx, ctypes.byref(r)) == 0
    return {0: "host", 1: "device", 2: "host after device"}[r.value]


def _solo(s, steps):
    r = ctypes.c_int32(-1)
    assert s._lib.msat_selftest_step_route(s._ctx, steps, ctypes.byref(r)) == 0
    return bool(r.value)


def _varied(seed, n, m, lo, hi, weighted):
    """Clauses of lo..hi distinct variables: consecutive ones from a random
    start, so that none repeats."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(lo, hi + 1, size=m)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    start = np.repeat(rng.integers(0, n, size=m), lens)
    var = (start + (np.arange(off[-1]) - np.repeat(off[:-1], lens)) * 7919) % n
    lits = ((var + 1) * rng.choice([-1, 1], size=off[-1])).astype(np.int32)
    return Cnf(n, off, lits, rng.integers(1, 1 << 20, size=m) if weighted else None)


def _empties(n, m, empty):
    """3-literal clauses with empty ones among them, which no light block
    groups."""
    c = _varied(7, n, m, 3, 3, True)
    lens = np.full(m + empty, 3)
    lens[np.random.default_rng(8).choice(m + empty, size=empty, replace=False)] = 0
    return Cnf(n, np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), c.lits,
               np.random.default_rng(9).integers(1, 50, size=m + empty))


def _doubled(cnf):
    j = int(np.flatnonzero(np.diff(cnf.off))[-1])
    end = cnf.off[j + 1]
    off = cnf.off.copy()
    off[j + 1:] += 1
    return Cnf(cnf.n, off, np.insert(cnf.lits, end, cnf.lits[cnf.off[j]]).astype(np.int32), cnf.weights)


# B=64 and 128: the store's rows are grouped (m B floats above 32 MiB)
FORMS = {
    "k4_weighted_rows": (lambda: _varied(1, 30000, 140000, 4, 4, True), 64, "device"),
    "k2_rows": (lambda: _varied(2, 50000, 140001, 2, 2, False), 64, "device"),
    "varied_rows": (lambda: _varied(3, 30000, 140003, 1, 8, False), 64, "device"),
    "varied_weighted_rows": (lambda: _varied(4, 30000, 140003, 1, 8, True), 64, "device"),
    "a_group_at_its_limit": (lambda: _empties(30000, 130000, 4096), 64, "device"),
    "a_group_past_its_limit": (lambda: _empties(30000, 130000, 4097), 64, "host after device"),
    "varied_weighted": (lambda: _varied(5, 30000, 140003, 1, 32, True), 1, "device"),
}


@pytest.mark.parametrize("name", sorted(FORMS))
def test_device_preparation_of_each_form(pkg, name):
    import torch
    make, B, want = FORMS[name]
    cnf = make()
    a = torch.randint(0, 2, (cnf.n, 70), device="cuda", dtype=torch.int8) * 2 - 1
    got = []
    for c, route in ((cnf, want), (_doubled(cnf), "host after device")):
        with pkg.Solver.from_cnf(c, restarts=B, lr=1e-2) as s:
            assert _prep(s) == route
            loss, cost = s.step(3, per_pass=True)
            got.append((loss, cost, s.x(), *s.best(), s.evaluate(a, "sparse").cpu().numpy()))
    for u, v in zip(*got):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("name", ["k4_weighted_rows", "varied_weighted"])
def test_first_tensor_core_evaluation_of_a_device_prepared_instance(pkg, name):
    """Targets and clause lengths come from the device's clause list."""
    import torch
    make, _, _ = FORMS[name]
    cnf = make()
    a = torch.randint(0, 2, (cnf.n, 33), device="cuda", dtype=torch.int8) * 2 - 1
    with pkg.Solver.from_cnf(cnf, restarts=1) as s:
        assert _prep(s) == "device"
        dense = s.evaluate(a, "dense").cpu().numpy()
        assert np.array_equal(dense, s.evaluate(a, "sparse").cpu().numpy())
    x = a.cpu().numpy() > 0
    clause = np.repeat(np.arange(cnf.m), np.diff(cnf.off))
    for b in (0, 32):
        sat = np.bincount(clause[x[np.abs(cnf.lits) - 1, b] == (cnf.lits > 0)], minlength=cnf.m)
        assert dense[b] == cnf.weights[sat == 0].sum()


@pytest.mark.parametrize("name", ["k4_weighted_rows", "varied_weighted", "k3"])
def test_device_preparation_in_the_serving_engine(pkg, name):
    """The engine's contexts (from the stream-ordered pool, rows in clause
    order) give the best costs of the instance alone."""
    cnf = uniform_ksat(60000, 258000, 3, seed=2) if name == "k3" else FORMS[name][0]()
    with pkg.Solver.from_cnf(cnf, restarts=2, seed_x=4, lr=1e-4) as s:
        assert _prep(s) == "device"
        s.step(9)
        want = s.best()
    with pkg.Server(restarts=2, chunk=4) as srv:
        r = srv.wait(srv.submit(cnf, 9, seed_x=4), 300)
    assert np.array_equal(r["best_costs"], want[1])


def test_solo_kernel_with_signs_apart_over_two_waves(pkg, oracle):
    """3-literal clauses whose signed pairs do not fit, more restarts than
    multiprocessors, an odd number of steps in one call."""
    cnf = uniform_ksat(5000, 21500, 3, seed=7)
    B, S, lr = 256, 41, 2e-2
    ref = oracle.solve(cnf, B, 1, S, mode=oracle.MODE_F32, lr=lr)
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr) as s:
        assert _solo(s, S)
        _, cost = s.step(S, want_loss=False)
        x = s.x()
        assign, best = s.best()
        assert not _solo(s, 1)  # and on from there
        s.step(1, want_loss=False)
        with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr) as p:
            p.step(S + 1, want_loss=False, per_pass=True)
            assert np.array_equal(s.x(), p.x())
    assert np.array_equal(cost, ref["cost_hist"][S])
    assert np.array_equal(x.astype(np.float64), ref["x_final"])
    assert np.array_equal(best, ref["best_cost"]) and np.array_equal(assign, ref["best_assign"])


@pytest.mark.parametrize("k", [3, 4, 5])
@pytest.mark.parametrize("B,shape", [(1, {}), (2, {}), (4, {}), (8, dict(fwd_vw=8)), (64, dict(fwd_vw=4)),
                                     (512, dict(fwd_vw=8))])
def test_heavy_variable_of_several_chunks(pkg, oracle, k, B, shape):
    """One variable in every clause (three chunks of 1024 occurrences, the last
    one short) at every width of the passes and fixed clause length."""
    rng = np.random.default_rng(20 + k)
    m, n = 2099, 60
    rest = 1 + (rng.integers(0, n - 1, size=m)[:, None] + np.arange(k - 1) * 13) % (n - 1)
    lits = (np.concatenate([np.zeros((m, 1), np.int64), rest], 1) + 1) * rng.choice([-1, 1], size=(m, k))
    cnf = Cnf(n, np.arange(m + 1, dtype=np.int64) * k, lits.reshape(-1).astype(np.int32))
    S, lr = 5, 2e-2
    ref = oracle.solve(cnf, B, 1, S, mode=oracle.MODE_F32, lr=lr)
    with pkg.Solver.from_cnf(cnf, restarts=B, lr=lr, **shape) as s:
        assert s.info()["max_degree"] == m
        cost = [s.step(1, want_loss=False, per_pass=True)[1] for _ in range(S)]
        assert np.array_equal(np.stack(cost), ref["cost_hist"][1:])
        assert np.array_equal(s.x().astype(np.float64), ref["x_final"])


@pytest.mark.parametrize("make,B,solo", [(lambda: uniform_ksat(1200, 25200, 5, seed=1), 16, False),
                                         (lambda: zipf_weighted(3000, 15000, seed=1), 1, False),
                                         (lambda: uniform_ksat(800, 7900, 4, seed=1), 1024, True),
                                         (lambda: uniform_ksat(1000, 4300, 3, seed=1), 16, True)])
def test_route_of_an_evaluation_alone(pkg, make, B, solo):
    """A call without steps takes the route that its evaluation alone is faster
    on; both give the same costs and best assignments."""
    cnf = make()
    got = []
    for per_pass in (False, True):
        with pkg.Solver.from_cnf(cnf, restarts=B, lr=1e-2) as s:
            assert _solo(s, 0) == solo
            s.step(2, want_loss=False, per_pass=True)
            got.append((s.step(0, want_loss=False, per_pass=per_pass)[1], *s.best()))
    for u, v in zip(*got):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("B,want", [(1, "device"), (1024, "host")])
def test_instance_of_heavy_variables_is_prepared_by_the_host(pkg, B, want):
    """With grouped rows (B=1024) and an average variable past the light
    blocks' reach, nearly every clause has heavy variables alone."""
    import torch
    cnf = uniform_ksat(3000, 63000, 5, seed=1)
    a = np.random.default_rng(1).choice(np.array([-1, 1], np.int8), size=(cnf.n, 2))
    with pkg.Solver.from_cnf(cnf, restarts=B) as s:
        assert _prep(s) == want
        got = s.evaluate(torch.from_numpy(a).cuda(), "sparse").cpu().numpy()
    sat = ((a[np.abs(cnf.lits) - 1] > 0) == (cnf.lits > 0)[:, None]).reshape(cnf.m, 5, 2).any(axis=1)
    assert np.array_equal(got, (~sat).sum(axis=0))
