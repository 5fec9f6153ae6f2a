"""What msat_create reads of the caller's arrays."""
import ctypes
import mmap

import numpy as np
import pytest

from synth import uniform_ksat

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


def _resident(buf, start, stop):
    """Pages of [start, stop) of a mapping that something has read or written."""
    libc = ctypes.CDLL(None, use_errno=True)
    base = ctypes.addressof(ctypes.c_char.from_buffer(buf))
    pages = (stop - start) // mmap.PAGESIZE
    vec = (ctypes.c_ubyte * pages)()
    assert libc.mincore(ctypes.c_void_p(base + start), ctypes.c_size_t(stop - start), vec) == 0, ctypes.get_errno()
    return sum(v & 1 for v in vec)


def test_no_literal_is_read_before_the_offsets_are_checked(pkg):
    """Offsets that decrease once and end far past the literals: refused
    without a look at what lies behind them.  The tail is a mapping that
    nothing has touched, so that a read of it shows in its residence (and
    stays inside the mapping)."""
    from paper_2402_03640_gb300 import MsatError
    cnf = uniform_ksat(60000, 258000, 3, seed=3)
    head, total = 8 << 20, 64 << 20
    assert 4 * cnf.lits.size <= head // 2
    buf = mmap.mmap(-1, total, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS)
    lits = np.frombuffer(buf, np.int32, count=total // 4)
    lits[:cnf.lits.size] = cnf.lits
    assert _resident(buf, head, total) == 0
    off = cnf.off.copy()
    off[100] = off[101] + 1
    off[-1] = total // 4
    with pytest.raises(MsatError) as e:
        pkg.Solver(cnf.n, off, lits, None, restarts=1)
    assert "non-decreasing at clause 100" in str(e.value)
    assert _resident(buf, head, total) == 0


def _route(s):
    r = ctypes.c_int32(-1)
    assert s._lib.msat_selftest_preparation(s._ctx, ctypes.byref(r)) == 0
    return {0: "host", 1: "device", 2: "host after device"}[r.value]


@pytest.mark.parametrize("what,want", [("clean", "device"), ("small", "host"), ("long", "host"), ("hot", "host"),
                                       ("doubled", "host"), ("one_doubled", "host after device"),
                                       ("just_past_a_warp", "host after device")])
def test_instances_for_the_host_are_seen_early(pkg, what, want):
    """A clause too long, variables in very many clauses and repeats in most
    clauses keep an instance off the device path before its literals are
    uploaded; a single repeat and a variable of 1025 occurrences are found
    there."""
    from synth import Cnf, zipf_weighted
    rng = np.random.default_rng(2)
    cnf = uniform_ksat(*((60000, 258000) if what != "small" else (300, 1290)), 3, seed=3)
    lits, off, w = cnf.lits.copy(), cnf.off, cnf.weights
    if what == "long":
        lits, off = np.concatenate([lits, np.arange(1, 34, dtype=np.int32)]), np.append(off, off[-1] + 33)
    elif what == "hot":
        z = zipf_weighted(20000, 60000, seed=4)
        assert np.bincount(np.abs(z.lits)).max() > 4096
        lits, off, w = z.lits, z.off, z.weights
    elif what == "doubled":
        lits[1::3] = lits[0::3]
    elif what == "one_doubled":
        lits[off[-2] + 1] = lits[off[-2]]
    elif what == "just_past_a_warp":
        cl = lits.reshape(-1, 3)
        have = (np.abs(cl) == 1).any(axis=1)
        add = rng.choice(np.flatnonzero(~have), size=1025 - have.sum(), replace=False)
        cl[add, 0] = 1
        assert (np.abs(lits) == 1).sum() == 1025
    n = z.n if what == "hot" else cnf.n
    with pkg.Solver(n, off, lits, w, restarts=1, lr=1e-2) as s:
        assert _route(s) == want
        a = rng.choice(np.array([-1, 1], np.int8), size=(n, 3))
        import torch
        got = s.evaluate(torch.from_numpy(a).cuda(), "sparse").cpu().numpy()
    clause = np.repeat(np.arange(off.size - 1), np.diff(off))
    for b in range(3):
        sat = np.bincount(clause[(a[np.abs(lits) - 1, b] > 0) == (lits > 0)], minlength=off.size - 1)
        assert got[b] == (np.ones(off.size - 1, np.int64) if w is None else w)[sat == 0].sum()


@pytest.mark.parametrize("m", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1])
@pytest.mark.parametrize("bad", ["first", "last", "wrap", "none"])
def test_offsets_on_both_sides_of_the_line(pkg, m, bad):
    """Offsets checked by the host (up to 2^17 clauses) and by the device: an
    offset that decreases, at the first clause, the last or by differences
    that are small modulo 2^64, is refused with the literals behind it
    untouched; without one the device prepares the instance."""
    from paper_2402_03640_gb300 import MsatError
    cnf = uniform_ksat(30000, m, 3, seed=3)
    off, total = cnf.off.copy(), 64 << 20
    buf = mmap.mmap(-1, total, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS)
    lits = np.frombuffer(buf, np.int32, count=total // 4)
    lits[:cnf.lits.size] = cnf.lits
    if bad == "none":
        with pkg.Solver(cnf.n, off, lits[:cnf.lits.size], None, restarts=1) as s:
            assert _route(s) == "device" and s.info()["uniform_len"] == 3
        return
    at = {"first": 0, "last": m - 1, "wrap": 1000}[bad]
    if bad == "first":
        off[1], off[2:] = -1, total // 4
        off[-1] = total // 4
    elif bad == "last":
        off[m - 1], off[m] = total // 4 + 1, total // 4
    else:
        off[at + 1:] = np.iinfo(np.int64).min + 3
        off[-1] = total // 4
    with pytest.raises(MsatError) as e:
        pkg.Solver(cnf.n, off, lits, None, restarts=1)
    assert "non-decreasing at clause %d" % at in str(e.value)
    assert _resident(buf, 8 << 20, total) == 0
