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
