"""The Python side of calls: sizes of field arrays and conversion of electron cases."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1008_1685_gb300 import binding as B


@pytest.mark.parametrize("cells", [20, 21])
@pytest.mark.parametrize("comp", range(8))
def test_field_takes_the_library_s_size(cells, comp):
    """A box of 20.5 cells: 21 in the library (halves away from zero), 20 by round()."""
    want = np.arange(cells + 1 if comp in B.NODE_COMPONENTS else cells, dtype=float)

    def call(c, cap, ptr, n):
        C.cast(n, C.POINTER(C.c_int64))[0] = len(want)
        if c != comp or cap < len(want):
            return -1
        C.memmove(ptr, want.ctypes.data, want.nbytes)
        return 0

    def check(rc):
        if rc:
            raise B.PicError(rc, "output too small")

    assert np.array_equal(B._field(call, check, 20, comp), want)
    if cells == 20:  # a refusal for another reason stays one
        with pytest.raises(B.PicError):
            B._field(lambda *a: -1, check, 20, comp)


def case(**kw):
    return dict(dict(wave=0, a0=1.0, tau=2.0, x0=3.0, p0=(4.0, 5.0, 6.0)), **kw)


@pytest.mark.parametrize("bad", [dict(a0=None), dict(tau=None), dict(x0=None), dict(p0=(1.0, None, 2.0)), dict(wave=None),
                                 dict(a0=np.timedelta64(5, "s")), dict(p0={1.0, 2.0, 3.0}), dict(p0=(1.0, 2.0)),
                                 dict(a0=1j)])
def test_electron_cases_refuse_what_is_no_number(bad):
    with pytest.raises((TypeError, IndexError)):
        B._electron_cases([case(), case(**bad), case()])


def test_electron_cases_keep_their_values():
    odd = [case(p0=[1, 2.5, np.float32(3)]), case(p0=np.arange(3)), case(p0={0: 7.0, 1: 8.0, 2: 9.0}), case(p0=(1, 2, 3, 4)),
           case(a0="1.5", wave="2"), {"wave": 1.9, "a0": True, "p0": (0, 0, 0)}, case(wave=2**32 + 1)]
    for cases in ([], odd, [case(a0=k / 7, wave=k % 3) for k in range(50)], *[[c] for c in odd]):
        got = B._electron_cases(cases)
        assert len(got) == max(1, len(cases))
        for a, c in zip(got, cases):
            assert (a["wave"], a["a0"], a["tau"], a["x0"]) == (int(c["wave"]) % 2**32, float(c["a0"]), c.get("tau", 0.0), c.get("x0", 0.0))
            assert list(a["p0"]) == [float(c["p0"][j]) for j in range(3)]


def test_electron_scan_reports_a_lack_of_host_memory():
    """An allocation that fails in the library comes back as an error of the call."""
    from paper_1008_1685_gb300 import build

    build.build()
    code = """
import resource
import numpy as np
from paper_1008_1685_gb300 import binding as B
L, n = B.library(), 1 << 22
cases, out = np.zeros(n, np.dtype(B.ElectronCase)), np.zeros(5)
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (4 << 20), resource.RLIM_INFINITY))
print(L.pic_electron_scan(cases.ctypes.data, n, 1, 0, 0.01, 0, 1, 0.8, 0, out.ctypes.data, 0))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(B.__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True)
    assert (r.returncode, r.stdout.strip()) == (0, "-3"), r.stderr  # PIC_ERR_OOM


@pytest.mark.gpu
def test_fields_of_a_box_with_half_a_cell():
    import __graft_entry__

    __graft_entry__.build()
    g = B.Sim(length_lambda=20.5, cells_per_lambda=1.0, source_node=8)
    for comp in range(8):
        assert len(g.field(comp)) == (22 if comp in B.NODE_COMPONENTS else 21)
    g.close()
