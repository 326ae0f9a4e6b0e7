"""The Python side of calls: sizes of field arrays."""
import ctypes as C

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


@pytest.mark.gpu
def test_fields_of_a_box_with_half_a_cell():
    import __graft_entry__

    __graft_entry__.build()
    g = B.Sim(length_lambda=20.5, cells_per_lambda=1.0, source_node=8)
    for comp in range(8):
        assert len(g.field(comp)) == (22 if comp in B.NODE_COMPONENTS else 21)
    g.close()
