"""The binding's C arrays of descriptors and integers: built in bulk, they take and refuse what building them
one by one takes and refuses."""
import ctypes
import types

import pytest

import paper_1412_0934_gb300 as hy


def _descriptors(struct, n):
    out = []
    for k in range(n):
        c = struct()
        c.nx, c.ny, c.nz, c.dx, c.level = 3 + k, 4 + k, 5 + k, 0.5 + k, k
        out.append(types.SimpleNamespace(c=c))
    return out


@pytest.mark.parametrize("n", [0, 1, 2, 5])
@pytest.mark.parametrize("struct", [hy.hydro_patch, hy.hydro_mhd_patch])
def test_descriptors_keep_their_values(struct, n):
    arr, count = hy._struct_array(struct, _descriptors(struct, n))
    assert count == n and len(arr) == n
    assert [(a.nx, a.ny, a.nz, a.dx, a.level) for a in arr] == [(3 + k, 4 + k, 5 + k, 0.5 + k, k) for k in range(n)]


@pytest.mark.parametrize("n", [1, 2, 5])
def test_descriptors_of_the_other_kind_are_refused(n):
    with pytest.raises(TypeError):
        hy._struct_array(hy.hydro_patch, _descriptors(hy.hydro_mhd_patch, n))
    with pytest.raises(TypeError):
        hy._struct_array(hy.hydro_mhd_patch, _descriptors(hy.hydro_patch, n))
    with pytest.raises(TypeError):
        hy._struct_array(hy.hydro_patch, _descriptors(hy.hydro_patch, n) + _descriptors(hy.hydro_mhd_patch, 1))


@pytest.mark.parametrize("convert", [list, tuple, iter, lambda r: map(float, r)])
@pytest.mark.parametrize("outer", [list, iter])
def test_integers_from_any_rows(convert, outer):
    """Rows may be iterators, and values anything int() takes."""
    rows = [(1, 2, 3), (4.0, 5, True), (7, 8.9, 2 ** 31)]
    got = hy._ints(outer([convert(r) for r in rows]))
    assert list(got) == [1, 2, 3, 4, 5, 1, 7, 8, ctypes.c_int(2 ** 31).value]
    assert list(hy._ints([])) == []
