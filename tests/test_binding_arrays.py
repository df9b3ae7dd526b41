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
