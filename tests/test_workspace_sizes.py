"""Caller-owned workspaces: the sizes that a caller may have fixed stay enough."""
import ctypes

import pytest

FORMS = ("fp64", "fp64tc", "tf32", "bf16x3", "bf16x6")
# (d, D, chi, Lx, Ly): bytes by form, as first published
SIZES = {
    (8, 2, 16, 2, 2): (9278976, 91330048, 81401344, 81434112, 78304768),
    (8, 3, 27, 2, 2): (80783104, 281474304, 198454016, 198486784, 173614848),
    (8, 4, 53, 2, 1): (812147456, 2262643456, 1420104448, 1423807232, 1177219840),
    (8, 5, 100, 2, 2): (6605875456, 17814526208, 11107250432, 11117768960, 9161636096),
    (1, 2, 100, 1, 1): (54487552, 159114752, 177529856, 179397632, 194104832),
    (1, 1, 200, 1, 1): (33044992, 116756992, 120208384, 121289728, 125241856),
}


@pytest.mark.parametrize("cell", sorted(SIZES))
@pytest.mark.parametrize("budget", [40, 64])
def test_workspace_is_no_larger_than_it_was(cell, budget):
    from paper_1711_04798_gb300 import binding as b
    lib = b.load_library()
    d, D, chi, lx, ly = cell
    for form, size in zip(FORMS, SIZES[cell]):
        c = b.Cell()
        c.Lx, c.Ly = lx, ly
        for i in range(lx * ly):
            c.pattern[i] = i
        c.n_tensors, c.d, c.D, c.dtype = lx * ly, d, D, 1
        ptrs = (ctypes.c_void_p * 4)(1, 1, 1, 1)
        c.tensors = ctypes.cast(ptrs, ctypes.POINTER(ctypes.c_void_p))
        opt = b._make_options(lib, chi, form, jacobi_max_sweeps=budget)
        n = ctypes.c_size_t()
        assert lib.ipeps_ctm_workspace_size(ctypes.byref(c), ctypes.byref(opt), ctypes.byref(n)) == 0
        assert n.value <= size, (form, n.value, size)
