"""CPU-only: which combinations of precision, dimension, materials and solid
the library builds.  dfv_create_grid refuses a combination that is not built
before it looks at the workspace, so that a missing workspace tells the two
apart without a GPU."""
import ctypes
import itertools

import pytest

B = pytest.importorskip("paper_2111_11806_gb300.binding")

WORKSPACE, UNSUPPORTED = -5, -6


@pytest.fixture(scope="module")
def lib():
    from paper_2111_11806_gb300 import _build
    _build.build()
    B._lib = None
    return B.load()


@pytest.mark.parametrize("prec,dim,nmat,solid", list(itertools.product((B.DFV_FP64, B.DFV_FP32), (1, 2, 3), (1, 2, 3), (0, 1, 2))))
def test_only_the_documented_forms_are_refused(lib, prec, dim, nmat, solid):
    refused = dim == 3 and (solid != 0 or (prec == B.DFV_FP64 and nmat == 3))
    opt = B.dfv_options(nmat, solid, 1, 1.6, 0, 0, 0, 0, 0, 0, 0)
    lo, hi = (ctypes.c_double * 3)(0.0, 0.0, 0.0), (ctypes.c_double * 3)(1.0, 1.0, 1.0)
    dp = ctypes.POINTER(ctypes.c_double)
    out = ctypes.c_void_p()
    st = lib.dfv_create_grid(dim, (ctypes.c_int * 3)(8, 8, 8), ctypes.cast(lo, dp), ctypes.cast(hi, dp), None, prec,
                             ctypes.byref(opt), None, 0, None, ctypes.byref(out))
    assert st == (UNSUPPORTED if refused else WORKSPACE)
