"""The largest mesh: the device's packed indices (4 x triangle + part, and the sign of an
edge's face) fit 32 bits below 2^29 triangles.  Only counts are looked at: the call with a
bad unit in it returns before it reads an array."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def pic():
    import paper_1701_03784_gb300 as pkg
    pkg.build()
    from paper_1701_03784_gb300 import pic as p
    return p


@pytest.mark.parametrize("n_tris,too_large", [(2 ** 29 - 1, False), (2 ** 29, True), (2 ** 30, True)])
def test_triangle_limit(pic, n_tris, too_large):
    a = np.zeros(8)
    u = pic.pic_units(-1.0, 1.0, 1.0, pic.PIC_FP32, 0)
    out = ctypes.c_void_p()
    p = pic._ptr(a)
    st = pic._lib.pic_mesh_create(p, 3, p, n_tris, p, p, 1, ctypes.byref(u), ctypes.byref(out))
    assert st == pic.PIC_ERR_ARG
    assert ("too large" in pic.pic_last_error()) == too_large
