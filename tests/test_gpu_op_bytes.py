"""The device bytes that an operator states are those it holds: the library's count of all its buffers before
and after the assembly."""
import ctypes

import numpy as np
import pytest

from workloads.meshes import cylinder_array, icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("case", ["sphere", "array", "glass", "inner"])
def test_stated_bytes_are_held(case, prec):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    layers, mats, f, nested = [(1.0, 1.0, 0.0, 0.0)], [(4.0, 1.0, 0.0, 0)], 300e6, 0
    if case in ("sphere", "inner"):
        m = sldm.Mesh(*icosphere(2, 0.1))
        nested = 300 if case == "inner" else -1
    else:
        m = sldm.Mesh(*cylinder_array(2, 2, 120e-9, 300e-9, 500e-9))
        mats, f = [(6.0, 1.0, 0.0, 0)] * 4, 299792458.0 / 1e-6
        if case == "glass":
            layers = layers + [(2.25, 1.0, 0.0, 0.0)]
    st = sldm.Stack(layers)
    before = sldm.device_bytes()
    op = sldm.Operator(m, st, mats, f, precision=prec, nested_min=nested)
    assert op.device_bytes == sldm.device_bytes() - before
    b = op.rhs_planewave([0, 0, -1.0], [1.0, 0, 0], np.zeros(op.N, complex))
    op.solve(b, np.zeros_like(b), tol=1e-3)
    info = sldm.OpInfo()
    op.L.check(op.L.lib.sldm_op_info_get(op.h, ctypes.byref(info)))
    assert info.device_bytes == sldm.device_bytes() - before  # with the Krylov workspace
