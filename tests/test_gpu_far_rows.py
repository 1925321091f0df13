"""The far field of pair operators streams Y11 alone, once per pass: the matrix bytes its product counts."""
import numpy as np
import pytest

from workloads.meshes import cylinder_array, ellipsoid, icosphere, merge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["two", "cyl4"])
def test_bytes_of_the_far_field_product(which):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    if which == "two":
        xyz, tri, obj = merge(ellipsoid(2, (0.06, 0.04, 0.05)), icosphere(1, 0.05, (0.15, 0.02, 0.0)))
        mats, f = [(6.0, 1.0, 0.05), (2.5, 1.0, 0.0)], 500e6
    else:
        xyz, tri, obj = cylinder_array(2, 2, 120e-9, 300e-9, 500e-9)
        mats, f = [(6.0, 1.0, 0.0)] * 4, 299792458.0 / 1e-6
    op = sldm.Operator(sldm.Mesh(xyz, tri, obj), sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), mats, f, precision=sldm.PREC_F32X2)
    y11 = sum(8.0 * (3 * n // 2) ** 2 for n in np.bincount(obj))
    for nr in (1, 8, 9, 32):
        x = np.zeros((nr, op.N), complex)
        sldm.timers_reset()
        sldm.timers_enable(True)
        op.farfield_n(x, [0.3], 0.0, nr)
        sldm.timers_enable(False)
        tc = sldm.timers_read().get("gemm_tc", (0, 0))[1]
        assert sldm.timer_units("gemv_y") == y11 * (1 if tc else (nr + 7) // 8), (nr, tc)
