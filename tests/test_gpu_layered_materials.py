"""Objects of one shape and height but different materials in a stack.  Their global blocks are filled once
and copied, the material blocks are each object's own: Y11 and Y21 depend on an object's shape, its
material and its background layer alone, so they must equal those of the object by itself, and
L^A_m, L^phi_m, which do not depend on materials, those of equal objects.  FP64 fills in another
summation order: 1e-10 (the parity tests' bound of Y)."""
import numpy as np
import pytest

from workloads.meshes import icosphere, merge

pytestmark = pytest.mark.gpu

MATS = [(4.0, 1.0, 0.0, 0), (2.5, 1.0, 0.01, 0), (4.0, 1.0, 0.0, 0)]


@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-4)])
def test_equal_shapes_of_two_materials(prec, tol):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    parts = [icosphere(1, 0.05, (0.3 * i, 0.0, 0.15)) for i in range(3)]
    st = sldm.Stack([(1.0, 1.0, 0.0, 0.0)], z_top=0.0, bottom=sldm.BOTTOM_PEC)
    m = sldm.Mesh(*merge(*parts))
    op = sldm.Operator(m, st, MATS, 300e6, precision=prec)
    same = sldm.Operator(m, st, MATS[:1] * 3, 300e6, precision=prec)
    for b in (sldm.BLOCK_LAM, sldm.BLOCK_LPM):
        ref = same.block(b)
        assert np.max(np.abs(op.block(b) - ref)) <= tol * np.max(np.abs(ref))
    for o, (part, mat) in enumerate(zip(parts, MATS)):
        one = sldm.Operator(sldm.Mesh(*part), st, [mat], 300e6, precision=prec)
        for b in (sldm.BLOCK_K, sldm.BLOCK_Y11, sldm.BLOCK_Y21):
            # the scaling length of M_l is the mesh's mean edge, the same here for one and three
            ref = one.block(b)
            assert np.max(np.abs(op.block(b, o) - ref)) <= tol * np.max(np.abs(ref)), (o, b)
