"""Far field of operators held as complex64 pairs: its product with Y has a plan of its own, on the
tensor cores in TF32 form or on the CUDA cores.  Both against the complex128 operator's far field:
each product term is within 3 x 2^-22 (TF32 pairs) or 2^-24 of |Y||e|, so the currents, and twice
that the cross-sections, are within 4e-6 of their norm."""
import numpy as np
import pytest

from workloads.meshes import cylinder_array

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [0, 9, 33])
def test_far_field_of_pairs(policy):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    xyz, tri, obj = cylinder_array(3, 3, 120e-9, 300e-9, 500e-9)
    m = sldm.Mesh(xyz, tri, obj)
    st = sldm.Stack([(1.0, 1.0, 0.0, 0.0)])
    ops = []
    for prec, p in ((0, 0), (2, policy)):
        sldm.set_tc_policy(p)
        try:
            ops.append(sldm.Operator(m, st, [(6.0, 1.0, 0.0)] * 9, 299792458.0 / 1e-6, precision=prec))
        finally:
            sldm.set_tc_policy(0)
    rng = np.random.default_rng(3)
    ell = float(np.linalg.norm(xyz[tri[:, 0]] - xyz[tri[:, 1]], axis=1).mean())
    th = np.linspace(0.0, np.pi, 37)
    for nr in (1, 9, 12, 20, 32):
        x = rng.standard_normal((nr, ops[0].N)) + 1j * rng.standard_normal((nr, ops[0].N))
        x[:, : m.ne] /= ell
        ref, got = (op.farfield_n(np.ascontiguousarray(x), th, 0.4, nr) for op in ops)
        assert np.linalg.norm(got - ref) <= 4e-6 * np.linalg.norm(ref), nr
