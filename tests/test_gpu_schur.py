"""The preconditioner's inverted Schur complements: by FP64 LU (255 charges), by refined FP32 LU
(259 and more), and shared by repeated objects.  A wrong inverse leaves the solution right (GMRES
measures true residuals) but costs iterations: the preconditioned solve must take fewer than the
plain one, and with two copies of an object, far apart so that they hardly couple, at most a
few more than with one."""
import numpy as np
import pytest

from workloads.meshes import box, merge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("cells", [(4, 4, 6), (5, 5, 4), (9, 8, 7)])
def test_refined_inverse_preconditions(prec, cells):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    one = box(0.1, 0.09, 0.08, *cells)
    far = (one[0] + [40.0, 0.0, 0.0], one[1])
    iters = []
    for mesh, n in ((one, 1), (merge(one, far), 2)):
        xyz, tri = mesh[0], mesh[1]
        m = sldm.Mesh(xyz, tri, mesh[2] if n > 1 else None)
        op = sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.01)] * n, 300e6, precision=prec)
        b = op.rhs_planewave((0, 0, -1), (1, 0, 0), np.zeros(op.N, complex))
        x, x0 = np.zeros(op.N, complex), np.zeros(op.N, complex)
        it = op.solve(b, x, tol=1e-6)["iters"]
        plain = op.solve(b, x0, tol=1e-6, precond=False)["iters"]
        assert 0 < it < plain, (it, plain)
        assert np.linalg.norm(x - x0) <= 1e-2 * np.linalg.norm(x0)  # two residuals of 1e-6, condition below 10^4
        iters.append(it)
    assert iters[1] <= 1.5 * iters[0] + 5, iters
