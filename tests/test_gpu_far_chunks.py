"""Far field of many directions (taken in chunks) and of every width of the groups of currents
against one direction and one current at a time: the same products, summed in the same order
of triangles, so equal to FP64 rounding of sums of ~10^4 terms: 1e-12 of the largest."""
import numpy as np
import pytest

from workloads.meshes import box, icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layered", [False, True])
@pytest.mark.parametrize("mesh,n", [("sphere", 1), ("sphere", 300), ("box", 700)])
def test_chunks_and_groups(layered, mesh, n):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    v, f = icosphere(0, 0.05) if mesh == "sphere" else box(0.1, 0.09, 0.08, 9, 8, 7)
    m = sldm.Mesh(v, f, None)
    layers = [(1.0, 1.0, 0.0, 0.0), (2.25, 1.0, 0.0, 0.0)] if layered else [(1.0, 1.0, 0.0, 0.0)]
    st = sldm.Stack(layers, z_top=float(v[:, 2].min()) - 0.05)
    op = sldm.Operator(m, st, [(4.0, 1.0, 0.0, 0)], 300e6)
    rng = np.random.default_rng(2)
    x = rng.standard_normal((9, op.N)) + 1j * rng.standard_normal((9, op.N))
    th = np.linspace(0.01, 1.5 if layered else 3.1, n)
    ph = np.linspace(0, 6, n)
    got = op.farfield_n(x, th, ph, 9)
    for a in {0, n // 2, n - 1}:
        for r in (0, 7, 8):
            ref = op.farfield(np.ascontiguousarray(x[r]), th[a:a + 1], ph[a:a + 1])[0]
            assert abs(got[r, a] - ref) <= 1e-12 * got[r].max(), (a, r)
