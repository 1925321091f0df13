"""The blocked LU of an object whose first panels are taller than a cluster's shared memory holds (above ~6,200 rows):
cooperative panels, then clusters.  Y formed by the FP64 LU against Y applied by inner solves, whose complex64
inverse comes from the same LU but whose result is M_l's own (refined to 1e-13): 1e-9, the
blocked LU's tolerance.  A wrong complex64 factor would not contract and Y would be formed there too."""
import pytest

from workloads.meshes import box

pytestmark = pytest.mark.gpu


def test_tall_panels():
    import torch
    from paper_2106_06184_gb300 import sldm
    v, f = box(0.2, 0.19, 0.05, 21, 21, 5, jitter=0.05, seed=4)
    m = sldm.Mesh(v, f)
    assert m.ne + m.nt - 1 > 6300
    st = sldm.Stack([(1.0, 1.0, 0.0, 0.0)])
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(2, m.n_unknowns, dtype=torch.complex128, device="cuda", generator=g)
    y = []
    for nested in (-1, 0):
        op = sldm.Operator(m, st, [(4.0, 1.0, 0.01)], 300e6, nested_min=nested)
        if nested == 0:
            with pytest.raises(sldm.SldmError) as e:
                op.block(sldm.BLOCK_Y11)
            assert e.value.code == sldm.ENOTSUP  # inner solves, not a formed Y
        y.append(op.apply(x, torch.empty_like(x), nrhs=2))
        op.close()
    d = y[0] - y[1]
    ne = m.ne
    for s in (slice(0, ne), slice(ne, 2 * ne), slice(2 * ne, None)):
        assert float(d[:, s].norm() / y[0][:, s].norm()) < 1e-9
