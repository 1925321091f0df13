"""A tensor-core product whose bounded wait runs out (here its flag, set after the product by
sldm_test_inject) is reported by the call that waits for that product, once, and the operator stays usable: products
and far fields of complex64 and pair operators, with host memory at once and with device memory at
the next call that waits."""
import numpy as np
import pytest

from workloads.meshes import icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2])
def test_a_lost_wait_is_reported_once(prec):
    import torch
    from paper_2106_06184_gb300 import sldm
    sldm.set_tc_policy(9)
    try:
        op = sldm.Operator(sldm.Mesh(*icosphere(2, 0.1)), sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.0)], 300e6, precision=prec)
    finally:
        sldm.set_tc_policy(0)
    rng = np.random.default_rng(1)
    x = rng.standard_normal((12, op.N)) + 1j * rng.standard_normal((12, op.N))
    y = np.zeros_like(x)
    th = np.linspace(0, 3, 4)
    dx, dy = torch.from_numpy(x).cuda(), torch.zeros(x.shape, dtype=torch.complex128, device="cuda")
    calls = {"apply": lambda: op.apply(x, y, nrhs=12), "farfield": lambda: op.farfield_n(x, th, 0.0, 12),
             "solve": lambda: op.solve(x, y, nrhs=12, tol=1e-4)}
    for name, call in calls.items():
        sldm.test_inject(sldm.INJECT_TC_WAIT, 1)
        try:
            with pytest.raises(sldm.SldmError) as e:
                call()
            assert e.value.code == sldm.ETIMEOUT, name
        finally:
            sldm.test_inject(sldm.INJECT_TC_WAIT, 0)
        call()  # reported once
    ref = op.apply(x, y, nrhs=12).copy()
    sldm.test_inject(sldm.INJECT_TC_WAIT, 2)  # both products of a call that does not wait
    try:
        op.apply(dx, dy, nrhs=12)
    finally:
        sldm.test_inject(sldm.INJECT_TC_WAIT, 0)
    with pytest.raises(sldm.SldmError) as e:
        op.farfield_n(x, th, 0.0, 12)
    assert e.value.code == sldm.ETIMEOUT
    op.farfield_n(x, th, 0.0, 12)
    assert np.array_equal(op.apply(x, y, nrhs=12), ref)
