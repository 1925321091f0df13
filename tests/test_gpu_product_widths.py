"""Products of every count of right-hand sides against the same columns one at a
time: each count up to 8 has a kernel of its own in FP64 and in the compensated
product, larger ones run as passes of 8 and a rest.  The two orders of summation
over N ~ 10^3 terms differ by at most N x 2^-53 ~ 1e-13 of sum |a||x| (FP64), and
the compensated sums carry 2^-48 (4e-15) per operation: 1e-12."""
import numpy as np
import pytest

from workloads.meshes import box, ellipsoid, merge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(0, 1e-13), (2, 1e-12)])
def test_every_width(prec, tol):
    import torch
    from paper_2106_06184_gb300 import sldm
    xyz, tri, obj = merge(box(0.1, 0.09, 0.05, 5, 4, 3, jitter=0.05, seed=5), ellipsoid(1, (0.05, 0.04, 0.03), (0.2, 0.0, 0.0)))
    m = sldm.Mesh(xyz, tri, obj)
    op = sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.01), (2.0, 1.0, 0.0)], 500e6, precision=prec)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(21, op.N, dtype=torch.complex128, device="cuda", generator=g)
    one = torch.stack([op.apply(x[i].contiguous(), torch.empty_like(x[i])) for i in range(21)])
    for n in (2, 3, 4, 5, 6, 7, 8, 9, 13, 16, 21):
        y = op.apply(x[:n].contiguous(), torch.empty(n, op.N, dtype=torch.complex128, device="cuda"), nrhs=n)
        assert float((y - one[:n]).abs().max() / one[:n].abs().max()) < tol, n
