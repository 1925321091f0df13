"""FP64-accurate products of complex64 block pairs on the tensor cores (passes of up to 16
right-hand sides, here forced from 3 on) against the same operator assembled with the tensor
cores switched off.

Both compute with 48-bit operators and vectors; per 128-column segment the tensor-core form drops
what lies below 2^-54 of the segment's largest entries, the compensated sums what lies below
2^-48 of each product: 1e-12 of the largest result, as for the widths of the compensated product.
Scaling x by a power of ten moves only exponents."""
import pytest

from workloads.meshes import box, cylinder_array, ellipsoid, merge

pytestmark = pytest.mark.gpu

CASES = {
    "two": lambda: (*merge(box(0.1, 0.09, 0.05, 5, 4, 3, jitter=0.05, seed=5), ellipsoid(1, (0.05, 0.04, 0.03), (0.2, 0.0, 0.0))),
                    [(4.0, 1.0, 0.01), (2.0, 1.0, 0.0)], 500e6),
    "cyl9": lambda: (*cylinder_array(3, 3, 120e-9, 300e-9, 500e-9), [(6.0, 1.0, 0.0)] * 9, 299792458.0 / 1e-6),
}


@pytest.mark.parametrize("name", ["two", "cyl9"])
@pytest.mark.parametrize("scale", [1.0, 1e22, 1e-22])
def test_tensor_cores_match_cuda_cores(name, scale):
    import torch
    from paper_2106_06184_gb300 import sldm
    xyz, tri, obj, mats, f = CASES[name]()
    m = sldm.Mesh(xyz, tri, obj)
    ops = []
    for policy in (3, 33):
        sldm.set_tc_policy(policy)
        try:
            ops.append(sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), mats, f, precision=2))
        finally:
            sldm.set_tc_policy(0)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = scale * torch.randn(32, ops[0].N, dtype=torch.complex128, device="cuda", generator=g)
    for n in (3, 13, 16, 18, 32):  # 18: 16 and 2 on the CUDA cores
        y = [op.apply(x[:n].contiguous(), torch.empty(n, op.N, dtype=torch.complex128, device="cuda"), nrhs=n) for op in ops]
        d = float((y[0] - y[1]).abs().max() / y[1].abs().max())
        assert 0.0 < d < 1e-12, (n, d)   # 0 would mean that one kernel computed both
