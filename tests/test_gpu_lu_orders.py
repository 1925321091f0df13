"""The direct solver at orders around its changes of form (side-by-side kernel below
160, blocked form above, ragged last panels): Y11 and Y21 of single boxes against
the oracle's dense solve, at the blocked LU's tolerances (FP64 1e-9; complex64 5e-4)."""
import numpy as np
import pytest

from oracle import system as S
from oracle.topology import Mesh as OMesh
from workloads.meshes import box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [(2, 2, 2), (3, 2, 2), (4, 3, 3), (5, 4, 3)])
def test_orders(cells):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    v, f = box(0.2, 0.15, 0.1, *cells, jitter=0.05, seed=2)
    A = S.assemble(OMesh(v, f), [S.Material(4.0, 1.0, 0.01)], S.Material(), 300e6)
    for prec, tol in ((0, 1e-9), (1, 5e-4)):
        op = sldm.Operator(sldm.Mesh(v, f), sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.01)], 300e6, precision=prec)
        for got, ref in ((op.block(sldm.BLOCK_Y11, 0), A.blocks[0]["Y11"]), (op.block(sldm.BLOCK_Y21, 0), A.blocks[0]["Y21"])):
            assert np.max(np.abs(got - ref)) < tol * np.max(np.abs(ref))
