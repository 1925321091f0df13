"""The refined solution of a complex64 operator solves the system of its stored blocks in FP64: with the
blocks copied out and the eliminated charge formed by B as the oracle does (B Y21's last row is minus
the sum of the others, exactly), the residual is the requested 1e-10 plus the product's 48 bits,
2^-44 of |Z| |x| with room for sums of a few hundred terms.  A last row stored in complex64
leaves 2^-25 of it instead."""
import copy

import numpy as np
import pytest

from oracle import system as S
from oracle.topology import Mesh as OMesh
from workloads.meshes import box, ellipsoid, merge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 12])
def test_residual_of_the_stored_blocks(nrhs):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    xyz, tri, obj = merge(box(0.1, 0.09, 0.05, 4, 3, 2, jitter=0.05, seed=5), ellipsoid(1, (0.05, 0.04, 0.03), (0.2, 0.0, 0.0)))
    mats, f = [(4.0, 1.0, 0.01), (2.0, 1.0, 0.0)], 500e6
    m = sldm.Mesh(xyz, tri, obj)
    op = sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), mats, f, precision=sldm.PREC_F32)
    A = copy.copy(S.assemble(OMesh(xyz, tri, obj), [S.Material(*mm) for mm in mats], S.Material(), f))
    A.LAm, A.LPm, A.Ix = op.block(sldm.BLOCK_LAM), op.block(sldm.BLOCK_LPM), op.block(sldm.BLOCK_IX)
    A.blocks = [dict(bl, LA=op.block(sldm.BLOCK_LA, o), LP=op.block(sldm.BLOCK_LP, o), K=op.block(sldm.BLOCK_K, o),
                     Y11=op.block(sldm.BLOCK_Y11, o), Y21=op.block(sldm.BLOCK_Y21, o)) for o, bl in enumerate(A.blocks)]
    Z = S.final_matrix(A)
    rng = np.random.default_rng(4)
    ell = float(np.linalg.norm(xyz[tri[:, 0]] - xyz[tri[:, 1]], axis=1).mean())
    dr = np.ones(op.N)
    dr[2 * op.ne:] = ell
    b = (rng.standard_normal((nrhs, op.N)) + 1j * rng.standard_normal((nrhs, op.N))) / dr
    x = np.zeros_like(b)
    info = op.solve(b, x, nrhs=nrhs, tol=1e-10)
    assert info["relres"] <= 1e-10
    for r in range(nrhs):
        bn = np.linalg.norm(dr * b[r])
        res = np.linalg.norm(dr * (b[r] - Z @ x[r])) / bn
        assert res <= 1e-10 + 2.0 ** -44 * np.linalg.norm(dr * (np.abs(Z) @ np.abs(x[r]))) / bn, (r, res)
