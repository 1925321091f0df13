"""The bulk fill's use of symmetry: half of the pairs of a symmetric block, blocks
that are the transpose or the repeat of another, and tiles at the edges of their
sizes, against the oracle (which integrates every pair).  FP64: rounding, 1e-10;
FP32: the fill's stated 1e-5."""
import numpy as np
import pytest

from oracle import system as S
from oracle.topology import Mesh as OMesh
from workloads.meshes import box, ellipsoid, icosphere, merge

pytestmark = pytest.mark.gpu


def _check(xyz, tri, obj, mats, bg, freq, prec):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    A = S.assemble(OMesh(xyz, tri, obj), [S.Material(*m) for m in mats], S.Material(*bg), freq)
    op = sldm.Operator(sldm.Mesh(xyz, tri, obj), sldm.Stack([(*bg, 0.0)]), mats, freq, precision=prec)
    tol = 1e-10 if prec == sldm.PREC_F64 else 1e-5
    got = [(op.block(sldm.BLOCK_LAM), A.LAm), (op.block(sldm.BLOCK_LPM), A.LPm)]
    got += [(op.block(sldm.BLOCK_K, o), A.blocks[o]["K"]) for o in range(len(mats))]
    for g, r in got:
        assert np.max(np.abs(g - r)) < tol * np.max(np.abs(r))


@pytest.mark.parametrize("prec", [0, 1])
def test_transposed_and_repeated_blocks(prec):
    """Objects A, B, A at equal spacing in a lossy background: (A, A') repeats, (B, A)
    is the transpose of (A, B), which differ in size."""
    a = icosphere(1, 0.05)
    xyz, tri, obj = merge(a, ellipsoid(0, (0.05, 0.04, 0.03), (0.15, 0.02, 0.0)), (a[0] + [0.3, 0.0, 0.0], a[1]))
    _check(xyz, tri, obj, [(4.0, 1.0, 0.0), (2.5, 1.0, 0.03), (4.0, 1.0, 0.0)], (1.3, 1.0, 0.004), 500e6, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("cells", [(2, 1, 1), (4, 4, 2), (5, 4, 2)])
def test_tile_edges(cells, prec):
    """20, 128 and 152 triangles: less than a warp, exactly one and just over one
    tile of 128 sources."""
    v, f = box(0.1, 0.09, 0.05, *cells, jitter=0.05, seed=3)
    _check(v, f, None, [(3.0, 1.0, 0.01)], (1.0, 1.0, 0.0), 700e6, prec)
