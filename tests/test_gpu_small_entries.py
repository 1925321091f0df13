"""Tensor-core products of rows whose entries span many orders: unit vectors pick single entries of K, which
fall to 10^-7 of their neighbours' within a 64-column segment.  The scaled FP16 pairs keep 22 bits of an entry down to
2^-29 of its segment's largest and 2^-51 of that largest below, so with factors of two for the
roundings a column of the product is within 2^-21 of each entry plus 2^-50 of the segment's largest."""
import numpy as np
import pytest

from workloads.meshes import box

pytestmark = pytest.mark.gpu


def test_unit_vectors_return_the_entries():
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    v, f = box(0.4, 0.03, 0.02, 24, 2, 2, jitter=0.05, seed=3)
    m = sldm.Mesh(v, f)
    sldm.set_tc_policy(9)
    try:
        op = sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.5)], 2e9, precision=sldm.PREC_F32)
    finally:
        sldm.set_tc_policy(0)
    K = op.block(sldm.BLOCK_K)
    ne = op.ne
    seg = np.abs(np.pad(K, ((0, 0), (0, -ne % 64)))).reshape(ne, -1, 64).max(2)
    small = 0
    for c0 in range(0, ne, 32):
        cols = np.arange(c0, min(ne, c0 + 32))
        x = np.zeros((32, op.N), complex)
        x[np.arange(len(cols)), ne + cols] = 1.0
        y = op.apply(x, np.zeros_like(x), nrhs=32)[: len(cols), ne:2 * ne].T  # row block 2: -K e
        a, top = K[:, cols], seg[:, cols // 64]
        small += int(np.sum((np.abs(a) > 0) & (np.abs(a) < 2.0 ** -18 * top)))
        err = np.maximum(np.abs((y + a).real), np.abs((y + a).imag))
        lim = 2.0 ** -21 * np.abs(a) + 2.0 ** -50 * top
        assert np.all(err <= lim), (c0, np.max(err / lim))
    assert small > 100  # the case has such entries
