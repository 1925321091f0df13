"""The preconditioner's inverse against P itself, built from the operator's blocks (Eq. pcext): one GMRES step from
zero returns a multiple of P^-1 b, so P x must be a multiple of b.

What is left over is the Schur complements' error.  Complex128: |I - S X| within 64 units of the
rounding of its terms, sqrt(n) of which add up, beside the rounding of the rest (100 eps of |P| |x|).
Complex64: the inverse and the vectors are rounded to 2^-24, 16 of which cover the products' sums."""
import numpy as np
import pytest

from workloads.meshes import box, icosphere

pytestmark = pytest.mark.gpu

MESHES = {
    "small": lambda: box(0.1, 0.09, 0.08, 4, 4, 6),                      # 255 charges: FP64 LU
    "sphere": lambda: icosphere(2, 0.1),                                 # 319: complex64 LU, refined
    "box": lambda: box(0.1, 0.09, 0.08, 9, 8, 7, jitter=0.1, seed=2),    # 763
    "graded": lambda: box(0.4, 0.02, 0.01, 30, 6, 3, grade=(13.0, 1.0, 1.0), jitter=0.01, seed=1),
}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name", ["small", "sphere", "box", "graded"])
def test_one_step_inverts_p(name, prec):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    v, f = MESHES[name]()
    m = sldm.Mesh(v, f)
    ne, nt = m.ne, m.nt
    nq = nt - 1
    op = sldm.Operator(m, sldm.Stack([(1.0, 1.0, 0.0, 0.0)]), [(4.0, 1.0, 0.01)], 300e6, precision=prec)
    dg = lambda b: np.diag(op.block(b))  # noqa: E731
    _, tp, tm = m.edges()
    D = np.zeros((nt, ne))
    D[tp, np.arange(ne)], D[tm, np.arange(ne)] = 1.0, -1.0
    B = np.vstack([np.eye(nq), -np.ones(nq)])
    FD = D[:nq]
    P13, P23 = D.T @ (dg(sldm.BLOCK_LPM)[:, None] * B), D.T @ (dg(sldm.BLOCK_LP)[:, None] * B)
    a, b_, c, d = dg(sldm.BLOCK_LAM), dg(sldm.BLOCK_IX), dg(sldm.BLOCK_LA), -dg(sldm.BLOCK_K)
    P = np.block([[np.diag(a), np.diag(b_), P13], [np.diag(c), np.diag(d), P23], [FD, np.zeros((nq, ne)), op.k0 ** 2 * np.eye(nq)]])
    det = a * d - b_ * c
    S = op.k0 ** 2 * np.eye(nq) - FD @ ((d / det)[:, None] * P13 - (b_ / det)[:, None] * P23)
    X = np.linalg.inv(S)
    ell = float(np.linalg.norm(v[f[:, 0]] - v[f[:, 1]], axis=1).mean())
    dr = np.ones(op.N)
    dr[2 * ne:] = ell  # the solver's scaling
    rng = np.random.default_rng(6)
    b = (rng.standard_normal(op.N) + 1j * rng.standard_normal(op.N)) / dr
    x = np.zeros(op.N, complex)
    op.solve(b, x, tol=1e-15, maxit=1, refine=False, check=False)
    y = P @ x
    alpha = np.vdot(dr * b, dr * y) / np.linalg.norm(dr * b) ** 2
    res = np.linalg.norm(dr * (y - alpha * b))
    t3 = np.abs(alpha) * (b[2 * ne:] - FD @ (d / det * b[:ne] - b_ / det * b[ne:2 * ne]))
    px = np.linalg.norm(dr * (np.abs(P) @ np.abs(x)))
    if prec == 0:
        lim = 64 * 2.0 ** -52 * np.max(np.abs(S)) * np.max(np.abs(X)) * np.sqrt(nq) * ell * np.linalg.norm(t3) + 100 * 2.0 ** -52 * px
    else:
        lim = 16 * 2.0 ** -24 * (ell * np.linalg.norm(np.abs(S) @ (np.abs(X) @ np.abs(t3))) + px)
    print(name, prec, res, lim, np.linalg.norm(dr * y))
    assert res <= lim, (res, lim)
