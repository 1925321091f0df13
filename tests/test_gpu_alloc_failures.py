"""Every device allocation of an assembly and of a far field, failing in turn.  A call either returns SLDM_ENOMEM with all
it took released, or goes its other way with the same result: the Schur complement's inverse by the FP64 LU
instead of the refined complex64 one (other launches; solutions within the solve's tolerance
times the conditioning, 1e-7), the far field with a smaller workspace (the same sums: 1e-12 of the largest)."""
import numpy as np
import pytest

from workloads.meshes import box, icosphere

pytestmark = pytest.mark.gpu


def _failing(sl, k, call):
    sl.test_inject(sl.INJECT_ALLOC, k)
    try:
        return call()
    except sl.SldmError as e:
        assert e.code == sl.ENOMEM
        return None
    finally:
        sl.test_inject(sl.INJECT_ALLOC, 0)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_assembly(prec):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    m, st = sldm.Mesh(*icosphere(2, 0.1)), sldm.Stack([(1.0, 1.0, 0.0, 0.0)])

    def launches(call):
        n = sldm.launch_count()
        op = call()
        return op, sldm.launch_count() - n

    def build():
        return sldm.Operator(m, st, [(4.0, 1.0, 0.01)], 300e6, precision=prec)

    def solved(op):
        b = op.rhs_planewave((0, 0, -1), (1, 0, 0), np.zeros(op.N, complex))
        x = np.zeros_like(b)
        it = op.solve(b, x, tol=1e-9)["iters"]
        return x, it

    build().close()  # the form of its products is measured once per shape
    ref, plain = launches(build)
    x_ref, it_ref = solved(ref)
    held = sldm.device_bytes()
    fallbacks = 0
    for k in range(1, 1000):
        op, n = launches(lambda: _failing(sldm, k, build))
        if op is None:
            assert sldm.device_bytes() == held, k
            continue
        if n == plain:
            break  # past the last allocation
        fallbacks += 1
        x, it = solved(op)
        assert abs(it - it_ref) <= 2, k  # the solve has converged, and as fast
        if prec != 1:  # (two FP32 fills are two operators: their atomics add in different orders)
            assert np.linalg.norm(x - x_ref) <= 1e-7 * np.linalg.norm(x_ref), k
        op.close()
    assert fallbacks >= 4 and k < 999, (fallbacks, k)  # the inverse's four buffers and its factorisation's


@pytest.mark.parametrize("layered", [False, True])
def test_far_field(layered):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    v, f = box(0.1, 0.09, 0.08, 9, 8, 7)
    layers = [(1.0, 1.0, 0.0, 0.0), (2.25, 1.0, 0.0, 0.0)] if layered else [(1.0, 1.0, 0.0, 0.0)]
    op = sldm.Operator(sldm.Mesh(v, f), sldm.Stack(layers, z_top=float(v[:, 2].min()) - 0.05), [(4.0, 1.0, 0.0, 0)], 300e6)
    rng = np.random.default_rng(2)
    x = rng.standard_normal((9, op.N)) + 1j * rng.standard_normal((9, op.N))
    th = np.linspace(0.01, 1.5, 700)
    ref = op.farfield_n(x, th, 0.3, 9)
    got = _failing(sldm, 1, lambda: op.farfield_n(x, th, 0.3, 9))
    assert got is not None and np.max(np.abs(got - ref)) <= 1e-12 * ref.max()
