"""An injected stall of the direct solver ends in SLDM_ETIMEOUT in the form of the solver that runs without it: the
blocked one for a single medium object, the side-by-side kernel for a small one and for many."""
import pytest

from workloads.meshes import icosphere, merge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub,n", [(0, 1), (1, 1), (1, 3)])
def test_the_stalled_solver_is_the_one_in_use(sub, n):
    import torch  # noqa: F401
    from paper_2106_06184_gb300 import sldm
    mats = [(4.0 + i, 1.0, 0.0) for i in range(n)]
    m = sldm.Mesh(*merge(*[icosphere(sub, 0.1, (0.4 * i, 0.0, 0.0)) for i in range(n)])) if n > 1 else sldm.Mesh(*icosphere(sub, 0.1))
    st = sldm.Stack([(1.0, 1.0, 0.0, 0.0)])

    def solvers(stall):
        sldm.timers_reset()
        sldm.timers_enable(True)
        sldm.test_inject(sldm.INJECT_LU_STALL, stall)
        try:
            if stall:
                with pytest.raises(sldm.SldmError) as e:
                    sldm.Operator(m, st, mats, 300e6)
                assert e.value.code == sldm.ETIMEOUT
            else:
                sldm.Operator(m, st, mats, 300e6)
        finally:
            sldm.test_inject(sldm.INJECT_LU_STALL, 0)
            sldm.timers_enable(False)
        t = sldm.timers_read()
        return [k for k in ("lu_blocked", "lu_coop") if t.get(k, (0, 0))[1] > 0]

    first = solvers(0)[0]
    assert solvers(1) == [first]  # the first launch failed: nothing came after it
