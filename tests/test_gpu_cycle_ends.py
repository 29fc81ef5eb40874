"""How the persistent Krylov cycle ends: full (its last step is the restart length), at the iteration limit, or
converged, for restart lengths from a single step.  Both arms run the same restarted method (the other one step
by step, chosen by asking for a second Gram-Schmidt pass) for the same number of steps.  They differ by rounding
only: the limit of 21 steps keeps the growth from step to step far below the 1e-9 allowed."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [2, 6, 15])
@pytest.mark.parametrize("restart,limit", [(1, 1), (1, 5), (2, 21), (3, 21), (7, 21), (64, 4)])
def test_cycle_ends_at_restart_and_iteration_limits(n, restart, limit):
    case = C.beltrami_case(n, seed=n)
    out = []
    for reorth in (0, 1):
        _, _, st = C.gpu_state(case, gmres_rtol=1e-30, gmres_restart=restart, gmres_max_iters=limit,
                               reorthogonalize=reorth)
        stats = st.step(allow_not_converged=True)
        assert stats["iterations"] == limit and not stats["converged"]
        u, p = st.get()
        out.append((u, p - p.mean()))
    assert rel(out[0][0], out[1][0]) < 1e-9 and rel(out[0][1], out[1][1]) < 1e-9


def test_many_short_cycles_repeat_bit_for_bit():
    """Three hundred cycles of one step and more, each ended by the verdict on its last step: the same bits
    every time."""
    case = C.beltrami_case(9, seed=4)
    _, _, st = C.gpu_state(case, gmres_rtol=1e-30, gmres_restart=1, gmres_max_iters=100)
    got = []
    for _ in range(3):
        st.set(case.u_hist, case.p_hist, case.t0)
        st.step(allow_not_converged=True)
        got.append(st.get())
    for u, p in got[1:]:
        assert np.array_equal(u, got[0][0]) and np.array_equal(p, got[0][1])
