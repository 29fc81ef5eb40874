"""The staged velocity smoothing pass where it runs: in solves that the persistent Krylov cycle does not take
(here those with a second Gram-Schmidt pass, and with a resistance outlet).  The launches of a step show that it is
the step-by-step form, and a tile's wait that runs out in one preconditioner application that this form stages.

* Against the oracle's step (1e-6, the mixed-step tolerance), and against the plain pass (the same sums in the
  same order: equal up to the rounding of the solver's own reductions, 1e-9).
* More tiles than resident CTAs, over three steps: the same Krylov counts as the plain pass, 1e-9, and 1e-6 of
  the FP64 step."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu

MIXED = dict(precision="mixed", smoother_bf16=1, gmres_rtol=1e-10, reorthogonalize=2)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def step(st):
    """A step's statistics, having checked that it ran launch by launch."""
    from paper_2304_12032_gb300 import lfx as L

    n = L.library().lfx_launch_count()
    stats = st.step()
    assert L.library().lfx_launch_count() - n > 10 * stats["iterations"] > 0
    return stats


@pytest.mark.parametrize("resistance", [0.0, 5.0])
def test_staged_pass_matches_oracle_and_plain_pass(resistance):
    from paper_2304_12032_gb300 import lfx as L

    case = C.vessel_case(6000, seed=23, resistance=resistance)
    opts = dict(MIXED, reorthogonalize=0 if resistance else 2)
    ost = C.oracle_step(case)
    outs = {}
    for staged in (1, 0):
        _, _, st = C.gpu_state(case, staged_f=staged, **opts)
        assert st.debug_staged_timeout() == (L.LFX_ERR_TIMEOUT if staged else L.LFX_ERR_INVALID_ARG)
        assert step(st)["converged"]
        outs[staged] = st.get()
    xref = ost.x.reshape(-1, 4)
    for i, ref in enumerate((xref[:, :3], xref[:, 3])):
        assert rel(outs[1][i], ref) <= 1e-6
        assert rel(outs[1][i], outs[0][i]) <= 1e-9


def test_staged_pass_with_several_tiles_per_cta():
    case = C.vessel_case(400000, seed=5, riis=False)
    assert case.mesh.n_nodes > 152 * 8 * 32      # more 32-row tiles than the staged kernel's resident CTAs
    states = {"staged": C.gpu_state(case, staged_f=1, **MIXED)[2], "plain": C.gpu_state(case, staged_f=0, **MIXED)[2],
              "fp64": C.gpu_state(case, gmres_rtol=1e-10)[2]}
    for k in range(3):
        its = {key: step(states[key])["iterations"] for key in ("staged", "plain")}
        states["fp64"].step()
        assert its["staged"] == its["plain"], (k, its)
        sol = {key: st.get() for key, st in states.items()}
        for i in range(2):
            assert rel(sol["staged"][i], sol["plain"][i]) <= 1e-9, (k, i)
            assert rel(sol["staged"][i], sol["fp64"][i]) <= 1e-6, (k, i)
