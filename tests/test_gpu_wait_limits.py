"""The bounded waits of the persistent Krylov cycle and of the lifting, made to run out (a target that nothing reaches, a limit of
milliseconds): the step reports LFX_ERR_TIMEOUT after a few launches instead of restarting an empty cycle until
the host's own limit of 100,000, the state keeps its time level, and its next step equals a fresh state's."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu

MIXED = dict(precision="mixed", smoother_bf16=1)
CASES = {"fp64": {}, "mixed-bf16": MIXED, "mixed-fp32": dict(MIXED, smoother_bf16=0),
         "newton": dict(MIXED, implicit=1), "newton-fp64": dict(implicit=1)}


def expect_timeout_then_recovery(prob, st, case):
    from paper_2304_12032_gb300 import lfx as L

    lib = L.library()
    st.debug_cycle_timeout(True)
    for _ in range(2):                       # the report clears the word: a second failure reports again
        n = lib.lfx_launch_count()
        with pytest.raises(L.LfxError) as err:
            st.step()
        assert err.value.status == L.LFX_ERR_TIMEOUT and "gave up" in str(err.value)
        assert lib.lfx_launch_count() - n < 3000
    st.debug_cycle_timeout(False)
    fresh = L.State(prob, case.u_hist, case.p_hist, case.t0)
    for tag, vals in (case.nodal or {}).items():
        fresh.set_dirichlet_nodal(tag, vals)
    if case.pin_node >= 0:
        fresh.set_pressure_pin(case.pin_value)
    assert st.step()["t"] == fresh.step()["t"]
    for a, b in zip(st.get(), fresh.get()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("name", list(CASES))
def test_cycle_waits_that_run_out(name):
    case = C.vessel_case(6000, seed=41)
    _, prob, st = C.gpu_state(case, **CASES[name])
    expect_timeout_then_recovery(prob, st, case)


@pytest.mark.parametrize("opts", [{}, MIXED], ids=["fp64", "mixed"])
def test_cycle_waits_that_run_out_in_a_batch(opts):
    from paper_2304_12032_gb300 import lfx as L
    from synthetic import batch, cube_kuhn

    m = batch([cube_kuhn(n, seed=n) for n in (3, 8)], tag_stride=0)
    V = m.n_nodes
    rng = np.random.default_rng(8)
    case = C.Case(m, 1.0, 0.05, 1e-2, 1, [], [], rng.standard_normal((1, V, 3)), rng.standard_normal((1, V)))
    bcs = [L.BC(tag=t, kind="noslip") for t in range(1, 6)] + [L.BC(tag=6, kind="neumann", time="constant", p=(0.0,))]
    prob = L.Problem(L.Mesh.from_synthetic(m), 1.0, 0.05, 1e-2, 1, bcs, [], L.default_options(**opts))
    st = L.State(prob, case.u_hist, case.p_hist, 0.0)
    expect_timeout_then_recovery(prob, st, case)


def test_cycle_waits_that_run_out_in_a_solve():
    from paper_2304_12032_gb300 import lfx as L

    _, _, st = C.gpu_state(C.vessel_case(6000, seed=42))
    st.debug_assemble(apply_bcs=True)
    st.debug_cycle_timeout(True)
    with pytest.raises(L.LfxError) as err:
        st.debug_solve()
    assert err.value.status == L.LFX_ERR_TIMEOUT
    st.debug_cycle_timeout(False)
    st.debug_assemble(apply_bcs=True)
    assert st.debug_solve()[1]["converged"]


@pytest.mark.parametrize("n", [2, 9, 24])
def test_lifting_waits_that_run_out(n):
    """One CTA, fewer rows than CTAs, a full grid.  The repeated step extends linear boundary data to the linear
    field, to the 1e-9 derived in the lifting's own test (two states' liftings differ in the last bits: their
    matrices are summed in the order of atomic additions)."""
    from paper_2304_12032_gb300 import lfx as L
    from synthetic import cube_kuhn

    m = cube_kuhn(n, seed=n)
    prob = L.Problem(L.Mesh.from_synthetic(m), 1.0, 1.0, 1e-3, 1, [L.BC(tag=t, kind="nodal") for t in range(1, 7)], [],
                     L.default_options(pin_pressure_node=0))
    V = m.n_nodes
    st = L.State(prob, np.zeros((1, V, 3)), np.zeros((1, V)), 0.0)
    st.set_displacement(np.zeros((1, V, 3)))
    d = m.nodes @ np.array([[0.02, 0.01, 0.0], [-0.01, 0.03, 0.0], [0.0, 0.02, -0.02]]) + 0.005
    bd = np.unique(m.bfaces.ravel())
    st.set_boundary_displacement(bd, d[bd])
    st.debug_lifting_timeout(True)
    for _ in range(2):
        with pytest.raises(L.LfxError) as err:
            st.step()
        assert err.value.status == L.LFX_ERR_TIMEOUT and "gave up" in str(err.value)
    assert not st.get_displacement()[0].any()              # the state keeps its time level
    st.debug_lifting_timeout(False)
    assert st.step(allow_not_converged=True)["t"] == 1e-3   # (and the prescribed data, for the repetition)
    assert np.abs(st.get_displacement()[0] - d).max() <= 1e-9 * np.abs(d).max()
