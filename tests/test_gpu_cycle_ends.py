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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_hard_member_beside_easy_ones(precision):
    """Members that converge early wait with zero basis vectors for the hardest one: each solution equals the
    member's own solve (both to 1e-11 of the right-hand side; 1e-7 as in the batch test of the cycle), and the
    batch takes no more steps than the hardest member alone, up to the different hierarchies."""
    from paper_2304_12032_gb300 import lfx as L
    from synthetic import batch, cube_kuhn

    sizes, rng = (3, 16, 2, 4), np.random.default_rng(2)
    ms = [cube_kuhn(n, seed=n) for n in sizes]
    hist = [(rng.standard_normal((1, m.n_nodes, 3)), rng.standard_normal((1, m.n_nodes))) for m in ms]
    opt = dict(precision=precision, gmres_rtol=1e-11, smoother_bf16=1)
    bcs = [L.BC(tag=t, kind="noslip") for t in range(1, 6)] + [L.BC(tag=6, kind="neumann", time="constant", p=(0.0,))]

    def solve(m, u, p):
        prob = L.Problem(L.Mesh.from_synthetic(m), 1.0, 0.05, 1e-2, 1, bcs, [], L.default_options(**opt))
        st = L.State(prob, u, p, 0.0)
        return st.step(), *st.get()

    union = batch(ms, tag_stride=0)
    stats, u, p = solve(union, np.concatenate([h[0] for h in hist], axis=1), np.concatenate([h[1] for h in hist], axis=1))
    assert stats["converged"]
    off, steps = union.meta["node_offsets"], []
    for i, m in enumerate(ms):
        a, ui, pi = solve(m, *hist[i])
        steps.append(a["iterations"])
        sl = slice(off[i], off[i] + m.n_nodes)
        assert rel(u[sl], ui) < 1e-7 and rel(p[sl], pi) < 1e-7
    assert min(steps) < max(steps)
    assert stats["iterations"] <= 1.25 * max(steps) + 4


@pytest.mark.parametrize("f_steps,more", [(2, 0), (3, 0), (4, 1), (6, 1)])
def test_cycle_statistics_count_what_was_timed(f_steps, more):
    """One product per Arnoldi step; the plain velocity passes of every step (all but the first), and those of the
    last, unfinished step before the verdict that ends a cycle (two cycles here)."""
    case = C.beltrami_case(9, seed=9)
    _, _, st = C.gpu_state(case, gmres_rtol=1e-30, gmres_restart=6, gmres_max_iters=12, f_steps=f_steps)
    stats = st.step(allow_not_converged=True)
    assert stats["iterations"] == 12 == stats["n_spmv"]
    assert stats["n_fpass"] == (f_steps - 2) * 12 + 2 * more
    assert 0.0 < stats["ms_spmv"] < stats["ms_solve"]
    assert stats["n_fpass"] * stats["ms_fpass_median"] < stats["ms_solve"]
