"""The persistent Krylov cycle against the step-by-step launches of the same method (chosen by asking for a
second Gram-Schmidt pass), at the sizes where its row partition changes shape: one CTA, 16, 8 or 4 lanes
per row, a full grid with uneven shares, and hierarchies of one, two and more multigrid levels.

Both solves stop at ||r|| <= 2e-12 ||b||, so they differ by at most 4e-12 times the amplification from
residual to solution.  That amplification, taken from the benchmark flows' own tolerance sweeps, stays
below 1e3 (velocity) and 1e4 (pressure of the pinned all-Dirichlet flow)."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,precision,opts", [
    (2, "fp64", {}),                                    # 27 nodes: fewer rows than a CTA's least share
    (6, "fp64", {}), (6, "mixed", {"smoother_bf16": 1}),   # the hierarchy is the dense inverse itself
    (15, "fp64", {}), (16, "fp64", {}),                 # FP64: 16 lanes per row, then ten rows a warp
    (12, "mixed", {"smoother_bf16": 1, "f_steps": 2}),  # two multigrid levels, the shortest smoother
    (20, "mixed", {"smoother_bf16": 1}), (21, "mixed", {"smoother_bf16": 1}),   # FP32: 16 lanes, 8 lanes
    (26, "mixed", {"smoother_bf16": 1}), (26, "mixed", {"smoother_bf16": 0}),   # 4 lanes
    (26, "fp64", {"amg_coarse_size": 40}),              # three levels and more
])
def test_cycle_matches_step_by_step(n, precision, opts):
    case = C.beltrami_case(n, seed=n)
    out = []
    for reorth in (0, 2 if precision == "mixed" else 1):
        _, _, st = C.gpu_state(case, precision=precision, gmres_rtol=1e-12, reorthogonalize=reorth, **opts)
        stats = st.step()
        u, p = st.get()
        out.append((u, p - p.mean(), stats))
    (u, p, a), (ur, pr, b) = out
    assert a["rel_residual"] <= 2e-12 and b["rel_residual"] <= 2e-12
    assert rel(u, ur) < 4e-9 and rel(p, pr) < 4e-8
    assert abs(a["iterations"] - b["iterations"]) <= 2 + b["iterations"] // 10
    assert a["outer_iterations"] == b["outer_iterations"]


@pytest.mark.parametrize("n,precision", [(56, "fp64"), (70, "mixed"), (84, "mixed")])
def test_cycle_with_row_data_in_global_memory(n, precision):
    """Sizes whose rows do not fit shared memory whole: some (56 in FP64, 70 in FP32) or all (84) of a row's
    data stays in global memory.  Solved to 1e-10 (the double-float operator's own rounding shows below
    1e-11 at these sizes); the bounds are the ones above, scaled."""
    case = C.beltrami_case(n, seed=n)
    out = []
    for reorth in (0, 2 if precision == "mixed" else 1):
        _, _, st = C.gpu_state(case, precision=precision, gmres_rtol=1e-10, reorthogonalize=reorth, smoother_bf16=1)
        st.step()
        u, p = st.get()
        out.append((u, p - p.mean()))
        del st
    assert rel(out[0][0], out[1][0]) < 4e-7 and rel(out[0][1], out[1][1]) < 4e-6


def test_cycle_repeats_bit_for_bit():
    """Fixed partitions and summation orders: the same step twice gives the same bits."""
    case = C.beltrami_case(14, seed=3)
    _, _, st = C.gpu_state(case, precision="mixed", smoother_bf16=1)
    got = []
    for _ in range(2):
        st.set(case.u_hist, case.p_hist, case.t0)
        st.step()
        got.append(st.get())
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("precision,opts", [("fp64", {}), ("mixed", {"smoother_bf16": 1}), ("mixed", {"smoother_bf16": 0})])
def test_cycle_of_a_batch_matches_step_by_step(precision, opts):
    """Pieces from one smaller than a CTA's share to one over many CTAs, one at rest (a zero right-hand side
    of its own: its solution is zero), each with its own basis, sums and stopping test."""
    from paper_2304_12032_gb300 import lfx as L
    from synthetic import batch, cube_kuhn

    sizes = (2, 3, 9, 14)
    m = batch([cube_kuhn(n, seed=n) for n in sizes], tag_stride=0)
    V = m.n_nodes
    rng = np.random.default_rng(5)
    u0, p0 = rng.standard_normal((1, V, 3)), rng.standard_normal((1, V))
    first = np.zeros(V, bool)
    first[np.unique(m.tets[: 6 * sizes[0] ** 3])] = True
    u0[0, first], p0[0, first] = 0.0, 0.0
    bcs = [L.BC(tag=t, kind="noslip") for t in range(1, 6)] + [L.BC(tag=6, kind="neumann", time="constant", p=(0.0,))]
    out = []
    for reorth in (0, 2 if precision == "mixed" else 1):
        opt = L.default_options(precision=precision, gmres_rtol=1e-11, reorthogonalize=reorth, **opts)
        prob = L.Problem(L.Mesh.from_synthetic(m), 1.0, 0.05, 1e-2, 1, bcs, [], opt)
        st = L.State(prob, u0, p0, 0.0)
        stats = st.step()
        out.append((*st.get(), stats))
    (u, p, a), (ur, pr, b) = out
    assert a["converged"] and b["converged"]
    assert np.abs(u[first]).max() == 0.0 and np.abs(p[first]).max() == 0.0
    assert rel(u, ur) < 4e-8 and rel(p, pr) < 4e-8
    assert abs(a["iterations"] - b["iterations"]) <= 2 + b["iterations"] // 10
