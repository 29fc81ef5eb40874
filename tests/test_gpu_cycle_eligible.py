"""When the persistent Krylov cycle's row partition is made, seen from the device bytes (2 bytes per block and
more on the mesh) and from the kernel launches of a step: a cycle takes one launch for all its Arnoldi steps, the
step-by-step form more than ten for each."""
import numpy as np
import pytest

from tests import cases as C
from tests.test_gpu_first_step_memory import Allocator

pytestmark = pytest.mark.gpu

MIXED = dict(precision="mixed", smoother_bf16=1)


def run(case, **opts):
    """(device bytes, launches of the second step, its Arnoldi steps, solution after it, blocks of the matrix)"""
    from paper_2304_12032_gb300 import lfx as L

    lib = L.library()
    mesh, _, st = C.gpu_state(case, assembly="chunks", **opts)
    st.step()
    n = lib.lfx_launch_count()
    its = st.step()["iterations"]
    return st.device_bytes(), lib.lfx_launch_count() - n, its, st.get(), mesh.info()["nnz_blocks"]


def one_launch_per_cycle(launches, its):
    assert its > 8
    return launches < 2 * its + 150        # (assembly, set-up and outer steps: about 100 launches)


@pytest.mark.parametrize("opts,unwanted", [
    ({}, dict(reorthogonalize=1)), (MIXED, dict(reorthogonalize=2)), ({}, dict(s_steps=2)), ({}, dict(f_steps=1)),
    ({}, dict(s_smoother="chebyshev", s_steps=6)),
])
def test_no_partition_where_no_cycle_can_run(opts, unwanted):
    case = C.vessel_case(6000, seed=51, riis=False)
    on, launches, its, _, nnzb = run(case, **opts)
    assert one_launch_per_cycle(launches, its)
    off, launches, its, _, _ = run(case, **opts, **unwanted)
    assert not one_launch_per_cycle(launches, its) and launches > 10 * its
    assert off <= on - 2 * nnzb


def test_no_partition_with_a_resistance_outlet():
    on, launches, its, _, nnzb = run(C.vessel_case(6000, seed=52, riis=False))
    assert one_launch_per_cycle(launches, its)
    off, launches, its, _, _ = run(C.vessel_case(6000, seed=52, riis=False, resistance=5.0))
    assert launches > 10 * its and off <= on - 2 * nnzb + 65536     # (the outlet's own arrays)


@pytest.mark.parametrize("opts", [{}, MIXED], ids=["fp64", "mixed"])
def test_a_partition_that_cannot_be_had_leaves_the_step_by_step_form(opts):
    """An allocator that refuses the local column indices: the problem is made all the same, and its steps are
    those of the launches (both solved to 1e-10; 1e-6 as in the tests against the oracle)."""
    case = C.vessel_case(6000, seed=53, riis=False)
    _, launches, its, want, nnzb = run(case, gmres_rtol=1e-10, **opts)
    assert one_launch_per_cycle(launches, its)
    hook = Allocator(refuse=2 * nnzb)
    try:
        _, launches, its, got, _ = run(case, gmres_rtol=1e-10, **opts)
    finally:
        hook.close()
    assert hook.refused >= 1 and launches > 10 * its
    for a, b in zip(got, want):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("n,precision,lanes,spill", [
    (2, "fp64", 16, 0), (15, "fp64", 16, 0), (16, "fp64", 4, 0), (20, "mixed", 16, 0), (21, "mixed", 8, 0),
    (26, "mixed", 4, 0), (56, "fp64", 4, 1), (70, "mixed", 4, 1), (84, "mixed", 4, 2)])
def test_shapes_of_the_cycle_tests(n, precision, lanes, spill):
    """The sizes at which the cycle is compared with the launches run the shapes that they are meant for."""
    case = C.beltrami_case(n, seed=n)
    mesh, _, st = C.gpu_state(case, precision=precision, smoother_bf16=1, assembly="chunks", gmres_rtol=1e-6)
    assert st.debug_cycle_plan()["ctas"] == 0          # (not planned before the first set-up)
    st.step()
    p = st.debug_cycle_plan()
    V = case.mesh.n_nodes
    assert p["ctas"] == max(1, min(151, V // (8 if precision == "fp64" else 32)))
    assert (p["lanes"], p["spill"], p["segments"]) == (lanes, spill, 1)
    part = mesh.cycle_partition(p["ctas"])
    assert (part["max_rows"], part["max_loc"]) == (p["max_rows"], p["max_loc"])


@pytest.mark.parametrize("opts", [{}, MIXED], ids=["fp64", "mixed"])
def test_shape_of_a_batch(opts):
    from paper_2304_12032_gb300 import lfx as L
    from synthetic import batch, cube_kuhn

    m = batch([cube_kuhn(n, seed=n) for n in (2, 3, 9, 14)], tag_stride=0)
    bcs = [L.BC(tag=t, kind="noslip") for t in range(1, 6)] + [L.BC(tag=6, kind="neumann", time="constant", p=(0.0,))]
    for segmented in (1, 0):
        prob = L.Problem(L.Mesh.from_synthetic(m), 1.0, 0.05, 1e-2, 1, bcs, [], L.default_options(batch_segmented=segmented, **opts))
        st = L.State(prob, np.ones((1, m.n_nodes, 3)), np.zeros((1, m.n_nodes)), 0.0)
        st.step()
        assert st.debug_cycle_plan()["segments"] == (4 if segmented else 1)
