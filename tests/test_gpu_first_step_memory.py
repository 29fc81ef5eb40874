"""Device memory that a first step takes: each of its allocations fails once (an allocator hook).  The step
reports LFX_ERR_OOM or does without, no pointer of a half-made buffer is used, and the repeated step equals a
fresh state's bit for bit."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu


class Allocator:
    """PyTorch's caching allocator behind the library's hook; the fail_at-th allocation fails, and those of just
    `refuse` bytes."""

    def __init__(self, refuse=0):
        import torch

        from paper_2304_12032_gb300 import lfx as L

        self.n, self.fail_at, self.refused, dev = 0, -1, 0, torch.cuda.current_device()

        def alloc(nbytes, ctx):
            self.n += 1
            if nbytes == refuse:
                self.refused += 1
                return None
            return None if self.n == self.fail_at else torch.cuda.caching_allocator_alloc(int(nbytes), dev)

        self.keep = L.ALLOC_FN(alloc), L.FREE_FN(lambda p, ctx: torch.cuda.caching_allocator_delete(p))
        L._check(L.library().lfx_set_allocator(*self.keep, None))

    def close(self):
        from paper_2304_12032_gb300 import lfx as L

        L._check(L.library().lfx_set_allocator(L.ALLOC_FN(), L.FREE_FN(), None))


@pytest.mark.parametrize("opts", [{}, dict(precision="mixed", smoother_bf16=1)], ids=["fp64", "mixed"])
def test_each_allocation_of_a_first_step_fails_once(opts):
    from paper_2304_12032_gb300 import lfx as L

    case = C.vessel_case(3000, seed=31)
    _, prob, st = C.gpu_state(case, assembly="persistent", **opts)
    st.step()
    want = st.get()
    hook = Allocator()
    try:
        k, failed = 0, 0
        while True:
            k += 1
            st = L.State(prob, case.u_hist, case.p_hist, case.t0)
            hook.n, hook.fail_at = 0, k
            try:
                st.step()
            except L.LfxError as e:
                assert e.status == L.LFX_ERR_OOM, k
                failed += 1
                hook.fail_at = -1
                st.step()
            reached, hook.fail_at = hook.n >= k, -1
            for a, b in zip(st.get(), want):
                assert np.array_equal(a, b), k
            del st
            if not reached:
                break
        assert failed >= 5
    finally:
        hook.close()


def gather_bytes(mesh):
    c = mesh.chunks()
    return 8 * (16 * len(c["run_row"]) + 4 * int((c["run_row"] == c["run_col"]).sum()))


@pytest.mark.parametrize("opts", [{}, dict(precision="mixed", smoother_bf16=1)], ids=["fp64", "mixed"])
def test_gather_scratch_is_held_only_where_the_persistent_launch_runs(opts):
    """16 values per run and 4 per diagonal run: present with the persistent launch, absent with the others, in
    the state's bytes and in the admission estimate (10 % slack on each); with the autotuner as its choice says."""
    from paper_2304_12032_gb300 import lfx as L

    case = C.vessel_case(20000, seed=33, riis=False)
    held, need, gather = {}, {}, 0
    for shape in ("colors", "chunks", "persistent", "auto"):
        mesh, prob, st = C.gpu_state(case, assembly=shape, **opts)
        gather = gather_bytes(mesh)
        before = L.problem_state_bytes(prob)
        st.step()
        held[shape], need[shape] = st.device_bytes(), (before, L.problem_state_bytes(prob))
        mode = prob.assembly_tuning()[0]
    assert held["colors"] == held["chunks"] == held["persistent"] - gather
    assert held["auto"] == held["persistent" if mode == 3 else "chunks"]
    slack = gather + gather // 10
    assert need["colors"] == need["chunks"] and need["colors"][0] == need["colors"][1]
    assert abs(need["persistent"][0] - need["colors"][0] - slack) <= 2
    assert need["auto"][0] == need["persistent"][0]
    assert need["auto"][1] == need["persistent" if mode == 3 else "chunks"][0]


@pytest.mark.parametrize("newton", [0, 1])
def test_a_gather_scratch_that_cannot_be_had_leaves_the_coloured_form(newton):
    """An allocator that refuses just that size: the persistent launch steps colour by colour, the same sums (the
    semi-implicit step bit for bit, the Newton step to the rounding of its right-hand side: 1e-9)."""
    from paper_2304_12032_gb300 import lfx as L

    case = C.vessel_case(3000, seed=35, riis=False)
    mesh, prob, st = C.gpu_state(case, assembly="persistent", implicit=newton)
    st.step()
    want = st.get()
    hook = Allocator(refuse=gather_bytes(mesh))
    try:
        st = L.State(prob, case.u_hist, case.p_hist, case.t0)
        for _ in range(2):
            st.set(case.u_hist, case.p_hist, case.t0)
            assert st.step()["converged"] and hook.refused == 1
            for a, b in zip(st.get(), want):
                assert np.array_equal(a, b) if not newton else np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)
        del st
    finally:
        hook.close()
