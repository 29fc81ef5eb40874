"""Device memory that a first step takes: each of its allocations fails once (an allocator hook).  The step
reports LFX_ERR_OOM or does without, no pointer of a half-made buffer is used, and the repeated step equals a
fresh state's bit for bit."""
import numpy as np
import pytest

from tests import cases as C

pytestmark = pytest.mark.gpu


class Allocator:
    """PyTorch's caching allocator behind the library's hook; the fail_at-th allocation fails."""

    def __init__(self):
        import torch

        from paper_2304_12032_gb300 import lfx as L

        self.n, self.fail_at, dev = 0, -1, torch.cuda.current_device()

        def alloc(nbytes, ctx):
            self.n += 1
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
