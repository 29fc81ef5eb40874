"""The FP64 row kernels of aSIMPLE (a lane per row component) against the preconditioner written out in
numpy, through the allocation-free entry point, on graphs whose rows hold one to about thirty blocks: sizes
below a warp's ten rows, at and past a CTA's eighty, and not a multiple of either.  Both sides round the
same operations in another order: five smoothing steps on rows of at most 100 terms, 1e-12 of the result."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def system(V, seed):
    rng = np.random.default_rng(seed)
    pairs = {(i, i) for i in range(V)}
    for i in range(V):
        for j in rng.integers(0, V, rng.integers(0, 14)):
            pairs |= {(i, int(j)), (int(j), i)}
    key = np.array(sorted(pairs))
    row, col = key[:, 0], key[:, 1]
    B = 0.02 * rng.standard_normal((len(key), 4, 4))
    on = row == col
    B[on] += np.diag([2.0, 2.5, 3.0, 1.5])
    return row, col, B, rng.standard_normal((V, 4))


def reference(row, col, B, r, f_steps, s_steps, f_ratio, s_ratio):
    V = len(r)
    A = np.zeros((V, 4, V, 4))
    A[row, :, col, :] = B
    F, G = A[:, :3, :, :3].reshape(3 * V, 3 * V), A[:, :3, :, 3].reshape(3 * V, V)
    D, Cc = A[:, 3, :, :3].reshape(V, 3 * V), A[:, 3, :, 3]
    dF = 1.0 / np.diag(F)
    S = Cc - (D * dF) @ G
    dS = 1.0 / np.diag(S)
    lf = (np.abs(dF) * np.abs(F).sum(1)).max()
    ls = (np.abs(dS) * (np.abs(Cc).sum(1) + np.abs(D) @ (np.abs(dF) * np.abs(G).sum(1)))).max()

    def smooth(M, d, b, lmax, ratio, steps):
        theta, delta = 0.5 * (lmax + lmax / ratio), 0.5 * (lmax - lmax / ratio)
        rho, res = delta / theta, d * b
        step = res / theta
        x = step
        for _ in range(1, steps):
            res = res - d * (M @ step)
            new = 1.0 / (2.0 * theta / delta - rho)
            step = new * rho * step + 2.0 * new / delta * res
            x, rho = x + step, new
        return x

    u = smooth(F, dF, r[:, :3].reshape(-1), lf, f_ratio, f_steps)
    p = smooth(S, dS, r[:, 3] - D @ u, ls, s_ratio, s_steps)
    return np.concatenate([(u - dF * (G @ p)).reshape(V, 3), p[:, None]], axis=1)


@pytest.mark.parametrize("f_steps,s_steps", [(1, 1), (2, 1), (6, 6)])
@pytest.mark.parametrize("V", [1, 9, 10, 11, 63, 80, 81, 333])
def test_matches_numpy(V, f_steps, s_steps):
    import torch

    from paper_2304_12032_gb300 import lfx as L

    row, col, B, r = system(V, V)
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=V))])
    key = row * V + col
    diag, trans = np.searchsorted(key, np.arange(V) * (V + 1)), np.searchsorted(key, col * V + row)
    dev = [torch.tensor(np.ascontiguousarray(a, dtype=np.int32), device="cuda") for a in (rp, col, diag, trans)]
    dev += [torch.tensor(a, device="cuda") for a in (B, r)]
    z = torch.full((V, 4), float("nan"), dtype=torch.float64, device="cuda")
    opt = L.default_options(s_smoother="chebyshev", f_steps=f_steps, s_steps=s_steps)
    rc = L.library().lfx_asimple_apply_noalloc(V, *(ctypes.c_void_p(t.data_ptr()) for t in (*dev, z)), ctypes.byref(opt), None)
    assert rc == 0, L.library().lfx_last_error()
    torch.cuda.synchronize()
    ref = reference(row, col, B, r, f_steps, s_steps, opt.f_ratio, opt.s_ratio)
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
