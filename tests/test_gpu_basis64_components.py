"""Components of FP64 solutions that are small because columns hardly mix: sources of one colour per
column under links exp(i eps H), whose solutions in the other colours are of order eps.  Solves without a
tolerance that stops them early, so that what is left is rounding: against a dense solve refined in
extended precision the stored basis (csrc/basis64.cu) is held to the larger of four times the
error of the updates in HBM (the same recursion with FP64 FMAs, whose own error varies by
as much with the order of its sums) and 1.3e-12 of the largest small component: 30
iterations at a condition number of 400, 400 x 30 x 2^-53."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import _lib
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

NATIVE = 5  # RHMC_TUNE_NATIVE_FP64_RESIDUALS


def _links(dims, eps):
    H = np.einsum("...a,aij->...ij", np.random.default_rng(6).standard_normal(dims[::-1] + (4, 8)), syn.gell_mann())
    Y, E = 0.5j * eps * H, np.eye(3)
    for k in range(12, 0, -1):
        E = np.eye(3) + Y @ E / k
    return np.ascontiguousarray(E)


def _dense(ctx):
    m = ctx.Vh * 3
    A = np.zeros((m, m), complex)
    ctx.tune_set(NATIVE, 1)
    for c in range(0, m, 16):
        X = np.zeros((m, 16), complex)
        X[c + np.arange(16), np.arange(16)] = 1
        A[:, c:c + 16] = ctx.apply_mdagm_mrhs(to_gpu(X.reshape(ctx.Vh, 3, 16)), 0.0, "fp64").cpu().numpy().reshape(m, 16)
    ctx.tune_set(NATIVE, 0)
    return A


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("shifts", [[0.0, 0.05], [0.0, 0.05, 0.4, 2.0]])
def test_small_components(eps, shifts):
    need_gpu()
    dims = (4, 4, 4, 4)
    ctx = make_ctx(dims, 0.1, _links(dims, eps))
    A, rng = _dense(ctx), np.random.default_rng(1)
    B = np.zeros((ctx.Vh, 3, 3), complex)
    for c in range(3):
        B[:, c, c] = rng.standard_normal(ctx.Vh) + 1j * rng.standard_normal(ctx.Vh)
    cross = np.broadcast_to(~np.eye(3, dtype=bool), B.shape)
    err = {}
    for iters in (0, 1):
        ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, iters)
        X, _ = ctx.block_multishift_cg(to_gpu(B), shifts, 1e-14, precision="fp64", allow_not_converged=True)
        err[iters] = X.cpu().numpy()
    ctx.close()
    for q, sig in enumerate(shifts):
        S = A + sig * np.eye(len(A))
        Y = np.linalg.solve(S, B.reshape(-1, 3)).astype(np.clongdouble)
        for _ in range(6):
            Y = Y + np.linalg.solve(S, (B.reshape(-1, 3) - S.astype(np.clongdouble) @ Y).astype(complex))
        Y = Y.reshape(B.shape)
        e = {k: float(np.abs(v[q] - Y)[cross].max() / np.abs(Y)[cross].max()) for k, v in err.items()}
        assert e[0] <= max(4 * e[1], 1.3e-12), (sig, e)
