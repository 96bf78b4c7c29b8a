"""Workspace sizes of the FP64 solves: they follow the context's own launch settings, as the
solves lay the workspace out, and a solve stays within the bytes it asked for.  No tolerances."""
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import _lib
from paper_1808_01829_gb300 import synthetic as syn
from paper_1808_01829_gb300.remez import rational_approx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own,wide", [(1100, 0), (1, 0), (0, 1), (24, 1100)])
def test_rational_workspace_follows_the_context(own, wide):
    torch = need_gpu()
    dims, n = (4, 4, 4, 4), 3
    ra = rational_approx(1.0 / 16, 1e-3, 64.0, 8)
    ctx = make_ctx(dims, 0.1, syn.random_links(dims, 0.3, 1700))
    size = lambda: ctx.lib.rhmc_rational_solve_bytes(ctx._h, n, len(ra.beta))
    key = _lib.RHMC_TUNE_BASIS_ITERS
    try:
        ctx.lib.rhmc_tune_set(key, own)  # the process-wide value, as a context without its own has it
        want = size()
        ctx.lib.rhmc_tune_set(key, wide)
        ctx.tune_set(key, own)
        if own:
            assert size() == want
        need, guard = size(), 1 << 20
        ws = torch.full((need + guard,), 0x5A, dtype=torch.uint8, device="cuda")
        Phi = to_gpu(syn.gaussian_pseudofermions(dims, n, 2800))
        ctx.rational_solve(Phi, ra.alpha0, ra.alpha, ra.beta, 1e-12, workspace=ws)
        assert bool((ws[need:] == 0x5A).all())
    finally:
        ctx.lib.rhmc_tune_set(key, 0)
        ctx.close()


def _solve(ctx, B, shifts, tol):
    X, info = ctx.block_multishift_cg(B, shifts, tol, precision="fp64")
    assert info.true_rel_resid_max <= tol
    return X, info


def test_fp64_basis_takes_the_memory_it_needs():
    """More than one piece of 64 MB, about as much kept as was needed; the solve without the basis agrees."""
    torch = need_gpu()
    dims, n, tol, shifts = (16, 16, 16, 16), 8, 1e-12, [0.0, 0.02, 0.3, 2.0]
    ctx = make_ctx(dims, 0.05, syn.random_links(dims, 0.5, 1701))
    B = to_gpu(syn.gaussian_pseudofermions(dims, n, 2801))
    block = ctx.Vh * 3 * n * 16
    assert ctx.workspace_bytes(n, len(shifts), "fp64") < 60 * block + (64 << 20)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, 1)
    H, off = _solve(ctx, B, shifts, tol)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, 0)
    free = torch.cuda.mem_get_info()[0]
    X, info = _solve(ctx, B, shifts, tol)
    kept = free - torch.cuda.mem_get_info()[0]
    assert info.iters == off.iters and info.iters * block > 200 << 20
    assert kept <= 2 * (info.iters + 24) * block + ctx.workspace_bytes(n, len(shifts), "fp64") + 3 * block
    # residuals of tol move a solution by at most tol |B| / (4 m^2 + sigma) each
    for q, sig in enumerate(shifts):
        assert (X[q] - H[q]).norm().item() <= 2 * tol * B.norm().item() / (4 * 0.05 ** 2 + sig)
    ctx.close()


@pytest.mark.parametrize("room", [1500 << 20, 500 << 20])
def test_fp64_basis_without_memory(room):
    """With 1.5 GB free the basis takes up to half of it and the solve goes on without; with 0.5 GB, which
    holds fewer than 24 blocks of 12.6 MB beside what has to stay free, it starts without."""
    torch = need_gpu()
    dims, n, tol, shifts = (16, 16, 16, 16), 8, 1e-12, [0.0, 0.02, 0.3, 2.0]
    U = syn.random_links(dims, 0.5, 1701)
    B = to_gpu(syn.gaussian_pseudofermions(dims, n, 2801))
    ctx = make_ctx(dims, 0.05, U)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, 10)  # (loads the kernels of both forms)
    H, off = _solve(ctx, B, shifts, tol)
    ctx.close()
    assert off.iters * ctx.Vh * 3 * n * 16 > 750 << 20
    ctx = make_ctx(dims, 0.05, U)
    ws = torch.empty(ctx.workspace_bytes(n, len(shifts), "fp64"), dtype=torch.uint8, device="cuda")
    X = torch.empty((len(shifts),) + tuple(B.shape), dtype=B.dtype, device="cuda")
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        _, info = ctx.block_multishift_cg(B, shifts, tol, precision="fp64", out=X, workspace=ws)
        left = torch.cuda.mem_get_info()[0]
    finally:
        del hold
        torch.cuda.empty_cache()
    assert info.true_rel_resid_max <= tol and info.iters == off.iters and left > 200 << 20
    for q, sig in enumerate(shifts):
        assert (X[q] - H[q]).norm().item() <= 2 * tol * B.norm().item() / (4 * 0.05 ** 2 + sig)
    ctx.close()
