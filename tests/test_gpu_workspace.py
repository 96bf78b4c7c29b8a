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
