"""Defect corrections that stop on the device (fields below 2^19 elements) against the same ones checked by
the host after every iteration (RHMC_TUNE_CORRECTION_CHECK_EVERY = 1): the same arithmetic and the
same stopping rule, so the same iterations and, to the rounding of one FP64 addition, the same
solutions; replayed chunks serve corrections of every shift, at every place of a chunk."""
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

CHECK_EVERY = 24  # RHMC_TUNE_CORRECTION_CHECK_EVERY


@pytest.mark.parametrize("dims,n", [((4, 4, 4, 4), 1), ((4, 6, 4, 8), 3), ((8, 8, 8, 8), 8), ((6, 4, 6, 4), 16)])
def test_device_and_host_stops_agree(dims, n):
    need_gpu()
    shifts = [0.0, 0.003, 0.05, 0.4, 3.0]
    ctx = make_ctx(dims, 0.03, syn.random_links(dims, 0.5, 1720))
    B = to_gpu(syn.gaussian_pseudofermions(dims, n, 2820))
    some = 0
    for tol in (1e-8, 3e-9, 1e-9, 2e-10, 1e-10, 3e-11, 1e-11, 1e-12):
        out = []
        for every in (0, 1):
            ctx.tune_set(CHECK_EVERY, every)
            out.append(ctx.block_multishift_cg(B, shifts, tol))
        (X, dev), (Y, host) = out
        assert dev.true_rel_resid_max <= tol and dev.refinements == host.refinements
        assert dev.refine_iters == host.refine_iters and dev.iters == host.iters
        assert (X - Y).abs().max().item() <= 2.0 ** -52 * Y.abs().max().item()
        some += dev.refine_iters
    assert some > 0
    ctx.close()
