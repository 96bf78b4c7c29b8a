"""A context with RHMC_TUNE_LINKS12 = 1 whose links change from SU(3) to scaled ones and back: the
captured solver chunks follow the records that the hop reads.  Criteria of the solver tests."""
import pytest

import oracle
from gpu_util import check_solution, make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

LINKS12 = 10  # RHMC_TUNE_LINKS12


@pytest.mark.parametrize("dims,n", [((8, 4, 4, 8), 4), ((4, 4, 4, 4), 1)])
def test_solves_follow_the_staged_links(dims, n):
    need_gpu()
    mass, tol, shifts = 0.05, 1e-9, [0.0, 0.1, 1.0]
    U = syn.random_links(dims, 0.4, 1710)
    B = syn.gaussian_pseudofermions(dims, n, 2810)
    ctx = make_ctx(dims, mass, U)
    ctx.tune_set(LINKS12, 1)
    for scale in (1.0, 1.2, 1.0):
        ctx.set_gauge(to_gpu(scale * U))
        X, info = ctx.block_multishift_cg(to_gpu(B), shifts, tol)
        Xo, _, rc = oracle.sbcgrq(dims, mass, scale * U, B, shifts, tol=1e-13)
        assert rc == 0
        check_solution(dims, mass, scale * U, B, shifts, X.cpu().numpy(), tol, Xo)
    ctx.close()
