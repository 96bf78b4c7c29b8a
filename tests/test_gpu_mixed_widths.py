"""Mixed-precision solves at every width: row groups per warp in the base step and the fused
block QR step (n <= 8), row slices of the Gram kernel (n <= 4), Gram partials summed by the
coefficient kernels (few CTAs) or by their own kernel, and ragged last row tiles.  Criteria of
the solver tests: true residuals by the oracle's operator, distance to the oracle's solutions."""
import pytest

import oracle
from gpu_util import check_solution, make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

SMALL = [((6, 2, 2, 2), n) for n in (1, 2, 3)] + [((6, 4, 2, 6), n) for n in range(1, 17)]
LARGE = [((12, 10, 6, 14), n) for n in (1, 2, 3, 4, 5, 8, 16)]


@pytest.mark.parametrize("dims,n", SMALL + LARGE)
def test_mixed_solve(dims, n):
    need_gpu()
    mass, tol, shifts = 0.15, 1e-9, [0.02, 0.3, 2.0]
    U = syn.random_links(dims, 0.4, 1700)
    B = syn.gaussian_pseudofermions(dims, n, 2800 + n)
    ctx = make_ctx(dims, mass, U)
    X, info = ctx.block_multishift_cg(to_gpu(B), shifts, tol, precision="mixed")
    assert info.true_rel_resid_max <= tol
    Xo, _, _ = oracle.sbcgrq(dims, mass, U, B, shifts, tol=1e-13)
    check_solution(dims, mass, U, B, shifts, X.cpu().numpy(), tol, Xo)
    ctx.close()
