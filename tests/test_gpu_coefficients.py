"""The n x n coefficient kernels of the FP64 solve at every width: Gram partials summed as
integers by them or added by their own kernel, the factorisation's real and imaginary parts on
warps of their own, and the stored basis's coefficients column by column.  Columns of very
different size give partials of very different exponents.  Criteria of the solver tests: true
residuals by the oracle's operator, distance to the oracle's solutions."""
import numpy as np
import pytest

import oracle
from gpu_util import check_solution, make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

# (enough rows that the Krylov space, rows / n blocks, is not used up before convergence)
SMALL = [((6, 2, 2, 2), n) for n in (1, 2, 3)] + [((6, 4, 4, 6), n) for n in range(1, 17)]
LARGE = [((12, 10, 6, 14), n) for n in (1, 2, 4, 5, 8, 16)]


@pytest.mark.parametrize("dims,n", SMALL + LARGE)
def test_fp64_solve(dims, n):
    need_gpu()
    mass, tol, shifts = 0.15, 1e-10, [0.02, 0.3, 2.0]
    U = syn.random_links(dims, 0.4, 1750)
    B = syn.gaussian_pseudofermions(dims, n, 2850 + n) * 10.0 ** (((np.arange(n) * 7) % 11) - 5)
    ctx = make_ctx(dims, mass, U)
    X, info = ctx.block_multishift_cg(to_gpu(B), shifts, tol, precision="fp64")
    assert info.true_rel_resid_max <= tol
    Xo, _, _ = oracle.sbcgrq(dims, mass, U, B, shifts, tol=1e-13)
    check_solution(dims, mass, U, B, shifts, X.cpu().numpy(), tol, Xo)
    ctx.close()
