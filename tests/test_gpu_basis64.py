"""The FP64 solve with the stored basis (csrc/basis64.cu): capacity reached in the middle of
a solve (updates in HBM from there on), widths whose rows leave idle lanes, and the summed
form of the rational solve, against the oracle and against the updates in HBM.

The criteria are those of the solver tests (true residuals and distance to the oracle's
solutions); the rational sums, solved to 1e-13, agree with the updates in HBM to 1e-12."""
import numpy as np
import pytest

import oracle
from gpu_util import check_solution, colrel, make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import _lib
from paper_1808_01829_gb300 import synthetic as syn
from paper_1808_01829_gb300.remez import rational_approx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 11, 16])
@pytest.mark.parametrize("cap", [0, 3, 14])
def test_shifted_solutions(n, cap):
    need_gpu()
    dims, mass, tol = (4, 6, 4, 4), 0.1, 1e-10
    shifts = [0.9, 0.01, 0.2, 4.0, 0.05, 30.0]
    U = syn.random_links(dims, 0.4, 1600)
    B = syn.gaussian_pseudofermions(dims, n, 2600 + n)
    ctx = make_ctx(dims, mass, U)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, cap)
    X, info = ctx.block_multishift_cg(to_gpu(B), shifts, tol, precision="fp64")
    order = np.argsort(shifts)  # the oracle takes ascending shifts
    Xs, _, _ = oracle.sbcgrq(dims, mass, U, B, [shifts[q] for q in order], tol=1e-13)
    Xo = np.empty_like(Xs)
    Xo[order] = Xs
    check_solution(dims, mass, U, B, shifts, X.cpu().numpy(), tol, Xo)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, 1)
    H, info1 = ctx.block_multishift_cg(to_gpu(B), shifts, tol, precision="fp64")
    assert info.iters == info1.iters
    check_solution(dims, mass, U, B, shifts, H.cpu().numpy(), tol, Xo)
    ctx.close()


@pytest.mark.parametrize("n,cap", [(2, 0), (4, 14), (7, 0), (16, 9)])
def test_rational_sum(n, cap):
    need_gpu()
    dims, mass, tol = (6, 4, 4, 4), 0.1, 1e-13
    ra = rational_approx(1.0 / 16, 1e-3, 64.0, 8)
    U = syn.random_links(dims, 0.4, 1601)
    Phi = syn.gaussian_pseudofermions(dims, n, 2700 + n)
    ctx = make_ctx(dims, mass, U)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, cap)
    Y, _ = ctx.rational_solve(to_gpu(Phi), ra.alpha0, ra.alpha, ra.beta, tol)
    ctx.tune_set(_lib.RHMC_TUNE_BASIS_ITERS, 1)
    Z, _ = ctx.rational_solve(to_gpu(Phi), ra.alpha0, ra.alpha, ra.beta, tol)
    assert colrel(Y.cpu().numpy(), Z.cpu().numpy()) <= 1e-12
    order = np.argsort(ra.beta)
    Xs, _, _ = oracle.sbcgrq(dims, mass, U, Phi, [ra.beta[q] for q in order], tol=1e-13)
    ref = ra.alpha0 * Phi + sum(ra.alpha[q] * x for q, x in zip(order, Xs))
    assert colrel(Y.cpu().numpy(), ref) <= 1e-10
    ctx.close()
