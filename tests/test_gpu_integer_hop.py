"""The FP64 operator on the integer units (csrc/fx.cuh): both launch forms (four lanes or one
per (site, right-hand side), Vh * n above or below 38912), remainders of the site tiles, and
the inputs that leave the integer form (zeros, infinities, NaN, subnormals, neighbours of
very different size), against the oracle and against the native FP64 kernel.

Tolerance: an output is a sum of 24 complex products of SU(3) entries (row norm 1) with values
held to 2^-55 of the largest neighbour, plus one FP64 rounding: below 100 x 2^-53 of the
neighbourhood's largest value, so 1e-13 relative per column for Gaussian fields."""
import numpy as np
import pytest

import oracle
from gpu_util import colrel, make_ctx, need_gpu, to_gpu

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 4), 1), ((4, 4, 4, 4), 16), ((2, 4, 6, 2), 3), ((8, 4, 6, 8), 5), ((8, 8, 8, 8), 11),
         ((12, 10, 8, 14), 5), ((12, 10, 8, 14), 7), ((14, 12, 8, 8), 16), ((24, 24, 24, 8), 1)]


NATIVE = 5  # RHMC_TUNE_NATIVE_FP64_RESIDUALS: the native FP64 kernel


@pytest.mark.parametrize("dims,n", CASES)
def test_operator_and_hop_match_the_oracle(dims, n):
    need_gpu()
    from paper_1808_01829_gb300 import synthetic as syn

    U = syn.random_links(dims, 0.5, 1400 + n)
    X = syn.gaussian_pseudofermions(dims, n, 2400 + n)
    ctx = make_ctx(dims, 0.05, U)
    Y = ctx.apply_mdagm_mrhs(to_gpu(X), 0.3, "fp64").cpu().numpy()
    assert colrel(Y, oracle.apply_A(dims, 0.05, U, X, sigma=0.3)) <= 1e-13
    for par in (0, 1):
        Z = ctx.hop(to_gpu(X), par, "df64")
        ctx.tune_set(NATIVE, 1)
        N = ctx.hop(to_gpu(X), par, "fp64")
        ctx.tune_set(NATIVE, 0)
        assert colrel(Z.cpu().numpy(), N.cpu().numpy()) <= 1e-13
    ctx.close()


@pytest.mark.parametrize("dims,n", [((4, 4, 4, 6), 3), ((12, 10, 8, 14), 7)])
@pytest.mark.parametrize("what", ["zero", "point", "huge", "subnormal", "spread", "nan", "inf"])
def test_special_inputs_match_native_fp64(dims, n, what):
    torch = need_gpu()
    from paper_1808_01829_gb300 import synthetic as syn

    X = syn.gaussian_pseudofermions(dims, n, 2500)
    rng = np.random.default_rng(3)
    if what == "zero":
        X = 0 * X
    elif what == "point":
        X = 0 * X
        X[5, 1, n - 1] = 1.0 - 2.0j
    elif what == "huge":
        X = X * 1e300
    elif what == "subnormal":
        X = X * 1e-310
    elif what == "spread":
        X = X * 2.0 ** rng.integers(-60, 60, size=(X.shape[0], 1, n))
    elif what == "nan":
        X[7, 2, 0] = np.nan
    elif what == "inf":
        X[9, 0, n - 1] = np.inf
    ctx = make_ctx(dims, 0.05, syn.random_links(dims, 0.5, 1401))
    Y = ctx.apply_mdagm_mrhs(to_gpu(X), 0.1, "fp64")
    ctx.tune_set(NATIVE, 1)
    N = ctx.apply_mdagm_mrhs(to_gpu(X), 0.1, "fp64")
    y, z = torch.view_as_real(Y).cpu().numpy(), torch.view_as_real(N).cpu().numpy()
    fine = np.isfinite(z)
    assert np.array_equal(fine, np.isfinite(y)) and np.array_equal(np.isnan(y), np.isnan(z))
    # per entry, relative to the largest value within two hops (the whole column where all sizes are alike)
    scale = np.abs(z[fine]).max() if fine.any() else 0.0
    assert np.abs(y[fine] - z[fine]).max(initial=0.0) <= 1e-13 * scale
    ctx.close()
