"""Accuracy of the FP64 operator and hop per component (csrc/fx.cuh): colours of very different
size under unit, weak and block-diagonal links, sites of different size, single colours, links with
small rows, on lattices below and above the size at which the input is converted in a pass of its own.

Reference: the native FP64 kernel, whose error is below 30 x 2^-53 of S per hop, S the same hop
of the entries' absolute values.  An integer sum of 24 products with |v| < 2^E loses at most
77 x 2^-55 x 2^(E + 1) (values, links and their alignment truncated at 2^-55, products of low words);
it is taken only where S >= 0.4 x 2^(E - 4), so it is within 1600 x 2^-53 of S, twice that with the
rounding of the intermediate field: 4e-13 S per hop, 8e-13 for an operator application."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

NATIVE = 5  # RHMC_TUNE_NATIVE_FP64_RESIDUALS


def _weak(dims, eps):
    """Links exp(i eps H) whose small entries are accurate."""
    H = np.einsum("...a,aij->...ij", np.random.default_rng(6).standard_normal(dims[::-1] + (4, 8)), syn.gell_mann())
    Y, E = 0.5j * eps * H, np.eye(3)
    for k in range(12, 0, -1):
        E = np.eye(3) + Y @ E / k
    return E


def _links(dims, kind):
    U = syn.random_links(dims, 0.5, 1460)
    if kind == "unit":
        U = syn.unit_links(dims)
    elif kind == "weak":
        U = _weak(dims, 1e-6)
    elif kind == "block":  # colour 2 apart from the others but for 1e-9
        B = np.zeros_like(U)
        B[..., :2, :2], B[..., 2, 2] = U[..., :2, :2], 1.0
        B[..., 2, 0], B[..., 1, 2] = 1e-9, 1e-9j
        U = B
    elif kind == "small rows":
        U = U.copy()
        U[..., 3, :, :] *= 1e-7
        U[0, 0, 0, 1, 2, 1, :] = 0.0
    return np.ascontiguousarray(U)


def _field(dims, n, kind):
    X = syn.gaussian_pseudofermions(dims, n, 2460)
    rng = np.random.default_rng(4)
    if kind == "colours":
        X = X * np.array([1.0, 1e-8, 1e-17])[:, None]
    elif kind == "steps":  # every distance of two colours' sizes up to 2^20
        X = X * 2.0 ** (np.array([0.0, -1.0, 0.0])[:, None] * (np.arange(X.shape[0]) % 21)[:, None, None])
    elif kind == "one colour":
        X = X * np.array([0.0, 1.0, 0.0])[:, None]
    elif kind == "sites":
        X = X * 2.0 ** rng.integers(-60, 60, size=(X.shape[0], 1, n))
    elif kind == "point":
        Z = 0 * X
        Z[5], Z[7, 2] = X[5], 1e-12 * X[7, 2]
        X = Z
    return X


def _abs_hop(dims, U, X, par):
    """sum_mu |U_mu(x)| |X(x + mu)| + |U_mu(x - mu)|^T |X(x - mu)| at the sites of parity par."""
    lx, ly, lz, lt = dims
    t, z, y, x = np.meshgrid(np.arange(lt), np.arange(lz), np.arange(ly), np.arange(lx), indexing="ij")
    odd = (x + y + z + t) % 2 == 1
    F = np.zeros((lt, lz, ly, lx) + X.shape[1:])
    other = odd if par == 0 else ~odd
    F[other] = X  # (x fastest: the order of a parity's sites)
    out = 0
    for mu in range(4):
        ax = 3 - mu
        u = np.abs(U[..., mu, :, :])
        out = out + np.einsum("...ab,...bn->...an", u, np.roll(F, -1, ax))
        out = out + np.roll(np.einsum("...ba,...bn->...an", u, F), 1, ax)
    return out[odd if par else ~odd]


@pytest.mark.parametrize("dims,n", [((4, 6, 4, 4), 3), ((12, 10, 8, 14), 7)])
@pytest.mark.parametrize("links", ["su3", "unit", "weak", "block", "small rows"])
@pytest.mark.parametrize("field", ["gauss", "colours", "steps", "one colour", "sites", "point"])
def test_against_the_sum_of_absolute_values(dims, n, links, field):
    need_gpu()
    U, X = _links(dims, links), _field(dims, n, field)
    ctx = make_ctx(dims, 0.05, U)
    hop, op = [], []
    for native in (0, 1):
        ctx.tune_set(NATIVE, native)
        hop.append(ctx.hop(to_gpu(X), 1, "fp64").cpu().numpy())
        op.append(ctx.apply_mdagm_mrhs(to_gpu(X), 0.3, "fp64").cpu().numpy())
    ctx.close()
    S1 = _abs_hop(dims, U, np.abs(X), 1)
    S2 = (4 * 0.05 ** 2 + 0.3) * np.abs(X) + _abs_hop(dims, U, S1, 0)
    assert np.all(np.abs(hop[0] - hop[1]) <= 4e-13 * S1)
    assert np.all(np.abs(op[0] - op[1]) <= 8e-13 * S2)
