"""Relative accuracy of the gauge force (a kick of P = 0) for strong, weak and nearly
block-diagonal links exp(i eps H), against extended precision.

Tolerance, per entry: a floating-point form rounds relative to the products it adds, so the
error of entry (i, j) is held to 32 x 2^-53 of S_ij + S_ji, S = |U| sum |X| |Y| |Z| over the six
staples with the entries' absolute values (three products of three-term complex sums, each at most
seven roundings, and the sum of six); on the diagonal, where only imaginary parts enter, to that
of the parts' products, the largest of the three."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

AXIS = {0: 3, 1: 2, 2: 1, 3: 0}


def _links(dims, kind, eps):
    lx, ly, lz, lt = dims
    h = np.random.default_rng(5).standard_normal((lt, lz, ly, lx, 4, 8))
    if kind == "block":  # colours 0 and 1 mix strongly, colour 2 weakly with them
        h[..., 3:7] *= eps
        eps = 0.8
    Y = (0.5j * eps / 16) * np.einsum("...a,aij->...ij", h, syn.gell_mann()).astype(np.clongdouble)
    E = np.eye(3, dtype=np.clongdouble)
    for k in range(18, 0, -1):
        E = np.eye(3) + _mm(Y, E) / k
    for _ in range(4):
        E = _mm(E, E)
    return np.ascontiguousarray(E.astype(np.complex128))


def _mm(a, b):
    return np.einsum("...ij,...jk->...ik", a, b)


def _dag(a):
    return np.conj(np.swapaxes(a, -1, -2))


def _staples(U, mu, dag):
    sh = lambda f, d, k: np.roll(f, -k, axis=AXIS[d])
    V = 0
    for nu in range(4):
        if nu != mu:
            n, m = U[..., nu, :, :], U[..., mu, :, :]
            V = V + _mm(_mm(sh(n, mu, 1), dag(sh(m, nu, 1))), dag(n))
            V = V + _mm(_mm(dag(sh(sh(n, mu, 1), nu, -1)), dag(sh(m, nu, -1))), sh(n, nu, -1))
    return V


@pytest.mark.parametrize("kind,eps", [("su3", e) for e in (3.0, 0.5, 0.3, 0.2, 0.1, 1e-2, 1e-4, 1e-8, 0.0)]
                         + [("block", e) for e in (0.2, 1e-2, 1e-5, 0.0)])
def test_force_relative_to_its_products(kind, eps):
    torch = need_gpu()
    from paper_1808_01829_gb300 import hmc

    dims = (6, 4, 2, 4)
    U = _links(dims, kind, eps)
    ctx = make_ctx(dims, 0.1, U)
    P = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    hmc.gauge_kick(ctx, to_gpu(U), P, -6.0, 1.0)  # P = TA(U V)
    P = P.cpu().numpy()
    ctx.close()
    X = U.astype(np.clongdouble)
    size, re, im = (f(U) for f in (lambda z: np.abs(z.real) + np.abs(z.imag), lambda z: np.abs(z.real),
                                   lambda z: np.abs(z.imag)))
    for mu in range(4):
        W = _mm(X[..., mu, :, :], _staples(X, mu, _dag))
        A = (W - _dag(W)) / 2
        A = A - np.trace(A, axis1=-2, axis2=-1)[..., None, None] / 3 * np.eye(3)
        err = np.abs(P[..., mu, :, :] - A).astype(float)
        turn = lambda z: np.swapaxes(z, -1, -2)
        S = _mm(size[..., mu, :, :], _staples(size, mu, turn))
        off = S + np.swapaxes(S, -1, -2)
        # real and imaginary parts apart: an imaginary product takes an odd number of the latter
        even, odd = re + im, re - im  # (a + b)(c + d) - (a - b)(c - d) = 2 (a d + b c)
        Dg = (_mm(even[..., mu, :, :], _staples(even, mu, turn)) - _mm(odd[..., mu, :, :], _staples(odd, mu, turn))) / 2
        dia = np.einsum("...ii->...i", Dg).max(-1)[..., None, None]
        bound = 32 * 2.0 ** -53 * np.where(np.eye(3, dtype=bool), dia, off)
        assert np.all(err <= bound), (mu, (err / np.where(bound > 0, bound, 1)).max())
