"""The link update exp(eps P) U where P alone is near the ends of the FP64 range (eps P is not),
and for P whose exponential is small (negative real parts), against a plain sum.

Tolerance: 1e-12 of the largest entry of each link's result: exp(Y) takes up to eight squarings of
a sum of unit size, 2^8 roundings of a three-term complex product (2^-53 x 2^8 x 8 = 2.3e-13), in
the kernel and in the reference."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def _check(P, eps, Y, decay=0.0):
    from paper_1808_01829_gb300 import hmc

    dims = (4, 2, 2, 6)
    U = syn.random_links(dims, 0.5, 1530)
    ctx = make_ctx(dims, 0.1, U)
    Ug = to_gpu(U)
    hmc.link_update(ctx, Ug, to_gpu(P), eps)
    E = np.broadcast_to(np.eye(3), Y.shape)
    for k in range(20, 0, -1):
        E = np.eye(3) + (Y / 64) @ E / k
    for _ in range(6):
        E = E @ E
    ref = np.exp(-decay) * (E @ U)
    err = np.abs(Ug.cpu().numpy() - ref).max((-1, -2))
    assert np.all(err <= 1e-12 * np.abs(ref).max((-1, -2)))
    ctx.close()


def _random():
    rng = np.random.default_rng(9)
    shape = (6, 2, 2, 4, 4, 3, 3)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


@pytest.mark.parametrize("power", [-130, -49, -51, 49, 51, 130])
def test_momenta_near_the_ends_of_the_range(power):
    need_gpu()
    H = _random()
    _check(H * 10.0 ** power, 0.1 / 10.0 ** power, 0.1 * H)

@pytest.mark.parametrize("decay", [0.1, 3.0, 30.0])
def test_small_exponentials(decay):
    need_gpu()
    H = 0.2 * _random()
    _check(10 * (H - decay * np.eye(3)), 0.1, H, decay)
