"""The gauge-force kick at the edges of its integer form's range (csrc/gauge.cu): staple sums
around 8, where both parts of an entry fill their high words, against the trajectory oracle.
Tolerance: the 1e-13 of test_gpu_gauge_kick.py, relative to the largest entry; a wrapped sum is
wrong by its whole size."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from oracle import trajectory as tr
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [-1e-8, 0.0, 1e-9, 3.7e-9, 3.8e-9, 1e-6, 0.5])
@pytest.mark.parametrize("entry", [0, 2])
def test_staple_sums_around_eight(gap, entry):
    need_gpu()
    from paper_1808_01829_gb300 import hmc

    dims, beta = (4, 2, 4, 2), 5.12
    U = syn.unit_links(dims)
    # the links of direction 1 are the conjugate of a sixth of the staple sum (8 - gap)(1 + i)
    U[..., 1, entry, entry] = (8 - gap) / 6 * (1 - 1j)
    U[0, 0, 0, 0, 1] = np.eye(3)  # (with the conjugate itself the wrapped word is multiplied by zero)
    ctx = make_ctx(dims, 0.1, U)
    P0 = tr.momenta(dims, 1520)
    P = to_gpu(P0)
    hmc.gauge_kick(ctx, to_gpu(U), P, beta, 0.3)
    ref = P0 + 0.3 * tr.momentum_force(U, tr.gauge_G(U, beta))
    assert np.abs(P.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
    ctx.close()
