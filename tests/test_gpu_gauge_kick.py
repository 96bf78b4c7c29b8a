"""The gauge-force kick's integer form (csrc/gauge.cu, k_gauge_momentum_fx) and its FP64 form
(links that are not SU(3)-sized, streams under capture), and the link update for matrices
that are not anti-Hermitian, against the trajectory oracle and a plain Taylor sum.

Tolerances: a staple sum is six products of three unit-size matrices, integers in units of
2^-54 rounded after each product: below 1e-14 of the largest entry of the kick; 1e-13 leaves
the FP64 form's roundings room.  The exponential's Taylor remainder is below 1e-19."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from oracle import trajectory as tr
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

BETA = 5.12


def _links(dims, what):
    rng = np.random.default_rng(7)
    U = syn.random_links(dims, 0.5, 1500)
    if what == "unit":
        U = syn.unit_links(dims)
    elif what == "scaled":
        U = 3.7 * U
    elif what == "small":
        U = 1e-3 * U
    elif what == "mixed":  # some links leave the integer form, their neighbours' kicks with them
        U = U.copy()
        U[0, 0, 1, 0, 2] *= 40.0
        U[-1, 0, 0, 1, 0] = 0.0
    elif what == "general":
        U = rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape)
    return np.ascontiguousarray(U)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 10), (8, 6, 4, 4)])
@pytest.mark.parametrize("what", ["su3", "unit", "scaled", "small", "mixed", "general"])
def test_kick_against_the_oracle(dims, what):
    need_gpu()
    from paper_1808_01829_gb300 import hmc

    U, P0, eps = _links(dims, what), tr.momenta(dims, 1501), 0.41
    ctx = make_ctx(dims, 0.1, U)
    P = to_gpu(P0)
    hmc.gauge_kick(ctx, to_gpu(U), P, BETA, eps)
    ref = P0 + eps * tr.momentum_force(U, tr.gauge_G(U, BETA))
    assert np.abs(P.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
    ctx.close()


def test_kick_under_capture_and_on_two_streams():
    torch = need_gpu()
    from paper_1808_01829_gb300 import hmc

    dims, eps = (4, 6, 4, 8), 0.2
    sets = [_links(dims, "su3"), _links(dims, "scaled")]
    ctx = make_ctx(dims, 0.1, sets[0])
    P0 = tr.momenta(dims, 1502)
    refs = [P0 + eps * tr.momentum_force(U, tr.gauge_G(U, BETA)) for U in sets]
    Us, Ps = [to_gpu(U) for U in sets], [to_gpu(P0), to_gpu(P0)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for U, P, s in zip(Us, Ps, streams):
        with torch.cuda.stream(s):
            hmc.gauge_kick(ctx, U, P, BETA, eps)
    torch.cuda.synchronize()
    for P, ref in zip(Ps, refs):
        assert np.abs(P.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
    P = to_gpu(P0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hmc.gauge_kick(ctx, Us[0], P, BETA, eps)
    P.copy_(to_gpu(P0))
    graph.replay()
    torch.cuda.synchronize()
    assert np.abs(P.cpu().numpy() - refs[0]).max() <= 1e-13 * np.abs(refs[0]).max()
    ctx.close()


@pytest.mark.parametrize("eps", [1e-9, 0.02, 0.3, 2.5])
def test_link_update_of_general_matrices(eps):
    need_gpu()
    from paper_1808_01829_gb300 import hmc

    dims = (4, 2, 2, 6)
    rng = np.random.default_rng(8)
    U = syn.random_links(dims, 0.5, 1503)
    P = 0.5 * (rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape))
    P[0, 0, 0, 0, 1] = 0.0
    ctx = make_ctx(dims, 0.1, U)
    Ug = to_gpu(U)
    hmc.link_update(ctx, Ug, to_gpu(P), eps)
    Y = eps * P / 256
    E = np.broadcast_to(np.eye(3), Y.shape)
    for k in range(16, 0, -1):
        E = np.eye(3) + Y @ E / k
    for _ in range(8):
        E = E @ E
    ref = E @ U
    # the plain sum's eight squarings leave it 256 roundings
    assert np.abs(Ug.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    ctx.close()
