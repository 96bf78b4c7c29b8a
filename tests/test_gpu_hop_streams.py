"""FP64 hops of one context on two streams at once, and as the first call of a captured stream
(nothing may be allocated there), below and above the size at which the input is converted in a
pass of its own (Vh * n = 38912), against the native FP64 kernel.  Tolerance as in test_gpu_integer_hop.py: 1e-13 per column for Gaussian fields."""
import pytest

from gpu_util import colrel, make_ctx, need_gpu, to_gpu
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

NATIVE = 5  # RHMC_TUNE_NATIVE_FP64_RESIDUALS
CASES = [((4, 6, 4, 8), 5), ((12, 10, 8, 14), 7), ((16, 16, 16, 16), 16)]


def _case(dims, n):
    U = syn.random_links(dims, 0.5, 1450)
    Xs = [to_gpu(syn.gaussian_pseudofermions(dims, n, 2450 + q)) for q in range(2)]
    ref = make_ctx(dims, 0.05, U)
    ref.tune_set(NATIVE, 1)
    Ys = [ref.hop(X, 1, "fp64").cpu().numpy() for X in Xs]
    ref.close()
    return make_ctx(dims, 0.05, U), Xs, Ys


@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("dims,n", CASES)
def test_two_streams(dims, n, precision):
    torch = need_gpu()
    ctx, Xs, refs = _case(dims, n)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = [[], []]
    for _ in range(8):
        for q, s in enumerate(streams):
            with torch.cuda.stream(s):
                outs[q].append(ctx.hop(Xs[q], 1, precision))
    torch.cuda.synchronize()
    for out, ref in zip(outs, refs):
        for Y in out:
            assert colrel(Y.cpu().numpy(), ref) <= 1e-13
    ctx.close()


@pytest.mark.parametrize("dims,n", CASES)
def test_first_call_under_capture(dims, n):
    torch = need_gpu()
    ctx, Xs, refs = _case(dims, n)
    X = Xs[0].clone()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        Y = ctx.hop(X, 1, "fp64")
    ctx.apply_mdagm_mrhs(X, 0.1, "fp64")  # another call's scratch does not concern the graph
    for q in range(2):
        X.copy_(Xs[q])
        graph.replay()
        torch.cuda.synchronize()
        assert colrel(Y.cpu().numpy(), refs[q]) <= 1e-13
    ctx.close()


@pytest.mark.parametrize("dims,n", CASES)
def test_operator_under_capture_with_the_pool_of_a_mixed_hop(dims, n):
    """The pool that a mixed hop left holds the intermediate field of an FP64 operator application and
    no more; under capture it cannot grow."""
    torch = need_gpu()
    ctx, Xs, _ = _case(dims, n)
    ctx.hop(Xs[0], 1, "mixed")
    X = Xs[0].clone()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        Y = ctx.apply_mdagm_mrhs(X, 0.2, "fp64")
    X.copy_(Xs[1])
    graph.replay()
    torch.cuda.synchronize()
    y = Y.cpu().numpy()
    ctx.tune_set(NATIVE, 1)
    assert colrel(y, ctx.apply_mdagm_mrhs(Xs[1], 0.2, "fp64").cpu().numpy()) <= 1e-13
    ctx.close()
