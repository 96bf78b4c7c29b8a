"""The gauge-force kick where the device has no room for the links' integer form (592 bytes per
site): it runs in FP64 without it, as it does under capture.  Tolerance: the 1e-13 of
test_gpu_gauge_kick.py, against the same kick with room."""
import pytest

from gpu_util import make_ctx, need_gpu, to_gpu
from oracle import trajectory as tr
from paper_1808_01829_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_kick_without_room_for_the_integer_links():
    torch = need_gpu()
    from paper_1808_01829_gb300 import hmc

    dims, eps, beta = (16, 16, 32, 64), 0.1, 5.12  # 310 MB of integer links
    U = torch.from_numpy(syn.random_links((4, 4, 4, 4), 0.5, 1510)).cuda().repeat(16, 8, 4, 4, 1, 1, 1).contiguous()
    P0 = torch.from_numpy(tr.momenta((4, 4, 4, 4), 1511)).cuda().repeat(16, 8, 4, 4, 1, 1, 1).contiguous()
    small = make_ctx((4, 4, 4, 4), 0.1, syn.random_links((4, 4, 4, 4), 0.5, 1510))
    ref, out = P0.clone(), P0.clone()
    ctx = make_ctx(dims, 0.1, U.cpu().numpy())
    hmc.gauge_kick(ctx, U, ref, beta, eps)
    ctx.close()
    graph = torch.cuda.CUDAGraph()  # (loads the FP64 kernel)
    Us, Ps = to_gpu(syn.random_links((4, 4, 4, 4), 0.5, 1510)), to_gpu(tr.momenta((4, 4, 4, 4), 1511))
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        hmc.gauge_kick(small, Us, Ps, beta, eps)
    graph.replay()
    torch.cuda.synchronize()
    small.close()
    ctx = make_ctx(dims, 0.1, U.cpu().numpy())
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (260 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < 300 << 20
        hmc.gauge_kick(ctx, U, out, beta, eps)
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert (out - ref).abs().max().item() <= 1e-13 * ref.abs().max().item()
    ctx.close()
