"""Dense loops over short prompts: their time has to follow the work.  Ratios of times on one GPU, not times: against a prompt that
fills it."""
import pytest

from paper_2609_29812_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def time_of(B, P, ctx, L, H, calls=16):
    """Best of several replays of a graph of `calls` dense loops without statistics, in us a call."""
    w = workloads.config2(L=L, n_heads=H)
    sh = P.shape_of(w)
    q, k, v = (torch.randn(L, H, 128, device="cuda").bfloat16() for _ in range(3))
    o, lse = torch.empty_like(q), torch.empty(H, L, device="cuda")
    call = lambda: B.fl_dense_loop_attention(ctx, sh, q, k, v, o, lse, None)
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(calls):
            call()
    best = float("inf")
    for _ in range(12):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / calls)
    return best


# halfway between the shares with a tile per CTA and those of pairs of tiles (0.114 and 0.147, 0.160 and 0.201, 0.245 and 0.305); many
# heads: between two CTAs per SM and one (0.11 to 0.14 and 0.21 to 0.28, 0.19 to 0.22 and 0.29 to 0.38 on two GPUs)
@pytest.mark.parametrize("L,H,share", [(129, 16, 0.130), (400, 16, 0.180), (1024, 4, 0.275), (64, 200, 0.175), (384, 96, 0.255)])
def test_short_prompts_do_not_wait_for_a_second_tile(L, H, share):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    ctx = B.Context(0)
    full, short = time_of(B, P, ctx, 4096, 16), time_of(B, P, ctx, L, H)
    ctx.close()
    assert short < share * full, f"{L} x {H}: {short:.2f} us, 4096 x 16: {full:.2f} us"
