"""Decode calls with little work: their time has to follow the work.  Ratios of times on one GPU, not times: twice the queries
where the GPU has room for them, and a short list against a longer one."""
import pytest

from paper_2609_29812_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def time_of():
    """Time of a decode call of one layer (8192 positions, 16 heads, loop 4, a tenth of the rows with payloads), by the number
    of queries and columns: the best of several replays of a graph of 32 calls, the mean over four draws of the columns (how many
    payloads meet in one warp moves a short call by 10%), in us."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    L, H, loops, calls = 8192, 16, 4, 32
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=loops)
    ctx = B.Context(0)
    st = P.LayerState(ctx, w)
    rand = lambda *s: torch.randn(*s, device="cuda").to(torch.bfloat16)
    st.k_base, st.v_base = rand(L, H, 128), rand(L, H, 128)
    order = torch.randperm(L, device="cuda")
    for r in range(2, loops + 1):
        act = torch.sort(order[:L // 10])[0]
        slot = torch.full((L,), -1, dtype=torch.int32, device="cuda")
        slot[act] = torch.arange(len(act), dtype=torch.int32, device="cuda")
        sel = P.TokenSelection(act.to(torch.int32), slot, None, len(act))
        st.alloc_stream(sel, rows=False)
        st.quantize(r, rand(len(act), H, 128), rand(len(act), H, 128), sel)

    def one(queries, c):
        idx = torch.sort(torch.topk(torch.rand(queries * H, L, device="cuda"), c, dim=1)[1], dim=1)[0].to(torch.int32)
        cnt = torch.full((queries, H), c, dtype=torch.int32, device="cuda")
        q, lse, out = rand(3, queries, H, 128), torch.full((queries, H), 9.5, device="cuda"), rand(queries, H, 128)
        lse_out = torch.empty_like(lse)
        call = lambda: B.fl_decode_attention(ctx, st.shape, loops, q[0], q[1], queries, st.store, idx, cnt, c, lse, lse_out, q[2], out)
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

    def measure(queries, c):
        return sum(one(queries, c) for _ in range(4)) / 4
    yield measure
    ctx.close()


def test_more_queries_do_not_wait_for_a_second_wave(time_of):
    t2, t4 = time_of(2, 512), time_of(4, 512)
    assert t4 < 1.6 * t2, f"two queries {t2:.1f} us, four {t4:.1f} us"          # 1.32 (ten runs); 1.92 when a list was split too far


def test_a_short_list_takes_less_than_a_longer_one(time_of):
    t64, t512 = time_of(1, 64), time_of(1, 512)
    # halfway between 0.64 to 0.72 (ten runs) and the 0.84 of one form for all lists (11.9 and 14.1 us)
    assert t64 < 0.78 * t512, f"64 columns {t64:.1f} us, 512 columns {t512:.1f} us"
