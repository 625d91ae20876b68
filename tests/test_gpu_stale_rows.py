"""Shrinking token sets: rows of tokens whose payloads are all from earlier loops, rebuilt once per launch when the workspace
has room for them.  Every code width, few and many heads, against the oracle and against the chain
inside the kernels (a context without a workspace)."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200 import workloads
from helpers import assert_attn_close, to_dev, to_np
from test_gpu_economy import run_oracle
from test_gpu_parity import oracle_selection, small_bf16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bits,group,H,L,loops", [(4, 128, 2, 700, 4), (2, 32, 4, 1201, 3), (8, 64, 2, 903, 4), (16, 128, 2, 700, 3),
                                                  (4, 32, 2, 803, 7)])
def test_rows_of_dropped_tokens(bits, group, H, L, loops):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=loops, q_block=256, col_budget=96, bits=bits, group=group,
                          changed_fracs=tuple(0.5 * 0.6 ** i for i in range(loops - 1)))
    x = workloads.make_layer_inputs(w, seed=L)
    k_tok = [max(8, int(L * 0.4 * 0.6 ** i)) for i in range(loops - 1)]
    ref = run_oracle(w, x, k_tok=k_tok)
    scores = {}
    for lent in (True, False):
        ctx = B.Context(0)
        st = P.LayerState(ctx, w, split=lent)
        assert not lent or B.fl_loop_attention_full_workspace_bytes(ctx, st.shape) >= 4 * L * w.d
        st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
        st.select_columns_dense()
        for r in range(2, loops + 1):
            rec, act = ref["loops"][r - 2], ref["active"][r - 2]
            sel = oracle_selection(P, w, ref, r)
            st.alloc_stream(sel)
            st.quantize(r, to_dev(x.K[r - 1][act], w), to_dev(x.V[r - 1][act], w), sel)
            csn = torch.zeros(H, st.nb, st.c, device="cuda")
            B.fl_loop_attention_indexed(ctx, st.shape, r, to_dev(x.Q[r - 1][act], w), st.q_store, st.q_store, sel.active_idx, sel.n,
                                        st.store, st.col_idx, st.col_cnt, st.c, st.lse, st.lse, st.o_store, st.o_store, csn,
                                        status=st.status)
            st.check_status()
            assert_attn_close(to_np(st.o_store)[act], rec["O_rows"], f"loop {r} lent {lent}", carried=r - 1)
            scores[r, lent] = csn
        ctx.close()
    for r in range(2, loops + 1):
        torch.testing.assert_close(scores[r, True], scores[r, False], rtol=2e-2, atol=1e-4)


@pytest.mark.parametrize("bits,group", [(2, 8), (2, 16), (2, 128), (4, 8), (4, 16), (4, 32), (8, 8), (8, 16), (8, 64), (16, 8)])
def test_rebuilt_rows_bit_exact(bits, group):
    """The rows behind the split's part of the workspace, on both sides of the 32 elements that a lane rebuilds at a time (one
    scale and offset, or one per 8 elements): the binary32 chain of the oracle, rounded once to bf16."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    rng = np.random.default_rng(bits * 256 + group)
    L, H, dh, loops = 421, 2, 128, 4
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=loops, q_block=256, col_budget=64, bits=bits, group=group)
    bf = fo.round_bf16
    draw = lambda n: bf(rng.standard_normal((n, H, dh)).astype(np.float32))
    ctx = B.Context(0)
    st = P.LayerState(ctx, w)
    hat = {"k": draw(L), "v": draw(L)}
    st.dense_loop(to_dev(draw(L), w), to_dev(hat["k"], w), to_dev(hat["v"], w))
    st.select_columns_dense()
    order, seen = rng.permutation(L), np.zeros(L, dtype=bool)
    for r in range(2, loops + 1):                       # nested sets: 60%, 30%, 20% of the rows
        act = np.sort(order[: int(0.6 * L / (r - 1))])
        new = {s: bf(hat[s][act] + 0.3 * draw(len(act))) for s in "kv"}
        sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(),
                               torch.from_numpy(fo.slot_map(act, L).astype(np.int32)).cuda(), None, len(act))
        st.alloc_stream(sel)
        st.quantize(r, to_dev(new["k"], w), to_dev(new["v"], w), sel)
        st.attention_indexed(r, to_dev(draw(len(act)), w), sel)
        st.check_status()
        for s in "kv":
            hat[s], _ = fo.residual_update(new[s], hat[s], act, bits, group)
        stale = np.setdiff1d(np.flatnonzero(seen), act)
        seen[act] = True
        if len(stale) == 0:
            continue
        full = B.fl_loop_attention_full_workspace_bytes(ctx, st.shape)
        rows = to_np(ctx._workspace[full - 4 * L * w.d:full].view(torch.bfloat16).view(2, L, H, dh))
        for i, s in enumerate("kv"):
            assert np.array_equal(rows[i, stale], bf(hat[s][stale])), (r, s)
    ctx.close()


def test_room_for_rows_comes_with_the_first_set_that_shrinks():
    """Sets of one size: the split's part of the workspace alone.  The first smaller set: room for the rebuilt rows, and what
    the context held before stays allocated (a captured graph may use it).  A detached context gets nothing."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    w = workloads.replace(workloads.config2(L=2000, n_heads=2), n_loops=4, q_block=256, col_budget=96)
    base = torch.zeros(w.L, 2, 128, dtype=torch.bfloat16, device="cuda")

    def sel(n):
        idx = torch.arange(n, dtype=torch.int32, device="cuda")
        return P.TokenSelection(idx, torch.full((w.L,), -1, dtype=torch.int32, device="cuda"), None, n)
    for split in (True, False):
        ctx = B.Context(0)
        st = P.LayerState(ctx, w)
        need, full = B.fl_loop_attention_workspace_bytes(ctx, st.shape), B.fl_loop_attention_full_workspace_bytes(ctx, st.shape)
        assert 0 < need < full and ctx._workspace.numel() == need
        st.k_base = st.v_base = base
        st.alloc_stream(sel(200))
        st.alloc_stream(sel(200))
        before = ctx._workspace
        assert before.numel() == need
        if not split:
            P.LayerState(ctx, w, split=False)
        st.alloc_stream(sel(100))
        if split:
            assert ctx._workspace.numel() == full and ctx._workspace_before is before and not ctx._workspace[:1024].any()
            assert ctx._lent == (ctx._workspace.data_ptr(), full)
        else:
            assert ctx._workspace is None and ctx._lent is None
        ctx.close()
