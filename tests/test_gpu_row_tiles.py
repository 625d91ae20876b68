"""Loop attention on blocks of several 128-row tiles, which a group of CTAs shares: row counts just below, at and above whole
tiles, a short last block with fewer tiles than CTAs, with and without the carried old term."""
import pytest

from paper_2609_29812_b200 import workloads
from helpers import assert_attn_close, to_dev, to_np
from test_gpu_economy import run_oracle
from test_gpu_parity import oracle_selection, small_bf16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("L,q_block,k_tok", [(1024, 256, 513), (1100, 512, 1100), (1300, 1024, 330), (1537, 512, 769)])
def test_shared_row_tiles(L, q_block, k_tok):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    ctx = B.Context(0)
    w = workloads.replace(small_bf16(L=L, H=2, R=3), q_block=q_block)
    x = workloads.make_layer_inputs(w, seed=L)
    ref = run_oracle(w, x, k_tok=[k_tok] * 2)
    for carry in (False, True):
        st = P.LayerState(ctx, w)
        st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
        st.select_columns_dense()
        for r in (2, 3):
            rec, act = ref["loops"][r - 2], ref["active"][r - 2]
            sel = oracle_selection(P, w, ref, r)
            o_rows, _ = st.sparse_loop(r, to_dev(x.Q[r - 1][act], w), to_dev(x.K[r - 1][act], w),
                                       to_dev(x.V[r - 1][act], w), sel, indexed=True,
                                       carry=("write" if r == 2 else "reuse") if carry else None)
            st.check_status()
            assert_attn_close(to_np(o_rows), rec["O_rows"], f"loop {r} carry {carry}", carried=1 if carry else r - 1)
    ctx.close()
