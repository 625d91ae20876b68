"""fl_decode_attention at the edges of its tensor-core path: tiles of 16 columns, lists split over a cluster of CTAs, columns
with and without payloads, one to four residual streams (and a fifth, which takes the general kernel), against the oracle."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200 import workloads
from helpers import assert_attn_close, to_dev, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("c,loops,bits,group", [(1, 2, 4, 128), (16, 3, 8, 64), (17, 2, 2, 32), (127, 4, 4, 32), (513, 5, 4, 128),
                                                (1100, 3, 16, 128), (257, 6, 4, 64)])
def test_tile_and_split_edges(c, loops, bits, group):
    run_case(c, loops, bits, group)


# pieces of at most a tile per warp, columns dealt evenly over the warps (few problems) or by whole tiles (many), no payload,
# some or nearly all columns with one, and the first sizes past them
@pytest.mark.parametrize("c,loops,bits,group,Bq,frac", [(3, 5, 8, 16, 3, 0.75), (63, 4, 4, 128, 2, 0.75), (64, 5, 2, 8, 2, 0.1),
                                                        (64, 2, 16, 128, 3, 0.3), (65, 3, 4, 64, 2, 0.75), (200, 5, 16, 128, 3, 0.75),
                                                        (20, 4, 4, 32, 130, 0.3), (64, 3, 8, 64, 120, 0.75), (50, 2, 4, 8, 240, 0.1),
                                                        (70, 4, 2, 64, 120, 0.3), (512, 4, 8, 128, 4, 0.1), (130, 5, 4, 16, 40, 0.5)])
def test_short_pieces(c, loops, bits, group, Bq, frac):
    run_case(c, loops, bits, group, Bq, frac)


def run_case(c, loops, bits, group, Bq=3, frac=0.75):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    rng = np.random.default_rng(c)
    L, H, dh = 1300, 2, 128
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=loops, bits=bits, group=group)
    bf = fo.round_bf16
    ctx = B.Context(0)
    st = P.LayerState(ctx, w)
    k1, v1 = (bf(rng.standard_normal((L, H, dh)).astype(np.float32)) for _ in range(2))
    st.k_base, st.v_base = to_dev(k1, w), to_dev(v1, w)
    order = rng.permutation(L)
    khat, vhat, k_prev, v_prev = k1.copy(), v1.copy(), None, None
    for r in range(2, loops + 1):                       # nested sets, from `frac` of the rows down
        act = np.sort(order[: int(frac * L / (r - 1))])
        kr, vr = (bf(x[act] + 0.3 * rng.standard_normal((len(act), H, dh)).astype(np.float32)) for x in (khat, vhat))
        sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(),
                               torch.from_numpy(fo.slot_map(act, L).astype(np.int32)).cuda(), None, len(act))
        st.alloc_stream(sel, rows=False)
        st.quantize(r, to_dev(kr, w), to_dev(vr, w), sel)
        k_prev, v_prev = khat, vhat
        khat, _ = fo.residual_update(kr, khat, act, bits, group)
        vhat, _ = fo.residual_update(vr, vhat, act, bits, group)
    q_old, q_new, o1 = (bf(rng.standard_normal((Bq, H, dh)).astype(np.float32)) for _ in range(3))
    col_idx = np.full((Bq, H, c), -1, dtype=np.int32)
    col_cnt = np.zeros((Bq, H), dtype=np.int32)
    sets, p_old = {}, {}
    lse = np.zeros((Bq, H))
    for t in range(Bq):
        for h in range(H):
            n = [c, max(0, c - 1), c // 2, min(c, 15), min(c, 16), 0][(t * H + h) % 6]
            S = np.sort(rng.permutation(L)[:n])
            col_idx[t, h, :n], col_cnt[t, h], sets[(t, h)] = S, n, S
            logits = (bf(k_prev[:, h]).astype(np.float64) @ q_old[t, h].astype(np.float64)) * w.sm_scale
            lse[t, h] = logits.max() + np.log(np.exp(logits - logits.max()).sum())
            p_old[(t, h)] = np.exp(logits[S] - lse[t, h])
    ref = fo.decode_sparse_attention(q_new, khat, vhat, v_prev, o1, sets, p_old, w.sm_scale, kv_round=bf)
    o, p_new = torch.zeros(Bq, H, dh, dtype=torch.bfloat16, device="cuda"), torch.full((Bq, H, c), 7.0, device="cuda")
    lse_out = torch.zeros(Bq, H, device="cuda")
    lse_in = torch.from_numpy(lse.astype(np.float32)).cuda()
    B.fl_decode_attention(ctx, st.shape, loops, to_dev(q_new, w), to_dev(q_old, w), Bq, st.store,
                          torch.from_numpy(col_idx).cuda(), torch.from_numpy(col_cnt).cuda(), c, lse_in, lse_out,
                          to_dev(o1, w), o, p_new)
    torch.cuda.synchronize()
    assert_attn_close(to_np(o), ref["O"], f"decode tiles c={c} loops={loops}", carried=1)
    got = to_np(p_new)
    for (t, h), pn in ref["p_new"].items():
        np.testing.assert_allclose(got[t, h, : len(pn)], pn, rtol=2e-3, atol=1e-7)
        assert np.all(got[t, h, len(pn):] == 0)
        want = ref["lse"][t, h] if len(pn) else lse[t, h]
        assert abs(to_np(lse_out)[t, h] - want) < 2e-3
    ctx.close()
