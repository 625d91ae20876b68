"""The quantizers at the edges of their kernels' ranges, bit for bit against the oracle: residual streams up to the ninth
(pipelined up to seven earlier ones, general beyond), row widths on both sides of the 16-element form, and the packed base
with short token groups, masks and every group size."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200 import workloads
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding, pipeline
    ctx = binding.Context(0)
    yield binding, pipeline, ctx
    ctx.close()


@pytest.mark.parametrize("H,bits,group,loops,n", [(4, 4, 128, 10, 37), (4, 2, 16, 9, 700), (8, 8, 64, 5, 300), (6, 4, 32, 4, 90),
                                                  (2, 8, 8, 3, 1), (4, 4, 8, 3, 65)])
def test_residual_chain_bit_exact(env, H, bits, group, loops, n):
    B, P, ctx = env
    rng = np.random.default_rng(n)
    L = 900
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=loops, bits=bits, group=group)
    st = P.LayerState(ctx, w, split=False)
    base = fo.round_bf16(rng.standard_normal((L, H, 128)).astype(np.float32))
    st.k_base, st.v_base = to_dev(base, w), to_dev(base[::-1].copy(), w)
    xhat = {"k": base, "v": base[::-1].copy()}
    order = rng.permutation(L)
    for r in range(2, loops + 1):
        act = np.sort(order[: max(1, n - (r - 2) * (n // 12))])
        new = {s: fo.round_bf16(xhat[s][act] + rng.standard_normal((len(act), H, 128)).astype(np.float32) *
                                10.0 ** rng.integers(-4, 2, (len(act), 1, 1)).astype(np.float32)) for s in "kv"}
        new["k"][0, 0, :] = fo.round_bf16(xhat["k"][act[0], 0, :])      # no change at all in the first loop: constant groups
        sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(),
                               torch.from_numpy(fo.slot_map(act, L).astype(np.int32)).cuda(), None, len(act))
        st.alloc_stream(sel)
        st.quantize(r, to_dev(new["k"], w), to_dev(new["v"], w), sel)
        torch.cuda.synchronize()
        for s, streams in (("k", st.k_streams), ("v", st.v_streams)):
            got = streams[-1]
            nxt, pay = fo.residual_update(new[s], xhat[s], act, bits, group)
            assert np.array_equal(to_np(got["codes"]), pay["packed"].reshape(len(act), -1)), (r, s)
            for m in ("scale", "zero"):
                assert np.array_equal(to_np(got[m]).view(np.uint16), pay[m].reshape(len(act), -1).view(np.uint16)), (r, s, m)
            assert np.array_equal(to_np(got["rows_prev"]), fo.round_bf16(xhat[s][act]).reshape(len(act), -1)), (r, s)
            assert np.array_equal(to_np(got["rows_cur"]), fo.round_bf16(nxt[act]).reshape(len(act), -1)), (r, s)
            xhat[s] = nxt


@pytest.mark.parametrize("Lq,group,bits,dtype", [(1, 64, 4, "bf16"), (31, 32, 2, "bf16"), (129, 128, 8, "bf16"), (700, 64, 2, "bf16"),
                                                 (333, 128, 4, "f32"), (65, 32, 8, "f32")])
def test_packed_base_and_masked_rebuild(env, Lq, group, bits, dtype):
    B, P, ctx = env
    rng = np.random.default_rng(Lq)
    H, dh = (2, 128) if dtype == "bf16" else (4, 64)
    L = Lq + 5
    w = workloads.replace(workloads.config2(L=L, n_heads=H), head_dim=dh, dtype=dtype, bits=bits, group=min(group, dh))
    rnd = fo.round_bf16 if dtype == "bf16" else (lambda a: a)
    k, v = (rnd(rng.standard_normal((L, H * dh)).astype(np.float32)) for _ in range(2))
    k[:, 3] = 0.25                                                  # a constant channel
    ref = fo.quantize_base(k, v, bits, group, 5, storage_round=rnd if dtype == "bf16" else None)
    st = P.LayerState(ctx, w, split=False)
    kd, vd = to_dev(k.reshape(L, H, dh), w), to_dev(v.reshape(L, H, dh), w)
    st.pack_base(kd, vd, group, 5)
    kc, ks, kz, vc, vs, vz, kt, vt = [to_np(t) for t in st.base_tensors]
    assert np.array_equal(kc, fo.pack_codes(ref["k_codes"], bits)) and np.array_equal(vc, fo.pack_codes(ref["v_codes"], bits))
    for got, name in ((ks, "k_scale"), (kz, "k_zero"), (vs, "v_scale"), (vz, "v_zero")):
        assert np.array_equal(got.view(np.uint16), ref[name].view(np.uint16)), name
    assert np.array_equal(kt, k[Lq:]) and np.array_equal(vt, v[Lq:])
    for mask in (None, rng.random((H, L)) < 0.4):
        k_out, v_out = torch.full_like(kd, 9.0), torch.full_like(vd, 9.0)
        words = None
        if mask is not None:
            bits_ = np.zeros((H, (L + 31) // 32 * 32), dtype=np.uint8)
            bits_[:, :L] = mask
            words = torch.from_numpy(np.packbits(bits_, axis=1, bitorder="little").view(np.int32).copy()).cuda()
        B.fl_dequant_kv_base(ctx, st.shape, st.base_q, k_out, v_out, row_mask=words)
        torch.cuda.synchronize()
        for got, want in ((k_out, ref["khat"]), (v_out, ref["vhat"])):
            want = want.reshape(L, H, dh).copy()
            if mask is not None:
                want[:Lq][~mask.T[:Lq]] = 9.0
            assert np.array_equal(to_np(got), want)
