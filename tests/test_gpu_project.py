"""GPU parity of fl_project_rows (one tensor-core GEMM with gathered A rows and an indexed, optionally accumulating
epilogue) against the oracle's fp64 projection of the listed rows (Section 4.4 / Appendix G).

Tolerance, element by element: the inputs are bf16 on both sides, the kernel accumulates in binary32 and rounds each
output once to bf16, so |got - ref| <= 2^-8 |ref| (half a bf16 ulp, relative to the value's binade) + the binary32
accumulation bound d_in * 2^-23 * sum_k |x_k w_k|."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200.workloads import round_to_bf16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding
    ctx = binding.Context(0)
    yield binding, ctx
    ctx.close()


def dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    return t.to(dtype) if dtype is not None else t


def make(seed, x_rows, y_rows, n, d_in, d_out, gather, scatter):
    rng = np.random.default_rng(seed)
    x = round_to_bf16(rng.standard_normal((x_rows, d_in)).astype(np.float32))
    w = round_to_bf16((rng.standard_normal((d_out, d_in)) / np.sqrt(d_in)).astype(np.float32))
    y = round_to_bf16(rng.standard_normal((y_rows, d_out)).astype(np.float32))
    src = np.sort(rng.choice(x_rows, size=n, replace=False)).astype(np.int32) if gather else None
    dst = np.sort(rng.choice(y_rows, size=n, replace=False)).astype(np.int32) if scatter else None
    return x, w, y, src, dst


def check(B, ctx, x, w, y, src, dst, n, accumulate, rows=None):
    d_in, d_out = x.shape[1], w.shape[0]
    xd, wd, yd = dev(x, torch.bfloat16), dev(w, torch.bfloat16), dev(y, torch.bfloat16)
    sd = dev(src) if src is not None else None
    dd = dev(dst) if dst is not None else None
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    B.fl_project_rows(ctx, xd, x.shape[0], sd, n, d_in, wd, d_out, yd, y.shape[0], dd, accumulate, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = yd.float().cpu().numpy()
    touched = (dst if dst is not None else np.arange(n)).astype(np.int64)
    mask = np.ones(y.shape[0], dtype=bool)
    mask[touched] = False
    assert np.array_equal(got[mask], y[mask]), "rows that are not listed must stay bit-identical"
    # the oracle, on all listed rows or on a sample of them
    pick = np.arange(n) if rows is None else rows
    s_pick = (src[pick] if src is not None else pick)
    d_pick = (dst[pick] if dst is not None else pick)
    ref = fo.project_rows(x, s_pick, w, y, d_pick, bool(accumulate))[d_pick]
    mag = np.abs(x[s_pick].astype(np.float64)) @ np.abs(w.astype(np.float64)).T
    bound = 2.0 ** -8 * np.abs(ref) + d_in * 2.0 ** -23 * (mag + np.abs(y[d_pick])) + 1e-30
    err = np.abs(got[d_pick].astype(np.float64) - ref)
    worst = float(np.max(err / bound))
    assert worst <= 1.0, f"worst error / bound = {worst:.3f}"
    return worst


@pytest.mark.parametrize("gather,scatter,accumulate", [(True, False, 0), (False, True, 1), (True, True, 0),
                                                       (True, True, 1), (False, False, 0)])
def test_project_rows_ragged_tiles(env, gather, scatter, accumulate):
    B, ctx = env
    n = 300                                     # 2 full row tiles + 44 rows
    x, w, y, src, dst = make(7, 1000 if gather else n, 1000 if scatter else n, n, 256, 520, gather, scatter)
    check(B, ctx, x, w, y, src, dst, n, accumulate)       # d_out = 2 x 256 + 8: a ragged column tile


def test_project_rows_several_tiles_per_cta(env):
    """357 wide output tiles (21 x 17, the last column tile 8 columns wide, the last row tile 40 rows high) on at most
    148 CTAs: two or three tiles each, so both accumulators are reused and the stage ring wraps many times (where pairs of
    CTAs run it, with tiles of 224 columns, about as many per pair)."""
    B, ctx = env
    n = 2600
    x, w, y, src, dst = make(8, 4000, 4000, n, 512, 4104, True, True)
    rows = np.sort(np.random.default_rng(1).choice(n, size=400, replace=False))
    check(B, ctx, x, w, y, src, dst, n, 1, rows=rows)


@pytest.mark.parametrize("n,d_out,gather,scatter,accumulate", [
    (1229, 2056, False, True, 1),    # one round; the last tile's second half starts beyond the last column
    (2500, 3000, True, True, 0),     # two tiles per pair, gathered; 88 columns in a last tile of 224
    (2561, 2048, False, True, 1),    # the last 256 rows hold one: nothing for the second CTA
    (3277, 6144, True, False, 0),
])
def test_project_rows_pairs_of_ctas(env, n, d_out, gather, scatter, accumulate):
    """Sizes for which pairs of CTAs share a tile: ragged rows and columns, accumulators used in turn."""
    B, ctx = env
    args = make(29, 2 * n if gather else n, 2 * n if scatter else n, n, 2048, d_out, gather, scatter)
    rows = np.unique(np.r_[0, 127, 128, 255, 256, n - 2, n - 1, np.arange(5, n, 97)])
    check(B, ctx, *args, n, accumulate, rows=rows)


@pytest.mark.parametrize("n,d_in,d_out,gather,scatter,accumulate,plan", [
    (643, 512, 6320, False, False, 0, 128),       # one CTA per tile, narrow: two rounds, 48 columns in the last tile
    (5000, 512, 4104, False, False, 0, 256),      # wide: five rounds, rows in order
    (5000, 512, 4104, True, True, 1, 256),        # the same gathered and added
    (386, 1024, 4776, False, True, 0, -160),      # pairs: one round, the last rows are two of the second CTA
    (391, 4096, 4840, True, True, 1, -160),
    (258, 256, 6472, False, True, 1, -192),       # four slabs; two rows in the last tile
    (1560, 512, 5992, True, True, 1, -224),
    (262, 1024, 17400, False, False, 0, -256),    # two rounds
    (1027, 4096, 6608, True, True, 1, -256),
    (1044, 4096, 6544, True, False, 0, -256),
])
def test_project_rows_by_the_kernel_that_runs_them(env, n, d_in, d_out, gather, scatter, accumulate, plan):
    """Every width of tiles, by one CTA (plan > 0) and by pairs (< 0), at other depths than the benchmark's."""
    B, ctx = env
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert B.lib.fl_internal_project_plan(148, n, d_in, d_out, int(gather), accumulate) == plan
    check_every_row(B, ctx, n, d_in, d_out, gather, scatter, accumulate)


def check_every_row(B, ctx, n, d_in, d_out, gather, scatter, accumulate, launches=1):
    """All outputs of rows drawn from twice as many against the product in binary64; every launch gives the same bits."""
    g = torch.Generator(device="cuda").manual_seed(5)
    x, w = (torch.randn(r, d_in, generator=g, device="cuda").bfloat16() for r in (2 * n, d_out))
    y0 = torch.randn(2 * n, d_out, generator=g, device="cuda").bfloat16()
    src, dst = (torch.sort(torch.randperm(2 * n, generator=g, device="cuda")[:n])[0].int() for _ in range(2))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs = []
    for _ in range(launches):
        y = y0.clone()
        B.fl_project_rows(ctx, x, 2 * n, src if gather else None, n, d_in, w, d_out, y, 2 * n, dst if scatter else None, accumulate, status)
        outs.append(y)
    assert int(status.item()) == 0 and all(torch.equal(outs[0], o) for o in outs[1:])
    at = dst.long() if scatter else torch.arange(n, device="cuda")
    xs, ws, old = (x[src.long()] if gather else x[:n]).double(), w.double(), y0[at].double() * accumulate
    ref, mag = xs @ ws.T + old, xs.abs() @ ws.abs().T + old.abs()
    assert ((outs[0][at].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + d_in * 2.0 ** -23 * mag).all()
    rest = torch.ones(2 * n, dtype=torch.bool, device="cuda")
    rest[at] = False
    assert torch.equal(outs[0][rest], y0[rest])


def test_project_rows_pairs_reuse_their_accumulators(env):
    """Five tiles per pair of CTAs, every row of every tile: an accumulator is overwritten only when the epilogues of BOTH CTAs have
    read it."""
    B, ctx = env
    check_every_row(B, ctx, 3277, 2048, 6144, True, True, 1, launches=4)


def test_project_rows_single_row_and_empty(env):
    B, ctx = env
    x, w, y, src, dst = make(9, 50, 50, 1, 64, 8, True, True)
    check(B, ctx, x, w, y, src, dst, 1, 0)
    yd = dev(y, torch.bfloat16)
    B.fl_project_rows(ctx, dev(x, torch.bfloat16), 50, None, 0, 64, dev(w, torch.bfloat16), 8, yd, 50, None, 0)
    torch.cuda.synchronize()
    assert np.array_equal(yd.float().cpu().numpy(), y)


def test_project_rows_benchmark_shape_sampled(env):
    """The QKV projection of the benchmark shape (3277 active rows of 32768, d = 2048, 3 d outputs) and the output
    projection with its residual add scattered back, checked on sampled rows."""
    B, ctx = env
    n, L, d = 3277, 32768, 2048
    rows = np.sort(np.random.default_rng(2).choice(n, size=48, replace=False))
    x, w, y, src, _ = make(10, L, n, n, d, 3 * d, True, False)
    check(B, ctx, x, w, y, src, None, n, 0, rows=rows)
    x, w, y, _, dst = make(11, n, L, n, d, d, False, True)
    check(B, ctx, x, w, y, None, dst, n, 1, rows=rows)


# ---- the stacked Q/K/V projection with the residual codec as its epilogue ---------------------------------------
from paper_2609_29812_b200 import workloads            # noqa: E402
from helpers import to_dev, to_np                       # noqa: E402
from test_gpu_parity import small_bf16                  # noqa: E402


@pytest.mark.parametrize("bits,group,H,n_loops", [(4, 128, 2, 3), (8, 64, 2, 2), (2, 32, 4, 2)])
def test_projection_with_codec_epilogue(env, bits, group, H, n_loops):
    """Loops 2..n_loops of one small layer through fl_project_qkv_quant.  Q and the new K | V rows against the oracle's
    fp64 projection; codes, scales, offsets and the materialized rows bit for bit against the oracle's residual codec
    applied to the kernel's own bf16 K | V rows (the reading: the codes are those of the GEMM's own outputs); and every
    output bit for bit against the unfused calls (fl_project_rows, then fl_quant_kv_residual)."""
    from paper_2609_29812_b200 import pipeline as P
    B, ctx = env
    w = small_bf16(L=700, H=H, R=n_loops, bits=bits, group=group)
    L, d = w.L, w.d
    rng = np.random.default_rng(31)
    hid = [round_to_bf16(rng.standard_normal((L, d)).astype(np.float32)) for _ in range(n_loops)]
    wqkv = round_to_bf16((rng.standard_normal((3 * d, d)) / np.sqrt(d)).astype(np.float32))
    k1 = round_to_bf16(rng.standard_normal((L, d)).astype(np.float32))
    v1 = round_to_bf16(rng.standard_normal((L, d)).astype(np.float32))
    shp = (L, w.n_heads, w.head_dim)
    st, st_ref = P.LayerState(ctx, w), P.LayerState(ctx, w)
    for s_ in (st, st_ref):
        s_.k_base, s_.v_base = to_dev(k1.reshape(shp), w), to_dev(v1.reshape(shp), w)
    wd = dev(wqkv, torch.bfloat16)
    khat, vhat = k1.reshape(shp).copy(), v1.reshape(shp).copy()
    act = np.arange(L)
    for r in range(2, n_loops + 1):
        act = np.sort(rng.choice(act, size=max(40, len(act) // 3), replace=False))     # nested, ragged against 128
        n = len(act)
        sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(),
                               torch.from_numpy(fo.slot_map(act, L)).cuda(), None, n)
        hd = dev(hid[r - 1], torch.bfloat16)
        st.alloc_stream(sel)
        q_out = torch.full((n, d), 5.0, dtype=torch.bfloat16, device="cuda:0")
        kv_out = torch.full((n, 2 * d), 5.0, dtype=torch.bfloat16, device="cuda:0")
        status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
        B.fl_project_qkv_quant(ctx, st.shape, r, hd, L, sel.active_idx, n, wd, q_out, kv_out, st.store, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        rows_prev = [to_np(st.k_streams[-1]["rows_prev"]).copy(), to_np(st.v_streams[-1]["rows_prev"]).copy()]
        rows_cur = [to_np(st.k_streams[-1]["rows_cur"]).copy(), to_np(st.v_streams[-1]["rows_cur"]).copy()]
        # (1) the projection itself
        ref = fo.project_rows(hid[r - 1], act, wqkv, np.zeros((n, 3 * d)), None, False)
        mag = np.abs(hid[r - 1][act].astype(np.float64)) @ np.abs(wqkv.astype(np.float64)).T
        got = np.concatenate([to_np(q_out), to_np(kv_out)], axis=1).astype(np.float64)
        assert np.max(np.abs(got - ref) / (2.0 ** -8 * np.abs(ref) + d * 2.0 ** -23 * mag + 1e-30)) <= 1.0
        # (2) the codec, on the kernel's own K | V rows
        kv = to_np(kv_out)
        for side, (streams, hat, new) in enumerate(((st.k_streams, khat, kv[:, :d]), (st.v_streams, vhat, kv[:, d:]))):
            hat_new, pay = fo.residual_update(new.reshape(n, w.n_heads, w.head_dim), hat, act, bits, group)
            got_s = streams[-1]
            assert np.array_equal(got_s["codes"].cpu().numpy().reshape(n, -1), pay["packed"].reshape(n, -1)), (r, side)
            assert np.array_equal(got_s["scale"].cpu().numpy().view(np.uint16).reshape(-1), pay["scale"].view(np.uint16).reshape(-1))
            assert np.array_equal(got_s["zero"].cpu().numpy().view(np.uint16).reshape(-1), pay["zero"].view(np.uint16).reshape(-1))
            assert np.array_equal(rows_prev[side].reshape(n, -1), fo.round_bf16(hat[act]).reshape(n, -1))
            assert np.array_equal(rows_cur[side].reshape(n, -1), fo.round_bf16(hat_new[act]).reshape(n, -1))
            if side == 0:
                khat = hat_new
            else:
                vhat = hat_new
        # (3) the unfused calls on a second store
        st_ref.alloc_stream(sel)
        qkv = torch.empty(n, 3 * d, dtype=torch.bfloat16, device="cuda:0")
        B.fl_project_rows(ctx, hd, L, sel.active_idx, n, d, wd, 3 * d, qkv, n, None, 0, status)
        k_new, v_new = qkv[:, d:2 * d].contiguous(), qkv[:, 2 * d:].contiguous()
        B.fl_quant_kv_residual(ctx, st_ref.shape, r, k_new, v_new, sel.active_idx, n, st_ref.store)
        torch.cuda.synchronize()
        assert torch.equal(qkv[:, :d], q_out) and torch.equal(qkv[:, d:], kv_out)
        for a_, b_ in ((st.k_streams[-1], st_ref.k_streams[-1]), (st.v_streams[-1], st_ref.v_streams[-1])):
            for key in ("codes", "scale", "zero"):
                assert torch.equal(a_[key], b_[key]), (r, key)
        assert np.array_equal(to_np(st_ref.k_streams[-1]["rows_cur"]), rows_cur[0])
        assert np.array_equal(to_np(st_ref.v_streams[-1]["rows_prev"]), rows_prev[1])


@pytest.mark.parametrize("bits,group", [(4, 128), (8, 64), (2, 32)])
def test_codec_epilogue_with_a_channel_that_is_not_finite(env, bits, group):
    """One K channel without a value (a weight that is not a number), one V channel beyond fp16: the epilogue's streams are
    those of the unfused calls, and the K channel's code is 0 and spoils no neighbour's."""
    from paper_2609_29812_b200 import pipeline as P
    B, ctx = env
    w = small_bf16(L=300, H=2, R=2, bits=bits, group=group)
    L, d = w.L, w.d
    rng = np.random.default_rng(bits)
    draw = lambda *s: round_to_bf16(rng.standard_normal(s).astype(np.float32))
    hd, wd = dev(draw(L, d), torch.bfloat16), dev(draw(3 * d, d) / 16, torch.bfloat16)
    act = np.sort(rng.permutation(L)[:70])
    sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(), torch.from_numpy(fo.slot_map(act, L)).cuda(), None, 70)
    k1, v1 = (to_dev(draw(L, w.n_heads, w.head_dim), w) for _ in range(2))
    codes = {}
    for name in ("finite", "fused", "unfused"):
        if name != "finite":
            wd[d + 6, 0], wd[2 * d + 9] = float("nan"), 1e30
        st = P.LayerState(ctx, w)
        st.k_base, st.v_base = k1, v1
        st.alloc_stream(sel)
        status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
        if name == "unfused":
            qkv = torch.empty(70, 3 * d, dtype=torch.bfloat16, device="cuda:0")
            B.fl_project_rows(ctx, hd, L, sel.active_idx, 70, d, wd, 3 * d, qkv, 70, None, 0, status)
            st.quantize(2, qkv[:, d:2 * d].contiguous(), qkv[:, 2 * d:].contiguous(), sel)
        else:
            q_out, kv_out = (torch.empty(70, m * d, dtype=torch.bfloat16, device="cuda:0") for m in (1, 2))
            B.fl_project_qkv_quant(ctx, st.shape, 2, hd, L, sel.active_idx, 70, wd, q_out, kv_out, st.store, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        codes[name] = [to_np(s["codes"]) for s in (st.k_streams[0], st.v_streams[0])]
        meta = [to_np(s[m]) for s in (st.k_streams[0], st.v_streams[0]) for m in ("scale", "zero")]
        if name == "fused":
            fused_meta = meta
    assert all(np.array_equal(a, b) for a, b in zip(codes["fused"], codes["unfused"]))
    assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(fused_meta, meta))
    k = fo.unpack_codes(codes["fused"][0], bits)
    assert not k[:, 6].any()
    other = np.arange(d) >= group                          # the channel is missing from its own group's range only
    assert np.array_equal(k[:, other], fo.unpack_codes(codes["finite"][0], bits)[:, other])
