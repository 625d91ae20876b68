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


SPECIALS = (np.nan, np.inf, -np.inf, 3.0e38, -3.0e38)     # the last two overflow the fp16 scale and offset


def plant(x, at, groups_of):
    """`x` [rows, d] with SPECIALS at `at`; the mask of the elements in a group with one that is no finite fp16 number
    (codes 0, metadata not finite); the not-a-number element counts for nobody but itself."""
    bad, lost = x.copy(), np.zeros(x.shape, dtype=bool)
    for value, (i, j) in zip(SPECIALS, at):
        bad[i, j] = value
        if not np.isnan(value):
            lost[groups_of(i, j)] = True
    return bad, lost


@pytest.mark.parametrize("H,bits,group,dtype", [(4, 4, 128, "bf16"), (4, 2, 32, "bf16"), (4, 8, 16, "bf16"), (2, 4, 8, "bf16"),
                                                (2, 8, 64, "bf16"), (4, 4, 32, "f32"), (4, 8, 64, "f32")])
def test_not_finite_elements_spoil_nothing_else(env, H, bits, group, dtype):
    """Residual rows with an element that is no number, or not finite in fp16: codes, metadata and rows of every other
    element (its neighbours in the same word) and group are those of rows without it; its own code is 0."""
    B, P, ctx = env
    rng = np.random.default_rng(bits)
    L, n, dh = 64, 16, 128 if dtype == "bf16" else 64
    w = workloads.replace(workloads.config2(L=L, n_heads=H), n_loops=2, head_dim=dh, dtype=dtype, bits=bits, group=group)
    rnd = fo.round_bf16 if dtype == "bf16" else (lambda a: a)
    hat = rnd(rng.standard_normal((L, H, dh)).astype(np.float32))
    act = np.sort(rng.permutation(L)[:n])
    new = rnd(hat[act] + rng.standard_normal((n, H, dh)).astype(np.float32)).reshape(n, H * dh)
    at = [(2 * i, 7 + 9 * i) for i in range(len(SPECIALS))]
    new[0, 7] = hat[act].reshape(n, -1)[0, 7]              # where the not-a-number goes: no extremum of its group
    bad, lost = plant(new, at, lambda i, j: (i, slice(j // group * group, (j // group + 1) * group)))
    _, pay = fo.residual_update(new.reshape(n, H, dh), hat, act, bits, group)
    codes = pay["codes"].reshape(n, -1).copy()
    codes[lost | np.isnan(bad)] = 0
    st = P.LayerState(ctx, w, split=False)
    st.k_base = st.v_base = to_dev(hat, w)
    sel = P.TokenSelection(torch.from_numpy(act.astype(np.int32)).cuda(),
                           torch.from_numpy(fo.slot_map(act, L).astype(np.int32)).cuda(), None, n)
    st.alloc_stream(sel)
    st.quantize(2, to_dev(bad.reshape(n, H, dh), w), to_dev(new.reshape(n, H, dh), w), sel)
    torch.cuda.synchronize()
    k, v, ok = st.k_streams[-1], st.v_streams[-1], ~lost.reshape(n, -1, group).any(axis=2)
    assert np.array_equal(to_np(k["codes"]), fo.pack_codes(codes, bits))
    assert np.array_equal(to_np(v["codes"]), pay["packed"].reshape(n, -1))
    for m in ("scale", "zero"):
        assert np.array_equal(to_np(k[m]).view(np.uint16)[ok], pay[m].reshape(n, -1).view(np.uint16)[ok]), m
    if dtype == "bf16":                                    # the rows are what a reader of the stream forms, code 0 included
        seen = (hat[act] + fo.dequantize_groups(codes.reshape(n, H, dh), pay["scale"], pay["zero"], group)).astype(np.float32)
        assert np.array_equal(to_np(k["rows_cur"])[~lost], fo.round_bf16(seen).reshape(n, -1)[~lost])


@pytest.mark.parametrize("bits,group,dtype", [(4, 64, "bf16"), (2, 32, "bf16"), (8, 128, "bf16"), (4, 32, "f32")])
def test_packed_base_with_elements_that_are_not_finite(env, bits, group, dtype):
    """The same for the packed base, where four neighbouring key codes belong to four groups."""
    B, P, ctx = env
    rng = np.random.default_rng(group)
    H, dh = (2, 128) if dtype == "bf16" else (4, 64)
    L, tail = 300, 11
    Lq = L - tail
    w = workloads.replace(workloads.config2(L=L, n_heads=H), head_dim=dh, dtype=dtype, bits=bits, group=min(group, dh))
    rnd = fo.round_bf16 if dtype == "bf16" else (lambda a: a)
    k, v = (rnd(rng.standard_normal((L, H * dh)).astype(np.float32)) for _ in range(2))
    at = [(3 + 40 * i, 5 + 9 * i) for i in range(len(SPECIALS))]
    k[3, 5], v[3, 5] = k[4, 5], v[3, 6]                    # the not-a-number takes no extremum away
    k_bad, k_lost = plant(k, at, lambda i, j: (slice(i // group * group, min(Lq, (i // group + 1) * group)), j))
    v_bad, v_lost = plant(v, at, lambda i, j: (i, slice(j // group * group, (j // group + 1) * group)))
    ref = fo.quantize_base(k, v, bits, group, tail, storage_round=rnd if dtype == "bf16" else None)
    st = P.LayerState(ctx, w, split=False)
    st.pack_base(to_dev(k_bad.reshape(L, H, dh), w), to_dev(v_bad.reshape(L, H, dh), w), group, tail)
    kc, ks, kz, vc, vs, vz = [to_np(t) for t in st.base_tensors[:6]]
    for got, name, bad, lost in ((kc, "k_codes", k_bad, k_lost), (vc, "v_codes", v_bad, v_lost)):
        codes = ref[name].copy()
        codes[lost[:Lq] | np.isnan(bad[:Lq])] = 0
        assert np.array_equal(got, fo.pack_codes(codes, bits)), name
    k_ok = ~np.stack([k_lost[g * group:min(Lq, (g + 1) * group)].any(axis=0) for g in range(ks.shape[0])])
    v_ok = ~v_lost[:Lq].reshape(Lq, -1, group).any(axis=2)
    for got, name, ok in ((ks, "k_scale", k_ok), (kz, "k_zero", k_ok), (vs, "v_scale", v_ok), (vz, "v_zero", v_ok)):
        assert np.array_equal(got.view(np.uint16)[ok], ref[name].view(np.uint16)[ok]), name


def _pack(B, P, ctx, w, k, v, group):
    st = P.LayerState(ctx, w, split=False)
    shape = (w.L, w.n_heads, w.head_dim)
    st.pack_base(to_dev(k.reshape(shape), w), to_dev(v.reshape(shape), w), group, 0)
    return [to_np(t) for t in st.base_tensors[:6]]


@pytest.mark.parametrize("bits", [2, 4, 8])
def test_quotients_at_and_beside_half_integers(env, bits):
    """binary32 values whose quotients are exact halves, and the numbers next to those on either side: the code is the rounded
    quotient, halves to even, as a division gives it."""
    B, P, ctx = env
    rng = np.random.default_rng(bits)
    n, L, d = 2 ** bits - 1, 512, 256
    s = np.exp2(rng.integers(-9, 4, L)) * (1 + rng.integers(0, 1024, L) / 1024.0)      # scales that fp16 holds
    half = (rng.integers(0, n, (L, d)) + 0.5) * s[:, None]
    v = half.astype(np.float32)
    v = np.choose(rng.integers(0, 3, (L, d)), [v, np.nextafter(v, np.float32(0)), np.nextafter(v, np.float32(np.inf))])
    v[:, ::32], v[:, 1::32] = 0.0, (n * s[:, None]).astype(np.float32)                 # every group spans 0 .. n s: its scale is s
    w = workloads.replace(workloads.config2(L=L, n_heads=4), head_dim=64, dtype="f32", bits=bits, group=32)
    ref = fo.quantize_base(v, v, bits, 32, 0)
    got = _pack(B, P, ctx, w, v, v, 32)
    assert np.array_equal(got[3], fo.pack_codes(ref["v_codes"], bits)) and np.array_equal(got[0], fo.pack_codes(ref["k_codes"], bits))
    assert np.array_equal(got[4].view(np.uint16), ref["v_scale"].view(np.uint16))


@pytest.mark.parametrize("L,group", [(40037, 32), (20003, 64)])
def test_packed_base_with_several_key_tiles_per_cta(env, L, group):
    B, P, ctx = env
    rng = np.random.default_rng(L)
    k, v = (fo.round_bf16(rng.standard_normal((L, 256)).astype(np.float32)) for _ in range(2))
    w = workloads.replace(workloads.config2(L=L, n_heads=2), bits=4, group=group)
    ref = fo.quantize_base(k, v, 4, group, 0, storage_round=fo.round_bf16)
    got = _pack(B, P, ctx, w, k, v, group)
    for g, name in zip(got, ("k_codes", "k_scale", "k_zero", "v_codes", "v_scale", "v_zero")):
        want = fo.pack_codes(ref[name], 4) if "codes" in name else ref[name]
        assert np.array_equal(np.ascontiguousarray(g).view(np.uint8), np.ascontiguousarray(want).view(np.uint8)), name


@pytest.mark.parametrize("L,H,group", [(15001, 16, 128), (64, 4, 128), (20003, 8, 64)])
def test_packed_base_with_and_without_tiles_asked_for_ahead(env, L, H, group):
    """CTAs of 1024 and 512 threads: up to seven tiles of 256 channels per CTA (the first from registers, the others from the slots),
    and a base of one tile per CTA, which has no slots. Channels of every tile against the oracle (keys are grouped per channel)."""
    B, P, ctx = env
    g = torch.Generator(device="cuda").manual_seed(L)
    d = H * 128
    k, v = (torch.randn(L, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    w = workloads.replace(workloads.config2(L=L, n_heads=H), bits=4, group=group)
    got = _pack(B, P, ctx, w, to_np(k), to_np(v), group)
    cols = np.linspace(0, d - 1, group).astype(int)
    part = to_np(k)[:, cols]
    ref = fo.quantize_base(part, part, 4, group, 0, storage_round=fo.round_bf16)
    assert np.array_equal(fo.unpack_codes(got[0], 4)[:, cols], ref["k_codes"])
    assert np.array_equal(got[1][:, cols].view(np.uint16), ref["k_scale"].view(np.uint16))
    assert np.array_equal(got[2][:, cols].view(np.uint16), ref["k_zero"].view(np.uint16))
