"""What a row's new probabilities are taken against: a number near its largest logit, from the previous loop's log-normaliser (one-term
kernel) or from the row's first columns as well. Rows for which it is none send their tile through two more passes: single
tiles, several tiles of a block, shared and split problems, the one-term and the two-term kernel, and what that costs."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200 import workloads
from helpers import assert_attn_close, to_dev, to_np
from test_gpu_economy import run_oracle
from test_gpu_parity import oracle_selection, small_bf16

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


def loop(st, w, x, P, ref, r, **kw):
    sel, act = oracle_selection(P, w, ref, r), ref["active"][r - 2]
    o, _ = st.sparse_loop(r, to_dev(x.Q[r - 1][act], w), to_dev(x.K[r - 1][act], w), to_dev(x.V[r - 1][act], w), sel,
                          indexed=True, **kw)
    st.check_status()
    return o


@pytest.mark.parametrize("L,q_block,k_tok,scale", [(1500, 256, None, 64.0), (1100, 512, 1100, 64.0), (700, 1024, 90, 1e-3)])
def test_queries_that_jump(env, L, q_block, k_tok, scale):
    """Loop 2's queries are `scale` times as long as the source loop's: logits hundreds of units above the log-normalisers
    that came before (or, from long queries to short ones, below), in some rows of a tile and not in others."""
    B, P, ctx = env
    w = workloads.replace(small_bf16(L=L, H=2, R=2), q_block=q_block)
    x = workloads.make_layer_inputs(w, seed=L)
    one = 64.0 if scale < 1 else 1.0
    x.Q[0] = workloads.round_to_bf16(x.Q[0] * np.float32(one))
    grow = np.where(np.arange(L)[:, None, None] % 3 == 0, np.float32(scale * one), np.float32(one))
    x.Q[1] = workloads.round_to_bf16(x.Q[1] * grow)
    ref = run_oracle(w, x, k_tok=None if k_tok is None else [k_tok])
    for carry in (None, "write"):
        st = P.LayerState(ctx, w)
        st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
        st.select_columns_dense()
        o = loop(st, w, x, P, ref, 2, carry=carry)
        assert_attn_close(to_np(o), ref["loops"][0]["O_rows"], f"queries that jump, carry {carry}", carried=1)


@pytest.mark.parametrize("rows", [True, False], ids=["one-term kernel", "two-term kernel"])
@pytest.mark.parametrize("L,q_block,k_tok", [(1500, 256, 400), (1100, 512, 1100)])
def test_reuse_without_useful_normalisers(env, rows, L, q_block, k_tok):
    """A reusing call takes lse_in as a hint: without it, and with numbers that are none, its results are the same up to the
    rounding of its probabilities (two bf16 roundings of every weight, 2^-8 together, against each other)."""
    B, P, ctx = env
    w = workloads.replace(small_bf16(L=L, H=2, R=3), q_block=q_block)
    x = workloads.make_layer_inputs(w, seed=L + 1)
    ref = run_oracle(w, x, k_tok=[k_tok] * 2)
    st = P.LayerState(ctx, w)
    st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
    st.select_columns_dense()
    loop(st, w, x, P, ref, 2, carry="write", rows=rows)
    lse2 = st.lse.clone()
    want = loop(st, w, x, P, ref, 3, carry="reuse", rows="cur" if rows else False).clone()
    want_lse = st.lse.clone()
    sel = oracle_selection(P, w, ref, 3)
    q = to_dev(x.Q[2][ref["active"][1]], w)
    far = torch.where(torch.arange(L, device="cuda") % 2 == 0, 1000.0, -1000.0) + lse2
    hints = {"none": None, "nan": torch.full_like(lse2, float("nan")), "inf": torch.full_like(lse2, float("inf")),
             "-inf": torch.full_like(lse2, float("-inf")), "far": far}
    act = torch.from_numpy(ref["active"][1]).cuda()
    for name, hint in hints.items():
        lse_out = torch.zeros_like(lse2)
        st.o_store.zero_()
        rc = B.fl_loop_attention_indexed_carry(ctx, st.shape, 3, q, None, None, sel.active_idx, sel.n, st.store, st.col_idx, st.col_cnt,
                                               st.c, hint, lse_out, None, st.o_store, B.make_carry(st.bg_store, st.mass, True), None,
                                               status=st.status)
        assert rc == 0
        st.check_status()
        got = st.o_store[act].float()
        rel = ((got - want.float()).norm() / want.float().norm()).item()
        assert rel <= 2.0 ** -8, (name, rel)
        assert_attn_close(to_np(st.o_store[act]), ref["loops"][1]["O_rows"], f"reuse, hint {name}", carried=1)
        seen = st.mass[:, act] > 0
        assert torch.allclose(lse_out[:, act][seen], want_lse[:, act][seen], rtol=1e-5, atol=1e-4), name


@pytest.mark.parametrize("two_pass", [False, True], ids=["two-term kernel", "one-term kernels"])
def test_normalisers_that_are_no_numbers(env, two_pass, monkeypatch):
    """A row whose previous log-normaliser is NaN or -inf has no old probabilities. It must not come out as numbers: the two-term
    kernel passes them on (output and log-normaliser are no finite numbers either), the one-term kernels leave a row without a mass
    as it was. The other rows, those of the same tile among them, keep their bits."""
    B, P, ctx = env
    if two_pass:
        monkeypatch.setenv("FL_TWO_PASS", "1")
        ctx = B.Context(0)
        monkeypatch.delenv("FL_TWO_PASS")
    w = workloads.replace(small_bf16(L=1100, H=2, R=2), q_block=256)
    x = workloads.make_layer_inputs(w, seed=77)
    ref = run_oracle(w, x)
    act = torch.from_numpy(ref["active"][0]).cuda()
    bad = {(0, len(act) - 9): float("nan"), (1, len(act) // 2): float("-inf"), (1, len(act) - 40): float("nan")}
    outs = []
    for spoil in (False, True):
        st = P.LayerState(ctx, w)
        st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
        st.select_columns_dense()
        before = st.o_store.clone()
        for (h, t), value in bad.items() if spoil else ():
            st.lse[h, act[t]] = value
        loop(st, w, x, P, ref, 2, carry="write")
        outs.append((st.o_store[act].clone(), st.lse[:, act].clone(), st.mass[:, act].clone()))
    (o, lse, mass), (o_bad, lse_bad, mass_bad) = outs
    assert torch.isfinite(o.float()).all() and torch.isfinite(lse).all()
    same = torch.ones(w.n_heads, len(act), dtype=torch.bool, device="cuda")
    for (h, t), value in bad.items():
        same[h, t] = False
        got, m = o_bad[t, h].float(), mass_bad[h, t].item()
        assert not (0.0 < m < float("inf")), (h, t, m)
        if two_pass and m == 0.0:
            assert torch.equal(o_bad[t, h], before[act[t], h]), (h, t)
        else:
            assert not torch.isfinite(got).any() and not torch.isfinite(lse_bad[h, t]), (h, t)
    assert torch.equal(o_bad.transpose(0, 1)[same], o.transpose(0, 1)[same])
    assert torch.equal(lse_bad[same], lse[same]) and torch.equal(mass_bad[same], mass[same])
    if two_pass:
        ctx.close()


def spiked(w, seed, k_tok):
    """Inputs in which one key column, and it alone, has weight in the first head dimension. Its logit is 8 in units of log2 for
    ordinary rows and 326 for every third row of a sparse loop (another third per loop), whose other logits stay within +-100: past the
    row's first 128 columns its largest logit grows by more than any reference chosen from them can take, so its tile needs all
    three passes. Returns the inputs, the oracle's record and the column."""
    x = workloads.make_layer_inputs(w, seed=seed)
    act = run_oracle(w, x, k_tok=k_tok)["active"]
    col = next(p for p in range(int(0.7 * w.L), w.L) if not any(p in a for a in act))
    for r in range(w.n_loops):
        q, k = x.Q[r], x.K[r]
        k[:, :, 0] = 0.0
        k[col, :, 0] = 16.0
        q[:, :, 0] = 4.0
        if r > 0:
            q[r % 3::3, :, 0] = 160.0
    ref = run_oracle(w, x, k_tok=k_tok)
    for r, rec in enumerate(ref["loops"], start=2):
        sent = 0
        for (h, b), S in rec["col_sets"].items():
            S, rows = np.asarray(S), rec["active"][rec["active"] // w.q_block == b]
            rows = rows[(rows >= col) & (rows % 3 == (r - 1) % 3)]
            if col not in S or len(rows) == 0:
                continue
            # references come from a row's first chunk (reusing calls: from its first two): this column comes later
            assert (S[~np.isin(S, act[0])] < col).sum() >= 128
            kh = fo.round_bf16(rec["khat"])[S[S != col]][:, h].astype(np.float64)
            logits = x.Q[r - 1][rows][:, h].astype(np.float64) @ kh.T * w.sm_scale * np.log2(np.e)
            assert np.abs(logits).max() < 100.0 and 160.0 * 16.0 * w.sm_scale * np.log2(np.e) > 300.0
            sent += len(rows)
        assert sent > 0, r
    return x, ref, col


# "rebuilt": no materialized rows, so chunks with payloads are rewritten in the ring (two slots each where the old term is computed
# again); "several tiles": blocks of 130 rows whose two tiles one CTA walks (112 problems on 148 SMs, 208 on 296 slots)
PASSES = {
    "two terms": dict(kw=dict(carry="write")),
    "two terms, whole problems": dict(split=False, kw=dict(carry="write")),
    "two terms, rebuilt": dict(kw=dict(rows=False)),
    "two terms, rebuilt, whole problems, 16 bits": dict(split=False, bits=16, kw=dict(rows=False)),
    "two terms, rebuilt, several tiles": dict(L=1792, H=16, k_tok=[930], kw=dict(rows=False, carry="write")),
    "two terms, compact": dict(kw=dict(indexed=False)),
    "two terms, compact, rebuilt": dict(split=False, kw=dict(indexed=False, rows=False)),
    "two terms, shrinking sets": dict(k_tok=[400, 150, 60], kw=dict(rows=False)),
    "two streams": dict(k_tok=[300, 300, 300], reuse=dict(rows=False)),
    "two streams, rebuilt, shrinking sets": dict(k_tok=[400, 150, 60], split=False, reuse=dict(rows=False)),
    "one term": dict(k_tok=[300, 300, 300], reuse=dict(rows="cur")),
    "one term, shrinking sets": dict(k_tok=[400, 150, 60], split=False, reuse=dict(rows="cur")),
    "one term, several tiles": dict(L=3328, H=16, cols=560, k_tok=[1740, 1700], reuse=dict(rows="cur")),
    "one term twice": dict(k_tok=[400, 150, 60], two_pass=True, kw=dict(carry="write")),
}


@pytest.mark.parametrize("name", list(PASSES))
def test_three_passes(env, name, monkeypatch):
    """Rows whose largest logit no reference from their first columns fits, in every form that a tile is worked on. (The column
    lies in the later half of the lists: of a split problem one CTA needs the passes and the other does not.)"""
    B, P, ctx = env
    c = PASSES[name]
    if c.get("two_pass"):
        monkeypatch.setenv("FL_TWO_PASS", "1")
        ctx = B.Context(0)
        monkeypatch.delenv("FL_TWO_PASS")
    k_tok = c.get("k_tok", [300])
    w = workloads.replace(small_bf16(L=c.get("L", 1100), H=c.get("H", 2), R=1 + len(k_tok), c=c.get("cols", 400), bits=c.get("bits", 4)),
                          changed_fracs=tuple(k / c.get("L", 1100) for k in k_tok))
    x, ref, col = spiked(w, 5, k_tok)
    st = P.LayerState(ctx, w, split=c.get("split", True))
    st.dense_loop(to_dev(x.Q[0], w), to_dev(x.K[0], w), to_dev(x.V[0], w))
    st.select_columns_dense()
    for r in range(2, w.n_loops + 1):
        rec, act = ref["loops"][r - 2], ref["active"][r - 2]
        kw = dict(indexed=True, **c["kw"]) if "kw" in c and "indexed" not in c["kw"] else dict(c.get("kw", {}))
        if "reuse" in c:
            kw = dict(indexed=True, carry="write") if r == 2 else dict(indexed=True, carry="reuse", **c["reuse"])
        sel = oracle_selection(P, w, ref, r)
        o, _ = st.sparse_loop(r, to_dev(x.Q[r - 1][act], w), to_dev(x.K[r - 1][act], w), to_dev(x.V[r - 1][act], w), sel, **kw)
        st.check_status()
        # (the carried output is rounded once per loop on the GPU side only; where the old term is taken over, once in all)
        assert_attn_close(to_np(o), rec["O_rows"], f"three passes, {name}, loop {r}", carried=1 if "reuse" in c else r - 1)
        ok = np.isfinite(rec["lse_rows"])
        np.testing.assert_allclose(to_np(st.lse)[:, act][ok], rec["lse_rows"][ok], rtol=0, atol=5e-3 * (r - 1))
    if c.get("two_pass"):
        ctx.close()


class Timed:
    """One layer of 16384 positions on random rows, a tenth of them active: what the tests of times share."""
    L, H, n, c = 16384, 16, 1638, 512

    def __init__(self):
        g = torch.Generator(device="cuda").manual_seed(3)
        self.draw = lambda m: torch.randn(m, self.H, 128, generator=g, device="cuda").bfloat16()
        self.q, self.k, self.v = self.draw(self.L), self.draw(self.L), self.draw(self.L)
        self.act = torch.sort(torch.randperm(self.L, generator=g, device="cuda")[:self.n])[0]
        self.slot = torch.full((self.L,), -1, dtype=torch.int32, device="cuda")
        self.slot[self.act] = torch.arange(self.n, dtype=torch.int32, device="cuda")
        self.w = workloads.replace(workloads.config2(L=self.L, n_heads=self.H), n_loops=3, col_budget=self.c, changed_fracs=(0.1, 0.1))
        self.flush = torch.empty(64 << 20, device="cuda")

    def of(self, f):
        times = []
        for i in range(11):
            self.flush.fill_(1.0)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            f()
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        return float(np.median(times[2:]))

    def loop(self, P, st, sel, r, rows):
        st.alloc_stream(sel, rows=rows)
        st.quantize(r, self.k[self.act] + 0.1 * self.draw(self.n), self.v[self.act] + 0.1 * self.draw(self.n), sel)


def test_jumps_cost_no_passes(env):
    """Queries 12 times as long as the ones before (logits some 17 units of log2 apart, where the log-normalisers know of 1.4) in
    the two-term kernel, and reusing calls without log-normalisers in both, keep to one pass: within 1.25 of the ordinary call's time,
    medians of nine calls on the same buffers (three passes take 2.3 to 2.6 times as long; a running maximum with its rescales took
    1.2 to 1.3 times). The one-term kernel with log-normalisers that know nothing of the queries does take its three passes."""
    B, P, ctx = env
    t = Timed()
    sel = P.TokenSelection(t.act.to(torch.int32), t.slot, None, t.n)
    for rows in (True, False):
        st = P.LayerState(ctx, t.w)
        st.dense_loop(t.q, t.k, t.v)
        st.select_columns_dense()
        bg, mass = st.carry_buffers()
        lse, o = torch.empty_like(st.lse), torch.empty_like(st.o_store)
        for r in (2, 3):
            t.loop(P, st, sel, r, rows)
            carry = B.make_carry(bg, mass, r == 3)
            q_new, q_far = t.q[t.act], 12 * t.q[t.act]

            def call(q_rows, lse_in):
                B.fl_loop_attention_indexed_carry(ctx, st.shape, r, q_rows, st.q_store, None, sel.active_idx, t.n, st.store, st.col_idx,
                                                  st.col_cnt, t.c, lse_in, lse, st.o_store, o, carry, None, status=st.status)

            plain = t.of(lambda: call(q_new, st.lse))
            far = {"12 x": t.of(lambda: call(q_far, st.lse))} if r == 2 or not rows else {}
            if r == 3:
                far["no hint"] = t.of(lambda: call(q_new, None))
                far["12 x, no hint"] = t.of(lambda: call(q_far, None))
            call(q_new, st.lse)             # leaves the background and the masses that loop 3 takes over
            st.check_status()
            for name, took in far.items():
                assert took <= 1.25 * plain, (rows, r, name, took, plain)


@pytest.mark.parametrize("rows", ["cur", False], ids=["one-term kernel", "two-term kernel"])
def test_rows_without_a_mass_cost_no_passes(env, rows):
    """A reusing call leaves a row whose carried mass is 0 at its background, so its logits, however far apart, are no reason to do
    its tile again: within 1.2 of the ordinary call's time."""
    B, P, ctx = env
    t = Timed()
    sel = P.TokenSelection(t.act.to(torch.int32), t.slot, None, t.n)
    t.k[:, :, :32] = 0.0
    st = P.LayerState(ctx, t.w)
    st.dense_loop(t.q, t.k, t.v)
    st.select_columns_dense()
    bg, mass = st.carry_buffers()
    bg.copy_(st.o_store)
    mass.fill_(0.5)
    for r in (2, 3):
        t.loop(P, st, sel, r, rows)
    # in every list a column past the first 128 without a payload; the block's later rows see it 816 above the others
    q_new = t.q[t.act]
    q_far, late = q_new.clone(), torch.zeros(t.H, t.n, dtype=torch.bool, device="cuda")
    for b in range(st.nb):
        in_block = t.act // t.w.q_block == b
        for h in range(t.H):
            cols = st.col_idx[h, b].long()
            col = cols[t.slot[cols] < 0][200]
            t.k[col, h, b] = 16.0
            late[h] |= in_block & (t.act > col)
            q_far[in_block & (t.act > col), h, b] = 400.0
    assert late.any(dim=1).all()
    o, lse = torch.zeros_like(st.o_store), torch.empty_like(st.lse)
    carry = B.make_carry(bg, mass, True)

    def call(q_rows):
        B.fl_loop_attention_indexed_carry(ctx, st.shape, 3, q_rows, None, None, sel.active_idx, t.n, st.store, st.col_idx, st.col_cnt,
                                          t.c, st.lse, lse, None, o, carry, None, status=st.status)

    plain = t.of(lambda: call(q_new))
    with_mass = t.of(lambda: call(q_far))
    mass[:, t.act] = torch.where(late, 0.0, mass[:, t.act])
    without = t.of(lambda: call(q_far))
    st.check_status()
    assert with_mass > 2.0 * plain, (with_mass, plain)          # the rows would need the passes
    assert without <= 1.2 * plain, (without, plain)
    assert torch.equal(o[t.act].transpose(0, 1)[late], bg[t.act].transpose(0, 1)[late])
    assert torch.isfinite(o[t.act].float()).all()
