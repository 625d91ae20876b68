"""The number that a row's new probabilities are taken against comes from the previous loop's log-normaliser. Rows for which it is
no estimate of the new logits (queries that jump between loops, no or useless log-normalisers in a reusing call) send their tile
through two more passes: single tiles, several tiles of a block, shared and split problems, the one-term and the two-term kernel."""
import numpy as np
import pytest

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
