"""Output and log-normalisers of the dense loop where its tiles end (pairs of 128 query rows, chunks of 128 keys: a single row,
a pair without its second tile, a second tile of one row) and with logits that make the reference move, against PyTorch in binary64;
and with logits, queries and values that are not finite."""
import pytest

from paper_2609_29812_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("boost", [1.0, 64.0])
@pytest.mark.parametrize("L,H", [(1, 1), (33, 3), (128, 2), (129, 1), (256, 2), (257, 16), (383, 4), (1025, 3), (2500, 8),
                                 (513, 64), (150, 96)])   # the last two: chunks of 64 keys, several per CTA
def test_dense_output_edges(L, H, boost):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    ctx = B.Context(0)
    w = workloads.config2(L=L, n_heads=H)
    sh = P.shape_of(w)
    g = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn(L, H, 128, generator=g, device="cuda") for _ in range(3))
    # later keys have the larger logits: with the boost the reference moves by more than 2^60 along a row
    k *= torch.linspace(0.2, 1.0, L, device="cuda")[:, None, None]
    q, k, v = (q * boost).bfloat16(), k.bfloat16(), v.bfloat16()
    o = torch.full_like(q, float("nan"))
    lse = torch.full((H, L), float("nan"), device="cuda")
    B.fl_dense_loop_attention(ctx, sh, q, k, v, o, lse, None)
    causal = torch.ones(L, L, dtype=torch.bool, device="cuda").tril_()
    for h in range(H):
        qh, kh, vh = q[:, h].double(), k[:, h].double(), v[:, h].double()
        s = ((qh @ kh.T) * w.sm_scale).masked_fill_(~causal, float("-inf"))
        ref_lse = torch.logsumexp(s, 1)
        p = torch.exp(s - ref_lse[:, None])
        # binary32 logits are off by at most (128 additions + 2) 2^-24 sum |q k| scale, and every probability by that factor;
        # P and O are rounded to bf16 (8 significant bits: half a unit in the last place is up to 2^-8 of the value), normaliser
        # and accumulator to binary32 (inside the added 2^-12)
        ds = 130 * 2.0 ** -24 * ((qh.abs() @ kh.abs().T) * w.sm_scale).amax(1)
        bound = (2.0 ** -8 + 2.0 ** -12 + 2 * ds)[:, None] * (p @ vh.abs()) + 2.0 ** -8 * (p @ vh).abs() + 1e-6
        assert ((o[:, h].double() - p @ vh).abs() <= bound).all()
        assert ((lse[h].double() - ref_lse).abs() <= ds + 2.0 ** -20 * (1 + ref_lse.abs())).all()
    ctx.close()


@pytest.mark.parametrize("H", [7, 48, 64])             # one query tile per CTA, pairs of them, one with chunks of 64 keys
def test_dense_output_not_finite(H):
    """Keys whose logits are -inf count for nothing, wherever a row's first finite logit stands (rows that see no other are zero); a key
    that is not a number or has a logit of +inf spoils the rows that see it, a query its own row, a value its own channel, and
    nothing else changes a bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    ctx = B.Context(0)
    L, inf = 700, float("inf")
    w = workloads.config2(L=L, n_heads=H)
    sh = P.shape_of(w)
    g = torch.Generator(device="cuda").manual_seed(H)
    q, k, v = (torch.randn(L, H, 128, generator=g, device="cuda") for _ in range(3))
    q[..., 0], k[..., 0] = 2.0 ** 100, 0.0             # channel 0: +-2^100 in a key makes its logits +-inf
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()

    def run(q, k, v):
        o, lse = torch.empty_like(q), torch.empty(H, L, device="cuda")
        B.fl_dense_loop_attention(ctx, sh, q, k, v, o, lse, None)
        return o, lse
    o, lse = run(q, k, v)
    assert torch.isfinite(o).all() and torch.isfinite(lse).all()

    firsts = (1, 32, 40, 64, 100, 128, 200)
    k2 = k.clone()
    for h, m in enumerate(firsts):
        k2[:m, h, 0] = -(2.0 ** 100)
    o2, lse2 = run(q, k2, v)
    causal = torch.ones(L, L, dtype=torch.bool, device="cuda").tril_()
    for h, m in enumerate(firsts):
        assert not o2[:m, h].any() and (lse2[h, :m] == -inf).all()
        qh, kh, vh = q[m:, h, 1:].double(), k[m:, h, 1:].double(), v[m:, h].double()
        s = ((qh @ kh.T) * w.sm_scale).masked_fill_(~causal[m:, m:], -inf)
        ref_lse = torch.logsumexp(s, 1)
        p = torch.exp(s - ref_lse[:, None])
        ds = 130 * 2.0 ** -24 * ((qh.abs() @ kh.abs().T) * w.sm_scale).amax(1)      # the bound of the test above
        bound = (2.0 ** -8 + 2.0 ** -12 + 2 * ds)[:, None] * (p @ vh.abs()) + 2.0 ** -8 * (p @ vh).abs() + 1e-6
        assert ((o2[m:, h].double() - p @ vh).abs() <= bound).all(), m
        assert ((lse2[h, m:].double() - ref_lse).abs() <= ds + 2.0 ** -20 * (1 + ref_lse.abs())).all(), m

    for j in (31, 130, 333, 511):
        q3, k3, v3 = q.clone(), k.clone(), v.clone()
        k3[j, 0, 7] = float("nan")
        k3[j, 1, 0] = 2.0 ** 100
        q3[j, 2, 9] = float("nan")
        v3[j, 3, 5] = inf
        o3, lse3 = run(q3, k3, v3)
        want, want_lse = o.clone(), lse.clone()
        for h, rows in ((0, slice(j, L)), (1, slice(j, L)), (2, slice(j, j + 1))):
            want[rows, h], want_lse[h, rows] = float("nan"), float("nan")
        assert not torch.isfinite(o3[j:, 3, 5]).any()
        t = j // 128 * 128                             # a masked key's probability is 0 and meets the value inside its tile of rows
        o3[t:, 3, 5] = want[t:, 3, 5] = 0
        assert torch.equal(torch.nan_to_num(o3, 9.0), torch.nan_to_num(want, 9.0)), j
        assert torch.equal(torch.nan_to_num(lse3, 9.0), torch.nan_to_num(want_lse, 9.0)), j
    ctx.close()
