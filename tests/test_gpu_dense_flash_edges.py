"""Output and log-normalisers of the dense loop where its tiles end (pairs of 128 query rows, chunks of 128 keys: a single row,
a pair without its second tile, a second tile of one row) and with logits that make the reference move, against binary32
PyTorch."""
import pytest

from paper_2609_29812_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("boost", [1.0, 64.0])
@pytest.mark.parametrize("L,H", [(1, 1), (33, 3), (128, 2), (129, 1), (256, 2), (257, 16), (383, 4), (1025, 3), (2500, 8)])
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
