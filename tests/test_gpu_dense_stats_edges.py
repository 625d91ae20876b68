"""Block column statistics of the dense loop at the edges of their kernels (512 and 128 keys per CTA, short last tiles,
blocks that do not align with tiles, one block, a key chunk beyond the last block of a group) against binary32 PyTorch."""
import pytest

from paper_2609_29812_b200 import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("L,H,q_block", [(1, 1, 64), (127, 2, 64), (300, 2, 128), (513, 16, 64), (1024, 16, 100), (1700, 16, 200),
                                         (1537, 16, 700), (2049, 12, 1024), (1281, 4, 2048), (7000, 16, 7000)])
def test_dense_column_statistics_edges(L, H, q_block):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    ctx = B.Context(0)
    w = workloads.replace(workloads.config2(L=L, n_heads=H), q_block=q_block)
    sh = P.shape_of(w)
    g = torch.Generator(device="cuda").manual_seed(L)
    q, k, v = (torch.randn(L, H, 128, generator=g, device="cuda").bfloat16() for _ in range(3))
    nb = -(-L // q_block)
    o = torch.empty_like(q)
    lse = torch.empty(H, L, device="cuda")
    scores = torch.full((H, nb, L), -1.0, device="cuda")
    B.fl_dense_loop_attention(ctx, sh, q, k, v, o, lse, scores)
    causal = torch.ones(L, L, dtype=torch.bool, device="cuda").tril_()
    for h in range(H):
        p = ((q[:, h].float() @ k[:, h].float().T) * w.sm_scale).masked_fill_(~causal, float("-inf"))
        p = torch.exp(p - torch.logsumexp(p, 1, keepdim=True))
        for b in range(nb):
            hi = min(L, (b + 1) * q_block)
            want = p[b * q_block:hi, :hi].double().sum(0).float()
            torch.testing.assert_close(scores[h, b, :hi], want, rtol=2e-3, atol=1e-5)
    ctx.close()
