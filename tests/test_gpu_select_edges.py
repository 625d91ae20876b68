"""Token selection at the edges of its kernels (one CTA, a cluster of CTAs with a short or empty last piece, all kept, ties
across pieces, few distinct scores, keys that share all or none of their leading bits), exact on its own scores."""
import numpy as np
import pytest

from oracle import flashloop_oracle as fo
from paper_2609_29812_b200 import workloads
from helpers import to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,k,kind", [(1, 1, "spread"), (33, 32, "spread"), (4096, 400, "spread"), (4097, 4096, "spread"),
                                      (4100, 1, "ties"), (33001, 3300, "ties"), (33001, 33001, "spread"), (70003, 7001, "narrow"),
                                      (9000, 4500, "equal"), (20001, 19999, "few")])
def test_token_selection_edges(n, k, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P
    rng = np.random.default_rng(n)
    L, d = n + 7, 256
    ctx = B.Context(0)
    w = workloads.replace(workloads.config1(), L=L)
    sh = P.shape_of(w)
    step = {"spread": lambda: 10.0 ** rng.uniform(-6, 3, L), "narrow": lambda: rng.uniform(0.30, 0.3001, L),
            "ties": lambda: np.where(np.arange(L) % 3 == 0, 0.5, rng.uniform(0, 1, L)), "equal": lambda: np.full(L, 0.25),
            "few": lambda: rng.integers(0, 4, L) * 0.125}[kind]().astype(np.float32)
    g = torch.Generator().manual_seed(n)
    row = torch.randn(1, d, generator=g)
    prev = (torch.ones(L, 1) * row).cuda()                       # equal rows: equal steps give exactly equal scores
    cur = (prev + torch.from_numpy(step)[:, None].cuda()).contiguous()
    cand_np = np.sort(rng.permutation(L)[:n])
    for cand in (torch.from_numpy(cand_np.astype(np.int32)).cuda(),) + ((None,) if kind == "spread" else ()):
        pos = cand_np if cand is not None else np.arange(L)
        sel = P.select_tokens(ctx, sh, 2, prev, cur, cand, k)
        want = pos[fo.topk_ascending(to_np(sel.scores), min(k, len(pos)))]
        assert np.array_equal(to_np(sel.active_idx), want)
        assert np.array_equal(to_np(sel.slot_of_pos), fo.slot_map(want, L))
    ctx.close()
