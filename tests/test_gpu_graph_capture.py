"""State made while a stream is being captured: nothing that the graph records may reach what is used outside it."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_status_words_made_under_capture(monkeypatch):
    """A word taken during the capture is cleared by every replay; one taken afterwards starts at zero and is not."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import pipeline as P
    monkeypatch.setattr(P, "_STATUS", {})
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        inside = P.status_word("cuda:0")
    with torch.cuda.stream(side):
        outside = [P.status_word("cuda:0") for _ in range(3)]
        assert all(int(w.item()) == 0 for w in outside)
        for w in outside:
            w.fill_(-5)
        inside.fill_(-5)
        graph.replay()
        assert int(inside.item()) == 0
        assert all(int(w.item()) == -5 for w in outside)


def test_workspace_lent_under_capture():
    """A context whose first layer state is made under capture: the next one made outside clears the arrival counters (the
    captured clear has not run; the fill stands for what the memory held)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_29812_b200 import binding as B, pipeline as P, workloads
    w = workloads.replace(workloads.config2(L=2000, n_heads=2), q_block=256, col_budget=96)
    ctx = B.Context(0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.LayerState(ctx, w)
    ws = ctx._workspace
    ws[:1024].fill_(127)
    P.LayerState(ctx, w)
    assert ctx._workspace is ws and not ws[:1024].any()
    ws[:1024].fill_(127)                      # held and cleared by now: every launch leaves the counters at zero itself
    P.LayerState(ctx, w)
    assert int(ws[0]) == 127
    ctx.close()
