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
