"""The pools that pipeline keeps for the process (status words, rows of a loop): one per device, whatever the caller calls
the device.  Allocations are recorded, no GPU is needed."""
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def two_gpus(monkeypatch):
    """pipeline on a machine with two GPUs: `made` receives the device of every allocation, `gpu[0]` is current."""
    from paper_2609_29812_b200 import binding as B, pipeline as P
    made, gpu = [], [0]
    real = torch.zeros

    def alloc(*size, dtype=None, device=None):
        dev = torch.device(device)
        made.append(gpu[0] if dev.index is None else dev.index)
        return real(*size, dtype=dtype)
    monkeypatch.setattr(P, "_STATUS", {})
    monkeypatch.setattr(P, "_ROWS_WS", {})
    monkeypatch.setattr(B, "_stream_of", lambda index: None)       # the default stream of either device
    monkeypatch.setattr(torch.cuda, "current_device", lambda: gpu[0])
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(torch, "zeros", alloc)
    monkeypatch.setattr(torch, "empty", alloc)
    return P, made, gpu


def test_status_words_of_two_devices(two_gpus):
    P, made, gpu = two_gpus
    first = P.status_word("cuda")
    gpu[0] = 1
    second = P.status_word("cuda")
    assert made == [0, 1] and first.data_ptr() != second.data_ptr()
    assert P.status_word(torch.device("cuda:1")).data_ptr() == second.data_ptr() + 4     # the same block by its full name
    assert P.status_word("cuda:0").data_ptr() == first.data_ptr() + 4 and made == [0, 1]


def test_rows_of_two_devices(two_gpus):
    P, made, gpu = two_gpus
    first = P.rows_workspace("cuda", 4, 8)
    gpu[0] = 1
    second = P.rows_workspace("cuda", 4, 8)
    assert made == [0] * 4 + [1] * 4
    assert P.rows_workspace("cuda:1", 2, 8) is second and P.rows_workspace("cuda:0", 2, 8) is first
