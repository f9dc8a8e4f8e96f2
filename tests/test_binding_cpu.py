"""The Python side of the binding that needs no GPU: routing tables and the stream handle."""
import pytest
import torch

from paper_2502_16927_b200 import binding


@pytest.mark.parametrize("E,k,T", [(8, 2, 16), (7, 3, 5), (64, 8, 4096), (1, 1, 1)])
def test_routing_tables(E, k, T):
    layer = binding.Layer.__new__(binding.Layer)
    layer.handle, layer.cfg, layer.device = None, dict(E=E, k=k), torch.device("cpu")
    R = layer.empty_routing(T)
    shapes = dict(topk_idx=T * k, topk_w=T * k, counts=E, offsets=E + 1, row_of_slot=T * k, slot_of_row=T * k, counts_chosen=E, aux_loss=1)
    assert {name: t.numel() for name, t in R.items()} == shapes
    spans = sorted((t.data_ptr(), t.data_ptr() + 4 * t.numel()) for t in R.values())
    assert all(a[1] <= b[0] for a, b in zip(spans, spans[1:]))                  # none overlaps another
    for name, t in R.items():
        assert t.is_contiguous() and t.data_ptr() % 16 == 0, name
        assert t.dtype == (torch.float32 if name in ("topk_w", "aux_loss") else torch.int32), name
    # what a program keeps of a step (its loss, its loads) does not keep the tables of all slots with it
    for name in ("aux_loss", "counts", "counts_chosen", "offsets"):
        assert R[name].untyped_storage().nbytes() <= 4 * (3 * (E + 3) + 5), name


def test_stream_handle_without_the_private_accessors(monkeypatch):
    class Stream:
        cuda_stream = 1234

    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: Stream)
    monkeypatch.setattr(binding, "_raw_stream", None)
    assert binding._stream() == 1234
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 10 * device)
    monkeypatch.setattr(binding, "_current_device", lambda: 7)
    assert binding._stream() == 70
