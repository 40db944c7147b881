"""The torch allocator behind the library's device memory, on a stand-in for
torch's caching allocator (no GPU)."""
import types

import pytest


@pytest.mark.parametrize("device", ["cuda", "cuda:0", 0], ids=str)
def test_a_device_without_an_index_is_the_current_one(monkeypatch, device):
    """Batch(device="cuda") and TorchAllocator("cuda"): the caching allocator takes
    a device only with its index, and a refusal there reads as out of memory."""
    import torch
    from torch.cuda._utils import _get_device_index
    from paper_1202_6130_gb300.sim import TorchAllocator
    calls = []

    def alloc(size, device=None, stream=None):
        calls.append((size, _get_device_index(device), stream))
        return 0x1000

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    a = TorchAllocator(device, types.SimpleNamespace(cuda_stream=7))
    assert a._alloc_cb(256, None) == 0x1000
    assert calls == [(256, 0, 7)]
