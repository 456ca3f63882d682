"""Where the function-style calls take their stream from: a CUDA device, an
index or nothing.  A host tensor is refused before any native call, so its
address never reaches a kernel."""
import pytest
import torch

from paper_2110_00511_gb300 import ash


@pytest.fixture
def streams(monkeypatch):
    monkeypatch.setattr(ash, "_stream_of", lambda index: 1000 + index)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 5)


@pytest.mark.parametrize("device,handle", [
    (None, 1005), (0, 1000), (3, 1003), (torch.device("cuda"), 1005), (torch.device("cuda", 2), 1002),
    ("cuda", 1005), ("cuda:1", 1001)])
def test_stream_of_a_cuda_device(streams, device, handle):
    assert ash._stream(device) == handle


@pytest.mark.parametrize("device", [torch.device("cpu"), torch.device("meta"), "cpu"])
def test_other_devices_are_refused(streams, device):
    with pytest.raises(ValueError):
        ash._stream(device)


def test_host_tensors_never_reach_the_library(streams, monkeypatch):
    called = []

    class Recorder:
        def __getattr__(self, name):
            return lambda *a: called.append(name) or 0

    monkeypatch.setattr(ash, "lib", lambda: Recorder())
    keys = torch.zeros((4, 3), dtype=torch.int32)
    idx, mask = torch.zeros(4, dtype=torch.int32), torch.zeros(4, dtype=torch.bool)
    for call in (lambda: ash.ash_find(None, keys, idx, mask), lambda: ash.ash_activate(None, keys, idx, mask),
                 lambda: ash.ash_insert(None, keys, [], idx, mask), lambda: ash.ash_erase(None, keys, mask),
                 lambda: ash.ash_gather_keys(None, idx, keys)):
        with pytest.raises(ValueError):
            call()
    assert not called
