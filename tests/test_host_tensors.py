"""exw_extrapolate_host addresses its host tensors item by item: what is too short for that, or has elements of another
size, is refused before anything is launched, and a tensor longer than the call needs keeps its own strides.

No GPU: the library call is replaced by one that records its descriptors, and the device staging tensors live on the host.
"""
import struct

import pytest
import torch

from paper_2307_12607_gb300 import binding

F, NF, H, W = 2, 2, 4, 6


class Recorder:
    def __init__(self):
        self.calls = []

    def exw_workspace_bytes(self, *args):
        return 256

    def exw_extrapolate_host(self, *args):
        self.calls.append(args)
        return 0


@pytest.fixture
def recorder(monkeypatch):
    rec = Recorder()

    def dev(t, name, dtype=None, shape=None):
        if tuple(t.shape) != tuple(shape) or t.dtype != dtype:
            raise ValueError(f"{name} does not fit")
        return t.data_ptr()

    monkeypatch.setattr(binding, "lib", lambda: rec)
    monkeypatch.setattr(binding, "_dev", dev)
    monkeypatch.setattr(binding, "_stream", lambda stream, device: 0)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    return rec


def tensors(**change):
    t = {"color": torch.zeros(F, 3, H, W), "depth": torch.zeros(F, H, W), "mv": torch.zeros(F, 2, H, W),
         "out": torch.zeros(F, NF, 3, H, W), "mask": torch.zeros(F, NF, H, W, dtype=torch.uint8)}
    t.update(change)
    return t


def call(t, direct):
    staging = tensors()
    return binding.exw_extrapolate_host(
        t["color"], t["depth"], t["mv"], nfrac=NF, out=t["out"], mask=t["mask"],
        dev_in=(staging["color"], staging["depth"], staging["mv"]), dev_out=(staging["out"], staging["mask"]),
        ws=torch.zeros(256, dtype=torch.uint8), stream=0, direct=direct)


BAD = {
    "depth": [torch.zeros(F - 1, H, W), torch.zeros(F, H - 1, W), torch.zeros(F), torch.zeros(F, H, W).half(),
              torch.zeros(F, H, W).double()],
    "mv": [torch.zeros(F - 1, 2, H, W), torch.zeros(F, 1, H, W), torch.zeros(F, 2, H, W).double()],
    "out": [torch.zeros(F - 1, NF, 3, H, W), torch.zeros(F, NF - 1, 3, H, W), torch.zeros(F, NF, 3, H, W - 1),
            torch.zeros(F * NF, 3, H, W), torch.zeros(F, NF, 3, H, W).half(), torch.zeros(F)],
    "mask": [torch.zeros(F - 1, NF, H, W, dtype=torch.uint8), torch.zeros(F, NF - 1, H, W, dtype=torch.uint8),
             torch.zeros(F, NF, H - 1, W, dtype=torch.uint8), torch.zeros(F, NF, H, W, dtype=torch.int32)],
    "color": [torch.zeros(F, 2, H, W)],
}


@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("name,index", [(n, i) for n, bad in BAD.items() for i in range(len(bad))])
def test_host_tensor_that_does_not_fit_is_refused(recorder, name, index, direct):
    with pytest.raises((ValueError, TypeError, IndexError), match=name):
        call(tensors(**{name: BAD[name][index]}), direct)
    assert recorder.calls == []


LONGER = {
    "depth": torch.zeros(F + 1, H, W),
    "mv": torch.zeros(F + 2, 3, H, W),
    "out": torch.zeros(F + 1, NF + 1, 4, H, W),
    "mask": torch.zeros(F, NF + 2, H, W, dtype=torch.bool),
    "color": torch.zeros(F, 4, H, W),
}


@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("name", [None] + list(LONGER))
def test_items_are_addressed_by_the_tensors_own_strides(recorder, name, direct):
    t = tensors(**({name: LONGER[name]} if name else {}))
    call(t, direct)
    host, _, nframes, nfrac, _, outs, dev_outs = recorder.calls[0][:7]
    assert (nframes, nfrac) == (F, NF) and (dev_outs is None) == direct
    frames = struct.unpack("@" + "PPPiii4x" * F, host)
    for f in range(F):
        assert frames[6 * f:6 * f + 6] == (t["color"][f].data_ptr(), t["depth"][f].data_ptr(), t["mv"][f].data_ptr(),
                                           W, H, binding._cdt(t["color"]))
    addresses = struct.unpack(f"@{2 * F * NF}P", outs)
    assert addresses == tuple(p for f in range(F) for j in range(NF)
                              for p in (t["out"][f, j].data_ptr(), t["mask"][f, j].data_ptr()))
