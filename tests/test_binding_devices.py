"""Memory of another GPU than the one a call runs on is refused before anything is launched (stand-ins for the tensors: this needs no GPU)."""
import pytest
import torch

import paper_2502_08141_b200 as lw


class OnDevice:
    is_cuda = True

    def __init__(self, index):
        self.index, self.device = index, f"cuda:{index}"

    def get_device(self):
        return self.index


def test_other_device(monkeypatch):
    monkeypatch.setattr(lw, "_current_device", lambda: 1)
    lw._here(OnDevice(1), "X")
    with pytest.raises(ValueError, match="X is on cuda:0, the call runs on cuda:1"):
        lw._here(OnDevice(0), "X")


def test_pageable_host_memory():
    with pytest.raises(ValueError, match="maps must be a CUDA tensor"):
        lw._extent(torch.zeros(16), 16, "maps", torch.float32)
    lw._extent(None, 16, "maps", torch.float32)     # the library says that a pointer is missing
