"""Scratch memory of the Python calls when the device has no room for what a call asks
for: FP64 forms, which also work in less, fall back to the caller's workspace; the others
report the lack of memory.  (Allocation is faked: no GPU.)"""
import pytest
import torch

from paper_0912_1459_gb300 import cdsigma


@pytest.fixture
def full(monkeypatch):
    def no_room(nbytes, device):
        raise torch.OutOfMemoryError("no room")
    monkeypatch.setattr(cdsigma, "_workspace", no_room)


def test_a_large_enough_workspace_is_used(full):
    ws = torch.empty(64, dtype=torch.uint8)
    assert cdsigma._scratch(64, ws, ws.device, False) is ws


def test_a_smaller_one_is_tried_where_there_is_no_room(full):
    ws = torch.empty(16, dtype=torch.uint8)
    assert cdsigma._scratch(64, ws, ws.device, True) is ws
    with pytest.raises(torch.OutOfMemoryError):
        cdsigma._scratch(64, ws, ws.device, False)
    with pytest.raises(torch.OutOfMemoryError):
        cdsigma._scratch(64, None, ws.device, True)


def test_a_smaller_one_is_replaced_where_there_is():
    ws = torch.empty(16, dtype=torch.uint8)
    got = cdsigma._scratch(64, ws, ws.device, True)
    assert got is not ws and got.numel() == 64
