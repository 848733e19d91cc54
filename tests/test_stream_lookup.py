"""The current stream's handle: what the first lookup keeps for the later ones is published by one store, so that another
thread finds all of it or none."""
import dis
import types

import torch

import paper_2204_06666_gb300 as eh


def test_lookups_are_published_at_once():
    stores = [i.argval for i in dis.get_instructions(eh._first_stream) if i.opname == "STORE_GLOBAL"]
    assert len(stores) == 1


def test_handle_of_the_current_stream(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=7))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 40 + dev, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 2, raising=False)
    monkeypatch.setattr(eh, "_lookups", None)
    assert eh._stream(None) == 7 and eh._stream(None) == 42
    assert eh._stream(5) == 5 and eh._stream(types.SimpleNamespace(cuda_stream=6)) == 6
