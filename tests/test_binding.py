"""The binding's packed descriptors and its loading of the library (no GPU)."""
import ctypes
import dis

import torch

import paper_2606_24647_gb300 as px


def _batch(a):
    return px.px_batch.from_address(a.buffer_info()[0])


def test_negative_row_count_reaches_the_library():
    for n in (0, 7, -1, -2**63, 2**31):
        a = px._pack([], n)
        assert _batch(a).nrows == n and _batch(a).ncols == 0
    # which refuses it, as any row count out of range, before it touches the device
    a, offsets = px._pack([], -1), ctypes.c_int64()
    px.load()
    st = px._calls.px_gather(px._at(a), None, None, px._at(a), None, 0, None)
    assert st == px.PX_ERR_UNSUPPORTED and "nrows -1" in px.last_error()


def test_library_appears_with_its_calls():
    """A thread that finds the library loaded finds the operator calls too: load() stores
    them first."""
    stores = [i.argval for i in dis.get_instructions(px.load) if i.opname == "STORE_GLOBAL"]
    assert stores == ["_calls", "_lib"]


def test_current_stream_without_the_private_call(monkeypatch):
    class Stream:
        cuda_stream = 0x1234
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    assert px._stream(None) == 0x1234 and px._stream(Stream) == 0x1234
