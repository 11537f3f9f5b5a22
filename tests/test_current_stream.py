"""The handle of the current torch stream, with and without the private
functions that give it without a Stream object."""
import sys
import types

import pytest


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",),
                                     ("_cuda_getCurrentRawStream", "_cuda_getDevice")])
def test_current_stream_of_any_torch(alp, monkeypatch, missing):
    state = {"device": 0, "streams": {0: 11, 1: 21}}
    c = {"_cuda_getCurrentRawStream": lambda d: state["streams"][d],
         "_cuda_getDevice": lambda: state["device"]}
    torch = types.ModuleType("torch")
    torch._C = types.SimpleNamespace(**{k: v for k, v in c.items() if k not in missing})
    torch.cuda = types.SimpleNamespace(current_stream=lambda: types.SimpleNamespace(
        cuda_stream=state["streams"][state["device"]]))
    monkeypatch.setitem(sys.modules, "torch", torch)
    for name in ("_torch_c", "_raw"):
        if hasattr(alp, name):
            monkeypatch.setattr(alp, name, None)
    assert alp._s(None) == 11
    state["streams"][0] = 12
    assert alp._s(None) == 12
    state["device"] = 1
    assert alp._s(None) == 21
    assert alp._s(7) == 7
