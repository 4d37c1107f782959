"""The binding's stream lookup without a GPU: torch's raw stream handle where torch
has it, else the handle of its current stream."""
import sys
import types

import pytest

import paper_2302_04180_gb300 as rbs


class Tensor:
    is_cuda = True
    device = "cuda:1"

    def get_device(self):
        return 1


@pytest.mark.parametrize("raw", [True, False])
def test_a_torch_without_the_raw_handle_still_works(monkeypatch, raw):
    torch = types.ModuleType("torch")
    torch._C = types.SimpleNamespace(**({"_cuda_getCurrentRawStream": lambda d: 100 + d} if raw else {}))
    torch.cuda = types.SimpleNamespace(current_stream=lambda d: types.SimpleNamespace(cuda_stream=200 + int(str(d)[-1])))
    monkeypatch.setitem(sys.modules, "torch", torch)
    monkeypatch.setattr(rbs, "_raw_stream", None)
    assert rbs._stream(None, None, Tensor()) == (101 if raw else 201)
    assert rbs._stream(None, Tensor()) == (101 if raw else 201)
    assert rbs._stream(7, Tensor()) == 7
