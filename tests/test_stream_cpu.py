"""The binding's stream handle does not depend on a private call of PyTorch."""
import types

import torch

from test_abi_cpu import W  # noqa: F401  (fixture)


def test_stream_handle_without_the_private_call(W, monkeypatch):  # noqa: F811
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=7))
    assert W._stream() == 7
    assert W._stream(types.SimpleNamespace(cuda_stream=9)) == 9
