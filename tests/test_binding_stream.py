"""The current stream's handle: through torch's public call first (it initialises CUDA) and wherever the functions
beneath it do not exist, through those otherwise."""
from types import SimpleNamespace

import pytest
import torch

from paper_2505_00347_b200 import binding as B


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",)])
def test_stream_handle_with_and_without_the_private_functions(monkeypatch, missing):
    public = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: public.append(1) or SimpleNamespace(cuda_stream=77))
    names = {"_cuda_getCurrentRawStream": lambda device: 100 + device, "_cuda_getDevice": lambda: 3}
    monkeypatch.setattr(torch, "_C", SimpleNamespace(**{k: v for k, v in names.items() if k not in missing}))
    monkeypatch.setattr(B, "_raw_stream", None, raising=False)
    assert B._stream() == 77
    assert [B._stream(), B._stream()] == ([77, 77] if missing else [103, 103])
    assert len(public) == (3 if missing else 1)
