"""The stream handle of a call without a stream, with and without PyTorch's
private way to it."""
import types

import pytest
import torch

from paper_1901_01488_gb300 import esc


@pytest.mark.parametrize("missing", [(), ("_raw_stream",), ("_get_device",), ("_raw_stream", "_get_device")])
def test_current_stream(monkeypatch, missing):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(esc, "_raw_stream", lambda d: 77 if d == 3 else 0)
    monkeypatch.setattr(esc, "_get_device", lambda: 3)
    for name in missing:
        monkeypatch.setattr(esc, name, None)
    assert esc._stream(None) == 77
    assert esc._stream(types.SimpleNamespace(cuda_stream=5)) == 5 and esc._stream(9) == 9


def test_without_the_private_names():
    """The module loads where PyTorch has neither."""
    import importlib.util
    held = {n: getattr(torch._C, n) for n in ("_cuda_getCurrentRawStream", "_cuda_getDevice") if hasattr(torch._C, n)}
    try:
        for n in held:
            delattr(torch._C, n)
        spec = importlib.util.spec_from_file_location("paper_1901_01488_gb300._esc_without", esc.__file__)
        m = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(m)
        assert m._raw_stream is None and m._get_device is None
    finally:
        for n, f in held.items():
            setattr(torch._C, n, f)


@pytest.mark.gpu
def test_both_ways_agree(monkeypatch):
    st = torch.cuda.Stream()
    for ctx in (torch.cuda.stream(st), torch.cuda.stream(torch.cuda.default_stream())):
        with ctx:
            fast = esc._stream(None)
            with monkeypatch.context() as m:
                m.setattr(esc, "_raw_stream", None)
                assert esc._stream(None) == fast == torch.cuda.current_stream().cuda_stream
