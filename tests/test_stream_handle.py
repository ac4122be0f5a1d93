"""The stream that a call without one runs on: the current stream's handle, with
and without torch's undocumented getter."""
import types

import pytest


def test_without_the_raw_getter(monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_1311_0380_gb300 import api
    monkeypatch.setattr(api, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    assert api._stream(None) == 77
    assert api._stream(types.SimpleNamespace(cuda_stream=5)) == 5


def test_import_without_the_raw_getter(monkeypatch):
    import importlib
    torch = pytest.importorskip("torch")
    from paper_1311_0380_gb300 import api
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    spec = importlib.util.spec_from_file_location("paper_1311_0380_gb300.api_again", api.__file__)
    again = importlib.util.module_from_spec(spec)
    monkeypatch.setitem(__import__("sys").modules, spec.name, again)
    spec.loader.exec_module(again)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=9))
    assert again._stream(None) == 9


@pytest.mark.gpu
@pytest.mark.parametrize("raw", [True, False])
def test_the_current_stream_is_taken(raw, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_0380_gb300 import api
    if not raw:
        monkeypatch.setattr(api, "_raw_stream", None)
    side = torch.cuda.Stream()
    assert api._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert api._stream(None) == side.cuda_stream == api._stream(side)
