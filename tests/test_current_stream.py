"""The default stream of a call comes from the public torch function where the
quick one is not there (host only)."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_1605_05320_gb300 import swadj as S


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_public_call_where_the_quick_one_is_missing(monkeypatch, missing):
    for name, fn in (("_cuda_getCurrentRawStream", lambda d: 11), ("_cuda_getDevice", lambda: 0)):
        monkeypatch.setattr(torch._C, name, fn, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda *a: types.SimpleNamespace(cuda_stream=22))
    assert S._stream(None) == 11
    monkeypatch.delattr(torch._C, missing)
    assert S._stream(None) == 22
