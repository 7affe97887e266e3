"""The binding's default stream is torch's current one, also with a torch that
lacks the private call for its raw handle."""
import types

import pytest

from paper_2601_16736_gb300 import gsopt

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("raw", [True, False])
def test_default_stream_is_the_current_one(monkeypatch, raw):
    handle = {0: 0x1000, 3: 0x3000}
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=handle[3]))
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: handle[d], raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert gsopt._stream(None).value == handle[3]
    assert gsopt._stream(0x42).value == 0x42
    assert gsopt._stream(types.SimpleNamespace(cuda_stream=0x43)).value == 0x43
