"""The default stream's handle, with and without torch's raw-handle functions
(private names, which a release may drop)."""
import pytest

from paper_2609_04910_gb300 import _binding

torch = pytest.importorskip("torch")


class _Stream:
    cuda_stream = 0x1234


@pytest.fixture
def _stand_ins(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: _Stream())
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0x5600 + d, raising=False)
    return monkeypatch


def test_raw_handle(_stand_ins):
    assert _binding._stream_ptr(None) == 0x5603
    assert _binding._stream_ptr(_Stream()) == 0x1234


@pytest.mark.parametrize("name", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_public_path_where_a_name_is_missing(_stand_ins, name):
    _stand_ins.delattr(torch._C, name)
    assert _binding._stream_ptr(None) == 0x1234


def test_public_path_before_initialisation(_stand_ins):
    _stand_ins.setattr(torch.cuda, "is_initialized", lambda: False)
    assert _binding._stream_ptr(None) == 0x1234
