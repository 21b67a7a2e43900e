"""The Python binding's own host work, without a GPU."""
import types

import pytest
import torch

from paper_2510_13161_b200 import binding


def test_accept_result_follows_its_tensors():
    """The addresses handed to the library are those of the tensors as they are now, however they came to lie elsewhere."""
    out = binding.AcceptResult(2, 3, "cpu")
    current = lambda: [getattr(out, f).data_ptr() for f, _ in binding.AcceptOut._fields_]        # noqa: E731
    passed = lambda: [getattr(out.struct(), f) for f, _ in binding.AcceptOut._fields_]           # noqa: E731
    assert passed() == current()
    out.emitted = torch.empty((2, 4), dtype=torch.int32)
    assert passed() == current()
    out.n_accepted.resize_(1 << 16)
    assert passed() == current()
    out.reuse_slot.set_(torch.empty(7, dtype=torch.int32))
    assert passed() == current()
    out.decide_row.data = torch.empty(5, dtype=torch.int32)
    assert passed() == current()


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_torchs_private_names(missing, monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 11 + device, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=22))
    assert binding._stream(None) == 14 and binding._stream(types.SimpleNamespace(cuda_stream=33)) == 33
    monkeypatch.delattr(torch._C, missing)
    assert binding._stream(None) == 22
