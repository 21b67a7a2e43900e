"""The Python binding's own host work, without a GPU."""
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
