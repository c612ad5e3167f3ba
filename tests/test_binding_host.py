"""The binding's own work on the host, without a GPU: output tensors and argument packing."""
import torch

from paper_2510_12966_b200 import binding


def test_outputs_are_tensors_of_their_own():
    a, b = binding._rows("cpu", torch.int32, (3,), 2)
    c, d = binding._rows("cpu", torch.int32, (3, 4), 2)
    assert [tuple(t.shape) for t in (a, b, c, d)] == [(3,), (3,), (3, 4), (3, 4)] and all(t.dtype == torch.int32 for t in (a, b, c, d))
    assert len({t.untyped_storage().data_ptr() for t in (a, b, c, d)}) == 4
    assert all(t.storage_offset() == 0 and t.is_contiguous() and t.untyped_storage().nbytes() == 4 * t.numel() for t in (a, b, c, d))
    d.view(torch.int64)                       # any of them as another type
    x, y = binding._rows("cpu", torch.float32, (2, 3), 2)
    x.zero_()
    w = torch.ones((2, 3), requires_grad=True)
    loss = (w * x).sum()
    y.clamp_(min=0)                           # one of them in place while autograd holds another
    loss.backward()
    y.detach_()
