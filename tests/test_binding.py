"""The native call path of the package, without a GPU: calls that return before anything is launched."""
import torch

import paper_2410_15704_b200 as rvq


def test_buffers_that_a_call_writes_get_storage_of_their_own():
    """A lazily cloned tensor shares its storage until the first write.  A call's outputs are written on the
    device, so they have to part with the original when the call takes their address; inputs need not."""
    cfg = rvq.make_config(128, 32, 0, 8, 1024, 16, rvq.F32, 0)
    original = torch.zeros(1 << 12)
    codes, books, out, status = (torch._lazy_clone(original) for _ in range(4))
    rvq.rvq_decode(cfg, codes, None, 0, books, 256, out, 128, status, stream=0)
    assert torch._C._is_cow_tensor(codes) and torch._C._is_cow_tensor(books)
    assert not torch._C._is_cow_tensor(out) and not torch._C._is_cow_tensor(status)
    assert out.data_ptr() != original.data_ptr()
