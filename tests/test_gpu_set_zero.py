"""The zeroed output of a ranker gradient: whole, ordered on its stream, refused without a pointer."""
import ctypes as C

import pytest
import torch

from paper_2403_18901_gb300 import qdec


def test_null_is_refused():
    L = qdec.lib()
    assert L.qd_set_zero(None, 4, None) != 0
    assert L.qd_set_zero(None, 0, None) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 3, 4095, 4096])
@pytest.mark.parametrize("side", [False, True])
def test_zeros(n, side):
    s = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(s):
        torch.full((n,), 3.0, device="cuda")  # the allocator's block for the next tensor
        z = qdec.zeros(n)
        assert z.dtype == torch.float32 and z.shape == (n,)
        assert torch.equal(z, torch.zeros_like(z))
        x = torch.ones(n + 2, device="cuda")
        assert qdec.lib().qd_set_zero(x.data_ptr() + 4, 4 * n, C.c_void_p(s.cuda_stream)) == 0
        assert x[0] == 1 and x[-1] == 1 and not x[1:-1].any()
