"""What the compiled marshalling refuses before it reaches the library (no GPU needed: host tensors are among the refusals)."""
import pytest
import torch

import paper_2603_15965_b200 as M
from paper_2603_15965_b200.binding import _ProjDescC

I = torch.zeros(3, dtype=torch.int32)
X = torch.zeros(3, 8)


class Pointer:
    """Device memory that is no torch tensor."""

    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


def test_null_and_foreign_pointers_are_the_librarys_to_judge():
    descs = (_ProjDescC * 1)(_ProjDescC(0x1000, 64, 0x2000, 64, 0x3000, 0x4000, 64, 64, 16, 1.0, None))
    empty, some = (descs, 0, 2, M.BF16), (descs, 5, 2, M.BF16)
    before = M.molora_launch_count()
    M.molora_apply_batched(None, I, None, stream=0, packed=empty)                  # no tokens: perm may be null
    M.molora_apply_batched(None, Pointer(0x1000), Pointer(0x1000), dev_status=Pointer(0x1000), stream=0, packed=empty)
    for offsets, perm in ((None, I), (I, None)):
        with pytest.raises(M.MoloraError, match="invalid argument"):
            M.molora_apply_batched(None, offsets, perm, stream=0, packed=some)
    with pytest.raises(AttributeError):
        M.molora_apply_batched(None, object(), I, stream=0, packed=empty)
    assert M.molora_launch_count() == before


@pytest.mark.parametrize("call,error", [
    (lambda: M.molora_route_vocab(I, I), ValueError),                                   # host tensor
    (lambda: M.molora_route_vocab(None, I), TypeError),
    (lambda: M.molora_route_composite(I, I, I, 2), ValueError),
    (lambda: M.molora_route_gate(X, torch.zeros(8, 2)), ValueError),
    (lambda: M.molora_route_mlp(X, X, None, X, None), ValueError),
    (lambda: M.molora_group(I, 2), ValueError),
    (lambda: M.molora_group_apply_batched(I, []), ValueError),
    (lambda: M.molora_apply_batched([M.ProjDesc(X, X, X, X)], I, I), ValueError),
    (lambda: M.molora_apply_batched([object()], I, I), AttributeError),
    (lambda: M.molora_topk_softmax(torch.zeros(3), 1), ValueError),                     # not two-dimensional
    (lambda: M.molora_apply_topk([M.ProjDesc(X, X, X, X)], I, X, 2), ValueError),
])
def test_refusals(call, error):
    before = M.molora_launch_count()
    with pytest.raises(error):
        call()
    assert M.molora_launch_count() == before
