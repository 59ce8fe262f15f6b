"""What the compiled marshalling refuses before it reaches the library (no GPU needed: host tensors are among the refusals)."""
import pytest
import torch

import paper_2603_15965_b200 as M

I = torch.zeros(3, dtype=torch.int32)
X = torch.zeros(3, 8)


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
