"""The compiled marshalling on a GPU: what a caller passes is what is used, and errors keep their types."""
import pytest
import torch

import paper_2603_15965_b200 as M

pytestmark = pytest.mark.gpu


def test_out_of_memory_is_torchs_own_error():
    ids, breaks = torch.zeros(50_000_000, dtype=torch.int32, device="cuda"), torch.tensor([0, 5], dtype=torch.int32, device="cuda")
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction(1e-4)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            M.molora_route_vocab(ids, breaks)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert not M.molora_route_vocab(ids, breaks).any()
