"""Grouping inside the apply kernels where it changes its form: around a token per thread of each kernel (256, 384, 448 threads), around
whole warps, at 1, 31, 32 and 33 adapters, with unrouted and flagged tokens -- bit-equal to the oracle, and y to the two-call form."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import dev_tensor

pytestmark = pytest.mark.gpu

KERNELS = {"stream": {"umma_min_tokens": 1000000, "small_path": 1}, "twophase": {"umma_min_tokens": 1000000, "small_path": 2},
           "jobs": {"umma_min_tokens": 1000000, "small_path": 3}, "umma": {"umma_min_tokens": 1}}


@pytest.fixture(autouse=True)
def _default_kernels_afterwards():
    yield
    for k in M.TUNING_NAMES:
        M.molora_debug_set(k, 0)


@pytest.mark.parametrize("kernel", list(KERNELS))
@pytest.mark.parametrize("N", [1, 31, 32, 33, 255, 256, 257, 383, 384, 385, 447, 448, 449, 1000])
@pytest.mark.parametrize("C", [1, 2, 5, 31, 32, 33])
def test_grouping_inside(kernel, N, C):
    for k, v in KERNELS[kernel].items():
        M.molora_debug_set(k, v)
    w = W.random_problem(N * 64 + C, N, C, 128, 192, 16, "bf16", unrouted_frac=0.1 if N > 10 else 0.0)
    r = w.r.copy()
    if N > 40:
        r[7], r[39], r[N - 1] = C, -7, 255
    clean = np.where((r >= 0) & (r < C), r, -1).astype(np.int32)
    p = w.projections[0]
    x, A, B = dev_tensor(w.inputs["x"], "bf16"), dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16")
    ya, yb = dev_tensor(p.y, "bf16"), dev_tensor(p.y, "bf16")
    counts, offsets, perm = M.molora_group(dev_tensor(clean, "i"), C)
    M.molora_apply(x, ya, A, B, offsets, perm)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = M.molora_group_apply_batched(dev_tensor(r, "i"), [M.ProjDesc(x, yb, A, B)], dev_status=status)
    c, o, q = oracle.group(clean, C)
    assert np.array_equal(got[0].cpu().numpy(), c) and np.array_equal(got[1].cpu().numpy(), o)
    assert np.array_equal(got[2].cpu().numpy()[: o[-1]], q[: o[-1]])
    assert torch.equal(ya, yb) and (int(status.item()) != 0) == (N > 40)
