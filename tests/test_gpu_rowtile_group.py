"""Grouping inside the CUDA-core apply (fp32 storage, or rank 8): both sides of its limits, against the two-call form and the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import assert_close, dev_tensor, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,d_in,d_out,rank,dtype,one", [
    (1, 1, 8, 8, 8, "f32", 1), (256, 2, 512, 512, 8, "f32", 1), (255, 3, 1032, 520, 8, "bf16", 1), (600, 100, 64, 72, 8, "bf16", 1),
    (300, 32, 256, 256, 16, "f32", 1), (290, 33, 256, 256, 32, "f32", 1), (33, 130, 64, 64, 64, "f32", 1), (2048, 20, 64, 96, 8, "f32", 1),
    (2049, 4, 64, 96, 8, "f32", 0), (2048, 21, 64, 96, 8, "f32", 0), (100, 7, 200, 264, 16, "bf16", 0),
])
def test_one_call_matches_two(N, C, d_in, d_out, rank, dtype, one):
    w = W.random_problem(N + C + rank, N, C, d_in, d_out, rank, dtype, unrouted_frac=0.1 if N > 10 else 0.0)
    p = w.projections[0]
    r, x, A, B = dev_tensor(w.r, "i"), dev_tensor(w.inputs["x"], dtype), dev_tensor(p.A, dtype), dev_tensor(p.B, dtype)
    ya, yb = dev_tensor(p.y, dtype), dev_tensor(p.y, dtype)
    counts, offsets, perm = M.molora_group(r, C)
    M.molora_apply(x, ya, A, B, offsets, perm)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    before = M.molora_launch_count()
    got = M.molora_group_apply_batched(r, [M.ProjDesc(x, yb, A, B)], dev_status=status)
    assert M.molora_launch_count() - before == (1 if one else 2)
    total = int(offsets[-1])
    assert torch.equal(got[0], counts) and torch.equal(got[1], offsets) and torch.equal(got[2][:total], perm[:total])
    assert torch.equal(ya, yb) and int(status.item()) == 0
    ref, _ = oracle.apply(w.inputs["x"], p.y, p.A, p.B, w.r)
    assert_close(to_f64(yb), ref)


def test_several_projections_and_bad_routes():
    N, C = 200, 5
    ws = [W.random_problem(i, N, C, 64, o, 8, "f32") for i, o in enumerate((64, 128, 8))]
    r = ws[0].r.copy()
    r[3], r[7] = C, -5                                  # flagged, and left alone as unrouted tokens are
    ys = [dev_tensor(w.projections[0].y, "f32") for w in ws]
    projs = [M.ProjDesc(dev_tensor(w.inputs["x"], "f32"), y, dev_tensor(w.projections[0].A, "f32"), dev_tensor(w.projections[0].B, "f32"))
             for w, y in zip(ws, ys)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    counts, offsets, perm = M.molora_group_apply_batched(dev_tensor(r, "i"), projs, dev_status=status)
    assert int(status.item()) != 0
    r[3] = r[7] = -1
    c, o, q = oracle.group(r, C)
    assert np.array_equal(counts.cpu().numpy(), c) and np.array_equal(offsets.cpu().numpy(), o) and np.array_equal(perm.cpu().numpy()[: o[-1]], q)
    for w, y in zip(ws, ys):
        p = w.projections[0]
        ref, _ = oracle.apply(w.inputs["x"], p.y, p.A, p.B, r)
        assert_close(to_f64(y), ref, 1e-5, 1e-4)
