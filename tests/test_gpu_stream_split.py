"""GPU parity of the streaming apply kernel against the CPU oracle where its tiling and its clusters can go wrong: segments around
the 16- and 32-row tiles, widths around a chunk (256, 512 or 1024 columns) and around a TMA box, every cluster size, more items
than clusters (the skewed order) and fewer."""
import numpy as np
import pytest
import torch

import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import dev_tensor, run_and_check

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _default_kernels_afterwards():
    yield
    for k in M.TUNING_NAMES:
        M.molora_debug_set(k, 0)


def force_stream(split, tile):
    for k, v in {"umma_min_tokens": 1000000, "small_path": 1, "stream_split": split, "stream_tile": tile}.items():
        M.molora_debug_set(k, v)


SEG_SIZES = [0, 1, 15, 16, 17, 31, 32, 33, 0, 63, 65]


@pytest.mark.parametrize("split", [1, 2, 4, 8])
@pytest.mark.parametrize("rank,tile", [(16, 16), (16, 32), (32, 16), (32, 32), (64, 16), (64, 32)])
@pytest.mark.parametrize("d_in,d_out", [(32, 32), (288, 544), (1056, 96), (4128, 1120)])
def test_segments_and_ragged_widths(rank, tile, split, d_in, d_out):
    force_stream(split, tile)
    r = W.segment_sizes_routing(SEG_SIZES)
    run_and_check(W.random_problem(split + rank + d_in, r.size, len(SEG_SIZES), d_in, d_out, rank, "bf16", r=r))


@pytest.mark.parametrize("split", [1, 2, 8])
@pytest.mark.parametrize("N,C", [(1, 1), (1, 256), (40, 33), (4096, 5), (4096, 256), (4097, 3)])
@pytest.mark.parametrize("rank", [16, 64])
def test_grouping_inside_and_many_items(N, C, rank, split):
    force_stream(split, 16)
    w = W.random_problem(N + C, N, C, 2080, 160, rank, "bf16", unrouted_frac=0.1 if N > 10 else 0.0)
    rows = None if N < 100 else np.random.default_rng(N).choice(N, 200, replace=False)
    run_and_check(w, rows=rows)
    # the one-call form writes the grouping of molora_group, bit for bit, and the same y
    p = w.projections[0]
    r = dev_tensor(w.r, "i")
    x, A, B = dev_tensor(w.inputs["x"], "bf16"), dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16")
    ya, yb = dev_tensor(p.y, "bf16"), dev_tensor(p.y, "bf16")
    counts, offsets, perm = M.molora_group(r, C)
    M.molora_apply(x, ya, A, B, offsets, perm)
    got = M.molora_group_apply_batched(r, [M.ProjDesc(x, yb, A, B)])
    total = int(offsets[-1])
    assert torch.equal(got[0], counts) and torch.equal(got[1], offsets) and torch.equal(got[2][:total], perm[:total])
    assert torch.equal(ya, yb)


@pytest.mark.parametrize("rank,split,d_in", [(32, 2, 1024), (32, 8, 4096), (64, 2, 512), (64, 4, 1024)])
def test_many_items_of_one_chunk_a_cta(rank, split, d_in):
    """The shortest items a cluster can have -- one shrink chunk a CTA and, for all but one CTA, no expand chunk -- and many of them,
    so that a slot of the exchange is reused as early as it can be."""
    force_stream(split, 16)
    w = W.random_problem(rank + split, 4000, 7, d_in, 32, rank, "bf16")
    run_and_check(w)
    p = w.projections[0]
    x, y, A, B = dev_tensor(w.inputs["x"], "bf16"), dev_tensor(p.y, "bf16"), dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16")
    _, offsets, perm = M.molora_group(dev_tensor(w.r, "i"), 7)
    first = M.molora_apply(x, y.clone(), A, B, offsets, perm)
    for _ in range(30):
        assert torch.equal(M.molora_apply(x, y.clone(), A, B, offsets, perm), first)
