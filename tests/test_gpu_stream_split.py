"""GPU parity of the streaming apply kernel against the CPU oracle where its tiling and its clusters can go wrong: segments around
the 16- and 32-row tiles, widths around a chunk (256, 512 or 1024 columns) and around a TMA box, every cluster size, more items
than clusters (the skewed order) and fewer."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import assert_close, dev_tensor, run_and_check, to_f64

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


@pytest.mark.parametrize("split", [1, 2, 4, 8])
@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("rank,k", [(16, 2), (32, 2), (16, 4)])
@pytest.mark.parametrize("N", [37, 500])
def test_adapter_sets_in_clusters(N, rank, k, tile, split):
    """Top-k in one pass: the adapters of a set side by side in a cluster's shares, their weights per token applied where the partials
    of the CTAs are summed."""
    force_stream(split, tile)
    C, d_in, d_out = 4, 2080, 1120
    rng = np.random.default_rng(N + rank + k)
    w = W.random_problem(700 + N + rank, N, C, d_in, d_out, rank, "bf16")
    p = w.projections[0]
    idx = np.stack([rng.permutation(C)[:k] for _ in range(N)], axis=1).astype(np.int32)
    weight = rng.random((k, N)).astype(np.float32)
    weight /= weight.sum(axis=0, keepdims=True)
    y = dev_tensor(p.y, "bf16")
    M.molora_apply_topk([M.ProjDesc(dev_tensor(w.inputs["x"], "bf16"), y, dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16"))],
                        dev_tensor(idx, "i"), dev_tensor(weight, "f32"), C)
    assert_close(to_f64(y), oracle.apply_topk(w.inputs["x"], p.y, p.A, p.B, idx, weight), what=f"top-{k} rank {rank}")


@pytest.mark.parametrize("split", [1, 2, 4, 8])
@pytest.mark.parametrize("rank", [32, 64])
def test_several_pitched_projections_in_clusters(rank, split):
    """Projections of different widths in one launch, rows of x and y further apart than they are wide, a LoRA scale and a factor per
    token; what lies between the rows of y stays as it is."""
    force_stream(split, 16)
    N, C = 333, 5
    rng = np.random.default_rng(rank)
    shapes = [(1056, 96), (4128, 1120), (2080, 4160), (1056, 32)]
    w = [W.random_problem(810 + i, N, C, a, b, rank, "bf16") for i, (a, b) in enumerate(shapes)]
    r, factor = w[0].r, rng.random(N).astype(np.float32)
    _, offsets, perm = M.molora_group(dev_tensor(r, "i"), C)
    descs, wide = [], []
    for v, (a, b) in zip(w, shapes):
        x = torch.full((N, a + 24), 3.0, dtype=torch.bfloat16, device="cuda")
        y = torch.full((N, b + 40), -7.0, dtype=torch.bfloat16, device="cuda")
        x[:, :a] = dev_tensor(v.inputs["x"], "bf16")
        y[:, :b] = dev_tensor(v.projections[0].y, "bf16")
        wide.append(y)
        descs.append(M.ProjDesc(x[:, :a], y[:, :b], dev_tensor(v.projections[0].A, "bf16"), dev_tensor(v.projections[0].B, "bf16"), 0.5,
                                dev_tensor(factor, "f32")))
    M.molora_apply_batched(descs, offsets, perm)
    for v, (a, b), y in zip(w, shapes, wide):
        p = v.projections[0]
        delta = oracle.apply(v.inputs["x"], np.zeros_like(p.y), p.A, p.B, r, 0.5)[0] * factor[:, None]
        assert_close(to_f64(y[:, :b]), p.y + delta, what=f"{a} -> {b}")
        assert bool((y[:, b:] == -7.0).all())
