"""Calls on both sides of the rules that choose kernel, tile and cluster from the sizes, against the CPU oracle: the library's own
choice throughout, several projections in one call, tokens spread evenly over the adapters."""
import numpy as np
import oracle
import pytest

import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import dev_tensor, run_and_check, to_f64

pytestmark = pytest.mark.gpu


def check(N, C, shapes, rank, rows=150):
    rng = np.random.default_rng(N + C + rank)
    r = rng.permutation(N).astype(np.int32) % C
    parts = [W.random_problem(N + C + i, N, C, a, b, rank, "bf16", r=r) for i, (a, b) in enumerate(shapes)]
    w = parts[0]
    for i, p in enumerate(parts):
        p.projections[0].x_key, p.projections[0].name = f"x{i}", f"proj{i}"
    w = W.Workload(name=f"choice-{N}-{C}-{rank}", N=N, C=C, dtype="bf16", router="given", inputs={f"x{i}": p.inputs["x"] for i, p in enumerate(parts)},
                   projections=[p.projections[0] for p in parts], r=r)
    run_and_check(w, rows=None if N <= rows else rng.choice(N, rows, replace=False), batched=True)


@pytest.mark.parametrize("N,C,shapes,rank", [
    # streaming kernel: output slices of one projection and of several, 16- and 32-row tiles, chunks that are partly empty
    (1, 1, [(1536, 1536), (1536, 4608)], 32), (1, 16, [(512, 512)], 16), (32, 4, [(512, 512), (512, 128)], 16),
    (200, 4, [(512, 512), (512, 128), (512, 512)], 16), (2500, 8, [(1024, 1024)], 32), (1500, 1, [(1024, 1024), (1024, 3072)], 16),
    (6000, 256, [(512, 512), (512, 256)], 16), (1500, 64, [(1536, 384), (1536, 1536)], 16),
])
def test_tiles_slices_and_clusters(N, C, shapes, rank):
    check(N, C, shapes, rank)


@pytest.mark.parametrize("d_in,d_out", [(1536, 5120), (2080, 4096), (1056, 5152), (2048, 6144)])
def test_linear_and_boxed_weights(d_in, d_out):
    """rank 16, short tiles: seven chunk jobs an item and eight, whole and ragged chunks"""
    check(60, 5, [(d_in, d_out)], 16)


@pytest.mark.parametrize("N,C,shapes,rank", [
    # rank 64, more than 64 adapters, one and two projections: two-launch, streaming and tcgen05 kernel
    (2399, 100, [(512, 320)], 64), (2400, 100, [(512, 320)], 64), (2400, 100, [(512, 320), (512, 96)], 64), (6399, 100, [(512, 320)], 64),
    (6400, 100, [(512, 320)], 64),
])
def test_many_adapters_of_rank_64(N, C, shapes, rank):
    check(N, C, shapes, rank)


@pytest.mark.parametrize("N,C,shapes,rank", [
    # rank 64, three and more projections below 680 tokens: 12 MB with 120 tokens per adapter, 60 MB with 60, and one token less
    (359, 3, [(2048, 2048), (2048, 2048), (2048, 1024)], 64), (360, 3, [(2048, 2048), (2048, 2048), (2048, 1024)], 64), (255, 2, [(4096, 4096)] * 3, 64),
    (256, 2, [(4096, 4096)] * 3, 64), (479, 8, [(4096, 4096)] * 6, 64), (480, 8, [(4096, 4096)] * 6, 64),
])
def test_mid_sized_layers_of_rank_64(N, C, shapes, rank):
    check(N, C, shapes, rank, rows=60)


@pytest.mark.parametrize("N,C,shapes,rank", [
    # rank 32, several projections from 60 MB: 3000 tokens with 300 per adapter, and one less of either
    (2999, 4, [(1024, 1024), (1024, 3072)], 32), (3000, 10, [(1024, 1024), (1024, 3072)], 32), (3000, 11, [(1024, 1024), (1024, 3072)], 32),
    (8000, 8, [(512, 512), (512, 128), (512, 128), (512, 512)], 32),
])
def test_narrow_layers_of_rank_32(N, C, shapes, rank):
    check(N, C, shapes, rank)


@pytest.mark.parametrize("N,C,rank,k,width", [
    # rank 32, top-2: more than 64 sets on both sides of 1024 tokens and of 45 MB, 36 sets on both sides of 100 MB
    (1023, 16, 32, 2, 4096), (1024, 16, 32, 2, 4096), (1831, 16, 32, 2, 4096), (1832, 16, 32, 2, 4096), (4096, 8, 32, 2, 4032), (4096, 8, 32, 2, 4160), (200, 4, 16, 4, 2048),
])
def test_topk_passes_and_kernels(N, C, rank, k, width):
    rng = np.random.default_rng(N + C)
    w = W.random_problem(N + width, N, C, width, width, rank, "bf16")
    p = w.projections[0]
    idx = np.argsort(rng.random((C, N)), axis=0)[:k].astype(np.int32)
    weight = rng.random((k, N)).astype(np.float32)
    weight /= weight.sum(axis=0, keepdims=True)
    y = dev_tensor(p.y, "bf16")
    M.molora_apply_topk([M.ProjDesc(dev_tensor(w.inputs["x"], "bf16"), y, dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16"))],
                        dev_tensor(idx, "i"), dev_tensor(weight, "f32"), C)
    rows = rng.choice(N, min(N, 80), replace=False)
    ref = oracle.apply_topk(w.inputs["x"][rows], p.y[rows], p.A, p.B, np.ascontiguousarray(idx[:, rows]), np.ascontiguousarray(weight[:, rows]))
    # The harness bound, and what y loses where there are several passes: it is rounded to bf16 after each of them, and rounding to
    # the nearest of 8 significant bits is off by at most 2^-8 of the value (half of a unit of 2^-7 in the last place, at a power of two).
    bound = 1e-3 + 2e-2 * np.abs(ref)
    for j in range(1, k):
        bound += 2.0 ** -8 * np.abs(oracle.apply_topk(w.inputs["x"][rows], p.y[rows], p.A, p.B, np.ascontiguousarray(idx[:j, rows]),
                                                      np.ascontiguousarray(weight[:j, rows])))
    assert np.all(np.abs(to_f64(y)[rows] - ref) <= bound)


@pytest.mark.parametrize("N,C,hidden,rank", [
    # a layer whose items pass one wave: widths cut in two and not, one chunk and ragged ones, few tiles and many
    (256, 8, 2048, 16), (257, 7, 2080, 16), (400, 3, 1056, 16), (150, 12, 1024, 16), (600, 2, 2048, 16), (330, 5, 960, 32),
])
def test_layers_of_more_items_than_a_wave(N, C, hidden, rank):
    check(N, C, [(hidden, hidden), (hidden, 512), (hidden, 512), (hidden, hidden), (hidden, 3 * hidden), (hidden, 3 * hidden), (3 * hidden, hidden)],
          rank, rows=60)


@pytest.mark.parametrize("N,C,shapes", [
    # one and two projections of rank 64 on both sides of 512 tokens, of 64 adapters and of 1024 columns
    (1, 1, [(512, 512)]), (90, 16, [(2080, 544)]), (511, 8, [(512, 512)]), (512, 8, [(512, 512)]), (511, 64, [(512, 320), (512, 512)]),
    (511, 65, [(512, 512)]), (511, 8, [(512, 480)]), (300, 3, [(1024, 1024), (1024, 2048)]),
])
def test_small_calls_of_rank_64(N, C, shapes):
    check(N, C, shapes, 64)
    # the scratch that these calls took before stays part of the call
    assert all(M.molora_apply_workspace_bytes(N, C, a, b, 64) > 0 for a, b in shapes)


@pytest.mark.parametrize("rank,kernel", [(16, {}), (64, {"umma_min_tokens": 1}), (32, {"umma_min_tokens": 1000000, "small_path": 1})])
@pytest.mark.parametrize("top", [1, 2])
def test_apply_started_under_the_launch_before_it(rank, kernel, top):
    """More tokens than a CTA groups: the apply starts while the grouping (or the launch that forms the adapter sets) still runs.  Calls in a
    row on the same buffers give what plain stream order gives, bit for bit."""
    N, C, d = 4500, 6, 256
    ws = [W.random_problem(rank + s, N, C, d, 320, rank, "bf16") for s in range(4)]
    xs = [dev_tensor(w.inputs["x"], "bf16") for w in ws]
    As, Bs = [dev_tensor(w.projections[0].A, "bf16") for w in ws], [dev_tensor(w.projections[0].B, "bf16") for w in ws]
    rng = np.random.default_rng(rank)
    idx = [dev_tensor(np.argsort(rng.random((C, N)), axis=0)[:top].astype(np.int32), "i") for _ in ws]
    weight = dev_tensor((rng.random((top, N)) / top).astype(np.float32), "f32")
    results = []
    try:
        for off in (1, 0):
            for k, v in dict(kernel, chained_launch_off=off).items():
                M.molora_debug_set(k, v)
            ys = [dev_tensor(w.projections[0].y, "bf16") for w in ws]
            for _ in range(5):
                for x, y, A, B, i in zip(xs, ys, As, Bs, idx):
                    if top == 1:
                        M.molora_group_apply_batched(i[0], [M.ProjDesc(x, y, A, B)])
                    else:
                        M.molora_apply_topk([M.ProjDesc(x, y, A, B)], i, weight, C)
            results.append([to_f64(y) for y in ys])
    finally:
        for k in M.TUNING_NAMES:
            M.molora_debug_set(k, 0)
    assert all(np.array_equal(a, b) for a, b in zip(*results))


@pytest.mark.parametrize("N,C,shapes", [(1, 1, [(4096, 12288)]), (32, 8, [(12288, 4096)]), (5, 4, [(4096, 4096), (4096, 12288)]), (33, 8, [(4096, 12288)])])
def test_few_items_of_wide_rank_64_projections(N, C, shapes):
    """On the two-launch pair, and one token more on the streaming kernel."""
    check(N, C, shapes, 64)
