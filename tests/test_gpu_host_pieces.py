"""molora_forward_host, one projection after the other and the last one in pieces (the last piece ragged, of one row, absent), and in one
piece: with projections that share x, on host buffers that overlap, and under capture -- against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import assert_close, dev_tensor

pytestmark = pytest.mark.gpu


def host(a):
    return torch.from_numpy(W.bf16_bits(a)).view(torch.bfloat16).pin_memory()


def problem(N, C, d, d_outs, rank, seed):
    parts = [W.random_problem(seed + i, N, C, d, o, rank, "bf16", unrouted_frac=0.1) for i, o in enumerate(d_outs)]
    return parts[0].inputs["x"], parts[0].r, [p.projections[0] for p in parts]


def check(x, r, ps, ys, rows):
    for p, y in zip(ps, ys):
        ref = oracle.apply_rows(x, p.y, p.A, p.B, r, rows)
        assert_close(y.float().numpy().astype(np.float64)[rows], ref, what=p.name)


@pytest.mark.parametrize("N,C,d,d_outs,rank", [
    (2048, 8, 2048, [1024, 512, 8192], 16),     # the last projection in four pieces of equal size
    (2049, 8, 2048, [1024, 512, 8192], 32),     # ... and a last one of one row
    (1500, 4, 2048, [2048, 512, 8192], 64),     # other kernels for a piece than for the call
    (4100, 5, 4096, [2048], 16),                # one projection
    (300, 3, 1024, [1024, 1024], 16),           # too few bytes: in one piece
    (6000, 5, 512, [520, 776], 16),             # CUDA-core kernel
])
@pytest.mark.parametrize("router", ["given", "gate"])
def test_pieces_match_the_oracle(N, C, d, d_outs, rank, router):
    x, r, ps = problem(N, C, d, d_outs, rank, N + rank)
    hx, hy = host(x), [host(p.y) for p in ps]
    projs = [M.HostProj(hx, y, dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16")) for p, y in zip(ps, hy)]
    rows = np.random.default_rng(N).choice(N, min(N, 200), replace=False)
    rows[:2] = 0, N - 1
    kw = {"route_src": torch.from_numpy(r).pin_memory()}
    if router == "gate":
        G = dev_tensor((np.random.default_rng(1).standard_normal((d, C)) * d ** -0.5).astype(np.float32), "f32")
        r = M.molora_route_gate(dev_tensor(x, "bf16"), G).cpu().numpy()       # the whole call is routed at once: the same decisions
        kw = {"G": G}
    code = M.ROUTE_GATE if router == "gate" else M.ROUTE_GIVEN
    arena = torch.zeros(M.molora_forward_host_arena_bytes(projs, code), dtype=torch.uint8, device="cuda")
    M.molora_forward_host(code, projs, arena, **kw)
    torch.cuda.synchronize()
    check(x, r, ps, hy, rows)


def test_results_that_replace_another_projections_input():
    """y of the first projection is x of the second: all of x is on its way before any result comes back."""
    N, C, d = 2048, 4, 2048
    x, r, ps = problem(N, C, d, [d, d], 16, 5)
    hx, h0, h1 = host(x), host(ps[0].y), host(ps[1].y)
    A, B = [dev_tensor(p.A, "bf16") for p in ps], [dev_tensor(p.B, "bf16") for p in ps]
    shifted = h0.view(-1)[d:].view(N - 1, d)                                   # overlaps rows 1.. of y at another row number
    projs = [M.HostProj(hx, h0, A[0], B[0]), M.HostProj(h0, h1, A[1], B[1])]
    arena = torch.zeros(M.molora_forward_host_arena_bytes(projs, M.ROUTE_GIVEN), dtype=torch.uint8, device="cuda")
    M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=torch.from_numpy(r).pin_memory())
    torch.cuda.synchronize()
    rows = np.arange(0, N, 37)
    check(x, r, ps[:1], [h0], rows)
    check(ps[0].y, r, ps[1:], [h1], rows)
    # ... and one row further: a piece in flight would read what an earlier piece has written
    h0.copy_(host(ps[0].y)), h1.copy_(host(ps[1].y))
    projs = [M.HostProj(hx[: N - 1], h0[: N - 1], A[0], B[0]), M.HostProj(shifted, h1[: N - 1], A[1], B[1])]
    M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=torch.from_numpy(r[: N - 1].copy()).pin_memory())
    torch.cuda.synchronize()
    check(ps[0].y[1:], r[: N - 1], ps[1:], [h1], rows[rows < N - 1])


def test_calls_in_a_row_on_one_arena_and_under_capture():
    N, C, d = 3000, 6, 1024
    x, r, ps = problem(N, C, d, [d, d], 16, 9)
    hx, hy, src = host(x), [host(p.y) for p in ps], torch.from_numpy(r).pin_memory()
    projs = [M.HostProj(hx, y, dev_tensor(p.A, "bf16"), dev_tensor(p.B, "bf16")) for p, y in zip(ps, hy)]
    arena = torch.zeros(M.molora_forward_host_arena_bytes(projs, M.ROUTE_GIVEN), dtype=torch.uint8, device="cuda")
    rows = np.arange(0, N, 41)
    M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=src)
    torch.cuda.synchronize()
    once = [y.clone() for y in hy]
    for y, p in zip(hy, ps):
        y.copy_(host(p.y))
    other = [M.HostProj(hx, host(p.y), q.A, q.B) for p, q in zip(ps, projs)]
    for _ in range(3):                                   # the next call's copies follow the last one's kernels on the same arena
        M.molora_forward_host(M.ROUTE_GIVEN, other, arena, route_src=src)
    M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=src)
    torch.cuda.synchronize()
    assert all(torch.equal(y, o) for y, o in zip(hy, once))
    for y, p in zip(hy, ps):
        y.copy_(host(p.y))
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=src)
    graph.replay()
    torch.cuda.synchronize()
    check(x, r, ps, hy, rows)
