"""Kernels launched under their predecessor: steps in a row whose inputs (activations, base projections, adapters, routing sources) are
rewritten in place between them, by copies and by other kernels, give bit for bit what plain stream order gives -- on one stream, on two at
once, from a graph, and from a graph whose step follows work of another stream."""
import pytest
import torch

import paper_2603_15965_b200 as M

pytestmark = pytest.mark.gpu

STEPS = 12


@pytest.fixture(autouse=True)
def _default_kernels_afterwards():
    yield
    for k in M.TUNING_NAMES:
        M.molora_debug_set(k, 0)


class Step:
    """One kind of step on buffers of its own; run(i) rewrites them with the i-th inputs and appends the results."""

    def __init__(self, kind, N, rank, dtype, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.kind, self.N, self.C, d = kind, N, 6, 512
        rand = lambda *shape, scale=1.0: (torch.randn(*shape, generator=g, device="cuda") * scale).to(dtype)
        self.x0, self.y0 = [rand(N, d) for _ in range(3)], [rand(N, 576) for _ in range(3)]
        self.A0, self.B0 = [rand(self.C, d, rank, scale=d ** -0.5) for _ in range(3)], [rand(self.C, rank, 576, scale=0.1) for _ in range(3)]
        self.ids0 = [torch.randint(0, 600, (N,), generator=g, device="cuda", dtype=torch.int32) for _ in range(3)]
        self.x, self.y, self.A, self.B, self.ids = (v[0].clone() for v in (self.x0, self.y0, self.A0, self.B0, self.ids0))
        self.breaks = torch.arange(0, 601, 100, device="cuda", dtype=torch.int32)
        self.W1, self.b1 = torch.randn(d, 64, generator=g, device="cuda") * d ** -0.5, torch.randn(64, generator=g, device="cuda")
        self.W2, self.b2 = torch.randn(64, self.C, generator=g, device="cuda") * 0.1, torch.randn(self.C, generator=g, device="cuda")
        self.G = torch.randn(d, self.C, generator=g, device="cuda") * d ** -0.5
        self.image = M.molora_route_mlp_prepare(dtype, self.W1, self.C) if kind == "mlp" else None
        self.logits = torch.empty(N, self.C, device="cuda")
        self.ws = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")
        self.out = []

    def step(self):
        proj = [M.ProjDesc(self.x, self.y, self.A, self.B)]
        if self.kind == "topk":
            M.molora_route_gate(self.x, self.G, logits_out=self.logits)
            idx, w = M.molora_topk_softmax(self.logits, 2)
            M.molora_apply_topk(proj, idx, w, self.C)
            return
        r = M.molora_route_mlp(self.x, self.W1, self.b1, self.W2, self.b2, prepared=self.image) if self.kind == "mlp" else \
            M.molora_route_vocab(self.ids, self.breaks)
        if self.kind == "grouped":
            _, offsets, perm = M.molora_group(r, self.C)
            M.molora_apply_batched(proj, offsets, perm, ws=self.ws)
            M.molora_apply_batched(proj, offsets, perm, ws=self.ws)
        else:
            M.molora_group_apply_batched(r, proj, ws=self.ws)

    def run(self, i):
        j = i % 3
        self.A.copy_(self.A0[j]), self.B.copy_(self.B0[j]), self.ids.copy_(self.ids0[j])
        self.y.copy_(self.y0[(i + 1) % 3]).mul_(0.5)
        torch.add(self.x0[j], 0.0, out=self.x)
        self.step()
        self.out.append(self.y.clone())


KINDS = [("vocab", 300, 16, torch.bfloat16), ("vocab", 5000, 64, torch.bfloat16), ("grouped", 700, 32, torch.bfloat16),
         ("grouped", 400, 8, torch.float32), ("vocab", 300, 8, torch.float32), ("mlp", 1300, 64, torch.bfloat16),
         ("topk", 900, 16, torch.bfloat16), ("topk", 5000, 32, torch.bfloat16), ("vocab", 90, 64, torch.bfloat16)]


def both(build):
    results = []
    for off in (1, 0):
        M.molora_debug_set("chained_launch_off", off)
        results.append(build())
        torch.cuda.synchronize()
    assert len(results[0]) == len(results[1]) and all(torch.equal(a, b) for a, b in zip(*results))


@pytest.mark.parametrize("kind,N,rank,dtype", KINDS)
def test_steps_in_a_row(kind, N, rank, dtype):
    def build():
        s = Step(kind, N, rank, dtype, 1)
        for i in range(STEPS):
            s.run(i)
        return s.out
    both(build)


def test_two_streams_at_once():
    def build():
        steps = [Step(*KINDS[k], seed=k) for k in (0, 1, 5, 6)]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(2)]
        for i in range(STEPS):
            for k, s in enumerate(steps):
                with torch.cuda.stream(streams[k % 2]):
                    s.run(i)
        torch.cuda.synchronize()
        return [y for s in steps for y in s.out]
    both(build)


@pytest.mark.parametrize("kind,N,rank,dtype", KINDS)
def test_graph_of_steps_that_follow_another_stream(kind, N, rank, dtype):
    def build():
        s, side = Step(kind, N, rank, dtype, 2), torch.cuda.Stream()
        s.step()                                                # first use of every kernel before the capture
        x1, x2 = s.x.clone(), s.x0[1]
        torch.cuda.synchronize()
        graph, capture = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=capture):
            s.y.copy_(s.y0[1])
            side.wait_stream(capture)
            with torch.cuda.stream(side):
                torch.add(x2, x1, out=s.x)                      # the step depends on a kernel of the other stream ...
                s.A.copy_(s.A0[2])                              # ... and on a copy
            s.B.copy_(s.B0[1])
            capture.wait_stream(side)
            s.step()
            s.step()
            out = s.y.clone()
        results = []
        for _ in range(3):
            graph.replay()
            results.append(out.clone())
        torch.cuda.synchronize()
        return results
    both(build)
