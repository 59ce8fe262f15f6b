"""Kernels launched under their predecessor, call forms beyond those of test_gpu_chained.py: several kernels in one call, the two-launch pair
behind a grouping that is itself chained, a prepared gate between layers, hot-set routing, and the streams of a host call.  Steps in a row
whose inputs are rewritten in place between them give bit for bit what plain stream order gives."""
import pytest
import torch

import paper_2603_15965_b200 as M

from test_gpu_chained import STEPS, _default_kernels_afterwards, both  # noqa: F401  (the fixture restores the overrides)

pytestmark = pytest.mark.gpu


class Form:
    """Projections of given (d_out, rank) on buffers of their own; run(i) rewrites them with the i-th inputs and keeps the results."""

    d = 512

    def __init__(self, N, C, projs, router, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        self.N, self.C, self.router = N, C, router
        rand = lambda *shape, scale=1.0: (torch.randn(*shape, generator=g, device="cuda") * scale).to(torch.bfloat16)
        self.x0 = [rand(N, self.d) for _ in range(3)]
        self.y0 = [[rand(N, o) for o, _ in projs] for _ in range(3)]
        self.A0 = [[rand(C, self.d, r, scale=self.d ** -0.5) for _, r in projs] for _ in range(3)]
        self.B0 = [[rand(C, r, o, scale=0.1) for o, r in projs] for _ in range(3)]
        # a few adapters with most of the tokens, many with a handful
        share = torch.tensor([1.0 / (c + 1) for c in range(C)], device="cuda")
        self.r0 = [torch.multinomial(share, N, replacement=True, generator=g).int() for _ in range(3)]
        self.x, self.r = self.x0[0].clone(), self.r0[0].clone()
        self.y, self.A, self.B = ([t.clone() for t in v[0]] for v in (self.y0, self.A0, self.B0))
        self.ids = torch.zeros(N, dtype=torch.int32, device="cuda")
        self.slots = torch.arange(C, dtype=torch.int32, device="cuda")
        self.one_range = torch.tensor([0, 10], dtype=torch.int32, device="cuda")
        self.G = torch.randn(self.d, min(C, 32), generator=g, device="cuda") * self.d ** -0.5
        self.image = M.molora_route_gate_prepare(torch.bfloat16, self.G) if router == "gate" else None
        self.ws = torch.zeros(64 << 20, dtype=torch.uint8, device="cuda")
        self.out = []

    def step(self):
        projs = [M.ProjDesc(self.x, y, A, B) for y, A, B in zip(self.y, self.A, self.B)]
        for layer in range(2):
            if self.router == "gate":
                r = M.molora_route_gate(self.x, self.G, prepared=self.image)
            elif self.router == "hotset":
                r = M.molora_route_hotset(self.ids, self.r, self.one_range, self.slots, self.C)
            else:
                r = self.r
            if layer:
                _, offsets, perm = M.molora_group(r, self.C)
                M.molora_apply_batched(projs, offsets, perm, ws=self.ws)
            else:
                M.molora_group_apply_batched(r, projs, C=self.C, ws=self.ws)
            self.x[:, :64] = self.y[0][:, :64]              # the next layer's input depends on this one's result

    def run(self, i):
        j = i % 3
        for to, of in zip(self.A + self.B, self.A0[j] + self.B0[j]):
            to.copy_(of)
        self.r.copy_(self.r0[j]), self.slots.copy_(torch.roll(torch.arange(self.C, dtype=torch.int32, device="cuda"), i))
        for to, of in zip(self.y, self.y0[(i + 1) % 3]):
            to.copy_(of)
        torch.add(self.x0[j], 0.0, out=self.x)
        self.step()
        self.out += [y.clone() for y in self.y]


@pytest.mark.parametrize("N,C,projs,router,kernels", [
    (1100, 6, [(576, 16), (512, 64), (520, 8), (320, 32)], "given", {}),                              # a launch per rank
    (3000, 100, [(576, 32), (256, 32)], "given", {"umma_min_tokens": 1}),                            # tcgen05 and streaming, by segment
    (3000, 100, [(576, 64), (256, 64)], "given", {"umma_min_tokens": 1, "small_path": 2}),           # tcgen05 and the pair, by segment
    (3000, 100, [(576, 64), (264, 64)], "given", {"umma_min_tokens": 1}),                            # ... and the CUDA-core kernel
    (1500, 7, [(576, 32), (256, 32)], "given", {"small_path": 2, "umma_min_tokens": 1000000}),       # the pair behind a grouping launch
    (700, 7, [(576, 64)], "given", {"small_path": 2, "umma_min_tokens": 1000000}),                   # ... and grouping inside
    (93, 16, [(576, 64), (512, 64), (512, 64)], "gate", {}),
    (2500, 16, [(576, 16), (512, 16)], "gate", {}),
    (5000, 24, [(576, 64), (512, 64)], "gate", {}),
    (400, 40, [(576, 16), (512, 16)], "hotset", {}),
    (5000, 5, [(576, 64)], "hotset", {}),
])
def test_steps_in_a_row(N, C, projs, router, kernels):
    def build():
        for k, v in kernels.items():
            M.molora_debug_set(k, v)
        f = Form(N, C, projs, router, N + C)
        for i in range(STEPS):
            f.run(i)
        return f.out
    both(build)


def test_steps_on_two_streams_at_once():
    def build():
        forms = [Form(1100, 6, [(576, 16), (512, 64), (520, 8)], "given", 1), Form(93, 16, [(576, 64)] * 3, "gate", 2),
                 Form(3000, 100, [(576, 32)], "hotset", 3), Form(300, 4, [(520, 8)], "given", 4)]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(2)]
        for i in range(STEPS):
            for k, f in enumerate(forms):
                with torch.cuda.stream(streams[k % 2]):
                    f.run(i)
        torch.cuda.synchronize()
        return [y for f in forms for y in f.out]
    both(build)


def host_calls(N, C, shapes, calls, seed):
    """(projections, routing source) of calls whose host buffers are their own."""
    g = torch.Generator().manual_seed(seed)
    rand = lambda *s, scale=1.0: (torch.randn(*s, generator=g) * scale).bfloat16()
    A, B = [rand(C, i, r, scale=i ** -0.5).cuda() for i, _, r in shapes], [rand(C, r, o, scale=0.1).cuda() for _, o, r in shapes]
    out = []
    for _ in range(calls):
        x = rand(N, shapes[0][0]).pin_memory()
        out.append(([M.HostProj(x, rand(N, o).pin_memory(), a, b) for (_, o, _), a, b in zip(shapes, A, B)],
                    torch.randint(-1, C, (N,), generator=g, dtype=torch.int32).pin_memory()))
    return out


@pytest.mark.parametrize("N,C,shapes", [
    (2000, 6, [(1024, 1024, 16), (1024, 576, 64), (1024, 520, 8), (1024, 1536, 16)]),
    (1300, 70, [(2048, 1024, 32), (2048, 2048, 64)]),
])
def test_host_calls_in_a_row_between_other_work(N, C, shapes):
    """The streams of a call, whose kernels are chained among themselves, against the caller's stream before and after it."""
    def build():
        calls = host_calls(N, C, shapes, 5, N)
        arena = torch.zeros(M.molora_forward_host_arena_bytes(calls[0][0], M.ROUTE_GIVEN), dtype=torch.uint8, device="cuda")
        device = Form(300, 5, [(576, 16)], "given", 8)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            for i, (projs, r) in enumerate(calls):
                device.run(i)
                M.molora_forward_host(M.ROUTE_GIVEN, projs, arena, route_src=r)
        torch.cuda.synchronize()
        return [p.y.clone() for projs, _ in calls for p in projs] + device.out
    both(build)
