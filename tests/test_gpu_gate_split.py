"""The gate of small calls (16 tokens per cluster, the k chunks spread over its warps) against the CPU oracle: token counts around
the 16-token groups, widths below, at and between the numbers of chunks the clusters take, every adapter padding."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import workloads as W

from _harness import dev_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 15, 16, 17, 93, 1023])
@pytest.mark.parametrize("d,C", [(8, 5), (136, 8), (1024, 6), (1032, 9), (2048, 16), (8264, 11), (520, 17), (4104, 32)])
def test_small_call_gate_matches_oracle(N, d, C):
    rng = np.random.default_rng(N * 7 + d + C)
    x = W.round_to_bf16(rng.standard_normal((N, d), dtype=np.float32))
    G = (rng.standard_normal((d, C)) * d ** -0.5).astype(np.float32)
    bias = (rng.standard_normal(C) * 0.1).astype(np.float32)
    xd, Gd, bd = dev_tensor(x, "bf16"), dev_tensor(G, "f32"), dev_tensor(bias, "f32")
    z = torch.empty(N, C, dtype=torch.float32, device="cuda")
    r = M.molora_route_gate(xd, Gd, bd, logits_out=z)
    z64 = x.astype(np.float64) @ G.astype(np.float64) + bias
    # three bf16 terms carry 24 bits of G; fp32 sums of d terms of magnitude d^-1/2
    np.testing.assert_allclose(z.cpu().numpy(), z64, rtol=0, atol=4e-6 * max(1.0, np.abs(z64).max()))
    order = np.sort(z64, axis=1)
    keep = order[:, -1] - order[:, -2] >= 1e-4
    assert np.array_equal(r.cpu().numpy()[keep], z64.argmax(axis=1)[keep])
    r_ref, _, margin = oracle.route_gate(x, G)
    r0 = M.molora_route_gate(xd, Gd)
    assert np.array_equal(r0.cpu().numpy()[margin >= 1e-3], r_ref[margin >= 1e-3])
    # equal logits go to the lowest adapter
    flat = M.molora_route_gate(xd, torch.ones(d, C, device="cuda"))
    assert not flat.any()


@pytest.mark.parametrize("N,d,C", [(1024, 2048, 8), (3173, 2048, 8), (3174, 2048, 8), (2441, 2048, 16), (2442, 2048, 16), (1500, 64, 17),
                                   # one wave of clusters of 1, 2 and 4 CTAs, the second wave of up to 8 adapters, and what lies past either
                                   (4736, 64, 8), (4737, 64, 8), (4736, 64, 16), (4737, 192, 16), (2368, 2048, 8), (2369, 2048, 8), (1184, 4096, 16),
                                   (1185, 4096, 16), (1185, 4096, 8), (8000, 512, 8), (8001, 512, 8), (16000, 64, 5)])
def test_both_sides_of_the_small_call_rule(N, d, C):
    rng = np.random.default_rng(N + C)
    x = W.round_to_bf16(rng.standard_normal((N, d), dtype=np.float32))
    G = (rng.standard_normal((d, C)) * d ** -0.5).astype(np.float32)
    z = torch.empty(N, C, dtype=torch.float32, device="cuda")
    r = M.molora_route_gate(dev_tensor(x, "bf16"), dev_tensor(G, "f32"), logits_out=z)
    r_ref, z_ref, margin = oracle.route_gate(x, G)
    np.testing.assert_allclose(z.cpu().numpy(), z_ref, rtol=0, atol=4e-6 * max(1.0, np.abs(z_ref).max()))
    assert np.array_equal(r.cpu().numpy()[margin >= 1e-3], r_ref[margin >= 1e-3])


@pytest.mark.parametrize("N", [40, 1500])
@pytest.mark.parametrize("C", [7, 16, 31])
def test_nan_and_infinite_logits_decide_as_a_scan_does(N, C):
    """Logits of NaN (an adapter whose gate column or bias is damaged) and of -inf (one that is masked): the winner is that of a scan
    from adapter 0 that replaces the best by what is greater."""
    rng = np.random.default_rng(C)
    d = 2048
    x = W.round_to_bf16(rng.standard_normal((N, d), dtype=np.float32))
    G = (rng.standard_normal((d, C)) * d ** -0.5).astype(np.float32)
    z64 = x.astype(np.float64) @ G.astype(np.float64)
    for bad in ([1], [2, 5], [0], [0, 3], list(range(C)), list(range(1, C))):
        for value in (np.nan, -np.inf, np.inf):
            bias = np.zeros(C, np.float32)
            bias[bad] = value
            r = M.molora_route_gate(dev_tensor(x, "bf16"), dev_tensor(G, "f32"), dev_tensor(bias, "f32")).cpu().numpy()
            z = z64 + bias
            want = np.zeros(N, np.int64)
            best = z[:, 0].copy()
            for c in range(1, C):
                more = z[:, c] > best
                want[more], best[more] = c, z[more, c]
            order = np.sort(np.where(np.isfinite(z), z, -1e30), axis=1)
            clear = order[:, -1] - order[:, -2] >= 1e-3
            assert np.array_equal(r[clear], want[clear]), (bad, value)


@pytest.mark.parametrize("N", [1, 63, 127, 128, 1000, 1792, 1793])
@pytest.mark.parametrize("d,H", [(64, 64), (2048, 64), (4096, 128)])
def test_mlp_router_of_small_calls(N, d, H):
    C = 5
    rng = np.random.default_rng(N + d)
    x = W.round_to_bf16(rng.standard_normal((N, d), dtype=np.float32))
    W1 = (rng.standard_normal((d, H)) * d ** -0.5).astype(np.float32)
    W2 = (rng.standard_normal((H, C)) * H ** -0.5).astype(np.float32)
    b1, b2 = (rng.standard_normal(H) * 0.1).astype(np.float32), (rng.standard_normal(C) * 0.1).astype(np.float32)
    xd, W1d, b1d, W2d, b2d = (dev_tensor(v, "bf16" if v is x else "f32") for v in (x, W1, b1, W2, b2))
    z = torch.empty(N, C, dtype=torch.float32, device="cuda")
    r = M.molora_route_mlp(xd, W1d, b1d, W2d, b2d, logits_out=z)
    r_ref, z_ref, margin = oracle.route_mlp(x, W1, b1, W2, b2)
    np.testing.assert_allclose(z.cpu().numpy(), z_ref, rtol=0, atol=1e-5 * max(1.0, np.abs(z_ref).max()))
    assert np.array_equal(r.cpu().numpy()[margin >= 1e-3], r_ref[margin >= 1e-3])


@pytest.mark.parametrize("N,d,H,launches", [(1, 64, 16, 1), (127, 64, 16, 1), (128, 64, 16, 2), (127, 64, 17, 2), (127, 128, 16, 2), (127, 128, 8, 2), (127, 64, 8, 1)])
def test_mlp_router_on_both_sides_of_the_tiny_rule(N, d, H, launches):
    C = 4
    rng = np.random.default_rng(N + H)
    x = W.round_to_bf16(rng.standard_normal((N, d), dtype=np.float32))
    W1 = (rng.standard_normal((d, H)) * d ** -0.5).astype(np.float32)
    W2 = (rng.standard_normal((H, C)) * H ** -0.5).astype(np.float32)
    xd, W1d, W2d = dev_tensor(x, "bf16"), dev_tensor(W1, "f32"), dev_tensor(W2, "f32")
    z = torch.empty(N, C, dtype=torch.float32, device="cuda")
    before = M.molora_launch_count()
    r = M.molora_route_mlp(xd, W1d, None, W2d, None, logits_out=z)
    assert M.molora_launch_count() - before == launches
    r_ref, z_ref, margin = oracle.route_mlp(x, W1, None, W2, None)
    np.testing.assert_allclose(z.cpu().numpy(), z_ref, rtol=0, atol=1e-5 * max(1.0, np.abs(z_ref).max()))
    assert np.array_equal(r.cpu().numpy()[margin >= 1e-3], r_ref[margin >= 1e-3])
    prepared, zp = M.molora_route_mlp_prepare(xd.dtype, W1d, C), torch.empty_like(z)
    assert torch.equal(M.molora_route_mlp(xd, W1d, None, W2d, None, logits_out=zp, prepared=prepared), r) and torch.equal(zp, z)
