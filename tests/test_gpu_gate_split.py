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
