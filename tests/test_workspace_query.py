"""The scratch that molora_apply_workspace_bytes reports, summed over the projections of a call, is enough for whatever kernels the call
is given to.  Host arithmetic on made-up pointers, so only where there is no GPU that the accepted calls could reach."""
import ctypes

import pytest
import torch

import paper_2603_15965_b200 as M
from paper_2603_15965_b200.binding import _ProjDescC

pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="the accepted calls would be launched")


@pytest.fixture(autouse=True)
def default_kernels_afterwards():
    yield
    for k in M.TUNING_NAMES:
        M.molora_debug_set(k, 0)


@pytest.mark.parametrize("umma_min_tokens", [0, 1, 512, 10 ** 6])
@pytest.mark.parametrize("small_path", [0, 1, 2, 3])
@pytest.mark.parametrize("shapes", [[(4096, 4096, 64)], [(2048, 2048, 64)], [(2080, 2048, 64)], [(2048, 2048, 16)], [(1024, 4096, 32)],
                                    [(4096, 4096, 64), (2048, 2048, 16)]])
def test_a_call_takes_the_scratch_it_asked_for(shapes, small_path, umma_min_tokens):
    M.molora_debug_set("small_path", small_path)
    M.molora_debug_set("umma_min_tokens", umma_min_tokens)
    lib, fake = M.load_library(), ctypes.c_void_p(0x10000)
    for P in (1, 2, 3, 7):
        descs = [_ProjDescC(0x10000, a, 0x20000, b, 0x30000, 0x40000, a, b, r, 1.0, None) for a, b, r in (shapes * P)[:P]]
        arr = (_ProjDescC * P)(*descs)
        for N in (1, 200, 256, 257, 512, 700, 1000, 1024, 1025, 1279, 1280, 3000, 5000):
            for C in (1, 4, 8, 16, 64, 65, 256):
                room = sum(M.molora_apply_workspace_bytes(N, C, d.d_in, d.d_out, d.rank) for d in descs)
                assert lib.molora_apply_batched(arr, P, M.BF16, N, C, fake, fake, fake, room, None, None) != 3, (P, N, C)
                assert lib.molora_group_apply_batched(fake, N, C, fake, fake, fake, arr, P, M.BF16, fake, room, None, None) != 3, (P, N, C)
