"""Which calls run as one grouping launch + apply and which as a single launch, on both sides of the rules that choose between the
tcgen05 and the streaming kernel (host arithmetic: no GPU)."""
import pytest

import paper_2603_15965_b200 as M
from paper_2603_15965_b200.binding import _ProjDescC


@pytest.mark.parametrize("N,C,shapes,expected", [
    # rank 16: the streaming kernel takes layers of any size; one projection of 150 MB with few adapters goes to tcgen05;
    # either is one launch up to 4096 tokens
    (4096, 8, [(2048, 2048, 16)] * 7, 1), (4097, 8, [(2048, 2048, 16)] * 7, 0), (4096, 4, [(8192, 8192, 16)], 1),
    # with more than 64 adapters the tcgen05 kernel does not group; few tokens per adapter go to the streaming kernel, which does
    (3001, 256, [(2048, 2048, 32)] * 4, 1), (3001, 256, [(2048, 2048, 64)] * 4, 1), (4096, 65, [(2048, 2048, 64)] * 4, 1),
    (4096, 64, [(2048, 2048, 64)] * 4, 1),
    # one rank-64 projection with few tokens per adapter: the two-launch kernels behind a grouping launch
    (3001, 256, [(2048, 2048, 64)], 0),
    # ... from 24 tokens per adapter the streaming kernel, up to 64 adapters the tcgen05 kernel as before
    (2399, 100, [(2048, 2048, 64)], 0), (2400, 100, [(2048, 2048, 64)], 1), (4096, 128, [(2048, 2048, 64)] * 2, 1), (4160, 65, [(2048, 2048, 64)], 0),
])
def test_one_launch(N, C, shapes, expected):
    lib = M.load_library()
    arr = (_ProjDescC * len(shapes))(*[_ProjDescC(0x1000, a, 0x2000, b, 0x3000, 0x4000, a, b, r, 1.0, None) for a, b, r in shapes])
    assert int(lib.molora_group_apply_is_one_launch(arr, len(shapes), M.BF16, N, C)) == expected


@pytest.mark.parametrize("N,C", [(1500, 64), (1500, 32), (2048, 4)])
def test_scratch_of_one_rank_64_projection_is_what_it_was(N, C):
    assert M.molora_apply_workspace_bytes(N, C, 2048, 2048, 64) == 0
