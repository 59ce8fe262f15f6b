"""The compiled marshalling on a GPU: what a caller passes is what is used, and errors keep their types."""
import threading
import time

import pytest
import torch

import paper_2603_15965_b200 as M

pytestmark = pytest.mark.gpu


def test_out_of_memory_is_torchs_own_error():
    ids, breaks = torch.zeros(50_000_000, dtype=torch.int32, device="cuda"), torch.tensor([0, 5], dtype=torch.int32, device="cuda")
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction(1e-4)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            M.molora_route_vocab(ids, breaks)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert not M.molora_route_vocab(ids, breaks).any()


@pytest.mark.parametrize("offset,size", [(1, 20), (1, 255), (1, 256), (0, 255), (256, 0)])
def test_topk_workspace_shorter_than_its_alignment_is_refused(offset, size):
    """(the workspace starts at its first 256-byte boundary, which may lie past its end)"""
    N, C = 40, 4
    x, y = torch.randn(N, 64, device="cuda").bfloat16(), torch.zeros(N, 64, dtype=torch.bfloat16, device="cuda")
    A, B = torch.randn(C, 64, 16, device="cuda").bfloat16(), torch.randn(C, 16, 64, device="cuda").bfloat16()
    idx, w = M.molora_topk_softmax(torch.randn(N, C, device="cuda"), 2)
    buffer = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    with pytest.raises(M.MoloraError, match="workspace"):
        M.molora_apply_topk([M.ProjDesc(x, y, A, B)], idx, w, C, ws=buffer[offset:offset + size])
    assert not y.any() and not buffer.any()


def test_other_threads_run_while_a_call_waits_for_the_launch_queue():
    ids, breaks = torch.zeros(64, dtype=torch.int32, device="cuda"), torch.tensor([0, 5], dtype=torch.int32, device="cuda")
    r = M.molora_route_vocab(ids, breaks)
    torch.cuda.synchronize()

    def launches():
        for _ in range(4000):                        # more than the queue holds: some call blocks until the kernel ahead ends
            M.molora_route_vocab(ids, breaks, r_out=r)

    torch.cuda._sleep(1_500_000_000)                 # ~0.8 s
    worker = threading.Thread(target=launches)
    start = last = time.perf_counter()
    longest = 0.0
    worker.start()
    while worker.is_alive():
        time.sleep(0.001)
        now = time.perf_counter()
        longest, last = max(longest, now - last), now
    worker.join()
    torch.cuda.synchronize()
    assert last - start > 0.3, "the queue never filled"
    assert longest < 0.15


@pytest.mark.parametrize("raw", [False, True])
def test_what_a_call_allocates_belongs_to_its_stream(raw):
    """Memory freed on the current stream is still read there when a call on another stream asks for an output of that size."""
    N = 1 << 20
    ids, breaks = torch.zeros(N, dtype=torch.int32, device="cuda"), torch.tensor([0, 5], dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    freed = torch.full((N,), 7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)
    copy = freed.clone()
    del freed
    r = M.molora_route_vocab(ids, breaks, stream=side.cuda_stream if raw else side)
    side.synchronize()
    assert not r.any()
    assert (copy == 7).all()


def test_callers_outputs_stream_and_workspace_are_used():
    N, C = 300, 5
    r = torch.randint(0, C, (N,), dtype=torch.int32, device="cuda")
    x, y = torch.randn(N, 512, device="cuda").bfloat16(), torch.randn(N, 256, device="cuda").bfloat16()
    A, B = torch.randn(C, 512, 64, device="cuda").bfloat16() * 0.05, torch.randn(C, 64, 256, device="cuda").bfloat16() * 0.1
    want = y.clone()
    M.molora_group_apply_batched(r, [M.ProjDesc(x, want, A, B)])
    counts, offsets, perm = (torch.full((n,), -9, dtype=torch.int32, device="cuda") for n in (C, C + 1, N))
    need = M.molora_apply_workspace_bytes(N, C, 512, 256, 64)
    assert need > 0
    ws = torch.full((need,), 255, dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    assert bool((counts == -9).all())                              # (its kernels are loaded before the time counts)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)
    got = M.molora_group_apply_batched(r, [M.ProjDesc(x, y, A, B)], counts=counts, offsets=offsets, perm=perm, ws=ws, stream=side)
    assert got[0] is counts and got[1] is offsets and got[2] is perm
    assert not side.query() and bool((counts == -9).all())         # it waits for what is ahead of it on that stream
    side.synchronize()
    assert torch.equal(y, want) and torch.equal(counts, torch.bincount(r, minlength=C).int()) and not bool((ws == 255).all())
    with pytest.raises(M.MoloraError, match="workspace"):
        M.molora_group_apply_batched(r, [M.ProjDesc(x, y, A, B)], ws=ws[:need - 16])
    ids, breaks = torch.arange(N, dtype=torch.int32, device="cuda"), torch.tensor([0, 100, 300], dtype=torch.int32, device="cuda")
    out = torch.full((N,), -9, dtype=torch.int32, device="cuda")
    assert M.molora_route_vocab(ids, breaks, r_out=out) is out and int(out.sum()) == 200
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    M.molora_route_vocab(ids + 1, breaks, r_out=out, dev_status=status)
    assert int(status) == 1 and int(out[-1]) == -1
