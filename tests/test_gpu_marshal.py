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
