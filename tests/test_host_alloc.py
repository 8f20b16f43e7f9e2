"""The allocating extension of the wrappers (no GPU needed)."""
import threading
import time

import pytest
import torch

from paper_2608_15522_b200 import binding as av


@pytest.fixture
def slow_allocations():
    """Uninitialised memory is filled, which makes an allocation as slow as its size says."""
    threads = torch.get_num_threads()
    torch.set_num_threads(1)
    torch.use_deterministic_algorithms(True)
    yield
    torch.use_deterministic_algorithms(False)
    torch.set_num_threads(threads)


@pytest.mark.parametrize("call", ["empty", "empty_as"])
def test_other_threads_run_during_an_allocation(slow_allocations, call):
    """A caching-allocator miss may wait for the GPU: the interpreter lock must be free meanwhile.  Another thread counts
    milliseconds; with the lock held it can do so once before and once behind the call."""
    like = torch.empty((1, 1, 1 << 13, 1 << 13), dtype=torch.bfloat16)
    counts, stop = [0], threading.Event()

    def count():
        while not stop.is_set():
            counts[0] += 1
            time.sleep(1e-3)

    counter = threading.Thread(target=count)
    counter.start()
    seen = []
    try:
        for _ in range(5):
            before = counts[0]
            x = av._empty(like, 0, 1, 1 << 13, 1 << 13) if call == "empty" else av._empty_as(like)
            seen.append(counts[0] - before)
            assert x.numel() == like.numel()
            del x      # (a tensor is freed without the lock: not beside the next call)
    finally:
        stop.set()
        counter.join()
    assert sorted(seen)[2] > 5, seen      # (50 to 100 ms each)


@pytest.mark.parametrize("call", [lambda: av._empty(torch.empty(1), 0, -1), lambda: av._empty(torch.empty(1), 0, 1 << 60)])
def test_a_failed_allocation_raises(call):
    with pytest.raises(RuntimeError):
        call()
