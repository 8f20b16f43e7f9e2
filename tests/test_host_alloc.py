"""The allocating extension of the wrappers (its allocations need no GPU, whole calls are made with tensors on one)."""
import ctypes
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


@pytest.fixture
def sleepy_calls():
    """The library's entry points replaced: the workspace queries sleep as many microseconds as there are batch items (and give back 0),
    without touching the interpreter lock; the calls are noted with what they were handed."""
    i, f, p, sz, T = ctypes.c_int, ctypes.c_float, ctypes.c_void_p, ctypes.c_size_t, av._Bf16Tensor4
    signatures = {"cross": [i] * 5 + [T] * 3 + [p] * 3 + [f] * 3 + [p, sz, p], "mask": [i] * 5 + [T] * 2 + [p, i, i, ctypes.c_uint, f] + [p] * 6 + [sz, p],
                  "sparse": [i] * 5 + [T] * 3 + [p] * 4 + [f, p, sz, p], "protected": [i] * 5 + [T] * 3 + [p, i, p, p, f, p, sz, p]}
    calls, keep = [], []

    def recorder(types):
        def entry(*args):
            calls.append([(a.ptr, a.stride_b, a.stride_h, a.stride_n) if isinstance(a, T) else a for a in args])
            return 0
        keep.append(ctypes.CFUNCTYPE(i, *types)(entry))
        return ctypes.cast(keep[-1], p).value

    sleep = ctypes.cast(ctypes.CDLL(None).usleep, p).value
    av._alloc().bind(*(recorder(s) for s in signatures.values()), *[sleep] * 4, torch._C._cuda_getCurrentRawStream)
    yield calls
    av._alloc_module = None      # bound to the library again
    av._alloc()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["cross", "mask", "sparse", "protected"])
def test_other_threads_run_during_a_whole_call_and_change_nothing_of_it(sleepy_calls, name):
    """From the first allocation to the launches a whole call holds no interpreter lock.  A thread that gives its tensors other data
    meanwhile does not reach it: sizes, strides and pointers are those of the beginning."""
    B, H, N, d = 200000, 1, 2, 64
    new = lambda: torch.empty((B, N, H, d), dtype=torch.bfloat16, device="cuda").transpose(1, 2)
    q, k, v, o, u8 = new(), new(), new(), new(), torch.empty((B, N), dtype=torch.uint8, device="cuda")
    i32 = torch.empty((B, 4), dtype=torch.int32, device="cuda")
    s = torch.empty((B, N), device="cuda")
    call, given = {"cross": (lambda: av.avsa_cross_attn_scores(q, k, v, scores=s), [q, k, v]), "mask": (lambda: av.avsa_build_block_mask(q, k, s, 1, 1, 64), [q, k]),
                   "sparse": (lambda: av.avsa_sparse_self_attn(q, k, v, i32, i32, 64), [q, k, v]),
                   "protected": (lambda: av.avsa_protected_rows_attn(q, k, v, u8, 1, 64, o), [q, k, v])}[name]
    others = [s] if name in ("cross", "mask") else [i32] if name == "sparse" else [u8, o]
    want = [(t.data_ptr(), *t.stride()[:3]) for t in given], [t.data_ptr() for t in others]
    small = {t.dtype: torch.empty((1, 1, 1, 64), dtype=t.dtype, device="cuda") for t in given + others}
    held = [t.data for t in given + others]      # the memory stays
    steps, stop = [], threading.Event()

    def change():
        for t in given + others:
            time.sleep(5e-3)
            t.data = small[t.dtype]
            steps.append(t)
        while not stop.is_set():
            time.sleep(1e-3)
            steps.append(None)
    changer = threading.Thread(target=change)
    changer.start()
    try:
        call()
        during = len(steps)
    finally:
        stop.set()
        changer.join()
    assert during > len(given + others) + 5      # 200 ms
    args, sizes = sleepy_calls.pop(), [B, H, N, N, d] if name == "cross" else [B, H, N, d]
    assert args[:len(sizes)] == sizes
    assert [x for x in args if isinstance(x, tuple)] == want[0]
    assert all(x in args for x in want[1])
    del held
