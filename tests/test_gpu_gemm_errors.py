"""A stand-alone product that is refused fails alone: its error and the one-call test hook end with it."""
import ctypes as C
import os
import subprocess
import sys
import threading
import time

import pytest
import torch

from synth_inputs import rng

pytestmark = pytest.mark.gpu


def _operands(T, N, K):
    x = rng.normal(31, 1, (T, K), 1.0, dtype=torch.float32).cuda()
    w = rng.normal_bf16(31, 2, (N, K), 0.02).cuda()
    return x, w, x.double() @ w.double().T


def _refused_call():
    """More row chunks than a grid has rows (65535 of 128 rows): the launch is refused on the host."""
    from paper_2507_22424_b200 import binding as B
    w = torch.zeros(4, 8, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.SpecVLAError) as e:
        B.gemm(torch.zeros(65536 * 128 + 1, 8, device="cuda"), w)
    assert e.value.code == -5                                           # SPECVLA_ERR_CUDA


@pytest.mark.parametrize("packed", [False, True])
def test_refused_launch_does_not_fail_later_calls(packed):
    from paper_2507_22424_b200 import binding as B
    T, N, K = 19, 512, 264
    x, w, ref = _operands(T, N, K)
    p = B.pack_weights(w)
    _refused_call()
    for _ in range(3):
        y = B.gemm_prepacked(x, p, N) if packed else B.gemm(x, w)
        assert (y.double() - ref).abs().max() < 1e-4 * 0.02 * (K ** 0.5) + 1e-6


def test_refused_call_takes_the_test_hook_with_it():
    """The hook holds for the next call, whether that call is launched or refused."""
    from paper_2507_22424_b200 import binding as B
    x, w, ref = _operands(16, 256, 512)
    _refused_call()
    assert B.lib.specvla_gemm_fault_test(2_000_000, 1) == 0
    _refused_call()
    y = B.gemm(x, w)                                                    # an ordinary call: no wait runs out
    assert (y.double() - ref).abs().max() < 1e-4 * 0.02 * (512 ** 0.5) + 1e-6


@pytest.mark.parametrize("T,N,K", [(1, 256, 8192), (512, 1024, 4096), (40000, 256, 512)])
def test_a_wait_limit_covers_the_product_alone(T, N, K):
    """A limit of 0.2 ms, far above any wait of the product itself, never runs out, however much the
    operand split in front of it has to do; the status word says so."""
    from paper_2507_22424_b200 import binding as B
    x, w, ref = _operands(T, N, K)
    for _ in range(5):
        assert B.lib.specvla_gemm_fault_test(200_000, -1) == 0          # no K block is withheld
        y = B.gemm(x, w)                                                # (raises on a timeout)
    assert (y.double() - ref).abs().max() < 1e-4 * 0.02 * (K ** 0.5) + 1e-6


def test_products_from_several_threads():
    """Products from several threads on streams of their own: each succeeds with its own result."""
    from paper_2507_22424_b200.binding import gemm_prepacked, pack_weights
    g = torch.Generator().manual_seed(3)
    w = torch.randn(256, 264, generator=g).to(torch.bfloat16).cuda()
    packed = pack_weights(w)
    xs = [torch.randn(n, 264, generator=g).cuda() for n in (1, 9, 33)]
    want = [gemm_prepacked(x, packed, 256) for x in xs]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(50):
                if not torch.equal(gemm_prepacked(xs[i], packed, 256), want[i]):
                    bad.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(xs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


def test_a_thread_may_end_inside_another_threads_capture():
    """The end of a thread that has read a status makes no call that a capture forbids."""
    from paper_2507_22424_b200 import binding as B
    x, w, ref = _operands(9, 256, 264)
    asked, end = threading.Event(), threading.Event()

    def work():
        B.gemm(x, w)
        asked.set()
        end.wait()

    thread = threading.Thread(target=work)
    thread.start()
    asked.wait()
    torch.cuda.synchronize()
    y = torch.ones(8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        y.mul_(2)
        end.set()
        thread.join()
        time.sleep(0.3)                                                 # (its thread-local objects go after the join)
        y.add_(1)
    graph.replay()
    assert y.tolist() == [3.0] * 8


# Contexts that come and go under one thread: each reads its own status, before and after the others.
CONTEXTS = """
import ctypes as C
import torch
from paper_2507_22424_b200 import binding as B

cu = C.CDLL("libcuda.so.1")


def ok(rc):
    assert rc == 0, rc


x = torch.ones(9, 264, device="cuda")
w = torch.ones(256, 264, device="cuda", dtype=torch.bfloat16)
primary = C.c_void_p()
for _ in range(20):                                         # more than have words of their own
    assert bool((B.gemm(x, w) == 264).all())
    ok(cu.cuCtxGetCurrent(C.byref(primary)))
    ctx, scratch = C.c_void_p(), C.c_uint64()
    ok(cu.cuCtxCreate_v2(C.byref(ctx), 0, 0))
    ok(cu.cuMemAlloc_v2(C.byref(scratch), C.c_size_t(4096)))
    for word, status in ((0, 0), (3, -6), (0, 0)):
        ok(cu.cuMemsetD32_v2(scratch, word, C.c_size_t(1024)))
        assert B.lib.specvla_gemm_status(C.c_void_p(scratch.value), None) == status
    ok(cu.cuMemsetD32_v2(scratch, 3, C.c_size_t(1024)))
    ok(cu.cuCtxSynchronize())
    ok(cu.cuCtxSetCurrent(primary))                         # memory of a context that is not the current one
    assert B.lib.specvla_gemm_status(C.c_void_p(scratch.value), None) == -6
    ok(cu.cuCtxSetCurrent(ctx))
    ok(cu.cuMemFree_v2(scratch))
    ok(cu.cuCtxDestroy_v2(ctx))
    ok(cu.cuCtxSetCurrent(primary))
assert bool((B.gemm(x, w) == 264).all())
"""


def test_status_in_contexts_that_come_and_go():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    done = subprocess.run([sys.executable, "-c", CONTEXTS], cwd=root, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]


@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_status_of_a_word_at_any_address(offset):
    """A word off a four-byte boundary is read as well."""
    from paper_2507_22424_b200 import binding as B
    buf = torch.zeros(64, dtype=torch.uint8, device="cuda")
    for value, status in ((0, 0), (1, -6), (0, 0)):
        buf[offset] = value
        assert B.lib.specvla_gemm_status(C.c_void_p(buf.data_ptr() + offset), B._stream()) == status


def test_status_belongs_to_the_asking_thread():
    """One product that timed out and one that did not, asked about at the same time by two threads."""
    from paper_2507_22424_b200 import binding as B
    T, N, K = 16, 256, 512
    x, w, ref = _operands(T, N, K)
    nb = B.lib.specvla_gemm_scratch_bytes(T, N, K)
    streams = [torch.cuda.Stream() for _ in range(2)]
    scratch = [torch.empty(nb + 1024, dtype=torch.uint8, device="cuda") for _ in range(2)]
    y = [torch.empty(T, N, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    at = [C.c_void_p((s.data_ptr() + 1023) // 1024 * 1024) for s in scratch]
    on = [C.c_void_p(s.cuda_stream) for s in streams]
    assert B.lib.specvla_gemm_fault_test(2_000_000, 1) == 0             # the first of the two products
    for i in range(2):
        assert B.lib.specvla_gemm(C.c_void_p(x.data_ptr()), C.c_void_p(w.data_ptr()), C.c_void_p(y[i].data_ptr()),
                                  T, N, K, at[i], nb, on[i]) == 0
    together, seen = threading.Barrier(2), [set(), set()]

    def ask(i):
        together.wait()
        for _ in range(500):
            seen[i].add(B.lib.specvla_gemm_status(at[i], on[i]))

    threads = [threading.Thread(target=ask, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert seen == [{-6}, {0}], seen
    assert (y[1].double() - ref).abs().max() < 1e-4 * 0.02 * (K ** 0.5) + 1e-6


def test_more_calls_at_a_time_than_words():
    """Seventy calls wait behind one kernel, each for its own word; twice, since the words come back."""
    from paper_2507_22424_b200 import binding as B
    n = 70
    words = torch.zeros(n, 64, dtype=torch.int32, device="cuda")
    words[::3] = 1
    streams = [torch.cuda.Stream() for _ in range(n)]
    torch.cuda.synchronize()
    for _ in range(2):
        got = [None] * n
        gate = torch.cuda.Event()
        torch.cuda._sleep(200_000_000)                                  # about 0.1 s
        gate.record()
        for s in streams:
            s.wait_event(gate)

        def ask(i):
            got[i] = B.lib.specvla_gemm_status(C.c_void_p(words[i].data_ptr()), C.c_void_p(streams[i].cuda_stream))

        threads = [threading.Thread(target=ask, args=(i,)) for i in range(n)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert got == [-6 if i % 3 == 0 else 0 for i in range(n)], got


def test_status_of_managed_memory():
    """Memory that is not the device's own alone is copied."""
    from paper_2507_22424_b200 import binding as B
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    scratch = C.c_uint64()
    assert cu.cuMemAllocManaged(C.byref(scratch), C.c_size_t(4096), 1) == 0
    try:
        for value, status in ((0, 0), (1, -6), (0, 0)):
            C.c_int.from_address(scratch.value).value = value
            assert B.lib.specvla_gemm_status(C.c_void_p(scratch.value), B._stream()) == status
            torch.cuda.synchronize()
    finally:
        assert cu.cuMemFree_v2(scratch) == 0
