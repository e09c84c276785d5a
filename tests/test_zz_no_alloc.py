"""specvla_gemm_static: the GEMM entry point for callers that may not allocate device memory
(stream captures, real-time loops, plug-ins that are handed only their buffers). Its scratch is
a fixed array inside the library, so this checks that it gives what specvla_gemm gives with
caller-allocated scratch, twice in a row on the shared array, and that it refuses shapes the
array cannot hold. Collected last on purpose: a failure here cannot hide another test."""
import os
import subprocess
import sys

import pytest
import torch

from synth_inputs import rng

pytestmark = pytest.mark.gpu


def _case(seed, T, N, K):
    x = rng.normal(seed, 1, (T, K), 1.0, "cuda", dtype=torch.float32)
    w = rng.normal_bf16(seed, 2, (N, K), 0.02, "cuda")
    return x, w


def test_static_scratch_gemm_matches_allocating_gemm_twice():
    from paper_2507_22424_b200 import binding as B
    # the second call is smaller and of another row-tile size, so planes and limbs left behind by
    # the first call would show up in its result if they were not rewritten
    for seed, (T, N, K) in enumerate([(27, 4096, 4096), (9, 1000, 520)]):
        x, w = _case(31 + seed, T, N, K)
        assert B.lib.specvla_gemm_scratch_bytes(T, N, K) <= B.STATIC_SCRATCH_BYTES
        y = torch.full((T, N), float("nan"), dtype=torch.float32, device="cuda")
        got = B.gemm_static(x, w, y).cpu().double()
        want = B.gemm(x, w).cpu().double()
        ref = x.cpu().double() @ w.cpu().double().T
        tol = 1e-4 * 0.02 * (K ** 0.5) + 1e-6          # the tolerance of the GEMM parity tests
        assert torch.isfinite(got).all()
        assert (got - want).abs().max() < tol, float((got - want).abs().max())
        assert (got - ref).abs().max() < tol, float((got - ref).abs().max())


def test_static_scratch_gemm_rejects_oversize():
    from paper_2507_22424_b200 import binding as B
    T, N, K = 1024, 256, 8192          # the two limbs of X alone need 32 MiB
    assert B.lib.specvla_gemm_scratch_bytes(T, N, K) > B.STATIC_SCRATCH_BYTES
    x = torch.zeros(T, K, dtype=torch.float32, device="cuda")
    w = torch.zeros(N, K, dtype=torch.bfloat16, device="cuda")
    y = torch.zeros(T, N, dtype=torch.float32, device="cuda")
    with pytest.raises(B.SpecVLAError) as e:
        B.gemm_static(x, w, y)
    assert e.value.code == -2


def test_static_scratch_gemm_asynchronous_then_status():
    """wait = 0 (the form a stream capture needs): the call returns at once; the status of the
    built-in scratch is asked for afterwards."""
    import ctypes as C
    from paper_2507_22424_b200 import binding as B
    T, N, K = 27, 1024, 1024
    x, w = _case(41, T, N, K)
    y = torch.full((T, N), float("nan"), dtype=torch.float32, device="cuda")
    rc = B.lib.specvla_gemm_static(C.c_void_p(x.data_ptr()), C.c_void_p(w.data_ptr()), C.c_void_p(y.data_ptr()),
                                   T, N, K, 0, B._stream())
    assert rc == 0
    assert B.lib.specvla_gemm_static_status(B._stream()) == 0
    want = B.gemm(x, w).cpu().double()
    assert (y.cpu().double() - want).abs().max() < 1e-4 * 0.02 * (K ** 0.5) + 1e-6


def test_static_scratch_gemm_in_a_captured_graph():
    """Two products in one captured graph (the second reads the first's result; both use the one
    array), replayed with new operands: as the same two calls outside."""
    import ctypes as C
    from paper_2507_22424_b200 import binding as B
    T, N, K = 27, 1024, 520
    x, w = _case(51, T, N, K)
    _, w2 = _case(52, 8, 512, N)
    y, z = torch.empty(T, N, device="cuda"), torch.empty(T, 512, device="cuda")

    def both():
        for a, b, c in ((x, w, y), (y, w2, z)):
            rc = B.lib.specvla_gemm_static(C.c_void_p(a.data_ptr()), C.c_void_p(b.data_ptr()), C.c_void_p(c.data_ptr()),
                                           a.shape[0], b.shape[0], a.shape[1], 0, B._stream())
            assert rc == 0

    both()                                                  # the device's first call is outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        both()
    for seed in (53, 54, 55):
        x.copy_(_case(seed, T, N, K)[0])
        y.fill_(float("nan"))
        z.fill_(float("nan"))
        for _ in range(3):                                  # replays back to back share the array
            graph.replay()
        assert B.lib.specvla_gemm_static_status(B._stream()) == 0
        want = B.gemm(B.gemm(x, w), w2)
        assert torch.equal(z, want)


# In a process of its own, where nothing else has mapped page-locked memory yet: the driver maps it from
# /dev/zero, two megabytes at least for the first four bytes.
ALLOCATES = """
import threading
import torch
from paper_2507_22424_b200 import binding as B

x = torch.randn(9, 264, device="cuda")
w = torch.randn(256, 264, device="cuda").to(torch.bfloat16)
y = torch.empty(9, 256, device="cuda")


def page_locked():
    return sorted(line.split()[0] for line in open("/proc/self/maps") if "/dev/zero" in line)


def calls():
    B.gemm_static(x, w, y)                                  # waits
    assert B.lib.specvla_gemm_static_status(B._stream()) == 0


rc = B.lib.specvla_gemm_static(x.data_ptr(), w.data_ptr(), y.data_ptr(), 9, 256, 264, 0, B._stream())
assert rc == 0
torch.cuda.synchronize()
y.cpu()                                                     # the device and the copy path are set up
before = page_locked()
calls()
thread = threading.Thread(target=calls)
thread.start()
thread.join()
assert page_locked() == before, (before, page_locked())
"""


def test_static_gemm_allocates_no_page_locked_memory():
    """A call that waits and the status call, on a thread's first use."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    done = subprocess.run([sys.executable, "-c", ALLOCATES], cwd=root, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
