"""A stand-alone product that is refused fails alone: its error and the one-call test hook end with it."""
import ctypes as C

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


def test_status_belongs_to_the_calling_thread():
    """Products from several threads on streams of their own: each reads its own status and result."""
    import threading
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
