"""The stand-alone product at the sizes where its launch plans change, against float64."""
import pytest
import torch

from synth_inputs import rng

pytestmark = pytest.mark.gpu


def _check(T, N, K, packed):
    from paper_2507_22424_b200.binding import gemm, gemm_prepacked, pack_weights
    x = rng.normal(21, 1, (T, K), 1.0, dtype=torch.float32)
    w = rng.normal_bf16(21, 2, (N, K), 0.02)
    ref = x.double() @ w.double().T
    y = (gemm_prepacked(x.cuda(), pack_weights(w.cuda()), N) if packed else gemm(x.cuda(), w.cuda())).cpu().double()
    # two-limb activations (2^-18 relative) and fp32 accumulation; outputs ~0.02 * sqrt(K)
    tol = 1e-4 * 0.02 * (K ** 0.5) + 1e-6
    assert (y - ref).abs().max() < tol, float((y - ref).abs().max())


# more row chunks than run side by side: a full group and a last one of one or several chunks, a ragged
# last chunk, one tile and several, with and without K slices
@pytest.mark.parametrize("T,N,K", [(1537, 512, 64), (1665, 1000, 256), (3100, 256, 1024), (2049, 768, 520)])
@pytest.mark.parametrize("packed", [True, False])
def test_many_row_chunks(T, N, K, packed):
    _check(T, N, K, packed)


# MMA widths of the 64-row instantiation: the next multiple of eight rows, first and last row of each
@pytest.mark.parametrize("T", [33, 40, 41, 57, 64, 65])
def test_widths_between_33_and_64_rows(T):
    _check(T, 1000, 520, True)


# the long instantiation sizes its ring by the rows: four stages up to 88, three above; 17 K blocks go
# through it, unsplit, so that every stage is refilled
@pytest.mark.parametrize("T", [65, 72, 80, 81, 88, 89, 96, 128])
def test_ring_sizes_of_long_tiles(T):
    _check(T, 20480, 1032, True)


# several chunks with a tail box of the same width
@pytest.mark.parametrize("T", [170, 176])
def test_ring_sizes_of_several_chunks(T):
    _check(T, 4096, 2056, True)


# a narrower tail box inside stages sized by the longer chunk: by the launch plan three chunks, unsplit, of 80
# (tail 64) and 88 rows (72) in four stages, of 104 (96) and 120 rows (104) in three, and two of 80 (72) over K slices
@pytest.mark.parametrize("T,N,K", [(220, 20480, 1032), (245, 20480, 1032), (300, 20480, 1032), (340, 20480, 1032),
                                   (150, 4096, 2056)])
def test_ring_with_a_narrower_tail(T, N, K):
    _check(T, N, K, True)


def test_operand_off_a_16_byte_boundary():
    """The split takes X four values at a time only where it starts on 16 bytes."""
    from paper_2507_22424_b200.binding import gemm
    T, N, K = 19, 256, 264
    x = rng.normal(22, 1, (T, K), 1.0, dtype=torch.float32)
    w = rng.normal_bf16(22, 2, (N, K), 0.02).cuda()
    buf = torch.empty(T * K + 1, dtype=torch.float32, device="cuda")
    off = buf[1:].view(T, K)
    off.copy_(x)
    assert off.data_ptr() % 16 == 4
    assert torch.equal(gemm(off, w), gemm(x.cuda(), w))
