"""Sliced launches whose last tile is partly past the matrix, or whose tiles are partly outside the scored id
range: threads whose values no output takes read their peers' partial sums like the others."""
import pytest
import torch

from oracle import quant as Q
from oracle.specvla import SpecVLAOracle, Tree
from synth_inputs import configs as C, data, rng

import gpu_helpers as G

pytestmark = pytest.mark.gpu


# 33 K blocks over clusters; 4 and 128 columns in the last tile, at each operand width
@pytest.mark.parametrize("T", [1, 9, 27, 60, 100])
@pytest.mark.parametrize("N", [4, 260, 384])
def test_product_with_a_ragged_last_tile(T, N):
    from paper_2507_22424_b200.binding import gemm, gemm_prepacked, pack_weights
    K = 2056
    x = rng.normal(61, 1, (T, K), 1.0, dtype=torch.float32)
    w = rng.normal_bf16(61, 2, (N, K), 0.02)
    ref = x.double() @ w.double().T
    tol = 1e-4 * 0.02 * (K ** 0.5) + 1e-6                   # two-limb activations and fp32 accumulation
    for y in (gemm(x.cuda(), w.cuda()), gemm_prepacked(x.cuda(), pack_weights(w.cuda()), N)):
        assert (y.cpu().double() - ref).abs().max() < tol


# width 640: QKV, O and down end with half a tile, gate/up with 48 of 128 columns, each over K slices; the
# scored ids start and end inside a tile of the head
@pytest.mark.parametrize("bits", [16, 8])
@pytest.mark.parametrize("n_rows", [1, 27, 60, 90])
def test_model_with_ragged_tiles(bits, n_rows):
    desc = C.ModelDesc(n_layers=2, d_model=640, n_heads=10, head_dim=64, d_ffn=2096, vocab=1024, action_base=702)
    w = data.make_weights(desc, 8)
    orc = SpecVLAOracle(desc, Q.quantize_target(w) if bits == 8 else w)
    gpu = G.make_gpu(desc, G.to_cuda(w), max_seq=256, max_episodes=1, max_rows=256, action_only=True, weight_bits=bits)
    tally = G.Tally()
    ids = torch.arange(40) * 7 % desc.action_base
    embeds = torch.zeros(40, desc.d_model, dtype=torch.bfloat16)
    ep, _, _ = G.prefill_both(orc, gpu, embeds.cuda(), ids, 0, tally, desc)
    tok, par, dep = data.random_tree(n_rows, desc, seed=n_rows, max_depth=8, root_token=ep.root)
    tree = Tree(tok, par, dep, [0.0] * n_rows)
    greedy = gpu.score_tree([0], [G.tree_dict(tree)])       # no logits: only the scored columns are stored
    G.verify_both(orc, gpu, ep, tree, 40, tally, desc, where=f"ragged({bits}, T={n_rows})")
    assert greedy == gpu.read_buffer(1, n_rows, torch.int32).tolist()
    # fp32 rounding only: a partial sum that was left out moves a logit by about 0.1
    assert tally.accepts == 1 and tally.caches == 1 and tally.max_logit_err < 2e-4, tally.max_logit_err
    gpu.close()
