"""The int8 expansion at the row counts where its launches change: the last width of one MMA operand
(64), the first launch of the long instantiation (65), its widest chunk (96) and the first launch of
two chunks (97), against the quantised oracle."""
import pytest
import torch

from oracle import quant as Q
from oracle.specvla import SpecVLAOracle, Tree
from synth_inputs import configs as C, data

import gpu_helpers as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rows", [64, 65, 96, 97])
def test_quantised_verify_at_chunk_edges(c0, n_rows):
    desc = c0["desc"]
    orc = SpecVLAOracle(C.TINY, Q.quantize_target(c0["weights"]))
    gpu = G.make_gpu(desc, G.to_cuda(c0["weights"]), max_seq=256, max_episodes=1, max_rows=256, action_only=True,
                     weight_bits=8)
    tally = G.Tally()
    ep, _, _ = G.prefill_both(orc, gpu, c0["embeds"].cuda(), c0["ids"], 0, tally, desc)
    tok, par, dep = data.random_tree(n_rows, desc, seed=n_rows, max_depth=8, root_token=ep.root)
    G.verify_both(orc, gpu, ep, Tree(tok, par, dep, [0.0] * n_rows), 40, tally, desc, where=f"q8.g(T={n_rows})")
    # one wrong code would move a logit by about 1e-3; identical codes leave fp32 rounding only
    assert tally.accepts == 1 and tally.caches == 1 and tally.max_logit_err < 2e-4, tally.max_logit_err
    gpu.close()


@pytest.mark.parametrize("n_rows", [1, 27, 64, 96])
def test_code_ring_is_refilled(n_rows):
    """A down projection of 94 K blocks over clusters of eight: eleven or twelve units per CTA, more than
    the ring of eight holds, so every slot a set has freed is written again; at each operand width."""
    desc = C.ModelDesc(n_layers=2, d_model=256, n_heads=4, head_dim=64, d_ffn=6008, vocab=1024, action_base=768)
    w = data.make_weights(desc, 5)
    orc = SpecVLAOracle(desc, Q.quantize_target(w))
    gpu = G.make_gpu(desc, G.to_cuda(w), max_seq=256, max_episodes=1, max_rows=256, action_only=True, weight_bits=8)
    tally = G.Tally()
    ids = torch.arange(40) * 7 % desc.action_base
    embeds = torch.zeros(40, desc.d_model, dtype=torch.bfloat16)
    ep, _, _ = G.prefill_both(orc, gpu, embeds.cuda(), ids, 0, tally, desc)
    tok, par, dep = data.random_tree(n_rows, desc, seed=n_rows, max_depth=8, root_token=ep.root)
    G.verify_both(orc, gpu, ep, Tree(tok, par, dep, [0.0] * n_rows), 40, tally, desc, where=f"q8.ring(T={n_rows})")
    # a unit whose codes were overwritten moves every logit by far more than rounding does
    assert tally.accepts == 1 and tally.caches == 1 and tally.max_logit_err < 2e-4, tally.max_logit_err
    gpu.close()


@pytest.mark.parametrize("k_blocks", [1, 2, 3])
def test_fewer_units_than_expanding_sets(k_blocks):
    """One to three K blocks per tile: some sets of expanding warps have no unit, or exactly one."""
    desc = C.ModelDesc(n_layers=2, d_model=64 * k_blocks, n_heads=2, head_dim=64, d_ffn=64 * k_blocks, vocab=1024,
                       action_base=768)
    w = data.make_weights(desc, 6)
    orc = SpecVLAOracle(desc, Q.quantize_target(w))
    gpu = G.make_gpu(desc, G.to_cuda(w), max_seq=256, max_episodes=1, max_rows=256, action_only=True, weight_bits=8)
    tally = G.Tally()
    ids = torch.arange(40) * 7 % desc.action_base
    embeds = torch.zeros(40, desc.d_model, dtype=torch.bfloat16)
    ep, _, _ = G.prefill_both(orc, gpu, embeds.cuda(), ids, 0, tally, desc)
    tok, par, dep = data.random_tree(27, desc, seed=k_blocks, max_depth=8, root_token=ep.root)
    G.verify_both(orc, gpu, ep, Tree(tok, par, dep, [0.0] * 27), 40, tally, desc, where=f"q8.units({k_blocks})")
    # a unit that was left out moves every logit by far more than rounding does (2e-4, as above)
    assert tally.accepts == 1 and tally.caches == 1 and tally.max_logit_err < 2e-4, tally.max_logit_err
    gpu.close()
