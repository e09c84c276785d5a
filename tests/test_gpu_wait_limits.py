"""Failure detection without a fault: one launch of a context withholds a tile under a wait limit of 2 ms.
The call must come back with SPECVLA_ERR_TIMEOUT, once, and the next ordinary call be as before."""
import functools
import random
import time

import pytest
import torch

from synth_inputs import configs as C, data

import gpu_helpers as G

pytestmark = pytest.mark.gpu


def _timed_out(call):
    from paper_2507_22424_b200.binding import SpecVLAError
    t0 = time.perf_counter()
    with pytest.raises(SpecVLAError) as e:
        call()
    assert e.value.code == -6, e.value                                  # SPECVLA_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 5.0


@functools.lru_cache(maxsize=None)
def _weights(desc, seed):
    return G.to_cuda(data.make_weights(desc, seed))


class Episodes:
    """A context with a batch of prefixes and one tree per episode."""

    def __init__(self, desc, lens, seed, rows, bits=16):
        from paper_2507_22424_b200 import binding as B
        rng = random.Random(seed)
        self.eps, self.lens = list(range(len(lens))), lens
        self.ids = [rng.randrange(desc.action_base) for _ in range(sum(lens))]
        self.embeds = torch.zeros(sum(lens), desc.d_model, dtype=torch.bfloat16, device="cuda")
        self.trees = []
        for e in self.eps:
            tok, par, dep = data.random_tree(rows, desc, seed=e, max_depth=8, root_token=desc.action_base + e)
            self.trees.append(dict(tokens=list(tok), parent=list(par), depth=list(dep)))
        self.gpu = G.make_gpu(desc, _weights(desc, seed), max_seq=512, max_episodes=len(lens),
                              max_rows=max(sum(lens), rows * len(lens)), action_only=True, weight_bits=bits)
        self.shape = B.make_shape((2, 2, 2), (1, 2, 4))

    def prefill(self):
        first, logits = self.gpu.prefill(self.eps, self.embeds, self.ids, self.lens, want_logits=True)
        return first, logits.cpu()

    def score(self):
        return self.gpu.score_tree(self.eps, self.trees)

    def chunk(self):
        return self.gpu.generate_action(self.eps, self.embeds, self.ids, self.lens, self.shape, 4, 7)[0]


def _exercise(s, option, index):
    from paper_2507_22424_b200 import binding as B
    first, logits = s.prefill()
    greedy = s.score()
    chunk = s.chunk()
    s.prefill()
    s.gpu.set_option(B.OPT_WAIT_LIMIT_NS, 2_000_000)

    s.gpu.set_option(option, index)
    _timed_out(s.prefill)
    with pytest.raises(B.SpecVLAError) as e:
        s.score()
    assert e.value.code == -4                                           # SPECVLA_ERR_BAD_STATE: prefill again
    f, l = s.prefill()
    assert f == first and torch.equal(l, logits)

    s.gpu.set_option(option, index)
    _timed_out(s.score)
    assert s.score() == greedy                                          # a scoring call changes no state

    s.gpu.set_option(option, index)
    _timed_out(lambda: s.gpu.verify_tree(s.eps, s.trees, 4))
    with pytest.raises(B.SpecVLAError) as e:
        s.gpu.verify_tree(s.eps, s.trees, 4)
    assert e.value.code == -4

    for device_loop in (1, 0):
        s.gpu.set_option(B.OPT_DEVICE_LOOP, device_loop)
        s.gpu.set_option(option, index)
        _timed_out(s.chunk)
        assert s.chunk() == chunk
    s.gpu.set_option(B.OPT_WAIT_LIMIT_NS, 2_000_000_000)
    f, l = s.prefill()
    assert f == first and torch.equal(l, logits) and s.score() == greedy
    s.gpu.close()


# first tile, second buffer, the first tile of a reused buffer, the third use of one
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("tile", [0, 1, 2, 4])
def test_withheld_key_tile(head_dim, tile):
    from paper_2507_22424_b200 import binding as B
    desc = C.ModelDesc(n_layers=2, d_model=8 * head_dim, n_heads=8, head_dim=head_dim, d_ffn=688, vocab=1024,
                       action_base=768)
    _exercise(Episodes(desc, [300 + 3 * i for i in range(14)], 41, 27), B.OPT_WITHHOLD_KEYS, tile)


# first unit of each of the three sets of expanding warps (64 rows at most), a later one of each, among them the
# first past the code ring (8), the last
@pytest.mark.parametrize("unit", [0, 1, 2, 6, 8, 9, 13, 15])
@pytest.mark.parametrize("bits,rows", [(8, 9), (8, 60), (16, 9)])
def test_withheld_weights(unit, bits, rows):
    """QKV of 128 K blocks over clusters of eight: sixteen units per CTA."""
    from paper_2507_22424_b200 import binding as B
    desc = C.ModelDesc(n_layers=1, d_model=8192, n_heads=4, head_dim=64, d_ffn=256, vocab=1024, action_base=768)
    _exercise(Episodes(desc, [40, 33], 42, rows, bits), B.OPT_WITHHOLD_GEMM, unit)
