"""Attention of launches with many rows (batched prefill, batched verification: blocks of 128 rows of one
episode, key tiles of 64 slots in two buffers) against the same episodes taken one at a time, and some
of them against the oracle itself. Episodes taken alone have at most 96 (32-row block, head) pairs and so
run the few-row kernel, which the oracle tests pin. Row counts sit at the edges of the 32- and 128-row blocks
and of the key tiles, with up to six tiles, so that both buffers are reused twice; trees of 128 rows
start before, on and after a tile edge, so that their masks lie across one to three tiles."""
import random

import pytest
import torch

from oracle.specvla import SpecVLAOracle
from synth_inputs import configs as C, data

import gpu_helpers as G

pytestmark = pytest.mark.gpu

DESCS = [C.ModelDesc(n_layers=2, d_model=8 * hd, n_heads=8, head_dim=hd, d_ffn=688, vocab=1024, action_base=768)
         for hd in (64, 128)]


def _batched_equals_single(desc, lens, tree_rows, seed, max_seq=320, oracle_eps=(1, 7)):
    """Prefill and scoring of all episodes in one call against one call per episode; logits of
    `oracle_eps` against the oracle."""
    w = data.make_weights(desc, 31)
    rng = random.Random(seed)
    n_ep = len(lens)
    ids = [[rng.randrange(desc.action_base) for _ in range(n)] for n in lens]
    gpu = G.make_gpu(desc, G.to_cuda(w), max_seq=max_seq, max_episodes=n_ep, max_rows=max(sum(lens), sum(tree_rows)),
                     action_only=True)
    embeds = torch.zeros(sum(lens), desc.d_model, dtype=torch.bfloat16, device="cuda")
    eps = list(range(n_ep))
    trees = []
    for e in eps:
        tok, par, dep = data.random_tree(tree_rows[e], desc, seed=e, max_depth=8, root_token=None)
        trees.append(dict(tokens=[desc.action_base + e] + list(tok)[1:], parent=list(par), depth=list(dep)))
    first, logits = gpu.prefill(eps, embeds, sum(ids, []), lens, want_logits=True)
    greedy = gpu.score_tree(eps, trees)
    margin = gpu.read_buffer(2, len(greedy), torch.float32)
    r0, checked = 0, 0
    for e in eps:
        f1, l1 = gpu.prefill([e], embeds[:lens[e]], ids[e], [lens[e]], want_logits=True)
        # both paths carry 16 mantissa bits per operand: 2 layers, logits of order 1
        assert (logits[e] - l1[0]).abs().max() < 1e-4, (e, lens[e])
        g1 = gpu.score_tree([e], [trees[e]])
        m1 = gpu.read_buffer(2, len(g1), torch.float32)
        for i, (a, b) in enumerate(zip(greedy[r0:r0 + len(g1)], g1)):
            if float(m1[i]) > 1e-3:
                assert a == b and abs(float(margin[r0 + i] - m1[i])) < 1e-3, (e, i)
                checked += 1
        r0 += len(g1)
    assert checked > 0.9 * len(greedy)
    orc = SpecVLAOracle(desc, w)
    for e in oracle_eps:
        embeds_e, ids_e = torch.zeros(lens[e], desc.d_model, dtype=torch.bfloat16), torch.tensor(ids[e])
        _, ref, _ = orc.prefill(embeds_e, ids_e, want_logits=True)
        assert (logits[e].cpu().double() - ref.reshape(-1)).abs().max() < 1e-3, (e, lens[e])
    gpu.close()


@pytest.mark.parametrize("desc", DESCS, ids=["head_dim64", "head_dim128"])
@pytest.mark.parametrize("n_ep", [16, 60])
def test_batched_rows_equal_single_episodes(desc, n_ep):
    edges = [65, 31, 97, 64, 33, 128, 96, 129, 63, 127]
    lens = [edges[i % len(edges)] if n_ep == 60 or i % 2 == 0 else 70 + i for i in range(n_ep)]
    _batched_equals_single(desc, lens, [[27, 40, 65][e % 3] for e in range(n_ep)], n_ep)


# prefixes of two and three row blocks and four to six key tiles; trees as wide as they get: the masks' upper
# half, first bits at every kind of offset within a tile
@pytest.mark.parametrize("desc", DESCS, ids=["head_dim64", "head_dim128"])
def test_long_prefixes_and_wide_trees(desc):
    lens = [255, 256, 257, 320, 319, 321, 191, 192, 193, 383, 128, 64, 63, 200]
    rows = [128, 128, 128, 128, 65, 127, 128, 33, 97, 64, 128, 128, 128, 1]
    _batched_equals_single(desc, lens, rows, 17, max_seq=520, oracle_eps=(2, 5, 9))


# 75 to 96 (row block, head) pairs: the few-row kernel with one slice; a block of one row, a full one and
# ragged ones, and the first and last count of it
@pytest.mark.parametrize("desc", DESCS, ids=["head_dim64", "head_dim128"])
@pytest.mark.parametrize("lens", [[32, 1, 31, 17, 5, 32, 29, 2, 32, 16], [64, 33, 31, 62, 1, 32, 64, 32]])
def test_one_slice_equals_single_episodes(desc, lens):
    blocks = sum((n + 31) // 32 for n in lens) * desc.n_heads
    assert 75 <= blocks <= 96, blocks
    _batched_equals_single(desc, lens, [[32, 27, 1][e % 3] for e in range(len(lens))], 3)


@pytest.mark.parametrize("desc", DESCS, ids=["head_dim64", "head_dim128"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_row_reaches_only_rows_that_see_it(desc, bad):
    """One input row that is not finite: the rows before it in its prefix, and the other prefixes, come out
    as without it, bit for bit; the rows from it on are NaN. Rows at both ends of a 128-row block and of a
    64-slot tile."""
    lens = [300, 130, 257, 200, 64, 129]
    rows = [0, 127, 128, 63, 64, 130, 199, 256, 299]
    gpu = G.make_gpu(desc, G.to_cuda(data.make_weights(desc, 31)), max_seq=320, max_episodes=len(lens), max_rows=sum(lens),
                     action_only=True)
    gen = torch.Generator().manual_seed(5)
    embeds = torch.randn(sum(lens), desc.d_model, generator=gen).mul_(0.5).to(torch.bfloat16).cuda()
    ids, eps = [-1] * sum(lens), list(range(len(lens)))

    def run(x):
        _, logits = gpu.prefill(eps, x, ids, lens, want_logits=True)
        # what the second layer wrote to the cache: the first layer's attention is in it
        return logits.cpu(), [[gpu.read_kv(e, 1, which, 0, lens[e]) for which in (0, 1)] for e in eps]

    good, kv = run(embeds)
    assert torch.isfinite(good).all()
    for e, row in [(0, r) for r in rows] + [(2, 255), (3, 198)]:
        if row >= lens[e]:
            continue
        x = embeds.clone()
        x[sum(lens[:e]) + row, 3] = bad
        logits, got = run(x)
        for other in eps:
            first_bad = row if other == e else lens[other]
            for which in (0, 1):
                assert torch.equal(got[other][which][:first_bad], kv[other][which][:first_bad]), (e, row, other)
                assert torch.isnan(got[other][which][first_bad:]).all(), (e, row, other)
            if other != e:
                assert torch.equal(logits[other], good[other])
        assert torch.isnan(logits[e]).all()
    gpu.close()
