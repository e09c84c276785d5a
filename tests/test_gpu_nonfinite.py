"""Inputs that are not finite: tokens are embedding row numbers, so every path must still return valid
ids, come to its end and leave the context as good as before."""
import pytest
import torch

from synth_inputs import configs as C

import gpu_helpers as G

pytestmark = pytest.mark.gpu

SHAPES = {"none": ((), (), 0), "static": ((2, 2, 2), (1, 2, 4), 0), "dynamic": ((8, 8, 8), (1, 8, 8), 20)}


@pytest.mark.parametrize("action_only", [True, False])
@pytest.mark.parametrize("bits,persistent", [(16, False), (16, True), (8, False)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_chunk_of_a_non_finite_image(c0, action_only, bits, persistent, bad):
    from paper_2507_22424_b200 import binding as B
    desc, n = c0["desc"], len(c0["ids"])
    gpu = G.make_gpu(desc, G.to_cuda(c0["weights"]), max_seq=256, max_episodes=2, max_rows=256, action_only=action_only,
                     weight_bits=bits)
    if persistent:
        gpu.set_option(B.OPT_PERSISTENT_FORWARD, 1)
    good, broken = c0["embeds"].cuda(), c0["embeds"].cuda().clone()
    broken[n // 2, 5] = bad
    lo, hi = (desc.action_base, desc.action_base + desc.n_bins) if action_only else (0, desc.vocab)
    for name, (branch, expand, keep) in SHAPES.items():
        shape = B.make_shape(branch, expand, keep=keep)
        want = gpu.generate_action([0], good, c0["ids"].tolist(), [n], shape, 4, 7)[0]
        pair = gpu.generate_action([0, 1], torch.cat((good, good)), c0["ids"].tolist() * 2, [n, n], shape, 4, 7)[0]
        for device_loop in (1, 0):
            gpu.set_option(B.OPT_DEVICE_LOOP, device_loop)
            toks, _, _ = gpu.generate_action([0], broken, c0["ids"].tolist(), [n], shape, 4, 7)
            assert all(lo <= t < hi for t in toks[0]), (name, toks)
            # two episodes in one call: the other one is not touched
            both = torch.cat((broken, good))
            toks, _, _ = gpu.generate_action([0, 1], both, c0["ids"].tolist() * 2, [n, n], shape, 4, 7)
            assert all(lo <= t < hi for t in toks[0]) and toks[1] == pair[1], (name, toks, pair)
            assert gpu.generate_action([0], good, c0["ids"].tolist(), [n], shape, 4, 7)[0] == want
    gpu.close()


def test_draft_tree_of_non_finite_features(c0):
    from paper_2507_22424_b200 import binding as B
    desc, n = c0["desc"], len(c0["ids"])
    gpu = G.make_gpu(desc, G.to_cuda(c0["weights"]), max_seq=256, max_episodes=1, max_rows=256, action_only=True)
    first = gpu.prefill([0], torch.full_like(c0["embeds"], float("nan")).cuda(), c0["ids"].tolist(), [n])
    assert first == [desc.action_base]                      # nothing comparable: the lowest id of the range
    for branch, expand, keep in list(SHAPES.values())[1:]:
        t = gpu.draft_tree([0], B.make_shape(branch, expand, keep=keep))[0]
        assert all(desc.action_base <= x < desc.action_base + desc.n_bins for x in t["tokens"])
        assert t["parent"][0] == -1 and all(0 <= t["parent"][i] < i for i in range(1, len(t["parent"])))
        gpu.prefill([0], torch.full_like(c0["embeds"], float("nan")).cuda(), c0["ids"].tolist(), [n])
    gpu.close()
