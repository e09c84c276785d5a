"""Timed workloads of the Spec-VLA decoding path, through the package's public entry points.

A case is a dict of plain values. Its "kind" says which call is timed:

  chunk    SpecVLA.generate_action: prefill, then draft tree -> verification -> acceptance until the
           action chunk is complete (what a robot controller calls once per control step)
  prefill  SpecVLA.prefill over one or many episodes, with the last rows' logits
  score    SpecVLA.score_tree: one verification forward over a draft tree (or a single row: an
           autoregressive step) against a committed prefix
  gemm     gemm_prepacked: the stand-alone weight-streaming product

One context per model and weight format is made once per process and serves every case, as a server
does; what a case's `prepare` makes from the seed are the episodes: image features, prompts, trees.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2507_22424_b200 import binding as B

# The two decoders of this repository's workloads (OpenVLA-7B-shaped, and the tiny one).
MODELS = {
    "7b": SimpleNamespace(n_layers=32, d_model=4096, n_heads=32, head_dim=128, d_ffn=11008, vocab=32064,
                          action_base=31744, n_bins=256, rms_eps=1e-6, rope_theta=1e4),
    "tiny": SimpleNamespace(n_layers=2, d_model=256, n_heads=4, head_dim=64, d_ffn=688, vocab=1024,
                            action_base=768, n_bins=256, rms_eps=1e-6, rope_theta=1e4),
}
# Draft trees: the static 14- and 26-node trees, the dynamic top-8 tree of depth 5 of which the 50
# best nodes are verified, and none (autoregressive decoding).
TREES = {
    "none": ((), (), 0),
    "static14": ((2, 2, 2), (1, 2, 4), 0),
    "static26": ((4, 2, 2, 1, 1), (1, 4, 3, 4, 4), 0),
    "dynamic50": ((8, 8, 8, 8, 8), (1, 8, 8, 8, 8), 50),
}
# Verification steps that a seven-token chunk takes with these trees on the weights below (mean over
# seeds, as measured; used only to count a chunk's work).
STEPS = {"none": 6.0, "static14": 2.0, "static26": 4.5, "dynamic50": 4.0}

MAX_SEQ, MAX_ROWS = 640, 5120


# ------------------------------------------------------------------------------------ the cases
def _chunk(**kw):
    return dict(dict(kind="chunk", model="7b", bits=16, episodes=1, visual=256, text_lo=34, text_hi=34,
                     tree="static26", r=0, tokens=7), **kw)


def _prefill(**kw):
    return dict(dict(kind="prefill", model="7b", bits=16, episodes=1, visual=256, text_lo=34, text_hi=34), **kw)


def _score(**kw):
    return dict(dict(kind="score", model="7b", bits=16, prefix=290, rows=27), **kw)


def listed():
    return [
        # the tiny decoder: nothing but launches and latency
        _chunk(name="chunk-tiny", model="tiny", visual=64, text_lo=0, text_hi=0, tree="static14", r=4),
        # a text-only prompt (language part of an instruction, no image)
        _prefill(name="prefill-34", visual=0),
        # one camera frame (256 patches) and a short instruction
        _prefill(name="prefill-290"),
        # a server's batch of sixteen ragged episodes
        _prefill(name="prefill-16x", episodes=16, text_lo=20, text_hi=60),
        # verification of one tree: an autoregressive step, the static tree, the widest tree
        _score(name="score-1", rows=1),
        _score(name="score-27"),
        _score(name="score-128", rows=128),
        # the int8 target on the same tree
        _score(name="score-27-int8", bits=8),
        # the control step: one episode, strict acceptance
        _chunk(name="chunk-26"),
        # the same with the dynamic tree and relaxed acceptance
        _chunk(name="chunk-dynamic-50", tree="dynamic50", r=9),
        # sixteen ragged episodes decoded together
        _chunk(name="chunk-16x", episodes=16, text_lo=20, text_hi=60, r=4),
        # the product alone: the down projection over the rows of a tree
        dict(name="gemm-27", kind="gemm", t=27, n=4096, k=11008),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("chunk", "prefill", "score", "score", "gemm"))
    if kind == "gemm":
        # N and K in the multiples the entry point asks for
        return dict(kind="gemm", t=_log_int(rng, 1, 512), n=4 * _log_int(rng, 64, 5504), k=8 * _log_int(rng, 32, 1376))
    if kind == "score":
        return _score(rows=_log_int(rng, 1, 128), prefix=_log_int(rng, 32, 480), bits=rng.choice((16, 16, 16, 8)))
    if kind == "prefill":
        n_ep = _log_int(rng, 1, 16)
        lo = rng.randint(4, 60)
        return _prefill(episodes=n_ep, visual=rng.choice((0, 256, 256)), text_lo=lo, text_hi=rng.randint(lo, 60))
    if rng.random() < 0.25:
        return _chunk(model="tiny", visual=rng.randint(16, 64), text_lo=0, text_hi=rng.randint(0, 32), tree="static14",
                      r=rng.choice((0, 1, 4, 9)), tokens=rng.randint(4, 14))
    lo = rng.randint(20, 60)
    return _chunk(episodes=rng.choice((1, 1, 1, 2, 4, 8)), text_lo=lo, text_hi=rng.randint(lo, 60),
                  tree=rng.choice(("none", "static26", "static26", "dynamic50")), r=rng.choice((0, 1, 2, 4, 5, 9)),
                  bits=rng.choice((16, 16, 16, 8)))


# ------------------------------------------------------------------------------------ contexts
_CONTEXTS, _WEIGHTS, _NEXT_EPISODE = {}, {}, {}


def _weights(name):
    """Weights of a decoder and its one-layer draft head: N(0, 0.02), the projections that write to the
    residual stream smaller by 2 sqrt(2 layers) (as decoders are initialised, so that the logits are
    as well conditioned as a trained model's), embeddings at the scale of the image features. The
    draft head's input layer passes the token's embedding on, so that draft and target agree on the
    next token about as often as a trained head does."""
    if name not in _WEIGHTS:
        m = MODELS[name]
        g = torch.Generator(device="cuda")
        g.manual_seed(20250722)
        d, f, hd = m.d_model, m.d_ffn, m.n_heads * m.head_dim
        res = 0.02 / (2.0 * math.sqrt(2.0 * m.n_layers))

        def mat(rows, cols, std=0.02):
            return torch.randn(rows, cols, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)

        def ones():
            return torch.ones(d, dtype=torch.float32, device="cuda")

        w = {"embed": mat(m.vocab, d, 0.5), "lm_head": mat(m.vocab, d), "final_norm": ones()}
        for p in ["layers.%d." % i for i in range(m.n_layers)] + ["draft.layer."]:
            w.update({p + "wqkv": mat(3 * hd, d), p + "wo": mat(d, hd, res), p + "wgu": mat(2 * f, d),
                      p + "wd": mat(d, f, res), p + "norm1": ones(), p + "norm2": ones()})
        fc = mat(d, 2 * d, 0.002)
        fc[:, d:] += torch.eye(d, device="cuda", dtype=torch.bfloat16)
        w["draft.fc"] = fc
        _WEIGHTS[name] = w
    return _WEIGHTS[name]


def _context(name, bits):
    key = (name, bits)
    if key not in _CONTEXTS:
        _CONTEXTS[key] = B.SpecVLA(MODELS[name], _weights(name), max_seq=MAX_SEQ, max_episodes=16, max_rows=MAX_ROWS,
                                   action_only=True, weight_bits=bits)
        _NEXT_EPISODE[key] = 0
    return _CONTEXTS[key]


def _prefix(m, lens, n_visual, g, rng):
    """Rows of the call's episodes: image features N(0, 0.5), then prompt tokens given by id."""
    ids = []
    for n in lens:
        ids += [-1] * n_visual + [rng.randrange(m.action_base) for _ in range(n - n_visual)]
    embeds = torch.randn(len(ids), m.d_model, generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.5)
    return embeds, ids


def _tree(m, rows, rng):
    """A draft tree of `rows` rows: random topology (at most eight levels), action tokens."""
    parent, depth = [-1], [0]
    for i in range(1, rows):
        p = rng.randrange(i)
        while depth[p] >= B.MAX_DEPTH:
            p = parent[p]
        parent.append(p)
        depth.append(depth[p] + 1)
    return dict(tokens=[m.action_base + rng.randrange(m.n_bins) for _ in range(rows)], parent=parent, depth=depth)


def prepare(case, seed):
    rng = random.Random(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "gemm":
        t, n, k = case["t"], case["n"], case["k"]
        x = torch.randn(t, k, generator=g, device="cuda", dtype=torch.float32)
        w = torch.randn(n, k, generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.02)
        return dict(kind="gemm", x=x, packed=B.pack_weights(w), n=n)
    m = MODELS[case["model"]]
    ctx = _context(case["model"], case["bits"])
    if case["kind"] == "score":
        key = (case["model"], case["bits"])
        ep = _NEXT_EPISODE[key]
        _NEXT_EPISODE[key] = (ep + 1) % 16
        n = case["prefix"]
        embeds, ids = _prefix(m, [n], min(256, n // 2), g, rng)
        ctx.prefill([ep], embeds, ids, [n])
        return dict(kind="score", ctx=ctx, episodes=[ep], trees=[_tree(m, case["rows"], rng)], rows=case["rows"])
    lens = [case["visual"] + rng.randint(case["text_lo"], case["text_hi"]) for _ in range(case["episodes"])]
    embeds, ids = _prefix(m, lens, case["visual"], g, rng)
    s = dict(kind=case["kind"], ctx=ctx, episodes=list(range(case["episodes"])), embeds=embeds, ids=ids, lens=lens)
    if case["kind"] == "chunk":
        branch, expand, keep = TREES[case["tree"]]
        s.update(shape=B.make_shape(branch, expand, keep=keep), r=case["r"], tokens=case["tokens"])
    return s


def run(s):
    if s["kind"] == "gemm":
        return B.gemm_prepacked(s["x"], s["packed"], s["n"])
    ctx = s["ctx"]
    if s["kind"] == "prefill":
        first, logits = ctx.prefill(s["episodes"], s["embeds"], s["ids"], s["lens"], want_logits=True)
        return dict(first=np.array(first), logits=logits)
    if s["kind"] == "score":
        # the greedy tokens, and the confidence (top-1 minus top-2 logit) of every row
        greedy = ctx.score_tree(s["episodes"], s["trees"])
        return dict(greedy=np.array(greedy), margin=ctx.read_buffer(B.BUF_MARGIN, s["rows"], torch.float32))
    tokens, actions, stats = ctx.generate_action(s["episodes"], s["embeds"], s["ids"], s["lens"], s["shape"], s["r"],
                                                 s["tokens"])
    return dict(tokens=np.array(tokens), actions=np.array(actions), iterations=stats.iterations,
                accepted=np.array(stats.accept_len[:]))


# ------------------------------------------------------------------------------------ in 64 bits
def _mat64(w, name, bits):
    """A weight matrix in float64; with bits = 8 as the quantised target holds it (per row: scale =
    max / 127, codes rounded half to even, scale and quotient in float32)."""
    t = w[name]
    if bits != 8:
        return t.double()
    f = t.float()
    top = f.abs().amax(dim=1, keepdim=True)
    scale = top / torch.full_like(top, 127.0)
    scale[scale == 0] = 1.0
    return (f / scale).round_().clamp_(-127, 127).double() * scale.double()


def _decode64(m, w, x, pos, parts, bits):
    """The decoder over the rows x at RoPE positions pos; parts = (first row, rows, mask) of every
    episode. Returns the final-norm output."""
    half, n = m.head_dim // 2, x.shape[0]
    ang = pos.double()[:, None] * m.rope_theta ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]

    def norm(v, gain):
        return v * torch.rsqrt((v * v).mean(dim=1, keepdim=True) + m.rms_eps) * w[gain].double()

    def rotate(v):
        a, b = v[..., :half], v[..., half:]
        return torch.cat((a * cos - b * sin, b * cos + a * sin), dim=-1)

    for i in range(m.n_layers):
        p = "layers.%d." % i
        q, k, v = (norm(x, p + "norm1") @ _mat64(w, p + "wqkv", bits).T).view(n, 3, m.n_heads, m.head_dim).unbind(1)
        q, k = rotate(q), rotate(k)
        out = torch.empty_like(v)
        for r0, rows, mask in parts:
            s = slice(r0, r0 + rows)
            a = torch.einsum("thd,shd->hts", q[s], k[s]) * m.head_dim ** -0.5
            a = a.masked_fill(~mask, -math.inf).softmax(dim=-1)
            out[s] = torch.einsum("hts,shd->thd", a, v[s])
        x = x + out.reshape(n, -1) @ _mat64(w, p + "wo", bits).T
        gate, up = (norm(x, p + "norm2") @ _mat64(w, p + "wgu", bits).T).chunk(2, dim=1)
        x = x + (torch.nn.functional.silu(gate) * up) @ _mat64(w, p + "wd", bits).T
    return norm(x, "final_norm")


def _inputs64(w, embeds, ids):
    ids = torch.tensor(ids, device="cuda")
    return torch.where((ids < 0)[:, None], embeds, w["embed"][ids.clamp(min=0)]).double()


def exact(case, seed):
    """What run() returns, in 64 bits. None for a chunk: its tokens are whole values."""
    if case["kind"] == "chunk":
        return None
    rng = random.Random(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "gemm":
        x = torch.randn(case["t"], case["k"], generator=g, device="cuda", dtype=torch.float32)
        w = torch.randn(case["n"], case["k"], generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.02)
        return x.double() @ w.double().T
    m, w, bits = MODELS[case["model"]], _weights(case["model"]), case["bits"]
    act = slice(m.action_base, m.action_base + m.n_bins)
    if case["kind"] == "score":
        n, rows = case["prefix"], case["rows"]
        embeds, ids = _prefix(m, [n], min(256, n // 2), g, rng)
        tree = _tree(m, rows, rng)
        mask = torch.ones(n + rows, n + rows, dtype=torch.bool, device="cuda").tril_()
        mask[n:, n:] = False
        sees = np.zeros((rows, rows), dtype=bool)
        for i, p in enumerate(tree["parent"]):
            if p >= 0:
                sees[i] = sees[p]
            sees[i, i] = True
        mask[n:, n:] = torch.from_numpy(sees).cuda()
        pos = torch.tensor(list(range(n)) + [n + d for d in tree["depth"]], device="cuda")
        x = _inputs64(w, torch.cat((embeds, embeds.new_zeros(rows, m.d_model))), ids + tree["tokens"])
        h = _decode64(m, w, x, pos, [(0, n + rows, mask)], bits)
        top = (h[n:] @ _mat64(w, "lm_head", bits)[act].T).topk(2, dim=1)
        return dict(greedy=(top.indices[:, 0] + m.action_base).cpu().numpy(),
                    margin=(top.values[:, 0] - top.values[:, 1]).cpu())
    lens = [case["visual"] + rng.randint(case["text_lo"], case["text_hi"]) for _ in range(case["episodes"])]
    embeds, ids = _prefix(m, lens, case["visual"], g, rng)
    parts, r0 = [], 0
    for n in lens:
        parts.append((r0, n, torch.ones(n, n, dtype=torch.bool, device="cuda").tril_()))
        r0 += n
    pos = torch.cat([torch.arange(n, device="cuda") for n in lens])
    h = _decode64(m, w, _inputs64(w, embeds, ids), pos, parts, bits)
    logits = h[[r + n - 1 for r, n, _ in parts]] @ _mat64(w, "lm_head", bits).T
    return dict(first=(logits[:, act].argmax(dim=1) + m.action_base).cpu().numpy(), logits=logits)


# ------------------------------------------------------------------------------------ work and tolerance
def _forward(m, rows, keys, n_ep, heads, bits):
    """(bytes, flops) of one forward of the target over `rows` rows of n_ep episodes with `keys` visible
    positions each: the weights once, the K/V rows read and written at two bytes an element, `heads`
    rows scored over the action ids."""
    hd = m.n_heads * m.head_dim
    layer = 4 * hd * m.d_model + 3 * m.d_model * m.d_ffn
    by = m.n_layers * (layer * bits // 8 + 4 * hd * (n_ep * keys + rows)) + m.n_bins * m.d_model * 2
    fl = m.n_layers * (2 * rows * layer + 4 * rows * keys * hd) + 2 * heads * m.n_bins * m.d_model
    return by, fl


def _draft_level(m, rows, keys, n_ep, heads):
    """The same of one forward of the draft head (its input layer, one decoder layer)."""
    hd = m.n_heads * m.head_dim
    p = 4 * hd * m.d_model + 3 * m.d_model * m.d_ffn + 2 * m.d_model * m.d_model
    by = 2 * p + 4 * hd * (n_ep * keys + rows) + 2 * m.n_bins * m.d_model
    return by, 2 * rows * p + 2 * heads * m.n_bins * m.d_model + 4 * rows * keys * hd


def work(case):
    if case["kind"] == "gemm":
        t, n, k = case["t"], case["n"], case["k"]
        return dict(bytes=2 * n * k + 4 * t * (k + n), flops=2 * t * n * k)
    m = MODELS[case["model"]]
    if case["kind"] == "score":
        by, fl = _forward(m, case["rows"], case["prefix"], 1, case["rows"], case["bits"])
        return dict(bytes=by, flops=fl)
    n_ep = case["episodes"]
    prefix = int(case["visual"] + 0.5 * (case["text_lo"] + case["text_hi"]))
    rows = n_ep * prefix
    # (causal: half the prefix is visible on average; its keys are the rows the call itself writes)
    by, fl = _forward(m, rows, prefix // 2, 0, n_ep, case["bits"])
    dby, dfl = _draft_level(m, rows, prefix // 2, 0, 0)
    by, fl = by + dby + 2 * rows * m.d_model, fl + dfl
    if case["kind"] == "chunk":
        branch, expand, keep = TREES[case["tree"]]
        nodes = sum(b * e for b, e in zip(branch, expand))
        steps = STEPS[case["tree"]] * (case["tokens"] - 1) / 6.0
        tree_rows = 1 + (min(keep, nodes) if keep else nodes)
        # (the rows of all episodes share one pass over the weights; every episode has its own keys)
        vby, vfl = _forward(m, n_ep * tree_rows, prefix, n_ep, n_ep * tree_rows, case["bits"])
        by, fl = by + steps * vby, fl + steps * vfl
        for e in expand:
            lby, lfl = _draft_level(m, n_ep * e, prefix, n_ep, n_ep * e)
            by, fl = by + steps * lby, fl + steps * lfl
    return dict(bytes=int(by), flops=int(fl))


def tolerance(case):
    """About four times what the same path shows against 64-bit arithmetic (weights bf16 or int8,
    activations 16 mantissa bits, float32 sums). Greedy tokens may differ where two logits tie."""
    if case["kind"] == "gemm":
        return dict(rel=1.2e-5)                                   # 3.1e-6 at 27 x 4096 x 11008
    if case["kind"] == "prefill":
        return dict(rel=6e-5, differ=0.01)                        # logits: 1.5e-5
    if case["kind"] == "score":
        # margins: 5.7e-5 over 27 rows, 4.8e-5 over 128. A margin is a difference of two logits and may
        # be small, so that its relative error says something only over several rows.
        return dict(rel=max(2.5e-4, 0.02 / case["rows"] ** 2), differ=0.01)
    # a chunk's tokens, and its actions, which are the tokens' bin centres
    return dict(rel=1e-6, differ=0.01)
