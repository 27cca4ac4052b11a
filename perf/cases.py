"""The work a user of this library has it do, as measurable cases.

A serving process loads a decoder once and keeps it; every utterance brings a paged cache.  One case is one pass
through the public entry points for one such situation:

  round  one verification round of one utterance: verify a draft tree, commit the accepted path
  batch  one round of several utterances in one call (with `top2`: one step of a draft model, which also wants the
         two most probable next tokens and their probabilities)
  fill   the context fill of a new utterance: audio-embedding vectors, then prompt text
  score  arg-max / accept / top-2 over a logits matrix that already exists

Rounds start by rewinding the cache to the case's length, so that a pass can be repeated on its state.
"""
import random
from types import SimpleNamespace

import torch

from paper_2507_18181_b200 import binding
from paper_2507_18181_b200.runtime import BatchVerifier, DeviceKV, DeviceModel

# name: layers, width, query heads, key/value heads, head size, feed-forward width, vocabulary
SHAPES = {
    "tiny": (2, 256, 4, 4, 64, 688, 4096),
    "0.5b": (24, 896, 14, 2, 64, 4864, 32000),
    "1b": (16, 2048, 32, 8, 64, 8192, 32000),
    "7b": (32, 4096, 32, 8, 128, 14336, 32000),
    "13b": (40, 5120, 40, 40, 128, 13824, 32000),
}


def _shape(name):
    keys = ("n_layers", "d_model", "n_heads", "n_kv_heads", "head_dim", "ffn", "vocab")
    return SimpleNamespace(name=name, eps=1e-6, rope_base=1e4, **dict(zip(keys, SHAPES[name])))


def listed():
    return [
        # the smallest decoder and context: launches and latency are all there is
        {"name": "tiny_tree15", "op": "round", "model": "tiny", "nodes": 15, "chain": False, "context": 72},
        # one autoregressive step of the draft model for eight utterances at once: what drafting consists of
        {"name": "draft_step_b8", "op": "batch", "model": "0.5b", "batch": 8, "nodes": 1, "chain": True,
         "shortest": 300, "longest": 1500, "top2": True},
        # plain speculative decoding on a small target: a chain of eight drafts under the root
        {"name": "chain9_1b", "op": "round", "model": "1b", "nodes": 9, "chain": True, "context": 782},
        # a new utterance on a small target: ragged audio prefix and prompt
        {"name": "fill_1b", "op": "fill", "model": "1b", "frames": 750, "text": 33},
        # decoding without a draft: one token on a large target
        {"name": "token_7b", "op": "round", "model": "7b", "nodes": 1, "chain": True, "context": 999},
        # a long draft on a long recording: a ragged chain near the longest cache
        {"name": "chain33_7b", "op": "round", "model": "7b", "nodes": 33, "chain": True, "context": 4063},
        # the headline workload: a sparse tree of 64 nodes on 1500 audio frames and 200 text tokens
        {"name": "tree64_7b", "op": "round", "model": "7b", "nodes": 64, "chain": False, "context": 1700},
        # the largest tree a call takes
        {"name": "tree256_7b", "op": "round", "model": "7b", "nodes": 256, "chain": False, "context": 2048},
        # the serving batch: eight utterances with 32-node trees on prefixes of different lengths
        {"name": "batch8x32_7b", "op": "batch", "model": "7b", "batch": 8, "nodes": 32, "chain": False,
         "shortest": 300, "longest": 1500, "top2": False},
        # a new utterance on a large target: half a minute of audio and the prompt
        {"name": "fill_7b", "op": "fill", "model": "7b", "frames": 1500, "text": 8},
        # the largest target, multi-head attention
        {"name": "tree64_13b", "op": "round", "model": "13b", "nodes": 64, "chain": False, "context": 1024},
        # logits computed elsewhere: accept rule for a tree and top-2 of every row
        {"name": "score64", "op": "score", "nodes": 64, "chain": False, "vocab": 32000},
    ]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    op = rng.choices(["round", "batch", "fill", "score"], [9, 5, 4, 2])[0]
    chain = rng.random() < 0.5
    if op == "round":
        model = rng.choice(["tiny", "0.5b", "1b", "7b", "7b", "13b"])
        longest = {"tiny": 1024, "13b": 2048}.get(model, 4096)
        return {"op": op, "model": model, "nodes": _between(rng, 1, 256), "chain": chain,
                "context": _between(rng, 16, longest)}
    if op == "batch":
        batch = rng.randint(2, 16)
        nodes = _between(rng, 1, min(32, 256 // batch))
        shortest = _between(rng, 50, 700)
        return {"op": op, "model": rng.choice(["0.5b", "1b", "7b"]), "batch": batch, "nodes": nodes, "chain": chain,
                "shortest": shortest, "longest": rng.randint(shortest, 1500),
                "top2": batch * nodes <= 64 and rng.random() < 0.5}
    if op == "fill":
        return {"op": op, "model": rng.choice(["0.5b", "1b", "7b"]), "frames": _between(rng, 30, 1500),
                "text": rng.randint(1, 8) if rng.random() < 0.5 else rng.randint(9, 64)}
    return {"op": op, "nodes": _between(rng, 1, 256), "chain": chain, "vocab": _between(rng, 520, 32000)}


# ---- what a program has in hand before the call ------------------------------------------------------------------
class _Weights:
    """Random-init weights, drawn on the GPU tensor by tensor: matrices 0.02 N(0,1) in bf16, gains 1 + 0.02 N(0,1)."""

    def __init__(self, cfg):
        c, q, kv = cfg, cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim
        self.shapes = {"wq": (q, c.d_model), "wk": (kv, c.d_model), "wv": (kv, c.d_model), "wo": (c.d_model, q),
                       "wg": (c.ffn, c.d_model), "wu": (c.ffn, c.d_model), "wd": (c.d_model, c.ffn),
                       "g_attn": (c.d_model,), "g_ffn": (c.d_model,), "g_final": (c.d_model,),
                       "embed": (c.vocab, c.d_model), "lm_head": (c.vocab, c.d_model)}

    def tensor(self, layer, name):
        gen = torch.Generator("cuda").manual_seed(1000 * (layer + 2) + sorted(self.shapes).index(name))
        z = torch.randn(self.shapes[name], generator=gen, device="cuda").mul_(0.02)
        if z.ndim == 1:
            return z.add_(1.0).cpu().numpy()
        return z.to(torch.bfloat16).view(torch.int16).cpu().numpy().view("uint16")


_models = {}


def _model(name):
    """The decoder a serving process has loaded; utterances come and go beside it."""
    if name not in _models:
        cfg = _shape(name)
        _models[name] = DeviceModel(cfg, _Weights(cfg), device="cuda:0")
    return _models[name]


def _tree(nodes, chain, rng):
    """Parent array: a chain, or root fan-out 4, then 2, then chains, half of whose nodes form the main trunk."""
    if chain:
        return list(range(-1, nodes - 1))
    parent = [-1] + [0] * min(4, nodes - 1)
    tops = range(1, len(parent))
    for t in tops:
        parent += [t] * max(0, min(2, nodes - len(parent)))
    ends = list(range(1 + len(tops), len(parent)))
    rest = nodes - len(parent)
    trunk = (rest + 1) // 2
    for k in range(rest):
        c = 0 if k < trunk or len(ends) < 2 else rng.randrange(1, len(ends))
        parent.append(ends[c])
        ends[c] = len(parent) - 1
    return parent


def _main_path(parent):
    path = [0]
    while path[-1] in parent[path[-1]:]:
        path.append(parent.index(path[-1]))
    return path


def _ints(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _utterance(model, context, longest, nodes, gen, max_nodes=256):
    """A cache for contexts up to `longest` that holds `context` positions: audio-embedding vectors, and text for the
    last tenth."""
    kv = DeviceKV(model, max_tokens=longest + nodes + 64, max_nodes=max_nodes)
    text = context // 10
    kv.prefill_embeds(torch.randn(context - text, model.cfg.d_model, generator=gen, device="cuda"))
    if text:
        kv.prefill_tokens(torch.randint(0, model.cfg.vocab, (text,), generator=gen, device="cuda", dtype=torch.int32))
    return kv


def _draft(model, kv, context, parent, gen):
    """Draft tokens: the main path follows the target's own greedy continuation, each position replaced by a random
    token with probability 0.2; the other nodes are random."""
    tokens = torch.randint(0, model.cfg.vocab, (len(parent),), generator=gen, device="cuda", dtype=torch.int32)
    path = _main_path(parent)[:17]
    wrong = torch.rand(len(path), generator=gen, device="cuda") < 0.2
    root = _ints([-1])
    cur = tokens[:1].clone()
    for k, node in enumerate(path[1:]):
        kv.verify(cur, root)
        kv.commit()
        cur = kv.out_argmax[:1].clone()
        tokens[node] = torch.where(wrong[k + 1], tokens[node], cur[0])
    kv.truncate(context)
    return tokens


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    rng = random.Random(seed)
    s = SimpleNamespace(op=case["op"], case=case)
    if case["op"] == "score":
        n = case["nodes"]
        s.logits = torch.randn(n, case["vocab"], generator=gen, device="cuda") * 1.3
        parent = _tree(n, case["chain"], rng)
        path = _main_path(parent)
        s.tokens = torch.randint(0, case["vocab"], (n,), generator=gen, device="cuda", dtype=torch.int32)
        right = torch.rand(n, generator=gen, device="cuda") < 0.8
        greedy = s.logits.argmax(-1).to(torch.int32)
        for a, b in zip(path, path[1:]):
            s.tokens[b] = torch.where(right[b], greedy[a], s.tokens[b])
        s.parent = _ints(parent)
        s.argmax, s.path = torch.empty_like(s.tokens), torch.empty_like(s.tokens)
        s.accept, s.bonus = _ints([0]), _ints([0])
        s.ids = torch.empty(n, 2, dtype=torch.int32, device="cuda")
        s.probs = torch.empty(n, 2, device="cuda")
        return s
    s.model = model = _model(case["model"])
    vocab = model.cfg.vocab
    if case["op"] == "fill":
        s.kv = DeviceKV(model, max_tokens=case["frames"] + case["text"] + 64)
        s.audio = torch.randn(case["frames"], model.cfg.d_model, generator=gen, device="cuda")
        s.text = torch.randint(0, vocab, (case["text"],), generator=gen, device="cuda", dtype=torch.int32)
    elif case["op"] == "round":
        n, s.context = case["nodes"], case["context"]
        s.kv = _utterance(model, s.context, s.context, max(n, 18), gen)
        parent = _tree(n, case["chain"], rng)
        s.parent = _ints(parent)
        s.tokens = _draft(model, s.kv, s.context, parent, gen)
        s.logits = torch.empty(n, vocab, device="cuda")
    else:
        b, n = case["batch"], case["nodes"]
        s.context = [rng.randint(case["shortest"], case["longest"]) for _ in range(b)]
        s.kvs = [_utterance(model, c, case["longest"], max(n, 18), gen) for c in s.context]
        parents = [_tree(n, case["chain"], rng) for _ in range(b)]
        s.parent = _ints([p for t in parents for p in t])
        s.tokens = torch.cat([_draft(model, kv, c, p, gen) for kv, c, p in zip(s.kvs, s.context, parents)])
        s.offsets = [n * i for i in range(b + 1)]
        s.bv = BatchVerifier(s.kvs)
        s.logits = None if case["top2"] else torch.empty(n * b, vocab, device="cuda")
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------
def run(s):
    if s.op == "score":
        stream = torch.cuda.current_stream().cuda_stream
        n, vocab = s.logits.shape
        binding.specasr_accept_logits_static(s.logits.data_ptr(), vocab, s.tokens.data_ptr(), s.parent.data_ptr(), n,
                                             s.argmax.data_ptr(), s.accept.data_ptr(), s.path.data_ptr(),
                                             s.bonus.data_ptr(), stream)
        binding.specasr_top2_probs(s.logits.data_ptr(), n, vocab, s.ids.data_ptr(), s.probs.data_ptr(), stream)
        return [s.argmax, s.accept, s.path, s.bonus, s.ids, s.probs]
    if s.op == "fill":
        s.kv.truncate(0)
        s.kv.prefill_embeds(s.audio)
        s.kv.prefill_tokens(s.text)
        return [s.kv.k_pool, s.kv.v_pool]
    if s.op == "round":
        kv, n = s.kv, s.tokens.shape[0]
        kv.truncate(s.context)
        kv.verify(s.tokens, s.parent, s.logits)
        kv.commit()
        return [s.logits, kv.out_argmax[:n], kv.out_accept, kv.out_path[:n], kv.out_bonus, kv.k_pool, kv.v_pool]
    bv, total = s.bv, s.tokens.shape[0]
    for kv, c in zip(s.kvs, s.context):
        kv.truncate(c)
    if s.logits is None:
        bv.verify_top2(s.tokens, s.parent, s.offsets)
        out = [bv.out_top2_ids[:total], bv.out_top2_probs[:total]]
    else:
        bv.verify(s.tokens, s.parent, s.offsets, s.logits)
        out = [s.logits]
    bv.commit()
    out += [bv.out_argmax[:total], bv.out_accept, bv.out_path[:total], bv.out_bonus]
    return out + [p for kv in s.kvs for p in (kv.k_pool, kv.v_pool)]


# ---- what a pass cannot do without -------------------------------------------------------------------------------
def work(case):
    if case["op"] == "score":
        cells = case["nodes"] * case["vocab"]
        return {"bytes": 4.0 * cells, "flops": 3.0 * cells}
    c = _shape(case["model"])
    layer = c.d_model * c.head_dim * (2 * c.n_heads + 2 * c.n_kv_heads) + 3 * c.d_model * c.ffn
    head = c.d_model * c.vocab
    slot = c.n_layers * 2 * c.n_kv_heads * c.head_dim * 4      # keys and values of one position, 4 bytes a value
    score = c.n_layers * 4 * c.n_heads * c.head_dim            # operations for one position one row looks at
    if case["op"] == "fill":
        n = case["frames"] + case["text"]
        return {"bytes": 2.0 * c.n_layers * layer + n * slot + 4 * case["frames"] * c.d_model,
                "flops": 2.0 * n * c.n_layers * layer + score * n * (n + 1) / 2}
    if case["op"] == "round":
        rows, length = [case["nodes"]], [case["context"]]
    else:
        rows = [case["nodes"]] * case["batch"]
        length = [(case["shortest"] + case["longest"]) / 2] * case["batch"]
    n = sum(rows)
    bytes_ = 2.0 * (c.n_layers * layer + head) + slot * (sum(length) + n) + 4 * n * c.vocab * (0 if case.get("top2") else 1)
    return {"bytes": bytes_, "flops": 2.0 * n * (c.n_layers * layer + head) + score * sum(r * (l + r) for r, l in zip(rows, length))}


def tolerance(case):
    """Measured between the library's two engines (up to 64 rows, and more), which add in different orders: logits agree
    to 1e-4, but the caches are compared as they are stored, in two bf16 planes (value = hi + lo), and a last-bit change
    that moves a hi value to its neighbour moves the lo value back by as much.  Largest of K and V: 1.8e-4 with 2
    layers, 3.2e-4 with 16, 5.1e-4 with 32, single entries 0.036 of the root mean square.  Four times that."""
    if case["op"] == "score":
        return {"rel": 1e-6}       # one soft-max in fp32 against fp64: 7e-8
    layers = SHAPES[case["model"]][0]
    return {"rel": 8e-4 + 4e-5 * layers, "max": 0.15, "differ": 0.01}
