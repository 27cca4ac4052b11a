"""Attention units at the edges of their ranges, against the oracle: cache lengths around multiples of 16 and 64 (chunks
and 16-key groups that end exactly, one key early, one key late), ranges of one and of up to 17 chunks, CTAs that run one
and several units, head sizes 64 and 128, pages larger than a 16-key group, up to 64 rows (fused stack) and more (separate
kernel), and a cache longer than the rest of the tests use.

`sharp` multiplies the query and key weights: with the plain random-init weights scores stay within a few units, so the
running maximum never has to be raised by more than 2^8 and the rescaling of the partial output would not run.  The
score error grows with the score (about |s| 2^-16 for operands of 16 bits: 2e-3 at 100), which the logit bound covers."""
import numpy as np
import pytest
import torch

import gen
from oracle import specasr_oracle as O
from test_gpu_batch import _run_batch
from test_gpu_parity import _check_against_oracle, _verify_gpu

pytestmark = pytest.mark.gpu


class _SharpStore(gen.WeightStore):
    """The seeded weights with wq and wk multiplied by a power of two (exact in bf16)."""

    def __init__(self, cfg, seed, factor):
        super().__init__(cfg, seed)
        self.factor = np.float32(factor)

    def _draw(self, layer, name):
        z = super()._draw(layer, name)
        if name in ("wq", "wk"):
            z = z * self.factor
        return z


@pytest.mark.parametrize("cfg_name,context,nodes,page_size,sharp", [
    ("small", 15, 1, 16, 1), ("small", 47, 17, 16, 1), ("small", 63, 2, 16, 1), ("small", 112, 16, 16, 1),
    ("tiny", 49, 15, 16, 1), ("tiny", 191, 64, 16, 1), ("tiny", 130, 63, 48, 1), ("small", 320, 70, 80, 1),
    ("small", 100, 33, 16, 1), ("tiny", 100, 48, 16, 1), ("small", 100, 49, 16, 1),      # row padding 32 | 48 | 64
    ("tiny", 400, 40, 16, 8), ("small", 400, 40, 16, 8), ("small", 700, 130, 16, 8), ("tiny", 701, 256, 16, 8),
])
def test_ranges_and_rescaling_match_the_oracle(cfg_name, context, nodes, page_size, sharp, heads=None):
    from paper_2507_18181_b200.runtime import DeviceKV, DeviceModel
    cfg = gen.get_config(cfg_name, **({"n_heads": heads, "n_kv_heads": heads} if heads else {}))
    store = _SharpStore(cfg, 0, sharp) if sharp != 1 else gen.WeightStore(cfg, 0)
    model = DeviceModel(cfg, store, page_size=page_size)
    kv = DeviceKV(model, max_tokens=context + nodes + 8, max_nodes=256, shuffle_pages_seed=5, poison=True)
    W = O.Weights(store, cache_layers=True)
    cache = O.KVCache(cfg)
    audio = gen.audio_prefix(context, cfg.d_model, 0)
    O.prefill(cfg, W, cache, audio.astype(np.float64))
    kv.prefill_embeds(torch.from_numpy(audio).cuda())
    parent = gen.sparse_tree(nodes, seed=2) if nodes > 2 else gen.chain_tree(nodes - 1)
    tokens = gen.fill_tree_tokens(parent, cfg.vocab, seed=3, root_token=5)
    want = O.verify_tree(cfg, W, cache, tokens, parent)
    _check_against_oracle(_verify_gpu(cfg, kv, tokens, parent), want, tokens, parent)


@pytest.mark.parametrize("heads,context,nodes,sharp", [
    (64, 400, 40, 8),         # fused stack, ranges of 4 chunks: the partial output is rescaled in the middle of a range
    (74, 900, 40, 1),         # ranges of 8 chunks, one unit on each of 148 CTAs
    (64, 900, 130, 8),        # separate kernel, one range of 17 chunks
    (100, 300, 256, 8),       # 200 units of 9 chunks: CTAs run a second unit behind the first
])
def test_ranges_of_many_chunks(heads, context, nodes, sharp):
    """As many KV heads as it takes to fill the GPU with few ranges per row, so that the ranges are long."""
    test_ranges_and_rescaling_match_the_oracle("tiny", context, nodes, 16, sharp, heads)


@pytest.mark.parametrize("nodes", [2, 4])
def test_ctas_with_several_units_of_different_lengths(nodes):
    """Twenty utterances with caches of 20 to 723 positions and eight KV heads: 296 units of one to five chunks, two per
    CTA, in the fused stack (40 rows) and in the separate kernel (80)."""
    from paper_2507_18181_b200.runtime import BatchVerifier, DeviceKV, DeviceModel
    cfg = gen.get_config("small", n_kv_heads=8, vocab=1000)
    store = gen.WeightStore(cfg, 0)
    model = DeviceModel(cfg, store)
    W = O.Weights(store, cache_layers=True)
    kvs, caches, trees = [], [], []
    for b in range(20):
        audio = gen.audio_prefix(20 + 37 * b, cfg.d_model, 0, utterance=b)
        kv = DeviceKV(model, max_tokens=800, max_nodes=128 if b == 0 else 16, shuffle_pages_seed=b)
        kv.prefill_embeds(torch.from_numpy(audio).cuda())
        cache = O.KVCache(cfg)
        O.prefill(cfg, W, cache, audio.astype(np.float64))
        parent = gen.chain_tree(nodes - 1)
        kvs.append(kv); caches.append(cache)
        trees.append((gen.fill_tree_tokens(parent, cfg.vocab, seed=b, root_token=3 + b), parent))
    for got, cache, (tokens, parent) in zip(_run_batch(BatchVerifier(kvs), trees, cfg.vocab), caches, trees):
        _check_against_oracle(got, O.verify_tree(cfg, W, cache, tokens, parent), tokens, parent)
    assert all(kv.status() == 0 for kv in kvs)


@pytest.mark.parametrize("nodes", [15, 70])
def test_cache_of_nine_thousand_positions(nodes):
    """The capacity is what the pages hold and the rotary table reaches; the oracle continues from the device's own cache
    (read back: hi + lo is what both sides see)."""
    from paper_2507_18181_b200.runtime import DeviceKV, DeviceModel
    cfg = gen.get_config("tiny")
    store = gen.WeightStore(cfg, 0)
    model = DeviceModel(cfg, store, max_positions=9100)
    kv = DeviceKV(model, max_tokens=9100, max_nodes=256, shuffle_pages_seed=1, poison=True)
    kv.prefill_embeds(torch.from_numpy(gen.audio_prefix(9000, cfg.d_model, 0)).cuda())
    cache = O.KVCache(cfg)
    for layer in range(cfg.n_layers):
        cache.K[layer], cache.V[layer] = kv.read_kv(layer, 9000)
    parent = gen.sparse_tree(nodes, seed=2)
    tokens = gen.fill_tree_tokens(parent, cfg.vocab, seed=3, root_token=5)
    want = O.verify_tree(cfg, O.Weights(store, cache_layers=True), cache, tokens, parent)
    _check_against_oracle(_verify_gpu(cfg, kv, tokens, parent), want, tokens, parent)
