"""Attention units at the edges of their ranges, against the oracle: cache lengths around multiples of 16 and 64 (chunks
and 16-key groups that end exactly, one key early, one key late), ranges of one and of many chunks, head sizes 64 and
128, pages larger than a 16-key group, up to 64 rows (fused stack) and more (separate kernel).

`sharp` multiplies the query and key weights: with the plain random-init weights scores stay within a few units, so the
running maximum never has to be raised by more than 2^8 and the rescaling of the partial output would not run.  The
score error grows with the score (about |s| 2^-16 for operands of 16 bits: 2e-3 at 100), which the logit bound covers."""
import numpy as np
import pytest
import torch

import gen
from oracle import specasr_oracle as O
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
def test_ranges_and_rescaling_match_the_oracle(cfg_name, context, nodes, page_size, sharp):
    from paper_2507_18181_b200.runtime import DeviceKV, DeviceModel
    cfg = gen.get_config(cfg_name)
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
