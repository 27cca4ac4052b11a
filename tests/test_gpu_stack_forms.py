"""The forms of the fused stack's kernel on either side of their rules, for both head sizes, against the oracle: residual rows that fill
one group of four columns per worker thread and half (2048), one group of columns more (2056) and a few only (8-wide
remainders); the smallest width and row count whose ring stages hold one sub-block (512, 33 rows) and their neighbours."""
import pytest
import torch

import gen
from oracle import specasr_oracle as O
from test_gpu_parity import _check_against_oracle, _verify_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_model,head_dim,nodes", [
    (2048, 64, 9), (2056, 64, 9), (2048, 128, 3), (2056, 128, 3), (2048, 64, 50), (2056, 64, 50), (2056, 128, 50),
    (512, 64, 32), (512, 64, 33), (504, 64, 33), (1032, 128, 64),
])
def test_forms_of_the_stack_match_the_oracle(d_model, head_dim, nodes):
    from paper_2507_18181_b200.runtime import DeviceKV, DeviceModel
    cfg = gen.get_config("small", d_model=d_model, head_dim=head_dim, n_heads=4, ffn=712, vocab=1000)
    store = gen.WeightStore(cfg, 0)
    model = DeviceModel(cfg, store)
    kv = DeviceKV(model, max_tokens=200, max_nodes=64, shuffle_pages_seed=5, poison=True)
    W = O.Weights(store, cache_layers=True)
    cache = O.KVCache(cfg)
    audio = gen.audio_prefix(70, cfg.d_model, 0)
    O.prefill(cfg, W, cache, audio.astype("float64"))
    kv.prefill_embeds(torch.from_numpy(audio).cuda())
    parent = gen.sparse_tree(nodes, seed=2)
    tokens = gen.fill_tree_tokens(parent, cfg.vocab, seed=3, root_token=5)
    want = O.verify_tree(cfg, W, cache, tokens, parent)
    _check_against_oracle(_verify_gpu(cfg, kv, tokens, parent), want, tokens, parent)
