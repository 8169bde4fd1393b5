"""The LM head's statistics and top-k lists in the dense kernel against the skinny one: the same bits for every row.  Vocabularies that
end inside a tile or a pair of tiles, the mask token in every place, equal logits (whose lower index wins), rows around the
dense kernel's 256-row tiles."""
import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu

BASE = wl.TINY.replace(name="lmhead", n_layers=1, d_model=328, n_heads=2, n_kv_heads=2, head_dim=128, d_ffn=128, prompt_len=40, weight_dtype="bf16")


@pytest.mark.parametrize("vocab,block,nodes", [(130, 1, 1), (257, 13, 13), (2048, 32, 8), (12801, 24, 11), (999, 37, 7), (19000, 32, 16)])
def test_dense_and_skinny_lm_head_give_the_same_bits(vocab, block, nodes):
    from paper_2510_04147_b200 import binding
    w = BASE.replace(vocab=vocab, block_len=block, gen_len=block, batch=1)
    rng = np.random.default_rng(vocab)
    ids = rng.integers(0, vocab - 1, (1, nodes, block))
    masked = np.ones(ids.shape, bool)
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=nodes - 1))
    out = []
    try:
        ssd.load_workload_weights(w)
        head = wl.make_tensor(w, "lm_head", "cuda")
        head[vocab // 2:] = head[:vocab - vocab // 2].clone()          # every logit twice, in another quarter, tile or pair
        ssd.load_weights("lm_head", head.contiguous())
        ssd.prefill(wl.make_prompts(w).numpy())
        for dense_rows in (1 << 20, 0):
            ssd.set_option("dense_rows", dense_rows)
            out.append([*ssd.verify_forward(ids, masked)[:2], *ssd.verify_forward_topk(ids, masked, 8), *ssd.verify_forward_topk(ids, masked, 3)])
    finally:
        ssd.destroy()
    assert np.isfinite(out[0][1]).all() and (out[0][0] < vocab - vocab // 2).all()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
