"""The tcgen05 attention's parts: a cluster of one CTA for every part, one for two parts, or one CTA for all of them, by the number of
query tiles.  A node's rows have the same bits in each (the others only change how many tiles share the machine)."""
import numpy as np
import pytest

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu

BASE = wl.TINY.replace(n_layers=1, vocab=512, d_model=256, d_ffn=256, head_dim=128, weight_dtype="bf16", batch=1)


@pytest.mark.parametrize("heads,kv_heads,prompt,block,counts", [
    # four parts of 5, 4 and 33 tiles, keys ending inside a tile: one, two, four, five query tiles
    (32, 32, 512, 32, (1, 2, 8, 9, 17)), (28, 4, 345, 24, (1, 3, 7, 12, 20)), (32, 8, 4090, 64, (1, 4, 5)),
    # eight parts; two parts (more heads than a cluster of four finds room for); fewer tiles than parts
    (16, 4, 1000, 32, (1, 5, 13, 30)), (40, 8, 700, 32, (1, 8, 13)), (32, 4, 130, 32, (1, 9, 17)),
])
def test_a_nodes_rows_do_not_depend_on_how_the_parts_are_shared(heads, kv_heads, prompt, block, counts):
    from paper_2510_04147_b200 import binding
    w = BASE.replace(name=f"parts{heads}", n_heads=heads, n_kv_heads=kv_heads, prompt_len=prompt, block_len=block, gen_len=block)
    rng = np.random.default_rng(prompt)
    ids = rng.integers(0, w.vocab - 1, (1, max(counts), block))
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=max(counts) - 1))
    out = []
    try:
        ssd.load_workload_weights(w)
        ssd.prefill(wl.make_prompts(w).numpy())
        for n in counts:
            out.append([x[:, :min(counts[1], n)] for x in ssd.verify_forward(ids[:, :n], np.ones((1, n, block), bool), want_logits=True)])
    finally:
        ssd.destroy()
    for o in out:
        assert all(np.isfinite(x).all() for x in o)
        assert all(np.array_equal(x[:, :1], y[:, :1]) for x, y in zip(o, out[0]))
    for o in out[2:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, out[1]))
