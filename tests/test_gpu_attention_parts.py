"""The tcgen05 attention's parts: a cluster of one CTA for every part, one for two parts, or one CTA for all of them, by the number of
query tiles, heads and sequences.  A node's rows have the same bits in each (the others only change how many tiles share the machine)."""
import numpy as np
import pytest

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu

BASE = wl.TINY.replace(n_layers=1, vocab=512, d_model=256, d_ffn=256, head_dim=128, weight_dtype="bf16", batch=1)


@pytest.mark.parametrize("heads,kv_heads,prompt,block,counts", [
    # four parts of 5, 4 and 33 tiles, keys ending inside a tile: one, two, four, five query tiles
    (32, 32, 512, 32, (1, 2, 8, 9, 17)), (28, 4, 345, 24, (1, 3, 7, 12, 20)), (32, 8, 4090, 64, (1, 4, 5)),
    # eight parts, in clusters of eight and of four; two parts (more heads than a cluster of four finds room for); fewer tiles than parts
    (8, 2, 900, 32, (1, 4, 9, 17)), (16, 4, 1000, 32, (1, 5, 13, 30)), (40, 8, 700, 32, (1, 8, 13)), (32, 4, 130, 32, (1, 9, 17)),
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


@pytest.mark.parametrize("prompt,counts", [(1024, (1, 4)), (1300, (2, 5))])
def test_a_sequences_rows_do_not_depend_on_a_second_one_from_1024_keys_on(prompt, counts):
    # 32 heads: four parts with one sequence and, from 1024 keys on, with two; 32 clusters of four CTAs, 64 pairs of more
    from paper_2510_04147_b200 import binding
    w = BASE.replace(name="parts_two", n_heads=32, n_kv_heads=8, prompt_len=prompt, block_len=32, gen_len=32, batch=2)
    rng = np.random.default_rng(prompt)
    ids = rng.integers(0, w.vocab - 1, (2, max(counts), 32))
    prompts = wl.make_prompts(w).numpy()
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=max(counts) - 1))
    try:
        ssd.load_workload_weights(w)
        for n in counts:
            out = []
            for batch in (1, 2):
                ssd.prefill(prompts[:batch])
                out.append(ssd.verify_forward(ids[:batch, :n], np.ones((batch, n, 32), bool), want_logits=True))
            assert np.isfinite(out[1][2]).all()
            assert all(np.array_equal(x[0], y[0]) for x, y in zip(*out))
    finally:
        ssd.destroy()


@pytest.mark.parametrize("form", ["chain_of_two_blocks", "hole", "window"])
def test_a_sequence_decodes_the_same_alone_and_among_others(form):
    # 8 heads, eight parts: with one sequence a CTA for each, with seven (56 pairs, still under the line for one part) fewer CTAs.
    # Finished blocks that ride in front of the next one's forward, the dual cache's hole, windows of two blocks.
    from paper_2510_04147_b200 import binding
    w = BASE.replace(name="parts_decode", n_layers=2, n_heads=8, n_kv_heads=2, prompt_len=900, block_len=24, gen_len=56, batch=7, lm_head_scale=8.0)
    prompts = wl.make_prompts(w).numpy()
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=5))
    out = []
    try:
        ssd.load_workload_weights(w)
        ssd.set_option("max_drafts", 2)
        for batch in (1, 7):
            ssd.set_option("dual_cache", 0)
            ssd.prefill(prompts[:batch])
            if form == "hole":
                ssd.set_option("dual_cache", w.prompt_len + w.gen_len)
            got = ssd.generate(binding.MODE_SSD, w.gen_len, w.block_len, batch, form == "window")
            caches = [x for l in range(w.n_layers) for x in ssd.read_cache(l, 0, w.prompt_len + (48 if form != "hole" else 0))]
            out.append([got[0][0]] + caches)
    finally:
        ssd.destroy()
    for x, y in zip(*out):
        assert np.isfinite(x).all() and np.array_equal(x, y)
