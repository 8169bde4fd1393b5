"""The evenly shared projections (q|k|v and gate|up of up to 256 rows) against the skinny kernel: the same K ranges in the same
order, so the bits of a forward are the same.  Row counts around the halves of a CTA pair (8-row steps, quarters of 32 rows, 128),
units that end inside a weight tile, one and two MMAs to a unit, one and four K splits, one to four units to a pair one after the
other.  (With dense_rows = 0 every projection that fits takes this kernel, whether that is faster or not; test_routes.py has the
units of these widths.)"""
import numpy as np
import pytest

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu

BASE = wl.TINY.replace(n_layers=2, vocab=512, head_dim=128, weight_dtype="bf16")
SHAPES = {
    # units of 16 couples (the least), most of the last ones missing; K ends inside a K block
    "narrow": BASE.replace(name="even_narrow", d_model=328, n_heads=4, n_kv_heads=2, d_ffn=200),
    # four K splits with accumulators of their own; units of 136 and of 256 couples (two MMAs)
    "splits": BASE.replace(name="even_splits", d_model=1024, n_heads=28, n_kv_heads=4, d_ffn=9664),
    "wide": BASE.replace(name="even_wide", d_model=512, n_heads=32, n_kv_heads=32, d_ffn=18944),
    # two units to a pair and one accumulator: of 136 couples over a single K block (each of the two producer warps has every
    # second unit to itself), of 200 over three and of 256 over five, more than the ring has stages
    "two_turns": BASE.replace(name="even_two_turns", n_layers=1, d_model=64, n_heads=2, n_kv_heads=1, d_ffn=19456),
    "two_turns_3": BASE.replace(name="even_two_turns_3", n_layers=1, d_model=184, n_heads=2, n_kv_heads=1, d_ffn=28672),
    "two_turns_5": BASE.replace(name="even_two_turns_5", n_layers=1, d_model=320, n_heads=2, n_kv_heads=1, d_ffn=37888),
    # four units to a pair, the last ones missing
    "four_turns": BASE.replace(name="even_four_turns", n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=60008),
}


@pytest.mark.parametrize("shape,prompt,block,nodes", [
    ("narrow", 5, 1, 1), ("narrow", 33, 13, 1), ("narrow", 250, 13, 13), ("narrow", 256, 24, 9),
    ("splits", 17, 16, 1), ("splits", 255, 23, 11), ("splits", 161, 32, 8),
    ("wide", 9, 9, 2), ("wide", 129, 24, 7), ("wide", 256, 16, 16),
    ("two_turns", 7, 3, 1), ("two_turns", 161, 32, 8), ("two_turns_3", 200, 23, 11), ("two_turns_5", 256, 32, 5), ("four_turns", 33, 32, 7),
])
def test_even_and_skinny_projections_give_the_same_bits(shape, prompt, block, nodes):
    from paper_2510_04147_b200 import binding
    w = SHAPES[shape].replace(prompt_len=prompt, batch=1, block_len=block, gen_len=block)
    prompts = wl.make_prompts(w).numpy()
    rng = np.random.default_rng(prompt)
    ids = rng.integers(0, w.vocab - 1, (1, nodes, block))
    masked = np.ones(ids.shape, bool)
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=nodes - 1))
    out = []
    try:
        ssd.load_workload_weights(w)
        for dense_rows in (1 << 20, 0):          # (0: every forward of up to 256 rows)
            ssd.set_option("dense_rows", dense_rows)
            ssd.prefill(prompts)
            caches = [x for l in range(w.n_layers) for x in ssd.read_cache(l, 0, prompt)]
            out.append(caches + [x for x in ssd.verify_forward(ids, masked, want_logits=True)])
    finally:
        ssd.destroy()
    assert all(np.isfinite(x).all() for x in out[0])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
