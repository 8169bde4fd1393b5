"""A sequence's rows are bit for bit the same beside a sequence whose rows are not finite."""
import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,width,nodes", [(128, 24, 1), (128, 17, 3), (128, 32, 2), (128, 40, 2), (128, 96, 1), (128, 160, 1), (64, 24, 2), (64, 16, 3)])
@pytest.mark.parametrize("ctas", [1, 1 << 20])
def test_nan_rows_stay_in_their_sequence(head_dim, width, nodes, ctas):
    from paper_2510_04147_b200 import binding as b
    w = wl.TINY.replace(d_model=192, n_kv_heads=2, head_dim=head_dim, d_ffn=160, vocab=512, prompt_len=150, block_len=width, batch=3, gen_len=256)
    poison = w.vocab - 2
    embed = wl.make_tensor(w, "embed", "cuda").clone()
    embed[poison] = float("nan")
    rng = np.random.default_rng(width)
    prompts = rng.integers(0, poison, (3, w.prompt_len)).astype(np.int32)
    ids = rng.integers(0, poison, (3, nodes, width))
    masked = np.ones(ids.shape, np.uint8)
    m = b.Ssd(b.config_from_workload(w, max_drafts=max(nodes - 1, 1), max_batch=3))
    try:
        m.set_option("attn_pipe_ctas", ctas)
        m.load_workload_weights(w)
        m.load_weights("embed", embed)
        m.prefill(prompts)
        clean = m.verify_forward(ids, masked, want_logits=True)
        ids[1] = poison
        dirty = m.verify_forward(ids, masked, want_logits=True)
    finally:
        m.destroy()
    assert np.isnan(dirty[2][1]).any()
    for x, y in zip(clean, dirty):
        assert np.array_equal(x[[0, 2]], y[[0, 2]]), "rows of one sequence reached another"
