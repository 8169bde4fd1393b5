"""A call that fails half way leaves forwards in flight; what goes wrong in them is not reported by the next call."""
import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_error_words_of_a_failed_call_are_not_the_next_calls():
    from paper_2510_04147_b200 import binding as b
    # enough layers that the first forward still runs when the next call begins
    w = wl.TINY.replace(n_layers=24, block_len=32)
    prompts = wl.make_prompts(w).numpy()
    m = b.Ssd(b.config_from_workload(w, max_drafts=3))
    try:
        m.load_workload_weights(w)
        m.load_weights("lm_head", torch.full((w.vocab, w.d_model), float("nan"), device="cuda"))
        m.set_option("mix_order", 1)               # six nodes for three drafts: more than the context was created for
        for _ in range(3):
            m.prefill(prompts)
            with pytest.raises(b.SsdError, match="nodes"):
                m.decode_block(b.MODE_SSD, 32, 1)  # its first forward (one node, NaN confidences) is enqueued, the second refused
            m.prefill(prompts)                     # reads no confidence
        m.set_option("mix_order", 0)
        with pytest.raises(b.SsdError, match="non-finite"):
            m.decode_block(b.MODE_SSD, 32, 1)
        m.load_weights("lm_head", wl.make_tensor(w, "lm_head", "cuda"))
        m.prefill(prompts)
        assert (m.decode_block(b.MODE_SSD, 32, 1)[0] >= 0).all() and np.isfinite(m.cache_length())
    finally:
        m.destroy()
