"""Options at the ends of what they accept: the value that stands for "never", and the one that brings a default back."""
import numpy as np
import pytest

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_the_largest_dense_rows_means_never():
    from paper_2510_04147_b200 import binding
    w = wl.TINY.replace(name="options", n_layers=1, vocab=512, n_heads=2, n_kv_heads=2, head_dim=128, prompt_len=40, gen_len=16)
    ids = np.arange(16, dtype=np.int32)[None, None]
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=0))
    try:
        ssd.load_workload_weights(w)
        ssd.prefill(wl.make_prompts(w).numpy())
        launches = []
        for dense_rows in (1 << 20, (1 << 30) - 1, 1 << 30, 2**31 - 1, 0):
            ssd.set_option("dense_rows", dense_rows)
            before = ssd.launch_count()
            ssd.verify_forward(ids, np.ones((1, 1, 16), np.uint8))
            launches.append(ssd.launch_count() - before)
        # (the evenly shared q|k|v projection needs no pass that finishes q, k and v)
        assert len(set(launches[:-1])) == 1 and launches[-1] < launches[0], launches
    finally:
        ssd.destroy()


def test_the_default_of_attn_pipe_ctas_can_be_set_again():
    # 64 pairs (head, sequence) over 1024 and more keys: the default keeps several parts, which a context with any lower line does not
    from paper_2510_04147_b200 import binding
    w = wl.TINY.replace(name="pipe_default", n_layers=1, vocab=512, n_heads=32, n_kv_heads=4, head_dim=128, prompt_len=1100, gen_len=16, batch=2)
    ids = np.random.default_rng(1).integers(0, w.vocab - 1, (2, 2, 16))
    ssd = binding.Ssd(binding.config_from_workload(w, max_drafts=1))
    try:
        ssd.load_workload_weights(w)
        ssd.prefill(wl.make_prompts(w).numpy())
        out = []
        for ctas in (None, 1, 64):
            if ctas:
                ssd.set_option("attn_pipe_ctas", ctas)
            out.append(ssd.verify_forward(ids, np.ones(ids.shape, np.uint8), want_logits=True)[2])
        assert not np.array_equal(out[0], out[1])
        assert np.array_equal(out[0], out[2])
        with pytest.raises(binding.SsdError):
            ssd.set_option("attn_pipe_ctas", 0)
    finally:
        ssd.destroy()
