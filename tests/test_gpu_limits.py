"""What a context accepts: the largest K split of the QKV projection, and the largest direct projection."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_qkv_splits_and_direct_projections_up_to_two_ctas_per_sm():
    from paper_2510_04147_b200 import binding as b
    # 48 tiles of q|k|v: six splits give two CTAs per SM, and 6 * 6144 floats a row are more than 16 * 2048
    w = wl.TINY.replace(n_layers=1, d_model=2048, n_heads=16, n_kv_heads=16, head_dim=128, d_ffn=256, vocab=512, prompt_len=40, gen_len=24)
    m = b.Ssd(b.config_from_workload(w, max_drafts=1, max_batch=1))
    try:
        m.load_workload_weights(w)
        prompts = wl.make_prompts(w).numpy()
        ids = np.arange(16, dtype=np.int32)[None, None]
        want = None
        for split in (1, 6):
            m.set_option("split_k_qkv", split)
            m.prefill(prompts)
            got = m.verify_forward(ids, np.ones((1, 1, 16), np.uint8), want_logits=True)[2]
            if want is not None:           # one layer in bf16: four roundings behind the sums and the LM head's input
                keep = np.arange(w.vocab) != w.mask_id
                assert np.linalg.norm((got - want)[..., keep]) < 1e-2 * np.linalg.norm(want[..., keep])
            want = got
        with pytest.raises(b.SsdError):
            m.set_option("split_k_qkv", 7)
        x = wl.normal_tensor(3, 1, (64, 64), 1.0, "cuda", torch.bfloat16)
        wt = wl.normal_tensor(3, 2, (36868, 64), 0.05, "cuda", torch.bfloat16)
        assert torch.allclose(m.gemm_bf16(x, wt[:36864]), x.float() @ wt[:36864].float().T, atol=1e-4)      # 64 rows of 6 * 6144 floats
        out = torch.empty(64, 36868, device="cuda")
        rc = m.lib.ssd_gemm_bf16(m._ctx, C.c_void_p(x.data_ptr()), C.c_void_p(wt.data_ptr()), C.c_void_p(out.data_ptr()), 64, 36868, 64, 1)
        assert rc == -5
    finally:
        m.destroy()
