"""A context's calls take no device memory after its creation: neither the first forward, nor the first one that ranks the most
probable tokens, nor the first acceptance-limit probe."""
import gc

import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_first_calls_of_a_context_allocate_nothing():
    from paper_2510_04147_b200 import binding as b
    # 512 vocabulary tiles and 640 rows: lists of 20 MB, far more than the driver's granules could hide
    w = wl.TINY.replace(vocab=65536, block_len=32, gen_len=96, batch=2)
    prompts = wl.make_prompts(w).numpy()
    rng = np.random.default_rng(5)
    ids = rng.integers(0, w.vocab - 1, (2, 4, 32))
    masked = np.ones((2, 4, 32), np.uint8)

    def calls(m):
        m.verify_forward(ids, masked)
        tok, prob = m.verify_forward_topk(ids, masked, 8)
        m.probe_acceptance_limit(32, 3, 8, 2)
        return tok, prob

    taken = []
    for _ in range(2):                 # the first context's calls make the driver load the kernels: only the second counts
        m = b.Ssd(b.config_from_workload(w, max_drafts=9, max_batch=2))
        try:
            m.load_workload_weights(w)
            m.prefill(prompts)
            gc.collect()
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            out = calls(m)
            taken.append(before - torch.cuda.mem_get_info()[0])
        finally:
            m.destroy()
        assert (out[0] >= 0).all() and np.isfinite(out[1]).all()
    assert taken[1] == 0
