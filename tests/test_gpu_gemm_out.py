"""Where the two projection calls write: a caller's output may begin at any float, rows may be of any length.  Every store form
(vectors, single floats; one K range, several summed in a cluster) gives the same bits and touches nothing beside the output."""
import ctypes as C

import pytest
import torch

from paper_2510_04147_b200 import workloads as wl

pytestmark = pytest.mark.gpu

GUARD = 8                                  # floats on either side that must stay as they are


def _call(b, ssd, entry, x, w, split, offset):
    """The output of one call into a buffer at `offset` floats past a 16-byte boundary, and whether the guards held."""
    rows, n = x.shape[0], w.shape[0]
    buf = torch.full((GUARD + 3 + rows * n + GUARD,), 7.5, device="cuda")
    assert buf.data_ptr() % 16 == 0
    first = GUARD + offset
    out = C.c_void_p(buf.data_ptr() + 4 * first)
    px, pw = C.c_void_p(x.data_ptr()), C.c_void_p(w.data_ptr())
    torch.cuda.synchronize()
    if entry == "context":
        rc = ssd.lib.ssd_gemm_bf16(ssd._ctx, px, pw, out, rows, n, x.shape[1], split)
    else:
        rc = ssd.lib.ssd_gemm_bf16_noalloc(px, pw, out, rows, n, x.shape[1], split, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == b.SSD_OK
    host = buf.cpu()
    assert (host[:first] == 7.5).all() and (host[first + rows * n:] == 7.5).all(), "a store beside the output"
    return host[first:first + rows * n].view(rows, n)


@pytest.mark.parametrize("rows,n,k", [(5, 256, 256), (17, 300, 520), (33, 130, 264), (40, 129, 328), (270, 134, 200)])
@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("entry", ["context", "noalloc"])
def test_output_may_begin_at_any_float(rows, n, k, split, entry):
    from paper_2510_04147_b200 import binding as b
    x = wl.normal_tensor(31, 1, (rows, k), 1.0, "cuda", torch.bfloat16)
    w = wl.normal_tensor(31, 2, (n, k), 0.05, "cuda", torch.bfloat16)
    ssd = b.Ssd(b.config_from_workload(wl.TINY, max_drafts=1, max_batch=2))
    try:
        aligned = _call(b, ssd, entry, x, w, split, 0)
        for offset in (1, 2, 3):
            assert torch.equal(_call(b, ssd, entry, x, w, split, offset), aligned), offset
    finally:
        ssd.destroy()
    ref = x.cpu().double() @ w.cpu().double().T
    # fp32 sums of k products: k * 2^-24 of the sum of magnitudes, itself about 0.04 * k
    assert (aligned.double() - ref).abs().max() < 2 * k * 2.0 ** -24 * 0.04 * k + 1e-6
