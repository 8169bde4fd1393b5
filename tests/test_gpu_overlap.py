"""Allocation-free projections that overlap: threads with streams of their own, the first calls on the device among them, and a call
that waits behind long work while more others come and go than there are error words."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (a process of its own: the calls that set the entry point up must be the overlapping ones)
SCRIPT = """
import threading
import torch
from paper_2510_04147_b200 import binding as b, workloads as wl

shapes = [(8, 256, 256, 1), (77, 1300, 3592, 3), (33, 130, 520, 4), (129, 512, 1032, 2)]
data, out, wrong = [], {}, []
for i, (r, n, k, s) in enumerate(shapes):
    data.append((wl.normal_tensor(i, 1, (r, k), 1.0, "cuda", torch.bfloat16), wl.normal_tensor(i, 2, (n, k), 0.05, "cuda", torch.bfloat16), s))
busy = torch.randn(8192, 8192, device="cuda")
torch.cuda.synchronize()
start = threading.Barrier(len(shapes) + 1)

def worker(i, calls):
    x, w, s = data[i]
    with torch.cuda.stream(torch.cuda.Stream()):
        y = torch.full((x.shape[0], w.shape[0]), float("nan"), device="cuda")
        torch.cuda.current_stream().synchronize()
        start.wait()
        first = None
        for _ in range(calls):
            if b.gemm_bf16_noalloc(x, w, y, s) != 0:
                wrong.append(("code", i))
            got = y.clone()
            first = got if first is None else first
            if not torch.equal(got, first):
                wrong.append(("bits", i))
        out[i] = first.cpu()

def waiting():
    x, w, s = data[0]
    with torch.cuda.stream(torch.cuda.Stream()):
        y = torch.full((x.shape[0], w.shape[0]), float("nan"), device="cuda")
        start.wait()
        for _ in range(40):
            busy @ busy
        if b.gemm_bf16_noalloc(x, w, y, s) != 0:
            wrong.append(("code", "waiting"))
        out["waiting"] = y.cpu()

threads = [threading.Thread(target=worker, args=(i, 400)) for i in range(len(shapes))] + [threading.Thread(target=waiting)]
for t in threads:
    t.start()
for t in threads:
    t.join()
assert not wrong, wrong[:5]
for i, (x, w, s) in enumerate(data):
    y = torch.full((x.shape[0], w.shape[0]), float("nan"), device="cuda")
    assert b.gemm_bf16_noalloc(x, w, y, s) == 0
    assert torch.equal(out[i], y.cpu()), i
assert torch.equal(out["waiting"], out[0])
print("overlap ok")
"""


def test_overlapping_calls_give_the_serial_results():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "overlap ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
