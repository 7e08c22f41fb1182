"""Handles driven from several host threads at once, each on a stream of its own: the first launches of a kernel on a
device (which set its attributes) may then come from any of them.  Every thread must end with the weights that the
same calls give one after the other, bit for bit (all sums are taken in a fixed order)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# In a process of its own, so that the threads make the process's first launches.
CHILD = r"""
import threading
import torch
import paper_2602_03515_b200 as br
from workloads import LayerSpec
from workloads.configs import GEOM_BI, SRC_SECOND

SETS = [([(64, 32)], "f32"), ([(9, 70)] * 3, "f32"), ([(130, 97), (33, 40)], "f32"), ([(128, 136), (72, 264)], "bf16")]
torch.manual_seed(0)
inputs = []
for shapes, grad in SETS:
    dt = torch.bfloat16 if grad == "bf16" else torch.float32
    inputs.append(([0.02 * torch.randn(m, n, device="cuda") for m, n in shapes],
                   [[(0.01 * torch.randn(m, n, device="cuda")).to(dt) for m, n in shapes] for _ in range(3)]))
torch.cuda.synchronize()

def train(i, start, out):
    shapes, grad = SETS[i]
    stream = torch.cuda.Stream()
    if start is not None:
        start.wait()
    with torch.cuda.stream(stream):
        weights = [w.clone() for w in inputs[i][0]]
        specs = [LayerSpec("w", m, n, GEOM_BI, SRC_SECOND, 1) for m, n in shapes]
        opt = br.BasisRotation(specs, weights, grad_dtype=grad, freq=3, stream=stream, use_torch_allocator=False,
                               gemm_prec=br.BR_GEMM_BF16 if grad == "bf16" else br.BR_GEMM_FP32)
        for c in range(8):
            opt.step(inputs[i][1][c % 3])
        opt.sync_status()
        opt.close()
    stream.synchronize()
    out[i] = weights

together = {}
start = threading.Barrier(len(SETS))
threads = [threading.Thread(target=train, args=(i, start, together)) for i in range(len(SETS))]
[t.start() for t in threads]
[t.join() for t in threads]
one_by_one = {}
for i in range(len(SETS)):
    train(i, None, one_by_one)
for i in range(len(SETS)):
    for a, b in zip(together[i], one_by_one[i]):
        assert torch.isfinite(a).all() and torch.equal(a, b), i
"""


def test_handles_of_several_threads():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]
