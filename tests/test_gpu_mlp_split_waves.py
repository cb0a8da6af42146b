"""K splits that would take nearly every SM: whole clusters have to find room in a GPC,
so such a split can need a second wave of them, and fewer rows of an MLP then take
longer than more rows do (1024 rows of 768 x 3072: 38.9 us, 1280 rows: 29.6)."""
import os
import statistics
import subprocess
import sys

import pytest
import torch

from paper_2609_13141_gb300 import sas, synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _us(layer, x, w1, w2):
    for _ in range(10):
        layer.mlp(x, w1, w2)
    times = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            layer.mlp(x, w1, w2)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 50)
    return statistics.median(times)


@pytest.mark.parametrize("rows,more,D,F", [(1024, 1280, 768, 3072)])
def test_fewer_rows_take_no_longer(rows, more, D, F):
    X, W1, W2, _, _ = (None if t is None else t.cuda() for t in synth.mlp(more, D, F, seed=2))
    layer = sas.SasLayer(1, 1, 64, 64, 0)
    t_more, t_rows = _us(layer, X, W1, W2), _us(layer, X[:rows].contiguous(), W1, W2)
    layer.close()
    assert t_rows <= 1.15 * t_more, (t_rows, t_more)


FIRST = """
import torch
from paper_2609_13141_gb300 import sas, synth
T, D, F = 130, 1088, 4352
X, W1, W2, _, _ = (None if t is None else t.cuda() for t in synth.mlp(T, D, F, seed=3))
Y, Z = torch.zeros_like(X), torch.zeros_like(X)
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    sas.sas_mlp_fwd_noalloc(X, W1, W2, Y)
graph.replay()
sas.sas_mlp_fwd_noalloc(X, W1, W2, Z)
torch.cuda.synchronize()
assert sas.sas_mlp_noalloc_get_device_status() == 0
assert torch.equal(Y, Z) and float(Y.float().abs().max()) > 0
print("captured")
"""


def test_first_call_of_a_process_under_capture():
    r = subprocess.run([sys.executable, "-c", FIRST], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr
