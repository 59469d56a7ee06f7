"""Calls of more samples than one small chunk: what they leave in the library's
pool, and the same sums in small chunks and in large ones."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
sys.path[:0] = [%r, %r]
import torch
from paper_2409_08975_gb300 import tc
import test_gpu_order as T
mot = tc.make_motif(T.C4)
parts = [1 << 27] * 8 + [600_077]  # each below a small chunk

def call(g, w):
    free, launches = torch.cuda.mem_get_info()[0], tc.tc_kernel_launches()
    whole = tc.tc_sample_estimate(g, mot, 3600, w, sum(parts), 5, 9)
    launches = tc.tc_kernel_launches() - launches
    free -= torch.cuda.mem_get_info()[0]
    total = dict(sum_x=0, sum_x2=0, hits=0, checked=0)
    for i, k in enumerate(parts):
        e = tc.tc_sample_estimate(g, mot, 3600, w, k, 5, 9 + sum(parts[:i]))
        for key in total:
            total[key] += e[key]
    assert {key: whole[key] for key in total} == total
    return free, launches

# a small graph: four small chunks (two order passes and a sampler each) and the rest (one pass)
g = T.graph(tc, "bursty")
w = tc.tc_path_weights(g, mot, 3600)
taken, launches = call(g, w)
assert taken <= 3 << 30 and launches == 4 * 3 + 2, (taken, launches)
# a large graph: larger chunks in the memory that its build has left
m = 120_000_000
torch.manual_seed(1)
src = torch.randint(0, 1 << 20, (m,), dtype=torch.int32, device="cuda")
dst = torch.randint(0, 1 << 20, (m,), dtype=torch.int32, device="cuda")
t = torch.randint(0, 1 << 20, (m,), dtype=torch.int64, device="cuda")
g = tc.tc_build_temporal_csr(1 << 20, src, dst, t)
w = tc.tc_path_weights(g, mot, 3600)
assert w.W > 1 << 24
taken, launches = call(g, w)
assert taken <= 1 << 26 and launches == 2 * 3 + 2, (taken, launches)
print("same sums")
"""


def test_large_calls_leave_no_more_in_the_pool_than_a_small_chunk_or_the_build():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CHILD % (ROOT, os.path.join(ROOT, "tests"))], capture_output=True, text=True)
    assert r.returncode == 0 and "same sums" in r.stdout, r.stdout + r.stderr
