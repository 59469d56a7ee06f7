"""Ordered sampling on the GPU: the sums of a call whose samples are taken by
buckets of their draws equal those of the same sample ids taken in id order
(calls too short to be ordered), at the switch between the two, with one and
with two partition passes, with fewer paths than buckets, with draws that span
more than 32 bits inside a bucket, and with buckets that outgrow their room."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C4 = [(0, 1), (1, 2), (2, 3), (3, 0)]
CHORD = [(0, 1), (1, 2), (2, 3), (0, 3)]
MULTI = [(0, 1), (1, 2), (1, 2), (2, 3), (3, 0), (0, 2)]
TRIANGLE = [(0, 1), (0, 2), (1, 2)]
ORDERED = 1 << 19  # kOrderedMinSamples
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def tc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08975_gb300 import _build
    _build.build()
    from paper_2409_08975_gb300 import tc as tcmod
    tcmod.lib()
    return tcmod


def graph(tc, name, scale=1):
    import torch
    from paper_2409_08975_gb300 import synth
    if name == "bursty":
        c = synth.scaled_mid(3000, 60_000, seed=21)
    elif name == "few_paths":  # a handful of edges: W far below the bucket count
        c = {"n": 5, "src": np.array([0, 1, 2, 3, 1, 0]), "dst": np.array([1, 2, 3, 0, 3, 2]), "t": np.array([1, 2, 3, 4, 3, 5])}
    else:  # "hub": few vertices, windows of thousands of edges, W above 2^41
        c = synth.dense_tiny(seed=5, n=24, m=200_000)
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)  # noqa: E731
    return tc.tc_build_temporal_csr(c["n"], dev(c["src"], torch.int32), dev(c["dst"], torch.int32),
                                    dev(c["t"].astype(np.int64) * scale, torch.int64))


def in_id_order(tc, g, mot, delta, w, k, seed, offset):
    total = dict(sum_x=0, sum_x2=0, hits=0, checked=0)
    for base in range(0, k, ORDERED - 1):
        e = tc.tc_sample_estimate(g, mot, delta, w, min(ORDERED - 1, k - base), seed, offset + base)
        for key in total:
            total[key] += e[key]
    return total


CASES = [("bursty", 1, C4, 3600, ORDERED - 1), ("bursty", 1, C4, 3600, ORDERED), ("bursty", 1, CHORD, 3600, ORDERED + 1),
         ("bursty", 1, MULTI, 86_400, 700_001), ("bursty", 1, TRIANGLE, 3600, 1_000_003),
         ("bursty", 1000, CHORD, 3_600_000, 600_011),         # 64-bit list times
         ("bursty", 1, CHORD, 3600, 4_700_003),               # two partition passes
         ("few_paths", 1, C4, 10, 600_001), ("hub", 1, C4, 1_000_000, ORDERED + 77)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%s_x%d_%d_%d" % (c[0], c[1], len(c[2]), c[4]))
def test_ordered_sums_equal_id_order(tc, case):
    name, scale, edges, delta, k = case
    g = graph(tc, name, scale)
    mot = tc.make_motif(edges)
    w = tc.tc_path_weights(g, mot, delta)
    assert w.W > 0
    if name == "hub":
        assert w.W >= 1 << 41  # beyond 2^31 draws a bucket for up to 1024 buckets
    e = tc.tc_sample_estimate(g, mot, delta, w, k, 31, 12_345)
    assert e["checked"] > 0
    assert {key: e[key] for key in ("sum_x", "sum_x2", "hits", "checked")} == in_id_order(tc, g, mot, delta, w, k, 31, 12_345)
    b = tc.Batch([(g, edges, delta, k, 31, 12_345), (g, edges, delta, 70_000, 31, 12_345)], block_size=256, tile=8192).run()
    assert all(b[0][key] == e[key] for key in ("sum_x", "sum_x2", "hits", "checked"))


CHILD = """
import sys
sys.path[:0] = [%r, %r]
import torch
from paper_2409_08975_gb300 import tc
tc.LIB_PATH = sys.argv[1]
import test_gpu_order as T
g = T.graph(tc, "bursty")
mot = tc.make_motif(T.CHORD)
w = tc.tc_path_weights(g, mot, 3600)
for k in (600_001, 4_700_003):
    e = tc.tc_sample_estimate(g, mot, 3600, w, k, 7, 3)
    assert {key: e[key] for key in ("sum_x", "sum_x2", "hits", "checked")} == T.in_id_order(tc, g, mot, 3600, w, k, 7, 3), k
    b = tc.Batch([(g, T.CHORD, 3600, k, 7, 3)], block_size=128, tile=2048).run()
    assert all(b[0][key] == e[key] for key in ("sum_x", "sum_x2", "hits", "checked")), k
print("same sums")
"""


def test_buckets_that_outgrow_their_room(tc, tmp_path):
    # a build whose buckets have room for their mean only, so that some always
    # overflow: the chunk is then taken in id order, with the same sums
    from paper_2409_08975_gb300 import _build
    obj = str(tmp_path / "tc_sample.o")
    src = os.path.join(_build.CSRC, "tc_sample.cu")
    subprocess.run([_build.nvcc()] + _build.ARCH + _build.FLAGS + ["-DTC_ORDER_SLACK=0", "-c", src, "-o", obj], check=True)
    rest = [os.path.join(_build.OBJ, f) for f in sorted(os.listdir(_build.OBJ)) if f.endswith(".o") and f != "tc_sample.o"]
    lib = str(tmp_path / "libtc_tight.so")
    subprocess.run([_build.nvcc()] + _build.ARCH + ["-shared", "-o", lib, obj] + rest + ["-cudart", "static"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD % (ROOT, os.path.join(ROOT, "tests")), lib], capture_output=True, text=True)
    assert r.returncode == 0 and "same sums" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("n,m,scale", [(6, 40, 1), (24, 900, 1), (24, 900, 1 << 33), (40, 5000, 1)])
def test_path_sum_steps_over_small_windows(tc, n, m, scale):
    # windows shorter than a warp's step, edges with fewer than 32 paths, and
    # runs that end inside an edge, against the oracle's path sum
    import torch
    import oracle
    from _graphs import small_random_graph
    s, d, t = small_random_graph(m, n, m, 10 * m, dup_frac=0.3)
    t = t * scale
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)  # noqa: E731
    g = tc.tc_build_temporal_csr(n, dev(s, torch.int32), dev(d, torch.int32), dev(t, torch.int64))
    og = oracle.build_csr(n, s, d, t)
    for edges in (C4, CHORD, MULTI, TRIANGLE):
        for delta in (20 * scale, 700 * scale):
            plan = oracle.compile_motif(edges)
            w = tc.tc_path_weights(g, tc.make_motif(edges), delta)
            e = tc.tc_exact_count(g, tc.make_motif(edges), delta, w)
            exp = oracle.path_sum(og, plan, delta)
            assert (e["sum_x"], e["sum_x2"], e["W"]) == (exp["C"], exp["sum_x2"], exp["paths"]), (edges, delta)


@pytest.mark.parametrize("name,m,delta", [("bursty", 60_000, 0), ("bursty", 60_000, 3600), ("bursty", 2047, 86_400),
                                          ("bursty", 2049, 1 << 40), ("hub", 400_000, 3000), ("hub", 400_000, 0)])
def test_features_of_32_and_64_bit_times_are_the_same(tc, name, m, delta):
    # the same graph in units a thousand times finer has times beyond 32 bits
    # and takes the other kernel; the counts, so the rows, are the same bits
    import torch
    from paper_2409_08975_gb300 import synth
    if name == "hub":  # lists of 200,000 entries on two vertices: saturated range words
        rng = np.random.default_rng(3)
        other = rng.integers(2, 5000, m)
        src, dst = np.where(rng.random(m) < 0.5, 0, other), np.where(rng.random(m) < 0.5, 1, rng.integers(2, 5000, m))
        keep = src != dst
        c = {"n": 5000, "src": src[keep], "dst": dst[keep], "t": rng.integers(0, 10_000_000, m)[keep]}
    else:
        c = synth.scaled_mid(max(100, m // 20), m, seed=m)
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)  # noqa: E731
    rows = []
    for scale in (1, 1000):
        g = tc.tc_build_temporal_csr(c["n"], dev(c["src"], torch.int32), dev(c["dst"], torch.int32),
                                     dev(c["t"].astype(np.int64) * scale, torch.int64))
        assert (g.t_max - g.t_min < 1 << 32) == (scale == 1)
        w = tc.tc_path_weights(g, tc.make_motif(CHORD, window=1), delta * scale)
        assert w.W > 0 or delta == 0
        rows.append(tc.tc_edge_features(g, tc.make_motif(CHORD, window=1), delta * scale, w).view(torch.int16))
    assert torch.equal(rows[0], rows[1])


@pytest.mark.parametrize("n,m,span", [(1, 1, 1), (2, 2, 1), (3, 4095, 5), (3, 4096, 1), (70_000, 4097, 1 << 20),
                                      (300, 40_961, (1 << 32) - 1), (5000, 9000, 1 << 32), (1 << 22, 50_000, 1 << 31)])
def test_lists_of_both_time_widths(tc, n, m, span):
    # record sorts (spans below 2^32) and pair sorts at tile edges, with one
    # vertex, one time, ties, and up to three digit passes, against the oracle
    import torch
    import oracle
    from test_gpu_parity import _check_csr
    rng = np.random.default_rng(m)
    s, d = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    t = rng.integers(0, span, m).astype(np.int64) - 7
    t[0], t[-1] = -7, span - 7  # the whole span, negative times included
    dev = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dt)  # noqa: E731
    g = tc.tc_build_temporal_csr(n, dev(s, torch.int32), dev(d, torch.int32), dev(t, torch.int64))
    _check_csr(tc, g, oracle.build_csr(n, s, d, t))


def test_chunks_of_2_30_samples(tc):
    # one call over a chunk bound against its parts, which are ordered apart
    g = graph(tc, "bursty")
    mot = tc.make_motif(C4)
    w = tc.tc_path_weights(g, mot, 3600)
    parts = [1 << 29, 1 << 29, 600_077]
    whole = tc.tc_sample_estimate(g, mot, 3600, w, sum(parts), 5, 9)
    total = dict(sum_x=0, sum_x2=0, hits=0, checked=0)
    for i, k in enumerate(parts):
        e = tc.tc_sample_estimate(g, mot, 3600, w, k, 5, 9 + sum(parts[:i]))
        for key in total:
            total[key] += e[key]
    assert {key: whole[key] for key in total} == total
