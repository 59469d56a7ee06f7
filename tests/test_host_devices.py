"""The library's host side on a fake CUDA runtime of two devices
(fake_cuda.cpp): what is set for one device is set for the next one too, and
what threads share is bounded.  Kernels do not run there; a launch is refused
as CUDA refuses it when its shared memory was not allowed on the current
device."""
import ctypes
import os
import subprocess
import threading

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
C4 = [(0, 1), (1, 2), (2, 3), (3, 0)]


def fake_library(folder):
    """The library's objects linked with the fake runtime, and its functions."""
    from paper_2409_08975_gb300 import _build, tc
    _build.build()
    obj, lib = str(folder / "fake_cuda.o"), str(folder / "libtc_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-I" + inc, "-c", os.path.join(HERE, "fake_cuda.cpp"), "-o", obj], check=True)
    objs = [os.path.join(_build.OBJ, os.path.basename(f)[:-3] + ".o") for f in sorted(os.listdir(_build.CSRC)) if f.endswith(".cu")]
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib, obj] + objs + ["-lpthread"], check=True)
    L, real = ctypes.CDLL(lib), tc.lib()
    for name in dir(real):
        if name.startswith("tc_"):
            getattr(L, name).argtypes, getattr(L, name).restype = getattr(real, name).argtypes, getattr(real, name).restype
    L.fake_launches.argtypes, L.fake_launches.restype = [ctypes.c_int, ctypes.c_char_p], ctypes.c_long
    return L


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_library(tmp_path_factory.mktemp("fake"))


def buffer(nbytes):  # 256-byte aligned "device" memory
    a = np.zeros(nbytes + 256, np.uint8)
    p = (a.ctypes.data + 255) & ~255
    return a, p


def make_graph(L, t, n=1 << 20):
    # (the fake does not run the kernel that finds the times' range: the build sees a span of 1)
    m = len(t)
    s, d, t = np.zeros(m, np.int32), np.ones(m, np.int32), np.asarray(t, np.int64)
    g = ctypes.c_void_p()
    st = L.tc_build_temporal_csr(n, m, s.ctypes.data, d.ctypes.data, t.ctypes.data, None, ctypes.byref(g))
    assert st == 0, L.tc_last_error()
    return g


def test_every_kernel_runs_on_the_second_device(fake):
    from paper_2409_08975_gb300 import tc
    L = fake
    mot = ctypes.byref(tc.make_motif(C4))
    k = 5_000_000  # two order passes
    for dev in (0, 1):
        assert L.cudaSetDevice(dev) == 0
        g = make_graph(L, [1, 2, 3])
        prefix, p = buffer(8 * 4)
        ib = ctypes.c_size_t()
        assert L.tc_sample_index_bytes(g, ctypes.byref(ib)) == 0
        index, ix = buffer(ib.value)
        W, est = ctypes.c_uint64(), tc.tc_estimate()
        assert L.tc_path_weights(g, mot, 10, None, p, ix, ctypes.byref(W), None) == 0, L.tc_last_error()
        assert L.tc_sample_estimate(g, mot, 10, p, ix, k, 1, 0, ctypes.byref(est), None) == 0, L.tc_last_error()
        mlp = ctypes.c_void_p()
        assert L.tc_mlp_create(1, ctypes.byref(mlp)) == 0, L.tc_last_error()
        feat, f = buffer(32 * 256)
        out, o = buffer(4 * 256)
        grad, gp = buffer(4 * 8192)
        loss = ctypes.c_float()
        assert L.tc_mlp_forward(mlp, f, None, 256, o, None) == 0, L.tc_last_error()
        for objective in (0, 1):
            assert L.tc_mlp_grad_ex(mlp, f, None, o, 256, objective, 0.1, gp, ctypes.byref(loss), None) == 0, L.tc_last_error()
        qb = ctypes.c_size_t()
        assert L.tc_proposal_index_bytes(g, ctypes.byref(qb)) == 0
        qindex, qx = buffer(qb.value)
        h, hp = buffer(2 * 3)
        q, qp = buffer(8 * 4)
        for kernel in (0, 1):  # k_proposal, k_mlp_umma
            L.tc_mlp_kernel(kernel)
            assert L.tc_proposal_weights(mlp, g, mot, 10, p, f, 0.1, 64, hp, qp, qx, ctypes.byref(W), None) == 0, L.tc_last_error()
        assert L.tc_sample_estimate_q(g, mot, 10, ix, hp, qp, qx, k, 1, 0, ctypes.byref(est), None, None, None) == 0, L.tc_last_error()
        assert L.tc_exact_count(g, mot, 10, p, ix, ctypes.byref(est), None) == 0, L.tc_last_error()
        for name in (b"k_rec_scatter", b"k_order_second", b"k_sample", b"k_mlp_umma", b"k_mlp_grad", b"k_proposal"):
            assert L.fake_launches(dev, name) > 0, name
        L.tc_mlp_destroy(mlp)
        L.tc_graph_destroy(g)


def test_batch_on_the_second_device(fake):
    from paper_2409_08975_gb300 import tc
    L = fake
    for dev in (0, 1):
        assert L.cudaSetDevice(dev) == 0
        g = make_graph(L, [1, 2, 3])
        for block_size in (128, 256, 512):
            q = (tc.tc_query * 1)(tc.tc_query(g, tc.make_motif(C4), 10, 5_000_000, 1, 0))
            opts = tc.tc_batch_options(block_size, 8192, 1, 0)
            b = ctypes.c_void_p()
            assert L.tc_batch_create(q, 1, ctypes.byref(opts), None, ctypes.byref(b)) == 0, L.tc_last_error()
            est = tc.tc_estimate()
            assert L.tc_batch_run(b, ctypes.byref(est), None) == 0, L.tc_last_error()
            L.tc_batch_destroy(b)
        assert L.fake_launches(dev, b"k_order_second") > 0 and L.fake_launches(dev, b"k_sample_batch") > 0
        L.tc_graph_destroy(g)


def test_read_back_buffers_are_shared_and_bounded(fake):
    from paper_2409_08975_gb300 import tc
    L = fake
    L.cudaSetDevice(0)
    g = make_graph(L, [1, 2, 3])
    mot = ctypes.byref(tc.make_motif(C4))
    prefix, p = buffer(8 * 4)
    ib = ctypes.c_size_t()
    assert L.tc_sample_index_bytes(g, ctypes.byref(ib)) == 0
    index, ix = buffer(ib.value)
    failed = []

    def call(dev=0):
        W = ctypes.c_uint64()
        if L.cudaSetDevice(dev) or L.tc_path_weights(g, mot, 10, None, p, ix, ctypes.byref(W), None):
            failed.append(L.tc_last_error())

    def threads(n, together):
        ts = [threading.Thread(target=call) for _ in range(n)]
        for t in ts:
            t.start()
            if not together:
                t.join()
        for t in ts:
            t.join()

    call()
    taken, given = L.fake_pinned_taken(), L.fake_pinned_given()
    threads(50, False)  # threads that come and go use the buffer that is there, and release none
    assert (L.fake_pinned_taken(), L.fake_pinned_given()) == (taken, given)
    threads(200, True)
    assert L.fake_pinned_taken() <= taken + 15 and L.fake_pinned_given() == given
    # a device reset takes the buffers with it (a use of one would fault here)
    taken = L.fake_pinned_taken()
    L.fake_reset()
    call()
    call(1)  # the other device's context has a buffer of its own
    assert L.fake_pinned_taken() == taken + 2
    for _ in range(20):  # more contexts than buffers: plain copies
        L.fake_reset()
        call()
    assert L.fake_pinned_taken() <= 16 and L.fake_pinned_given() == given and not failed


def test_large_calls_do_not_grow_the_pool_beyond_a_small_chunk(fake):
    from paper_2409_08975_gb300 import tc
    L = fake
    L.fake_reserved.restype, L.fake_limit.argtypes = ctypes.c_size_t, [ctypes.c_size_t]
    L.cudaSetDevice(1)
    g = make_graph(L, [1, 2, 3])
    mot, est = ctypes.byref(tc.make_motif(C4)), tc.tc_estimate()
    prefix, p = buffer(8 * 4)
    ib = ctypes.c_size_t()
    assert L.tc_sample_index_bytes(g, ctypes.byref(ib)) == 0
    index, ix = buffer(ib.value)
    k = (1 << 30) + 600_001  # a ragged last chunk

    def chunks(g, ix):
        before = L.fake_launches(1, b"k_order_first")
        status = L.tc_sample_estimate(g, mot, 10, p, ix, k, 1, 0, ctypes.byref(est), None)
        return status, L.fake_launches(1, b"k_order_first") - before

    before = L.fake_reserved()
    L.fake_limit(2 << 30)  # not even a small chunk: an error, as ever
    assert chunks(g, ix) == (2, 0)
    L.fake_limit(ctypes.c_size_t(-1).value)
    for _ in range(2):
        assert chunks(g, ix) == (0, 5)
        assert L.fake_reserved() <= before + (3 << 30)
    # on a large graph the chunks take the memory that its build has left, and no more
    for m, expected in ((120_000_000, 3), (240_000_000, 2)):
        s, t = np.zeros(m, np.int32), np.zeros(m, np.int64)
        big = ctypes.c_void_p()
        assert L.tc_build_temporal_csr(m, m, s.ctypes.data, s.ctypes.data, t.ctypes.data, None, ctypes.byref(big)) == 0
        assert L.tc_sample_index_bytes(big, ctypes.byref(ib)) == 0
        index, ix = buffer(ib.value)
        held = L.fake_reserved()
        assert chunks(big, ix) == (0, expected)
        assert L.fake_reserved() == held
        if m > 200_000_000:  # memory is short after all: smaller chunks
            L.fake_limit(held - 52 * m + (9 << 30))  # of the build's scratch, 9 GB are left
            assert chunks(big, ix) == (0, 3)
            L.fake_limit(ctypes.c_size_t(-1).value)
        L.tc_graph_destroy(big)
    L.tc_graph_destroy(g)
