"""The orders that the sampler takes: every sample once, and no bucket beyond
its room; and in a build whose buckets have room
for their mean only, the overflow word that sends a chunk into id order."""
import ctypes
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COUNTS = (65_536, 600_001, 4_062_208, 4_700_003)  # one partition pass and two, at the switch


class OrderView(ctypes.Structure):
    _fields_ = [("head", ctypes.c_void_p), ("sizes", ctypes.c_void_p), ("ids", ctypes.c_void_p),
                ("nb", ctypes.c_uint32), ("room", ctypes.c_uint32)]


def order(L, count, wave):
    """(overflow word, bucket sizes, ids by bucket) of samples 9 .. 9 + count."""
    import torch
    u64, u32, vp = ctypes.c_uint64, ctypes.c_uint32, ctypes.c_void_p
    nbytes, nscratch, view, run = (L._ZN2tc11order_bytesEmj, L._ZN2tc19order_scratch_bytesEmj, L._ZN2tc10order_viewEmjPv,
                                   L._ZN2tc13order_samplesEmmmjPvS0_P11CUstream_st)
    nbytes.argtypes = nscratch.argtypes = [u64, u32]
    nbytes.restype = nscratch.restype = ctypes.c_size_t
    view.argtypes, view.restype = [u64, u32, vp], OrderView
    run.argtypes = [u64, u64, u64, u32, vp, vp, vp]
    out = torch.zeros(nbytes(count, wave), dtype=torch.uint8, device="cuda")
    scratch = torch.zeros(max(nscratch(count, wave), 1), dtype=torch.uint8, device="cuda")
    assert run(7, 9, count, wave, scratch.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    v, words = view(count, wave, out.data_ptr()), out.view(torch.int32)
    at = lambda p, n: words[(p - out.data_ptr()) // 4:][:n]  # noqa: E731
    return int(at(v.head, 1)[0]), at(v.sizes, v.nb), at(v.ids, v.nb * v.room).view(v.nb, v.room)


def test_every_sample_is_in_one_bucket():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08975_gb300 import _build, tc
    _build.build()
    L = ctypes.CDLL(tc.LIB_PATH)
    for count in COUNTS:
        for wave in (1, 456):
            over, sizes, ids = order(L, count, wave)
            nb, room = ids.shape
            assert over == 0 and int(sizes.max()) <= room and int(sizes.sum()) == count, (count, wave)
            taken = ids[torch.arange(room, device="cuda")[None, :] < sizes[:, None]]
            assert torch.equal(taken.sort().values, torch.arange(count, dtype=torch.int32, device="cuda")), (count, wave)


CHILD = """
import ctypes, sys
sys.path[:0] = [%r, %r]
import test_gpu_order_rooms as T
L = ctypes.CDLL(sys.argv[1])
for count in T.COUNTS:
    over, sizes, ids = T.order(L, count, 1)
    assert over == 1 and int(sizes.max()) > ids.shape[1], count
print("overflowed")
"""


def test_a_full_bucket_sets_the_overflow_word(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08975_gb300 import _build
    _build.build()
    obj, lib = str(tmp_path / "tc_sample.o"), str(tmp_path / "libtc_tight.so")
    subprocess.run([_build.nvcc()] + _build.ARCH + _build.FLAGS + ["-DTC_ORDER_SLACK=0", "-c", os.path.join(_build.CSRC, "tc_sample.cu"),
                    "-o", obj], check=True)
    rest = [os.path.join(_build.OBJ, f) for f in sorted(os.listdir(_build.OBJ)) if f.endswith(".o") and f != "tc_sample.o"]
    subprocess.run([_build.nvcc()] + _build.ARCH + ["-shared", "-o", lib, obj] + rest + ["-cudart", "static"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD % (ROOT, os.path.join(ROOT, "tests")), lib], capture_output=True, text=True)
    assert r.returncode == 0 and "overflowed" in r.stdout, r.stdout + r.stderr
