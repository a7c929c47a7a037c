"""What the allocation-free sort says of its waits: nothing in ordinary use, and
an error once, after which it works as before, when a wait of its blocks for one
another runs out (a library whose wait limit is none).  And its one cooperative
kernel on a stream that has only some of the multiprocessors."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import workloads as W  # noqa: F401  (the tests' path)

pytestmark = pytest.mark.gpu


def sort(lib, torch, k):
    d_in = torch.from_numpy(k.view(np.int64)).cuda()
    d_out, d_perm = torch.full_like(d_in, -1), torch.full((len(k),), -1, dtype=torch.int32, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.gpet_sort_times_noalloc(C.c_void_p(d_in.data_ptr()), C.c_uint64(len(k)), C.c_void_p(d_out.data_ptr()),
                                       C.c_void_p(d_perm.data_ptr()), st) == 0
    status = lib.gpet_sort_times_noalloc_status(st)
    return status, np.array_equal(d_out.cpu().numpy().view(np.uint64), np.sort(k))


def test_status(tmp_path):
    torch = pytest.importorskip("torch")
    from paper_2603_07327_gb300 import build as B
    B.build()
    import paper_2603_07327_gb300 as G
    k = np.random.default_rng(3).integers(0, 1 << 46, 100_001, dtype=np.uint64)
    assert sort(G.load(), torch, k) == (0, True)
    obj, lib = str(tmp_path / "sort_noalloc.cu.o"), str(tmp_path / "libgpet_nowait.so")
    flags = [*B.ARCH, *B.FLAGS, "-DGPET_GRID_WAIT_POLLS=0"]
    subprocess.run([B._nvcc(), *flags, "-c", os.path.join(B.CSRC, "sort_noalloc.cu"), "-o", obj], check=True)
    rest = [os.path.join(B.BUILD, os.path.basename(s) + ".o") for s in B.sources() if not s.endswith("sort_noalloc.cu")]
    subprocess.run([B._nvcc(), *B.ARCH, "-shared", "-o", lib, obj, *rest, "-lcudart"], check=True)
    nowait = C.CDLL(lib)
    nowait.gpet_last_error.restype = C.c_char_p
    status, whole = sort(nowait, torch, k)
    assert status == -4 and not whole, (status, whole)
    assert b"incomplete" in nowait.gpet_last_error()
    # told once; a sort of one block has no one to wait for
    assert sort(nowait, torch, k[:500]) == (0, True)
    assert sort(G.load(), torch, k) == (0, True)


@pytest.mark.parametrize("n", [500, 9_000, 300_007])
def test_stream_of_a_part_of_the_multiprocessors(n):
    torch = pytest.importorskip("torch")
    import paper_2603_07327_gb300 as G
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    dev, groups, parts, desc, ctx, st = C.c_int(), (C.c_ubyte * 1024)(), C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    whole, rest = (C.c_ubyte * 1024)(), (C.c_ubyte * 1024)()     # (CUdevResource has 144 bytes)
    sm, non_blocking = 1, 1
    for code in (cu.cuDeviceGet(C.byref(dev), 0), cu.cuDeviceGetDevResource(dev, whole, sm),
                 cu.cuDevSmResourceSplitByCount(groups, C.byref(parts), whole, rest, 0, 16),
                 cu.cuDevResourceGenerateDesc(C.byref(desc), groups, 1),
                 cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1),
                 cu.cuGreenCtxStreamCreate(C.byref(st), ctx, non_blocking, 0)):
        if code:
            pytest.skip(f"no stream of a green context (CUresult {code})")
    k = np.random.default_rng(n).integers(0, 1 << 46, n, dtype=np.uint64)
    d_in = torch.from_numpy(k.view(np.int64)).cuda()
    d_out = torch.full_like(d_in, -1)
    torch.cuda.synchronize()
    code = G.load().gpet_sort_times_noalloc(C.c_void_p(d_in.data_ptr()), n, C.c_void_p(d_out.data_ptr()), None, st)
    assert code == 0, G.load().gpet_last_error().decode()
    assert G.load().gpet_sort_times_noalloc_status(st) == 0
    assert np.array_equal(d_out.cpu().numpy().view(np.uint64), np.sort(k))
    assert cu.cuStreamDestroy_v2(st) == 0 and cu.cuGreenCtxDestroy(ctx) == 0
