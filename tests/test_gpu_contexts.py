"""What a launch needs (a kernel's limit of dynamic shared memory, the cluster
size) belongs to a context and its device, not to the process: no flag says
"done" for every device, host threads share none, and nc_gemm_tc, which has no
context of the library, sets the limit of the variant it launches.  A second
driver context on the same GPU is given every variant."""
import ctypes as C
import re
import threading
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2602_19626_gb300" / "csrc"


def test_no_launch_state_per_process():
    """No mutable flag of a function or file outlives a context (the pool of
    status words and the cached address of the allocation-free quantiser are
    keyed by device under a mutex; the allocation budget is a test hook)."""
    for f in sorted(CSRC.glob("*.cu")) + sorted(CSRC.glob("*.cuh")):
        flags = re.findall(r"^\s*static (?:bool|int|int32_t)\s+\w+\s*=.*$", f.read_text(), re.M)
        assert not flags, (f.name, flags)


def _gemm(nc, W, X, M, N, K, bn, alloc, put, get):
    w, x, y = alloc(W.nbytes), alloc(X.nbytes), alloc(4 * M * N)
    put(w, W)
    put(x, X)
    st = nc.lib.nc_gemm_tc(w, x, None, None, 0, M, N, K, bn, y, None)
    out = np.empty((N, M), np.float32)
    get(out, y)
    return st, out


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(160, 100, 192), (5000, 1000, 72)])
def test_gemm_in_a_second_context(gpu_lib, M, N, K):
    """Every tile, 3D and 2D maps, one and two CTAs per SM: the bits of the
    first context."""
    nc = gpu_lib
    cu = C.CDLL("libcuda.so.1")
    rng = np.random.default_rng(K)
    W, X = ((rng.normal(0, 1, s).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16) for s in ((M, K), (N, K)))

    def check(r):
        assert r == 0, r

    def alloc(n):
        p = C.c_uint64(0)
        check(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(n)))
        return p.value

    def put(p, a):
        check(cu.cuMemcpyHtoD_v2(C.c_uint64(p), C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes)))

    def get(a, p):
        check(cu.cuMemcpyDtoH_v2(C.c_void_p(a.ctypes.data), C.c_uint64(p), C.c_size_t(a.nbytes)))

    import torch
    torch.zeros(1, device="cuda")                    # the primary context is current here
    first, second, errors = {}, {}, []
    for bn in (32, 64, 128, 256):
        first[bn] = _gemm(nc, W, X, M, N, K, bn, alloc, put, get)

    def other():
        ctx = C.c_void_p()
        try:
            check(cu.cuCtxCreate_v2(C.byref(ctx), C.c_uint(0), C.c_int(0)))
            for bn in (32, 64, 128, 256):
                second[bn] = _gemm(nc, W, X, M, N, K, bn, alloc, put, get)
        except Exception as e:                       # shown below, in the test's own thread
            errors.append(e)
        finally:
            if ctx:
                cu.cuCtxDestroy_v2(ctx)

    t = threading.Thread(target=other)
    t.start()
    t.join()
    assert not errors
    for bn in (32, 64, 128, 256):
        assert first[bn][0] == nc.NC_OK and second[bn][0] == nc.NC_OK, bn
        assert np.array_equal(first[bn][1], second[bn][1]), bn
