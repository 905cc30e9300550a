"""A K-SVM solve on a stream that has part of the GPU's SMs: the resident grid needs all of its blocks at
once, so where they do not fit the solve takes the steps of separate kernels; the iterates are the
oracle's either way (1e-10, the FP64 form's tolerance)."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2406_18001_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Resource(C.Structure):  # CUdevResource, with room to spare
    _fields_ = [("type", C.c_int), ("rest", C.c_ubyte * 508)]


@pytest.fixture
def half_stream():
    """A stream of a green context that holds about half of the SMs."""
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    dev, ctx, st, desc = C.c_int(), C.c_void_p(), C.c_void_p(), C.c_void_p()
    assert cu.cuDeviceGet(C.byref(dev), 0) == 0
    full, part, rest = Resource(), Resource(), Resource()
    if cu.cuDeviceGetDevResource(dev, C.byref(full), 1) != 0:  # 1: SMs
        pytest.skip("no partitions on this driver")
    n = C.c_uint(1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(n), C.byref(full), C.byref(rest), 0, sms // 2) == 0
    assert cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), 1) == 0
    assert cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1) == 0  # 1: CU_GREEN_CTX_DEFAULT_STREAM
    assert cu.cuGreenCtxStreamCreate(C.byref(st), ctx, 1, 0) == 0  # 1: CU_STREAM_NON_BLOCKING
    yield st.value
    cu.cuStreamSynchronize(st)
    cu.cuStreamDestroy_v2(st)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("m,n,s", [(2000, 64, 8), (300, 16, 1)])
def test_solve_on_part_of_the_gpu(half_stream, m, n, s):
    from paper_2406_18001_gb300 import binding as B
    p = inputs.blobs(m=m, n=n, seed=m)
    H = 40 * s + (s > 1)
    A, y = torch.from_numpy(p.A).cuda(), torch.from_numpy(p.y).cuda()
    k = B.kernel("rbf", gamma=0.5 / n)
    al, al2, gr = (torch.zeros(m, dtype=torch.float64, device="cuda") for _ in range(3))
    torch.cuda.synchronize()
    _, _, info, _ = B.svm_solve(A, y, k, 1, 1.0, s, H, seed=4, prec="fp64", alpha=al, grad=gr, stream=half_stream)
    torch.cuda.synchronize()
    want = oracle.dcd_svm(p.A, p.y, oracle.kernel("rbf", gamma=0.5 / n), 1, 1.0, H, seed=4)
    assert info["iters_done"] == H
    assert np.linalg.norm(al.cpu().numpy() - want) < 1e-10 * np.linalg.norm(want)
    side = torch.cuda.Stream()
    _, _, whole, _ = B.svm_solve(A, y, k, 1, 1.0, s, H, seed=4, prec="fp64", alpha=al2, grad=gr,
                                 stream=side.cuda_stream)
    torch.cuda.synchronize()
    assert whole["gpu_launches_per_step"] == 1  # the resident grid, where the whole GPU is there
    assert np.linalg.norm(al2.cpu().numpy() - want) < 1e-10 * np.linalg.norm(want)
