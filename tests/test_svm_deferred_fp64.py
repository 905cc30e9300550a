"""The deferred K-SVM step on dense FP64 problems above the resident grid's range: every kernel, data that
the slices take and data that they leave to the direct block, the longest step, pieces, host buffers;
against the oracle's DCD on the same index sequence (1e-10, the FP64 form's tolerance)."""
import numpy as np
import pytest

import oracle
from paper_2406_18001_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNELS = {"rbf": dict(gamma=0.5), "poly": dict(coef0=1.0, degree=3), "linear": {}}


def B():
    from paper_2406_18001_gb300 import binding
    return binding


def data(m, n, direct, kind):
    p = inputs.blobs(m=m, n=n, seed=m)
    A = p.A / np.sqrt(n)
    if direct and kind == "rbf":
        A += 10.0  # gamma |a|^2 beyond the expansion's range
    elif direct:
        A[:, ::4] *= 1e-6  # and half of each row's magnitude in few features
        A[:, 1::4] *= 1e-6
        A[:, 2::4] *= 1e-6
    return A, p.y


@pytest.mark.parametrize("kind", ["rbf", "poly", "linear"])
@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("m,n,s,loss", [(500, 40, 64, 1), (300, 33, 128, 2), (2500, 320, 8, 2)])
def test_solve_matches_oracle(kind, direct, m, n, s, loss):
    A, y = data(m, n, direct, kind)
    H = 6 * s + 3
    st = torch.cuda.Stream()
    Ad, yd = torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        al, _, info, _ = B().svm_solve(Ad, yd, B().kernel(kind, **KERNELS[kind]), loss, 0.7, s, H, seed=6, prec="fp64")
    torch.cuda.synchronize()
    assert info["gpu_launches_per_step"] > 1  # steps of separate kernels
    want = oracle.dcd_svm(A, y, oracle.kernel(kind, **KERNELS[kind]), loss, 0.7, H, seed=6)
    assert np.linalg.norm(al.cpu().numpy() - want) < 1e-10 * np.linalg.norm(want)


@pytest.mark.parametrize("direct", [False, True])
def test_pieces_and_host_buffers_give_the_bits_of_one_call(direct):
    A, y = data(900, 48, direct, "rbf")
    k, s = B().kernel("rbf", gamma=0.5), 64
    H = 13 * s + 9
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        Ad, yd = torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda()
        ref = B().Plan(0, Ad, yd, k, 1.0, 1, s, H, seed=8, prec="fp64", loss=2)
        ref.run(-1)
        pl = B().Plan(0, Ad, yd, k, 1.0, 1, s, H, seed=8, prec="fp64", loss=2)
        assert pl.enqueue(4) == 4
        pl.run(3)
        assert pl.enqueue(2) == 2
        info, _ = pl.run(-1)
        ah, gh, _, _ = B().svm_solve(np.ascontiguousarray(A), y.copy(), k, 2, 1.0, s, H, seed=8, prec="fp64",
                                     flags=B().FLAG_HOST_IO, stream=st.cuda_stream)
        st.synchronize()
    assert info["outer_steps"] == 14 and info["gpu_launches_per_step"] > 1
    assert torch.equal(ref.alpha, pl.alpha) and torch.equal(ref.grad, pl.grad)
    assert np.array_equal(ref.alpha.cpu().numpy(), ah) and np.array_equal(ref.grad.cpu().numpy(), gh)
    ref.close()
    pl.close()
