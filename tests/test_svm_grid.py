"""Resident K-SVM steps (small dense FP64 problems: many outer steps per launch) against the oracle's
DCD on the same index stream, at the shapes where the split over CTAs, warps and lanes turns: one
row, fewer rows than a CTA takes, a last CTA with one row; one coordinate a step, more than one
warp's, the most the recurrence takes; one feature, odd ones; repeats within and across steps; more
steps than a launch holds.  Iterates 1e-10 relative (the FP64 form's tolerance)."""
import numpy as np
import pytest

import oracle
from paper_2406_18001_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def B():
    from paper_2406_18001_gb300 import binding
    return binding


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("m,n,s,H", [(1, 3, 1, 5), (5, 1, 4, 41), (33, 16, 1, 90), (300, 16, 1, 256), (257, 7, 8, 400),
                                     (2000, 64, 8, 800), (120, 40, 33, 33 * 7 + 2), (90, 20, 64, 64 * 6),
                                     (40, 9, 128, 128 * 5 + 1), (30, 5, 1, 9000)])
@pytest.mark.parametrize("loss", [1, 2])
@pytest.mark.parametrize("own_stream", [False, True])
def test_solve_matches_oracle(m, n, s, H, loss, own_stream):
    p = inputs.blobs(m=max(m, 2), n=n, seed=m)
    A, y = p.A[:m].copy(), p.y[:m].copy()
    st = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    Ad, yd = torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        al, gr, info, _ = B().svm_solve(Ad, yd, B().kernel("rbf", gamma=0.5 / n), loss, 0.8, s, H, seed=3, prec="fp64")
    st.synchronize()
    ko = oracle.kernel("rbf", gamma=0.5 / n)
    want = oracle.dcd_svm(A, y, ko, loss, 0.8, H, seed=3)
    assert info["iters_done"] == H and info["outer_steps"] == -(-H // s)
    assert rel(al.cpu().numpy(), want) < 1e-10
    gw = oracle.svm_gradient(A, y, ko, loss, 0.8, want)
    assert np.max(np.abs(gr.cpu().numpy() - gw)) < 1e-10 * max(1.0, np.max(np.abs(gw)))


@pytest.mark.parametrize("kind,kw", [("rbf", dict(gamma=0.5)), ("poly", dict(coef0=1.0, degree=3)), ("linear", {})])
@pytest.mark.parametrize("shift", [0.0, 10.0])
def test_kernels_and_data_away_from_the_origin(kind, kw, shift):
    """shift: gamma |a|^2 beyond the expansion's range, so that distances come from differences."""
    p = inputs.blobs(m=250, n=20, seed=4)
    A = p.A / np.sqrt(20.0) + shift / np.sqrt(20.0)
    al, _, _, _ = B().svm_solve(torch.from_numpy(A).cuda(), torch.from_numpy(p.y).cuda(), B().kernel(kind, **kw), 2, 0.7,
                                16, 16 * 20 + 3, seed=9, prec="fp64")
    want = oracle.dcd_svm(A, p.y, oracle.kernel(kind, **kw), 2, 0.7, 16 * 20 + 3, seed=9)
    assert rel(al.cpu().numpy(), want) < 1e-10


def test_pieces_give_the_bits_of_one_call():
    p = inputs.blobs(m=400, n=30, seed=2)
    k = B().kernel("rbf", gamma=0.05)
    A, y = torch.from_numpy(p.A).cuda(), torch.from_numpy(p.y).cuda()
    ref = B().Plan(0, A, y, k, 1.0, 1, 8, 8 * 50 + 5, seed=1, prec="fp64")
    ref.run(-1)
    pl = B().Plan(0, A, y, k, 1.0, 1, 8, 8 * 50 + 5, seed=1, prec="fp64")
    assert pl.enqueue(7) == 7
    pl.run(1)
    pl.run(-1)
    assert torch.equal(ref.alpha, pl.alpha) and torch.equal(ref.grad, pl.grad)
    ref.close()
    pl.close()
