"""The FP64 form's kernel block from exact slice products (tensor cores) against the FP64 oracle.

Shapes sit on the edges of the block's tiles: 128 rows, 32 columns (the step's coordinates), 64
features per k-block, n = 512 (the last one whose sums are exact) and 513 (the direct block), with
ragged rows, columns and features, and at the line in m sb n from which the form is taken.

Tolerances: iterates 1e-10 relative (the FP64 form's).  Gradient of a given alpha: every kernel
value is within a few ulp (norms and dot products rounded once, exp within about one ulp; 16 ulp =
4e-15 allowed) and a row's sum of at most 800 terms adds 800 * 2^-53 = 9e-14, both relative to
sum_j |K_ij w_j|; 1e-12 of the size of the gradient's parts covers them.
"""
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


KERNELS = {"rbf": dict(gamma=0.5), "poly": dict(degree=3, coef0=1.0), "linear": {}}


@pytest.mark.parametrize("m,n,b,s", [(300, 65, 8, 8), (385, 64, 16, 5), (128, 512, 8, 17), (129, 513, 8, 17),
                                     (257, 512, 4, 13), (640, 33, 8, 16), (511, 1, 32, 64)])
@pytest.mark.parametrize("kind", ["rbf", "poly", "linear"])
def test_krr_steps_match_oracle(m, n, b, s, kind):
    p = inputs.krr_dense(m=m, n=n, seed=m + n, dtype=np.float64)
    H = 3 * s + 1  # full steps and a short last one
    al, gr, st, _ = B().krr_solve(torch.from_numpy(p.A).cuda(), torch.from_numpy(p.y).cuda(),
                                  B().kernel(kind, **KERNELS[kind]), 1e-2, b, s, H, seed=5, prec="fp64")
    want = oracle.bdcd_krr(p.A, p.y, oracle.kernel(kind, **KERNELS[kind]), 1e-2, b, H, seed=5)
    assert rel(al.cpu().numpy(), want) < 1e-10


@pytest.mark.parametrize("m,n,s", [(385, 48, 64), (300, 100, 40), (4000, 300, 8)])
@pytest.mark.parametrize("own_stream", [False, True])
def test_svm_steps_match_oracle(m, n, s, own_stream):
    p = inputs.blobs(m=m, n=n, seed=m)
    st = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    A, y = torch.from_numpy(p.A).cuda(), torch.from_numpy(p.y).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        al, _, _, _ = B().svm_solve(A, y, B().kernel("rbf", gamma=0.5 / n), 1, 1.0, s, 6 * s + 3, seed=3, prec="fp64")
    st.synchronize()
    want = oracle.dcd_svm(p.A, p.y, oracle.kernel("rbf", gamma=0.5 / n), 1, 1.0, 6 * s + 3, seed=3)
    assert rel(al.cpu().numpy(), want) < 1e-10


@pytest.mark.parametrize("case", ["plain", "zero rows", "uneven rows", "far from the origin", "duplicates"])
def test_gradient_of_a_given_alpha(case):
    """The full pass over all columns, on data that the form takes and on data that it leaves to the
    direct block (gamma |a|^2 beyond the expansion's range)."""
    m, n, lam = 700, 70, 1e-2
    g = np.random.Generator(np.random.PCG64(7))
    A = g.standard_normal((m, n)) / np.sqrt(n)
    if case == "zero rows":
        A[::5] = 0.0
    elif case == "uneven rows":  # entries of a row over eight decades, rows over four
        A *= 10.0 ** g.uniform(-8, 0, (m, n)) * 10.0 ** g.uniform(-4, 0, (m, 1))
    elif case == "far from the origin":
        A += 10.0
    elif case == "duplicates":
        A[1::2] = A[::2]
    al0 = g.standard_normal(m)
    y = g.standard_normal(m)
    ko = oracle.kernel("rbf", gamma=0.5)
    al, gr, _, _ = B().krr_solve(torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda(), B().kernel("rbf", gamma=0.5),
                                 lam, 8, 8, 0, prec="fp64", alpha=torch.from_numpy(al0).cuda())
    want = oracle.krr_gradient(A, y, ko, lam, al0)
    K = oracle.kernel_block(ko, A, np.arange(m))
    size = np.linalg.norm(np.abs(K) @ np.abs(al0)) / lam + m * np.linalg.norm(al0) + np.linalg.norm(y)
    assert np.linalg.norm(gr.cpu().numpy() - want) < 1e-12 * size
