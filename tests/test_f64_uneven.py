"""The FP64 form where its slices would cost digits: the results stay those of FP64 sums.

The slices hold a value relative to its row's largest magnitude, so a dot product made of features that
are tiny beside others loses digits; such data belong to the direct block.  Compared row by row, with
sum_j sum_k |a_ik a_jk| (the polynomial's power of it) as the size of what is summed: an FP64 sum of n
products, d powers and m terms is within d (n + m + 16) 2^-53 of that size, and so is the oracle's,
together twice as much.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNELS = {"linear": {}, "poly": dict(degree=3, coef0=1.0), "rbf": dict(gamma=0.5)}


def B():
    from paper_2406_18001_gb300 import binding
    return binding


def gradient(A, al0, y, kind, kw, lam):
    """The gradient of a given alpha: full passes of the block that a step of 64 coordinates takes."""
    _, g, _, _ = B().krr_solve(torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda(), B().kernel(kind, **kw), lam, 8, 8,
                               0, prec="fp64", alpha=torch.from_numpy(al0).cuda())
    return g.cpu().numpy()


def data(case, m, n, g):
    A = g.standard_normal((m, n)) / 8
    if case.startswith("large"):  # one feature of size F in every second row, 0 in the others
        A[:, 5] = 0.0
        A[::2, 5] = float(case.split()[1])
    elif case == "disjoint":  # large features of one row meet small ones of the other
        A *= 1e-7
        A[::2, :n // 2] *= 1e7
        A[1::2, n // 2:] *= 1e7
    elif case == "decades":
        A *= 10.0 ** g.uniform(-12, 0, (m, n))
    elif case == "whole numbers":  # exact in the slices whatever their sizes
        A = np.rint(A * 3) * (g.random((m, n)) < 0.3)
        A[::2, 5] = 2.0 ** 26 - 1
    return A


@pytest.mark.parametrize("kind", ["linear", "poly", "rbf"])
@pytest.mark.parametrize("case", ["plain", "large 1e6", "large 1e9", "large 1e12", "disjoint", "decades", "whole numbers"])
def test_rows_of_uneven_features(case, kind):
    m, n, lam = 600, 64, 1e-2
    g = np.random.Generator(np.random.PCG64(11))
    A, al0, y = data(case, m, n, g), g.standard_normal(m), g.standard_normal(m)
    kw = KERNELS[kind]
    got = gradient(A, al0, y, kind, kw, lam)
    want = oracle.krr_gradient(A, y, oracle.kernel(kind, **kw), lam, al0)
    if kind == "rbf":
        size = oracle.kernel_block(oracle.kernel(kind, **kw), A, np.arange(m)) @ np.abs(al0)
    else:
        size = np.abs(A) @ np.abs(A).T
        if kind == "poly":
            size = (size + kw["coef0"]) ** kw["degree"]
        size = size @ np.abs(al0)
    size = size / lam + m * np.abs(al0) + np.abs(y)
    d = kw.get("degree", 1)
    assert np.max(np.abs(got - want) / size) < 2 * d * (n + m + 16) * 2.0 ** -53
