"""The RBF values of the FP64 form at the edges of its slices' range."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def B():
    from paper_2406_18001_gb300 import binding
    return binding


def test_one_large_feature():
    """Values against one row, read off the gradient of a unit alpha.  Allowed: four roundings of an exponent
    made of gamma |a|^2 + gamma |b|^2 <= 16 (the expansion's error), which a kernel value near 1 shows."""
    m, n, j = 200, 512, 7
    g = np.random.Generator(np.random.PCG64(3))
    A = g.standard_normal((m, n)) * 1e-3
    A[:, 100] = 2.05
    gamma = 7.9 / 2.05 ** 2
    al0 = np.zeros(m)
    al0[j] = 1.0
    _, gr, _, _ = B().krr_solve(torch.from_numpy(A).cuda(), torch.ones(m, dtype=torch.float64).cuda(),
                                B().kernel("rbf", gamma=gamma), 1.0, 8, 8, 0, prec="fp64",
                                alpha=torch.from_numpy(al0).cuda())
    got = gr.cpu().numpy() + 1.0
    want = oracle.kernel_block(oracle.kernel("rbf", gamma=gamma), A, np.array([j]))[:, 0]
    assert np.max(np.abs(got - want)[np.arange(m) != j]) < 4 * 16 * 2.0 ** -53
