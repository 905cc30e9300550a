"""The FP64 form with an RBF width far beyond the data's: K = 1 to rounding, against the oracle (1e-10,
the FP64 form's tolerance for iterates)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma,scale", [(1e-170, 1e-100), (1e-250, 1e-50), (1e-300, 1.0), (5e-324, 1.0)])
def test_tiny_gamma(gamma, scale):
    from paper_2406_18001_gb300 import binding as B
    m, n, b, s = 300, 65, 8, 8
    g = np.random.Generator(np.random.PCG64(5))
    A, y = g.standard_normal((m, n)) * scale, g.standard_normal(m)
    al, _, _, _ = B.krr_solve(torch.from_numpy(A).cuda(), torch.from_numpy(y).cuda(), B.kernel("rbf", gamma=gamma), 1e-2,
                              b, s, 3 * s, seed=2, prec="fp64")
    want = oracle.bdcd_krr(A, y, oracle.kernel("rbf", gamma=gamma), 1e-2, b, 3 * s, seed=2)
    assert np.linalg.norm(al.cpu().numpy() - want) < 1e-10 * np.linalg.norm(want)
