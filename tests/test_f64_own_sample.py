"""The RBF value of a row against itself is exactly 1 in the FP64 form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(300, 65), (129, 512)])
def test_a_row_against_itself(m, n):
    """alpha = e_j and lambda = 2^-40: g_j = 2^40 K_jj + m - 1, so that the last bit of K_jj shows."""
    from paper_2406_18001_gb300 import binding as B
    g = np.random.Generator(np.random.PCG64(9))
    A = torch.from_numpy(g.standard_normal((m, n)) / np.sqrt(n)).cuda()
    y = torch.ones(m, dtype=torch.float64).cuda()
    for j in list(range(0, m, 7)) + [m - 1]:
        al0 = torch.zeros(m, dtype=torch.float64).cuda()
        al0[j] = 1.0
        _, gr, _, _ = B.krr_solve(A, y, B.kernel("rbf", gamma=4.0), 2.0 ** -40, 8, 8, 0, prec="fp64", alpha=al0)
        assert float(gr[j]) == 2.0 ** 40 + m - 1
