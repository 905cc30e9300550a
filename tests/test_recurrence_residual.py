"""dcd_bdcd_recurrence on an FP64 Gram with ill-conditioned diagonal blocks (near-duplicate rows, a small
lambda): every block's system is solved to the residual of a Cholesky solve.

Allowed, in units of 2^-53: b for the block's own product |G_jj| |Delta_j| (a Cholesky solve stays near 1),
and, as rounding of the right-hand side, the number of terms for each earlier |G_jt| |Delta_t|.  The
residual is worked out in extended precision.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,nblk", [(2, 9), (4, 8), (7, 5), (8, 16), (16, 4), (16, 64), (31, 3), (32, 6)])
@pytest.mark.parametrize("lam,dup", [(1e-2, 1.0), (1e-6, 1e-2), (1e-9, 1e-3), (1e-11, 1e-5), (1e-13, 1e-6)])
def test_block_residuals(b, nblk, lam, dup):
    from paper_2406_18001_gb300 import binding as B
    r = np.random.Generator(np.random.PCG64(b * nblk))
    sb, mdiag = b * nblk, 50.0
    X = r.standard_normal((sb, 24)) / 6
    X[1::2] = X[::2][:len(X[1::2])] + dup * r.standard_normal(X[1::2].shape) / 6
    K = np.exp(-0.5 * ((X[:, None] - X[None]) ** 2).sum(2))
    g = r.standard_normal(sb)
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    delta, w = torch.empty(sb, dtype=torch.float64, device="cuda"), torch.empty(sb, dtype=torch.float64, device="cuda")
    B.bdcd_recurrence(d(K), d(np.arange(sb, dtype=np.int32)), b, lam, mdiag, d(g), delta, w)
    x = delta.cpu().numpy()
    G = K.astype(np.longdouble) / np.longdouble(lam) + np.longdouble(mdiag) * np.eye(sb, dtype=np.longdouble)
    size = np.linalg.norm(G.astype(float).reshape(nblk, b, nblk, b), axis=(1, 3)) * np.linalg.norm(x.reshape(nblk, b), axis=1)
    for j in range(nblk):
        s = slice(j * b, (j + 1) * b)
        res = -g[s] - G[s, :(j + 1) * b] @ x[:(j + 1) * b].astype(np.longdouble)
        allowed = b * size[j, j] + (j * b + b) * size[j, :j].sum() + np.linalg.norm(g[s])
        assert float(np.linalg.norm(res.astype(float))) <= allowed * 2.0 ** -53
