"""The K-RR recurrence on one thread-block cluster against an FP64 block forward substitution: every
super-block size (20, 24, 28 and 32 rows), a last super-block that is not full, one super-block, an
odd number of them, the most a cluster takes and one more, with few and with many repeated rows.
The FP32 solve is refined once by an exact residual: an error of (n eps32)^2 kappa^2 for panels of
n = 32 and K / lambda + m I with kappa < 3, below 1e-10."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nblk,b", [(1, 4), (8, 4), (9, 4), (250, 4), (45, 8), (3, 12), (41, 12), (63, 16), (64, 16),
                                    (66, 16), (50, 20), (40, 24), (7, 28), (1, 32), (2, 32), (31, 32), (33, 32)])
@pytest.mark.parametrize("rows", [20000, 300])
def test_recurrence_matches_fp64_substitution(nblk, b, rows):
    from paper_2406_18001_gb300 import binding as B
    r = np.random.default_rng(nblk * b + rows)
    cnt, lam, m = nblk * b, 0.05, 20000.0
    S = np.concatenate([r.choice(rows, b, replace=False) for _ in range(nblk)]).astype(np.int32)
    X = r.standard_normal((rows, 24)) / 24 ** 0.5
    n2 = (X[S] ** 2).sum(1)
    K = np.exp(-0.5 * np.maximum(n2[:, None] + n2[None] - 2 * X[S] @ X[S].T, 0)).astype(np.float32)
    G = K.astype(np.float64) / lam + m * (S[:, None] == S[None, :])
    g = r.standard_normal(rows)[S]
    want = np.zeros(cnt)
    for k in range(nblk):
        i = slice(k * b, k * b + b)
        want[i] = np.linalg.solve(G[i, i], -g[i] - G[i, :k * b] @ want[:k * b])
    d = lambda x: torch.from_numpy(x).cuda()
    delta, w = torch.empty(cnt, dtype=torch.float64).cuda(), torch.empty(cnt, dtype=torch.float64).cuda()
    B.bdcd_recurrence(d(K), d(S), b, lam, m, d(g), delta, w)
    torch.cuda.synchronize()
    got = delta.cpu().numpy()
    assert np.linalg.norm(got - want) < 1e-10 * np.linalg.norm(want)
    assert np.array_equal(w.cpu().numpy(), got / lam)
