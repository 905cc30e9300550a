"""dcd_dcd_recurrence with y other than +-1 (the entry point takes any weights): theta follows the couplings
y_t y_j K_tj and w = y theta, on both sides of the 128 coordinates up to which the chain runs in registers.

Tolerance: a pending gradient is a sum of at most cnt + 1 terms, each within 2^-52 of the largest
|y_t y_j K_tj theta_j| seen; 1e-11 of the size of theta covers that for cnt <= 200 with the steps' own
amplification (couplings below 1/4 of the diagonal).  w is the one product y theta: exact.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def reference(K, S, y, al, g, omega, nu):
    cnt = len(S)
    al, g, th = al.copy(), g.copy(), np.zeros(cnt)
    for j in range(cnt):
        eta = K[j, j] + omega
        if min(max(al[j] - g[j], 0.0), nu) != al[j]:
            th[j] = min(max(al[j] - g[j] / eta, 0.0), nu) - al[j]
        same = S == S[j]
        g += y * y[j] * K[:, j] * th[j] + omega * th[j] * same
        al += th[j] * same
    return th


@pytest.mark.parametrize("cnt", [1, 5, 32, 40, 128, 129, 200])
@pytest.mark.parametrize("loss", [1, 2])
@pytest.mark.parametrize("weights", ["labels", "any", "some zero"])
@pytest.mark.parametrize("f64", [True, False])
def test_recurrence_takes_any_weights(cnt, loss, weights, f64):
    from paper_2406_18001_gb300 import binding as B
    r = np.random.Generator(np.random.PCG64(cnt))
    X = r.standard_normal((cnt, 64)) / 16
    S = r.integers(0, max(cnt // 2, 1) + 3, cnt).astype(np.int32)
    X = X[S % cnt]  # a repeated id is the same row
    K = X @ X.T
    K[S[:, None] == S[None, :]] = 1.0
    if not f64:
        K = K.astype(np.float32).astype(np.float64)
    y = np.where(r.random(cnt) < 0.5, 1.0, -1.0)
    if weights != "labels":
        y *= r.uniform(0.3, 1.2, cnt)
    if weights == "some zero":
        y[::3] = 0.0
    y = y[np.unique(S, return_index=True)[1]][np.unique(S, return_inverse=True)[1]]  # one weight a row
    C = 0.8
    al = r.uniform(0, C, cnt)[np.unique(S, return_inverse=True)[1]]
    g = r.standard_normal(cnt)[np.unique(S, return_inverse=True)[1]]
    omega, nu = (0.0, C) if loss == 1 else (0.5 / C, np.inf)
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    theta, w = torch.empty(cnt, dtype=torch.float64, device="cuda"), torch.empty(cnt, dtype=torch.float64, device="cuda")
    B.dcd_recurrence(d(K if f64 else K.astype(np.float32)), d(S), d(y), d(al), d(g), loss, C, theta, w)
    theta, w = theta.cpu().numpy(), w.cpu().numpy()
    want = reference(K, S, y, al, g, omega, nu)
    assert np.max(np.abs(theta - want)) <= 1e-11 * max(np.max(np.abs(want)), 1.0)
    assert np.array_equal(w, y * theta)
