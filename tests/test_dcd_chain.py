"""The K-SVM recurrence of up to 128 coordinates against Algorithm 2 one coordinate at a time: groups
of 32 and their edges, repeated rows within and across groups, coordinates that cannot move (at a
bound, a diagonal that is not positive), and Grams scaled by a power of two, which leaves the steps as
they are and takes the recurrence to and past the range in which it keeps scaled gradients.  Both
sides are FP64 sums of at most 128 terms of size one: 1e-12 absolute."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def reference(K, S, y, alpha, g, omega, nu):
    al, gr, th = alpha.copy(), g.copy(), np.zeros(len(S))
    for t in range(len(S)):
        eta = K[t, t] + omega
        r = al[S[t]]
        if eta > 0 and min(max(r - gr[t], 0.0), nu) != r:
            th[t] = min(max(r - gr[t] / eta, 0.0), nu) - r
        al[S[t]] += th[t]
        for q in range(t + 1, len(S)):
            gr[q] += y[S[q]] * y[S[t]] * K[q, t] * th[t] + (omega * th[t] if S[q] == S[t] else 0.0)
    return th


@pytest.mark.parametrize("cnt", [1, 2, 31, 32, 33, 64, 65, 100, 128])
@pytest.mark.parametrize("loss", [1, 2])
@pytest.mark.parametrize("shift", [0, -19, -21, -40, 299, 302])
@pytest.mark.parametrize("f64", [True, False])
def test_recurrence_matches_one_coordinate_at_a_time(cnt, loss, shift, f64):
    from paper_2406_18001_gb300 import binding as B
    if not f64 and shift > 100:
        pytest.skip("past FP32's range")
    r = np.random.default_rng(cnt + 7 * loss)
    m = max(cnt - cnt // 8, 1)
    S = r.permutation(np.concatenate([np.arange(m), r.integers(0, m, cnt - m)])).astype(np.int32)
    X = r.standard_normal((m, 40)) / 8
    K = (X @ X.T + 1.0 + np.diag(r.random(m)))[np.ix_(S, S)]
    bad = r.random(m) < 0.1
    K[bad[S][:, None] & (S[:, None] == S[None, :])] = -3.0  # such a row's coordinates do not move
    K = K.astype(np.float32).astype(np.float64)
    y = np.where(r.random(m) < 0.5, -1.0, 1.0)
    C = 0.75
    alpha = np.where(r.random(m) < 0.5, r.random(m) * C, np.where(r.random(m) < 0.5, 0.0, C if loss == 1 else 0.3))
    alpha[0] = -0.0
    g = r.standard_normal(m) * 0.3
    omega = 0.0 if loss == 1 else 0.25
    sc = 2.0 ** shift
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    want = reference(K, S, y, alpha, g[S], omega, C if loss == 1 else np.inf)
    th, w = torch.empty(cnt, dtype=torch.float64).cuda(), torch.empty(cnt, dtype=torch.float64).cuda()
    Kd = d(K * sc) if f64 else d((K * sc).astype(np.float32))
    B.dcd_recurrence(Kd, d(S), d(y[S]), d(alpha[S]), d(g[S] * sc), loss, C if loss == 1 else 2.0 / sc, th, w)
    torch.cuda.synchronize()
    assert np.max(np.abs(th.cpu().numpy() - want)) < 1e-12
    assert np.array_equal(w.cpu().numpy(), y[S] * th.cpu().numpy())
