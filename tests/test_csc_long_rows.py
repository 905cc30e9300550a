"""CSR data with rows of more than 131071 nonzeros: the apply through the transposed copy is taken where it
reads less, as with short rows, and gives the bits of the full pass; elements too far into their tile for
a key send that tile to the full pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def matrix(m, n, nnz, long_rows, length, seed):
    """m rows of nnz nonzeros, those in long_rows of `length`; sorted distinct columns, unit rows (FP32)."""
    g = np.random.default_rng(seed)
    rp, ci, va = [0], [], []
    for i in range(m):
        k = length if i in long_rows else nnz
        step = n // k
        c = np.arange(k, dtype=np.int64) * step + g.integers(0, step, k)
        v = g.random(k) + 0.1
        ci.append(c.astype(np.int32))
        va.append((v / np.linalg.norm(v)).astype(np.float32))
        rp.append(rp[-1] + k)
    return np.array(rp, np.int64), np.concatenate(ci), np.concatenate(va)


# one long row; a tile of long rows (6.4 M nonzeros, beyond the 2^22 a key holds); the longest rows that the
# scatter's launch takes, and longer ones (the full pass)
@pytest.mark.parametrize("m,n,long_rows,length,through", [
    (3000, 600000, [1700], 131072, True), (3000, 16000000, range(64, 96), 200000, True),
    (3000, 1200000, [2999], 262140, True), (3000, 1200000, [2999], 262141, False)])
@pytest.mark.parametrize("prec", ["bf16x3", "fp64"])
def test_long_rows(m, n, long_rows, length, through, prec):
    from paper_2406_18001_gb300 import binding as B
    rp, ci, va = matrix(m, n, 20, set(long_rows), length, 7)
    d = lambda x: torch.from_numpy(x).cuda()
    A = B.Csr(d(rp), d(ci), d(va.astype(np.float64 if prec == "fp64" else np.float32)), n)
    y = d(np.where(np.random.default_rng(1).random(m) < 0.5, 1.0, -1.0))
    res = []
    for flags in (0, B.FLAG_CSR_FULL_PASS):
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            al, gr, info, _ = B.svm_solve(A, y, B.kernel("poly", coef0=1.0, degree=3), 2, 0.5, 8, 8 * 40, seed=3,
                                          prec=prec, flags=flags)
        torch.cuda.synchronize()
        res.append((al, gr, info["gpu_launches_per_step"]))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    assert res[0][2] == res[1][2] + (1 if through else 0)  # the scatter
