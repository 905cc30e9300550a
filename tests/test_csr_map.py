"""The sampled rows' column map and Gram on CSR data against the oracle's DCD, at the shapes where
they change form: one row; columns that two, and that many, sampled rows hold; empty rows; more
coordinates than a warp has lanes; the register map's last size (4096 positions; 262144 columns) and
the first past each.  FP64 iterates 1e-10 relative, FP32 1e-5 (the CSR solver's tolerances)."""
import numpy as np
import pytest

import oracle
from paper_2406_18001_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def B():
    from paper_2406_18001_gb300 import binding
    return binding


def ragged(m, n, max_nnz, seed):
    """Rows of 0 .. max_nnz sorted columns, every seventh empty, the last one full."""
    g = np.random.default_rng(seed)
    rp, ci, va = [0], [], []
    for i in range(m):
        k = max_nnz if i == m - 1 else 0 if i % 7 == 3 else int(g.integers(1, max_nnz + 1))
        ci.extend(np.sort(g.choice(n, size=k, replace=False)).tolist())
        va.extend((g.standard_normal(k) * 0.3).tolist())
        rp.append(len(ci))
    return inputs.CsrProblem(np.array(rp, np.int64), np.array(ci, np.int32), np.array(va, np.float64), n,
                             np.where(g.random(m) < 0.5, -1.0, 1.0))


@pytest.mark.parametrize("prec,dtype,tol", [("fp64", np.float64, 1e-10), ("bf16x3", np.float32, 1e-5)])
@pytest.mark.parametrize("m,n,max_nnz,s", [(1, 5, 3, 1), (70, 40, 9, 31), (70, 40, 9, 33), (400, 3000, 12, 32),
                                           (40, 30, 12, 128), (90, 262144, 64, 64), (90, 262145, 64, 64),
                                           (90, 1000, 64, 64), (90, 1000, 65, 64), (64, 2000, 130, 32)])
def test_svm_iterates_match_oracle(m, n, max_nnz, s, prec, dtype, tol):
    p = ragged(m, n, max_nnz, seed=m + n)
    va = p.values.astype(dtype)
    A = inputs.CsrProblem(p.row_ptr, p.col_idx, va.astype(np.float64), p.n, p.y).to_dense()
    Ad = B().Csr(torch.from_numpy(p.row_ptr).cuda(), torch.from_numpy(p.col_idx).cuda(), torch.from_numpy(va).cuda(), n)
    H = 6 * s + min(s - 1, 3)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        al, _, info, _ = B().svm_solve(Ad, torch.from_numpy(p.y).cuda(), B().kernel("rbf", gamma=0.3), 2, 0.5, s, H,
                                       seed=5, prec=prec)
    st.synchronize()
    want = oracle.dcd_svm(A, p.y, oracle.kernel("rbf", gamma=0.3), 2, 0.5, H, seed=5)
    assert info["iters_done"] == H
    assert np.linalg.norm(al.cpu().numpy() - want) < tol * np.linalg.norm(want)
