"""K-RR in the tensor-core forms with block sizes that do not divide the Gram's 128-row tiles: diagonal blocks
lie across tile edges, and the recurrences read them whole though the Gram is written by its lower
triangle.  Against the oracle at 1e-4 relative (the split forms' tolerance for alpha), with the deferred
and the in-order look-ahead and on one stream, on one cluster and in panels (s b > 1024), with memory
that earlier calls have left full of other values."""
import numpy as np
import pytest

import oracle
from paper_2406_18001_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,s", [(12, 11), (12, 30), (20, 7), (20, 32), (20, 50), (24, 6), (24, 41), (28, 5), (28, 36),
                                 (20, 60), (28, 50)])
@pytest.mark.parametrize("mode", ["deferred", "in order", "one stream"])
def test_solve_matches_oracle(b, s, mode):
    from paper_2406_18001_gb300 import binding as B
    p = inputs.krr_dense(m=1500, n=40, seed=b, dtype=np.float32)
    lam, H = 1e-3, 4 * s + 1
    k = B.kernel("rbf", gamma=0.5)
    A, y = torch.from_numpy(p.A).cuda(), torch.from_numpy(p.y).cuda()
    st = torch.cuda.current_stream() if mode == "one stream" else torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        # what the library's memory holds next: another problem's kernel values
        B.krr_solve(A * 3, y, B.kernel("poly", degree=4, coef0=1.0), 1.0, b, s, 4 * s, seed=1, prec="bf16x3")
        al, _, _, _ = B.krr_solve(A, y, k, lam, b, s, H, seed=3, prec="bf16x3",
                                  flags=B.FLAG_NO_DEFER if mode == "in order" else 0)
        st.synchronize()
    want = oracle.bdcd_krr(p.A.astype(np.float64), p.y, oracle.kernel("rbf", gamma=0.5), lam, b, H, seed=3)
    assert np.linalg.norm(al.cpu().numpy() - want) < 1e-4 * np.linalg.norm(want)
