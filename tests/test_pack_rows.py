"""Operands packed four rows a warp (32768 rows and more; also with a last warp that is not full, a
strided matrix, columns past a multiple of 32) against FP64: K(A, A_S) w, where a row's wrong norm or
place shows as an error of order one.  Tolerances: the forms' unit roundoffs (fp16 2^-11, bf16 2^-8,
split bf16 2^-16) times 8 for the exponent's size, on sums of positive terms."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [32767, 32768, 32769, 32770, 32771])
@pytest.mark.parametrize("n,ld", [(33, 33), (64, 70), (300, 300)])
@pytest.mark.parametrize("prec,tol", [("fp16", 8 * 2.0 ** -11), ("bf16", 8 * 2.0 ** -8), ("bf16x3", 8 * 2.0 ** -16)])
def test_rows_and_norms(m, n, ld, prec, tol):
    from paper_2406_18001_gb300 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    A = (torch.randn(m, ld, generator=gen, device="cuda") / n ** 0.5)[:, :n]
    cols = torch.randint(0, m, (40,), generator=gen, device="cuda", dtype=torch.int32)
    w = torch.rand(40, generator=gen, device="cuda", dtype=torch.float64) + 0.5
    g = torch.zeros(m, device="cuda", dtype=torch.float64)
    B.kernel_block_apply(A, B.kernel("rbf", gamma=0.5), prec, cols, w, g)
    D = A.double()
    d2 = (D * D).sum(1)[:, None] + (D[cols.long()] ** 2).sum(1)[None] - 2 * D @ D[cols.long()].T
    want = torch.exp(-0.5 * d2.clamp(min=0)) @ w
    assert float(((g - want).abs() / want).max()) < tol
