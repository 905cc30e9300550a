"""The deferred K-RR step's split of the SMs between the block and the next step's Gram (the more
CTAs for the Gram, the narrower its items): sizes for which the block is the longer path, the side
path is, and neither fills the chip, against in-order steps.  1e-5 relative, the deferred step's bound
(its sums are those of the in-order step in another association)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEFER_TOL = 1e-5


@pytest.mark.parametrize("m,n,b,s,prec", [
    (300, 17, 4, 60, "bf16x3"), (1700, 512, 16, 64, "fp16"), (8000, 300, 16, 44, "bf16x3"),
    (20000, 512, 16, 44, "tf32x3"), (40000, 384, 32, 32, "tf32x3"), (30000, 512, 32, 16, "bf16x3")])
def test_deferred_steps_match_in_order_steps(m, n, b, s, prec):
    from paper_2406_18001_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn(m, n, generator=g, device="cuda") / n ** 0.5
    y = torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        runs = [B.krr_solve(A, y, B.kernel("rbf", gamma=0.5), 1e-3, b, s, 6 * s, seed=7, prec=prec, flags=f,
                            stream=st.cuda_stream)[:2] for f in (B.FLAG_NO_DEFER, 0)]
    st.synchronize()
    (a0, g0), (a1, g1) = runs
    assert float((a1 - a0).norm()) <= DEFER_TOL * float(a0.norm())
    assert float((g1 - g0).norm()) <= DEFER_TOL * float(y.norm())
