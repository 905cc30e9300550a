"""The library's memory pool: calls from several threads on streams of their own give the bits of one
call, and after calls that need more than it keeps no more than that stays allocated."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def apply(B, A, cols, w, st):
    with torch.cuda.stream(st):
        g = torch.zeros(A.shape[0], dtype=torch.float64, device="cuda")
        B.kernel_block_apply(A, B.kernel("rbf", gamma=0.3), "fp16", cols, w, g)
    st.synchronize()
    return g


@pytest.mark.parametrize("threads", [1, 4])
def test_threads_and_streams_share_the_pool(threads):
    from paper_2406_18001_gb300 import binding as B
    gen = torch.Generator(device="cuda").manual_seed(5)
    jobs = []
    for i in range(threads):
        A = torch.randn(2000 + 777 * i, 60, generator=gen, device="cuda") / 8
        cols = torch.arange(0, 900, 3, device="cuda", dtype=torch.int32)
        w = torch.randn(300, generator=gen, device="cuda", dtype=torch.float64)
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        jobs.append((A, cols, w, st, apply(B, A, cols, w, st)))
    bad = []

    def work(job):
        A, cols, w, st, want = job
        for _ in range(20):
            if not torch.equal(apply(B, A, cols, w, st), want):
                bad.append(A.shape)

    ts = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


def test_what_stays_allocated_is_bounded():
    from paper_2406_18001_gb300 import binding as B
    A = torch.randn(1 << 20, 512, device="cuda")  # 1 GB of packed fp16
    cols = torch.arange(64, device="cuda", dtype=torch.int32)
    w = torch.ones(64, device="cuda", dtype=torch.float64)
    g = torch.zeros(1 << 20, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    B.kernel_block_apply(A, B.kernel("linear"), "fp16", cols, w, g)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= (512 << 20) + (64 << 20)  # and the driver's own granules
