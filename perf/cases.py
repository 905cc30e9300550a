"""What is timed of this framework: solves, plans and kernel blocks as a program calls them.

Every case goes through the Python binding's public entry points on one GPU.
A plan case advances a resident solve by a few outer steps (the plan is what a
training program keeps); a solve case is one whole call, set-up included.  The
sizes are those of the benchmark's five workloads and of the tests' ragged and
small problems; draw() gives further ones of the same ranges.  exact() works
the paper's iteration out in 64 bits with plain torch and numpy on the same
index stream.
"""
import numpy as np
import torch

from paper_2406_18001_gb300 import binding as B

BUDGET = 1 << 40  # a plan's iteration budget: never used up here


def listed():
    return [
        # a first try on a few hundred rows, one coordinate at a time, on the default stream: launches and set-up
        {"name": "svm-small-solve", "kind": "svm", "m": 300, "n": 16, "s": 1, "H": 256, "loss": 1, "prec": "fp64",
         "kernel": "rbf", "own_stream": False},
        # the K-SVM blobs workload: 20000 coordinate updates in FP64, s = 8, as one call
        {"name": "svm-blobs-fp64", "kind": "svm", "m": 2000, "n": 64, "s": 8, "H": 20000, "loss": 1, "prec": "fp64",
         "kernel": "rbf", "own_stream": True},
        # the same data with the squared hinge in split bf16 and long steps (the form that reaches a gap fastest)
        {"name": "svm-blobs-split", "kind": "svm", "m": 2000, "n": 64, "s": 64, "H": 16384, "loss": 2,
         "prec": "bf16x3", "kernel": "rbf", "own_stream": True},
        # K-SVM on uniformly sparse CSR rows (text-like data), polynomial kernel, FP32 block
        {"name": "svm-csr", "kind": "csr", "m": 200000, "n": 50000, "nnz": 50, "s": 32, "steps": 16,
         "prec": "bf16x3"},
        # the headline: K-RR steps of 1024 coordinates on a dense matrix, fp16 kernel block
        {"name": "krr-dense-fp16", "kind": "krr", "m": 50000, "n": 512, "b": 16, "s": 64, "steps": 8, "prec": "fp16",
         "kernel": "rbf"},
        # odd sizes in split bf16 with the polynomial kernel: no tile, chunk or k-block is full
        {"name": "krr-ragged-split", "kind": "krr", "m": 20011, "n": 301, "b": 8, "s": 45, "steps": 16,
         "prec": "bf16x3", "kernel": "poly"},
        # the FP64 form of K-RR (the reference results of a study), moderate size
        {"name": "krr-dense-fp64", "kind": "krr", "m": 6000, "n": 512, "b": 16, "s": 16, "steps": 4, "prec": "fp64",
         "kernel": "rbf"},
        # the largest: FP8 storage, steps of 4096 coordinates
        {"name": "krr-stress-fp8", "kind": "stress", "m": 400000, "n": 2048, "b": 32, "s": 128, "steps": 1,
         "prec": "fp8"},
        # a hyperparameter sweep: uneven independent problems in one batched call
        {"name": "krr-sweep", "kind": "sweep", "count": 32, "n": 128, "m_lo": 1000, "m_hi": 20000, "H": 512,
         "prec": "fp16"},
        # a whole solve from pinned host arrays to relative residual 1e-6, recomputed gradient included
        {"name": "krr-to-tolerance", "kind": "tolerance", "m": 20000, "n": 512, "b": 16, "s": 64, "prec": "fp16"},
        # predictions of a fitted model: K(A, A_S) w in one call, nothing kept between calls
        {"name": "predict-fp16", "kind": "apply", "m": 50000, "n": 512, "cols": 1024, "prec": "fp16",
         "kernel": "rbf"},
        # an explicit kernel block for another program's use, odd sizes
        {"name": "kernel-block-split", "kind": "block", "m": 12001, "n": 257, "cols": 999, "prec": "bf16x3",
         "kernel": "rbf"},
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread over the logarithm of the range, odd as often as even."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["svm", "svm", "csr", "krr", "krr", "krr", "fp64", "stress", "sweep", "tolerance", "apply",
                       "block"])
    dense = rng.choice(["fp16", "bf16", "bf16x3", "tf32x3", "fp16", "bf16x3"])
    kernel = rng.choice(["rbf", "rbf", "rbf", "poly", "linear"])
    if kind == "svm":
        s = rng.choice([1, 4, 8, 16, 32, 64])
        return {"kind": "svm", "m": _log(rng, 200, 6000), "n": _log(rng, 8, 200), "s": s,
                "H": s * _log(rng, 100, 1000), "loss": rng.choice([1, 2]),
                "prec": rng.choice(["fp64", "fp64", "bf16x3", "fp16"]), "kernel": "rbf", "own_stream": rng.random() < 0.8}
    if kind == "csr":
        return {"kind": "csr", "m": _log(rng, 10000, 200000), "n": _log(rng, 3000, 50000),
                "nnz": rng.randint(10, 50), "s": rng.choice([1, 8, 16, 32]), "steps": 16,
                "prec": rng.choice(["fp64", "bf16x3"])}
    if kind == "krr":
        b = rng.choice([4, 8, 16, 32])
        return {"kind": "krr", "m": _log(rng, 2000, 50000), "n": _log(rng, 30, 512), "b": b,
                "s": rng.randint(max(1, 64 // b), 1024 // b), "steps": 8, "prec": dense, "kernel": kernel}
    if kind == "fp64":
        return {"kind": "krr", "m": _log(rng, 600, 6000), "n": _log(rng, 30, 512), "b": rng.choice([8, 16]),
                "s": rng.randint(1, 16), "steps": 4, "prec": "fp64", "kernel": kernel}
    if kind == "stress":
        return {"kind": "stress", "m": _log(rng, 40000, 200000), "n": _log(rng, 700, 2048), "b": 32,
                "s": rng.choice([32, 64, 128]), "steps": 1, "prec": rng.choice(["fp8", "bf16"])}
    if kind == "sweep":
        return {"kind": "sweep", "count": rng.randint(6, 32), "n": _log(rng, 64, 128), "m_lo": 1000,
                "m_hi": _log(rng, 4000, 20000), "H": _log(rng, 128, 512), "prec": dense}
    if kind == "tolerance":
        return {"kind": "tolerance", "m": _log(rng, 4000, 20000), "n": _log(rng, 256, 512), "b": 16,
                "s": rng.choice([16, 32, 64]), "prec": rng.choice(["fp16", "bf16x3"])}
    if kind == "apply":
        return {"kind": "apply", "m": _log(rng, 1000, 50000), "n": _log(rng, 30, 512), "cols": _log(rng, 16, 1024),
                "prec": dense, "kernel": kernel}
    return {"kind": "block", "m": _log(rng, 500, 12000), "n": _log(rng, 30, 512), "cols": _log(rng, 16, 1024),
            "prec": dense, "kernel": kernel}


# ---------------------------------------------------------------- inputs ---
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _gauss(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _blobs(c, seed):
    """Two Gaussian blobs (means +-0.5 in every coordinate, unit variance), labels +-1 (FP64)."""
    g = _gen(seed)
    y = torch.where(torch.rand(c["m"], generator=g, device="cuda") < 0.5, 1.0, -1.0).double()
    return _gauss(g, c["m"], c["n"], dtype=torch.float64) + 0.5 * y[:, None], y


def _regression(m, n, seed):
    """A ~ N(0, 1) / sqrt(n) in FP32, y = sin(A w) + 0.1 N(0, 1) with w ~ N(0, I)."""
    g = _gen(seed)
    A = _gauss(g, m, n) / float(n) ** 0.5
    w = _gauss(g, n)
    return A, torch.sin(A @ w).double() + 0.1 * _gauss(g, m, dtype=torch.float64)


def _sparse(c, seed):
    """Rows of nnz distinct uniform columns (one in each of nnz equal bands), U(0, 1) values scaled to unit norm,
    labels from a random hyperplane with 5% flips."""
    g = _gen(seed)
    m, n, k = c["m"], c["n"], c["nnz"]
    band = n // k
    cols = torch.arange(k, device="cuda")[None] * band + torch.randint(0, band, (m, k), generator=g, device="cuda")
    vals = torch.rand(m, k, generator=g, device="cuda", dtype=torch.float64) + 1e-3
    vals = (vals / vals.norm(dim=1, keepdim=True)).float()
    w = _gauss(g, n) * (torch.rand(n, generator=g, device="cuda") < 0.01)
    y = torch.where((vals * w[cols]).sum(1) >= 0, 1.0, -1.0)
    y = torch.where(torch.rand(m, generator=g, device="cuda") < 0.05, -y, y).double()
    ptr = torch.arange(0, (m + 1) * k, k, device="cuda", dtype=torch.int64)
    return ptr, cols.reshape(-1).int(), vals.reshape(-1), y


def _stress(c, seed):
    """Ill-conditioned rows z^T diag(sig) W^T (sig log-spaced over four decades, E||a||^2 = 64), stored BF16."""
    g = _gen(seed)
    n = c["n"]
    W, _ = torch.linalg.qr(_gauss(g, n, n))
    sig = torch.logspace(-4, 0, n, device="cuda")
    sig = sig * (64.0 / sig.square().sum()).sqrt()
    mix = sig[:, None] * W.T
    w = _gauss(g, n) / 8.0
    A = torch.empty(c["m"], n, device="cuda", dtype=torch.bfloat16)
    y = torch.empty(c["m"], device="cuda", dtype=torch.float64)
    for r in range(0, c["m"], 65536):
        rows = _gauss(g, min(65536, c["m"] - r), n) @ mix
        A[r:r + 65536] = rows.bfloat16()
        y[r:r + 65536] = torch.sin(rows @ w).double()
    return A, y + 0.1 * _gauss(g, c["m"], dtype=torch.float64)


def _e4m3(A):
    """Per-row FP8 storage: scale = max|a| / 448, codes of a / scale."""
    q = torch.empty(A.shape, device="cuda", dtype=torch.uint8)
    sc = torch.empty(A.shape[0], device="cuda", dtype=torch.float32)
    for r in range(0, A.shape[0], 65536):
        a = A[r:r + 65536].float()
        s = a.abs().amax(1) / 448.0
        sc[r:r + 65536] = s
        q[r:r + 65536] = (a / s[:, None]).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
    return q, sc


def _sweep(c, seed):
    """The problems of a sweep: m uneven, A and y ~ N(0, 1), sigma and lambda over log ranges, b 8 or 32 (the grid
    is the case's, the data the seed's)."""
    out = []
    for p in range(c["count"]):
        g = _gen(seed * 1009 + p)
        r = np.random.RandomState(p)
        m = int(r.randint(c["m_lo"], c["m_hi"] + 1))
        sig, lam = 10.0 ** r.uniform(-1, 1), 10.0 ** r.uniform(-6, -1)
        b = 8 if p % 2 == 0 else 32
        out.append({"A": _gauss(g, m, c["n"]), "y": _gauss(g, m, dtype=torch.float64), "gamma": 0.5 / sig ** 2,
                    "lam": lam, "b": b, "s": 1024 // b, "H": c["H"], "seed": p})
    return out


def _columns(c, seed):
    """The distinct rows that a fitted model keeps, and their coefficients."""
    g = _gen(seed + 77)
    cols = torch.randperm(c["m"], generator=g, device="cuda")[:c["cols"]].sort().values.int()
    return cols, _gauss(g, cols.numel(), dtype=torch.float64)


def _kernel_args(c):
    """(kind, gamma, coef0, degree) of a case's kernel."""
    if c["kind"] == "svm":
        return "rbf", 0.5 / c["n"], 0.0, 2
    if c["kind"] == "csr":
        return "poly", 1.0, 1.0, 3
    if c["kind"] == "stress":
        return "rbf", 1.0 / 128, 0.0, 2
    return {"rbf": ("rbf", 0.5, 0.0, 2), "poly": ("poly", 1.0, 1.0, 2), "linear": ("linear", 1.0, 0.0, 2)}[
        c.get("kernel", "rbf")]


def _kernel(c):
    kind, gamma, coef0, degree = _kernel_args(c)
    return B.kernel(kind, gamma=gamma, coef0=coef0, degree=degree)


LAMBDA = {"krr": 1e-4, "stress": 1e-6, "tolerance": 1e-4}
SVM_C = {"svm": 1.0, "csr": 0.5}


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c, "kernel": _kernel(c), "seed": int(seed)}
    if kind == "svm":
        st["A"], st["y"] = _blobs(c, seed)
        st["stream"] = torch.cuda.Stream() if c["own_stream"] else torch.cuda.current_stream()
    elif kind == "apply" or kind == "block":
        st["A"], _ = _regression(c["m"], c["n"], seed)
        st["cols"], st["w"] = _columns(c, seed)
        st["g0"] = torch.zeros(c["m"], device="cuda", dtype=torch.float64)
    elif kind == "sweep":
        st["stream"] = torch.cuda.Stream()
        st["problems"] = [dict({k: v for k, v in p.items() if k != "gamma"}, k=B.kernel("rbf", gamma=p["gamma"]))
                          for p in _sweep(c, seed)]
    elif kind == "tolerance":
        A, y = _regression(c["m"], c["n"], seed)
        st["stream"] = torch.cuda.Stream()
        st["A"], st["y"] = A.cpu().pin_memory(), y.cpu().pin_memory()
    else:  # resident plans, on a stream of their own
        stream = st["stream"] = torch.cuda.Stream()
        if kind == "csr":
            ptr, cols, vals, y = _sparse(c, seed)
            A = B.Csr(ptr, cols, vals, c["n"])
        elif kind == "stress":
            A, y = _stress(c, seed)
            if c["prec"] == "fp8":
                A = B.Fp8(*_e4m3(A))
        else:
            A, y = _regression(c["m"], c["n"], seed)
            A = A.double() if c["prec"] == "fp64" else A
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            if kind == "csr":
                st["plan"] = B.Plan(0, A, y, st["kernel"], SVM_C[kind], 1, c["s"], BUDGET, seed=st["seed"],
                                    prec=c["prec"], loss=2, stream=stream.cuda_stream)
            else:
                st["plan"] = B.Plan(1, A, y, st["kernel"], LAMBDA[kind], c["b"], c["s"], BUDGET, seed=st["seed"],
                                    prec=c["prec"], stream=stream.cuda_stream)
    torch.cuda.synchronize()
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "svm":
        with torch.cuda.stream(state["stream"]):
            alpha, grad, _, _ = B.svm_solve(state["A"], state["y"], state["kernel"], c["loss"], SVM_C[kind], c["s"],
                                            c["H"], seed=state["seed"], prec=c["prec"])
        return {"alpha": alpha, "grad": grad}
    if kind == "sweep":
        with torch.cuda.stream(state["stream"]):
            alphas, grads, _, _ = B.krr_solve_batched(state["problems"], prec=c["prec"])
        return {"alpha": alphas, "grad": grads}
    if kind == "tolerance":
        alpha, grad, _, _ = B.krr_solve(state["A"].numpy(), state["y"].numpy(), state["kernel"], LAMBDA[kind], c["b"],
                                        c["s"], 400 * c["m"], seed=state["seed"], prec=c["prec"], tol=1e-6,
                                        check_every=max(1, 256 // c["s"]), flags=B.FLAG_HOST_IO | B.FLAG_REFRESH,
                                        stream=state["stream"].cuda_stream)
        return {"alpha": alpha, "grad": grad}
    if kind == "apply":
        g = state["g0"].clone()
        return {"f": B.kernel_block_apply(state["A"], state["kernel"], c["prec"], state["cols"], state["w"], g)}
    if kind == "block":
        return {"K": B.kernel_block(state["A"], state["kernel"], c["prec"], state["cols"])}
    plan = state["plan"]
    plan.run(c["steps"])
    return {"alpha": plan.alpha, "grad": plan.grad}


# -------------------------------------------------------------- the work ---
WIDTH = {"fp64": 8, "tf32": 4, "tf32x3": 8, "bf16x3": 4, "bf16": 2, "fp16": 2, "fp8": 1}


def work(case):
    """Each outer step (a kernel block of all rows against the step's) needs every row once, the vectors once a pass;
    two operations for each product of the block."""
    c, kind = case, case["kind"]
    if kind == "svm":
        steps = -(-c["H"] // c["s"])
        row = c["n"] * WIDTH[c["prec"]]
        fits = c["m"] * row < 100e6  # a matrix that stays in L2 is read from memory once
        return {"bytes": c["m"] * (row * (1 if fits else steps) + 24.0), "flops": 2.0 * c["m"] * c["n"] * c["H"]}
    if kind == "csr":
        width = 8 if c["prec"] == "fp64" else 4
        # the nonzeros that meet a sampled row, index and value, per step; the vectors once
        hits = c["m"] * c["nnz"] * min(1.0, c["s"] * c["nnz"] / c["n"])
        return {"bytes": c["steps"] * hits * (4 + width) + 24.0 * c["m"], "flops": 2.0 * c["steps"] * hits}
    if kind == "sweep":
        m = (c["m_lo"] + c["m_hi"]) / 2
        return {"bytes": c["count"] * m * (4.0 * c["n"] + 24), "flops": c["count"] * 2.0 * m * c["n"] * c["H"] * 20}
    if kind == "tolerance":
        # how often the rows are visited depends on the data: about 35 epochs
        return {"bytes": c["m"] * (4.0 * c["n"] + 24), "flops": 2.0 * c["m"] * c["n"] * 35 * c["m"]}
    if kind == "apply":
        return {"bytes": c["m"] * (4.0 * c["n"] + 16), "flops": 2.0 * c["m"] * c["n"] * min(c["m"], c["cols"])}
    if kind == "block":
        return {"bytes": c["m"] * 4.0 * (c["n"] + min(c["m"], c["cols"])),
                "flops": 2.0 * c["m"] * c["n"] * min(c["m"], c["cols"])}
    row = c["n"] * WIDTH[c["prec"]]
    fits = c["m"] * row < 100e6
    sb = c["s"] * c["b"]
    return {"bytes": c["m"] * (row * (1 if fits else c["steps"]) + 24.0),
            "flops": 2.0 * c["m"] * c["n"] * sb * c["steps"]}


# ------------------------------------------------- the iteration, 64 bits ---
_MASK = (1 << 64) - 1


def _splitmix(state, k):
    """Output k of the SplitMix64 sequence from `state` (Steele, Lea and Flood 2014)."""
    z = (state + k * 0x9E3779B97F4A7C15) & _MASK
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _MASK
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _MASK
    return z ^ (z >> 31)


def _coordinates(seed, m, count):
    start = _splitmix(seed & _MASK, 1)
    return [(_splitmix(start, t + 1) * m) >> 64 for t in range(count)]


def _blocks(seed, m, b, count):
    out = []
    for t in range(count):
        start, got = _splitmix(seed & _MASK, 2 * (t + 1) + 1), []
        for q in range(b):
            top = m - b + q
            r = (_splitmix(start, q + 1) * (top + 1)) >> 64
            got.append(top if r in got else r)
        out += got
    return out


def _k64(dots, ni, nj, args):
    """Kernel values from dot products and squared norms, in place where that helps."""
    kind, gamma, coef0, degree = args
    if kind == "rbf":
        d2 = dots.mul_(-2.0).add_(ni[:, None]).add_(nj[None, :])
        return d2.clamp_(min=0.0).mul_(-gamma).exp_()
    return dots if kind == "linear" else dots.add_(coef0).pow_(degree)


def _k_times(A, S, w, args, rows=8192):
    """K(A, A_S) w for all rows; A a function from a range of rows to their FP64 values."""
    AS, out, r = S, [], 0
    nS = AS.square().sum(1)
    while (a := A(r, r + rows)) is not None:
        out.append(_k64(a @ AS.T, a.square().sum(1), nS, args) @ w)
        r += rows
    return torch.cat(out)


def _krr64(A, m, y, args, lam, b, blocks, seed):
    """alpha and the gradient after `blocks` block updates from zero: the updates on the sampled rows alone, then
    the gradient of all."""
    S = _blocks(seed, m, b, blocks)
    uniq, inv = np.unique(np.array(S), return_inverse=True)
    pick = torch.from_numpy(uniq).cuda()
    AS = torch.cat([a[pick[(pick >= r) & (pick < r + 8192)] - r] for r in range(0, m, 8192)
                    for a in [A(r, r + 8192)]])
    nS = AS.square().sum(1)
    K = _k64(AS @ AS.T, nS, nS, args)
    if args[0] == "rbf":
        K.fill_diagonal_(1.0)
    K.div_(lam)
    K.diagonal().add_(float(m))
    g, al = -y[pick], torch.zeros(len(uniq), device="cuda", dtype=torch.float64)
    where = torch.from_numpy(inv.reshape(blocks, b)).cuda()
    G = K[where[:, :, None], where[:, None, :]]
    L = torch.linalg.cholesky(G)
    for t in range(blocks):
        ix = where[t]
        d = torch.cholesky_solve(-g[ix][:, None], L[t])[:, 0]
        al[ix] += d
        g += K[:, ix] @ d
    alpha = torch.zeros(m, device="cuda", dtype=torch.float64)
    alpha[pick] = al
    grad = _k_times(A, AS, al / lam, args) + m * alpha - y
    return {"alpha": alpha, "grad": grad}


def _svm_updates(K, y, S, C, loss):
    """The DCD updates on the rows K describes; their alpha (numpy)."""
    omega, top = (0.0, C) if loss == 1 else (0.5 / C, np.inf)
    Q = K * y[:, None] * y[None, :]
    al, g = np.zeros(len(y)), -np.ones(len(y))
    for i in S:
        eta = Q[i, i] + omega
        new = min(max(al[i] - g[i] / eta, 0.0), top)
        if new != al[i]:
            g += Q[i] * (new - al[i])
            g[i] += omega * (new - al[i])
            al[i] = new
    return al


def _rows(A, scale=None):
    def get(r0, r1):
        if r0 >= A.shape[0]:
            return None
        a = A[r0:r1]
        if scale is None:
            return a.double()
        return a.view(torch.float8_e4m3fn).to(torch.float32).double() * scale[r0:r1].double()[:, None]
    return get


def exact(case, seed):
    c, kind, args = case, case["kind"], _kernel_args(case)
    if kind == "svm":
        A, y = _blobs(c, seed)
        nA = A.square().sum(1)
        K = _k64(A @ A.T, nA, nA, args).fill_diagonal_(1.0)
        yn = y.cpu().numpy()
        al = torch.from_numpy(_svm_updates(K.cpu().numpy(), yn, _coordinates(int(seed), c["m"], c["H"]), 1.0,
                                           c["loss"])).cuda()
        omega = 0.0 if c["loss"] == 1 else 0.5
        return {"alpha": al, "grad": y * (K @ (y * al)) - 1.0 + omega * al}
    if kind == "csr":
        ptr, cols, vals, y = _sparse(c, seed)
        m, n, C = c["m"], c["n"], SVM_C[kind]
        S = np.array(_coordinates(int(seed), m, c["s"] * c["steps"]))
        uniq, inv = np.unique(S, return_inverse=True)
        pick = torch.from_numpy(uniq).cuda()
        cols2, vals2 = cols.view(m, -1).long(), vals.view(m, -1).double()
        AS = torch.zeros(len(uniq), n, device="cuda", dtype=torch.float64)
        AS.scatter_(1, cols2[pick], vals2[pick])
        T = AS.T.contiguous()

        def dots(c2, v2):
            out = torch.zeros(c2.shape[0], len(uniq), device="cuda", dtype=torch.float64)
            for q in range(c2.shape[1]):
                out += v2[:, q, None] * T[c2[:, q]]
            return out

        K = _k64(dots(cols2[pick], vals2[pick]), None, None, args)
        ys = y[pick]
        al = torch.from_numpy(_svm_updates(K.cpu().numpy(), ys.cpu().numpy(), inv.reshape(-1), C, 2)).cuda()
        Kw = torch.cat([_k64(dots(cols2[r:r + 8192], vals2[r:r + 8192]), None, None, args) @ (ys * al)
                        for r in range(0, m, 8192)])
        alpha = torch.zeros(m, device="cuda", dtype=torch.float64)
        alpha[pick] = al
        return {"alpha": alpha, "grad": y * Kw - 1.0 + 0.5 / C * alpha}
    if kind == "sweep":
        probs = _sweep(c, seed)
        got = [_krr64(_rows(p["A"]), p["A"].shape[0], p["y"], ("rbf", p["gamma"], 0.0, 2), p["lam"], p["b"], p["H"],
                      p["seed"]) if i < 6 else {"alpha": None, "grad": None} for i, p in enumerate(probs)]
        return {k: [g[k] for g in got] for k in ("alpha", "grad")}
    if kind == "tolerance":  # the solution that the solve stops near; its gradient is zero
        A, y = _regression(c["m"], c["n"], seed)
        A = A.double()
        nA = A.square().sum(1)
        K = _k64(A @ A.T, nA, nA, args).fill_diagonal_(1.0).div_(LAMBDA[kind])
        K.diagonal().add_(float(c["m"]))
        return {"alpha": torch.cholesky_solve(y[:, None], torch.linalg.cholesky(K))[:, 0], "grad": None}
    if kind in ("apply", "block"):
        A, _ = _regression(c["m"], c["n"], seed)
        cols, w = _columns(c, seed)
        AS = A[cols.long()].double()
        if kind == "apply":
            return {"f": _k_times(_rows(A), AS, w, args)}
        A = A.double()
        return {"K": _k64(A @ AS.T, A.square().sum(1), AS.square().sum(1), args)}
    if kind == "stress":
        A, y = _stress(c, seed)
        rows = _rows(*_e4m3(A)) if c["prec"] == "fp8" else _rows(A)
    else:
        A, y = _regression(c["m"], c["n"], seed)
        rows = _rows(A)
    return _krr64(rows, c["m"], y, args, LAMBDA[kind], c["b"], c["s"] * c["steps"], int(seed))
