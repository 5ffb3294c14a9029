"""What a user of this library has it do, as cases that can be timed: analyses of every
precision and variant from a 40-variable cycling problem to a 1024 x 1024 grid, a batch of
uneven problems, and the training step of the learned warm start.

listed() names the fixed cases, draw(rng) gives one more of the same ranges, prepare(case,
seed) makes the inputs and the handle a program keeps, run(state) is one pass through the
public entry points and returns its outputs whole, work(case) is what a pass cannot do
without, and exact(case, seed) is the same result from plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2606_19224_gb300 as enkf


# ------------------------------------------------------------------ the cases
def _grf(name, side, N, m, ell, r_lo, r_hi, precision, **kw):
    """An analysis of a Gaussian random field ensemble on a side x side grid."""
    c = dict(name=name, kind="grf", side=side, N=N, m=m, ell=float(ell), r_lo=r_lo, r_hi=r_hi, precision=precision,
             variant="cgd", precondition=1, reduce_order=0, tol=1e-8, weights=1)
    c.update(kw)
    return c


def listed():
    return [
        # one cycle of a Lorenz-96 twin experiment, the smallest call: launch and latency bound
        dict(name="l96_fp64", kind="l96", n=40, N=20, every=2, tol=1e-10),
        # the benchmark workload in its fastest mode: 512 x 512 field, 64 members, 65,536 point
        # observations, FP16 contractions with refinement
        _grf("grf512_n64_fp16", 512, 64, 65536, 16, 0.5, 1.5, "fp16", reduce_order=1),
        # the same analysis in the product's default single precision, bitwise repeatable
        _grf("grf512_n64_fp32", 512, 64, 65536, 16, 0.5, 1.5, "fp32"),
        # the paper's plain CG in FP32 with an odd ensemble size, ragged rows and a general
        # operator (one to three weighted entries per observation)
        _grf("csr_n37_fp32_plain", 101, 37, 3001, 6, 0.5, 1.5, "fp32", precondition=0, weights=3),
        # the paper's plain CG in FP64, the library's default configuration, on a 256 x 256 field
        _grf("grf256_n64_fp64_plain", 256, 64, 16384, 8, 0.5, 1.5, "fp64", precondition=0),
        # the mixed-precision workload: 1024 x 1024 field, 128 members, 262,144 observations
        _grf("grf1024_n128_bf16", 1024, 128, 262144, 24, 0.25, 1.0, "bf16"),
        # the same workload in single precision, the largest analysis
        _grf("grf1024_n128_fp32", 1024, 128, 262144, 24, 0.25, 1.0, "fp32"),
        # many independent analyses of uneven shape in one launch (an ensemble of regions or of
        # experiments): n from 4,096 to 262,144, N of 16 to 128
        dict(name="batch48", kind="batch", count=48, n_lo=4096, n_hi=262144, shapes=1),
        # the reduced form of the method on the benchmark workload
        _grf("grf512_n64_reduced", 512, 64, 65536, 16, 0.5, 1.5, "fp32", variant="reduced"),
        # correlated observation noise (tridiagonal R, H = I) in FP64, the paper's Example 2b
        dict(name="tridiag_p10000_fp64", kind="tridiag", p=10000, N=100, tol=1e-13),
        # an analysis from the learned start, as a cycling program with a trained model runs it
        dict(name="warm_n64_fp32", kind="warm", side=512, N=64, m=65536, ell=16.0, K=1024, hidden=512, layers=3),
        # one training step of that model: loss and gradient of a minibatch
        dict(name="mlp_grad_b256", kind="mlp", batch=256, K=1024, N=64, hidden=512, layers=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["l96", "refine", "refine", "refine", "plain32", "fp64", "batch", "gram", "tridiag", "warm", "mlp"])
    N = _log_int(rng, 8, 128)
    if kind == "l96":
        return dict(kind="l96", n=4 * _log_int(rng, 10, 100), N=_log_int(rng, 10, 64), every=rng.choice([1, 2, 4]), tol=1e-10)
    if kind in ("refine", "gram"):
        side = _log_int(rng, 48, 1024 if N <= 100 else 700)
        c = _grf("", side, N, max(16, int(side * side * rng.uniform(0.1, 0.25))), rng.uniform(0.015, 0.06) * side,
                 rng.choice([0.25, 0.5]), rng.choice([1.0, 1.5]), "fp32", weights=rng.choice([1, 1, 2]))
        if kind == "refine":
            c.update(precision=rng.choice(["fp32", "fp16", "bf16"]), reduce_order=rng.choice([0, 1]))
        else:
            c.update(variant=rng.choice(["reduced", "senkf"]), precision=rng.choice(["fp32", "fp64"]) if side < 400 else "fp32")
    elif kind in ("plain32", "fp64"):
        side = _log_int(rng, 40, 200)
        c = _grf("", side, N, max(16, int(side * side * rng.uniform(0.1, 0.25))), rng.uniform(0.03, 0.06) * side,
                 0.5, 1.5, "fp32" if kind == "plain32" else "fp64", weights=rng.choice([1, 2, 3]),
                 precondition=0 if kind == "plain32" else rng.choice([0, 1]))
    elif kind == "batch":
        lo = _log_int(rng, 1024, 8192)
        return dict(kind="batch", count=rng.randint(5, 48), n_lo=lo, n_hi=lo * rng.randint(4, 24), shapes=rng.randint(2, 1 << 20))
    elif kind == "tridiag":
        return dict(kind="tridiag", p=_log_int(rng, 500, 12000), N=N, tol=1e-13)
    elif kind == "warm":
        side = _log_int(rng, 64, 512)
        return dict(kind="warm", side=side, N=N, m=side * side // 4, ell=rng.uniform(0.025, 0.05) * side, K=rng.choice([128, 500, 1024]),
                    hidden=rng.choice([128, 512]), layers=rng.randint(2, 3))
    else:
        return dict(kind="mlp", batch=_log_int(rng, 32, 256), K=_log_int(rng, 100, 1024), N=N, hidden=rng.choice([128, 300, 512]),
                    layers=rng.randint(1, 3))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _fields(side, ell, count, gen, chunk=32):
    """`count` periodic fields of unit variance and covariance exp(-d^2 / (2 ell^2)) on a
    side x side grid by circulant embedding, [side^2][count] in FP32."""
    k = torch.arange(side, device="cuda", dtype=torch.float64)
    d = torch.minimum(k, side - k)
    lam = torch.fft.fft(torch.exp(-d * d / (2.0 * ell * ell))).real.clamp_min(0.0)
    root = torch.sqrt(torch.outer(lam, lam[: side // 2 + 1]))
    out = torch.empty((side * side, count), dtype=torch.float32, device="cuda")
    for c0 in range(0, count, chunk):
        c = min(chunk, count - c0)
        w = torch.randn((c, side, side), generator=gen, device="cuda", dtype=torch.float64)
        x = torch.fft.irfft2(torch.fft.rfft2(w) * root, s=(side, side))
        out[:, c0:c0 + c] = x.reshape(c, side * side).T
    return out


def _operator(n, m, weights, gen):
    """m observations of n grid points: distinct points in ascending order with weight 1, or
    rows of one to `weights` entries with random weights. CSR arrays on the host."""
    if weights == 1:
        col = torch.sort(torch.randperm(n, generator=gen, device="cuda")[:m]).values
        return np.arange(m + 1, dtype=np.int32), col.cpu().numpy().astype(np.int32), np.ones(m)
    per = torch.randint(1, weights + 1, (m,), generator=gen, device="cuda")
    rowptr = np.zeros(m + 1, dtype=np.int32)
    rowptr[1:] = torch.cumsum(per, 0).cpu().numpy()
    nnz = int(rowptr[-1])
    col = torch.randint(0, n, (nnz,), generator=gen, device="cuda").cpu().numpy().astype(np.int32)
    w = (0.2 + torch.rand((nnz,), generator=gen, device="cuda", dtype=torch.float64)).cpu().numpy()
    return rowptr, col, w


def _observe(truth, op, r, gen):
    rowptr, col, w = op
    rows = torch.from_numpy(np.repeat(np.arange(rowptr.size - 1), np.diff(rowptr))).cuda()
    hx = torch.zeros(rowptr.size - 1, dtype=torch.float64, device="cuda")
    hx.index_add_(0, rows, torch.from_numpy(w).cuda() * truth[torch.from_numpy(col.astype(np.int64)).cuda()])
    return hx + torch.sqrt(r) * torch.randn(r.shape, generator=gen, device="cuda", dtype=torch.float64)


def _field_problem(c, seed, dtype):
    """Forecast ensemble, operator, variances of R and observation of one analysis."""
    side, N, m = c["side"], c["N"], c["m"]
    X = _fields(side, c["ell"], N + 1, _gen(seed, 1))
    truth = X[:, N].double()
    X = X[:, :N].contiguous().to(dtype)
    op = _operator(side * side, m, c.get("weights", 1), _gen(seed, 2))
    lo, hi = c.get("r_lo", 0.5), c.get("r_hi", 1.5)
    r = lo + (hi - lo) * torch.rand((m,), generator=_gen(seed, 3), device="cuda", dtype=torch.float64)
    return X, op, r, _observe(truth, op, r, _gen(seed, 4))


def _l96_step(x, dt, steps):
    f = lambda v: (torch.roll(v, -1, 0) - torch.roll(v, 2, 0)) * torch.roll(v, 1, 0) - v + 8.0  # noqa: E731
    for _ in range(steps):
        k1 = f(x)
        k2 = f(x + 0.5 * dt * k1)
        k3 = f(x + 0.5 * dt * k2)
        k4 = f(x + dt * k3)
        x = x + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return x


def _l96_problem(c, seed):
    """A Lorenz-96 forecast of a truth plus unit noise and every k-th variable observed, R = I."""
    n, N = c["n"], c["N"]
    g = _gen(seed, 5)
    truth = _l96_step(8.0 + torch.randn((n, 1), generator=g, device="cuda", dtype=torch.float64), 0.05, 40)
    X = truth + torch.randn((n, N), generator=g, device="cuda", dtype=torch.float64)
    X, truth = _l96_step(X, 0.05, 5), _l96_step(truth, 0.05, 5)
    col = np.arange(0, n, c["every"], dtype=np.int32)
    op = (np.arange(col.size + 1, dtype=np.int32), col, np.ones(col.size))
    r = torch.ones(col.size, dtype=torch.float64, device="cuda")
    return X.contiguous(), op, r, _observe(truth[:, 0], op, r, g)


def _tridiag_problem(c, seed, sigma=0.3, rho=0.2):
    """Example 2b: an FP64 Lorenz-96 ensemble, H = I, R tridiagonal with sigma^2 on the diagonal
    and sigma^2 rho beside it."""
    p, N = c["p"], c["N"]
    g = _gen(seed, 6)
    truth = _l96_step(torch.randn((p, 1), generator=g, device="cuda", dtype=torch.float64), 0.01, 20)
    X = truth + 0.1 * torch.randn((p, N), generator=g, device="cuda", dtype=torch.float64)
    X, truth = _l96_step(X, 0.01, 1), _l96_step(truth, 0.01, 1)
    op = (np.arange(p + 1, dtype=np.int32), np.arange(p, dtype=np.int32), np.ones(p))
    r = np.full(p, sigma * sigma)
    off = np.full(p - 1, sigma * sigma * rho)
    xi = torch.randn((p,), generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    d, e = _bidiagonal(r, off)
    v = d * xi
    v[1:] += e * xi[:-1]
    return X.contiguous(), op, r, off, truth[:, 0] + torch.from_numpy(v).cuda()


def _bidiagonal(r, off):
    """Diagonal and subdiagonal of L with L L^T the tridiagonal R."""
    d, e = np.empty(r.size), np.empty(r.size - 1)
    d[0] = math.sqrt(r[0])
    for i in range(1, r.size):
        e[i - 1] = off[i - 1] / d[i - 1]
        d[i] = math.sqrt(r[i] - e[i - 1] ** 2)
    return d, e


def _batch_specs(c):
    rng = np.random.default_rng(c["shapes"])
    specs = []
    for _ in range(c["count"]):
        side = int(round(math.sqrt(math.exp(rng.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]))))))
        specs.append(dict(side=side, N=int(rng.choice((16, 32, 64, 128))), m=side * side // 4, ell=float(rng.uniform(4.0, 32.0))))
    return specs


def _mlp_params(c, seed, scale=1.0):
    """Weights of the size that training starts from, and the features' standardisation."""
    g = _gen(seed, 7)
    dims = [c["K"] + c["N"]] + [c["hidden"]] * c["layers"] + [c["N"]]
    parts = []
    for fi, fo in zip(dims[:-1], dims[1:]):
        parts += [torch.randn((fo * fi,), generator=g, device="cuda") * (scale * math.sqrt(2.0 / fi)), torch.zeros(fo, device="cuda")]
    for d in (dims[0], dims[-1]):
        parts += [0.1 * torch.randn((d,), generator=g, device="cuda"), 0.5 + torch.rand((d,), generator=g, device="cuda")]
    return tuple([dims[0], c["hidden"], c["layers"], c["N"]]), torch.cat(parts)


def _mlp_data(c, seed):
    g = _gen(seed, 8)
    rows = 4 * c["batch"]
    X = torch.randn((rows, c["K"] + c["N"]), generator=g, device="cuda")
    T = torch.randn((rows, c["N"]), generator=g, device="cuda")
    pick = torch.randperm(rows, generator=g, device="cuda")[: c["batch"]].to(torch.int32)
    return X, T, pick


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(kind=kind, seed=int(seed) & 0x7FFFFFFF, counter=int(seed) % 7)
    if kind == "mlp":
        s["shape"], s["params"] = _mlp_params(c, seed)
        s["X"], s["T"], s["rows"] = _mlp_data(c, seed)
        return s
    if kind == "batch":
        specs = _batch_specs(c)
        probs = [_field_problem(p, 97 * seed + i, torch.float32) for i, p in enumerate(specs)]
        s["Xf"], s["y"] = [p[0] for p in probs], [p[3] for p in probs]
        s["seeds"] = [s["seed"] + i for i in range(len(probs))]
        s["an"] = enkf.BatchAnalysis([dict(n=p[0].shape[0], m=p[2].numel(), N=p[0].shape[1], rowptr=p[1][0], col=p[1][1],
                                           w=p[1][2], r=p[2].cpu().numpy()) for p in probs])
        return s
    if kind == "tridiag":
        X, op, r, off, y = _tridiag_problem(c, seed)
        an = enkf.Analysis(c["p"], c["p"], c["N"], *op, r, r_off=off, precision="fp64", variant="reduced", tol=c["tol"])
    elif kind == "l96":
        X, op, r, y = _l96_problem(c, seed)
        an = enkf.Analysis(c["n"], r.numel(), c["N"], *op, r.cpu().numpy(), precision="fp64", tol=c["tol"])
    elif kind == "warm":
        X, op, r, y = _field_problem(c, seed, torch.float32)
        an = enkf.Analysis(c["side"] ** 2, c["m"], c["N"], *op, r.cpu().numpy(), precision="fp32", precondition=1, tol=1e-8, warm_start=1)
        shape, params = _mlp_params(c, seed, 0.3)
        an.set_warm_model(shape, params)
    else:
        X, op, r, y = _field_problem(c, seed, torch.float64 if c["precision"] == "fp64" else torch.float32)
        kw = dict(precondition=c["precondition"], reduce_order=c["reduce_order"]) if c["variant"] == "cgd" else {}
        an = enkf.Analysis(c["side"] ** 2, c["m"], c["N"], *op, r.cpu().numpy(), precision=c["precision"], variant=c["variant"],
                           tol=c["tol"], **kw)
    s.update(an=an, Xf=X, y=y)
    return s


def run(state):
    s = state
    if s["kind"] == "mlp":
        loss, grad = enkf.mlp_loss_grad(s["shape"], s["params"], s["X"], s["T"], rows=s["rows"])
        return dict(loss=loss, grad=grad)
    if s["kind"] == "batch":
        return s["an"].analyze(s["Xf"], s["y"], s["seeds"])
    return s["an"].analyze(s["Xf"], s["y"], seed=s["seed"], counter=s["counter"])


# ------------------------------------------------------------------ what a pass cannot do without
def _analysis_work(n, m, N, size, nnz):
    """X_f and the operator, R and y read once, X_a written once; the two tall products of the
    observed anomalies (with themselves and with the innovations) and the update."""
    return 2 * n * N * size + 16 * m + 12 * nnz, 4.0 * m * N * N + 2.0 * n * N * N


def work(case):
    c, kind = case, case["kind"]
    if kind == "mlp":
        dims = [c["K"] + c["N"]] + [c["hidden"]] * c["layers"] + [c["N"]]
        pairs = [a * b for a, b in zip(dims[:-1], dims[1:])]
        count = sum(pairs) + sum(dims[1:])
        return dict(bytes=4 * (2 * count + c["batch"] * (dims[0] + dims[-1])), flops=2.0 * c["batch"] * (3 * sum(pairs) - pairs[0]))
    if kind == "batch":
        each = [_analysis_work(p["side"] ** 2, p["m"], p["N"], 4, p["m"]) for p in _batch_specs(c)]
        return dict(bytes=sum(b for b, _ in each), flops=sum(f for _, f in each))
    if kind == "l96":
        m = -(-c["n"] // c["every"])
        b, f = _analysis_work(c["n"], m, c["N"], 8, m)
    elif kind == "tridiag":
        b, f = _analysis_work(c["p"], c["p"], c["N"], 8, c["p"])
    else:
        size = 8 if c.get("precision") == "fp64" else 4
        b, f = _analysis_work(c["side"] ** 2, c["m"], c["N"], size, c["m"] * (c.get("weights", 1) + 1) / 2)
        if kind == "warm":
            dims = [c["K"] + c["N"]] + [c["hidden"]] * c["layers"] + [c["N"]]
            count = sum(a * d for a, d in zip(dims[:-1], dims[1:]))
            b, f = b + 4 * count, f + 2.0 * c["N"] * count
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------ the same results in 64 bits
def _philox_normals(m, N, seed, counter):
    """The analysis's perturbation stream: Philox4x32-10 at counter (i, j >> 1, counter lo, hi)
    under key (seed lo, hi), two 53-bit uniforms, Box-Muller (cos for even j, sin for odd)."""
    mask = 0xFFFFFFFF
    half = (N + 1) // 2
    c0 = torch.arange(m, device="cuda", dtype=torch.int64)[:, None].expand(m, half)
    c1 = torch.arange(half, device="cuda", dtype=torch.int64)[None, :].expand(m, half)
    c2, c3 = torch.full_like(c0, counter & mask), torch.full_like(c0, (counter >> 32) & mask)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57   # modulo 2^64: both halves are exact
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
    u1 = (((c0 << 21) | (c1 >> 11)).double() + 0.5) * 2.0 ** -53
    u2 = ((c2 << 21) | (c3 >> 11)).double() * 2.0 ** -53
    rho, ang = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
    return torch.stack([rho * torch.cos(ang), rho * torch.sin(ang)], dim=2).reshape(m, 2 * half)[:, :N]


def _exact_analysis(X, op, r, y, seed, counter, senkf=False, off=None):
    """X_f + A HA^T (HA HA^T / (N-1) + R)^{-1} D / (N-1) through the N x N identity (or Algorithm 3,
    the diagonal inverse), all in FP64."""
    X = X.double()
    n, N = X.shape
    rowptr, col, w = op
    m = rowptr.size - 1
    cols = torch.from_numpy(col.astype(np.int64)).cuda()
    if col.size == m and np.all(np.diff(rowptr) == 1):
        Zo = X[cols] * torch.from_numpy(w).cuda()[:, None]
    else:
        rows = torch.from_numpy(np.repeat(np.arange(m), np.diff(rowptr))).cuda()
        Zo = torch.zeros((m, N), dtype=torch.float64, device="cuda")
        Zo.index_add_(0, rows, torch.from_numpy(w).cuda()[:, None] * X[cols])
    zbar = Zo.mean(1, keepdim=True)
    HA = Zo - zbar
    xi = _philox_normals(m, N, seed, counter)
    if off is not None:   # whiten the rows with L L^T = R; E = L xi
        d, e = _bidiagonal(r, off)
        B = torch.cat([HA, y[:, None] - zbar], 1).cpu().numpy()
        B[0] /= d[0]
        for i in range(1, m):
            B[i] = (B[i] - e[i - 1] * B[i - 1]) / d[i]
        B = torch.from_numpy(B).cuda()
        HA, D = B[:, :N].contiguous(), B[:, N:] - B[:, :N] + xi
        r = torch.ones(m, dtype=torch.float64, device="cuda")
    else:
        D = y[:, None] - Zo + torch.sqrt(r)[:, None] * xi
    A = X - X.mean(1, keepdim=True)
    if senkf:
        s = (HA * HA).sum(1) + (N - 1) * r
        return X + A @ (HA.T @ (D / s[:, None]))
    G = HA.T @ (HA / r[:, None]) / (N - 1) + torch.eye(N, dtype=torch.float64, device="cuda")
    F = HA.T @ (D / r[:, None]) / (N - 1)
    return X + A @ torch.linalg.solve(G, F)


def _exact_mlp(c, seed):
    shape, params = _mlp_params(c, seed)
    X, T, rows = _mlp_data(c, seed)
    dims = [shape[0]] + [shape[1]] * shape[2] + [shape[3]]
    P = params.double().requires_grad_(True)
    at, layers = 0, []
    for fi, fo in zip(dims[:-1], dims[1:]):
        layers.append((P[at:at + fo * fi].view(fo, fi), P[at + fo * fi:at + fo * fi + fo]))
        at += fo * fi + fo
    tail = params[at:].double()
    mu_in, sd_in, mu_out, sd_out = torch.split(tail, [dims[0], dims[0], dims[-1], dims[-1]])
    h = (X[rows.long()].double() - mu_in) / sd_in
    for l, (W, b) in enumerate(layers):
        h = h @ W.T + b
        if l < len(layers) - 1:
            h = torch.nn.functional.gelu(h)
    loss = ((h - (T[rows.long()].double() - mu_out) / sd_out) ** 2).mean()
    grad, = torch.autograd.grad(loss, P)
    return dict(loss=loss.detach().reshape(1), grad=grad)


def exact(case, seed):
    c, kind = case, case["kind"]
    key, counter = int(seed) & 0x7FFFFFFF, int(seed) % 7
    if kind == "mlp":
        return _exact_mlp(c, seed)
    if kind == "batch":
        out = []
        for i, p in enumerate(_batch_specs(c)):
            X, op, r, y = _field_problem(p, 97 * seed + i, torch.float32)
            out.append(_exact_analysis(X, op, r, y, key + i, 0))
        return out
    if kind == "tridiag":
        X, op, r, off, y = _tridiag_problem(c, seed)
        return _exact_analysis(X, op, r, y, key, counter, off=off)
    if kind == "l96":
        X, op, r, y = _l96_problem(c, seed)
    else:
        X, op, r, y = _field_problem(c, seed, torch.float64 if c.get("precision") == "fp64" else torch.float32)
    return _exact_analysis(X, op, r, y, key, counter, senkf=c.get("variant") == "senkf")
