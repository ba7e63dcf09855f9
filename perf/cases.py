"""The work that a user of this framework has it do, as cases that can be timed.

Three kinds of cases: the building blocks of Algorithm 1 (the gradient passes, the sketches, AAb_Solver, the
backward pass), each through its own entry point; the gradient of the dual form; and two whole calls (sketch, then a
refined solve; sketch, λ-paths and their refinement for a batch of problems).  Sizes are those of the benchmark, the
workloads module and the tests, with ragged ones among them.

Iterations are compared number by number, so the cases are posed where the numbers are fixed by the inputs and not by
the path that rounding takes: a single AAb_Solver call runs a fixed number of passes on a sketch with condition
κ(SAᵀSA + λI) ≈ 10 (Algorithm 5 does not reorthogonalise: at κ ≫ 10³ two fp32 runs with different summation orders
part after a dozen passes), and the whole calls end in the compensated refinement, whose fixed point is x* itself.

Every matrix is A = G·diag(σ)·Vᵀ/√n with G Gaussian and V orthogonal, b = A·x0 + noise, drawn on the GPU.
"""
import math

import torch

from paper_1912_03514_gb300 import mihs

DEV = "cuda"


def listed():
    return [
        # The 4096×256 problem of the benchmark: one gradient of 4 MB, all launches and latency.
        dict(name="gradient-4096x256", kind="gradient", n=4096, d=256, pad=0),
        # The gradient of the dual form (wide matrices, n ≤ d) at the benchmark's n, d ragged.
        dict(name="dual-gradient-2000x200001", kind="dual", n=2000, d=200001),
        # The gradients of a 16-value λ-path in one pass, a middling matrix of the batched workload.
        dict(name="path-gradient-65536x512", kind="path", n=65536, d=512, nl=16),
        # The compensated gradient of refinement solves, at the benchmark's size.
        dict(name="refined-gradient-262144x1024", kind="refined", n=262144, d=1024),
        # The three sketch families: once per matrix and solve.  Gaussian and CountSketch at the benchmark's
        # size, SRHT at an n that is not a power of two (its usual case) with d = 1000.
        dict(name="gaussian-262144x1024", kind="sketch", family="gaussian", prec="fp32", n=262144, d=1024, m=588),
        dict(name="countsketch-262144x1024", kind="sketch", family="countsketch", prec="fp32", n=262144, d=1024,
             m=588),
        dict(name="srht-200000x1000", kind="sketch", family="srht", prec="fp32", n=200000, d=1000, m=600),
        # The inner solver: a sketch that one thread-block cluster holds (the benchmark's 588×1024) and the
        # largest of the mixed-precision workload (3076×2048), which is spread over the whole GPU.
        dict(name="aab-588x1024", kind="aab", prec="fp32", m=588, d=1024, passes=30),
        dict(name="aab-3076x2048", kind="aab", prec="fp32", m=3076, d=2048, passes=30),
        # The pass that differentiates the solution, for 1000 features and an intercept: rows that are not
        # a multiple of 16 bytes.
        dict(name="backward-200003x1001", kind="backward", n=200003, d=1001),
        # Whole call: a new matrix arrives, is sketched and solved with refinement to 1e-12.
        dict(name="solve-262144x1024", kind="solve", family="countsketch", n=262144, d=1024, m=588, power=1.0,
             lam=1e-4, tol=1e-12),
        # Whole call: λ-paths of a batch of problems in fp32, then every λ refined.
        dict(name="batch-4x32768x256", kind="batch", count=4, n=32768, d=256, nl=8, decades=3.0, tol=1e-11),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A number of columns: one of the usual powers of two, or anything between."""
    if rng.random() < 0.4:
        return rng.choice([w for w in (64, 128, 256, 512, 1024, 2048) if lo <= w <= hi])
    return _log(rng, lo, hi)


def _rows(rng, lo, hi, d, most):
    """A number of rows, log-uniform, such that the matrix has at most `most` elements."""
    return max(d, min(_log(rng, lo, hi), most // d))


def draw(rng):
    kind = rng.choice(["gradient", "gradient", "dual", "path", "refined", "sketch", "sketch", "sketch", "aab", "aab",
                       "backward", "solve", "batch"])
    big = 1 << 28  # elements: 1 GB
    if kind == "gradient":
        d = _width(rng, 64, 2048)
        return dict(kind=kind, n=_rows(rng, 4096, 262144, d, big), d=d, pad=rng.choice([0, 0, 4]))
    if kind == "dual":
        n = _log(rng, 128, 2048)
        return dict(kind=kind, n=n, d=max(n, _log(rng, 8192, 262144)))
    if kind == "path":
        d = _width(rng, 64, 1024)
        return dict(kind=kind, n=_rows(rng, 8192, 262144, d, big // 4), d=d, nl=rng.choice([4, 9, 16, 16]))
    if kind == "refined":
        d = _width(rng, 64, 1024)
        return dict(kind=kind, n=_rows(rng, 8192, 262144, d, big), d=d)
    if kind == "sketch":
        d = _width(rng, 64, 1024)
        n = _rows(rng, 8192, 262144, d, big)
        family = rng.choice(["gaussian", "countsketch", "srht"])
        prec = rng.choice(["fp32", "fp32", "bf16", "fp8"]) if family == "gaussian" else "fp32"
        return dict(kind=kind, family=family, prec=prec, n=n, d=d, m=_log(rng, 32, min(1024, 2 * d)))
    if kind == "aab":
        d = _width(rng, 128, 2048)
        return dict(kind=kind, prec=rng.choice(["fp32", "fp32", "bf16", "fp8"]), d=d, m=_log(rng, d // 2, 3 * d // 2),
                    passes=30)
    if kind == "backward":
        d = _width(rng, 64, 1024)
        return dict(kind=kind, n=_rows(rng, 8192, 200003, d, 200 << 20), d=d)
    if kind == "solve":
        d = _width(rng, 128, 1024)
        power = rng.choice([1.0, 1.5])
        lam = rng.choice([1e-4, 1e-3])
        sd = sum(1.0 / (1.0 + lam * i ** (2.0 * power)) for i in range(1, d + 1))
        m = int(math.ceil(4 * sd / 4)) * 4
        return dict(kind=kind, family=rng.choice(["gaussian", "countsketch", "srht"]),
                    n=max(4 * m, _rows(rng, 8192, 262144, d, big)), d=d, m=m, power=power, lam=lam, tol=1e-12)
    d = _width(rng, 64, 256)
    return dict(kind=kind, count=rng.choice([2, 3, 4]), n=_log(rng, 8192, 32768), d=d, nl=rng.choice([4, 8]),
                decades=rng.choice([2.0, 3.0]), tol=1e-11)


# ------------------------------------------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & (2**63 - 1))


def _orth(d, g):
    q, r = torch.linalg.qr(torch.randn(d, d, generator=g, device=DEV))
    return q * torch.sign(torch.diagonal(r))


def _pitch(d, pad=0):
    return (d + 3) // 4 * 4 + pad


def _rows_of(n, d, sigma, g, pad=0):
    """A (n × d, row pitch a multiple of 4) = G·diag(σ)·Vᵀ/√n."""
    basis = (sigma.unsqueeze(1) * _orth(d, g).t()) / math.sqrt(n)
    full = torch.zeros(n, _pitch(d, pad), device=DEV)
    for r in range(0, n, 1 << 16):
        e = min(n, r + (1 << 16))
        full[r:e, :d] = torch.randn(e - r, d, generator=g, device=DEV) @ basis
    return full[:, :d]


def _exponential(d, decades):
    return 10.0 ** (-decades * torch.arange(d, device=DEV, dtype=torch.float32) / max(d - 1, 1))


def _polynomial(d, power):
    return torch.arange(1, d + 1, device=DEV, dtype=torch.float32) ** (-power)


def _ridge(n, d, sigma, g, pad=0, snr_db=40.0):
    A = _rows_of(n, d, sigma, g, pad)
    x0 = torch.randn(d, generator=g, device=DEV)
    b = A @ x0
    w = torch.randn(n, generator=g, device=DEV)
    b = b + w * (b.norm() / w.norm() / 10.0 ** (snr_db / 20.0))
    return A, b, x0


def _lambdas(nl):
    """nl values, log-spaced over [1e-4, 1e-1]."""
    return [10.0 ** (-4.0 + 3.0 * i / max(nl - 1, 1)) for i in range(nl)]


def _sds(sigma, lams):
    s2 = sigma.double() ** 2
    return [float((s2 / (s2 + lam)).sum()) for lam in lams]


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    st = dict(case=case, seed=int(seed))
    if kind == "gradient":
        A, b, x0 = _ridge(case["n"], case["d"], _polynomial(case["d"], 1.0), g, case["pad"])
        st.update(A=A, b=b, x=0.5 * x0, lam=1e-2)
    elif kind == "dual":
        n, d = case["n"], case["d"]
        A = torch.zeros(n, _pitch(d), device=DEV)[:, :d]
        scale = _polynomial(n, 0.5) / math.sqrt(d)
        for r in range(0, n, 256):
            e = min(n, r + 256)
            A[r:e] = torch.randn(e - r, d, generator=g, device=DEV) * scale[r:e].unsqueeze(1)
        st.update(A=A, b=torch.randn(n, generator=g, device=DEV), nu=torch.randn(n, generator=g, device=DEV),
                  lam=1e-2)
    elif kind == "path":
        A, b, x0 = _ridge(case["n"], case["d"], _polynomial(case["d"], 1.0), g)
        X = torch.randn(case["nl"], case["d"], generator=g, device=DEV) * 0.3 + 0.5 * x0
        st.update(A=A, b=b, X=X, lams=_lambdas(case["nl"]))
    elif kind == "refined":
        A, b, x0 = _ridge(case["n"], case["d"], _polynomial(case["d"], 1.0), g)
        x = x0.double() + 1e-3 * torch.randn(case["d"], generator=g, device=DEV, dtype=torch.float64)
        st.update(A=A, b=b, x=x, lam=1e-4)
    elif kind == "sketch":
        st.update(A=_rows_of(case["n"], case["d"], _polynomial(case["d"], 1.0), g))
    elif kind == "aab":
        m, d = case["m"], case["d"]
        sigma, V = _exponential(d, 2.0), _orth(d, g)
        SA = torch.zeros(m, _pitch(d), device=DEV)[:, :d]
        SA.copy_((torch.randn(m, d, generator=g, device=DEV) / math.sqrt(m) * sigma) @ V.t())
        rhs = V @ (sigma**2 * torch.randn(d, generator=g, device=DEV))
        rhs = rhs + 0.01 * (V @ (sigma * torch.randn(d, generator=g, device=DEV)))
        st.update(SA=SA, g=rhs, lam=0.1)
        if case["prec"] != "fp32":
            st["q"], st["scales"] = mihs.quantize_sa(SA, case["prec"])
    elif kind == "backward":
        A, b, x0 = _ridge(case["n"], case["d"], _polynomial(case["d"], 1.0), g)
        st.update(A=A, b=b, x=0.9 * x0, v=torch.randn(case["d"], generator=g, device=DEV))
    elif kind == "solve":
        sigma = _polynomial(case["d"], case["power"])
        A, b, _ = _ridge(case["n"], case["d"], sigma, g)
        st.update(A=A, b=b, sd=_sds(sigma, [case["lam"]])[0],
                  sk=mihs.Sketch(A, case["family"], case["m"], int(seed)),
                  x=torch.empty(case["d"], dtype=torch.float64, device=DEV))
    elif kind == "batch":
        sigma, lams = _exponential(case["d"], case["decades"]), _lambdas(case["nl"])
        sds = _sds(sigma, lams)
        m = min(case["n"], int(math.ceil(4 * max(sds) / 4)) * 4)
        probs = []
        for _ in range(case["count"]):
            A, b, _ = _ridge(case["n"], case["d"], sigma, g, snr_db=30.0)
            probs.append((mihs.Sketch(A, "countsketch", m, int(seed)), A, b,
                          torch.empty(case["nl"], case["d"], device=DEV)))
        st.update(probs=probs, lams=lams, sds=[sds] * case["count"])
    else:
        raise ValueError(kind)
    return st


# ------------------------------------------------------------------------------------------------- passes


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "gradient":
        return mihs.gradient(st["A"], st["b"], st["x"], st["lam"])
    if kind == "dual":
        return mihs.gradient_dual(st["A"], st["b"], st["nu"], st["lam"])
    if kind == "path":
        return mihs.gradient_path(st["A"], st["b"], st["X"], st["lams"])
    if kind == "refined":
        return mihs.gradient_refined(st["A"], st["b"], st["x"], st["lam"])
    if kind == "sketch":
        if case["prec"] == "bf16":
            return mihs.sketch_gaussian_bf16(st["A"], case["m"], st["seed"])
        if case["prec"] == "fp8":
            return mihs.sketch_gaussian_fp8(st["A"], case["m"], st["seed"])
        return mihs.sketch_apply(st["A"], case["family"], case["m"], st["seed"])
    if kind == "aab":
        if case["prec"] == "fp32":
            return mihs.aab_solve(st["SA"], st["g"], st["lam"], eps_sub=0.0, max_inner=case["passes"])
        return mihs.aab_solve_q(st["q"], case["prec"], st["scales"], case["d"], st["g"], st["lam"], eps_sub=0.0,
                                max_inner=case["passes"])
    if kind == "backward":
        return mihs.backward_grads(st["A"], st["b"], st["x"], st["v"])
    if kind == "solve":
        st["sk"].resketch(st["A"], st["seed"])
        x, _ = st["sk"].solve_refined(st["A"], st["b"], case["lam"], st["sd"], tol=case["tol"], x=st["x"])
        return x
    for sk, A, _, _ in st["probs"]:
        sk.resketch(A, st["seed"])
    mihs.solve_batched(st["probs"], st["lams"], st["sds"], tol=1e-6)
    mihs.refine_batched(st["probs"], st["lams"], [case["tol"]] * case["nl"], st["sds"])
    return [X for _, _, _, X in st["probs"]]


def work(case):
    """What a pass cannot do without: inputs read once, outputs written once, multiplications and additions of the
    plain formula.  An iterative solve reads its matrix once a step, for as many steps as the method's rate √(sd/m) =
    1/2 needs."""
    kind, d = case["kind"], case["d"]
    n = case.get("n", 0)
    if kind == "gradient":
        return dict(bytes=4 * (n * d + n + 2 * d), flops=4 * n * d)
    if kind == "dual":
        return dict(bytes=4 * (n * d + 3 * n), flops=4 * n * d)
    if kind == "path":
        return dict(bytes=4 * (n * d + n + 2 * case["nl"] * d), flops=4 * n * d * case["nl"])
    if kind == "refined":
        return dict(bytes=4 * (n * d + n) + 16 * d, flops=4 * n * d)
    if kind == "sketch":
        m = case["m"]
        flops = {"gaussian": 2 * m * n * d, "countsketch": n * d,
                 "srht": n * d * math.log2(max(n, 2))}[case["family"]]
        return dict(bytes=4 * (n * d + m * d), flops=flops)
    if kind == "aab":
        size = {"fp32": 4, "bf16": 2, "fp8": 1}[case["prec"]]
        return dict(bytes=size * case["m"] * d + 8 * d, flops=4 * case["m"] * d * (case["passes"] + 1))
    if kind == "backward":
        return dict(bytes=8 * (n * d + n) + 8 * d, flops=8 * n * d)
    if kind == "solve":
        steps = math.ceil(math.log2(1 / case["tol"]))
        return dict(bytes=4 * n * d * (steps + 1), flops=4 * n * d * steps)
    # a path to 1e-6 reads each matrix once a step for all λ, a refined λ from there to its tolerance on its own
    steps = 20 + case["nl"] * math.ceil(math.log2(1e-6 / case["tol"]))
    return dict(bytes=4 * n * d * case["count"] * (steps + 1),
                flops=4 * n * d * case["count"] * case["nl"] * math.ceil(math.log2(1 / case["tol"])))


# ------------------------------------------------------------------------------ the same in 64 bits, without the library


def _mulhilo(a, b):
    """High and low words of the 64-bit product of the 32-bit number a and the 32-bit words b (held in int64)."""
    lo16, hi16 = b & 0xFFFF, b >> 16
    p0, p1 = a * lo16, a * hi16  # both below 2⁴⁸
    low = p0 + ((p1 & 0xFFFF) << 16)
    return ((p1 >> 16) + (low >> 32)) & 0xFFFFFFFF, low & 0xFFFFFFFF


def _philox(c0, c1, c2, seed):
    """Philox4x32-10 words (w0 … w3) for counters (c0, c1, c2, 0); int64 tensors of 32-bit words."""
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    x = [c0, c1, torch.full_like(c0, c2), torch.zeros_like(c0)]
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, x[0])
        h1, l1 = _mulhilo(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x


def _box_muller(a, b):
    u1, u2 = ((a >> 8) + 1).double() * 2.0**-24, (b >> 8).double() * 2.0**-24
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


def _sketch64(A, family, m, seed):
    n, d = A.shape
    A = A.double()
    out = torch.zeros(m, d, device=DEV, dtype=torch.float64)
    if family == "gaussian":
        step = max(4, ((1 << 25) // m) // 4 * 4)  # columns of S at a time
        for j in range(0, n, step):
            e = min(n, j + step)
            q = torch.arange(j // 4, (e + 3) // 4, device=DEV).unsqueeze(0).expand(m, -1)
            i = torch.arange(m, device=DEV).unsqueeze(1).expand_as(q)
            w = _philox(q, i, 0, seed)
            S = torch.stack((*_box_muller(w[0], w[1]), *_box_muller(w[2], w[3])), dim=2).reshape(m, -1)[:, : e - j]
            out += S @ A[j:e]
        return out / math.sqrt(m)
    j = torch.arange(n, device=DEV)
    if family == "countsketch":
        w = _philox(j, torch.zeros_like(j), 1, seed)
        sign = 1.0 - 2.0 * (w[1] & 1).double()
        return out.index_add_(0, (w[0] * m) >> 32, A * sign.unsqueeze(1))
    bits = max(0, (n - 1).bit_length())
    w = _philox(j, torch.zeros_like(j), 2, seed)
    Y = torch.zeros(1 << bits, d, device=DEV, dtype=torch.float64)
    Y[:n] = A * (1.0 - 2.0 * (w[0] & 1).double()).unsqueeze(1)
    del A
    for s in range(bits):
        V = Y.view(-1, 2, 1 << s, d)
        top = V[:, 0] + V[:, 1]
        V[:, 1] = V[:, 0] - V[:, 1]
        V[:, 0] = top
    i = torch.arange(m, device=DEV)
    r = _philox(i, torch.zeros_like(i), 3, seed)[0] >> (32 - bits) if bits else torch.zeros_like(i)
    return Y[r] / math.sqrt(m)


def _aab64(SA, g, lam, passes):
    """Algorithm 5: `passes` loop passes of the bidiagonalisation, Eldén's rotation and forward substitution."""
    theta1 = g.norm()
    v = g / theta1
    w = SA @ v
    rho = w.norm()
    p = w / rho
    rhobar = torch.sqrt(rho**2 + lam)
    c, s, phi = rho / rhobar, math.sqrt(lam) / rhobar, theta1 / rhobar
    dv = v / rhobar
    x = phi * dv
    for _ in range(passes):
        z = SA.t() @ p - rho * v
        theta = z.norm()
        v = z / theta
        w = SA @ v - theta * p
        rho = w.norm()
        p = w / rho
        lambar = torch.sqrt(lam + (s * theta) ** 2)
        thetabar = c * theta
        rhobar = torch.sqrt(rho**2 + lambar**2)
        c, s, phi = rho / rhobar, lambar / rhobar, -phi * thetabar / rhobar
        dv = (v - thetabar * dv) / rhobar
        x = x + phi * dv
    return x


def _ridge64(A, b, lams):
    """x*(λ) for each λ: Cholesky of the normal equations and two steps of refinement."""
    A, b = A.double(), b.double()
    gram, rhs = A.t() @ A, A.t() @ b
    eye = torch.eye(A.shape[1], device=DEV, dtype=torch.float64)
    xs = []
    for lam in lams:
        L = torch.linalg.cholesky(gram + lam * eye)
        x = torch.cholesky_solve(rhs.unsqueeze(1), L).squeeze(1)
        for _ in range(2):
            r = A.t() @ (b - A @ x) - lam * x
            x = x + torch.cholesky_solve(r.unsqueeze(1), L).squeeze(1)
        xs.append(x)
    return torch.stack(xs)


def _decoded(st):
    """The stored sketch of an AAb_Solver case as 64-bit numbers."""
    case = st["case"]
    if case["prec"] == "fp32":
        return st["SA"].double()
    m, d = case["m"], case["d"]
    if case["prec"] == "bf16":
        return st["q"][:, :d].double()
    q = st["q"].view(torch.float8_e4m3fn)[:, :d].float().double()
    s = st["scales"].double().repeat_interleave(128, 0)[:m].repeat_interleave(128, 1)[:, :d]
    return q * s


def exact(case, seed):
    kind, st = case["kind"], prepare(case, seed)
    if kind in ("gradient", "refined"):
        A, b, x = st["A"].double(), st["b"].double(), st["x"].double()
        return A.t() @ (b - A @ x) - st["lam"] * x
    if kind == "dual":
        A, b, nu = st["A"].double(), st["b"].double(), st["nu"].double()
        return b - A @ (A.t() @ nu) - st["lam"] * nu
    if kind == "path":
        A, X = st["A"].double(), st["X"].double()
        lams = torch.tensor(st["lams"], device=DEV, dtype=torch.float64).unsqueeze(1)
        return (st["b"].double().unsqueeze(1) - A @ X.t()).t() @ A - lams * X
    if kind == "sketch":
        return _sketch64(st["A"], case["family"], case["m"], st["seed"])
    if kind == "aab":
        return _aab64(_decoded(st), st["g"].double(), st["lam"], case["passes"])
    if kind == "backward":
        A, b, x, v = (st[k].double() for k in ("A", "b", "x", "v"))
        q = A @ v
        dA = torch.outer(b - A @ x, v)
        dA -= torch.outer(q, x)
        return dA, q, -(x * v).sum()
    if kind == "solve":
        return _ridge64(st["A"], st["b"], [case["lam"]])[0]
    return [_ridge64(A, b, st["lams"]) for _, A, b, _ in st["probs"]]
