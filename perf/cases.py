"""What this library is timed on: calls of its public entry points as a user's program makes them.

A case names one call (`kind`) and its sizes.  `prepare` makes the inputs and the handle
that such a program keeps, `run` makes the call, `exact` gives the same outputs from
plain torch in binary64, `work` counts what the call cannot do without.

Kinds
  apply          r = A x - y and g = A^T r with a handle's encoder (a caller with its own
                 outer loop, one step at a time)
  noalloc        the same from the caller's own matrix, without a handle
  apply_batched  the same for several images that share A (bf16 hi+lo storage)
  solve          one reconstruction with a stored A (IADM, or FTVCS), fixed iterations
  continuation   FTVCS or IADM with beta raised stage by stage, each warm-started
  batch          many images that share A, solved together (tensor-core products)
  uneven         several problems of different sizes whose A is regenerated from a seed
  dct            one reconstruction with the partial-DCT encoder
  oneshot        a new encoder used once: create (A copied, step size found), solve, destroy

The iteration counts are fixed (tol = 0), as in the repository's benchmark, so that
every run of a case does the same work.  Sizes come from the named workloads, the tests
and the paper's sampling ratios (m / n^2 from 0.05 to 0.6).
"""
import math
import random

import numpy as np
import torch

import paper_1001_1774_gb300 as tv

PRECISIONS = {"fp32": tv.TVCS_PREC_FP32, "bf16x2": tv.TVCS_PREC_BF16X2, "fp8": tv.TVCS_PREC_FP8_BF16}
BYTES = {"fp32": 4, "bf16x2": 4, "fp8": 3}     # per entry of A in the handle's storage
ON_CHIP = 32e6   # bytes of A that the SMs' shared memories hold together


def listed():
    return [
        # the smallest call: one application of a 16 x 16 operator, where latency is all there is
        dict(name="apply_n16", kind="apply", n=16, m=77, precision="fp32"),
        # a caller's own matrix at a ragged size (A about the size of the L2 cache)
        dict(name="noalloc_n96", kind="noalloc", n=96, m=2765),
        # a few images through the shared-A products
        dict(name="apply_batched_n64", kind="apply_batched", n=64, m=1229, count=40),
        # the 32 x 32 workload (ratio 0.3, up to 500 iterations), measurements and image on the host
        dict(name="solve_n32", kind="solve", n=32, m=307, precision="fp32", algo="iadm", iters=500,
             mu=1e3, beta=10.0, host=True),
        # the paper's 64 x 64 FTVCS practice: beta = 2^4 .. 2^7
        dict(name="continuation_n64", kind="continuation", n=64, m=1229, algo="ftvcs", stages=4,
             iters=60, mu=200.0, beta=16.0),
        # the default benchmark: 128 x 128, ratio 0.3, A in binary32 (322 MB), 300 iterations
        dict(name="solve_n128", kind="solve", n=128, m=4915, precision="fp32", algo="iadm",
             iters=300, mu=1e3, beta=10.0, host=False),
        # one image on the handle that a shared-A batch keeps (A as bf16 hi + lo)
        dict(name="solve_n128_bf16x2", kind="solve", n=128, m=4915, precision="bf16x2", algo="iadm",
             iters=100, mu=1e3, beta=10.0, host=False),
        # the large image with the smallest storage (2.6 GB of A), ratio 0.2
        dict(name="solve_n256_fp8", kind="solve", n=256, m=13107, precision="fp8", algo="iadm",
             iters=20, mu=5e2, beta=10.0, host=False),
        # the partial-DCT experiment of the paper at 128 x 128
        dict(name="dct_n128", kind="dct", n=128, m=4915, algo="iadm", iters=300, mu=500.0, beta=64.0),
        # 256 images sharing one A: throughput reconstruction
        dict(name="batch_n128", kind="batch", n=128, m=4915, count=256, iters=60, beta=10.0),
        # problems of mixed sizes whose matrices are never stored
        dict(name="uneven_6", kind="uneven", count=6, shapes=6, iters=10, mu=1e3, beta=10.0),
        # a new encoder for one image: setting up counts as much as solving
        dict(name="oneshot_n48", kind="oneshot", n=48, m=691, algo="iadm", iters=100, mu=1e3,
             beta=10.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["apply", "noalloc", "apply_batched", "solve", "solve", "continuation", "batch",
                       "uneven", "dct", "oneshot"])
    ratio = _log(rng, 0.05, 0.6 if kind == "dct" else 0.5)

    def m_of(n):
        return max(1, int(ratio * n * n) + rng.randrange(-3, 4))

    mu, beta = rng.choice([2e2, 5e2, 1e3]), rng.choice([8.0, 10.0, 16.0])
    algo = rng.choice(["iadm", "iadm", "ftvcs"])
    if kind == "apply":
        n = rng.choice([16, 32, 48, 64, 96, 128, 192])
        p = rng.choice(["fp32", "fp32", "bf16x2", "fp8"]) if n in (32, 64, 128, 192) else "fp32"
        return dict(kind=kind, n=n, m=m_of(n), precision=p)
    if kind == "noalloc":
        n = rng.choice([16, 32, 48, 64, 96, 128])
        return dict(kind=kind, n=n, m=m_of(n))
    if kind == "apply_batched":
        n = rng.choice([32, 64, 128])
        return dict(kind=kind, n=n, m=m_of(n), count=int(_log(rng, 1, 300)))
    if kind == "solve":
        n = rng.choice([16, 32, 48, 64, 96, 128, 192, 256])
        p = rng.choice(["fp32", "fp32", "bf16x2", "fp8"]) if n in (32, 64, 128, 192, 256) else "fp32"
        m = m_of(n)
        iters = int(min(_log(rng, 10, 400), max(4, 5e10 / (4.0 * m * n * n))))
        return dict(kind=kind, n=n, m=m, precision=p, algo=algo, iters=iters, mu=mu, beta=beta,
                    host=rng.random() < 0.5)
    if kind == "continuation":
        n = rng.choice([32, 48, 64, 96])
        return dict(kind=kind, n=n, m=m_of(n), algo=algo, stages=rng.randrange(2, 5),
                    iters=rng.randrange(20, 81), mu=mu, beta=rng.choice([4.0, 8.0, 16.0]))
    if kind == "batch":
        n = rng.choice([32, 64, 128])
        count = int(_log(rng, 2, 300))
        m = m_of(n)
        iters = int(min(_log(rng, 5, 50), max(2, 4e12 / (4.0 * m * n * n * count))))
        return dict(kind=kind, n=n, m=m, count=count, iters=iters, beta=beta)
    if kind == "uneven":
        return dict(kind=kind, count=rng.randrange(2, 9), shapes=rng.randrange(1 << 20),
                    iters=rng.randrange(3, 15), mu=mu, beta=beta)
    if kind == "dct":
        n = rng.choice([16, 32, 48, 64, 96, 128])
        return dict(kind=kind, n=n, m=max(1, min(n * n, m_of(n))), algo=algo,
                    iters=int(_log(rng, 20, 400)), mu=mu, beta=rng.choice([16.0, 64.0]))
    n = rng.choice([16, 32, 48, 64, 96])
    return dict(kind=kind, n=n, m=m_of(n), algo=algo, iters=int(_log(rng, 20, 200)), mu=mu, beta=beta)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(((int(seed) * 1_000_003) ^ (what * 7919)) & (2**62 - 1))


def _matrix(seed, m, N):
    """Gaussian encoder, entries N(0, 1/m), binary32."""
    return torch.randn(m, N, generator=_gen(seed, 1), device="cuda").mul_(1.0 / math.sqrt(m))


def _phantoms(seed, count, n, shapes=10):
    """Piecewise-constant images in [0, 1]: random ellipses painted one over the other."""
    p = torch.rand(shapes, 6, count, 1, 1, generator=_gen(seed, 2), device="cuda", dtype=torch.float64)
    t = (2.0 * torch.arange(n, device="cuda", dtype=torch.float64) + 1.0) / n - 1.0
    X, Y = t.view(1, 1, n), t.view(1, n, 1)
    img = torch.zeros(count, n, n, device="cuda", dtype=torch.float64)
    for cx, cy, ax, ay, th, val in p:
        c, s = torch.cos(math.pi * th), torch.sin(math.pi * th)
        dx, dy = X - (1.4 * cx - 0.7), Y - (1.4 * cy - 0.7)
        a, b = (dx * c + dy * s) / (0.05 + 0.45 * ax), (dy * c - dx * s) / (0.05 + 0.45 * ay)
        img = torch.where(a * a + b * b <= 1.0, val.expand_as(img), img)
    return img.reshape(count, n * n)


def _times(A, X):
    """X A^T in binary64 (rows of X are images), by slabs of A's rows."""
    return torch.cat([X @ a.double().T for a in A.split(max(1, (1 << 26) // A.shape[1]))], dim=1)


def _measure(seed, clean, level=1e-3):
    """Measurements with Gaussian noise of `level` times their RMS, binary32."""
    noise = torch.randn(clean.shape, generator=_gen(seed, 3), device="cuda", dtype=torch.float64)
    rms = clean.square().mean(dim=1, keepdim=True).sqrt()
    return (clean + level * rms * noise).float().contiguous()


def _mus(count):
    return [(2e2, 5e2, 1e3, 2e3)[b % 4] for b in range(count)]


def _dct_matrix(n):
    k = torch.arange(n, device="cuda", dtype=torch.float64).view(n, 1)
    j = torch.arange(n, device="cuda", dtype=torch.float64).view(1, n)
    C = math.sqrt(2.0 / n) * torch.cos(math.pi * (2 * j + 1) * k / (2 * n))
    C[0] = math.sqrt(1.0 / n)
    return C


def _dct_rows(seed, n, m):
    rows = np.random.default_rng([int(seed), 17]).choice(n * n, size=m, replace=False)
    return np.sort(rows).astype(np.int32)


def _shapes(case):
    """(n, m) of each problem of an uneven case."""
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        n = r.choice([64, 64, 96, 128])
        out.append((n, int(r.choice([0.1, 0.2, 0.3]) * n * n)))
    return out


def _philox_matrix(seed, m, N):
    """The matrix that a seed stands for (Philox4x32-10 and Box-Muller, entry e from block
    e >> 2; the recipe stated in include/tvcs.h's generator), in binary64."""
    mask = 0xFFFFFFFF

    def mul(a, b):   # 32 x 32 -> (high, low)
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        t = p1 + (p0 >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)

    out = torch.empty(m * N, device="cuda", dtype=torch.float64)
    step = 1 << 23
    for e0 in range(0, m * N, step):
        e1 = min(m * N, e0 + step)
        b = torch.arange(e0 >> 2, (e1 + 3) >> 2, device="cuda", dtype=torch.int64)
        c = [b & mask, b >> 32, torch.zeros_like(b), torch.zeros_like(b)]
        k0, k1 = seed & mask, seed >> 32
        for _ in range(10):
            h0, l0 = mul(0xD2511F53, c[0])
            h1, l1 = mul(0xCD9E8D57, c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        z = []
        for xa, xb in ((c[0], c[1]), (c[2], c[3])):
            rad = torch.sqrt(-2.0 * torch.log(((xa >> 8) + 1).double() * 2.0**-24))
            ang = (2.0 * math.pi * 2.0**-24) * (xb >> 8).double()
            z += [rad * torch.cos(ang), rad * torch.sin(ang)]
        out[e0:e1] = torch.stack(z, dim=1).reshape(-1)[: e1 - e0]
    return out.view(m, N).mul_(float(np.float32(1.0 / math.sqrt(m))))


def _problem_seed(seed, i):
    return (int(seed) * 64 + i + 1) & (2**40 - 1)


def _edge_tau(n, m):
    """Step size below 1 / lambda_max(A^T A) from the edge of the Marchenko-Pastur law."""
    return 0.9 / (1.0 + n / math.sqrt(m)) ** 2


def _inputs(case, seed):
    """What a case is about: the encoder (or what names it) and the measurements."""
    kind, n = case["kind"], case.get("n", 0)
    N = n * n
    if kind == "uneven":
        mats, fs = [], []
        for i, (k, m) in enumerate(_shapes(case)):
            s = _problem_seed(seed, i)
            A = _philox_matrix(s, m, k * k)
            fs.append(_measure(s, _phantoms(s, 1, k) @ A.T)[0])
            mats.append(A)
        return mats, fs
    if kind == "dct":
        rows = _dct_rows(seed, n, case["m"])
        C = _dct_matrix(n)
        Z = C @ _phantoms(seed, 1, n).view(n, n) @ C.T
        return rows, _measure(seed, Z.reshape(1, N)[:, torch.from_numpy(rows).cuda().long()])[0]
    A = _matrix(seed, case["m"], N)
    count = case.get("count", 1)
    X = _phantoms(seed, count, n)
    f = _measure(seed, _times(A, X))
    if kind in ("apply", "noalloc", "apply_batched"):
        return A, f, X.float().contiguous() + 0.01 * torch.randn(count, N, generator=_gen(seed, 4), device="cuda")
    return A, f


def _options(case, precision="fp32", tau=0.0):
    o = tv.tvcs_default_options()
    o.precision = PRECISIONS[precision]
    o.algo = tv.TVCS_ALGO_FTVCS if case.get("algo") == "ftvcs" else tv.TVCS_ALGO_IADM
    o.max_iter = case.get("iters", 0)
    o.tau = tau
    return o


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def prepare(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    N = n * n
    if kind == "uneven":
        _, fs = _inputs(case, seed)
        hs = []
        for i, (k, m) in enumerate(_shapes(case)):
            opt = _options(case, tau=_edge_tau(k, m))
            opt.a_mode = tv.TVCS_A_REGENERATE
            hs.append(tv.tvcs_create(None, _problem_seed(seed, i), m, k, case["mu"], case["beta"], 0.0, opt))
        return dict(kind=kind, hs=hs, f=fs, u=[torch.empty(h.N, device="cuda") for h in hs])
    if kind == "dct":
        rows, f = _inputs(case, seed)
        h = tv.tvcs_create_partial_dct(rows, n, case["mu"], case["beta"], 0.0, _options(case, tau=1.9))
        return dict(kind="solve", h=h, f=f, u=torch.empty(N, device="cuda"))
    if kind in ("apply", "noalloc", "apply_batched"):
        A, f, X = _inputs(case, seed)
        s = dict(kind=kind, n=n, m=case["m"], x=X, y=f, r=torch.empty_like(f), g=torch.empty_like(X))
        if kind == "noalloc":
            s["A"] = A
        else:
            p = case.get("precision", "bf16x2")
            # the step size is not used by the products: a given one spares the search for it
            s["h"] = tv.tvcs_create(A, 0, case["m"], n, 1.0, 1.0, 0.0, _options(case, p, tau=0.1))
        return s
    A, f = _inputs(case, seed)
    if kind == "oneshot":
        return dict(kind=kind, A=A, f=f[0], u=torch.empty(N, device="cuda"), n=n, m=case["m"],
                    mu=case["mu"], beta=case["beta"], opt=_options(case))
    if kind == "batch":
        h = tv.tvcs_create(A, 0, case["m"], n, 1e3, case["beta"], 0.0, _options(case, "bf16x2"))
        return dict(kind=kind, h=h, f=f, u=torch.empty(case["count"], N, device="cuda"),
                    mu=_mus(case["count"]))
    h = tv.tvcs_create(A, 0, case["m"], n, case["mu"], case["beta"], 0.0,
                       _options(case, case.get("precision", "fp32")))
    if kind == "continuation":
        return dict(kind=kind, h=h, f=f[0], u=torch.empty(N, device="cuda"),
                    betas=[case["beta"] * 2**k for k in range(case["stages"])])
    if case["host"]:
        return dict(kind=kind, h=h, f=f[0].cpu().numpy(), u=np.empty(N, np.float32))
    return dict(kind=kind, h=h, f=f[0], u=torch.empty(N, device="cuda"))


def run(s):
    kind = s["kind"]
    if kind == "apply":
        tv.tvcs_apply(s["h"], s["x"], s["y"], s["r"], s["g"])
        return s["r"], s["g"]
    if kind == "noalloc":
        tv.tvcs_apply_noalloc(s["A"], s["m"], s["n"], s["x"], s["y"], s["r"], s["g"])
        return s["r"], s["g"]
    if kind == "apply_batched":
        tv.tvcs_apply_batched(s["h"], s["x"].shape[0], s["x"], s["y"], s["r"], s["g"])
        return s["r"], s["g"]
    if kind == "solve":
        res = tv.tvcs_solve(s["h"], s["f"], s["u"])
        return s["u"], res.objective
    if kind == "continuation":
        res = tv.tvcs_solve_continuation(s["h"], s["f"], s["u"], s["betas"])
        return s["u"], res[-1].objective
    if kind == "batch":
        f, u = s["f"], s["u"]
        res = tv.tvcs_solve_batched([s["h"]] * f.shape[0], list(f), list(u), s["mu"])
        return u, np.array([r.objective for r in res])
    if kind == "uneven":
        res = tv.tvcs_solve_batched(s["hs"], s["f"], s["u"])
        return s["u"], np.array([r.objective for r in res])
    h = tv.tvcs_create(s["A"], 0, s["m"], s["n"], s["mu"], s["beta"], 0.0, s["opt"])
    res = tv.tvcs_solve(h, s["f"], s["u"])
    tau = tv.tvcs_get_tau(h)
    tv.tvcs_destroy(h)
    return s["u"], res.objective, tau


def work(case):
    """One product pair reads A once (what of it does not fit in the SMs' shared memories
    has to come again in every iteration); A counts in the handle's storage."""
    kind = case["kind"]
    if kind == "uneven":
        iters = case["iters"]
        flops = sum(4.0 * m * n * n for n, m in _shapes(case)) * (iters + 2)
        return {"bytes": sum(4.0 * (m + n * n) for n, m in _shapes(case)), "flops": flops}
    n, m = case["n"], case["m"]
    N = n * n
    per = 2.0 * 5 * N * math.log2(N) + 40.0 * N   # the FFT pair and the point-wise steps
    if kind == "dct":
        per += 4 * 2.0 * n**3
        return {"bytes": 4.0 * (2 * m + N), "flops": per * case["iters"]}
    a = float(m) * N * BYTES[case.get("precision", "bf16x2" if kind in ("apply_batched", "batch") else "fp32")]
    count = case.get("count", 1)
    vec = 4.0 * count * (m + N)
    if kind in ("apply", "noalloc", "apply_batched"):
        return {"bytes": a + 2 * vec, "flops": 4.0 * m * N * count}
    passes = case["iters"] * case.get("stages", 1) + 2
    if kind == "oneshot":
        passes += 101   # the power iteration that finds the step size
    return {"bytes": (a if a <= ON_CHIP else a + (a - ON_CHIP) * (passes - 1)) + vec,
            "flops": passes * count * (4.0 * m * N + per)}


# --------------------------------------------------------------------------
# the same in binary64
# --------------------------------------------------------------------------

def _objective(u, resid, mu):
    d1, d2 = torch.roll(u, -1, 2) - u, torch.roll(u, -1, 1) - u
    return torch.sqrt(d1 * d1 + d2 * d2).sum(dim=(1, 2)) + 0.5 * mu.view(-1) * resid.square().sum(dim=1)


def _iterate(mul, mult, f, n, mu, betas, tau, iters, algo):
    """Algorithm 2 (1 where algo is ftvcs), stage by stage in beta, for images u[b]; mul and
    mult apply A and A^T to rows."""
    mu = mu.view(-1, 1, 1)
    s = 4.0 * torch.sin(math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n).square()
    lam_dd = s.view(n, 1) + s.view(1, n)
    u = mult(f).view(-1, n, n)
    l1, l2 = torch.zeros_like(u), torch.zeros_like(u)
    for beta in betas:
        for _ in range(iters):
            z1 = torch.roll(u, -1, 2) - u + l1 / beta
            z2 = torch.roll(u, -1, 1) - u + l2 / beta
            nz = torch.sqrt(z1 * z1 + z2 * z2)
            k = torch.where(nz > 1.0 / beta, (nz - 1.0 / beta) / nz.clamp_min(1e-300), torch.zeros_like(nz))
            w1, w2 = k * z1, k * z2
            g = mult(mul(u.view(-1, n * n)) - f).view(-1, n, n)
            y1, y2 = w1 - l1 / beta, w2 - l2 / beta
            c = mu / (beta * tau)
            rhs = torch.roll(y1, 1, 2) - y1 + torch.roll(y2, 1, 1) - y2 + c * (u - tau * g)
            u = torch.fft.ifft2(torch.fft.fft2(rhs) / (lam_dd + c)).real
            if algo == "iadm":
                l1 = l1 - beta * (w1 - (torch.roll(u, -1, 2) - u))
                l2 = l2 - beta * (w2 - (torch.roll(u, -1, 1) - u))
    return u, _objective(u, mul(u.reshape(-1, n * n)) - f, mu)


def _tau(A, rounds=100):
    v = torch.full((1, A.shape[1]), 1.0 / math.sqrt(A.shape[1]), device="cuda", dtype=torch.float64)
    for _ in range(rounds):
        v = (v @ A.T) @ A
        v = v / v.norm()
    return float(1.0 / (1.01 * (v @ A.T).square().sum()))


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "uneven":
        mats, fs = _inputs(case, seed)
        us, objs = [], []
        for (k, m), A, f in zip(_shapes(case), mats, fs):
            mu = torch.tensor([case["mu"]], device="cuda", dtype=torch.float64)
            u, o = _iterate(lambda x: x @ A.T, lambda r: r @ A, f.double().view(1, -1), k, mu, [case["beta"]],
                            _edge_tau(k, m), case["iters"], "iadm")
            us.append(u.reshape(-1))
            objs.append(float(o))
        return us, np.array(objs)
    if kind == "dct":
        rows, f = _inputs(case, seed)
        C, at = _dct_matrix(n), torch.from_numpy(rows).cuda().long()

        def mul(x):
            return (C @ x.view(n, n) @ C.T).reshape(1, -1)[:, at]

        def mult(r):
            S = torch.zeros(n * n, device="cuda", dtype=torch.float64)
            S[at] = r[0]
            return (C.T @ S.view(n, n) @ C).reshape(1, -1)

        mu = torch.tensor([case["mu"]], device="cuda", dtype=torch.float64)
        u, o = _iterate(mul, mult, f.double().view(1, -1), n, mu, [case["beta"]], 1.9, case["iters"], case["algo"])
        return u.reshape(-1), float(o)
    if kind in ("apply", "noalloc", "apply_batched"):
        A, f, X = _inputs(case, seed)
        A = A.double()
        r = X.double() @ A.T - f.double()
        return r, r @ A
    A, f = _inputs(case, seed)
    A, f = A.double(), f.double()
    tau = _tau(A)
    mus = _mus(case["count"]) if kind == "batch" else [case["mu"]]
    mu = torch.tensor(mus, device="cuda", dtype=torch.float64)
    betas = [case["beta"] * 2**k for k in range(case.get("stages", 1))]
    u, o = _iterate(lambda x: x @ A.T, lambda r: r @ A, f, n, mu, betas, tau, case["iters"], case.get("algo", "iadm"))
    if kind == "batch":
        return u.reshape(len(mus), n * n), o.cpu().numpy()
    u, o = u.reshape(-1), float(o)
    return (u, o, tau) if kind == "oneshot" else (u, o)
