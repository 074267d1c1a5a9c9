"""Performance cases of the library: the calls that its users make, from the smallest to the largest.

Every case is one call (one pass) through `paper_2609_21102_b200.binding.Context`. `kind` says which entry point:

  polar    defl_polar_batched: the deflated polar factor of a batch of device matrices
  host     defl_polar_batched_host: the same for pinned host buffers, copies included
  muon     defl_muon_step_batched: one Deflated Muon step on a shape group, weights and momentum updated in place
  psd      defl_psd_project: one deflated PSD projection, the basis tracked from call to call
  invroot  defl_inv_root: one deflated inverse matrix root, the basis tracked from call to call
  admm     defl_admm_diag_sdp: a few ADMM iterations on a max-cut type SDP

`exact` restates the algorithms in fp64 torch operations.
"""
import math

import numpy as np
import torch

from paper_2609_21102_b200 import binding, schedules

MUON = [list(binding.MUON_QUINTIC)]
CLASSICAL = [list(binding.CLASSICAL_QUINTIC)]
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
LR, MU, DECAY = 0.02, 0.95, 0.1

_context = None


def _ctx():
    """The one context a single-stream program keeps for the life of the process."""
    global _context
    if _context is None:
        _context = binding.Context(0)
    return _context


def _schedule(case):
    if case["schedule"] == "minimax":
        # per-step minimax quintics from [1e-3, 1], as the tests and the benchmark build them
        return [list(c) for c in schedules.remez_sign_schedule(1e-3, case["steps"], margin=0.01)[0]]
    return (MUON if case["schedule"] == "muon" else CLASSICAL) * case["steps"]


def listed():
    polar = {"kind": "polar", "schedule": "muon", "steps": 5, "gamma": 1.01, "mode": "padded", "tau": 0.0,
             "symmetry": True, "sketch": "given", "dtype": "bf16"}
    return [
        # the smallest batch: a few small fp32 matrices (unit tests, small layers), where latency is all; default options
        dict(polar, name="tiny_fp32", b=4, m=128, n=256, dtype="fp32", k=4, p=4, J=1, spectrum="head4", symmetry=False, sketch="seed"),
        # fp32 storage at the size of a small model's layer, with the additive restore of Eq. 3
        dict(polar, name="fp32_add", b=4, m=512, n=384, dtype="fp32", k=8, p=8, J=1, spectrum="spiked", mode="add"),
        # attention-sized square layers of a small transformer, with the deflation gate deciding how many to deflate
        dict(polar, name="square_gated", b=12, m=768, n=768, k=16, p=8, J=1, spectrum="spiked", tau=0.2),
        # layers whose sides are multiples of nothing, stored tall, library defaults
        dict(polar, name="ragged_tall", b=4, m=1003, n=517, k=10, p=6, J=2, spectrum="power", symmetry=False),
        # MLP layers of a medium transformer with the steep per-step minimax schedule
        dict(polar, name="wide_minimax", b=24, m=1024, n=4096, k=16, p=8, J=1, spectrum="power08", schedule="minimax", gamma=1.1),
        # the two shape groups of a GPT-2-XL-sized Muon batch; the wide one is the largest call
        dict(polar, name="xl_square", b=48, m=1600, n=1600, k=32, p=16, J=2, spectrum="power"),
        dict(polar, name="xl_wide", b=48, m=1600, n=6400, k=32, p=16, J=2, spectrum="power"),
        # host-resident gradients: the copies count
        dict(polar, name="host_wide", kind="host", b=12, m=768, n=3072, k=8, p=8, J=1, spectrum="spiked", sketch="seed"),
        # an optimizer step: tall MLP layers, bf16 momentum with Nesterov, fp32 master weights, weight decay, library-drawn sketch
        dict(polar, name="muon_tall", kind="muon", b=12, m=3072, n=768, k=8, p=8, J=1, spectrum="spiked", sketch="seed"),
        # one projection inside a large SDP solver (tf32 filter)
        {"name": "psd_4096", "kind": "psd", "n": 4096, "k": 8, "K": 16, "schedule": "classical", "steps": 7, "gamma": 1.1,
         "half": False, "symmetry": True},
        # a Shampoo-type preconditioner block: inverse 4-th root of a covariance with a dominant head
        {"name": "invroot_1024", "kind": "invroot", "n": 1024, "k": 8, "K": 16, "root": 4, "steps": 8, "gamma": 1.1},
        # a stretch of a small SDP solve, with the filter in half precision
        {"name": "admm_1000", "kind": "admm", "n": 1000, "k": 8, "K": 16, "iters": 5, "schedule": "classical", "steps": 7,
         "gamma": 1.1, "half": True, "symmetry": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["polar", "polar", "polar", "polar32", "ragged", "muon", "host", "psd", "invroot", "admm"])
    if kind in ("psd", "invroot", "admm"):
        # rows of n fp32 values: multiples of 4 are what the tensor engine takes, other sizes stay small
        n = 8 * _log_int(rng, 16, 320) if kind != "admm" else 8 * _log_int(rng, 16, 128)
        if kind != "admm" and rng.random() < 0.25:
            n = _log_int(rng, 100, 500)
        K = rng.choice([8, 12, 16, 24])
        k = rng.choice([4, 6, 8])
        if kind == "invroot":
            return {"kind": kind, "n": n, "k": k, "K": K, "root": rng.choice([1, 2, 4]), "steps": rng.choice([8, 9, 10]), "gamma": 1.1}
        c = {"kind": kind, "n": n, "k": k, "K": K, "schedule": "classical", "steps": rng.randint(5, 8), "gamma": 1.1,
             "half": n % 8 == 0 and rng.random() < 0.4, "symmetry": rng.random() < 0.7}
        if kind == "admm":
            c["iters"] = rng.randint(2, 6)
        return c
    fp32 = kind == "polar32"
    if fp32:
        ms, ratio, b = _log_int(rng, 32, 400), rng.uniform(1.0, 3.0), rng.randint(1, 6)
    elif kind == "ragged":
        ms, ratio, b = _log_int(rng, 65, 520), rng.uniform(1.0, 2.5), rng.randint(1, 4)
    else:
        ms, ratio, b = 8 * _log_int(rng, 8, 160), rng.choice([1.0, 1.0, 1.5, 2.0, 3.0, 4.0, rng.uniform(1.0, 4.0)]), _log_int(rng, 1, 24)
    ml = int(ms * ratio)
    if not fp32 and kind != "ragged":
        ml = (ml + 7) // 8 * 8
    else:
        ms, ml = ms | 1, ml | 1
        if rng.random() < 0.3:
            ms, ml = ms + 1, ml + 1
    ml = max(ms, ml)
    m, n = (ms, ml) if rng.random() < 0.5 else (ml, ms)
    cap = min(24, ms // 5)
    case = {"kind": "polar" if kind in ("polar32", "ragged") else kind, "b": b, "m": m, "n": n, "dtype": "fp32" if fp32 else "bf16",
            "k": rng.randint(4, max(4, cap)), "p": rng.randint(4, 12), "J": rng.randint(1, 2), "schedule": "muon", "steps": 5,
            "gamma": 1.01, "mode": "padded", "tau": 0.0, "symmetry": rng.random() < 0.7, "sketch": rng.choice(["given", "seed"]),
            "spectrum": rng.choice(["spiked", "power", "power08"])}
    if case["kind"] == "polar":
        if rng.random() < 0.15:
            case["k"], case["p"], case["J"] = 0, 0, 0      # the plain filter (past the deflation cutoff)
        elif fp32 and rng.random() < 0.4:
            case["mode"] = "add"
        elif rng.random() < 0.2:
            case["spectrum"], case["k"], case["tau"] = "spiked", max(10, case["k"]), 0.2
        if not fp32 and ms >= 256 and rng.random() < 0.25:
            case["schedule"], case["gamma"] = "minimax", 1.1
    return case


# ---- inputs -----------------------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _heads(g, b, rows, r):
    """[b, rows, r] with orthonormal columns."""
    q = torch.linalg.qr(_randn(g, b, rows, r))[0]
    return q


def _matrices(case, g):
    """Momentum-like matrices: a few dominant directions over a bulk (spiked), or singular values that fall like a power
    of the index down to a noise floor (power, power08), or four values far above the rest (head4)."""
    b, m, n = case["b"], case["m"], case["n"]
    ms, ml = min(m, n), max(m, n)
    kind = case["spectrum"]
    bulk = _randn(g, b, m, n)
    if kind == "spiked":
        sigma = torch.full((min(8, ms // 4),), 30.0 * math.sqrt(ms), device="cuda")
    elif kind == "head4":
        bulk *= 0.5 / (math.sqrt(ms) + math.sqrt(ml))
        sigma = torch.tensor([100.0, 50.0, 30.0, 20.0], device="cuda")
    else:
        r = min(96, ms // 2)
        top, power = (200.0, 1.0) if kind == "power" else (50.0, 0.8)
        sigma = top * torch.arange(1, r + 1, device="cuda", dtype=torch.float32) ** -power
        bulk *= top * (r + 1.0) ** -power / (math.sqrt(ms) + math.sqrt(ml))     # the bulk's norm continues the law
    u, v = _heads(g, b, m, sigma.numel()), _heads(g, b, n, sigma.numel())
    return torch.baddbmm(bulk, u * sigma, v.transpose(1, 2)).to(DTYPES[case["dtype"]])


def _width(case):
    return min(min(case["m"], case["n"]), case["k"] + case["p"]) if case["k"] else 0


def _symmetric(n, g, heads=8, magnitude=1000.0):
    """A symmetric matrix with `heads` dominant eigenvalues of either sign over a bulk in about [-1, 1], and the basis a
    solver has tracked so far: those directions, a little off, and directions of the bulk."""
    a = _randn(g, n, n)
    x = (a + a.T) * (0.5 / math.sqrt(2.0 * n))
    u = _heads(g, 1, n, heads)[0]
    sign = torch.where(torch.rand(heads, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    size = magnitude * (0.5 + 0.5 * torch.rand(heads, generator=g, device="cuda"))
    x = x + (u * (sign * size)) @ u.T
    return 0.5 * (x + x.T), u


def _basis(u, K, g):
    n, h = u.shape
    h = min(h, K)
    v = torch.cat([u[:, :h] + 1e-4 / math.sqrt(n) * _randn(g, n, h), _randn(g, n, K - h) / math.sqrt(n)], dim=1)
    return torch.linalg.qr(v)[0].contiguous()


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": dict(case), "ctx": _ctx(), "seed": int(seed)}
    if kind in ("polar", "host", "muon"):
        s["schedule"] = _schedule(case)
        G = _matrices(case, g)
        l = _width(case)
        s["sketch"] = _randn(g, case["b"], min(case["m"], case["n"]), l) if case["sketch"] == "given" and l else None
        if kind == "polar":
            s["G"] = G
        elif kind == "host":
            s["G"] = G.cpu().pin_memory()
            s["out"] = torch.empty_like(s["G"]).pin_memory()
        else:
            # a momentum in its steady state and a gradient that agrees with it up to noise
            s["M"] = G
            s["grad"] = ((1.0 - MU) * (G.float() + 0.3 * G.float().std() * _randn(g, *G.shape))).to(G.dtype)
            s["W"] = _randn(g, *G.shape) * 0.02
        return s
    n = case["n"]
    if kind == "psd":
        s["schedule"] = _schedule(case)
        s["X"], u = _symmetric(n, g, case["k"])
        s["V"], s["start"] = _basis(u, case["K"], g), _randn(g, n)
    elif kind == "invroot":
        # gradient statistics: a Wishart bulk (twice as many samples as rows), damping, and a dominant head
        w = _randn(g, n, 2 * n)
        u = _heads(g, 1, n, case["k"])[0]
        lam = 300.0 + 1700.0 * torch.rand(case["k"], generator=g, device="cuda")
        a = w @ w.T / (2.0 * n) + (u * lam) @ u.T
        a = 0.5 * (a + a.T)
        a.diagonal().add_(0.05)
        s["A"] = a
        s["V"], s["start"] = _basis(u, case["K"], g), _randn(g, n)
        for _ in range(2):      # two block steps: the basis of a root that has been taken before
            s["V"] = torch.linalg.qr(a @ s["V"])[0].contiguous()
    else:
        # max-cut: the weighted adjacency of a random graph, unit diagonal, cold start
        s["schedule"] = _schedule(case)
        w = torch.triu((torch.rand(n, n, generator=g, device="cuda") < 0.3).float() * torch.rand(n, n, generator=g, device="cuda"), 1)
        s["C"] = (w + w.T) / 4.0
        s["rhs"] = torch.ones(n, device="cuda")
        s["X"], s["S"] = torch.zeros(n, n, device="cuda"), torch.zeros(n, n, device="cuda")
        s["V"] = torch.linalg.qr(_randn(g, n, case["K"]))[0].contiguous()
        s["start"] = _randn(g, n)
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind in ("polar", "host", "muon"):
        kw = dict(sketch=s["sketch"], seed=s["seed"], gamma=case["gamma"], exploit_symmetry=case["symmetry"],
                  restore_mode=binding.RESTORE_ADD if case["mode"] == "add" else binding.RESTORE_PADDED)
        if kind == "polar":
            return ctx.defl_polar_batched(s["G"], case["k"], case["p"], case["J"], s["schedule"], tau=case["tau"], **kw)
        if kind == "host":
            return ctx.defl_polar_batched_host(s["G"], s["out"], case["k"], case["p"], case["J"], s["schedule"], **kw)
        ctx.defl_muon_step_batched(s["W"], s["M"], s["grad"], LR, MU, case["k"], case["p"], case["J"], s["schedule"],
                                   nesterov=True, weight_decay=DECAY, **kw)
        return s["W"], s["M"]
    if kind == "psd":
        P = ctx.defl_psd_project(s["X"], case["k"], s["V"], s["schedule"], gamma=case["gamma"], lanczos_start=s["start"],
                                 exploit_symmetry=case["symmetry"], half_filter=case["half"])
        return P, s["V"]
    if kind == "invroot":
        return ctx.defl_inv_root(s["A"], case["root"], case["k"], s["V"], case["steps"], gamma=case["gamma"],
                                 lanczos_start=s["start"]), s["V"]
    y, residuals = ctx.defl_admm_diag_sdp(s["C"], s["rhs"], 1.0, case["iters"], s["X"], s["S"], case["k"], s["V"], s["schedule"],
                                          warmup_iters=2, gamma=case["gamma"], lanczos_start=s["start"],
                                          exploit_symmetry=case["symmetry"], half_filter=case["half"])
    return s["X"], s["S"], y, residuals


# ---- what a pass cannot do without ------------------------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("polar", "host", "muon"):
        b, m, n, L = case["b"], case["m"], case["n"], case["steps"]
        ms, ml, es = min(m, n), max(m, n), 2 if case["dtype"] == "bf16" else 4
        l = _width(case)
        # a filter step: the Gram matrix and its square (symmetric: half of each), then the product with X; two steps
        # can also share one pass over X, with four more short-side products, which is less where X is long
        single = 3 * ms * ms * ml + ms ** 3
        both = min(2 * single, 3 * ms * ms * ml + 5 * ms ** 3)
        flops = b * ((L // 2) * both + (L % 2) * single)
        if l:
            flops += b * (2 * m * n * l * (2 * case["J"] + 2) + 2 * m * n * case["k"])
        size = b * m * n * es
        # a Muon step reads gradient, momentum and fp32 weights and writes momentum and weights
        moved = 2 * size if kind != "muon" else 3 * size + 2 * b * m * n * 4
        return {"bytes": moved, "flops": flops}
    n, K = case["n"], case["K"]
    if kind == "invroot":
        products = (case["steps"] - 1) * {1: 2, 2: 3, 4: 4}[case["root"]]
        return {"bytes": 8 * n * n, "flops": products * n ** 3 + 2 * n * n * (K + 40 + case["k"])}
    one = 3 * case["steps"] * n ** 3 + n ** 3 + 2 * n * n * (K + 40 + 3 * case["k"])
    if kind == "psd":
        return {"bytes": 8 * n * n, "flops": one}
    return {"bytes": 20 * n * n, "flops": case["iters"] * one}


def tolerance(case):
    """About four times the distance from `exact` that was measured over the listed cases and some hundred and twenty drawn ones."""
    kind = case["kind"]
    if kind in ("polar", "host"):
        # 16-bit iterates: 3e-3 .. 1.2e-2, single values up to 5e-2; fp32 storage: 1e-6 .. 6e-5, up to 3.3e-4
        return {"rel": 3e-2, "max": 0.25} if case["dtype"] == "bf16" else {"rel": 2.5e-4, "max": 1.5e-3}
    if kind == "muon":
        return {"rel": 2.2e-3, "max": 1.3e-2}        # 6e-5 .. 5.4e-4 of the weights, whose update is a small part of them
    if kind == "psd":
        return {"rel": 1.5e-4, "max": 2e-3}          # 1e-6 .. 5e-6 of the projection, 1e-5 .. 3.5e-5 of the basis
    if kind == "invroot":
        return {"rel": 4e-3, "max": 2e-2}            # 7e-4 .. 1e-3, single values up to 4.2e-3
    return {"rel": 1e-2, "max": 3e-2}                # ADMM: iterates 2e-4 .. 5e-4, multipliers 2.4e-4 .. 2.7e-3, up to 6.5e-3


# ---- the same results in fp64 -----------------------------------------------------------------------------------


def _gaussian(seed, count):
    """The documented counter-based generator (values 0 .. count-1 of stream `seed`), rounded to fp32."""
    u64 = np.uint64

    def h(x):
        x = x + u64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> u64(30))) * u64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> u64(27))) * u64(0x94D049BB133111EB)
        return x ^ (x >> u64(31))

    with np.errstate(over="ignore"):
        base = h(np.array([seed], dtype=np.uint64))
        pair = np.arange((count + 1) // 2, dtype=np.uint64)
        r1, r2 = h(base ^ (u64(2) * pair)), h(base ^ (u64(2) * pair + u64(1)))
    u1 = ((r1 >> u64(11)).astype(np.float64) + 1.0) * 2.0 ** -53
    u2 = (r2 >> u64(11)).astype(np.float64) * 2.0 ** -53
    rad = np.sqrt(-2.0 * np.log(u1))
    v = np.stack([rad * np.cos(2.0 * np.pi * u2), rad * np.sin(2.0 * np.pi * u2)], axis=1).reshape(-1)[:count]
    return v.astype(np.float32)


def _orth(y):
    """The QR factor with positive diagonal."""
    q, r = torch.linalg.qr(y)
    return q * torch.sign(torch.diagonal(r))


def _polar64(G, omega, case, sched):
    """Algorithm 3, then Algorithm 1 (or Eq. 3) on one fp64 matrix."""
    tall = G.shape[0] >= G.shape[1]
    A = G if tall else G.T
    k, head = case["k"], None
    R = A
    if k:
        q = _orth(A @ omega)
        for _ in range(case["J"]):
            q = _orth(A @ _orth(A.T @ q))
        B = q.T @ A
        lam, e = torch.linalg.eigh(B @ B.T)
        sv, e = lam.flip(0).clamp(min=0).sqrt(), e.flip(1)
        if case["tau"] > 0:
            k = int((sv[:k] > case["tau"] * sv[0]).sum()) if float(sv[k - 1]) < case["tau"] * float(sv[0]) else 0
        u, v = q @ e[:, :k], (B.T @ e[:, :k]) / sv[:k]
        head = u @ v.T
        R = A - (u * sv[:k]) @ v.T
    X = R / torch.linalg.norm(R)
    if head is not None and case["mode"] == "padded":
        X = X + head / case["gamma"]
    for a, b, c in sched:
        S = X.T @ X
        X = a * X + X @ (b * S + c * (S @ S))
    if head is not None and case["mode"] == "add":
        X = X + head
    return X if tall else X.T


def _polar64_batch(D, s, case):
    ms, l = min(case["m"], case["n"]), _width(case)
    out = torch.empty(D.shape, dtype=torch.float64, device="cuda")
    for i in range(case["b"]):
        omega = None
        if l:
            omega = s["sketch"][i] if s["sketch"] is not None else torch.from_numpy(_gaussian(s["seed"] + i, ms * l).reshape(ms, l)).cuda()
            omega = omega.double()
        out[i] = _polar64(D[i].cuda().double(), omega, case, s["schedule"])
    return out


def _theta64(R, start, n):
    """Upper estimate of the spectral norm: Lanczos on R^2, the largest Ritz value plus its residual, square root."""
    steps = min(20, n)
    Q = [start / torch.linalg.norm(start)]
    T = torch.zeros(steps, steps, dtype=torch.float64, device="cuda")
    for j in range(steps):
        w = R @ (R @ Q[j])
        T[j, j] = Q[j] @ w
        for _ in range(2):
            for q in Q:
                w = w - (q @ w) * q
        beta = torch.linalg.norm(w)
        if j + 1 == steps or float(beta) <= 1e-12 * abs(float(T[0, 0])):
            break
        T[j, j + 1] = T[j + 1, j] = beta
        Q.append(w / beta)
    lam, e = torch.linalg.eigh(T[:len(Q), :len(Q)])
    v = torch.stack(Q, dim=1) @ e[:, -1]
    return torch.sqrt(lam[-1].clamp(min=0) + torch.linalg.norm(R @ (R @ v) - lam[-1] * v))


def _ritz64(Z, V, case, deflate):
    V = _orth(V)
    Y = Z @ V
    H = V.T @ Y
    lam, e = torch.linalg.eigh(0.5 * (H + H.T))
    keep = torch.argsort(lam.abs(), descending=True)[:case["k"] if deflate else 0]
    return V @ e[:, keep], lam[keep], _orth(Y)


def _psd64(Z, V, start, case, sched, deflate=True):
    u, lam, basis = _ritz64(Z, V, case, deflate)
    R = Z - (u * lam) @ u.T
    X = R / _theta64(R, start, case["n"]) + (u * (torch.sign(lam) / case["gamma"])) @ u.T
    for a, b, c in sched:
        S = X @ X
        X = a * X + X @ (b * S + c * (S @ S))
    P = 0.5 * (R + R @ X) + (u * lam.clamp(min=0)) @ u.T
    return 0.5 * (P + P.T), basis


def _inv_root64(A, V, start, case):
    p, n = case["root"], case["n"]
    u, lam, basis = _ritz64(A, V, case, True)
    R = A - (u * lam) @ u.T
    theta = _theta64(R, start, n)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    M, Z = R / theta + (u @ u.T) / case["gamma"], eye
    pad, zpad = 1.0 / case["gamma"], 1.0
    for _ in range(case["steps"]):
        T = ((p + 1) * eye - M) / p
        t = (p + 1 - pad) / p
        Z, zpad = Z @ T, zpad * t
        for _ in range(p):
            M, pad = T @ M, pad * t
    out = theta ** (-1.0 / p) * (Z - zpad * (u @ u.T)) + (u * lam ** (-1.0 / p)) @ u.T
    return 0.5 * (out + out.T), basis


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "polar":
        return _polar64_batch(s["G"], s, case)
    if kind == "host":
        return _polar64_batch(s["G"], s, case).cpu()
    if kind == "muon":
        # the stored momentum and the look-ahead are bf16 numbers: what the step is a function of
        grad = s["grad"].double()
        M = (MU * s["M"].double() + grad).to(s["M"].dtype)
        D = (grad + MU * M.double()).to(M.dtype)
        return (1.0 - LR * DECAY) * s["W"].double() - LR * _polar64_batch(D, s, case), M.double()
    start = s["start"].double()
    if kind == "psd":
        return _psd64(s["X"].double(), s["V"].double(), start, case, s["schedule"])
    if kind == "invroot":
        return _inv_root64(s["A"].double(), s["V"].double(), start, case)
    C, rhs, X, S, V = (s[q].double() for q in ("C", "rhs", "X", "S", "V"))
    residuals = []
    for it in range(case["iters"]):
        y = rhs - torch.diagonal(X + S - C)
        S, V = _psd64(C - torch.diag(y) - X, V, start, case, s["schedule"], deflate=it >= 2)
        r = S + torch.diag(y) - C
        X = X + r
        obj, by = float((C * X).sum()), float(rhs @ y)
        residuals.append([float(torch.linalg.norm(torch.diagonal(X) - rhs)) / (1.0 + float(torch.linalg.norm(rhs))),
                          float(torch.linalg.norm(r)) / (1.0 + float(torch.linalg.norm(C))),
                          abs(obj - by) / (1.0 + abs(obj) + abs(by))])
    return X, S, y, torch.tensor(residuals, dtype=torch.float64)
