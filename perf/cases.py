"""Performance cases of the framework: what users of the collision operator have it do.

Each case is one pass through the public binding (paper_2004_11239_gb300): a collide, an RK4
step, a batched RK4 step, a Strang step of the inhomogeneous solver, or the creation of a plan.
Fields are complex64: the per-term arithmetic is FP32, and that is the type a caller keeps them
in when FP32 results are what is wanted.

`exact` evaluates the same operators in 64 bits with plain torch: the quadrature terms, the
weights F by the split of the paper's Sec. 4.1, the FFT convolution of eq. realQ, RK4 and the
spectral free streaming.
"""
import math

import numpy as np
import torch

import paper_2004_11239_gb300 as bz

SPHERE = (8, 12, 16, 18, 32, 50)          # points of the sphere rules in use (12: the icosahedron)
SPHERE_ODD = (9, 25, 49)                  # odd rules, complex data only
EPS = math.pi / 1000.0


def listed():
    return [
        # one evaluation of a small operator: the latency of a call (two Maxwellians, L = 10)
        dict(name="collide_n16", kind="collide", N=16, N_rho=16, M=12, gamma=0.0, s=0.5, R=9.0616, real=False),
        # serving geometry between the powers of two, soft potential, complex data
        dict(name="collide_n24", kind="collide", N=24, N_rho=24, M=12, gamma=-1.0, s=0.25, R=9.0616, real=False),
        # serving geometry on the chunked pipeline, real data
        dict(name="collide_n48_real", kind="collide", N=48, N_rho=48, M=12, gamma=-2.0, s=0.5, R=9.0616, real=True),
        # the largest grid, in both data forms
        dict(name="collide_n64_real", kind="collide", N=64, N_rho=32, M=12, gamma=-1.0, s=0.5, R=9.0616, real=True),
        dict(name="collide_n64", kind="collide", N=64, N_rho=16, M=12, gamma=-1.0, s=0.25, R=9.0616, real=False),
        # the headline solve: RK4 on the BKW domain at N = 32 with 1024 terms, in both data forms
        dict(name="rk4_n32_real", kind="rk4", N=32, N_rho=32, M=32, gamma=0.0, s=0.5, R=6.0, real=True, steps=2),
        dict(name="rk4_n32", kind="rk4", N=32, N_rho=32, M=32, gamma=0.0, s=0.5, R=6.0, real=False, steps=1),
        # many cells at once, gamma of their own: the collision step of a spatial solver
        dict(name="batch_n16", kind="batch", N=16, N_rho=16, M=32, gamma=0.0, s=0.5, R=6.0, real=False,
             capacity=256, active=251),
        dict(name="batch_n32_real", kind="batch", N=32, N_rho=32, M=12, gamma=0.0, s=0.25, R=6.0, real=True,
             capacity=16, active=16),
        # one Strang step of the spatially inhomogeneous solver
        dict(name="inhom_n16", kind="inhom", N=16, N_rho=16, M=12, gamma=0.0, s=0.5, R=6.0, real=False, nx=32),
        # the 2D operator
        dict(name="collide_2d_n64", kind="collide2d", N=64, N_rho=64, M=32, gamma=0.0, kernel="b4", R=6.0),
        # a new operator: what a solve with parameters of its own waits for first
        dict(name="plan_n32_real", kind="plan", N=32, N_rho=32, M=12, gamma=0.0, s=0.5, R=6.0, real=True),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["collide", "collide", "collide", "rk4", "rk4", "batch", "batch", "inhom", "collide2d", "plan"])
    c = dict(kind=kind, gamma=rng.choice([0.0, -1.0, -2.0]), R=rng.choice([6.0, 9.0616]))
    while True:
        if kind == "collide2d":
            c.update(N=rng.choice([8, 16, 32, 64]), N_rho=log_int(8, 64), M=rng.randint(8, 48),
                     kernel=rng.choice(["b1", "b2", "b3", "b4"]))
            if c["N_rho"] * c["M"] <= 2048:
                return c
            continue
        real = rng.random() < 0.5
        c.update(N=rng.choice([8, 16, 24, 32, 48, 64] if kind == "collide" else [8, 16, 24, 32]), N_rho=log_int(4, 64),
                 M=rng.choice(SPHERE if real else SPHERE + SPHERE_ODD), s=rng.choice([0.25, 0.5, 0.75]), real=real)
        unit = c["N_rho"] * c["M"] * c["N"] ** 3
        if kind == "collide" and unit <= 1.0e8:
            return c
        if kind == "rk4" and unit <= 3.3e7:
            c["steps"] = rng.randint(1, 2)
            return c
        if kind == "batch" and unit <= 6.0e6:
            c["capacity"] = min(256, log_int(3, max(4, 5.0e8 / unit)))
            c["active"] = rng.randint((c["capacity"] + 1) // 2, c["capacity"])
            return c
        if kind == "inhom" and unit <= 6.0e6:
            c["nx"] = rng.choice([8, 16, 24, 32])
            return c
        if kind == "plan" and unit <= 1.2e7:
            return c


def box_L(case):
    return (3.0 + math.sqrt(2.0)) * case["R"] / 4.0


def signed(N, device="cpu"):
    k = torch.arange(N, device=device, dtype=torch.float64)
    return torch.where(k < N // 2, k, k - N)


def device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def mixture(N, d, L, gen, count):
    """[count, N, ...] coefficients of two Maxwellians of mass 1/2 drifting apart at a speed near 2 in a
    direction of their own, temperatures near 1: the relaxation problem the solver is used for."""
    w = math.pi * signed(N, device()) / L
    u = torch.randn(count, d, generator=gen, dtype=torch.float64)
    u = u / u.norm(dim=1, keepdim=True) * (1.8 + 0.4 * torch.rand(count, 1, generator=gen, dtype=torch.float64))
    f = 0
    for side in (1.0, -1.0):
        c = (side * u).to(device())
        T = (0.8 + 0.4 * torch.rand(count, 1, generator=gen, dtype=torch.float64)).to(device())
        axes = [torch.exp(-1j * c[:, a:a + 1] * w - 0.5 * T * w * w) for a in range(d)]
        g = axes[0]
        for a in axes[1:]:
            g = g.unsqueeze(-1) * a.reshape(count, *([1] * (g.dim() - 1)), N)
        f = f + 0.5 * g
    return f / (2.0 * L) ** d


def inputs(case, seed):
    """The fields (complex64) and, for a batch, the slots and their gammas."""
    gen = torch.Generator().manual_seed(int(seed))
    N, L = case["N"], box_L(case)
    d = 2 if case["kind"] == "collide2d" else 3
    count = case.get("capacity", case.get("nx", 1))
    f = mixture(N, d, L, gen, count)
    if case["kind"] == "inhom":
        # a density wave over one profile whose cells differ a little
        wave = 1.0 + 0.2 * torch.cos(2 * math.pi * (torch.arange(count) / count + torch.rand(1, generator=gen)))
        f = (0.8 * f[:1] + 0.2 * f) * wave.to(f).reshape(count, 1, 1, 1)
    f = f.to(torch.complex64).contiguous()
    if case["kind"] != "batch":
        return (f if case["kind"] == "inhom" else f[0].clone()), None, None
    slots = torch.randperm(count, generator=gen)[:case["active"]].tolist()
    gammas = [[0.0, -1.0][int(v)] for v in torch.randint(0, 2, (count,), generator=gen)]
    return f, slots, gammas


def make_plan(case):
    if case["kind"] == "collide2d":
        return bz.bz_plan_create_ex(case["N"], box_L(case), case["R"], case["gamma"], 0.0, case["N_rho"], case["M"],
                                    kernel={"b1": bz.BZ_KERNEL_B1, "b2": bz.BZ_KERNEL_B2, "b3": bz.BZ_KERNEL_B3,
                                            "b4": bz.BZ_KERNEL_B4}[case["kernel"]], dim=2)
    return bz.bz_plan_create_ex(case["N"], box_L(case), case["R"], case["gamma"], case["s"], case["N_rho"], case["M"],
                                data=bz.BZ_DATA_REAL if case["real"] else bz.BZ_DATA_COMPLEX)


def prepare(case, seed):
    f, slots, gammas = inputs(case, seed)
    state = {"case": case, "f0": f, "slots": slots, "out": torch.empty_like(f)}
    if case["kind"] == "plan":
        # the operator's potential varies with the seed: a plan is made for parameters of its own
        state["case"] = dict(case, gamma=plan_gamma(case, seed))
        return state
    state["plan"] = make_plan(case)
    if case["kind"] in ("batch", "inhom"):
        state["batch"] = bz.bz_batch_create(state["plan"], case.get("capacity", case.get("nx")), 0)
        for slot, g in enumerate(gammas or []):
            bz.bz_batch_set_gamma(state["batch"], slot, g)
    return state


def plan_gamma(case, seed):
    return case["gamma"] + 0.01 * float(torch.rand(1, generator=torch.Generator().manual_seed(int(seed))))


DT = 0.01
LX = 4.0


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "plan":
        plan = make_plan(case)
        alpha = bz.bz_plan_alpha(plan, 0, plan.P)
        plan.close()
        return alpha
    out = state["out"]
    if kind in ("collide", "collide2d"):
        bz.bz_collide(state["plan"], state["f0"], out)
        return out
    out.copy_(state["f0"])                     # the solvers work in place
    if kind == "rk4":
        bz.bz_step_rk(state["plan"], out, 0.0, DT, case["steps"])
    elif kind == "batch":
        bz.bz_batch_step_rk(state["batch"], state["slots"], out, DT, 1)
    else:
        bz.bz_inhom_step(state["batch"], case["nx"], LX, out, DT, 1)
    return out


def work(case):
    """Fields in and out and the operator's weights once; the FFTs and products of every term, half of
    them where real data let two terms share a transform.  A new plan has its table to write."""
    N, P, d = case["N"], case["N_rho"] * case["M"], 2 if case["kind"] == "collide2d" else 3
    n = N ** d
    weights = 8.0 * n * P
    if case["kind"] == "plan":
        return {"bytes": weights, "flops": 0.0}
    half = 0.5 if case.get("real") else 1.0
    collides = {"rk4": 4 * case.get("steps", 1), "batch": 4 * case.get("active", 1),
                "inhom": 4 * case.get("nx", 1)}.get(case["kind"], 1)
    fields = case.get("active", case.get("nx", 1))
    flops = half * collides * P * n * (2 * 5 * d * math.log2(N) + 26)
    return {"bytes": half * weights + 16.0 * n * fields, "flops": flops}


# --- 64-bit evaluation -------------------------------------------------------------------------

def gauss(n, a, b):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (b - a) * x + 0.5 * (a + b), 0.5 * (b - a) * w


def directions(M, d):
    if d == 2:
        phi = 2 * math.pi * (np.arange(M) + 0.5) / M
        return np.stack([np.cos(phi), np.sin(phi)], 1), np.full(M, 2 * math.pi / M)
    if M == 12:
        g = (1 + math.sqrt(5)) / 2
        v = [p for a in (-1, 1) for b in (-1, 1) for p in ((0, a, b * g), (a, b * g, 0), (b * g, 0, a))]
        return np.array(v) / math.hypot(1, g), np.full(12, 4 * math.pi / 12)
    n = round(math.sqrt(M / 2))
    nt, npz = (n, 2 * n) if 2 * n * n == M else (math.isqrt(M), math.isqrt(M))
    ct, wt = gauss(nt, -1, 1)
    phi = 2 * math.pi * (np.arange(npz) + 0.5) / npz
    st = np.sqrt(1 - ct ** 2)
    q = np.stack([np.outer(st, np.cos(phi)), np.outer(st, np.sin(phi)), np.outer(ct, np.ones(npz))], -1)
    return q.reshape(-1, 3), np.repeat(wt, npz) * 2 * math.pi / npz


def angular(case):
    """g(theta) and its moments over [0, EPS]: (1 - cos), (1 - cos)^2, sin^2 (the Taylor part)."""
    if case["kind"] == "collide2d":
        c, b, cosine = {"b1": (1 / (2 * math.pi), 0.0, 0), "b2": (3 / 32, -1.0, 0), "b3": (1 / (8 * math.pi), -2.0, 0),
                        "b4": (5 / 256, -2.5, 1)}[case["kernel"]]
    else:
        s = case["s"]
        beta = math.exp(math.lgamma(1 - s) + math.lgamma(1.5) - math.lgamma(2.5 - s))
        c, b, cosine = 1 / (12 * math.pi * beta), -1 - 2 * s, 0

    def g(t):
        return c * np.sin(t / 2) ** b * (np.abs(np.cos(t / 2)) if cosine else 1.0)

    def moment(m):                             # int_0^EPS g (2 sin^2(t/2))^m dt with t = EPS u^4
        u, w = gauss(48, 0, 1)
        t = EPS * u ** 4
        return float(np.sum(w * 4 * EPS * u ** 3 * g(t) * (2 * np.sin(t / 2) ** 2) ** m))

    return g, (moment(1), moment(2), 2 * moment(1) - moment(2))


def theta_rule(z, g):
    width = min(0.25, 8.0 / max(z, 1e-9))
    edges = [EPS]
    while edges[-1] < 0.25:
        edges.append(min(2 * edges[-1], edges[-1] + width, 0.25))
    edges += list(np.linspace(0.25, math.pi, math.ceil((math.pi - 0.25) / width) + 1)[1:])
    t, w = (np.concatenate(v) for v in zip(*(gauss(20, a, b) for a, b in zip(edges, edges[1:]))))
    return t, w * g(t)


def weights(case):
    """c_p F(k, r_i, q_j) for every term and mode, [P, N, ...] complex128, with beta's axes [P, d, N]
    and r_i per term."""
    dev, N, L, M = device(), case["N"], box_L(case), case["M"]
    d = 2 if case["kind"] == "collide2d" else 3
    g, A = angular(case)
    r, wr = gauss(case["N_rho"], 0.0, case["R"])
    q, wq = directions(M, d)
    # half of the grid widened to -N/2 .. N/2 on every axis: F(-k) = conj F(k) gives the rest
    pos = torch.arange(0, N // 2 + 1, device=dev, dtype=torch.float64)
    full = torch.arange(-N // 2, N // 2 + 1, device=dev, dtype=torch.float64)
    ks = torch.stack(torch.meshgrid(pos, *([full] * (d - 1)), indexing="ij"), -1).reshape(-1, d)
    idx = torch.stack(torch.meshgrid(*([signed(N, dev).long()] * d), indexing="ij"), -1).reshape(-1, d)
    neg = idx[:, 0] < 0
    at = torch.where(neg[:, None], -idx, idx)
    flat = at[:, 0]
    for a in range(1, d):
        flat = flat * (N + 1) + at[:, a] + N // 2
    qd = torch.tensor(q, device=dev)
    out = torch.empty(case["N_rho"] * M, N ** d, dtype=torch.complex128, device=dev)
    kk = (ks * ks).sum(-1)
    group = max(1, (1 << 18) // ks.shape[0])
    for i in range(case["N_rho"]):
        a = math.pi * r[i] / (2 * L)
        t, W = (torch.tensor(v, device=dev) for v in theta_rule(a * math.sqrt(d) * N / 2, g))
        omc, sn = 2 * torch.sin(t / 2) ** 2, torch.sin(t)
        for j in range(0, M, group):
            kap = qd[j:j + group] @ ks.T
            if d == 3:
                perp = (kk - kap * kap).clamp(min=0).sqrt()
            else:
                perp = torch.stack([-qd[j:j + group, 1], qd[j:j + group, 0]], 1) @ ks.T
            x, y = (a * kap).reshape(-1, 1), (a * perp).reshape(-1, 1)
            re = torch.zeros_like(x[:, 0])
            im = torch.zeros_like(re)
            for n in range(0, len(t), 16):
                ys = y * sn[n:n + 16]
                if d == 3:
                    u = -0.25 * ys * ys
                    series = u * (1 + u / 4 * (1 + u / 9 * (1 + u / 16 * (1 + u / 25 * (1 + u / 36)))))
                    jm = torch.where(ys.abs() < 0.25, series, torch.special.bessel_j0(ys) - 1)
                else:
                    jm = -2 * torch.sin(ys / 2) ** 2
                h = 0.5 * x * omc[n:n + 16]
                sh, ch = torch.sin(h), torch.cos(h)
                re += (jm - 2 * sh * sh * (1 + jm)) @ W[n:n + 16]
                im += (2 * sh * ch * (1 + jm)) @ W[n:n + 16]
            x, y = x[:, 0], y[:, 0]
            c1, c2 = (0.25, 2 * math.pi) if d == 3 else (0.5, 2.0)
            re = c2 * (re - 0.5 * x * x * A[1] - c1 * y * y * A[2])
            im = c2 * (im + x * A[0])
            F = torch.complex(re, im).reshape(-1, ks.shape[0])[:, flat]
            F = torch.where(neg, F.conj(), F)
            c = torch.tensor(wr[i] * wq[j:j + group] * r[i] ** (case["gamma"] + d - 1), device=dev)
            out[i * M + j:i * M + min(j + group, M)] = c[:, None] * F
    m = signed(N, dev)
    rp = torch.tensor(np.repeat(r, M), device=dev)
    beta = torch.exp(-1j * math.pi / L * rp[:, None, None] * qd.repeat(case["N_rho"], 1)[:, :, None] * m)
    return out.reshape(-1, *([N] * d)), beta, rp


def operator(case, gammas=None):
    """Q of a [count, N, ...] field, eq. realQ term by term; gammas: one exponent per field."""
    alpha, beta, rp = weights(case)
    d, n = alpha.dim() - 1, alpha[0].numel()
    axes = tuple(range(1, d + 1))
    scale = None
    if gammas is not None:
        scale = rp[:, None] ** (torch.tensor(gammas, device=rp.device, dtype=torch.float64) - case["gamma"])

    def Q(f):
        if case.get("real"):                   # the band-limited real part of the data
            N = case["N"]
            f = 0.5 * (f + f.flip(axes).roll((1,) * d, axes).conj())
            keep = torch.arange(N, device=f.device) != N // 2
            f = f * (keep[:, None, None] & keep[:, None] & keep)
        h = torch.fft.ifftn(f, dim=axes) * n
        out = torch.zeros_like(f)
        for p in range(alpha.shape[0]):
            b = beta[p, 0]
            for a in range(1, d):
                b = b.unsqueeze(-1) * beta[p, a]
            u = torch.fft.fftn(torch.fft.ifftn(f * b, dim=axes) * h, dim=axes) * alpha[p]
            out += u if scale is None else u * scale[p].reshape(-1, *([1] * d))
        return out

    return Q


def rk4(Q, f, steps):
    for _ in range(steps):
        k1 = Q(f)
        k2 = Q(f + 0.5 * DT * k1)
        k3 = Q(f + 0.5 * DT * k2)
        k4 = Q(f + DT * k3)
        f = f + DT / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return f


def stream(f, L, t):
    """Free streaming of the [nx, N, N, N] cells along v_1, exact at the velocity nodes."""
    nx, N = f.shape[:2]
    sign = (1 - 2 * (torch.arange(N, device=f.device) % 2)).reshape(1, N, 1, 1).to(f)
    v = -L + 2 * L * torch.arange(N, device=f.device, dtype=torch.float64) / N
    g = torch.fft.fft(torch.fft.ifft(f * sign, dim=1), dim=0)
    g = g * torch.exp(-2j * math.pi * t / LX * signed(nx, f.device)[:, None] * v)[:, :, None, None]
    return torch.fft.fft(torch.fft.ifft(g, dim=0), dim=1) * sign


def exact(case, seed):
    if case["kind"] == "plan":
        w = weights(dict(case, gamma=plan_gamma(case, seed)))[0]
        return w / case["N"] ** 3
    f, slots, gammas = inputs(case, seed)
    f = f.to(torch.complex128)
    if case["kind"] in ("collide", "collide2d"):
        return operator(case)(f[None])[0]
    if case["kind"] == "rk4":
        return rk4(operator(case), f[None], case["steps"])[0]
    if case["kind"] == "batch":
        out = f.clone()
        out[slots] = rk4(operator(case, [gammas[b] for b in slots]), f[slots], 1)
        return out
    L = box_L(case)
    return stream(rk4(operator(case), stream(f, L, DT / 2), 1), L, DT / 2)
