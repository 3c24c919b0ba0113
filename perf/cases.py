"""The work that users of this framework have it do, as timed cases.

A case is one call of a public entry point on inputs shaped like the framework's workloads: the
dynamic projector pair (forward and back-projection), the four-dimensional TV operators, the
filtered back-projection start, and whole solves (ADMM-CG and Chambolle-Pock).  Sizes come from the
repository's named workloads, its batched and serving streams and its tests.

Inputs are moving ellipsoids: coefficient volumes hold their masks times decaying temporal
coefficients (plus a little noise), projection data their closed-form line integrals plus noise.
"""
import math

import numpy as np
import torch

from paper_1809_09725_gb300 import dynrecon as dr

LAMBDA1, LAMBDA2 = 1e-3, 1.0
RHO = 10.0 * LAMBDA1
PRECS = {"f32": dr.F32, "bf16": dr.BF16, "f64": dr.F64, "f32_bf16fields": dr.F32 | dr.FIELDS_BF16}
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64, "f32_bf16fields": torch.float32}


def _case(name, op, nx, ny, nz, ns, K, halfturns, basis, m, nt, prec="f32", iters=0, n_cg=0, windows=0):
    return {"name": name, "op": op, "nx": nx, "ny": ny, "nz": nz, "ns": ns, "K": K, "halfturns": halfturns,
            "basis": basis, "m": m, "nt": nt, "prec": prec, "iters": iters, "n_cg": n_cg, "windows": windows}


def listed():
    return [
        # the smallest reconstruction: one 64^2 slice, 256 projections over 4 half-turns (host and launch latency)
        _case("solve_64_slice", "admm", 64, 64, 1, 64, 256, 4, "fourier", 4, 4, iters=3, n_cg=2),
        # an ordinary scan, 16 slices of 256^2, 10 half-turns: each operator of the pair by itself
        _case("forward_256", "fwd", 256, 256, 16, 256, 1800, 10, "fourier", 8, 10),
        _case("backward_256", "adj", 256, 256, 16, 256, 1800, 10, "fourier", 8, 10),
        # the same scan reconstructed: two ADMM iterations of 2 conjugate-gradient steps (more steps of a solve
        # amplify the rounding of single precision beyond what two runs can be compared at)
        _case("solve_256", "admm", 256, 256, 16, 256, 1800, 10, "fourier", 8, 10, iters=2, n_cg=2),
        # a chunk of slices of the large volume, 20 half-turns: the largest operator calls
        _case("forward_1024", "fwd", 1024, 1024, 8, 1024, 6000, 20, "legendre", 16, 20),
        _case("backward_1024", "adj", 1024, 1024, 8, 1024, 6000, 20, "legendre", 16, 20),
        # the shrink and dual update on that volume's frames (memory)
        _case("prox_1024", "prox", 1024, 1024, 8, 1024, 600, 20, "legendre", 16, 20),
        # a batched job with a ragged grid and angles that never repeat mod pi
        _case("backward_ragged", "adj", 203, 187, 9, 251, 721, 5, "legendre", 7, 6),
        # storage in bfloat16, a few small slices of a serving request
        _case("forward_128_bf16", "fwd", 128, 128, 6, 128, 720, 8, "legendre", 8, 8, prec="bf16"),
        # the filtered back-projection that starts a reconstruction, one window per half-turn
        _case("fbp_512", "fbp", 512, 512, 4, 512, 1800, 5, "legendre", 8, 5, windows=5),
        # Chambolle-Pock with the dual fields in bfloat16, as larger serving jobs run
        _case("primal_dual_256", "cp", 256, 256, 12, 256, 1080, 6, "fourier", 16, 6, prec="f32_bf16fields", iters=3),
        # the double-precision plan that results are checked with: forward of a small volume
        _case("forward_96_f64", "fwd", 96, 96, 4, 96, 480, 4, "fourier", 4, 4, prec="f64"),
    ]


def _cost(c):
    """Rough seconds of one pass, to keep drawn cases at most as dear as the largest listed one."""
    pairs = float(c["nx"]) * c["ny"] * c["nz"] * _distinct(c)
    field = 64.0 * c["nx"] * c["ny"] * c["nz"] * c["nt"]
    proj = pairs * c["m"]
    if c["prec"] == "f64":  # one transform per projection, on the double-precision pipe
        proj = 4.3 * float(c["nx"]) * c["ny"] * c["nz"] * c["K"] * (c["m"] + 10)
    times = {"fwd": 1, "adj": 1, "fbp": 2, "grad": 0, "grad_adj": 0, "normal": 0, "prox": 0}
    n = times.get(c["op"], 2 * max(c["iters"], 1) * (c["n_cg"] + 1))
    return proj * n / 1.2e12 + field * max(c["iters"], 1) / 4e12


def draw(rng):
    """One more case: any operator, sizes over the whole range of the listed ones."""
    top = 0.5 * max(_cost(c) for c in listed())
    while True:
        def log(a, b):
            return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

        op = rng.choice(["fwd", "fwd", "adj", "adj", "admm", "admm", "cp", "prox", "grad", "grad_adj", "normal", "fbp"])
        nx = log(48, 1024)
        ny = nx if rng.random() < 0.6 else max(48, min(1024, int(nx * rng.uniform(0.7, 1.4))))
        nz = log(1, 24)
        ns = max(nx, ny) if rng.random() < 0.6 else int(max(nx, ny) * rng.uniform(0.9, 1.4))
        halfturns = rng.randint(4, 20)
        # whole numbers of projections per half-turn repeat the angles mod pi; others never do
        K = halfturns * log(24, 300) if rng.random() < 0.75 else log(120, 1500)
        m = rng.choice([4, 8, 16, 16, 8, 12, 24, 32, 5, 7, 10])
        prec = rng.choice(["f32", "f32", "f32", "f32", "bf16", "f32_bf16fields", "f64"])
        c = _case("", op, nx, ny, nz, min(ns, 2048), K, halfturns, rng.choice(["fourier", "legendre"]), m, rng.randint(3, 20), prec)
        if op in ("fwd", "adj", "fbp") and prec == "f32_bf16fields":
            c["prec"] = "f32"
        if op in ("admm", "cp"):
            c["iters"] = 2 if op == "admm" else rng.randint(2, 3)
            c["n_cg"] = rng.randint(1, 2) if op == "admm" else 0
        if op == "fbp":
            c["windows"] = halfturns if rng.random() < 0.5 else 1
        del c["name"]
        if prec == "f64" and c["nx"] * c["ny"] * c["nz"] > 1 << 19:
            continue
        if _cost(c) <= top and c["nx"] * c["ny"] * c["nz"] * max(c["m"], 4 * c["nt"]) <= 1 << 30:
            return c


# --------------------------------------------------------------------------- inputs
def _geometry(c):
    k = np.arange(c["K"], dtype=np.float64)
    return math.pi * c["halfturns"] * k / c["K"], k / c["K"]


def _distinct(c):
    return c["K"] // math.gcd(c["K"], c["halfturns"])


def _basis(c, t):
    """phi_j(t): real Fourier or shifted Legendre, as an array [len(t)][m]."""
    t = np.asarray(t, dtype=np.float64)
    out = np.ones((t.size, c["m"]))
    if c["basis"] == "fourier":
        for j in range(1, c["m"]):
            a = 2.0 * math.pi * ((j + 1) // 2) * t
            out[:, j] = np.cos(a) if j & 1 else np.sin(a)
        return out
    return np.polynomial.legendre.legvander(2.0 * t - 1.0, c["m"] - 1)


def _blobs(c, seed):
    r = np.random.RandomState(seed % (1 << 32))
    lim = 0.5 * min(c["nx"], c["ny"])
    out = []
    for _ in range(12):
        A, B = r.uniform(0.06, 0.3, 2) * lim
        rad, ph = (lim - max(A, B)) * math.sqrt(r.uniform()), r.uniform(0, 2 * math.pi)
        sp, di = r.uniform(0, 0.06) * lim, r.uniform(0, 2 * math.pi)
        out.append(dict(A=A, B=B, C=max(2.0, r.uniform(0.3, 1.0) * c["nz"]), x=rad * math.cos(ph), y=rad * math.sin(ph),
                        z=r.uniform(-0.5, 0.5) * c["nz"], vx=sp * math.cos(di), vy=sp * math.sin(di),
                        psi=r.uniform(0, math.pi), a=r.uniform(0.2, 1.0) * (1.0 if r.uniform() < 0.7 else -0.5),
                        coef=r.standard_normal(c["m"])))
    return out


def _centres(n):
    return torch.arange(n, dtype=torch.float32, device="cuda") - 0.5 * (n - 1)


def _volume(c, seed, gen):
    """Coefficient volumes [nz][ny][nx][m]: ellipsoids times decaying coefficients, plus noise."""
    u = torch.randn((c["nz"], c["ny"], c["nx"], c["m"]), generator=gen, device="cuda").mul_(1e-3)
    X, Y, Z = _centres(c["nx"]), _centres(c["ny"]), _centres(c["nz"])
    decay = 1.0 / (1.0 + np.arange(c["m"])) ** 2
    for b in _blobs(c, seed):
        dx, dy = X[None, :] - b["x"], Y[:, None] - b["y"]
        cp, sp = math.cos(b["psi"]), math.sin(b["psi"])
        r2 = ((dx * cp + dy * sp) / b["A"]) ** 2 + ((dy * cp - dx * sp) / b["B"]) ** 2
        mask = (r2[None] + (((Z - b["z"]) / b["C"]) ** 2)[:, None, None] <= 1.0).float()
        amp = b["a"] * decay * (0.3 * b["coef"])
        amp[0] = b["a"]
        u.addcmul_(mask[..., None], torch.tensor(amp, dtype=torch.float32, device="cuda"))
    return u


def _data(c, seed, gen):
    """Projection data [nz][K][ns]: closed-form line integrals of the moving ellipsoids, 1 % noise."""
    theta, t = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in _geometry(c))
    g = torch.zeros((c["nz"], c["K"], c["ns"]), device="cuda")
    s, Z = _centres(c["ns"]), _centres(c["nz"])
    ct, st = torch.cos(theta), torch.sin(theta)
    for b in _blobs(c, seed):
        sc = torch.sqrt(torch.clamp(1.0 - ((Z - b["z"]) / b["C"]) ** 2, min=0.0))
        cen = (b["x"] + b["vx"] * t) * ct + (b["y"] + b["vy"] * t) * st
        q = (b["A"] * torch.cos(theta - b["psi"])) ** 2 + (b["B"] * torch.sin(theta - b["psi"])) ** 2
        d2 = (s[None, :] - cen[:, None]) ** 2
        amp = b["a"] * (1.0 + 0.3 * torch.sin(2 * math.pi * t + float(b["coef"][0])))
        for z in range(c["nz"]):
            f = float(sc[z])
            if f > 0.05:
                q2 = q * f * f
                chord = torch.sqrt(torch.clamp(q2[:, None] - d2, min=0.0))
                g[z].addcmul_(chord, (2.0 * b["A"] * b["B"] * f * f * amp / q2)[:, None])
    sigma = 0.01 * float(g.abs().max())
    for z in range(c["nz"]):
        g[z].add_(torch.randn((c["K"], c["ns"]), generator=gen, device="cuda"), alpha=sigma)
    return g


def _inputs(case, seed):
    """The call's input tensors, in the precision that the call takes."""
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dt = TORCH[c["prec"]]
    calc = torch.float64 if c["prec"] == "f64" else torch.float32
    fields = (c["nz"], c["nt"], c["ny"], c["nx"], 4)
    if c["op"] == "fwd" or c["op"] == "grad":
        return {"u": _volume(c, seed, gen).to(dt)}
    if c["op"] == "normal":
        return {"u": _volume(c, seed, gen).to(calc)}
    if c["op"] == "grad_adj":
        return {"p": torch.randn(fields, generator=gen, device="cuda").to(calc).mul_(LAMBDA1)}
    if c["op"] == "prox":
        mu = torch.randn(fields, generator=gen, device="cuda").to(calc).mul_(0.5 * LAMBDA1)
        return {"u": _volume(c, seed, gen).to(dt), "mu": mu}
    return {"g": _data(c, seed, gen).to(dt)}


def prepare(case, seed):
    c = case
    s = {"case": dict(c), **_inputs(c, seed)}
    theta, t = _geometry(c)
    s["plan"] = plan = dr.Plan(c["nx"], c["ny"], c["nz"], c["ns"], theta, t,
                               dr.FOURIER if c["basis"] == "fourier" else dr.LEGENDRE, c["m"], c["nt"], PRECS[c["prec"]])
    dt = getattr(torch, plan.storage_dtype)
    calc = getattr(torch, plan.field_dtype)
    if c["op"] in ("fwd", "adj", "fbp", "admm", "cp"):
        plan.autotune()
    if c["op"] == "fwd":
        s["out"] = torch.empty(plan.g_shape(), dtype=dt, device="cuda")
    elif c["op"] in ("adj", "fbp"):
        s["out"] = torch.empty(plan.u_shape(), dtype=dt, device="cuda")
    elif c["op"] == "grad":
        s["out"] = torch.empty(plan.field_shape(), dtype=calc, device="cuda")
    elif c["op"] == "grad_adj":
        s["out"] = torch.empty(plan.u_shape(), dtype=dt, device="cuda")
    elif c["op"] == "normal":
        s["out"] = torch.empty(plan.u_shape(), dtype=calc, device="cuda")
    elif c["op"] == "prox":
        s["out"] = torch.empty(plan.field_shape(), dtype=calc, device="cuda")
    else:
        s["out"] = torch.empty(plan.u_shape(), dtype=dt, device="cuda")
        if c["op"] == "admm":
            s["params"] = dr.solve_params(dr.ADMM_CG, iters=c["iters"], n_cg=c["n_cg"], lambda1=LAMBDA1, lambda2=LAMBDA2, rho=RHO)
        else:
            s["params"] = dr.solve_params(dr.CHAMBOLLE_POCK, iters=c["iters"], lambda1=LAMBDA1, lambda2=LAMBDA2, op_norm=_norm_bound(c))
    return s


def run(state):
    s, c, plan = state, state["case"], state["plan"]
    if c["op"] == "fwd":
        return dr.dyn_radon_fwd(plan, s["u"], s["out"])
    if c["op"] == "adj":
        return dr.dyn_radon_adj(plan, s["g"], s["out"])
    if c["op"] == "fbp":
        return dr.fbp_init(plan, s["g"], s["out"], c["windows"])
    if c["op"] == "grad":
        return dr.tv4d_grad(plan, s["u"], s["out"], LAMBDA2)
    if c["op"] == "grad_adj":
        return dr.tv4d_grad_adj(plan, s["p"], s["out"], LAMBDA2)
    if c["op"] == "normal":
        return dr.tv4d_normal(plan, s["u"], s["out"], LAMBDA2)
    if c["op"] == "prox":
        dr.tv4d_prox(plan, s["u"], s["mu"], s["out"], RHO, LAMBDA1, LAMBDA2)
        return {"mu": s["mu"], "w": s["out"]}
    s["out"].zero_()  # a reconstruction starts from zero
    res = dr.admm_solve(plan, s["g"], s["out"], s["params"])
    return {"u": s["out"], "objective": res["objective"]}


def work(case):
    """Bytes: each input read and each output written once.  Operations: the projector pair with one static transform
    per distinct angle mod pi (or per projection, whichever is less), 2 taps a sample; the stencils' sums over m."""
    c = case
    size = {"f32": 4, "bf16": 2, "f64": 8, "f32_bf16fields": 4}[c["prec"]]
    calc = 8 if c["prec"] == "f64" else 4
    V = float(c["nx"]) * c["ny"] * c["nz"]
    nu, ng, nf = V * c["m"], float(c["nz"]) * c["K"] * c["ns"], 4.0 * V * c["nt"]
    pair = min(4.0 * c["m"] * _distinct(c) * V + 2.0 * c["m"] * ng, c["K"] * V * (2.0 * c["m"] + 4.0))
    if c["op"] in ("fwd", "adj"):
        return {"bytes": (nu + ng) * size, "flops": pair}
    if c["op"] == "fbp":  # the filter as a convolution by fast transforms: 5 n log2 n each way
        n = 2.0 ** math.ceil(math.log2(2 * c["ns"]))
        return {"bytes": (nu + ng) * size, "flops": pair + ng / c["ns"] * 10.0 * n * math.log2(n)}
    sums = 2.0 * nf * c["m"]
    if c["op"] == "normal":
        return {"bytes": 2 * nu * calc, "flops": 4.0 * nu * c["m"]}
    if c["op"] == "grad":
        return {"bytes": nu * size + nf * calc, "flops": sums}
    if c["op"] == "grad_adj":
        return {"bytes": nu * size + nf * calc, "flops": sums / 2}
    if c["op"] == "prox":
        return {"bytes": nu * size + 3 * nf * calc, "flops": sums}
    field = 2 if c["prec"] == "f32_bf16fields" else calc
    if c["op"] == "admm":
        n = c["iters"]
        return {"bytes": (nu + ng) * size + n * 3 * nf * field, "flops": n * (2.0 * pair * (c["n_cg"] + 1) + 1.5 * sums)}
    return {"bytes": (nu + ng) * size + c["iters"] * 2 * nf * field, "flops": c["iters"] * (4.0 * pair + 2.5 * sums)}


# --------------------------------------------------------------------------- the same in 64 bits
def _groups(c):
    """Distinct angles mod pi with their projections: [(theta0, [(k, flipped)])]."""
    theta, _ = _geometry(c)
    out = {}
    for k, th in enumerate(theta):
        n = math.floor(th / math.pi + 1e-12)
        key = round((th - n * math.pi) * 1e9)
        out.setdefault(key, (th - n * math.pi, []))[1].append((k, n % 2 == 1))
    return list(out.values())


def _rays(c, th):
    """The Joseph samples of one angle: along-line pixel index below each sample and its fraction, [lines][ns]."""
    co, si = math.cos(th), math.sin(th)
    X = torch.arange(c["nx"], dtype=torch.float64, device="cuda") - 0.5 * (c["nx"] - 1)
    Y = torch.arange(c["ny"], dtype=torch.float64, device="cuda") - 0.5 * (c["ny"] - 1)
    s = torch.arange(c["ns"], dtype=torch.float64, device="cuda") - 0.5 * (c["ns"] - 1)
    rows = abs(co) >= abs(si)
    pos = ((s[None, :] - Y[:, None] * si) / co + 0.5 * (c["nx"] - 1)) if rows else ((s[None, :] - X[:, None] * co) / si + 0.5 * (c["ny"] - 1))
    low = torch.floor(pos)
    return rows, low.long(), pos - low, 1.0 / max(abs(co), abs(si))


def _static(c, u, th):
    """R_theta of every channel: u [nz][ny][nx][m] -> [nz][ns][m]."""
    rows, low, w, scale = _rays(c, th)
    v = u if rows else u.transpose(1, 2)
    n = v.shape[2]
    r = torch.arange(v.shape[1], device="cuda")[:, None]
    out = torch.zeros((u.shape[0], c["ns"], u.shape[3]), dtype=torch.float64, device="cuda")
    for i, wt in ((low, 1.0 - w), (low + 1, w)):
        wt = torch.where((i >= 0) & (i < n), wt, torch.zeros_like(wt))
        i = i.clamp(0, n - 1)
        for z in range(u.shape[0]):
            for j in range(0, r.shape[0], 128):
                out[z] += (v[z][r[j:j + 128], i[j:j + 128]] * wt[j:j + 128, :, None]).sum(0)
    return out * scale


def _static_adj(c, h, th):
    """The transpose of _static: h [nz][ns][m] -> [nz][ny][nx][m], written from the pixels' side."""
    co, si = math.cos(th), math.sin(th)
    X = torch.arange(c["nx"], dtype=torch.float64, device="cuda") - 0.5 * (c["nx"] - 1)
    Y = torch.arange(c["ny"], dtype=torch.float64, device="cuda") - 0.5 * (c["ny"] - 1)
    pos = X[None, :] * co + Y[:, None] * si + 0.5 * (c["ns"] - 1)
    half = max(abs(co), abs(si))
    low = torch.floor(pos)
    out = None
    for d in (0, 1):
        b = low + d
        wt = torch.clamp(1.0 - (pos - b).abs() / half, min=0.0) / half
        wt = torch.where((b >= 0) & (b < c["ns"]), wt, torch.zeros_like(wt))
        part = h[:, b.long().clamp(0, c["ns"] - 1)] * wt[None, :, :, None]
        out = part if out is None else out.add_(part)
    return out


def _fwd64(c, u):
    Phi = torch.tensor(_basis(c, _geometry(c)[1]), device="cuda")
    g = torch.empty((c["nz"], c["K"], c["ns"]), dtype=torch.float64, device="cuda")
    for th, members in _groups(c):
        r = _static(c, u, th)
        for k, flip in members:
            v = r @ Phi[k]
            g[:, k] = v.flip(1) if flip else v
    return g


def _adj64(c, g, table=None):
    Phi = torch.tensor(_basis(c, _geometry(c)[1]) if table is None else table, device="cuda")
    u = torch.zeros((c["nz"], c["ny"], c["nx"], c["m"]), dtype=torch.float64, device="cuda")
    for th, members in _groups(c):
        h = torch.zeros((c["nz"], c["ns"], c["m"]), dtype=torch.float64, device="cuda")
        for k, flip in members:
            h += (g[:, k].flip(1) if flip else g[:, k])[..., None] * Phi[k]
        u += _static_adj(c, h, th)
    return u


def _frames(c):
    P = _basis(c, np.arange(c["nt"]) / c["nt"])
    return torch.tensor(P, device="cuda")


def _diff(f, dim):
    d = torch.zeros_like(f)
    n = f.shape[dim]
    if n > 1:
        d.narrow(dim, 0, n - 1).copy_(f.narrow(dim, 1, n - 1) - f.narrow(dim, 0, n - 1))
    return d


def _diff_adj(p, dim):
    d = torch.zeros_like(p)
    n = p.shape[dim]
    if n > 1:
        d.narrow(dim, 0, n - 1).sub_(p.narrow(dim, 0, n - 1))
        d.narrow(dim, 1, n - 1).add_(p.narrow(dim, 0, n - 1))
    return d


def _grad64(c, u):
    """D u: [nz][nt][ny][nx][4]."""
    f = torch.einsum("lj,zyxj->zlyx", _frames(c), u)
    return torch.stack([_diff(f, 3), _diff(f, 2), _diff(f, 0), LAMBDA2 * _diff(f, 1)], -1)


def _grad_adj64(c, p):
    f = _diff_adj(p[..., 0], 3) + _diff_adj(p[..., 1], 2) + _diff_adj(p[..., 2], 0) + LAMBDA2 * _diff_adj(p[..., 3], 1)
    return torch.einsum("lj,zlyx->zyxj", _frames(c), f)


def _prox64(c, u, mu):
    d = _grad64(c, u)
    v = d + mu / RHO
    n = v.square().sum(-1, keepdim=True).sqrt()
    psi = v * torch.where(n > 0, torch.clamp(1.0 - (LAMBDA1 / RHO) / n, min=0.0), torch.zeros_like(n))
    mu = mu + RHO * (d - psi)
    return mu, psi - mu / RHO


def _norm_bound(c):
    """A bound on the norm of [R; D]: by its row and column sums, as a program that knows its geometry gives it."""
    Phi = _basis(c, _geometry(c)[1])
    P = _basis(c, np.arange(c["nt"]) / c["nt"])
    proj = math.sqrt(2.0) * math.hypot(c["nx"], c["ny"]) * np.linalg.norm(Phi, 2) ** 2
    return math.sqrt(proj + (12.0 + 4.0 * LAMBDA2 ** 2) * np.linalg.norm(P, 2) ** 2)


def _admm64(c, g):
    u = torch.zeros((c["nz"], c["ny"], c["nx"], c["m"]), dtype=torch.float64, device="cuda")
    mu = torch.zeros((c["nz"], c["nt"], c["ny"], c["nx"], 4), dtype=torch.float64, device="cuda")
    w = mu.clone()
    objective = []
    for _ in range(c["iters"]):
        r = _adj64(c, g - _fwd64(c, u)) + RHO * _grad_adj64(c, w - _grad64(c, u))
        p, rr = r.clone(), float(r.square().sum())
        for _ in range(c["n_cg"]):
            q = _adj64(c, _fwd64(c, p)) + RHO * _grad_adj64(c, _grad64(c, p))
            pq = float((p * q).sum())
            if not (pq > 0 and rr > 0):
                break
            u += rr / pq * p
            r -= rr / pq * q
            new = float(r.square().sum())
            p = r + new / rr * p
            rr = new
        mu, w = _prox64(c, u, mu)
        objective.append(_objective64(c, u, g))
    return u, objective


def _cp64(c, g):
    """Chambolle-Pock with step 0.99 / norm for both variables and extrapolation 1."""
    step = 0.99 / _norm_bound(c)
    u = torch.zeros((c["nz"], c["ny"], c["nx"], c["m"]), dtype=torch.float64, device="cuda")
    ut, h1 = u.clone(), torch.zeros_like(g)
    h2 = torch.zeros((c["nz"], c["nt"], c["ny"], c["nx"], 4), dtype=torch.float64, device="cuda")
    objective = []
    for _ in range(c["iters"]):
        h1 = (h1 + step * (_fwd64(c, ut) - g)) / (1.0 + step)
        h2 = h2 + step * _grad64(c, ut)
        n = h2.square().sum(-1, keepdim=True).sqrt()
        h2 = h2 * torch.where(n > LAMBDA1, LAMBDA1 / n, torch.ones_like(n))
        new = u - step * (_adj64(c, h1) + _grad_adj64(c, h2))
        ut, u = 2.0 * new - u, new
        objective.append(_objective64(c, u, g))
    return u, objective


def _objective64(c, u, g):
    tv = _grad64(c, u).square().sum(-1).sqrt().sum()
    return 0.5 * float((_fwd64(c, u) - g).square().sum()) + LAMBDA1 * float(tv)


def _fbp64(c, g):
    n = np.arange(-(c["ns"] - 1), c["ns"])
    taps = torch.tensor(-2.0 / (math.pi ** 2 * (4.0 * n * n - 1.0)), device="cuda")
    length = 4 * c["ns"]
    q = torch.fft.irfft(torch.fft.rfft(g, length) * torch.fft.rfft(taps, length), length)[..., c["ns"] - 1:2 * c["ns"] - 1]
    Phi = _basis(c, _geometry(c)[1])
    win = np.clip(np.floor(_geometry(c)[1] * c["windows"]), 0, c["windows"] - 1).astype(int)
    S = np.zeros((c["K"], c["windows"]))
    S[np.arange(c["K"]), win] = 1.0
    A = np.linalg.pinv(Phi, rcond=1e-6) @ S
    return _adj64(c, q, (math.pi / S.sum(0)[win])[:, None] * A[:, win].T)


def exact(case, seed):
    c = case
    # a solve in bfloat16 has its own rounding, and a large one takes too long
    pairs = float(c["nx"]) * c["ny"] * c["nz"] * c["m"] * _distinct(c)
    n = {"admm": 2 * c["iters"] * (c["n_cg"] + 2), "cp": 3 * c["iters"], "prox": 0, "grad": 0, "grad_adj": 0, "normal": 0}.get(c["op"], 1)
    if pairs * n > 2.5e11 or (n > 0 and _distinct(c) * n > 60000):
        return None
    x = {k: v.double() for k, v in _inputs(c, seed).items()}
    if c["op"] == "fwd":
        return _fwd64(c, x["u"])
    if c["op"] == "adj":
        return _adj64(c, x["g"])
    if c["op"] == "fbp":
        return _fbp64(c, x["g"])
    if c["op"] == "grad":
        return _grad64(c, x["u"])
    if c["op"] == "grad_adj":
        return _grad_adj64(c, x["p"])
    if c["op"] == "normal":
        return _grad_adj64(c, _grad64(c, x["u"]))
    if c["op"] == "prox":
        mu, w = _prox64(c, x["u"], x["mu"])
        return {"mu": mu, "w": w}
    u, objective = (_admm64 if c["op"] == "admm" else _cp64)(c, x["g"])
    return {"u": u, "objective": np.array(objective)}
