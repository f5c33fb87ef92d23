"""Performance cases: what users of the solver run, through its Python entry points.

Every case names one call on inputs of one size.  The kinds:
  apply   one LS-apply y = H u (Sec. 2): FP32 ("f32", the iteration's operator in mixed
          precision), FP64 ("fp64") or double-float ("df", the refinement residuals)
  inner   the inner level alone: GMRES on C v = A f preconditioned by Algorithm 2
  solve   the two-level solve H u = f, one right-hand side or a batch that shares H
  group   independent problems of different sizes solved concurrently
  net     one gradient evaluation of the learned step's network (forward, backward)

Sizes follow the repository's configurations (64^2, 1024^2 and 2048^2 at 10.24 points per
wavelength, the n/50-layer series 200..1600, the uneven sizes 256..1024 at n/64 layers)
with sizes in between, powers of two or not.  Media are seeded Gaussian bumps in a disk, or
one Gaussian disk for the layer series.
"""
import math

import numpy as np
import torch

from paper_1602_07652_gb300 import binding

PPW = 10.24     # grid points per wavelength
EXT = 10        # extension rows of a layer
DEV = "cuda"


def listed():
    return [
        # the smallest call: one operator application of a small problem in a user's own iteration
        {"name": "apply_f32_64", "kind": "apply", "form": "f32", "n": 64, "layers": 4},
        # a size that is no power of two (the layer series has t = 50 rows a layer)
        {"name": "apply_f32_800", "kind": "apply", "form": "f32", "n": 800, "layers": 16},
        # the operator of the mixed iteration at the benchmark's size
        {"name": "apply_f32_2048", "kind": "apply", "form": "f32", "n": 2048, "layers": 32},
        # the FP64-accurate apply behind the refinement residuals at the benchmark's size
        {"name": "apply_df_2048", "kind": "apply", "form": "df", "n": 2048, "layers": 32},
        # the FP64 operator of the all-FP64 configuration
        {"name": "apply_fp64_1024", "kind": "apply", "form": "fp64", "n": 1024, "layers": 16},
        # the inner level alone, as the layer series measures it
        {"name": "inner_fp64_400", "kind": "inner", "n": 400, "layers": 8, "tol": 1e-6},
        # the smallest full solve, all FP64
        {"name": "solve_fp64_64", "kind": "solve", "precision": "fp64", "n": 64, "layers": 4, "rhs": 1, "tol": 1e-8},
        # one right-hand side in mixed precision
        {"name": "solve_mixed_768", "kind": "solve", "precision": "mixed", "n": 768, "layers": 12, "rhs": 1, "tol": 1e-8},
        # many incident directions in one call, converged well below the discretisation error
        {"name": "solve_mixed_1024_b32", "kind": "solve", "precision": "mixed", "n": 1024, "layers": 16, "rhs": 32,
         "tol": 1e-10},
        # the benchmark's problem with a small batch of directions
        {"name": "solve_mixed_2048_b8", "kind": "solve", "precision": "mixed", "n": 2048, "layers": 32, "rhs": 8,
         "tol": 1e-10},
        # independent problems of different sizes in one call
        {"name": "group_mixed", "kind": "group", "sizes": "256,768,512,256", "tol": 1e-8},
        # the learned step's network: forward and backward of a batch of residual fields
        {"name": "net_grad_256", "kind": "net", "n": 256, "batch": 4, "channels": 32},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _layered(rng, lo, hi):
    """n = layers * t with t rows a layer in 24..80 and n near a log-uniform size in [lo, hi]."""
    t = rng.randint(24, 80)
    layers = max(1, min(round(_log(rng, lo, hi) / t), hi // t, 32))
    return layers * t, layers


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "inner", "solve", "solve", "solve", "group", "net"])
    if kind == "apply":
        form = rng.choice(["f32", "f32", "df", "fp64"])
        n, layers = _layered(rng, 48, {"f32": 2048, "df": 2048, "fp64": 1024}[form])
        return {"kind": kind, "form": form, "n": n, "layers": layers}
    if kind == "inner":
        n, layers = _layered(rng, 100, 500)
        return {"kind": kind, "n": n, "layers": layers, "tol": 1e-6}
    if kind == "solve":
        if rng.random() < 0.25:
            n, layers = _layered(rng, 48, 400)
            return {"kind": kind, "precision": "fp64", "n": n, "layers": layers, "rhs": rng.randint(1, 3), "tol": 1e-8}
        rhs = int(round(_log(rng, 1, 32)))
        n, layers = _layered(rng, 100, 1024)
        return {"kind": kind, "precision": "mixed", "n": n, "layers": layers, "rhs": rhs, "tol": 1e-8 if rhs == 1 else 1e-10}
    if kind == "group":
        return {"kind": kind, "sizes": ",".join(str(64 * rng.randint(2, 12)) for _ in range(rng.randint(2, 6))), "tol": 1e-8}
    return {"kind": kind, "n": 64 * rng.randint(2, 6), "batch": rng.randint(1, 4), "channels": rng.choice([16, 32])}


# ---------------------------------------------------------------- inputs
def _nodes(n):
    c = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) / n
    return c[None, :], c[:, None]   # x, z


def _bumps(n, rng):
    """20 seeded Gaussian bumps (sigma 0.02..0.08, amplitude -0.3..0.3) in the disk of radius 0.4."""
    x, z = _nodes(n)
    m = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    for _ in range(20):
        s, a = rng.uniform(0.02, 0.08), rng.uniform(-0.3, 0.3)
        r, p = (0.4 - 2 * s) * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        cx, cz = 0.5 + r * math.cos(p), 0.5 + r * math.sin(p)
        m += a * torch.exp(-(x - cx) ** 2 / (2 * s * s)) * torch.exp(-(z - cz) ** 2 / (2 * s * s))
    m[(x - 0.5) ** 2 + (z - 0.5) ** 2 > 0.16] = 0.0
    return m


def _disk(n, rng):
    """One Gaussian disk of either sign (the layer series' medium)."""
    x, z = _nodes(n)
    r2 = (x - 0.5) ** 2 + (z - 0.5) ** 2
    m = rng.choice([-0.2, 0.2]) * torch.exp(-r2 / (2 * rng.uniform(0.08, 0.12) ** 2))
    m[r2 > 0.09] = 0.0
    return m


def _wave(n, omega, theta):
    x, z = _nodes(n)
    return torch.exp(1j * omega * math.cos(theta) * x) * torch.exp(1j * omega * math.sin(theta) * z)


def _field(n, omega, rng, seed):
    """An oscillating field as the iteration sees it: a few plane waves and some noise."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    u = 0.1 * torch.randn((n, n), dtype=torch.complex128, device=DEV, generator=g)
    for _ in range(3):
        u += rng.uniform(0.3, 1.0) * _wave(n, omega, rng.uniform(0, 2 * math.pi))
    return u


def _omega(case, n):
    return 2 * math.pi * n / (10.0 if case["kind"] == "inner" else PPW)


def _sizes(case):
    return [int(s) for s in case["sizes"].split(",")]


def _draws(case, seed):
    """The seeded medium, angles and fields of a case: the same for prepare and exact."""
    rng = np.random.default_rng([seed, 1602])
    kind = case["kind"]
    if kind == "apply":
        n = case["n"]
        w = _omega(case, n)
        return _bumps(n, rng), _field(n, w, rng, seed)
    if kind == "inner":
        return _disk(case["n"], rng), rng.uniform(0, 2 * math.pi)
    if kind == "solve":
        base = rng.uniform(0, 2 * math.pi)
        return _bumps(case["n"], rng), [base + 2 * math.pi * k / case["rhs"] for k in range(case["rhs"])]
    if kind == "group":
        return [(_bumps(n, rng), rng.uniform(0, 2 * math.pi)) for n in _sizes(case)]
    n, b = case["n"], case["batch"]
    w = 2 * math.pi * n / PPW
    r = torch.stack([_field(n, w, rng, seed * 8 + k) for k in range(b)])
    e = torch.stack([_field(n, w, rng, seed * 8 + 4 + k) for k in range(b)])
    return r, torch.stack([_bumps(n, rng) for _ in range(b)]), e


def _net(case, seed):
    return binding.Net(levels=4, c0=case["channels"], max_batch=case["batch"], H=case["n"], W=case["n"], train=True,
                       seed=seed % 1000 + 1)


def prepare(case, seed):
    d = _draws(case, seed)
    kind = case["kind"]
    if kind == "group":
        torch.cuda.synchronize()   # the media, before the problems' own streams read them
        solvers, fs = [], []
        for n, (m, theta) in zip(_sizes(case), d):
            s = binding.Solver(m, _omega(case, n), layers=n // 64, ext=EXT, precision=binding.LS_MIXED,
                               stream=torch.cuda.Stream())
            s.ls_factor()
            solvers.append(s)
            fs.append(s.ls_incident_rhs(theta))
        torch.cuda.synchronize()
        return {"kind": kind, "solvers": solvers, "f": fs, "tol": case["tol"]}
    if kind == "net":
        r, m, e = d
        return {"kind": kind, "net": _net(case, seed), "r": r, "m": m, "e": e}
    n = case["n"]
    if kind == "apply":
        m, u = d
        fp64 = case["form"] == "fp64"
        s = binding.Solver(m, _omega(case, n), layers=case["layers"], ext=EXT,
                           precision=binding.LS_FP64 if fp64 else binding.LS_MIXED)
        u = u.to(torch.complex64) if case["form"] == "f32" else u
        call = {"f32": s.ls_apply_f32, "fp64": s.ls_apply, "df": s.ls_apply_double_float}[case["form"]]
        return {"kind": kind, "solver": s, "call": call, "u": u, "y": torch.empty_like(u)}
    m, theta = d
    if kind == "inner":
        s = binding.Solver(m, _omega(case, n), layers=case["layers"], ext=EXT, precision=binding.LS_FP64)
        s.ls_factor()
        g = s.ls_apply_A(s.ls_incident_rhs(theta))
        return {"kind": kind, "solver": s, "g": g, "tol": case["tol"]}
    o = binding.default_opts()
    if case["rhs"] > 1:   # above the iteration counts of these problems; bounds a batch's Krylov memory
        o.outer_restart, o.inner_restart = 10, 10
    mixed = case["precision"] == "mixed"
    s = binding.Solver(m, _omega(case, n), layers=case["layers"], ext=EXT, opts=o,
                       precision=binding.LS_MIXED if mixed else binding.LS_FP64)
    s.ls_factor()
    f = torch.stack([s.ls_incident_rhs(t) for t in theta]).contiguous()
    return {"kind": kind, "solver": s, "f": f, "u": torch.empty_like(f), "tol": case["tol"]}


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["call"](state["u"], state["y"])
    if kind == "inner":
        return state["solver"].ls_inner_solve(state["g"], state["tol"])[0]
    if kind == "solve":
        return state["solver"].ls_solve_batch(state["f"], state["tol"], state["u"])[0]
    if kind == "group":
        return binding.solve_group(state["solvers"], state["f"], state["tol"])[0]
    # learning rate 0: the gradients, for an optimiser of the caller's own
    loss = state["net"].train_step(state["r"], state["m"], state["e"], 0.0)
    return {"loss": loss, "grads": state["net"].get_grads()}


# ---------------------------------------------------------------- what a pass cannot do without
def _apply_work(n, cbytes):
    """u, y, m and the kernel's spectral quadrant once; zero-padded 2n x 2n transforms there and back."""
    return {"bytes": n * n * (2.5 * cbytes) + (n + 1.0) ** 2 * cbytes, "flops": 60.0 * n * n * math.log2(2 * n)}


def _factors_work(n, layers, cbytes, rhs):
    """Every factor matrix once, and one application of Algorithm 2 per right-hand side."""
    q = n // layers + 2 * EXT
    mats = 2.0 * layers * 3 * n
    return {"bytes": mats * q * q * cbytes, "flops": rhs * 2.0 * (2 * layers - 1) * 3.5 * n * 8 * q * q}


def _net_shapes(c0, levels=4):
    ch = [c0 * 2 ** l for l in range(levels)]
    out, prev = [], 3
    for l in range(levels):
        out += [("enc%d_a" % l, ch[l], prev, l), ("enc%d_b" % l, ch[l], ch[l], l)]
        prev = ch[l]
    for l in range(levels - 2, -1, -1):
        out += [("dec%d_up" % l, ch[l], ch[l + 1], l), ("dec%d_a" % l, ch[l], 2 * ch[l], l), ("dec%d_b" % l, ch[l], ch[l], l)]
    return out + [("head", 2, ch[0], 0)]


def work(case):
    kind = case["kind"]
    if kind == "apply":
        return _apply_work(case["n"], 8 if case["form"] == "f32" else 16)
    if kind == "net":
        px = case["batch"] * case["n"] ** 2
        macs = sum(9.0 * o * c * px / 4 ** l for _, o, c, l in _net_shapes(case["channels"]))
        params = sum(9 * o * c + o for _, o, c, _ in _net_shapes(case["channels"]))
        return {"bytes": px * (16 + 8 + 16) + params * 8.0, "flops": 6 * macs}
    parts = []
    if kind == "group":
        for n in _sizes(case):
            parts += [_apply_work(n, 8), _factors_work(n, n // 64, 8, 1), {"bytes": 32.0 * n * n, "flops": 0}]
    else:
        n, rhs = case["n"], case.get("rhs", 1)
        c = 8 if case.get("precision") == "mixed" else 16
        parts = [_factors_work(n, case["layers"], c, rhs), {"bytes": 32.0 * n * n * rhs, "flops": 0}]
        if kind == "solve":
            a = _apply_work(n, c)
            parts.append({"bytes": a["bytes"], "flops": rhs * a["flops"]})
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _hankel0(x):
    """H_0^(1)(x), x >= 0.3: its Laplace-type integral (2 / sqrt(pi)) int_0^oo e^(-t^2) / sqrt(1 + i t^2 / 2x) dt
    by the trapezoidal rule (the integrand is even and analytic for |Im t| < sqrt(x))."""
    step, acc = 0.0625, torch.full_like(x, 0.5, dtype=torch.complex128)
    for k in range(1, 104):
        t2 = (k * step) ** 2
        acc += math.exp(-t2) / torch.sqrt(torch.complex(torch.ones_like(x), t2 / (2 * x)))
    return acc * (2 * step / math.sqrt(math.pi)) * torch.sqrt(2 / (math.pi * x)) * torch.exp(1j * (x - math.pi / 4))


class _Convolution:
    """w^2 G * v on the n x n grid: the quadrature's kernel on a 2n x 2n torus by torch's FFT."""

    def __init__(self, n, omega):
        h = 1.0 / n
        d = torch.arange(n + 1, dtype=torch.float64, device=DEV)
        r = (d[None, :] ** 2 + d[:, None] ** 2).sqrt() * h * omega
        r[0, 0] = 1.0
        k = h * h * -0.25j * _hankel0(r)
        z0 = -math.log(2 * math.pi) - 2 * math.log(math.gamma(0.25) ** 2 / (2 * math.pi * math.sqrt(2.0)))
        c = math.log(omega * h / 2) + 0.57721566490153286061 + 0.5 * z0
        k[0, 0] = h * h * complex(c / (2 * math.pi), -0.25)
        k[n, :] = 0.0
        k[:, n] = 0.0
        fold = torch.cat([torch.arange(n + 1), torch.arange(n - 1, 0, -1)]).to(DEV)   # |offset| on the torus
        self.n, self.k = n, torch.fft.fft2(k[fold][:, fold]) * omega ** 2

    def __call__(self, v):
        n = self.n
        return torch.fft.ifft2(self.k * torch.fft.fft2(v, s=(2 * n, 2 * n)))[:n, :n]


def _gmres(op, b, tol=1e-13, most=1200):
    """Plain GMRES without restarts; None if it does not get to tol."""
    nb = torch.linalg.norm(b).item()
    V = torch.zeros((most + 1, b.numel()), dtype=b.dtype, device=b.device)
    V[0] = b.reshape(-1) / nb
    H = np.zeros((most + 1, most), dtype=np.complex128)
    for j in range(most):
        w = op(V[j].reshape(b.shape)).reshape(-1)
        for _ in range(2):
            c = V[:j + 1].conj() @ w
            w = w - c @ V[:j + 1]
            H[:j + 1, j] += c.cpu().numpy()
        H[j + 1, j] = torch.linalg.norm(w).item()
        V[j + 1] = w / H[j + 1, j].real
        if j % 10 == 9:
            e = np.zeros(j + 2, dtype=np.complex128)
            e[0] = nb
            y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
            if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= tol * nb:
                return (torch.from_numpy(y).to(b.device) @ V[:j + 1]).reshape(b.shape)
    return None


def _field_of(m, omega, theta):
    """The scattered field of one plane wave: u + w^2 G (m u) = -w^2 G (m u_I)."""
    n = m.shape[0]
    g = _Convolution(n, omega)
    return _gmres(lambda u: u + g(m * u), -g(m * _wave(n, omega, theta)))


def _net_exact(case, seed):
    r, m, e = _draws(case, seed)
    net = _net(case, seed)
    flat = net.get_params().double().to(DEV)
    net.close()
    p, at = {}, 0
    for name, o, c, _ in _net_shapes(case["channels"]):
        p[name] = (flat[at:at + 9 * o * c].reshape(o, c, 3, 3).requires_grad_(), flat[at + 9 * o * c:at + 9 * o * c + o].clone().requires_grad_())
        at += 9 * o * c + o
    s = r.abs().square().mean(dim=(1, 2), keepdim=True).sqrt()
    x = torch.stack([(r / s).real, (r / s).imag, m], dim=1)
    t = torch.stack([(e / s).real, (e / s).imag], dim=1)

    def conv(v, name):
        """A 3x3 convolution with zero padding, as nine products."""
        w, b = p[name]
        H, W = v.shape[2:]
        v = torch.nn.functional.pad(v, (1, 1, 1, 1))
        y = sum(torch.einsum("oc,bchw->bohw", w[:, :, i, j], v[:, :, i:i + H, j:j + W]) for i in range(3) for j in range(3))
        return y + b[None, :, None, None]

    skips, h = [], x
    for l in range(4):
        h = torch.nn.functional.avg_pool2d(h, 2) if l else h
        h = torch.relu(conv(torch.relu(conv(h, "enc%d_a" % l)), "enc%d_b" % l))
        skips.append(h)
    for l in (2, 1, 0):
        up = h.repeat_interleave(2, 2).repeat_interleave(2, 3)
        h = torch.cat([torch.relu(conv(up, "dec%d_up" % l)), skips[l]], dim=1)
        h = torch.relu(conv(torch.relu(conv(h, "dec%d_a" % l)), "dec%d_b" % l))
    loss = 0.5 * (conv(h, "head") - t).square().mean()
    loss.backward()
    return {"loss": loss.item(), "grads": torch.cat([g.grad.reshape(-1) for q in p.values() for g in q])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        m, u = _draws(case, seed)
        if case["form"] == "f32":
            u = u.to(torch.complex64).to(torch.complex128)
        return u + _Convolution(case["n"], _omega(case, case["n"]))(m * u)
    if kind == "inner":
        return None   # the sparsified operator has no form outside this repository
    if kind == "solve":
        if case["rhs"] * case["n"] ** 2 > 700000:
            return None
        m, thetas = _draws(case, seed)
        us = [_field_of(m, _omega(case, case["n"]), t) for t in thetas]
        return None if any(u is None for u in us) else torch.stack(us)
    if kind == "group":
        if sum(n * n for n in _sizes(case)) > 1200000:
            return None
        return [_field_of(m, _omega(case, n), t) for n, (m, t) in zip(_sizes(case), _draws(case, seed))]
    return _net_exact(case, seed)
