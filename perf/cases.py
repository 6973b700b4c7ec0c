"""The calls by which this library's speed is judged, and their 64-bit values.

A case is a dict of plain values.  `kind` says which public entry point it
takes, the other keys its sizes and options:

  step      Solver.set_state -> step(steps) -> get_state, page-locked buffers
  run       the same with run(): Algorithm 1's loop with energy and Delta m
  sweep     Batch.step over solvers of several sizes, parameters and seeds
  adjoint   Solver.adjoint: gradients of a loss on m(T)
  spectrum  hc_spectrum_noalloc: one transform on device buffers

Every pass starts from the same state (set_state is part of it), so a pass
repeats.  The fields follow the library's workloads: a source and a sink, or
one centred source, as Gaussians; a smooth permeability between 0.05 and 0.15,
or r = 0.1; m0 uniform.  The seed moves the sources and draws r and m0.

`exact` evaluates the scheme in 64 bits with torch alone: the pressure solved
to rounding instead of to the case's tolerance, the gradients by autograd.
"""
from __future__ import annotations

import ctypes
import itertools
import math

import torch

import paper_2606_06720_gb300 as hc
from paper_2606_06720_gb300 import _binding as abi  # the C entry points under their own names

DEV = "cuda:0"
F64 = torch.float64

# The parameter sweep: (c, D, gamma) triples over three grid sizes.
SWEEP = list(itertools.product((5.0, 10.0, 25.0, 50.0), (0.01, 0.02, 0.05, 0.1), (0.5, 0.75, 1.0)))
SWEEP_SIZES = (128, 256, 512)

# CG iterations that a step's solve takes, as `work` counts them: the loop's
# length depends on the data, and between 5 and 20 is ordinary.
NOMINAL_ITERATIONS = 10


def _step(name, n, precision, steps, **kw):
    case = {"name": name, "kind": "step", "n": "x".join(str(v) for v in n), "precision": precision,
            "steps": steps, "c": 25.0, "D": 0.02, "gamma": 0.5, "dt": 5e-4, "rtol": 1e-8,
            "precond": "kbar", "m_max": 0.5, "r": "smooth", "source": "pair"}
    case.update(kw)
    return case


def listed():
    return [
        # One small transform inside a host program that lends no memory: the
        # smallest call, two kernels.
        {"name": "spectrum_256", "kind": "spectrum", "n": "256x256"},
        # The smallest problem: 64^2 in plain FP64 to 1e-10, a teaching or
        # regression run, where launches and loop control count.
        _step("step_64_fp64", (64, 64), "fp64", 10, c=10.0, D=0.05, gamma=0.75, dt=1e-3, rtol=1e-10,
              precond="scalar", m_max=1.0, r="const", source="centre"),
        # An ordinary simulation: 512^2 with the defaults.
        _step("step_512", (512, 512), "fp32_refined", 10, precond="scalar"),
        # Production size: 2048^2, refined, several steps between two reads of
        # the state.
        _step("step_2048", (2048, 2048), "fp32_refined", 10),
        # The same grid coupled to a host program that takes the state every
        # step.
        _step("exchange_2048", (2048, 2048), "fp32_refined", 1),
        # Plain FP64, the mode for reference solutions.
        _step("step_1024_fp64", (1024, 1024), "fp64", 4),
        # Double-float refinement on a rectangle.
        _step("step_1024x512_df", (1024, 512), "fp32_refined_df", 10),
        # The paper's grid-convergence study: N = 400, not a power of two.
        _step("convergence_400", (400, 400), "fp64", 4, c=100.0, D=0.01, gamma=0.75, dt=0.05,
              rtol=1e-7, r="const", source="sink", m_max=1.0),
        # Algorithm 1 with its stopping rules watched: four sinks at 512^2.
        {"name": "run_512", "kind": "run", "n": "512x512", "precision": "fp32_refined", "steps": 8,
         "c": 200.0, "D": 0.0025, "gamma": 1.0, "dt": 0.005, "rtol": 1e-7, "precond": "kbar",
         "m_max": 1.0, "r": "const", "source": "four"},
        # 48 parameter triples at once, 16 on each of three grid sizes.
        {"name": "sweep_48", "kind": "sweep", "members": 48, "steps": 3, "dt": 1e-3, "rtol": 1e-8},
        # Gradients for fitting parameters and fields: checkpointed adjoint.
        dict(_step("adjoint_1024", (1024, 1024), "fp32_refined", 6), kind="adjoint", every=3),
        # The 3D case, refined.
        _step("step_256_3d", (256, 256, 256), "fp32_refined", 2, D=0.03, gamma=0.75, r="const",
              precond="scalar"),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def _smooth_size(rng, lo, hi):
    """A size in [lo, hi] with no prime factor above 5, spread over the logarithm."""
    sizes = sorted({2 ** a * 3 ** b * 5 ** c for a in range(12) for b in range(7) for c in range(5)
                    if lo <= 2 ** a * 3 ** b * 5 ** c <= hi})
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sizes, key=lambda v: abs(math.log(v / target)))


def draw(rng):
    kind = rng.choice(["spectrum", "step", "step", "step", "step3d", "generic", "run", "sweep",
                       "adjoint"])
    gamma = rng.choice([0.5, 0.5, 0.75, 1.0, 0.9, 1.5])
    common = {"c": round(math.exp(rng.uniform(math.log(5.0), math.log(50.0))), 3),
              "D": round(math.exp(rng.uniform(math.log(0.01), math.log(0.1))), 4),
              "gamma": gamma, "dt": rng.choice([2e-4, 5e-4, 1e-3]), "rtol": 1e-8,
              "precond": rng.choice(["kbar", "scalar"]), "m_max": rng.choice([0.5, 1.0]),
              "r": rng.choice(["smooth", "const"]), "source": rng.choice(["pair", "centre", "four"])}
    if kind == "spectrum":
        lx = rng.randint(3, 12)
        ly = rng.randint(3, min(12, 16 - lx))
        return {"kind": kind, "n": f"{1 << lx}x{1 << ly}"}
    if kind == "sweep":
        return {"kind": kind, "members": rng.randint(4, 48), "steps": rng.randint(1, 3), "dt": 1e-3,
                "rtol": 1e-8}
    if kind == "generic":
        nx, ny = _smooth_size(rng, 12, 800), _smooth_size(rng, 12, 800)
        if nx & (nx - 1) == 0 and ny & (ny - 1) == 0:
            nx = nx * 3 // 2  # both powers of two would take the other path
        return dict(common, kind="step", n=f"{nx}x{ny}", precision="fp64", steps=rng.randint(1, 4))
    precision = rng.choice(["fp32_refined", "fp32_refined", "fp64", "fp32_refined_df"])
    if kind == "step3d":
        lx, ly, lz = (rng.randint(4, 8) for _ in range(3))
        while lx + ly + lz > 22:
            lx, ly, lz = max(lx - 1, 4), max(ly - 1, 4), max(lz - 1, 4)
        return dict(common, kind="step", n=f"{1 << lx}x{1 << ly}x{1 << lz}", precision=precision,
                    steps=rng.randint(1, 2))
    if kind == "step":
        nx, ny = _pow2(rng, 5, 11), _pow2(rng, 5, 11)
        if precision == "fp64" and nx * ny > 1 << 20:
            nx //= 2
        most = 2 if precision == "fp64" else (4 if nx * ny > 1 << 20 else 10)
        return dict(common, kind=kind, n=f"{nx}x{ny}", precision=precision,
                    steps=rng.randint(1, most))
    nx, ny = _pow2(rng, 5, 10), _pow2(rng, 5, 10)
    if kind == "run":
        return dict(common, kind=kind, n=f"{nx}x{ny}", precision=rng.choice(["fp32_refined", "fp64"]),
                    steps=rng.randint(2, 8))
    steps = rng.randint(1, 6)
    return dict(common, kind=kind, n=f"{nx}x{ny}", precision=rng.choice(["fp32_refined", "fp64"]),
                steps=min(steps, 4), every=rng.randint(1, 4))


# ---------------------------------------------------------------- inputs


def _size(case):
    return tuple(int(v) for v in case["n"].split("x"))


def _members(case):
    """The sweep's members as cases of their own."""
    out = []
    for i in range(case["members"]):
        c, D, gamma = SWEEP[i]
        n = SWEEP_SIZES[i % 3]
        out.append({"kind": "step", "n": f"{n}x{n}", "precision": "fp32_refined", "c": c, "D": D,
                    "gamma": gamma, "dt": case["dt"], "rtol": case["rtol"], "precond": "scalar",
                    "m_max": 1.0, "r": "const", "source": "centre", "steps": case["steps"]})
    return out


def _nodes(n):
    """Coordinates x, y(, z) of the nodes of the unit square (cube), each
    shaped to broadcast over a field, x last."""
    dim = len(n)
    out = []
    for a, na in enumerate(n):
        shape = [1] * dim
        shape[dim - 1 - a] = na
        out.append((torch.arange(na, dtype=F64, device=DEV) / na).reshape(shape))
    return out


def _gaussian(xs, centre, inv):
    """exp(-inv |x - centre|^2) with the minimum-image distance."""
    d2 = 0.0
    for x, c in zip(xs, centre):
        d = x - c
        d = d - torch.round(d)
        d2 = d2 + d * d
    return torch.exp(-inv * d2)


def _fields(case, seed):
    """r, S, m0, p0 (and an adjoint's dL/dm(T)) of a case, FP64 on the GPU."""
    n = _size(case)
    dim, shape = len(n), tuple(reversed(n))
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * seed + 17)
    u = torch.rand(64, generator=g, device=DEV, dtype=F64).cpu().tolist()
    xs = _nodes(n)
    jit = [0.05 * (v - 0.5) for v in u[:6]]
    mid = [0.5 + jit[a] for a in range(dim)]
    if case["source"] == "pair":
        a, b = list(mid), list(mid)
        a[0], b[0] = 0.3 + jit[3], 0.7 + jit[4]
        S = _gaussian(xs, a, 200.0) - _gaussian(xs, b, 200.0)
    elif case["source"] == "centre":
        S = _gaussian(xs, mid, 200.0)
    elif case["source"] == "sink":
        S = _gaussian(xs, mid, 1000.0) - math.pi / 1000.0
    else:
        S = _gaussian(xs, mid, 1000.0)
        for cx, cy in ((0.2, 0.2), (0.2, 0.8), (0.8, 0.2), (0.8, 0.8)):
            S = S - 0.25 * _gaussian(xs, ([cx + jit[0], cy + jit[1]] + [0.5])[:dim], 1000.0)
    S = (S - S.mean()).expand(shape).contiguous()
    if case["r"] == "const":
        r = torch.full(shape, 0.1, dtype=F64, device=DEV)
    else:  # a trigonometric polynomial scaled into [-1, 1]
        f = 0.0
        for i in range(12):
            k = [1 + (i * 5 + a * 3 + int(8 * u[8 + i])) % 8 for a in range(dim)]
            phase = 2.0 * math.pi * u[24 + i]
            f = f + (0.5 + u[40 + i]) * torch.cos(
                2.0 * math.pi * sum((-1) ** (i + a) * k[a] * xs[a] for a in range(dim)) + phase)
        r = torch.clamp(0.1 + 0.05 * f / f.abs().max(), min=0.05).expand(shape).contiguous()
    m0 = case["m_max"] * torch.rand((dim,) + shape, generator=g, device=DEV, dtype=F64)
    out = {"r": r, "S": S, "m0": m0, "p0": torch.zeros(shape, dtype=F64, device=DEV)}
    if case["kind"] == "adjoint":  # 2 (m(T) - target) of two uniform fields
        target = case["m_max"] * torch.rand((dim,) + shape, generator=g, device=DEV, dtype=F64)
        out["lam"] = 2.0 * (m0 - target)
    return out


def _pinned(t):
    return torch.empty(t.shape, dtype=F64, pin_memory=True).copy_(t)


def _solver(case, fields, stream=None):
    s = hc.Solver(_size(case), c=case["c"], D=case["D"], gamma=case["gamma"], dt=case["dt"],
                  precision=case["precision"], cg_rtol=case["rtol"], precond=case["precond"],
                  device=DEV, stream=stream)
    s.set_r(fields["r"].cpu())
    s.set_source(fields["S"].cpu())
    return s


# ---------------------------------------------------------------- the calls


def prepare(case, seed):
    if case["kind"] == "spectrum":
        nx, ny = _size(case)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        f = torch.randn((ny, nx), generator=g, device=DEV, dtype=F64)
        return {"case": case, "f": f, "nx": nx, "ny": ny,
                "out": torch.empty((ny, nx // 2, 2), device=DEV, dtype=F64)}
    members = _members(case) if case["kind"] == "sweep" else [case]
    state = {"case": case, "solvers": [], "m": [], "p": [], "m_out": [], "p_out": []}
    for i, mc in enumerate(members):
        f = _fields(mc, seed + 7919 * i)
        state["solvers"].append(_solver(mc, f))
        state["m"].append(_pinned(f["m0"]))
        state["p"].append(_pinned(f["p0"]))
        if case["kind"] == "adjoint":
            state["lam"] = _pinned(f["lam"])
        elif case["kind"] != "sweep":
            state["m_out"].append(_pinned(f["m0"]))
            state["p_out"].append(_pinned(f["p0"]))
    if case["kind"] == "sweep":
        state["batch"] = hc.Batch(state["solvers"])
        # one result buffer per grid size, a slice for each member
        count = [len(range(k, len(members), 3)) for k in range(3)]
        state["all"] = [(torch.empty((count[k], 2, n, n), dtype=F64, pin_memory=True),
                         torch.empty((count[k], n, n), dtype=F64, pin_memory=True))
                        for k, n in enumerate(SWEEP_SIZES)]
        for i in range(len(members)):
            m, p = state["all"][i % 3]
            state["m_out"].append(m[i // 3])
            state["p_out"].append(p[i // 3])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "spectrum":
        rc = abi.hc_spectrum_noalloc(
            ctypes.cast(ctypes.c_void_p(state["f"].data_ptr()), ctypes.POINTER(ctypes.c_double)),
            ctypes.cast(ctypes.c_void_p(state["out"].data_ptr()), ctypes.POINTER(ctypes.c_double)),
            state["nx"], state["ny"],
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise hc.HuCaiError(rc, "hc_spectrum_noalloc")
        return state["out"]
    for s, m, p in zip(state["solvers"], state["m"], state["p"]):
        s.set_state(m, p)
    s = state["solvers"][0]
    if kind == "adjoint":
        g = s.adjoint(case["steps"], state["lam"], case["every"])
        return {"dc2": g["dc2"], "dD2": g["dD2"], "dr": g["dr"], "dS": g["dS"], "dm0": g["dm0"]}
    extra = {}
    if kind == "sweep":
        state["batch"].step(case["steps"])
    elif kind == "run":
        st = s.run(case["steps"], eps=1e-4, stop_on_energy=True)
        extra = {"energy": st.energy, "delta_m": st.delta_m}
    else:
        s.step(case["steps"])
    out = [s.get_state(m, p) for s, m, p in zip(state["solvers"], state["m_out"], state["p_out"])]
    if kind == "sweep":
        return [{"m": m, "p": p} for m, p in state["all"]]
    return dict({"m": out[0][0], "p": out[0][1]}, **extra)


def work(case):
    """Bytes: the fields in and out, once.  Flops: the real transforms of the
    solve and of the split step, 2.5 N log2 N each."""
    if case["kind"] == "sweep":
        parts = [work(c) for c in _members(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    n = _size(case)
    npts, dim = math.prod(n), len(n)
    fft = 2.5 * npts * math.log2(npts)
    if case["kind"] == "spectrum":
        return {"bytes": 16 * npts, "flops": fft}
    per_step = fft * (2 * dim * (NOMINAL_ITERATIONS + 1) + 3 * dim)
    sweeps = 3 if case["kind"] == "adjoint" else 1  # forward, recomputation, reverse
    return {"bytes": 8 * npts * (2 * (dim + 1) + 2), "flops": per_step * case["steps"] * sweeps}


# ---------------------------------------------------------------- 64-bit values


class _Spectral:
    """The scheme's Fourier variables on the unit square (cube), torch FP64.
    The first derivative is 0 at the Nyquist index; the diffusion keeps it."""

    def __init__(self, n):
        self.n, self.dim = n, len(n)
        self.shape = tuple(reversed(n))
        self.axes = tuple(range(-self.dim, 0))
        self.xi, self.xi2 = [], 0.0
        null = torch.ones(1, dtype=torch.bool, device=DEV)
        for a, na in enumerate(n):
            k = torch.arange(na // 2 + 1, device=DEV, dtype=F64)
            if a > 0:
                k = torch.fft.fftfreq(na, 1.0 / na, device=DEV, dtype=F64)
            shape = [1] * self.dim
            shape[self.dim - 1 - a] = k.numel()
            k = k.reshape(shape)
            d = torch.where(2 * k.abs() == na, torch.zeros_like(k), k)
            self.xi.append(2.0 * math.pi * d)
            self.xi2 = self.xi2 + (2.0 * math.pi * k) ** 2
            null = null & (d == 0)
        self.keep = (~null).to(F64)

    def fwd(self, f):
        return torch.fft.rfftn(f, dim=self.axes)

    def inv(self, F):
        return torch.fft.irfftn(F, s=self.shape, dim=self.axes)

    def project(self, f):
        return self.inv(self.fwd(f) * self.keep)

    def grad(self, f):
        F = self.fwd(f)
        return [self.inv(1j * x * F) for x in self.xi]

    def heat(self, f, D2, dt):
        return self.inv(self.fwd(f) * torch.exp(-D2 * dt * self.xi2))

    def apply(self, m, r, f):
        g = self.grad(f)
        mg = sum(a * b for a, b in zip(m, g))
        q = [mg * a + r * b for a, b in zip(m, g)]
        return -self.inv(sum(1j * x * self.fwd(v) for x, v in zip(self.xi, q)))

    def solve(self, m, r, S, p):
        """A p = S to rounding: CG preconditioned with the mean coefficient
        tensor, then once more on the residual."""
        dim = self.dim
        sym = 0.0
        for a in range(dim):
            for b in range(dim):
                k = (m[a] * m[b]).mean() + (r.mean() if a == b else 0.0)
                sym = sym + k * self.xi[a] * self.xi[b]
        pinv = torch.where(sym > 0, 1.0 / torch.where(sym > 0, sym, torch.ones_like(sym)),
                           torch.zeros_like(sym))
        S = self.project(S)
        target = 1e-15 * S.norm()
        for _ in range(2):
            res = S - self.apply(m, r, p)
            x = torch.zeros_like(p)
            d, rho = None, None
            best = res.norm()
            for it in range(400):
                z = self.inv(self.fwd(res) * pinv)
                rho_new = (res * z).sum()
                d = z if d is None else z + (rho_new / rho) * d
                rho = rho_new
                q = self.apply(m, r, d)
                alpha = rho / (d * q).sum()
                x = x + alpha * d
                res = res - alpha * q
                if it % 4 == 3:
                    now = res.norm()
                    if now <= target or not now < 1e3 * best:
                        break
                    best = torch.minimum(best, now)
            p = p + x
        return self.project(p)


def _relax(m, gamma, dt):
    n2 = sum(a * a for a in m)
    if gamma == 1.0:
        f = math.exp(-dt)
        return [a * f for a in m]
    e = 2.0 * (1.0 - gamma)
    pos = n2 > 0
    safe = torch.where(pos, n2, torch.ones_like(n2))
    x = -e * dt * safe ** (-0.5 * e)
    live = pos & (x > -1.0)
    f = torch.where(live, torch.exp(torch.log1p(torch.where(live, x, torch.zeros_like(x))) / e),
                    torch.zeros_like(x))
    return [a * f for a in m]


def _split(sp, m, p, c2, D2, gamma, dt):
    g = sp.grad(p)
    mg = sum(a * b for a, b in zip(m, g))
    z = c2 * dt * sum(b * b for b in g)
    small = z < 1e-8
    zs = torch.where(small, torch.ones_like(z), z)
    phi = torch.where(small, 1.0 + 0.5 * z, torch.expm1(zs) / zs)
    m = [a + c2 * dt * phi * mg * b for a, b in zip(m, g)]
    return [sp.heat(a, D2, dt) for a in _relax(m, gamma, dt)]


class _Solve(torch.autograd.Function):
    """p of A(m, r) p = S, differentiated as an exact solve."""

    @staticmethod
    def forward(ctx, sp, m, r, S, p0):
        p = sp.solve(list(m), r, S, p0)
        ctx.sp = sp
        ctx.save_for_backward(m, r, p)
        return p

    @staticmethod
    def backward(ctx, lam):
        sp = ctx.sp
        m, r, p = ctx.saved_tensors
        mu = sp.solve(list(m), r, lam, torch.zeros_like(p))
        gp, gu = sp.grad(p), sp.grad(mu)
        mp = sum(a * b for a, b in zip(m, gp))
        mu_m = sum(a * b for a, b in zip(m, gu))
        dm = torch.stack([-(mp * u + mu_m * q) for u, q in zip(gu, gp)])
        dr = -sum(u * q for u, q in zip(gu, gp))
        return None, dm, dr, mu, None


def _energy(sp, case, m, p, r):
    h = 1.0 / math.prod(sp.n)
    gp = sp.grad(p)
    mg = sum(a * b for a, b in zip(m, gp))
    gm2 = sum((b * b).sum() for a in m for b in sp.grad(a))
    n2 = sum(a * a for a in m)
    return float(h * (0.5 * case["D"] ** 2 * gm2 + 0.5 * case["c"] ** 2 *
                      ((r * sum(b * b for b in gp)).sum() + (mg * mg).sum()) +
                      (n2 ** case["gamma"]).sum() / (2.0 * case["gamma"])))


def _advance(case, seed):
    f = _fields(case, seed)
    sp = _Spectral(_size(case))
    m, p = list(f["m0"]), f["p0"]
    info = {}
    for _ in range(case["steps"]):
        p = sp.solve(m, f["r"], f["S"], p)
        new = _split(sp, m, p, case["c"] ** 2, case["D"] ** 2, case["gamma"], case["dt"])
        if case["kind"] == "run":
            info["energy"] = _energy(sp, case, m, p, f["r"])
            d2 = sum(((a - b) ** 2).sum() for a, b in zip(new, m))
            m2 = sum((b * b).sum() for b in m)
            info["delta_m"] = float(torch.sqrt(d2 / m2) / case["dt"])
        m = new
    return dict({"m": torch.stack(m).cpu(), "p": p.cpu()}, **info)


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        nx, ny = _size(case)
        F = torch.fft.fft2(prepare(case, seed)["f"])
        out = F[:, :nx // 2].clone()
        out[:, 0] = F[:, 0] + 1j * F[:, nx // 2]
        return torch.view_as_real(out).contiguous()
    if kind == "sweep":
        each = [_advance(c, seed + 7919 * i) for i, c in enumerate(_members(case))]
        return [{k: torch.stack([e[k] for e in each[size::3]]) for k in ("m", "p")}
                for size in range(3)]
    if kind != "adjoint":
        return _advance(case, seed)
    f = _fields(case, seed)
    sp = _Spectral(_size(case))
    m0, r, S = (f[k].clone().requires_grad_(True) for k in ("m0", "r", "S"))
    c2 = torch.tensor(case["c"] ** 2, dtype=F64, device=DEV, requires_grad=True)
    D2 = torch.tensor(case["D"] ** 2, dtype=F64, device=DEV, requires_grad=True)
    m, p = m0, f["p0"]
    for _ in range(case["steps"]):
        p = _Solve.apply(sp, m, r, S, p.detach())
        m = torch.stack(_split(sp, list(m), p, c2, D2, case["gamma"], case["dt"]))
    (m * f["lam"]).sum().backward()
    return {"dc2": float(c2.grad), "dD2": float(D2.grad), "dr": r.grad.cpu(), "dS": S.grad.cpu(),
            "dm0": m0.grad.cpu()}
