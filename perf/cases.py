"""Performance cases: whole passes through the public entry points of this package.

A forward pass is what a user's program does for one piece of a run: it sets the state to
the equilibrium of given fields, advances a number of steps and reads the density, the
velocity and the stored state (a restart file). A monitored pass reads the FP64 conserved
sums between groups of steps. A gradient pass is a differentiable rollout of the discrete
adjoint with its backward pass.
"""
from __future__ import annotations

import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_1312_3297_gb300 import D2Q9, D2Q9Cascaded, D3Q19
from paper_1312_3297_gb300.autograd import Rollout

AMP, PERIOD = 0.03, 1000.0  # prescribed relative velocity: A u~0(x) cos(2 pi t / P)


def _case(name, kind="run", lattice="d2q9", nx=64, ny=64, nz=1, mode="fluid", storage="fp32",
          flow="sine", steps=100):
    case = {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "mode": mode,
            "storage": storage, "flow": flow, "steps": steps}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the 64^2 parity workload: a unit-sized flow, bound by launches and latency
        _case("sine_64", nx=64, ny=64, steps=100),
        # a tiny ragged lattice for a few steps: the shortest call of an interactive session
        _case("ragged_63x41", nx=63, ny=41, mode="zero", steps=20),
        # the 512^2 crop of the reduced-precision workload
        _case("uniform_512_bf16", nx=512, ny=512, storage="bf16", flow="uniform", steps=200),
        # the headline: 4096^2 Taylor-Green vortex, analytic prescribed relative velocity
        _case("tg_4096", nx=4096, ny=4096, mode="analytic", flow="tg", steps=100),
        # the reduced-precision workload at full size, the largest
        _case("uniform_8192_fp16", nx=8192, ny=8192, storage="fp16", flow="uniform", steps=100),
        # Geier's cascaded scheme at a production size
        _case("cascaded_2048", lattice="cascaded", nx=2048, ny=2048, flow="tg", steps=100),
        # a channel-like lattice with a caller's relative-velocity field
        _case("field_1536x1000", nx=1536, ny=1000, mode="field", steps=50),
        # rows that no vector pack divides, 16-bit storage
        _case("ragged_4097x1999_fp16", nx=4097, ny=1999, storage="fp16", flow="uniform",
              steps=50),
        # the 3D Taylor-Green workload
        _case("tg3_256", lattice="d3q19", nx=256, ny=256, nz=256, flow="tg", steps=50),
        # a mid-sized 3D box in 16-bit storage whose rows leave a partial segment
        _case("uniform3_200x150x100_bf16", lattice="d3q19", nx=200, ny=150, nz=100,
              storage="bf16", flow="uniform", steps=50),
        # the adjoint workload: gradients of the final kinetic energy
        _case("gradient_1024", kind="gradient", nx=1024, ny=1024, mode="analytic", flow="shear",
              steps=200),
        # a run watched through its conserved sums every ten steps
        _case("monitor_1024x768", kind="monitor", nx=1024, ny=768, flow="uniform", steps=100),
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi]; half of the sizes rounded to a multiple of 8, the rest as
    they fall."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(8, v // 8 * 8) if rng.random() < 0.5 else v


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "run", "gradient", "monitor"])
    lattice = "d2q9" if kind == "gradient" else rng.choice(["d2q9", "d2q9", "cascaded", "d3q19"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    flow = rng.choice(["sine", "tg", "uniform"])
    if kind == "monitor" or storage != "fp32":
        flow = "uniform"  # sums of a mean flow; the flow that 16-bit storage is meant for
    steps = int(round(math.exp(rng.uniform(0.0, math.log(200.0)))))
    if lattice == "d3q19":
        nx, ny, nz = (_size(rng, 12, 288) for _ in range(3))
        nz = min(nz, (1 << 24) // (nx * ny))
        mode = rng.choice(["zero", "fluid", "field"])
        steps = min(steps, 50)
    else:
        nx, ny, nz = _size(rng, 24, 4096), _size(rng, 24, 4096), 1
        mode = rng.choice(["zero", "fluid", "analytic", "field"])
        if kind == "gradient":
            nx, ny = min(nx, 1024), min(ny, 1024)
            mode, flow, storage = rng.choice(["fluid", "analytic"]), "shear", "fp32"
            steps = max(4, min(steps, 100))
    if kind == "monitor":
        steps = max(10, steps // 10 * 10)
    return _case(None, kind, lattice, nx, ny, nz, mode, storage, flow, steps)


# ---------------------------------------------------------------- inputs
def _grid(case, dtype):
    """Angles 2 pi x / nx, ... of the nodes, shaped to broadcast over the lattice."""
    def axis(n):
        return torch.arange(n, device="cuda", dtype=dtype) * (2.0 * math.pi / n)

    x, y, z = axis(case["nx"]), axis(case["ny"]), axis(case["nz"])
    if case["lattice"] == "d3q19":
        return x[None, None, :], y[None, :, None], z[:, None, None]
    return x[None, :], y[:, None], None


def _shape(case):
    if case["lattice"] == "d3q19":
        return case["nz"], case["ny"], case["nx"]
    return case["ny"], case["nx"]


def _rates(case):
    if case["lattice"] == "d3q19":
        return [0, 0, 0, 0, 1.2] + [1.7] * 5 + [1.9] * 6 + [1.4] * 3
    return [0, 0, 0, 1.4, 1.8, 1.8, 1.2, 1.2, 1.4]


def _inputs(case, seed):
    """Seeded FP32 fields: rho, the velocity components and the base field u~0 (or None)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = _shape(case)
    dim = len(shape)

    def noise(scale):
        return scale * torch.randn(shape, generator=gen, device="cuda")

    x, y, z = _grid(case, torch.float32)
    flow = case["flow"]
    if flow == "uniform":
        rho = 1.0 + noise(1e-3)
        u = [U + noise(1e-3) for U in (0.05, 0.02, 0.01)[:dim]]
    elif flow == "sine":
        rho = 1.0 + noise(0.01)
        args = (y, x) if dim == 2 else (y, z, x)
        u = [0.05 * torch.sin(a) + noise(0.005) for a in args]
    elif flow == "shear":
        rho = torch.ones(shape, device="cuda")
        u = [0.05 * torch.sin(y) + noise(0.01), noise(0.01)]
    else:  # Taylor-Green vortex; the seed moves its centre and sets its strength
        a, b, c = (2.0 * math.pi * torch.rand(3, generator=gen, device="cuda")).tolist()
        u0 = 0.04 * (0.9 + 0.1 * float(torch.rand(1, generator=gen, device="cuda")))
        x, y = x + a, y + b
        if dim == 2:
            u = [-u0 * torch.cos(x) * torch.sin(y), u0 * torch.sin(x) * torch.cos(y)]
            rho = 1.0 - 0.75 * u0 * u0 * (torch.cos(2 * x) + torch.cos(2 * y))
        else:
            z = z + c
            u = [u0 * torch.sin(x) * torch.cos(y) * torch.cos(z),
                 -u0 * torch.cos(x) * torch.sin(y) * torch.cos(z),
                 torch.zeros(shape, device="cuda")]
            rho = 1.0 + (3.0 / 16.0) * u0 * u0 * (torch.cos(2 * x) + torch.cos(2 * y)) * (
                torch.cos(2 * z) + 2.0)
        u = [c.contiguous() for c in u]
        rho = rho.contiguous()
    ut0 = None
    if case["mode"] == "field":
        x, y, z = _grid(case, torch.float32)
        parts = [torch.sin(x + y), torch.cos(x) + 0.0 * y]
        if dim == 3:
            parts = [torch.sin(x + y + z), torch.cos(x + y + z), torch.sin(z - x + 0.0 * y)]
        ut0 = torch.stack([(p + noise(0.1)) for p in parts]).contiguous()
    return rho, u, ut0


def prepare(case, seed):
    rho, u, ut0 = _inputs(case, seed)
    mode = "prescribed" if case["mode"] in ("analytic", "field") else case["mode"]
    kw = {"mode": mode, "storage": case["storage"]}
    if case["lattice"] == "d3q19":
        sim = D3Q19(case["nx"], case["ny"], case["nz"], _rates(case), **kw)
    else:
        cls = D2Q9 if case["lattice"] == "d2q9" else D2Q9Cascaded
        sim = cls(case["nx"], case["ny"], _rates(case), **kw)
    if mode == "prescribed":
        sim.set_utilde(ut0, AMP, PERIOD)
    state = {"case": case, "sim": sim, "rho": rho, "u": u}
    if case["kind"] == "gradient":
        state["u0"] = torch.stack(u).requires_grad_()
        state["s_nu"] = torch.tensor(1.8, requires_grad=True)
        state["amp"] = torch.tensor(AMP, requires_grad=True)
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    n = case["steps"]
    if case["kind"] == "gradient":
        rho, u = Rollout.apply(state["u0"], state["s_nu"], state["amp"], sim, n, 0,
                               state["rho"])
        loss = 0.5 * (rho * (u * u).sum(0)).sum()
        g_u0, g_s, g_a = torch.autograd.grad(loss, (state["u0"], state["s_nu"], state["amp"]))
        return {"rho": rho, "u": u, "loss": loss, "g_u0": g_u0, "g_s_nu": g_s, "g_amp": g_a}
    sim.init_equilibrium(state["rho"], *state["u"])
    out = {}
    if case["kind"] == "monitor":
        out["sums"] = [sim.step_conserved(10) for _ in range(n // 10)][-1]
    else:
        sim.step(n)
    rho, *u = sim.moments()
    out.update({"rho": rho, "u": list(u), "state": sim.state()})
    return out


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the relaxation."""
    n = case["nx"] * case["ny"] * case["nz"]
    dim, q = (3, 19) if case["lattice"] == "d3q19" else (2, 9)
    size = 4 if case["storage"] == "fp32" else 2
    fields = 4 * (1 + dim) * n
    field = 4 * dim * n if case["mode"] == "field" else 0
    # floating-point operations of one relaxation, a fused multiply-add as two
    flops = {"d2q9": 160, "cascaded": 170, "d3q19": 340}[case["lattice"]] * n * case["steps"]
    if case["kind"] == "gradient":  # forward and a reverse step of about twice its arithmetic
        return {"bytes": 2 * fields + 4 * dim * n, "flops": 3 * flops}
    return {"bytes": 2 * fields + field + q * size * n, "flops": flops}


# ---------------------------------------------------------------- the scheme in 64 bits
_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
       (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_M2 = [(0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1), (1, 2), (2, 1), (2, 2)]
_M3 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2),
       (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 2, 0), (1, 0, 2), (2, 1, 0), (0, 1, 2),
       (2, 0, 1), (0, 2, 1), (2, 2, 0), (2, 0, 2), (0, 2, 2)]
# moment bases on the monomials of _M2 (x^3 = x and so on hold on the velocities only, so
# every polynomial is written with powers up to 2 per axis)
_BASIS = {
    "cascaded": [{0: 1}, {1: 1}, {2: 1}, {3: 1, 4: 1}, {3: 1, 4: -1}, {5: 1}, {6: 1}, {7: 1},
                 {8: 1}],
    "d3q19": [{0: 1}, {1: 1}, {2: 1}, {3: 1}, {4: 1, 5: 1, 6: 1}, {4: 1, 5: -1},
              {5: 1, 6: -1}] + [{k: 1} for k in range(7, 19)],
}


class _Exact:
    """The scheme of Section 1.2 in FP64 torch: moments m = M(0) d of the distance d to the
    equilibrium, shifted to the frame moving at u~ (m_k(u~) = sum_j P_k(v_j - u~) d_j),
    relaxed diagonally and shifted back (the shifts form a group)."""

    def __init__(self, lattice, s):
        self.lattice = lattice
        self.c = _C3 if lattice == "d3q19" else _C2
        self.dim = len(self.c[0])
        self.q = len(self.c)
        f64 = {"dtype": torch.float64, "device": "cuda"}
        self.w = [(1 / 3, 1 / 18, 1 / 36)[sum(map(abs, c))] if self.dim == 3
                  else (4 / 9, 1 / 9, 1 / 36)[sum(map(abs, c))] for c in self.c]
        self.s = s if torch.is_tensor(s) else torch.tensor(s, **f64)
        self.V = torch.tensor(self._matrix(), **f64)
        self.Vinv = torch.linalg.inv(self.V)
        self.D = [self._derivative(a) for a in range(self.dim)]

    def _poly(self, k, p):
        """Polynomial k at the point p."""
        if self.lattice == "d2q9":
            x, y = p
            r2 = x * x + y * y
            return [1.0, x, y, 3 * r2 - 4, x * x - y * y, x * y, x * (3 * r2 - 5),
                    y * (3 * r2 - 5), 4.5 * r2 * r2 - 10.5 * r2 + 4][k]
        mono = _M3 if self.dim == 3 else _M2
        return sum(a * math.prod(p[i] ** e for i, e in enumerate(mono[m]))
                   for m, a in _BASIS[self.lattice][k].items())

    def _matrix(self, axis=0, h=0.0):
        """P_k(v_j + h e_axis)."""
        return [[float(self._poly(k, [v + (h if a == axis else 0.0) for a, v in enumerate(c)]))
                 for c in self.c] for k in range(self.q)]

    def _derivative(self, axis):
        """Entries (k, l, D_kl) of dP_k / dX_axis = sum_l D_kl P_l, by the five-point
        difference that is exact for polynomials of degree 4."""
        f64 = {"dtype": torch.float64, "device": "cuda"}
        M = {h: torch.tensor(self._matrix(axis, h), **f64) for h in (-2.0, -1.0, 1.0, 2.0)}
        D = ((M[-2.0] - M[2.0] + 8.0 * (M[1.0] - M[-1.0])) / 12.0 @ self.Vinv).cpu()
        return [(k, l, float(D[k, l])) for k in range(self.q) for l in range(self.q)
                if abs(float(D[k, l])) > 1e-9]

    def shift(self, m, u, sign):
        """Moments in the frame moving at sign u from those at rest, P_k(v - sign u): the
        Taylor series exp(-sign u . D) m, which ends at the polynomials' degree 4."""
        out, term = list(m), list(m)
        for order in range(1, 5):
            nxt = [None] * self.q
            for a in range(self.dim):
                for k, l, v in self.D[a]:
                    if term[l] is not None:
                        t = (-sign * v / order) * u[a] * term[l]
                        nxt[k] = t if nxt[k] is None else nxt[k] + t
            term = nxt
            out = [o if t is None else o + t for o, t in zip(out, term)]
        return torch.stack(out)

    def moments(self, f):
        rho = f.sum(0)
        u = []
        for a in range(self.dim):
            plus = [j for j in range(self.q) if self.c[j][a] == 1]
            minus = [j for j in range(self.q) if self.c[j][a] == -1]
            u.append((sum(f[j] for j in plus) - sum(f[j] for j in minus)) / rho)
        return rho, u

    def feq(self, rho, u):
        out = []
        uu = sum(v * v for v in u)
        for w, c in zip(self.w, self.c):
            if self.lattice == "cascaded":
                fac = [2 / 3 - v * v if k == 0 else 0.5 * (1 / 3 + v * v + k * v)
                       for k, v in zip(c, u)]
                out.append(rho * fac[0] * fac[1])
            else:
                cu = sum(k * v for k, v in zip(c, u) if k) if any(c) else 0.0
                out.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu))
        return torch.stack(out)

    def _local(self, d, ut):
        """M(0)^{-1} T(-u~) S T(u~) M(0) d of every node."""
        m = torch.tensordot(self.V, d, 1)
        s = self.s.view((-1,) + (1,) * (d.dim() - 1))
        m = s * (m if ut is None else self.shift(m, ut, 1.0))
        return torch.tensordot(self.Vinv, m if ut is None else self.shift(m, ut, -1.0), 1)

    def step(self, f, ut):
        """One step: exact transport, then the relaxation. ut: "fluid", None or a list."""
        dims = tuple(range(self.dim))
        f = torch.stack([torch.roll(f[j], tuple(reversed(self.c[j])), dims) if any(self.c[j])
                         else f[j] for j in range(self.q)])
        rho, u = self.moments(f)
        return f - self._local(f - self.feq(rho, u), u if ut == "fluid" else ut)


def _relative(case, ut0, amp, k):
    if case["mode"] == "zero":
        return None
    if case["mode"] == "fluid":
        return "fluid"
    f = amp * math.cos(2.0 * math.pi * k / PERIOD)
    if case["mode"] == "field":
        return [f * c for c in ut0.double()]
    x, y, _ = _grid(case, torch.float64)
    one = torch.ones(_shape(case), dtype=torch.float64, device="cuda")
    return [f * torch.cos(y) * one, f * torch.sin(x) * one]


def exact(case, seed):
    n = case["nx"] * case["ny"] * case["nz"]
    # FP64 passes over the lattice: about 20 seconds at this many node steps
    cost = n * case["steps"] * (3.0 if case["lattice"] == "d3q19" else 1.0)
    if cost * (4.0 if case["kind"] == "gradient" else 1.0) > 4e9:
        return None
    rho, u, ut0 = _inputs(case, seed)
    rho, u = rho.double(), [v.double() for v in u]
    s = [float(v) for v in _rates(case)]
    if case["kind"] == "gradient":
        u0 = torch.stack(u).requires_grad_()
        s_nu = torch.tensor(1.8).double().cuda().requires_grad_()
        amp = torch.tensor(AMP).double().cuda().requires_grad_()
        one = torch.ones((), dtype=torch.float64, device="cuda")
        scheme = _Exact(case["lattice"], torch.stack(
            [s_nu if k in (4, 5) else one * v for k, v in enumerate(s)]))
        f = scheme.feq(rho, list(u0))
        for k in range(1, case["steps"] + 1):
            # s_nu and amp are reached through the closure: non-reentrant checkpoints keep them
            f = checkpoint(lambda g, k=k: scheme.step(g, _relative(case, ut0, amp, k)), f,
                           use_reentrant=False)
        r, v = scheme.moments(f)
        loss = 0.5 * (r * sum(c * c for c in v)).sum()
        used = (u0, s_nu, amp) if case["mode"] == "analytic" else (u0, s_nu)
        g = torch.autograd.grad(loss, used)
        g_amp = g[2] if len(g) == 3 else torch.zeros((), dtype=torch.float64)
        return {"rho": r.detach(), "u": torch.stack(v).detach(), "loss": loss.detach(),
                "g_u0": g[0], "g_s_nu": g[1], "g_amp": g_amp}
    with torch.no_grad():
        scheme = _Exact(case["lattice"], s)
        mean = [float((rho * c).sum() / rho.sum()) for c in u]
        one = torch.ones((1,) * len(_shape(case)), dtype=torch.float64, device="cuda")
        ref = scheme.feq(one, [m * one for m in mean])  # what the stored state is relative to
        f = scheme.feq(rho, u)
        for k in range(1, case["steps"] + 1):
            f = scheme.step(f, _relative(case, ut0, AMP, k))
        r, v = scheme.moments(f)
        out = {}
        if case["kind"] == "monitor":
            q = [float((r * c).sum()) for c in v] + [0.0] * (3 - len(v))
            out["sums"] = [float(r.sum()), *q, 0.0]
        out.update({"rho": r, "u": v, "state": f - ref})
        return out

