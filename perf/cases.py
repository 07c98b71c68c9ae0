"""What a user of this framework has it do, as cases that can be timed and
checked: runs of the stream + collide step from given macroscopic fields to the
fields some steps later, runs with diagnostics on the way, restarts from saved
populations, and gradients through a run, through the package's public entry
points.  Sizes and options are those of bench.py, of the tests and of the
workloads they name; ``draw`` gives more cases of the same ranges.

``exact`` is a plain torch FP64 restatement of the method (Bauer & Ruede,
arXiv:1803.04937: Eq. 14-17 and 22, Sec. 3.2-3.3, Sec. 5.1) that shares no code
with the package.
"""
import itertools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

DEVICE = "cuda"

# ---------------------------------------------------------------- cases

_DEFAULTS = dict(kind="run", precision="f32", pattern="ab", collision="srt", equilibrium="improved", tau=0.8,
                 walls="", force_x=0.0, stencil=19, samples=1)


def _case(**kw):
    return dict(_DEFAULTS, **kw)


def _channel_force(tau, ny):
    """Body force that drives a channel of ny layers to a centre velocity of 0.05."""
    return 8.0 * (tau - 0.5) / 3.0 * 0.05 / ny ** 2


def listed():
    return [
        # the smallest lattice of the tests and the smoke run: a vortex followed for 100 short steps
        _case(name="vortex_32_f32", nx=32, ny=32, nz=32, steps=100),
        # the headline workload of bench.py (periodic 256^3, SRT, tau 0.8, two grids) in its FP32 storage ...
        _case(name="wave_256_f32", nx=256, ny=256, nz=256, steps=100),
        # ... and in 16-bit storage, the throughput mode
        _case(name="wave_256_f16", nx=256, ny=256, nz=256, steps=100, precision="f16s"),
        # the walled channel of bench.py: half-way bounce-back in y, TRT, body force
        _case(name="channel_512_f32", nx=512, ny=256, nz=256, steps=50, collision="trt", tau=0.6, walls="y",
              force_x=_channel_force(0.6, 256)),
        # decaying turbulence on bench.py's largest lattice, one grid (in-place AA) to save memory
        _case(name="turbulence_768_f32", nx=768, ny=768, nz=768, steps=16, tau=0.51, pattern="aa"),
        # the same flow at the resolution of the long runs, 16-bit and in place, its energy and enstrophy
        # written down on the way
        _case(name="turbulence_192_f16_monitored", nx=192, ny=192, nz=192, steps=25, samples=4, tau=0.51,
              precision="f16s", pattern="aa", kind="monitor"),
        # the paper's square duct (Sec. 5.1) in FP64: invariant along x, so only four cells long
        _case(name="duct_96_f64", nx=4, ny=96, nz=96, steps=200, precision="f64", collision="trt", tau=0.8,
              walls="yz", force_x=1e-6),
        # a closed box (walls on all axes) with the second 16-bit type and the standard equilibrium
        _case(name="box_256x192x160_bf16", nx=256, ny=192, nz=160, steps=50, precision="bf16s", collision="trt",
              equilibrium="standard", tau=0.7, walls="xyz", force_x=1e-6),
        # a lattice whose rows fit no vector width (190 = 2 mod 4)
        _case(name="ragged_190x131x97_f16", nx=190, ny=131, nz=97, steps=50, precision="f16s", tau=0.7),
        # the 27-velocity comparison lattice of the paper's cost remark (Sec. 6)
        _case(name="d3q27_256_f32", nx=256, ny=256, nz=256, steps=40, stencil=27, equilibrium="standard"),
        # multi-relaxation-time run continued in place from saved populations and saved again
        _case(name="restart_mrt_160x144x99_f32", nx=160, ny=144, nz=99, steps=50, collision="mrt", tau=0.65,
              pattern="aa", kind="restart"),
        # gradient of a final-velocity misfit with respect to the initial velocity and tau, on the lattice of
        # bench.py's adjoint workload
        _case(name="gradient_128_f32", nx=128, ny=128, nz=128, steps=49, tau=0.7, kind="gradient"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["run", "monitor", "restart", "gradient"], [6, 1, 1, 1])[0]
    precision = rng.choices(["f32", "f16s", "bf16s", "f64"], [5, 4, 2, 1])[0]
    collision = rng.choice(["srt", "trt", "mrt"])
    stencil = 19
    pattern = rng.choice(["ab", "aa"])
    if kind == "run" and rng.random() < 0.15:
        stencil, pattern = 27, "ab"
    if kind == "gradient":
        pattern = "ab"
        precision = rng.choice(["f32", "f32", "f64"])
    if (stencil == 27 or kind == "gradient") and collision == "mrt":
        collision = "trt"
    # cells of the lattice, then its edges: from thin ducts to cubes, any remainder
    most = {"gradient": 128 ** 3, "monitor": 192 ** 3}.get(kind, 512 * 256 * 256)
    if precision == "f64":
        most = min(most, 96 ** 3)
    while True:
        nx, ny, nz = _log_int(rng, 4, 768), _log_int(rng, 4, 512), _log_int(rng, 4, 512)
        if 16 ** 3 <= nx * ny * nz <= most:
            break
    if rng.random() < 0.4:
        nx = max(4, nx // 4 * 4)
    steps = rng.randint(10, 25) if kind == "monitor" else rng.randint(10, 100)
    if kind == "gradient" and nx * ny * nz > 64 ** 3:
        steps = min(steps, 49)
    if nx * ny * nz > 256 ** 3:
        steps = min(steps, 50)
    walls = rng.choice(["", "", "y", "yz", "xyz"])
    return _case(nx=nx, ny=ny, nz=nz, steps=steps, samples=rng.randint(2, 4) if kind == "monitor" else 1, kind=kind,
                 precision=precision, pattern=pattern, collision=collision, stencil=stencil,
                 equilibrium="standard" if stencil == 27 else rng.choice(["improved", "improved", "standard"]),
                 tau=rng.choice([0.55, 0.6, 0.7, 0.8, 1.0]), walls=walls, force_x=rng.choice([0.0, 1e-6]))


# ---------------------------------------------------------------- inputs

_AMPLITUDE = 0.01
_MODES = 6


def _field_dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _velocity(case, seed, dtype):
    """Smooth divergence-free velocity: a mean flow and a few solenoidal plane waves of integer wave vectors
    |n_i| <= 3, drawn from the seed; components of about 0.02, as in the workloads of bench.py.  Along an
    axis of fewer than 16 cells the flow is uniform."""
    rng = np.random.default_rng(seed)
    n = (case["nx"], case["ny"], case["nz"])
    u = torch.empty((3, n[2], n[1], n[0]), dtype=dtype, device=DEVICE)
    mean = rng.uniform(-0.03, 0.03, 3)
    for i in range(3):
        u[i] = float(mean[i])
    axes = [torch.arange(m, dtype=torch.float64, device=DEVICE) * (2 * math.pi / m) for m in n]
    for _ in range(_MODES):
        k = rng.integers(-3, 4, 3) * np.array([m >= 16 for m in n])
        a = rng.standard_normal(3)
        phase = rng.uniform(0, 2 * math.pi)
        if k.any():
            a = a - k * (a @ k) / (k @ k)
        a = _AMPLITUDE * a / max(np.linalg.norm(a), 1e-3)
        # sin(kx X + ky Y + kz Z + phase), expanded so that no full-size phase array is needed
        yz = (float(k[2]) * axes[2]).view(-1, 1) + (float(k[1]) * axes[1]).view(1, -1) + phase
        s, c = torch.sin(yz).to(dtype).unsqueeze(-1), torch.cos(yz).to(dtype).unsqueeze(-1)
        cx, sx = torch.cos(float(k[0]) * axes[0]).to(dtype), torch.sin(float(k[0]) * axes[0]).to(dtype)
        for i in range(3):
            u[i].addcmul_(s, cx, value=float(a[i])).addcmul_(c, sx, value=float(a[i]))
    return u


_STORAGE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}


def _saved_populations(case, seed):
    """A saved state: equilibrium populations of a smooth flow with a non-equilibrium part of a few per cent
    of their size, in the storage type and the order that get_pdfs gives."""
    method = _Method(case)
    u = _velocity(case, seed, torch.float64)
    f = method.equilibrium(torch.zeros_like(u[0]), u)
    gen = torch.Generator(device=DEVICE).manual_seed(seed + 1)
    f += 1e-5 * torch.randn(f.shape, generator=gen, dtype=torch.float32, device=DEVICE)
    return f.to(_STORAGE[case["precision"]])


def _simulation(case):
    from paper_1803_04937_gb300.lbm import Simulation
    walls = tuple(a in case["walls"] for a in "xyz")
    return Simulation(case["nx"], case["ny"], case["nz"], equilibrium=case["equilibrium"],
                      collision=case["collision"], tau=case["tau"], precision=case["precision"],
                      force=(case["force_x"], 0.0, 0.0), walls=walls, pattern=case["pattern"],
                      stencil=case["stencil"], device=DEVICE)


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "gradient":
        state["u0"] = _velocity(case, seed, _field_dtype(case)).requires_grad_(True)
        state["tau"] = torch.tensor(case["tau"], dtype=torch.float64, requires_grad=True)
        state["target"] = _velocity(case, seed + 1000003, _field_dtype(case))
        return state
    state["sim"] = _simulation(case)
    if case["kind"] == "restart":
        state["pdfs"] = _saved_populations(case, seed)
    else:
        state["u"] = _velocity(case, seed, _field_dtype(case))
    return state


# ---------------------------------------------------------------- a pass

def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        from paper_1803_04937_gb300.adjoint import simulate
        u0, tau = state["u0"], state["tau"]
        walls = tuple(a in case["walls"] for a in "xyz")
        rho, u = simulate(u0, tau, case["steps"], case["nx"], case["ny"], case["nz"],
                          equilibrium=case["equilibrium"], collision=case["collision"], precision=case["precision"],
                          force=(case["force_x"], 0.0, 0.0), walls=walls)
        loss = 0.5 * ((u - state["target"]) ** 2).sum()
        grad_u0, grad_tau = torch.autograd.grad(loss, (u0, tau))
        return {"rho": rho.detach(), "u": u.detach(), "grad_u0": grad_u0, "grad_tau": grad_tau}
    sim = state["sim"]
    if case["kind"] == "restart":
        sim.set_pdfs(state["pdfs"])
        sim.step(case["steps"])
        return {"pdfs": sim.get_pdfs()}
    sim.init(None, state["u"])
    out = {}
    if case["kind"] == "monitor":
        for i in range(case["samples"]):
            sim.step(case["steps"])
            r = sim.reduce()
            out["sample_%d" % i] = {"mass": r["mass"], "energy": r["energy"], "momentum": list(r["momentum"]),
                                    "umax": r["umax"], "nonfinite": r["nonfinite"], "enstrophy": sim.enstrophy()}
    else:
        sim.step(case["steps"])
    out["rho"], out["u"] = sim.moments(_field_dtype(case))
    return out


def work(case):
    """Bytes: the fields (or populations) that go in and those that come out, once; the state between the
    steps of a pass need not leave the chip.  Operations: those of the collisions (a pair of populations takes
    about twenty), for a gradient also those of the recomputed steps and of their adjoint."""
    cells = case["nx"] * case["ny"] * case["nz"]
    field = 8 if case["precision"] == "f64" else 4
    steps = case["steps"] * case["samples"]
    per_cell = 200 if case["stencil"] == 19 else 300
    if case["collision"] == "mrt":
        per_cell += 40
    if case["kind"] == "gradient":
        # u0 and the target in; rho, u and dL/du0 out; forward, recomputed forward, adjoint
        return {"bytes": cells * field * (3 + 3 + 4 + 3), "flops": cells * steps * (2 * per_cell + 400)}
    if case["kind"] == "restart":
        size = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}[case["precision"]]
        return {"bytes": 2 * cells * size * case["stencil"], "flops": cells * steps * per_cell}
    extra = case["samples"] * 60 if case["kind"] == "monitor" else 0
    return {"bytes": cells * field * (3 + 4), "flops": cells * (steps * per_cell + extra)}


# ---------------------------------------------------------------- 64-bit reference

def _velocities(stencil):
    """Rest, faces, edges (and corners), every velocity followed by its opposite: the order of get_pdfs."""
    pairs = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
    if stencil == 27:
        pairs += [(1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]
    c = [(0, 0, 0)]
    for p in pairs:
        c += [p, tuple(-x for x in p)]
    return c


class _Method:
    """The method in FP64 on shifted populations f_q - w_q, as [Q, nz, ny, nx]."""

    def __init__(self, case):
        self.case = case
        self.c = _velocities(case["stencil"])
        weight = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[case["stencil"]]
        self.w = [weight[sum(x * x for x in c)] for c in self.c]
        self.opp = [self.c.index(tuple(-x for x in c)) for c in self.c]
        self.improved = case["equilibrium"] == "improved" and case["stencil"] == 19
        self.accel = (case["force_x"], 0.0, 0.0)

    def moments(self, f):
        drho = f.sum(0)
        u = []
        for i in range(3):
            j = sum(f[q] for q, c in enumerate(self.c) if c[i] > 0) - \
                sum(f[q] for q, c in enumerate(self.c) if c[i] < 0)
            u.append(j + 0.5 * self.accel[i])
        return drho, torch.stack(u)

    def equilibrium(self, drho, u):
        """Eq. 14, or Eq. 22 written as Eq. 14 plus its fourth-order-moment terms."""
        sq = u * u
        uu = sq.sum(0)
        out = []
        for c, w in zip(self.c, self.w):
            cu = sum(c[i] * u[i] for i in range(3) if c[i])
            e = w * (drho - 1.5 * uu)
            if any(c):
                e = e + w * (3.0 * cu + 4.5 * cu * cu)
            if self.improved:
                order = sum(x * x for x in c)
                if order == 0:
                    e = e + uu / 6.0
                elif order == 1:
                    e = e - (uu - sq[[abs(x) for x in c].index(1)]) / 12.0
                else:
                    e = e + sq[c.index(0)] / 24.0
            out.append(e)
        return torch.stack(out)

    def rates(self, tau):
        """(omega+, omega-) of SRT or of the odd/even split with magic parameter 3/16."""
        plus = 1.0 / tau
        return plus, plus if self.case["collision"] == "srt" else 1.0 / (0.5 + (3.0 / 16.0) / (tau - 0.5))

    def moment_operator(self, tau):
        """MRT: M^-1 S M over the monomials with exponents 0, 1, 2 that D3Q19 resolves; trace and fourth-order
        moments at rate 1, odd moments at omega-, the deviator at omega+."""
        plus, minus = self.rates(tau)
        c = np.array(self.c, dtype=float)
        rows, rate = [], []
        sq = c * c
        rows += [sq.sum(1), sq[:, 0] - sq[:, 1], sq[:, 0] + sq[:, 1] - 2 * sq[:, 2]]
        rate += [1.0, plus, plus]
        for e in itertools.product(range(3), repeat=3):
            row = np.prod([c[:, i] ** e[i] for i in range(3)], axis=0)
            if sum(e) == 2 and max(e) == 2 or not row.any():
                continue
            rows.append(row)
            rate.append(0.0 if sum(e) == 0 else minus if sum(e) % 2 else plus if sum(e) == 2 else 1.0)
        # exponents that vanish on the lattice's velocities drop out; the rest must span the 19 populations
        m = np.array(rows)
        keep = []
        for i in range(len(m)):
            if np.linalg.matrix_rank(m[keep + [i]]) == len(keep) + 1:
                keep.append(i)
        m, s = m[keep], np.array(rate)[keep]
        assert m.shape == (19, 19)
        return np.linalg.solve(m, s[:, None] * m)

    def step(self, f, tau):
        plus, minus = self.rates(tau)
        drho, u = self.moments(f)
        neq = f - self.equilibrium(drho, u)
        if self.case["collision"] == "mrt":
            k = torch.as_tensor(self.moment_operator(tau), dtype=torch.float64, device=f.device)
            post = f - torch.matmul(k, neq.flatten(1)).view_as(f)
        elif self.case["collision"] == "srt":
            post = f - plus * neq
        else:
            other = neq[self.opp]
            post = f - (0.5 * plus) * (neq + other) - (0.5 * minus) * (neq - other)
        del neq
        out = []
        for q, c in enumerate(self.c):
            p = post[q]
            ca = sum(c[i] * self.accel[i] for i in range(3))
            out.append(p + (1.0 - 0.5 * minus) * 3.0 * self.w[q] * ca if ca else p)
        return self._stream(out)

    def _stream(self, post):
        """Periodic shift, with half-way bounce-back on the walled axes."""
        n = (self.case["nx"], self.case["ny"], self.case["nz"])
        out = []
        for q, c in enumerate(self.c):
            moved = torch.roll(post[q], (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else post[q]
            blocked = None
            for i, axis in enumerate("xyz"):
                if axis in self.case["walls"] and c[i]:
                    shape = [1, 1, 1]
                    shape[2 - i] = n[i]
                    edge = torch.zeros(n[i], dtype=torch.bool, device=moved.device)
                    edge[0 if c[i] > 0 else n[i] - 1] = True
                    blocked = edge.view(shape) if blocked is None else blocked | edge.view(shape)
            out.append(moved if blocked is None else torch.where(blocked, post[self.opp[q]], moved))
        return torch.stack(out)

    def enstrophy(self, u):
        def diff(i, axis):
            dim = 2 - axis
            up, down = torch.roll(u[i], -1, dim), torch.roll(u[i], 1, dim)
            if "xyz"[axis] in self.case["walls"]:
                m = u.shape[1 + dim]
                up.select(dim, m - 1).copy_(-u[i].select(dim, m - 1))
                down.select(dim, 0).copy_(-u[i].select(dim, 0))
            return 0.5 * (up - down)
        w = (diff(2, 1) - diff(1, 2)) ** 2
        w += (diff(0, 2) - diff(2, 0)) ** 2
        w += (diff(1, 0) - diff(0, 1)) ** 2
        return 0.5 * float(w.mean())


def exact(case, seed):
    cells = case["nx"] * case["ny"] * case["nz"]
    if cells * case["steps"] * case["samples"] > 2.0e9:
        return None
    method = _Method(case)
    if case["kind"] == "gradient":
        return _exact_gradient(case, method, seed)
    with torch.no_grad():
        if case["kind"] == "restart":
            f = _saved_populations(case, seed).double()
            for _ in range(case["steps"]):
                f = method.step(f, case["tau"])
            return {"pdfs": f}
        u = _velocity(case, seed, _field_dtype(case)).double()
        f = method.equilibrium(torch.zeros_like(u[0]), u)
        out = {}
        for i in range(case["samples"]):
            for _ in range(case["steps"]):
                f = method.step(f, case["tau"])
            if case["kind"] == "monitor":
                drho, u = method.moments(f)
                uu = (u * u).sum(0)
                out["sample_%d" % i] = {
                    "mass": float(cells + drho.sum()), "energy": 0.5 * float(uu.sum()),
                    "momentum": [float(u[k].sum()) - 0.5 * method.accel[k] * cells for k in range(3)],
                    "umax": float(uu.max().sqrt()), "nonfinite": 0, "enstrophy": method.enstrophy(u)}
        drho, u = method.moments(f)
        out["rho"], out["u"] = 1.0 + drho, u
        return out


def _exact_gradient(case, method, seed):
    u0 = _velocity(case, seed, _field_dtype(case)).double().requires_grad_(True)
    target = _velocity(case, seed + 1000003, _field_dtype(case)).double()
    tau = torch.tensor(case["tau"], dtype=torch.float64, device=DEVICE, requires_grad=True)
    f = method.equilibrium(torch.zeros_like(u0[0]), u0)
    for _ in range(case["steps"]):
        f = checkpoint(method.step, f, tau, use_reentrant=False)
    drho, u = method.moments(f)
    loss = 0.5 * ((u - target) ** 2).sum()
    grad_u0, grad_tau = torch.autograd.grad(loss, (u0, tau))
    return {"rho": (1.0 + drho).detach(), "u": u.detach(), "grad_u0": grad_u0, "grad_tau": grad_tau.cpu()}
