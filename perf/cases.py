"""Performance cases: the work a user of this library has it do, through its
public entry points, on one GPU.

Kinds of case (the ``kind`` value):
  solve     Context.solve: one cold multigrid solve of a random right-hand side
  run       Context.run: quasi-static projection steps from a developed state
  explicit  Context.explicit_step: forward-Euler steps of the comparison scheme
  grad      plastic_work(...).backward(): plastic work and its gradient
  transfer  mg_residual_restrict_static: residual and restriction, no allocation

``exact`` restates each of them in plain FP64 torch.  The projection system is
solved directly there: the operator is periodic with constant coefficients in
x and y, so a Fourier transform leaves one block-tridiagonal system in z (3 x 3
blocks) per wave number, which block elimination solves.
"""
import ctypes
import math

import torch

from paper_1904_03808_gb300 import MG_FP64, MG_MIXED, Context, binding, make_state, plastic_work
from paper_1904_03808_gb300 import inputs as I

DEV = "cuda"
F64 = torch.float64
MAT = I.TABLE1
K, MU, RHO = MAT["K"], MAT["mu"], MAT["rho"]
LAM = K - 2.0 * MU / 3.0
KB = 1.380649e-23
L = 0.01                                # half width of the sample (m)
TS = L / math.sqrt(MU / RHO)            # shear time unit (s)


def listed():
    return [
        # one step of the smallest grid that still has two levels to descend:
        # an interactive or unit-sized run, all latency
        dict(name="step 16^3 mixed", kind="run", nx=16, ny=16, nz=16, precision="mixed", walls=0,
             steps=1, advect=False, tol=1e-10),
        # the cold verification solve of a small grid in plain FP64
        dict(name="solve 32^3 fp64", kind="solve", nx=32, ny=32, nz=32, precision="fp64",
             tol=1e-10),
        # the same kind of solve at an ordinary size in the default mixed precision
        dict(name="solve 64^3 mixed", kind="solve", nx=64, ny=64, nz=64, precision="mixed",
             tol=1e-10),
        # a host program's own residual and restriction without allocations
        dict(name="transfer 64^3", kind="transfer", nx=64, ny=64, nz=64),
        # the comparison geometry of the explicit scheme
        dict(name="explicit 64x64x32", kind="explicit", nx=64, ny=64, nz=32, steps=10),
        # the differentiation workload, a few steps with one recomputed segment
        dict(name="grad 64^3 fp64", kind="grad", nx=64, ny=64, nz=64, precision="fp64", steps=3,
             every=2, tol=1e-12),
        # a grid whose rows and coarse levels are no powers of two
        dict(name="run 160x80x80 mixed", kind="run", nx=160, ny=80, nz=80, precision="mixed",
             walls=0, steps=2, advect=False, tol=1e-10),
        # a step of the general constitutive law with stress advection
        dict(name="advect 96^3 mixed", kind="run", nx=96, ny=96, nz=96, precision="mixed", walls=0,
             steps=1, advect=True, tol=1e-10),
        # the verification run in plain FP64
        dict(name="run 128^3 fp64", kind="run", nx=128, ny=128, nz=128, precision="fp64", walls=0,
             steps=1, advect=False, tol=1e-10),
        # the benchmark's workload: consecutive simple-shear steps
        dict(name="run 256^3 mixed", kind="run", nx=256, ny=256, nz=256, precision="mixed",
             walls=0, steps=2, advect=False, tol=1e-10),
        # friction welding: disc walls on a wide, flat grid, the largest state
        dict(name="disc 512x512x256 mixed", kind="run", nx=512, ny=512, nz=256, precision="mixed",
             walls=1, steps=1, advect=False, tol=1e-10),
    ]


def _grid(rng, lo, hi):
    """A grid of lo .. hi cells that halves down to a small coarsest level."""
    while True:
        a, b, c = rng.choice([4, 5, 6, 7, 8, 10, 12, 16]), rng.choice([4, 5, 6, 7, 8]), \
            rng.choice([4, 5, 6, 7])
        if a * b * (c - 1) > 200:       # the dense coarsest solve stays small
            continue
        m = 1 << rng.randint(1, 6)
        nx, ny, nz = a * m, b * m, c * m
        if nx <= 512 and lo <= nx * ny * nz <= hi:
            return dict(nx=nx, ny=ny, nz=nz)


def draw(rng):
    def size(most):
        # the number of cells is drawn over its logarithm, then a grid near it
        n = math.exp(rng.uniform(math.log(1000), math.log(most / 1.5)))
        return _grid(rng, n / 1.5, 1.5 * n)

    kind = rng.choice(["solve", "run", "run", "run", "explicit", "grad", "transfer"])
    if kind == "solve":
        p = rng.choice(["fp64", "mixed"])
        return dict(kind=kind, precision=p, tol=1e-10,
                    **size(2e6 if p == "fp64" else 1.6e7))
    if kind == "run":
        p = rng.choice(["fp64", "mixed", "mixed"])
        advect = rng.random() < 0.2
        g = size(2e6 if p == "fp64" else 1.6e7)
        big = g["nx"] * g["ny"] * g["nz"] > 4e6
        return dict(kind=kind, precision=p, walls=rng.choice([0, 0, 1, 2, 3]),
                    steps=1 if advect or big else rng.randint(1, 3), advect=advect, tol=1e-10, **g)
    if kind == "explicit":
        return dict(kind=kind, steps=rng.randint(2, 10), **size(1e6))
    if kind == "grad":
        return dict(kind=kind, precision="fp64", steps=rng.randint(2, 3), every=rng.randint(1, 3),
                    tol=1e-12, **size(2.7e5))
    while True:                         # transfer: any even sizes that fit its array
        nx, ny, nz = (2 * int(math.exp(rng.uniform(math.log(2), math.log(64)))) for _ in range(3))
        if 3 * (nz + 1) * ny * nx <= 2097152:
            return dict(kind=kind, nx=nx, ny=ny, nz=nz)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _smooth(gen, shape, lc):
    """Random fields of unit variance with correlation exp(-r^2 / (2 lc^2))."""
    out = torch.empty(shape, dtype=F64, device=DEV)
    h = [torch.exp(-(2.0 * math.pi * torch.fft.fftfreq(n, dtype=F64, device=DEV) * lc) ** 2 / 4.0)
         for n in shape[1:]]
    norm = math.prod(math.sqrt(float((t * t).mean())) for t in h)
    for c in range(shape[0]):
        w = torch.randn(shape[1:], generator=gen, dtype=F64, device=DEV)
        f = torch.fft.rfftn(w)
        f *= h[0][:, None, None]
        f *= h[1][:, None]
        f *= h[2][:shape[3] // 2 + 1]
        out[c] = torch.fft.irfftn(f, s=tuple(shape[1:]))
    return out / norm


class Problem:
    """The numbers and arrays of one case: geometry, material, walls, state."""

    def __init__(self, case, seed):
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        self.case = case
        self.nx, self.ny, self.nz = nx, ny, nz = case["nx"], case["ny"], case["nz"]
        self.h = 2.0 * L / nx
        H = nz * self.h
        kind = case["kind"]
        if kind in ("solve", "transfer"):
            def rnd():
                return 2.0 * torch.rand((3, nz + 1, ny, nx), generator=gen, dtype=F64,
                                        device=DEV) - 1.0
            self.b = rnd()
            if kind == "transfer":
                self.x = rnd()
                return
            self.b[:, 0] = 0.0
            self.b[:, nz] = 0.0
            self.v = torch.zeros_like(self.b)
            self.v[0, 0], self.v[0, nz] = -1.0, 1.0
            return
        walls = case.get("walls", 0)
        self.zeta = 1e4 if kind == "explicit" else 1.0
        self.stz = dict(tau0=MAT["tau0"] / self.zeta, eps0=MAT["eps0"], c0=MAT["c0"],
                        Delta_K=MAT["Delta_K"], Omega=MAT["Omega"], T=MAT["T"],
                        chi_inf=MAT["chi_inf"], ez_K=MAT["ez_K"], sY=MAT["sY"], l=self.h, kB=KB)
        self.dt = (2e3 if walls else 200.0) * TS
        U = 0.02 * H / (2.0 * 50 * 200.0 * TS)   # 2% shear strain over 50 steps
        if kind == "explicit":
            self.dt = TS * self.h ** 2 / (20.0 * L * L)
            self.kappa = 4.8 * L / TS * self.h
            U = 1e-7 * self.zeta * L / TS
        R = 1.0 / 3.0
        omega = 2.0 * math.pi / (1e8 * TS)
        self.bc = dict(kind=walls, U_B=U, t_ramp=TS, omega=omega if walls else 0.0, R=R,
                       lambda_w=16.0 * math.log(10.0) / (1.0 - R * R) ** 2)
        self.t0 = TS
        # a state in mid-run: the chi field of the paper's random inclusions, a
        # shear stress about the yield stress (above it for simple shear) with
        # smooth variations, the linear shear profile with smooth deviations
        lc = min(4.0, nx / 8.0, ny / 8.0, nz / 8.0)
        self.chi = 600.0 + 30.0 * _smooth(gen, (1, nz, ny, nx), lc)[0]
        self.sigma = 2e7 * _smooth(gen, (6, nz, ny, nx), lc)
        self.sigma[4] += 0.8e9 if walls else 1.2e9
        V = omega * L if walls else U
        v = 0.02 * V * _smooth(gen, (3, nz + 1, ny, nx), lc)
        if not walls:
            zk = (torch.arange(nz + 1, dtype=F64, device=DEV) - nz / 2.0) * self.h
            v[0] += (2.0 * U / H * zk)[:, None, None]
        self.v = _walls(self, v, self.t0)

    def context(self):
        c = self.case
        if c["kind"] == "solve":
            return Context(self.nx, self.ny, self.nz, self.h, K, MU, precision=_prec(c))
        flags = binding.MG_FLAG_ADVECT_STRESS if c.get("advect") else 0
        return Context(self.nx, self.ny, self.nz, self.h, K, MU, bc=self.bc, stz=self.stz,
                       precision=_prec(c), flags=flags)


def _prec(case):
    return MG_MIXED if case.get("precision") == "mixed" else MG_FP64


def prepare(case, seed):
    p = Problem(case, seed)
    s = dict(case=case, p=p)
    if case["kind"] == "transfer":
        s["bc"] = torch.empty((3, p.nz // 2 + 1, p.ny // 2, p.nx // 2), dtype=F64, device=DEV)
        s["grid"] = binding.mg_grid(p.nx, p.ny, p.nz, p.h)
        s["moduli"] = binding.mg_moduli(K, MU)
        return s
    s["ctx"] = p.context()
    if case["kind"] == "solve":
        s["v"] = torch.empty_like(p.v)
    elif case["kind"] == "grad":
        s["chi"] = p.chi.clone().requires_grad_()
    else:
        s["work"] = [torch.empty_like(a) for a in (p.v, p.sigma, p.chi)]
    return s


def run(s):
    case, p = s["case"], s["p"]
    kind = case["kind"]
    if kind == "solve":
        s["v"].copy_(p.v)
        s["ctx"].solve(p.b, s["v"], tol=case["tol"])
        return s["v"]
    if kind == "transfer":
        stream = torch.cuda.current_stream()
        st = binding.lib().mg_residual_restrict_static(
            ctypes.byref(s["grid"]), ctypes.byref(s["moduli"]), ctypes.c_void_p(p.b.data_ptr()),
            ctypes.c_void_p(p.x.data_ptr()), ctypes.c_void_p(s["bc"].data_ptr()),
            ctypes.c_void_p(stream.cuda_stream))
        if st != binding.MG_OK:
            raise binding.QSMGError(st, "mg_residual_restrict_static")
        return s["bc"]
    if kind == "grad":
        s["chi"].grad = None
        W = plastic_work(s["ctx"], p.v, p.sigma, s["chi"], p.t0, case["steps"], p.dt,
                         tol=case["tol"], checkpoint_every=case["every"])
        W.backward()
        return W.detach(), s["chi"].grad
    # every pass starts from the same stored state, as the members of a
    # parameter study do
    for w, a in zip(s["work"], (p.v, p.sigma, p.chi)):
        w.copy_(a)
    state = make_state(*s["work"], p.t0)
    if kind == "explicit":
        s["ctx"].explicit_step(state, p.dt, RHO, p.kappa, nsteps=case["steps"])
    else:
        s["ctx"].run(state, case["steps"], p.dt, tol=case["tol"])
    return tuple(s["work"])


def work(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nc, nv = nx * ny * nz, nx * ny * (nz + 1)
    node = 90.0                         # operations of the 19-point operator at a node
    # a V-cycle: four sweeps and a residual a level, 27-point blocks (about
    # 310 operations a node) on the coarse ones; some 0.36 contraction a cycle
    cycle = nc * 5.0 * (node + 310.0 / 7.0)

    def solve(tol, start):
        return max(1.0, math.log(tol / start) / math.log(0.36)) * cycle

    state = 8.0 * (3 * nv + 7 * nc)
    kind = case["kind"]
    if kind == "transfer":
        return dict(bytes=8.0 * (6 * nv + 3 * nv / 8), flops=(node + 10.0) * nv)
    if kind == "solve":
        return dict(bytes=8.0 * 9 * nv, flops=solve(case["tol"], 1.0))
    if kind == "explicit":
        return dict(bytes=2 * state, flops=case["steps"] * 900.0 * nc)
    if kind == "grad":
        n = case["steps"]
        return dict(bytes=state + 8.0 * nc,
                    flops=n * (2 * solve(case["tol"], 1.0) + 1100.0 * nc))
    point = 450.0 + (250.0 if case["advect"] else 0.0)
    return dict(bytes=2 * state, flops=case["steps"] * (solve(case["tol"], 1e-2) + point * nc))


# ---------------------------------------------------------------------------
# the same results in plain FP64 torch
# ---------------------------------------------------------------------------

def _walls(p, v, t):
    """v with the wall velocities of time t on the planes k = 0 and nz."""
    nx, ny, nz, bc = p.nx, p.ny, p.nz, p.bc
    v = v.clone()
    v[:, 0], v[:, nz] = 0.0, 0.0
    if bc["kind"] == 0:
        U = bc["U_B"] * min(t / bc["t_ramp"], 1.0)
        v[0, 0], v[0, nz] = -U, U
        return v
    W = 0.5 * nx * p.h
    x = -W + torch.arange(nx, dtype=F64, device=DEV) * p.h
    y = (-0.5 * ny * p.h + torch.arange(ny, dtype=F64, device=DEV) * p.h)[:, None]
    r2 = (x * x + y * y) / (W * W)
    R2 = bc["R"] ** 2
    f = torch.where(r2 < R2, torch.ones_like(r2), torch.exp(-bc["lambda_w"] * (r2 - R2) ** 2))
    v[0, nz], v[1, nz] = -bc["omega"] * y * f, bc["omega"] * x * f
    sign = {1: 0.0, 2: 1.0, 3: -1.0}[bc["kind"]]
    v[:2, 0] = sign * v[:2, nz]
    return v


def _gradient(p, v):
    """G[a][b] = d v_a / d x_b at cell centres."""
    f = 0.25 / p.h
    c = [[[v[:, dz:dz + p.nz].roll((-dy, -dx), (2, 3)) for dx in (0, 1)] for dy in (0, 1)]
         for dz in (0, 1)]
    gx = sum(c[z][y][1] - c[z][y][0] for z in (0, 1) for y in (0, 1)) * f
    gy = sum(c[z][1][x] - c[z][0][x] for z in (0, 1) for x in (0, 1)) * f
    gz = sum(c[1][y][x] - c[0][y][x] for y in (0, 1) for x in (0, 1)) * f
    return [[gx[a], gy[a], gz[a]] for a in range(3)]


_COMP = ((0, 5, 4), (5, 1, 3), (4, 3, 2))       # stored component of (a, b)
_PAIR = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))


def _divergence(p, s):
    """Divergence of a cell stress at the interior corners."""
    f = 0.25 / p.h
    c = [[[s[:, dz:dz + p.nz - 1].roll((1 - dy, 1 - dx), (2, 3)) for dx in (0, 1)]
          for dy in (0, 1)] for dz in (0, 1)]

    def comp(a):
        m0, m1, m2 = _COMP[a]
        return (sum(c[z][y][1][m0] - c[z][y][0][m0] for z in (0, 1) for y in (0, 1)) +
                sum(c[z][1][x][m1] - c[z][0][x][m1] for z in (0, 1) for x in (0, 1)) +
                sum(c[1][y][x][m2] - c[0][y][x][m2] for y in (0, 1) for x in (0, 1))) * f
    return torch.stack([comp(a) for a in range(3)])


def _sbar(s):
    m = (s[0] + s[1] + s[2]) / 3.0
    return torch.sqrt(0.5 * ((s[0] - m) ** 2 + (s[1] - m) ** 2 + (s[2] - m) ** 2) +
                      s[3] ** 2 + s[4] ** 2 + s[5] ** 2)


def _rate(p, sbar, chi):
    z = p.stz
    on = (sbar > z["sY"]) & (chi > 0)
    sb, ch = torch.where(on, sbar, z["sY"]), torch.where(on, chi, 1.0)
    x, y = z["Omega"] * z["eps0"] / (z["kB"] * z["T"]) * sb, -z["ez_K"] / ch
    D = 0.5 * math.exp(-z["Delta_K"] / z["T"]) / z["tau0"] * \
        (torch.exp(x + y) + torch.exp(y - x)) * (1.0 - z["sY"] / sb)
    return torch.where(on, D, torch.zeros_like(D))


def _objective_rate(p, G, s, D, sbar):
    """L s + s L^T - tr(L) s - 2 mu D s0 / sbar, per stored component."""
    tr = G[0][0] + G[1][1] + G[2][2]
    m = (s[0] + s[1] + s[2]) / 3.0
    pl = torch.where(D > 0, 2.0 * MU * D / torch.where(D > 0, sbar, 1.0), torch.zeros_like(D))
    out = []
    for a, b in _PAIR:
        S = s[_COMP[a][b]]
        r = -tr * S - pl * (S - m if a == b else S)
        for e in range(3):
            r = r + G[a][e] * s[_COMP[e][b]] + s[_COMP[a][e]] * G[b][e]
        out.append(r)
    return out


def _elastic(G, a, b):
    tr = G[0][0] + G[1][1] + G[2][2]
    return (LAM * tr if a == b else 0.0) + MU * (G[a][b] + G[b][a])


def _chi_update(p, s, chi, D, sbar):
    z = p.stz
    # z ghost layers: stress and chi continued linearly, D their STZ rate
    def ghost(a, b):
        sg, cg = 2.0 * s[:, a] - s[:, b], 2.0 * chi[a] - chi[b]
        return cg[None], _rate(p, _sbar(sg), cg)[None]
    (cl, Dl), (ch, Dh) = ghost(0, 1), ghost(-1, -2)
    ce, De = torch.cat([cl, chi, ch]), torch.cat([Dl, D, Dh])
    acc = sum(0.5 * (D + De[1 + d:1 + d + p.nz]) * (ce[1 + d:1 + d + p.nz] - chi) for d in (-1, 1))
    for ax in (1, 2):
        for d in (-1, 1):
            acc = acc + 0.5 * (D + D.roll(d, ax)) * (chi.roll(d, ax) - chi)
    growth = 2.0 * D * sbar / z["sY"] * (z["chi_inf"] - chi)
    return chi + p.dt / z["c0"] * (growth + (z["l"] / p.h) ** 2 * acc)


def _direct_solve(b, v):
    """Solution of the scaled projection system for interior right-hand side b
    (3, nz-1, ny, nx), the walls of v kept."""
    nz1, ny, nx = b.shape[1:]
    lp, kq = (LAM + 2.0 * MU) / MU, (LAM + MU) / (4.0 * MU)
    ty = 2.0 * math.pi * torch.fft.fftfreq(ny, dtype=F64, device=DEV)[:, None]
    tx = 2.0 * math.pi * torch.fft.rfftfreq(nx, dtype=F64, device=DEV)[None, :]
    sx, sy = torch.sin(tx) + 0.0 * ty, torch.sin(ty) + 0.0 * tx
    cx, cy = 2.0 * torch.cos(tx) + 0.0 * ty, 2.0 * torch.cos(ty) + 0.0 * tx
    B = torch.zeros(ny, nx // 2 + 1, 3, 3, dtype=torch.complex128, device=DEV)
    up = torch.zeros_like(B)            # the coupling to plane k + 1
    for a in range(3):
        B[..., a, a] = 2.0 * lp + 4.0 - (lp if a == 0 else 1.0) * cx - (lp if a == 1 else 1.0) * cy
        up[..., a, a] = -lp if a == 2 else -1.0
    B[..., 0, 1] = B[..., 1, 0] = 4.0 * kq * sx * sy
    up[..., 0, 2] = up[..., 2, 0] = -2j * kq * sx
    up[..., 1, 2] = up[..., 2, 1] = -2j * kq * sy
    lo = up.mH
    r = torch.fft.rfft2(b).permute(1, 2, 3, 0).contiguous()[..., None]
    w = torch.fft.rfft2(v[:, [0, -1]]).permute(1, 2, 3, 0)[..., None]
    r[0] -= lo @ w[0]
    r[-1] -= up @ w[1]
    inv = []
    for k in range(nz1):                # block elimination, then back substitution
        M = B if k == 0 else B - lo @ (inv[-1] @ up)
        if k:
            r[k] -= lo @ (inv[-1] @ r[k - 1])
        inv.append(torch.linalg.inv(M))
    for k in range(nz1 - 1, -1, -1):
        r[k] = inv[k] @ (r[k] - up @ r[k + 1] if k + 1 < nz1 else r[k])
    x = torch.fft.irfft2(r[..., 0].permute(3, 0, 1, 2), s=(ny, nx))
    return torch.cat([v[:, :1], x, v[:, -1:]], dim=1)


class _Solve(torch.autograd.Function):
    """The solve as a differentiable function of b: its matrix is symmetric."""

    @staticmethod
    def forward(ctx, b, v):
        return _direct_solve(b, v)

    @staticmethod
    def backward(ctx, g):
        zero = torch.zeros_like(g)
        return _direct_solve(g[:, 1:-1], zero)[:, 1:-1], None


def _exact_step(p, v, s, chi, t, advect):
    G = _gradient(p, v)
    sbar = _sbar(s)
    D = _rate(p, sbar, chi)
    rate = _objective_rate(p, G, s, D, sbar)
    if advect:
        adv = _stress_advection(p, v, s)
        rate = [r - a for r, a in zip(rate, adv)]
    star = torch.stack([s[n] + p.dt * rate[n] for n in range(6)])
    chi1 = _chi_update(p, s, chi, D, sbar)
    b = p.h ** 2 / (MU * p.dt) * _divergence(p, star)
    v1 = _Solve.apply(b, _walls(p, v.detach(), t + p.dt))
    G1 = _gradient(p, v1)
    s1 = torch.stack([star[_COMP[a][b_]] + p.dt * _elastic(G1, a, b_) for a, b_ in _PAIR])
    return v1, s1, chi1, (D * sbar).sum()


def _eno(f, u, axis, h, ghost):
    """Second-order ENO derivative along `axis` of f (n fields, nz, ny, nx);
    `ghost` continues f by two layers on each side in z."""
    if axis == 1:
        e = ghost(f)
        n = f.shape[1]
        m2, m1, p1, p2 = (e[:, 2 + d:2 + d + n] for d in (-2, -1, 1, 2))
    else:
        m2, m1, p1, p2 = (f.roll(-d, axis) for d in (-2, -1, 1, 2))
    cm, c0, cp = (f - 2 * m1 + m2).abs(), (p1 - 2 * f + m1).abs(), (p2 - 2 * p1 + f).abs()
    d = p1 - m1
    d = torch.where((u > 0) & (c0 > cm), 3 * f - 4 * m1 + m2, d)
    d = torch.where((u < 0) & (c0 > cp), -p2 + 4 * p1 - 3 * f, d)
    return d / (2.0 * h)


def _cell_ghost(f):
    a, b = f[:, 1:2] - f[:, :1], f[:, -1:] - f[:, -2:-1]
    return torch.cat([f[:, :1] - 2 * a, f[:, :1] - a, f, f[:, -1:] + b, f[:, -1:] + 2 * b], dim=1)


def _corner_ghost(f):
    lo, hi = 2 * f[:, :1], 2 * f[:, -1:]
    return torch.cat([lo - f[:, 2:3], lo - f[:, 1:2], f, hi - f[:, -2:-1], hi - f[:, -3:-2]], dim=1)


def _stress_advection(p, v, s):
    u = sum(v[:, z:z + p.nz].roll((-y, -x), (2, 3)) for z in (0, 1) for y in (0, 1)
            for x in (0, 1)) / 8.0
    out = 0.0
    for c, axis in ((0, 3), (1, 2), (2, 1)):
        out = out + u[c] * _eno(s, u[c][None], axis, p.h, _cell_ghost)
    return out


def _exact_explicit(p, v, s, chi, t):
    G = _gradient(p, v)
    sbar = _sbar(s)
    D = _rate(p, sbar, chi)
    rate = _objective_rate(p, G, s, D, sbar)
    adv = _stress_advection(p, v, s)
    s1 = torch.stack([s[n] + p.dt * (rate[n] - adv[n] + _elastic(G, *_PAIR[n])) for n in range(6)])
    chi1 = _chi_update(p, s, chi, D, sbar)
    acc = 0.0
    for c, axis in ((0, 3), (1, 2), (2, 1)):
        acc = acc - v[c] * _eno(v, v[c][None], axis, p.h, _corner_ghost)
    acc = acc[:, 1:-1]
    w = v[:, 1:-1]
    lap = v[:, 2:] - 2 * w + v[:, :-2]
    for axis in (2, 3):
        lap = lap + w.roll(1, axis) - 2 * w + w.roll(-1, axis)
    v1 = v.clone()
    v1[:, 1:-1] = w + p.dt * (acc + _divergence(p, s) / RHO + p.kappa / p.h ** 2 * lap)
    return _walls(p, v1, t + p.dt), s1, chi1


def _exact_transfer(p):
    lp, kq = (LAM + 2.0 * MU) / MU, (LAM + MU) / (4.0 * MU)
    x, nz = p.x, p.nz

    def at(c, dx, dy, dz):
        return x[c, 1 + dz:nz + dz].roll((-dy, -dx), (1, 2))

    unit = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
    r = torch.zeros_like(x)
    for a in range(3):
        o = (2.0 * lp + 4.0) * at(a, 0, 0, 0)
        for b in range(3):
            for s in (-1, 1):
                o = o - (lp if a == b else 1.0) * at(a, *(s * e for e in unit[b]))
                if a != b:
                    for q in (-1, 1):
                        o = o - kq * s * q * at(b, *(q * i + s * j
                                                     for i, j in zip(unit[a], unit[b])))
        r[a, 1:nz] = p.b[a, 1:nz] - o
    for axis in (3, 2):
        r = 0.5 * r.roll(1, axis) + r + 0.5 * r.roll(-1, axis)
    r = r[:, :, ::2, ::2]
    out = torch.zeros((3, nz // 2 + 1) + tuple(r.shape[2:]), dtype=F64, device=DEV)
    out[:, 1:-1] = 0.5 * r[:, 1:nz - 2:2] + r[:, 2:nz - 1:2] + 0.5 * r[:, 3:nz:2]
    return out


def exact(case, seed):
    p = Problem(case, seed)
    kind = case["kind"]
    if kind == "transfer":
        return _exact_transfer(p)
    if kind == "solve":
        return _direct_solve(p.b[:, 1:-1], p.v)
    if kind == "grad":
        chi0 = p.chi.clone().requires_grad_()
        state, t, W = (p.v, p.sigma, chi0), p.t0, 0.0
        for _ in range(case["steps"]):
            *state, w = _exact_step(p, *state, t, False)
            W = W + 2.0 * p.dt * p.h ** 3 * w
            t += p.dt
        W.backward()
        return W.detach(), chi0.grad
    state, t = (p.v, p.sigma, p.chi), p.t0
    for _ in range(case["steps"]):
        if kind == "explicit":
            state = _exact_explicit(p, *state, t)
        else:
            state = _exact_step(p, *state, t, case["advect"])[:3]
        t += p.dt
    return tuple(state)
