"""Workloads of the finite-volume solver, as a program that uses it runs them.

``listed()`` holds the workloads, ``draw()`` gives more of the same kinds.
A case is a dict:

* ``kind``: the problem (``vortex``, ``inlet``, ``mms``, ``batch``,
  ``periodic``, ``ogrid``) and ``op``: what a pass does with it - ``step``
  (``steps`` Runge-Kutta time steps of four stages, graph-replayed, then the
  state read back), ``residual`` (one residual evaluation) or ``adjoint``
  (``stages`` differentiable stages and their gradient);
* ``ni``, ``nj``, ``nk``: cells (for ``batch``: ``nblocks`` blocks of ``lo``
  to ``hi`` cells an axis); ``precision``: arithmetic form;
* options: ``autotune`` (launch autotuned once, when the program starts),
  ``monitor`` (residual norms recorded and read every pass), ``flux``,
  ``limiter``, ``kappa``, ``fix_all``, ``visc`` (laminar terms, no-slip walls).

``exact()`` evaluates the same scheme in plain 64-bit torch, written here from
the method (Section 2 and Eq. (flux) of arXiv 2012.02925) without any of the
package's code.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

GAMMA = 1.4
ALPHA = (0.25, 1.0 / 3.0, 0.5, 1.0)
INFLOW, OUTFLOW, SLIP, FARFIELD, NOSLIP = 1, 2, 3, 4, 5
AIR = {"mu": 1.716e-5, "prandtl": 0.72, "r_gas": 287.0, "t_ref": 273.15, "s_suth": 110.4}


def listed():
    return [
        # the smallest call: the 64^2 isentropic vortex, 100 stages (latency and launches)
        dict(name="vortex_64_fp64", kind="vortex", op="step", ni=64, nj=64, nk=1, precision="fp64", steps=25),
        # 2D supersonic inlet with walls, inflow and outflow at an ordinary grid
        dict(name="inlet_416x128_fp64", kind="inlet", op="step", ni=416, nj=128, nk=1, precision="fp64", steps=5),
        # transonic wing-like O-grid, odd sizes: curvilinear 3D with a periodic cut, walls and a farfield
        dict(name="ogrid_151x49x27_fp64", kind="ogrid", op="step", ni=151, nj=49, nk=27, precision="fp64", steps=2),
        # the headline block: 128^3 curvilinear with a source, in each arithmetic form;
        # the binary64 run autotunes its launch as a long production run does
        dict(name="mms_128_fp64", kind="mms", op="step", ni=128, nj=128, nk=128, precision="fp64", steps=1,
             autotune=True),
        # a run that follows its convergence: residual norms of every step
        dict(name="mms_128_df64_monitor", kind="mms", op="step", ni=128, nj=128, nk=128, precision="df64", steps=1,
             monitor=True),
        dict(name="mms_128_fp32flux", kind="mms", op="step", ni=128, nj=128, nk=128, precision="fp32flux", steps=4),
        # many uneven blocks with rotated connections in one launch
        dict(name="batch_64_fp64", kind="batch", op="step", nblocks=64, lo=16, hi=96, layout=2012,
             precision="fp64", steps=1),
        dict(name="batch_64_fp32flux", kind="batch", op="step", nblocks=64, lo=16, hi=96, layout=2012,
             precision="fp32flux", steps=2),
        # the largest: one 67-million-cell periodic block, throughput form
        dict(name="periodic_512x512x256_fp32flux", kind="periodic", op="step", ni=512, nj=512, nk=256,
             precision="fp32flux", steps=1),
        # laminar Navier-Stokes around the wing-like section, adiabatic no-slip walls
        dict(name="ogrid_ns_256x96x48_df64", kind="ogrid", op="step", ni=256, nj=96, nk=48, precision="df64",
             steps=1, visc=1),
        # gradient of a time step: differentiable stages forward and backward
        dict(name="adjoint_96", kind="mms", op="adjoint", ni=96, nj=96, nk=96, precision="fp64", stages=4,
             limiter=2, fix_all=1, sweeps="df64"),
        # one residual of another scheme (van Leer splitting, van Albada, kappa = 1/3), odd sizes
        dict(name="residual_97x61x53_fp64", kind="mms", op="residual", ni=97, nj=61, nk=53, precision="fp64",
             flux=1, limiter=2, kappa=1.0 / 3.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    form = rng.choice(["fp64", "fp64", "df64", "fp32flux"])
    kind = rng.choice(["vortex", "inlet", "ogrid", "ogrid_ns", "mms", "mms", "batch", "periodic", "adjoint",
                       "residual"])
    if kind == "vortex":
        n = size(24, 384)
        return dict(kind="vortex", op="step", ni=n, nj=n, nk=1, precision=form, steps=rng.randint(4, 25))
    if kind == "inlet":
        return dict(kind="inlet", op="step", ni=size(52, 1200), nj=size(16, 400), nk=1, precision=form,
                    steps=rng.randint(1, 5))
    if kind in ("ogrid", "ogrid_ns"):
        c = dict(kind="ogrid", op="step", ni=size(48, 300), nj=size(20, 100), nk=size(9, 50), precision=form,
                 steps=rng.randint(1, 2))
        if kind == "ogrid_ns":
            c["visc"] = 1
        return c
    if kind == "mms":
        c = dict(kind="mms", op="step", ni=size(17, 150), nj=size(17, 150), nk=size(17, 150), precision=form,
                 steps=rng.randint(1, 3))
        if rng.random() < 0.25:
            c["autotune"] = True
        if rng.random() < 0.25:
            c["monitor"] = True
        return c
    if kind == "batch":
        lo = rng.randint(8, 24)
        return dict(kind="batch", op="step", nblocks=size(4, 48), lo=lo, hi=lo + rng.randint(8, 56),
                    layout=rng.randint(1, 10 ** 6), precision=form, steps=1)
    if kind == "periodic":
        return dict(kind="periodic", op="step", ni=size(40, 256), nj=size(40, 256), nk=size(40, 256),
                    precision=form, steps=1)
    if kind == "adjoint":
        return dict(kind="mms", op="adjoint", ni=size(16, 80), nj=size(16, 80), nk=size(16, 80), precision="fp64",
                    stages=rng.randint(2, 4), limiter=2, fix_all=1, sweeps=rng.choice(["fp64", "df64"]))
    return dict(kind="mms", op="residual", ni=size(16, 140), nj=size(16, 140), nk=size(16, 140), precision="fp64",
                flux=rng.choice([0, 1, 2]), limiter=rng.choice([0, 1, 2]),
                kappa=rng.choice([-1.0, 0.0, 1.0 / 3.0]))


# ---------------------------------------------------------------------------
# the problems: blocks, connections, boundaries, state, source, time step
# ---------------------------------------------------------------------------

def _block(ni, nj, nk, nodes=None, h=(1.0, 1.0, 1.0)):
    return SimpleNamespace(ni=ni, nj=nj, nk=nk, nodes=nodes, x0=(0.0, 0.0, 0.0), h=h)


def _conn(db, df, lo, hi, sb, sf, slo, t=(1, 2)):
    return SimpleNamespace(dst_block=db, dst_face=df, dst_lo=lo, dst_hi=hi, src_block=sb, src_face=sf, src_lo=slo,
                           transform=t)


def _patch(face, hi, kind, state=(0.0,) * 5):
    return SimpleNamespace(block=0, face=face, lo=(0, 0), hi=hi, kind=kind, state=tuple(map(float, state)))


def _extent(b):
    return (b.ni, b.nj, b.nk)


def _other(a):
    return [x for x in range(3) if x != a]


def _periodic(b, axes):
    out = []
    for a in axes:
        hi = tuple(_extent(b)[x] for x in _other(a))
        out.append(_conn(0, 2 * a, (0, 0), hi, 0, 2 * a + 1, (0, 0)))
        out.append(_conn(0, 2 * a + 1, (0, 0), hi, 0, 2 * a, (0, 0)))
    return out


def _cons(rho, u, v, w, p):
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w)])


def _dt(rho, u, v, w, p, h, dim):
    c = torch.sqrt(GAMMA * p / rho)
    s = (u.abs() + c) / h[0] + (v.abs() + c) / h[1] + ((w.abs() + c) / h[2] if dim == 3 else 0.0)
    return 0.5 / float(s.max())


def _axis(lo, hi, h=1.0, x0=0.0):
    return x0 + h * torch.arange(lo, hi, dtype=torch.float64, device="cuda")


def _grid(z, y, x):
    return torch.meshgrid(z, y, x, indexing="ij")


def _vortex(case, seed):
    """2D isentropic vortex in uniform flow at 45 degrees, periodic (strength,
    centre and Mach number from the seed)."""
    rng = np.random.default_rng(seed)
    n, h = case["ni"], 10.0 / case["ni"]
    b = _block(n, n, 1, None, (h, h, 1.0))
    beta, mach, cx, cy = 5.0 + rng.uniform(-0.5, 0.5), rng.uniform(0.4, 0.6), *rng.uniform(-0.5, 0.5, 2)
    x = _axis(-2, n + 2, h, -5.0 + 0.5 * h)
    _, Y, X = _grid(_axis(-2, 3), x - cy, x - cx)
    r2 = X * X + Y * Y
    e = torch.exp(0.5 * (1.0 - r2))
    u0 = mach * math.sqrt(GAMMA / 2.0)
    T = 1.0 - (GAMMA - 1.0) * beta ** 2 / (8.0 * GAMMA * math.pi ** 2) * torch.exp(1.0 - r2)
    rho = T ** (1.0 / (GAMMA - 1.0))
    V = (rho, u0 - beta / (2 * math.pi) * Y * e, u0 + beta / (2 * math.pi) * X * e, torch.zeros_like(X), rho ** GAMMA)
    return dict(dim=2, blocks=[b], conns=_periodic(b, (0, 1)), q=[_cons(*V)], dt=_dt(*V, b.h, 2))


def _ripple(shape, rng, dim):
    """1 + a few smooth waves over the index space (1 %), whole periods an axis."""
    n = [_axis(-2, s - 2) / (s - 4) for s in shape]
    out = 0.0
    for _ in range(3):
        k = rng.integers(1, 4, 3)
        ph = rng.uniform(0, 2 * math.pi, 3)
        w = [torch.sin(2 * math.pi * float(k[a]) * n[a] + float(ph[a])) for a in range(3)]
        out = out + 0.01 * (w[0].view(-1, 1, 1) if dim == 3 else 1.0) * w[1].view(1, -1, 1) * w[2].view(1, 1, -1)
    return 1.0 + out.expand(shape)


def _stream(mach, p, T, alpha_deg):
    rho = p / (AIR["r_gas"] * T)
    c = math.sqrt(GAMMA * p / rho)
    a = math.radians(alpha_deg)
    return (rho, mach * c * math.cos(a), mach * c * math.sin(a), 0.0, p)


def _disturbed(V0, shape, rng, dim):
    """The free stream with smooth disturbances of a percent or so."""
    speed = math.hypot(V0[1], V0[2])
    V = [V0[0] * _ripple(shape, rng, dim), *(V0[a] + speed * (_ripple(shape, rng, dim) - 1.0) for a in (1, 2, 3)),
         V0[4] * _ripple(shape, rng, dim)]
    if dim == 2:
        V[3] = torch.zeros_like(V[3])
    return V


def _spacing(nodes, dim):
    d = [float(torch.linalg.vector_norm(torch.diff(nodes, dim=ax), dim=-1).min()) for ax in (2, 1, 0)[:dim]]
    return d + [1.0] * (3 - dim)


def _inlet(case, seed):
    """2D channel with a 10 degree ramp, Mach-4 inflow, outflow, slip walls."""
    rng = np.random.default_rng(seed)
    ni, nj = case["ni"], case["nj"]
    x = 3.0 * _axis(0, ni + 1) / ni
    lower = torch.clamp(x - 1.0, min=0.0) * math.tan(math.radians(10.0))
    s = _axis(0, nj + 1) / nj
    eta = (torch.exp(2.0 * s) - 1.0) / (math.exp(2.0) - 1.0)
    nodes = torch.zeros((2, nj + 1, ni + 1, 3), dtype=torch.float64, device="cuda")
    nodes[..., 0] = x
    nodes[..., 1] = lower + (1.0 - lower) * eta.view(-1, 1)
    nodes[1, ..., 2] = 1.0
    V0 = _stream(4.0, 12270.0, 217.0, 0.0)
    V = _disturbed(V0, (5, nj + 4, ni + 4), rng, 2)
    b = _block(ni, nj, 1, nodes.cpu().numpy())
    bcs = [_patch(0, (nj, 1), INFLOW, V0), _patch(1, (nj, 1), OUTFLOW), _patch(2, (ni, 1), SLIP),
           _patch(3, (ni, 1), SLIP)]
    return dict(dim=2, blocks=[b], conns=[], bcs=bcs, q=[_cons(*V)], dt=_dt(*V, _spacing(nodes, 2), 2))


def _ogrid(case, seed):
    """O-grid around a 12 % ellipse extruded over a unit span, transonic wing
    free stream; walls slip, or no-slip with the laminar terms."""
    rng = np.random.default_rng(seed)
    ni, nj, nk = case["ni"], case["nj"], case["nk"]
    th = -2.0 * math.pi * _axis(0, ni + 1) / ni
    w = (torch.exp(6.0 * _axis(0, nj + 1) / nj) - 1.0) / (math.exp(6.0) - 1.0)
    nodes = torch.zeros((nk + 1, nj + 1, ni + 1, 3), dtype=torch.float64, device="cuda")
    w = w.view(-1, 1)
    nodes[..., 0] = (1.0 - w) * 0.5 * torch.cos(th) + w * 20.0 * torch.cos(th)
    nodes[..., 1] = (1.0 - w) * 0.06 * torch.sin(th) + w * 20.0 * torch.sin(th)
    nodes[:, :, ni] = nodes[:, :, 0]
    nodes[..., 2] = (_axis(0, nk + 1) / nk).view(-1, 1, 1)
    V0 = _stream(0.8395, 315979.763, 255.556, 3.06)
    V = _disturbed(V0, (nk + 4, nj + 4, ni + 4), rng, 3)
    b = _block(ni, nj, nk, nodes.cpu().numpy())
    wall = NOSLIP if case.get("visc") else SLIP
    bcs = [_patch(2, (ni, nk), wall), _patch(3, (ni, nk), FARFIELD, V0), _patch(4, (ni, nj), wall),
           _patch(5, (ni, nj), wall)]
    return dict(dim=3, blocks=[b], conns=_periodic(b, (0,)), bcs=bcs, q=[_cons(*V)],
                dt=_dt(*V, _spacing(nodes, 3), 3))


# phi = phi0 + phix sin(ax pi x + p) + phiy cos(ay pi y + p) + phiz sin(az pi z + p)
_FIELDS = ((1.0, 0.15, -0.1, 0.1, 1.0, 0.5, 1.0 / 3.0), (0.4, 0.05, 0.03, 0.02, 1.5, 0.6, 0.5),
           (0.3, -0.04, 0.05, 0.02, 0.5, 2.0 / 3.0, 1.0), (0.25, 0.03, 0.02, -0.04, 1.0 / 3.0, 1.0, 0.5),
           (1.0 / GAMMA, 0.02, 0.01, -0.015, 2.0, 1.0, 1.5))


def _mms(case, seed):
    """Smooth manufactured flow in a perturbed unit cube: ghosts fixed to the
    fields, source = the divergence of their Euler flux (phases from the seed)."""
    rng = np.random.default_rng(seed)
    ph = rng.uniform(-0.4, 0.4, (5, 3))
    n = (case["ni"], case["nj"], case["nk"])
    Z, Y, X = _grid(*(_axis(-2, m + 3) / m for m in reversed(n)))
    tp = 2.0 * math.pi
    N = torch.stack([X + 0.1 / n[0] * torch.sin(tp * Y) * torch.sin(tp * Z),
                     Y + 0.1 / n[1] * torch.sin(tp * Z) * torch.sin(tp * X),
                     Z + 0.1 / n[2] * torch.sin(tp * X) * torch.sin(tp * Y)], dim=-1)
    c = N[:-1] + N[1:]
    c = c[:, :-1] + c[:, 1:]
    c = 0.125 * (c[:, :, :-1] + c[:, :, 1:])
    V, D = [], []
    for f, p in zip(_FIELDS, ph):
        a = [f[4 + x] * math.pi for x in range(3)]
        t = [a[x] * c[..., x] + float(p[x]) for x in range(3)]
        V.append(f[0] + f[1] * torch.sin(t[0]) + f[2] * torch.cos(t[1]) + f[3] * torch.sin(t[2]))
        D.append([f[1] * a[0] * torch.cos(t[0]), -f[2] * a[1] * torch.sin(t[1]), f[3] * a[2] * torch.cos(t[2])])
    rho, vel, p = V[0], V[1:4], V[4]
    k2 = 0.5 * sum(u * u for u in vel)
    H = GAMMA / (GAMMA - 1.0) * p + rho * k2
    S = [torch.zeros_like(rho) for _ in range(5)]
    for a in range(3):
        dm = D[0][a] * vel[a] + rho * D[1 + a][a]
        S[0] = S[0] + dm
        for x in range(3):
            S[1 + x] = S[1 + x] + dm * vel[x] + rho * vel[a] * D[1 + x][a] + (D[4][a] if x == a else 0.0)
        dH = (GAMMA / (GAMMA - 1.0) * D[4][a] + D[0][a] * k2
              + rho * sum(vel[x] * D[1 + x][a] for x in range(3)))
        S[4] = S[4] + D[1 + a][a] * H + vel[a] * dH
    src = torch.stack(S)[:, 2:-2, 2:-2, 2:-2].contiguous()
    inner = [v[2:-2, 2:-2, 2:-2] for v in V]
    b = _block(*n, N[2:-2, 2:-2, 2:-2].contiguous().cpu().numpy())
    return dict(dim=3, blocks=[b], conns=[], q=[_cons(*V)], source=[src], dt=_dt(*inner, [1.0 / m for m in n], 3))


def _batch(case, seed):
    """Uneven Cartesian blocks; half of the faces joined in pairs by rotated or
    flipped connections, fixed free-stream ghosts elsewhere (layout from the
    case); Mach-0.5 flow with 1 % noise (from the seed)."""
    rng = np.random.default_rng(case["layout"])
    h = (1.0 / 64,) * 3
    blocks = [_block(*map(int, d), None, h) for d in rng.integers(case["lo"], case["hi"] + 1, (case["nblocks"], 3))]
    faces = [(b, f) for b in range(len(blocks)) for f in range(6)]
    order = [faces[x] for x in rng.permutation(len(faces))]
    conns = []

    def ext(face):
        return [_extent(blocks[face[0]])[x] for x in _other(face[1] // 2)]

    for A, B in zip(order[0:len(order) // 2:2], order[1:len(order) // 2:2]):
        first = int(rng.integers(1, 3))
        T = [int(s) * t for s, t in zip(rng.choice([-1, 1], 2), (first, 3 - first))]
        ea, eb = ext(A), ext(B)
        L = [min(ea[t], eb[abs(T[t]) - 1]) for t in (0, 1)]
        lo = [int(rng.integers(0, ea[t] - L[t] + 1)) for t in (0, 1)]
        slo, rlo, rhi, rsrc, rT = [0, 0], [0, 0], [0, 0], [0, 0], [0, 0]
        for t in (0, 1):
            u = abs(T[t]) - 1
            at = int(rng.integers(0, eb[u] - L[t] + 1))
            slo[u] = at if T[t] > 0 else at + L[t] - 1
            rlo[u], rhi[u] = at, at + L[t]
            rsrc[t] = lo[t] if T[t] > 0 else lo[t] + L[t] - 1
            rT[u] = (1 if T[t] > 0 else -1) * (t + 1)
        conns.append(_conn(*A, lo, [lo[0] + L[0], lo[1] + L[1]], *B, slo, T))
        conns.append(_conn(*B, rlo, rhi, *A, rsrc, rT))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    one = torch.ones((1, 1, 1), dtype=torch.float64, device="cuda")
    V0 = [one, *(0.5 / math.sqrt(3.0) * one for _ in range(3)), one / GAMMA]
    q = []
    for b in blocks:
        s = _cons(*V0).expand(5, b.nk + 4, b.nj + 4, b.ni + 4).clone()
        noise = torch.rand((5, b.nk, b.nj, b.ni), generator=gen, dtype=torch.float64, device="cuda")
        s[:, 2:-2, 2:-2, 2:-2] *= 1.0 + 0.01 * (2.0 * noise - 1.0)
        q.append(s)
    return dict(dim=3, blocks=blocks, conns=conns, q=q, dt=_dt(*V0, h, 3) / 1.05)


def _waves(case, seed):
    """Periodic box, Mach-2 flow along x carrying eight density bumps."""
    rng = np.random.default_rng(seed)
    n = (case["ni"], case["nj"], case["nk"])
    h = 1.0 / n[0]
    b = _block(*n, None, (h, h, h))
    rho = 1.0
    for at in rng.uniform(0.0, 1.0, (8, 3)):
        g = []
        for a in range(3):
            d = _axis(-2, n[a] + 2, h, 0.5 * h) - float(at[a]) * n[a] * h
            d = d - n[a] * h * torch.round(d / (n[a] * h))
            g.append(torch.exp(-d * d / (2 * 0.05 ** 2)))
        rho = rho + 0.1 * g[2].view(-1, 1, 1) * g[1].view(1, -1, 1) * g[0].view(1, 1, -1)
    q = torch.zeros((5, *rho.shape), dtype=torch.float64, device="cuda")
    q[0] = rho
    q[1] = 2.0 * rho
    q[4] = 1.0 / GAMMA / (GAMMA - 1.0) + 2.0 * rho
    one = torch.ones(1, dtype=torch.float64)
    return dict(dim=3, blocks=[b], conns=_periodic(b, (0, 1, 2)), q=[q],
                dt=_dt(one, 2.0 * one, 0.0 * one, 0.0 * one, one / GAMMA, b.h, 3))


_PROBLEMS = {"vortex": _vortex, "inlet": _inlet, "ogrid": _ogrid, "mms": _mms, "batch": _batch, "periodic": _waves}


def _params(case):
    p = {"gamma": GAMMA, "eps": 1.0, "kappa": case.get("kappa", -1.0), "limiter": case.get("limiter", 1),
         "harten": 0.1, "fix_all": case.get("fix_all", 0), "flux": case.get("flux", 0), "alpha": ALPHA,
         "va_delta2": 1e-12}
    if case.get("visc"):
        p.update(visc=1, sutherland=1, **AIR)
    return p


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------

def _flat(arrays):
    return torch.cat([a.reshape(-1) for a in arrays])


def _cotangent(q, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand(q.shape, generator=gen, dtype=torch.float64, device="cuda") - 0.5


def prepare(case, seed):
    import paper_2012_02925_gb300 as fv
    pb = _PROBLEMS[case["kind"]](case, seed)
    s = fv.Solver(pb["blocks"], pb["conns"], pb["dim"], _params(case), precision=case["precision"])
    if pb.get("bcs"):
        s.set_boundaries(pb["bcs"])
    q = _flat(pb["q"])
    s.set_state(q)
    if pb.get("source"):
        s.set_source(_flat(pb["source"]))
    if case.get("autotune"):
        s.autotune(pb["dt"])
        s.set_state(q)
    if case.get("monitor"):
        s.set_monitor(True)
    state = {"case": case, "solver": s, "dt": pb["dt"]}
    if case["op"] == "adjoint":
        s.set_adjoint_arith(case["sweeps"])
        state["q"] = q.requires_grad_()
        state["cotangent"] = _cotangent(q, seed)
    torch.cuda.synchronize()
    return state


def run(state):
    case, s = state["case"], state["solver"]
    if case["op"] == "residual":
        return {"residual": s.residual(0)}
    if case["op"] == "adjoint":
        from paper_2012_02925_gb300 import autograd
        out = autograd.run_stages(s, state["q"], state["dt"], case["stages"])
        (grad,) = torch.autograd.grad(out, state["q"], state["cotangent"])
        return {"state": out.detach(), "gradient": grad}
    for _ in range(case["steps"]):
        s.rk_step(state["dt"])
    out = {"state": s.get_state(0)}
    if case.get("monitor"):
        out["l2"], out["linf"] = s.monitor_norms()
    return out


def _dims(case):
    if case["kind"] == "batch":
        rng = np.random.default_rng(case["layout"])
        return rng.integers(case["lo"], case["hi"] + 1, (case["nblocks"], 3)).astype(float)
    return np.array([[case["ni"], case["nj"], case["nk"]]], dtype=float)


def work(case):
    """Floating-point operations of the scheme per cell and stage (a face: 391;
    recovery, sums and update: 58; a viscous face: 195; a reverse face: three
    forward ones), and the state read and written once, the curvilinear face
    vectors and volume (104 B a cell) and the source (40 B) read once."""
    n = float(_dims(case).prod(axis=1).sum())
    dim = 2 if case["kind"] in ("vortex", "inlet") else 3
    flops = dim * (391.0 + (195.0 if case.get("visc") else 0.0)) + 58.0
    per = 80.0 + (104.0 if case["kind"] in ("inlet", "ogrid", "mms") else 0.0) + (40.0 if case["kind"] == "mms" else 0.0)
    stages = 1 if case["op"] == "residual" else case.get("stages", 4 * case.get("steps", 1))
    if case["op"] == "adjoint":
        flops, per = 4.0 * flops, per + 80.0
    return {"bytes": n * per, "flops": n * stages * flops}


# ---------------------------------------------------------------------------
# the same scheme in plain 64-bit torch
# ---------------------------------------------------------------------------

class _Exact:
    def __init__(self, case, pb):
        self.P = SimpleNamespace(**_params(case))
        self.visc, self.dim = bool(case.get("visc")), pb["dim"]
        self.blocks, self.conns, self.bcs = pb["blocks"], pb["conns"], pb.get("bcs") or []
        self.source = pb.get("source")
        self.S, self.vol, self.geo = [], [], []
        for b in self.blocks:
            S, vol = self._metrics(b)
            self.S.append(S)
            self.vol.append(vol)
            self.geo.append(self._padded_geometry(b, S, vol) if self.visc else None)

    @staticmethod
    def _metrics(b):
        if b.nodes is None:
            hx, hy, hz = b.h
            area = (hy * hz, hx * hz, hx * hy)
            S = []
            for a in range(3):
                v = torch.zeros((3, 1, 1, 1), dtype=torch.float64, device="cuda")
                v[a] = area[a]
                S.append(v)
            return S, torch.full((1, 1, 1), hx * hy * hz, dtype=torch.float64, device="cuda")
        N = torch.from_numpy(np.ascontiguousarray(b.nodes)).cuda().permute(3, 0, 1, 2)   # (3, k, j, i)
        lo, hi = slice(None, -1), slice(1, None)
        full = slice(None)
        corners = [  # the four nodes of a face, in order, per direction (k, j, i slices)
            ((lo, lo, full), (lo, hi, full), (hi, hi, full), (hi, lo, full)),
            ((lo, full, lo), (hi, full, lo), (hi, full, hi), (lo, full, hi)),
            ((full, lo, lo), (full, lo, hi), (full, hi, hi), (full, hi, lo))]
        S, vol = [], 0.0
        for a in range(3):
            p = [N[(full, *c)] for c in corners[a]]
            f = 0.5 * torch.linalg.cross(p[2] - p[0], p[3] - p[1], dim=0)
            S.append(f)
            flow = (0.25 * (p[0] + p[1] + p[2] + p[3]) * f).sum(0)
            vol = vol + torch.diff(flow, dim=2 - a) / 3.0
        return S, vol

    def _padded_geometry(self, b, S, vol):
        """(Omega, mean face vectors) of every cell and one layer of ghosts:
        the donor's across a periodic connection, else the neighbour's."""
        planes = [vol.unsqueeze(0)]
        for a in range(3):
            d = 3 - a
            planes.append(0.5 * (S[a].narrow(d, 0, S[a].shape[d] - 1) + S[a].narrow(d, 1, S[a].shape[d] - 1)))
        G = torch.cat(planes)
        joined = {c.dst_face // 2 for c in self.conns}
        for a in range(3):
            d, n = 3 - a, _extent(b)[a]
            first, last = G.narrow(d, 0, 1), G.narrow(d, n - 1, 1)
            G = torch.cat([last, G, first] if a in joined else [first, G, last], dim=d)
        return G

    # -- ghosts ---------------------------------------------------------------
    def fill(self, q):
        for c in self.conns:
            D, S = q[c.dst_block], q[c.src_block]
            da, sa = c.dst_face // 2, c.src_face // 2
            n = _extent(self.blocks[c.src_block])[sa]
            m = _extent(self.blocks[c.dst_block])[da]
            a = torch.arange(c.dst_hi[0] - c.dst_lo[0], device="cuda").view(1, -1)
            bb = torch.arange(c.dst_hi[1] - c.dst_lo[1], device="cuda").view(-1, 1)
            t = [None, None]
            for step, T in ((a, c.transform[0]), (bb, c.transform[1])):
                u = abs(T) - 1
                t[u] = c.src_lo[u] + (step if T > 0 else -step) + 2
            for d in (1, 2):
                face = S.select(3 - sa, (n - d if c.src_face & 1 else d - 1) + 2)
                ghost = D.select(3 - da, (m - 1 + d if c.dst_face & 1 else -d) + 2)
                ghost[:, c.dst_lo[1] + 2:c.dst_hi[1] + 2, c.dst_lo[0] + 2:c.dst_hi[0] + 2] = face[:, t[1], t[0]]
        for p in self.bcs:
            self._boundary(p, q[0])
        if self.visc:
            self._edges(q[0])

    def _boundary(self, p, q):
        b = self.blocks[0]
        a, side = p.face // 2, p.face & 1
        n = _extent(b)[a]

        def at(t):   # interior tangential cells of the layer at coordinate t
            return q.select(3 - a, t + 2)[:, 2:-2, 2:-2]

        S = self.S[0][a].select(3 - a, n if side else 0)
        nrm = S / torch.linalg.vector_norm(S, dim=0)
        near = at(n - 1 if side else 0).clone()
        state = torch.tensor(p.state, dtype=torch.float64, device="cuda").view(5, 1, 1)
        if p.kind == INFLOW:
            fixed = _cons(*state).expand_as(near)
        elif p.kind == OUTFLOW:
            fixed = near
        elif p.kind == FARFIELD:
            fixed = _cons(*self._farfield(self._prim(near), state, nrm if side else -nrm))
        for d in (1, 2):
            mirror = at(n - d if side else d - 1)
            if p.kind == SLIP:
                g = mirror.clone()
                g[1:4] -= 2.0 * (mirror[1:4] * nrm).sum(0) * nrm
            elif p.kind == NOSLIP:
                g = mirror * torch.tensor([1.0, -1.0, -1.0, -1.0, 1.0], dtype=torch.float64, device="cuda").view(5, 1, 1)
            else:
                g = fixed
            at(n - 1 + d if side else -d).copy_(g)

    @staticmethod
    def _farfield(Vi, Vf, n):
        ci, cf = torch.sqrt(GAMMA * Vi[4] / Vi[0]), torch.sqrt(GAMMA * Vf[4] / Vf[0])
        vi, vf = (Vi[1:4] * n).sum(0), (Vf[1:4] * n).sum(0)
        k = 2.0 / (GAMMA - 1.0)
        rp, rm = vi + k * ci, vf - k * cf
        vb, cb = 0.5 * (rp + rm), 0.25 * (GAMMA - 1.0) * (rp - rm)
        out = vb >= 0.0
        ref = torch.where(out, Vi, Vf.expand_as(Vi))
        rho = ref[0] * (cb / torch.where(out, ci, cf.expand_as(ci))) ** k
        vel = ref[1:4] + (vb - torch.where(out, vi, vf.expand_as(vi))) * n
        sub = torch.cat([rho.unsqueeze(0), vel, (rho * cb * cb / GAMMA).unsqueeze(0)])
        return torch.where(vi >= ci, Vi, torch.where(vi <= -ci, Vf.expand_as(Vi), sub))

    def _edges(self, q):
        """First-layer edge ghosts: across a periodic direction the donor's
        ghost, else the mean of the two adjacent face ghosts."""
        joined = {c.dst_face // 2 for c in self.conns}
        ext = _extent(self.blocks[0])
        new = []
        for a, b in ((0, 1), (0, 2), (1, 2)):
            c = 3 - a - b
            for sa in (0, 1):
                for sb in (0, 1):
                    ea, eb = (ext[a] if sa else -1), (ext[b] if sb else -1)

                    def line(ia, ib):
                        at = [slice(None)] * 4
                        at[3 - a], at[3 - b], at[3 - c] = ia + 2, ib + 2, slice(2, 2 + ext[c])
                        return tuple(at)

                    if a in joined:
                        v = q[line(0 if sa else ext[a] - 1, eb)]
                    elif b in joined:
                        v = q[line(ea, 0 if sb else ext[b] - 1)]
                    else:
                        v = 0.5 * (q[line(ea, ext[b] - 1 if sb else 0)] + q[line(ext[a] - 1 if sa else 0, eb)])
                    new.append((line(ea, eb), v.clone()))
        for at, v in new:
            q[at] = v

    # -- residual -------------------------------------------------------------
    @staticmethod
    def _prim(q):
        u = [q[x] / q[0] for x in (1, 2, 3)]
        return torch.stack([q[0], *u, (GAMMA - 1.0) * (q[4] - 0.5 * (q[1] * u[0] + q[2] * u[1] + q[3] * u[2]))])

    def _limited(self, a, b):
        """Psi(a/b) b"""
        if self.P.limiter == 0:
            return b
        if self.P.limiter == 1:
            same = a * b > 0
            return torch.where(same, 2.0 * a * b / torch.where(same, a + b, torch.ones_like(a)), torch.zeros_like(a))
        return b * (a * a + a * b) / (a * a + b * b + self.P.va_delta2)

    def _reconstruct(self, v):
        dm, d0, dp = v[1] - v[0], v[2] - v[1], v[3] - v[2]
        km, kp = 0.25 * self.P.eps * (1.0 - self.P.kappa), 0.25 * self.P.eps * (1.0 + self.P.kappa)
        L, R = v[1] + km * self._limited(d0, dm), v[2] - km * self._limited(d0, dp)
        if kp:
            L, R = L + kp * self._limited(dm, d0), R - kp * self._limited(dp, d0)
        return L, R

    def _roe(self, L, R, n):
        def side(V):
            Vn = (V[1:4] * n).sum(0)
            h = GAMMA / (GAMMA - 1.0) * V[4] / V[0] + 0.5 * (V[1:4] ** 2).sum(0)
            return Vn, h, torch.cat([(V[0] * Vn).unsqueeze(0), V[0] * Vn * V[1:4] + V[4] * n,
                                     (V[0] * Vn * h).unsqueeze(0)])

        VnL, hL, F = side(L)
        VnR, hR, FR = side(R)
        F = F + FR
        del FR
        w = torch.sqrt(R[0] / L[0])
        rho = L[0] * w
        u = (L[1:4] + w * R[1:4]) / (1.0 + w)
        h = (hL + w * hR) / (1.0 + w)
        q2 = 0.5 * (u * u).sum(0)
        c2 = (GAMMA - 1.0) * (h - q2)
        c = torch.sqrt(c2)
        Vn = (u * n).sum(0)
        lam = [(Vn - c).abs(), Vn.abs(), (Vn + c).abs()]
        d = self.P.harten * c
        for x in range(3):
            if x != 1 or self.P.fix_all:
                lam[x] = torch.where(lam[x] < d, (lam[x] ** 2 + d * d) / (2.0 * d), lam[x])
        dV = R - L
        dn = VnR - VnL
        a1 = lam[0] * (dV[4] - rho * c * dn) / (2.0 * c2)
        a5 = lam[2] * (dV[4] + rho * c * dn) / (2.0 * c2)
        a2, a3 = lam[1] * (dV[0] - dV[4] / c2), lam[1] * rho
        du = dV[1:4] - dn * n
        D = torch.cat([(a1 + a2 + a5).unsqueeze(0), a1 * (u - c * n) + a5 * (u + c * n) + a2 * u + a3 * du,
                       (a1 * (h - c * Vn) + a5 * (h + c * Vn) + a2 * q2
                        + a3 * ((u * dV[1:4]).sum(0) - Vn * dn)).unsqueeze(0)])
        return 0.5 * (F - D)

    def _split(self, V, n, sg):
        """Flux-vector splittings F+ (sg = 1) and F- (sg = -1)."""
        rho, vel, p = V[0], V[1:4], V[4]
        c = torch.sqrt(GAMMA * p / rho)
        Vn = (vel * n).sum(0)
        q2 = (vel * vel).sum(0)
        H = c * c / (GAMMA - 1.0) + 0.5 * q2
        if self.P.flux == 1:
            full = torch.cat([(rho * Vn).unsqueeze(0), rho * Vn * vel + p * n, (rho * Vn * H).unsqueeze(0)])
            f = 0.25 * sg * rho * c * (Vn / c + sg) ** 2
            e = ((GAMMA - 1.0) * Vn + 2.0 * sg * c) ** 2 / (2.0 * (GAMMA ** 2 - 1.0)) + 0.5 * (q2 - Vn * Vn)
            part = torch.cat([f.unsqueeze(0), f * (vel + n * (2.0 * sg * c - Vn) / GAMMA), (f * e).unsqueeze(0)])
            beyond = sg * Vn >= c
            return torch.where(beyond, full, torch.where(-sg * Vn >= c, torch.zeros_like(full), part))
        l1, l2, l5 = (0.5 * (x + sg * x.abs()) for x in (Vn - c, Vn, Vn + c))
        a2 = 2.0 * (GAMMA - 1.0) * l2
        k = rho / (2.0 * GAMMA)
        return torch.cat([(k * (a2 + l1 + l5)).unsqueeze(0), k * ((a2 + l1 + l5) * vel + (l5 - l1) * c * n),
                          (k * (0.5 * a2 * q2 + (l1 + l5) * H + (l5 - l1) * c * Vn)).unsqueeze(0)])

    def _viscous(self, Q, G, a, n, S):
        """tau.S and Theta.S of the faces along axis a (Q: u, v, w, T and G:
        geometry, both with one ghost layer)."""
        d = 3 - a
        others = [x for x in range(3) if x != a][: self.dim - 1]

        def cells(A, shift, side=0, x=None):   # L (side 0) or R (side 1) cells, moved by `shift` along x
            for y in range(3):
                m = A.shape[3 - y] - 2
                if y == a:
                    A = A.narrow(3 - y, side, m + 1)
                else:
                    A = A.narrow(3 - y, 1 + (shift if y == x else 0), m)
            return A

        QL, QR, gL, gR = cells(Q, 0), cells(Q, 0, 1), cells(G, 0), cells(G, 0, 1)
        om, A = 0.5 * (gL[0] + gR[0]), 0.5 * (gL[1:] + gR[1:])
        grad = (QR - QL).unsqueeze(1) * A[3 * a:3 * a + 3]
        for b in others:
            D = 0.25 * (cells(Q, 1, 0, b) - cells(Q, -1, 0, b) + cells(Q, 1, 1, b) - cells(Q, -1, 1, b))
            grad = grad + D.unsqueeze(1) * A[3 * b:3 * b + 3]
        grad = grad / om
        Qf = 0.5 * (QL + QR)
        T = Qf[3]
        mu = self.P.mu * (T / self.P.t_ref) ** 1.5 * (self.P.t_ref + self.P.s_suth) / (T + self.P.s_suth)
        k = mu * GAMMA * self.P.r_gas / (GAMMA - 1.0) / self.P.prandtl
        div = grad[0, 0] + grad[1, 1] + grad[2, 2]
        tS = []
        for x in range(3):
            t = sum((grad[x, y] + grad[y, x]) * S[y] for y in range(3)) - 2.0 / 3.0 * div * S[x]
            tS.append(mu * t)
        heat = k * sum(grad[3, y] * S[y] for y in range(3))
        return torch.stack([torch.zeros_like(heat), *tS, sum(tS[x] * Qf[x] for x in range(3)) + heat])

    def residual(self, q):
        out = []
        for bi, b in enumerate(self.blocks):
            V = self._prim(q[bi])
            R = 0.0
            if self.visc:
                Q = torch.cat([V[1:4], (V[4] / (V[0] * self.P.r_gas)).unsqueeze(0)])[:, 1:-1, 1:-1, 1:-1]
            for a in range(self.dim):
                W = V
                for x in range(3):
                    if x != a:
                        W = W.narrow(3 - x, 2, _extent(b)[x])
                d, n = 3 - a, _extent(b)[a]
                stencil = [W.narrow(d, s, n + 1) for s in range(4)]
                S = self.S[bi][a]
                area = torch.linalg.vector_norm(S, dim=0)
                nrm = S / area
                L, Rt = self._reconstruct(stencil)
                if self.P.flux == 0:
                    F = self._roe(L, Rt, nrm) * area
                else:
                    F = (self._split(L, nrm, 1.0) + self._split(Rt, nrm, -1.0)) * area
                del L, Rt
                for p in self.bcs:
                    if p.face // 2 == a and p.kind in (SLIP, NOSLIP, FARFIELD):
                        side = p.face & 1
                        Sf = S.select(d, n if side else 0)
                        face = F.select(d, n if side else 0)
                        if p.kind == FARFIELD:
                            g = W.select(d, n + 2 if side else 1)
                            Vn = (g[1:4] * Sf).sum(0)
                            h = GAMMA / (GAMMA - 1.0) * g[4] / g[0] + 0.5 * (g[1:4] ** 2).sum(0)
                            new = torch.cat([(g[0] * Vn).unsqueeze(0), g[0] * Vn * g[1:4] + g[4] * Sf,
                                             (g[0] * Vn * h).unsqueeze(0)])
                        else:
                            p1, p2 = (W[4].select(d - 1, n + 1 - x if side else 2 + x) for x in (0, 1))
                            z = torch.zeros_like(p1)
                            new = torch.stack([z, *((1.5 * p1 - 0.5 * p2) * Sf[x] for x in range(3)), z])
                        face.copy_(new)
                if self.visc:
                    F = F - self._viscous(Q, self.geo[bi], a, n, S)
                R = R + torch.diff(F, dim=d)
                del F
            if self.source:
                R = R - self.source[bi] * self.vol[bi]
            out.append(R)
        return out

    def stage(self, q0, R, m, dt):
        """Interior of Q^(m) per block."""
        return [q[:, 2:-2, 2:-2, 2:-2] - ALPHA[m] * dt / v * r for q, v, r in zip(q0, self.vol, R)]

    def step(self, q, dt):
        """One time step of the packed states q in place (ghosts of q as the
        first stage filled them); the residual of the step's start."""
        start = [x.clone() for x in q]
        cur = q
        for m in range(4):
            self.fill(cur)
            R = self.residual(cur)
            if m == 0:
                first = R
            new = self.stage(q, R, m, dt)
            if m == 3:
                for x, y in zip(q, new):
                    x[:, 2:-2, 2:-2, 2:-2] = y
            else:
                cur = [x.clone() for x in start]
                for x, y in zip(cur, new):
                    x[:, 2:-2, 2:-2, 2:-2] = y
        return first


def exact(case, seed):
    pb = _PROBLEMS[case["kind"]](case, seed)
    E, q, dt = _Exact(case, pb), pb["q"], pb["dt"]
    if case["op"] == "residual":
        return {"residual": _flat(E.residual(q))}
    if case["op"] == "adjoint":
        # fixed ghosts: the interior is what the gradient is taken of
        base = q[0]
        x = base[:, 2:-2, 2:-2, 2:-2].clone().requires_grad_()

        def whole(i):
            return torch.nn.functional.pad(i, (2,) * 6) + edge

        edge = base.clone()
        edge[:, 2:-2, 2:-2, 2:-2] = 0.0
        q0 = cur = whole(x)
        for st in range(case["stages"]):
            m = st % 4
            if m == 0:
                q0 = cur
            cur = whole(E.stage([q0], E.residual([cur]), m, dt)[0])
        lam = _cotangent(_flat([base]), seed).view(base.shape)[:, 2:-2, 2:-2, 2:-2]
        (g,) = torch.autograd.grad(cur[:, 2:-2, 2:-2, 2:-2], x, lam)
        return {"state": cur.detach().reshape(-1), "gradient": torch.nn.functional.pad(g, (2,) * 6).reshape(-1)}
    for _ in range(case["steps"]):
        R = E.step(q, dt)
    out = {"state": _flat(q)}
    if case.get("monitor"):
        r = torch.cat([x.reshape(5, -1) for x in R], dim=1)
        out["l2"] = torch.sqrt((r * r).mean(dim=1)).cpu().numpy()
        out["linf"] = r.abs().amax(dim=1).cpu().numpy()
    return out
