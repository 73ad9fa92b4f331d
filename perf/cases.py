"""Performance cases: what a user of the library has it do, through the calls of
paper_2203_00879_gb300.nopcs, and the same results in 64 bits from plain torch.

A case is a dict of plain values:
  what   "step"     RK4 steps of a box already on the device, then its state
         "boxes"    one RK4 step of a batch of independent boxes, then their states
         "member"   a state in, a step, a filter, diagnostics, the state out
         "rhs"      one right-hand side of a given state
         "grad"     the derivative of one field along x, y and z
  nx, ny, nz, sub   grid and NOHAP sub-domain length (0: whole lines)
  prec   "mixed" or "f64" (grad: the field's type, "f32" or "f64")
  steps, gravity, compact, order, count: what the kinds below use
"""
import math

import numpy as np
import torch

from paper_2203_00879_gb300 import nopcs as N

# the two-temperature Rayleigh-Taylor problem of the benchmark (arXiv 2203.00879, Sec. 2)
TS_KELVIN, MU_S_SI, S_SUTH = 300.0, 1.8459162511975804e-05, 110.4 / 300.0
RE, MACH, PR, GAMMA = 12080.6, 0.0034939, 0.712, 1.4
T_LOW, ALPHA_F = 500.0 / 300.0, 0.135
DT = 7.69e-8 / math.sqrt(0.15 / 9.81)
# edges and heights of the batched workload's boxes
EDGES = (32, 48, 64, 96, 128)


def listed():
    return [
        # the smallest workload of the repository (48^3): a step is a chain of
        # small kernels, so launches and latency count
        dict(name="step-48-mixed", what="step", nx=48, ny=48, nz=48, sub=24, prec="mixed", steps=1, gravity=2, compact=0),
        # an ordinary box in the paper's own precision
        dict(name="step-128-f64", what="step", nx=128, ny=128, nz=128, sub=64, prec="f64", steps=1, gravity=2, compact=0),
        # odd sizes, gravity along y, a few steps between two outputs
        dict(name="step-ragged-mixed", what="step", nx=201, ny=263, nz=171, sub=32, prec="mixed", steps=4, gravity=1,
             compact=0),
        # the mid-size box of the benchmark's configurations
        dict(name="step-512-mixed", what="step", nx=512, ny=512, nz=512, sub=64, prec="mixed", steps=1, gravity=2,
             compact=0),
        # the largest: lines of 1024 points, as in the headline run
        dict(name="step-1024-mixed", what="step", nx=1024, ny=512, nz=512, sub=64, prec="mixed", steps=1, gravity=2,
             compact=0),
        # the option of compact viscous terms
        dict(name="step-compact-mixed", what="step", nx=256, ny=256, nz=256, sub=64, prec="mixed", steps=1, gravity=2,
             compact=1),
        # a parameter study: independent uneven boxes advanced together
        dict(name="boxes-16-mixed", what="boxes", nx=0, ny=0, nz=0, sub=64, prec="mixed", steps=1, gravity=2, compact=0,
             count=16),
        # one ensemble member: its state comes in, is advanced, filtered and
        # diagnosed, and goes out
        dict(name="member-256-mixed", what="member", nx=256, ny=256, nz=256, sub=64, prec="mixed", steps=1, gravity=2,
             compact=0),
        # a caller with its own time integration takes right-hand sides
        dict(name="rhs-ragged-mixed", what="rhs", nx=321, ny=257, nz=203, sub=64, prec="mixed", gravity=2, compact=0),
        # gradient of one field: the 512^3 derivative workload in single
        # precision, a ragged one in double
        dict(name="grad-512-f32", what="grad", nx=512, ny=512, nz=512, sub=64, prec="f32", order=1),
        dict(name="grad-ragged-f64", what="grad", nx=257, ny=193, nz=301, sub=64, prec="f64", order=1),
        # the three compact second derivatives of a small field (order 3)
        dict(name="second-96-f32", what="grad", nx=96, ny=80, nz=72, sub=32, prec="f32", order=3),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["step", "step", "step", "boxes", "member", "rhs", "grad", "grad"])
    n = [_size(rng, 24, 640) for _ in range(3)]
    prec = "mixed"
    if what == "grad":
        prec = rng.choice(["f32", "f32", "f64"])
    elif what in ("step", "rhs", "member") and rng.random() < 0.2:
        prec = "f64"
    most = {"mixed": 6e7, "f32": 1.3e8, "f64": 2e7 if what == "grad" else 3e6}[prec]
    while n[0] * n[1] * n[2] > most:
        n[max(range(3), key=lambda d: n[d])] //= 2
    if rng.random() < 0.25:  # long x lines, as in the headline run
        n[0] = 1024 + rng.randrange(0, 65)
        n[1] = min(n[1], 128)
        n[2] = min(n[2], 128 if prec != "f64" else 20)
    c = dict(what=what, nx=n[0], ny=n[1], nz=n[2], sub=rng.choice([24, 32, 64, 64, 128]), prec=prec)
    if max(n) <= 256 and rng.random() < 0.2:
        c["sub"] = 0
    if what == "grad":
        c["order"] = rng.choice([1, 1, 2, 3])
        return c
    c["gravity"] = rng.choice([2, 2, 2, 0, 1])
    c["compact"] = 1 if what in ("step", "rhs") and rng.random() < 0.25 else 0
    if what == "step":
        c["steps"] = rng.choice([1, 1, 2, 5])
    elif what == "member":
        c["steps"] = 1
    elif what == "boxes":
        c.update(nx=0, ny=0, nz=0, steps=1, gravity=2, sub=rng.choice([32, 64]), count=rng.randrange(2, 25))
    return c


# ---- inputs ---------------------------------------------------------------------
def _shapes(case):
    """(nx, ny, nz) of the case's boxes."""
    if case["what"] != "boxes":
        return [(case["nx"], case["ny"], case["nz"])]
    out = []
    for b in range(case["count"]):
        e = EDGES[(3 * b + 1) % len(EDGES)]
        out.append((e, e, 2 * int(e * (1.0 + (0.37 * b + 0.21) % 1.0) / 2.0)))
    return out


def _params(case, n):
    h = 1.0 / (n[0] - 1)
    return dict(n=n, len=tuple(h * (v - 1) for v in n), gravity_axis=case.get("gravity", 2), sub_n=(case["sub"],) * 3,
                Re=RE, M=MACH, Pr=PR, gamma=GAMMA, suth_S=S_SUTH, mub_scale=1.0, mu_s_si=MU_S_SI, Ts_kelvin=TS_KELVIN,
                T_upper=1.0, T_lower=T_LOW, g=1.0, dt=DT, filter_every=50, filter_alpha=ALPHA_F,
                base_subtract=1 if case["prec"] == "mixed" else 0, seed=1, perturb_amp=0.0,
                visc_compact=case.get("compact", 0))


def _along(v, d):
    """A profile along axis d (0 = x) as a factor of a (z, y, x) field."""
    return v.reshape([-1 if a == 2 - d else 1 for a in range(3)])


def _base(p):
    """Hydrostatic density and pressure along the gravity axis."""
    d = p["gravity_axis"]
    z = torch.arange(p["n"][d], dtype=torch.float64, device="cuda") * (p["len"][d] / (p["n"][d] - 1))
    zi, gm2 = 0.5 * p["len"][d], GAMMA * MACH * MACH
    T = torch.where(z < zi, torch.full_like(z, p["T_lower"]), torch.full_like(z, p["T_upper"]))
    pr = torch.exp(-gm2 * p["g"] * (z - zi) / T) / gm2
    return _along(gm2 * pr / T, d), _along(pr, d)


def _waves(n, gen, kmax):
    """A smooth field of values around 1 in size: a few waves with random phases and amplitudes."""
    out = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    for d in range(3):
        x = torch.linspace(0.0, 1.0, n[d], dtype=torch.float64, device="cuda")
        ph = torch.rand(kmax, generator=gen, dtype=torch.float64, device="cuda")
        am = torch.rand(kmax, generator=gen, dtype=torch.float64, device="cuda")
        k = torch.arange(1, kmax + 1, dtype=torch.float64, device="cuda")
        out += _along((am[:, None] / k[:, None] * torch.sin(2 * math.pi * (k[:, None] * x + ph[:, None]))).sum(0), d)
    return out


def _state(p, seed, index=0):
    """A disturbed box: density and energy off the hydrostatic base by about 1e-4, velocities of about 1e-3, zero
    on the walls; waves, a mean flow and a little noise."""
    n = p["n"]
    gen = torch.Generator(device="cuda").manual_seed(1000 * (seed % (1 << 40)) + index)

    def field(amp):
        f = _waves(n, gen, 8)
        f += 0.05 * torch.randn(f.shape, generator=gen, dtype=torch.float64, device="cuda")
        return f.mul_(amp)

    q = torch.empty((5, n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    rho, pr = _base(p)
    q[0] = rho * field(1e-4).add_(1.0)
    q[4] = pr / (GAMMA - 1.0) * field(1e-4).add_(1.0)
    bump = 2e-3
    for d in range(3):
        bump = bump * _along(torch.sin(torch.linspace(0.0, math.pi, n[d], dtype=torch.float64, device="cuda")), d)
    for k in range(1, 4):
        q[k] = q[0] * (field(1e-3) + bump)
        for d in range(3):
            q[k].select(2 - d, 0).zero_()
            q[k].select(2 - d, n[d] - 1).zero_()
    return q


def _field(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    gen = torch.Generator(device="cuda").manual_seed(seed % (1 << 40))
    f = _waves(n, gen, 48)
    f += 1e-3 * torch.randn(f.shape, generator=gen, dtype=torch.float64, device="cuda")
    return f if case["prec"] == "f64" else f.float()


class _Context:
    """Owns a library context."""

    def __init__(self, boxes, prec):
        self.handle = N.nopcs_init(boxes, prec=prec, stream=torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "handle", None):
            N.nopcs_destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    boxes = [_params(case, n) for n in _shapes(case)]
    s = dict(case=case, ctx=_Context(boxes, N.NOPCS_FP64 if case["prec"] == "f64" else N.NOPCS_MIXED))
    if case["what"] == "grad":
        s["f"] = _field(case, seed)
        s["out"] = [torch.empty_like(s["f"]) for _ in range(3)]
        return s
    s["q"] = [_state(p, seed, b) for b, p in enumerate(boxes)]
    if case["what"] == "rhs":
        s["out"] = [torch.empty_like(s["q"][0], dtype=torch.float64 if case["prec"] == "f64" else torch.float32)]
        return s
    s["out"] = [torch.empty_like(q) for q in s["q"]]
    if case["what"] != "member":
        torch.cuda.synchronize()
        for b, q in enumerate(s["q"]):
            N.nopcs_set_state(s["ctx"].handle, b, q.data_ptr())
        del s["q"]
    return s


def run(s):
    case, ctx, out = s["case"], s["ctx"].handle, s["out"]
    if case["what"] == "grad":
        st = torch.cuda.current_stream().cuda_stream
        for d in range(3):
            N.nopcs_derivative(ctx, 0, d, case["order"], 1 if case["prec"] == "f32" else 0, s["f"].data_ptr(),
                               out[d].data_ptr(), st)
        return out
    if case["what"] == "rhs":
        N.nopcs_rhs(ctx, 0, s["q"][0].data_ptr(), out[0].data_ptr())
        return out
    if case["what"] == "member":
        N.nopcs_set_state(ctx, 0, s["q"][0].data_ptr())
        N.nopcs_set_step(ctx, 0, 0)
        N.nopcs_rk_step(ctx, case["steps"])
        N.nopcs_filter(ctx, 0)
        diag = N.nopcs_diagnostics(ctx, 0)
        N.nopcs_get_state(ctx, 0, out[0].data_ptr())
        return {"q": out[0], "diag": diag}
    N.nopcs_rk_step(ctx, case["steps"])
    for b, q in enumerate(out):
        N.nopcs_get_state(ctx, b, q.data_ptr())
    return out


def work(case):
    """Bytes: derivatives read and write each field once.  A right-hand side reads the FP64 state and writes five
    fields.  A classical RK4 step of a state that no chip holds reads and writes, per point, stage 1: the stage state
    in, slope sum and next stage state out; stages 2 and 3: stage state, slope sum and the state's copy in the compute
    precision in, slope sum and next stage state out; stage 4: stage state, slope sum and FP64 state in, FP64 state
    out.  Operations: about 10 for each derivative and field, 250 for the other terms of a stage."""
    pts = float(sum(n[0] * n[1] * n[2] for n in _shapes(case)))
    es = 4.0 if case["prec"] in ("mixed", "f32") else 8.0
    if case["what"] == "grad":
        times = 2.0 if case["order"] == 2 else 1.0
        return {"bytes": 3 * 2 * es * pts, "flops": 3 * 10.0 * times * pts}
    stage = (3 * 5 * 10.0 + (24 * 10.0 if case["compact"] else 0.0) + 250.0) * pts
    if case["what"] == "rhs":
        return {"bytes": (40.0 + 5 * es) * pts, "flops": stage}
    step = (5 * es * (3 + 5 + 5 + 2) + 80.0) * pts
    more = (40.0 + 80.0 + 40.0) * pts if case["what"] == "member" else 0.0
    return {"bytes": case["steps"] * step + more, "flops": case["steps"] * 4 * stage}


# ---- the same in 64 bits ----------------------------------------------------------
def _tri_solve(alpha, implicit, rhs):
    """Lines along the first axis of rhs: x[i] + alpha (x[i-1] + x[i+1]) = rhs[i] where implicit[i], x[i] = rhs[i]
    elsewhere.  In place."""
    n = rhs.shape[0]
    cp = [0.0] * n
    for i in range(n):
        a = alpha if implicit[i] else 0.0
        den = 1.0 - (a * cp[i - 1] if i else 0.0)
        cp[i] = a / den
        if a:
            rhs[i].sub_(rhs[i - 1], alpha=a).div_(den)
    for i in range(n - 2, -1, -1):
        if cp[i]:
            rhs[i].sub_(rhs[i + 1], alpha=cp[i])
    return rhs


def _lines(f, d):
    """A copy of the (z, y, x) field with axis d first."""
    return f.movedim(2 - d, 0).contiguous()


def _first(f, d, h):
    """The OUCS3 first derivative of a field along d, whole lines."""
    a, b1, b2, be = 0.3793894912, 0.7877868952, 0.045801298, -0.025
    f = _lines(f, d)
    n = f.shape[0]
    r = torch.empty_like(f)
    r[2:-2] = b1 * (f[3:-1] - f[1:-3]) + b2 * (f[4:] - f[:-4])
    e0 = (-1.5, 2.0, -0.5)
    e1 = (2 * be / 3 - 1.0 / 3, -(8 * be / 3 + 0.5), 4 * be + 1, -(8 * be / 3 + 1.0 / 6), 2 * be / 3)
    r[0] = sum(c * f[j] for j, c in enumerate(e0))
    r[-1] = -sum(c * f[n - 1 - j] for j, c in enumerate(e0))
    r[1] = sum(c * f[j] for j, c in enumerate(e1))
    r[-2] = -sum(c * f[n - 1 - j] for j, c in enumerate(e1))
    _tri_solve(a, [2 <= i <= n - 3 for i in range(n)], r)
    return r.div_(h).movedim(0, 2 - d)


def _second(f, d, h):
    """The sixth-order compact second derivative."""
    a, b = 12.0 / 11.0, 3.0 / 11.0
    f = _lines(f, d)
    n = f.shape[0]
    r = torch.empty_like(f)
    r[1:-1] = f[2:] - 2 * f[1:-1] + f[:-2]
    r[2:-2] = a * r[2:-2] + 0.25 * b * (f[4:] - 2 * f[2:-2] + f[:-4])
    r[0] = 2 * f[0] - 5 * f[1] + 4 * f[2] - f[3]
    r[-1] = 2 * f[-1] - 5 * f[-2] + 4 * f[-3] - f[-4]
    _tri_solve(2.0 / 11.0, [2 <= i <= n - 3 for i in range(n)], r)
    return r.div_(h * h).movedim(0, 2 - d)


def _filtered(f, d, af):
    """The sixth-order implicit filter; three points next to each wall stay."""
    f = _lines(f, d)
    n = f.shape[0]
    r = f.clone()
    if n > 6:
        r[3:-3] = (11 + 10 * af) / 16 * f[3:-3] + (15 + 34 * af) / 64 * (f[4:-2] + f[2:-4]) \
            + (-3 + 6 * af) / 32 * (f[5:-1] + f[1:-5]) + (1 - 2 * af) / 64 * (f[6:] + f[:-6])
        _tri_solve(af, [3 <= i <= n - 4 for i in range(n)], r)
    return r.movedim(0, 2 - d)


def _explicit(f, d, h):
    """Second-order differences, one-sided on the walls."""
    r = torch.empty_like(f)
    g, o = f.movedim(2 - d, 0), r.movedim(2 - d, 0)
    o[1:-1] = g[2:] - g[:-2]
    o[0] = -3 * g[0] + 4 * g[1] - g[2]
    o[-1] = 3 * g[-1] - 4 * g[-2] + g[-3]
    return r.div_(2 * h)


def _walls(f, d):
    return f.select(2 - d, 0), f.select(2 - d, f.shape[2 - d] - 1)


def _right_side(p, q):
    """The right-hand side of the compressible equations, momentum held on the walls."""
    gm2, ga = GAMMA * MACH * MACH, p["gravity_axis"]
    h = [p["len"][d] / (p["n"][d] - 1) for d in range(3)]
    rho_b, p_b = _base(p) if p["base_subtract"] else (0.0, 0.0)
    rho, V = q[0], [q[k] / q[0] for k in (1, 2, 3)]
    pr = (GAMMA - 1) * (q[4] - 0.5 * (q[1] * V[0] + q[2] * V[1] + q[3] * V[2]))
    R = torch.zeros_like(q)
    for d in range(3):
        R[0] -= _first(q[1 + d], d, h[d])
        for k in range(3):
            F = q[1 + d] * V[k]
            R[1 + k] -= _first(F + (pr - p_b) if k == d else F, d, h[d])
        R[4] -= _first((q[4] + pr) * V[d], d, h[d])
    T = gm2 * pr / rho
    mu = T * torch.sqrt(T) * (1 + S_SUTH) / (T + S_SUTH)
    mub = 1e-4 * (3.381 * T * TS_KELVIN - 7.383) / MU_S_SI
    kap = -mu / ((GAMMA - 1) * PR * RE * MACH * MACH)
    diff = _first if p["visc_compact"] else _explicit
    g = [[diff(V[k], d, h[d]) for k in range(3)] for d in range(3)]  # g[d][k] = dV_k / dx_d
    div = g[0][0] + g[1][1] + g[2][2]
    for d in range(3):
        tau = []
        for k in range(3):
            t = mu * (g[d][k] + g[k][d])
            if k == d:
                t += (mub - 2.0 / 3.0 * mu) * div
            tau.append(t.div_(RE))
        heat = kap * diff(T, d, h[d])
        for w in _walls(heat, d):
            w.zero_()
        for k in range(3):
            R[1 + k] += diff(tau[k], d, h[d])
        R[4] += diff(V[0] * tau[0] + V[1] * tau[1] + V[2] * tau[2] - heat, d, h[d])
    R[1 + ga] -= (rho - rho_b) * p["g"]
    R[4] -= q[1 + ga] * p["g"]
    for k in (1, 2, 3):
        for d in range(3):
            for w in _walls(R[k], d):
                w.zero_()
    return R


def _wall_state(p, q):
    """No-slip adiabatic walls: faces, then edges from the faces, then corners from the edges."""
    n, gm2 = p["n"], GAMMA * MACH * MACH

    def temp(at):
        v = q[(slice(None),) + at]
        return gm2 * (GAMMA - 1) * (v[4] - 0.5 * (v[1] ** 2 + v[2] ** 2 + v[3] ** 2) / v[0]) / v[0]

    for axes in ([(0,), (1,), (2,)], [(0, 1), (0, 2), (1, 2)], [(0, 1, 2)]):
        done = []
        for ds in axes:
            for sides in range(1 << len(ds)):
                at = [slice(1, -1)] * 3  # z, y, x
                for j, d in enumerate(ds):
                    at[2 - d] = n[d] - 1 if sides >> j & 1 else 0
                tw = 0.0
                for j, d in enumerate(ds):
                    one, two = list(at), list(at)
                    one[2 - d], two[2 - d] = (n[d] - 2, n[d] - 3) if sides >> j & 1 else (1, 2)
                    tw = tw + (4 * temp(tuple(one)) - temp(tuple(two))) / 3
                done.append((tuple(at), tw / len(ds)))
        for at, tw in done:
            for k in (1, 2, 3):
                q[(k,) + at] = 0.0
            q[(4,) + at] = q[(0,) + at] * tw / (GAMMA * (GAMMA - 1) * MACH * MACH)
    return q


def _advance(p, q, steps):
    for _ in range(steps):
        k = _right_side(p, q)
        total = k.clone()
        for c, w in ((0.5, 2.0), (0.5, 2.0), (1.0, 1.0)):
            k = _right_side(p, _wall_state(p, torch.add(q, k, alpha=c * DT)))
            total.add_(k, alpha=w)
        q = _wall_state(p, q.add_(total, alpha=DT / 6))
    return q


def _filter_state(p, q):
    dev = q.clone()
    if p["base_subtract"]:
        rho, pr = _base(p)
        dev[0] -= rho
        dev[4] -= pr / (GAMMA - 1)
    for k in range(5):
        f = dev[k]
        for d in range(3):
            f = _filtered(f, d, ALPHA_F)
        q[k] += f - dev[k]
    return q


def _diagnose(p, q, step):
    h = [p["len"][d] / (p["n"][d] - 1) for d in range(3)]
    vol = h[0] * h[1] * h[2]
    ga = p["gravity_axis"]
    z = _along(torch.arange(p["n"][ga], dtype=torch.float64, device="cuda") * h[ga], ga)
    s2 = (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0] ** 2
    pr = (GAMMA - 1) * (q[4] - 0.5 * q[0] * s2)
    return dict(mass=float(q[0].sum()) * vol, momentum=[float(q[k].sum()) * vol for k in (1, 2, 3)],
                energy_total=float((q[4] + q[0] * p["g"] * z).sum()) * vol, max_speed=math.sqrt(float(s2.max())),
                max_dp=float((pr - _base(p)[1]).abs().max()),
                max_mach=math.sqrt(float((s2 * q[0] / (GAMMA * pr)).max())), step=step,
                nonfinite=int(not bool(np.isfinite(float(q.sum())))))


def exact(case, seed):
    boxes = [_params(case, n) for n in _shapes(case)]
    if case["what"] == "grad":
        f = _field(case, seed).double()
        p, out = boxes[0], []
        for d in range(3):
            h = p["len"][d] / (p["n"][d] - 1)
            if case["order"] == 3:
                g = _second(f, d, h)
            else:
                g = _first(f, d, h)
                if case["order"] == 2:
                    g = _first(g, d, h)
            out.append(g.contiguous())
        return out
    # a step of a larger box would take too long, or not fit
    if case["what"] != "rhs" and case["nx"] * case["ny"] * case["nz"] * case["steps"] > 4e7:
        return None
    qs = [_state(p, seed, b) for b, p in enumerate(boxes)]
    if case["what"] == "rhs":
        return [_right_side(boxes[0], qs[0])]
    qs = [_advance(p, q, case["steps"]) for p, q in zip(boxes, qs)]
    if case["what"] == "member":
        q = _filter_state(boxes[0], qs[0])
        return {"q": q, "diag": _diagnose(boxes[0], q, case["steps"])}
    return qs
