"""Performance cases of the solver: what a user has it do, from the smallest
box to the largest, through the public Python binding.

Kinds of case
* ``step``: a state held in device memory goes in, some RK3 steps are taken,
  the new state comes out (``Solver.set_state``, ``rk3_step`` or
  ``rk3_step_forced``, ``get_state``); with ``adaptive`` the time step is taken
  anew from the state before every step (``Solver.cfl_dt``).
* ``batch``: many uneven periodic boxes advanced together (``Batch``).
* ``train``: one optimiser step of the correction network, or its loss and
  gradients (``CNN.train_step``, ``CNN.gradients``).
* ``corrected``: coarse steps with the network's correction after each
  (``CNN.step_corrected``).
* ``pairs``: one training pair: a fine state, filtered and advanced one coarse
  step, and the filtered fine state one coarse step later (``box_filter``).

``exact`` restates the method in plain 64-bit torch: central differences by
``torch.roll``, the 2N-storage RK3 scheme, the network by rolled copies.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1707_08900_gb300 import gbfd

TWO_PI = 2.0 * math.pi
CS = 1.0
CFL, CNU = 0.4, 0.25
ALPHA = (0.0, -5.0 / 9.0, -153.0 / 128.0)
BETA = (1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0)
TAPS = [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
PARAMS = ("W1", "b1", "W2", "b2", "W3", "b3")
WIDTHS = ((32, 5), (32, 32), (5, 32))  # output and input channels of the layers


# ------------------------------------------------------------------- the cases

def _step(name, shape, precision, steps, form="55p", entropy=1, bc="periodic", forced=False,
          adaptive=False, even=True, nu=5e-3):
    nz, ny, nx = shape
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "form": form, "entropy": entropy, "bc": bc, "forced": forced, "adaptive": adaptive,
            "even": even, "nu": nu, "steps": steps}


def listed():
    return [
        # the smallest double-precision run: ten steps of a 32^3 box, the size
        # a user checks a set-up with; launches and latency count
        _step("fp64 32^3, 10 steps", (32,) * 3, "fp64", 10),
        # the plain coarse run beside the learned one
        _step("fp32 64^3, 10 steps", (64,) * 3, "fp32", 10),
        # the headline box, four steps (one coarse step's worth)
        _step("fp32 256^3, 4 steps", (256,) * 3, "fp32", 4),
        # the large production box
        _step("fp32 512^3, 2 steps", (512,) * 3, "fp32", 2),
        # the same flow in double precision, for reference solutions
        _step("fp64 256^3, 1 step", (256,) * 3, "fp64", 1),
        # forced turbulence in the two-pass form, new draws every step
        _step("fp32 19p forced 256^3", (256,) * 3, "fp32", 3, form="19p", forced=True, nu=1.4e-4),
        # a walled channel with uneven sides and spacings, no passive scalar,
        # the time step taken from the state before every step
        _step("fp32 walls 200x136x105", (105, 136, 200), "fp32", 4, entropy=0, bc="wall",
              adaptive=True, even=False),
        # double-precision update registers over single-precision storage
        _step("fp32_acc64 256^3, 1 step", (256,) * 3, "fp32_acc64", 1),
        # a parameter study: 96 boxes of three sizes in one call
        {"name": "batch of 96 boxes", "kind": "batch", "na": 32, "ca": 32, "nb": 64, "cb": 32,
         "nc": 128, "cc": 32, "steps": 4},
        # one optimiser step on a mini-batch of eight 64^3 pairs
        {"name": "train 64^3 x 8", "kind": "train", "n": 64, "batch": 8, "nf": 5,
         "entry": "train_step"},
        # five corrected coarse steps: how the trained network is used
        {"name": "corrected 64^3, 5 steps", "kind": "corrected", "n": 64, "steps": 5},
        # training data from a fine run
        {"name": "pair 256^3 to 64^3", "kind": "pairs", "n": 256, "ratio": 4},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mult(v, m, lo):
    return max(lo, int(round(v / m)) * m)


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["batch", "train", "train", "corrected", "pairs"])
    if kind == "batch":
        sizes = [_mult(_log_uniform(rng, 16, 132), 4, 16) for _ in range(3)]
        counts = [rng.randint(1, 32) for _ in range(3)]
        return {"kind": kind, "na": sizes[0], "ca": counts[0], "nb": sizes[1], "cb": counts[1],
                "nc": sizes[2], "cc": counts[2], "steps": rng.randint(1, 4)}
    if kind == "train":
        n = int(_log_uniform(rng, 12, 97))
        most = max(1, min(8, 8 * 64 ** 3 // n ** 3))
        return {"kind": kind, "n": n, "batch": rng.randint(1, most), "nf": rng.choice([4, 5]),
                "entry": rng.choice(["train_step", "gradients"])}
    if kind == "corrected":
        return {"kind": kind, "n": _mult(_log_uniform(rng, 24, 128), 4, 24),
                "steps": rng.randint(1, 8)}
    if kind == "pairs":
        ratio = rng.choice([2, 4])
        return {"kind": kind, "n": _mult(_log_uniform(rng, 64, 288), 4 * ratio, 64), "ratio": ratio}
    precision = rng.choice(["fp32"] * 6 + ["fp64"] * 2 + ["fp32_acc64", "fp32_accff"])
    form = rng.choice(["55p", "55p", "55p", "19p"]) if precision in ("fp32", "fp64") else "55p"
    bc = rng.choice(["periodic", "periodic", "periodic", "wall"])
    forced = bc == "periodic" and rng.random() < 0.25
    # what a pass may cost, in updates: the largest listed cases
    most = {"fp32": 2 * 512 ** 3, "fp64": 256 ** 3, "fp32_acc64": 2 * 256 ** 3,
            "fp32_accff": 512 ** 3}[precision]
    if form == "19p":
        most //= 2
    base = _log_uniform(rng, 16, 0.9 * most ** (1.0 / 3.0))
    side = [base * math.exp(rng.uniform(-0.35, 0.35)) for _ in range(3)]
    whole = rng.random() < 0.5  # whole tiles, or any size that is taken
    nx = _mult(side[0], 32 if whole else 4, 32 if whole else 12)
    ny = _mult(side[1], 8 if whole else 1, 16 if whole else 9)
    nz = _mult(side[2], 1, 9)
    while nx * ny * nz > most:
        nz = nz * 3 // 4
    steps = rng.randint(1, max(1, min(10, most // (nx * ny * nz))))
    c = _step("", (nz, ny, nx), precision, steps, form=form, entropy=rng.choice([0, 1, 1]), bc=bc,
              forced=forced, adaptive=not forced and rng.random() < 0.2, even=rng.random() < 0.6,
              nu=1.4e-4 if forced else 5e-3)
    del c["name"]
    return c


# ------------------------------------------------------------------ the inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _shell_field(g, shape, k2, p=-2.0):
    """Random field with shell energy ~ k^p over 1 <= |k| <= k2 (float64)."""
    nz, ny, nx = shape
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device="cuda", dtype=torch.float64)[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device="cuda", dtype=torch.float64)[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device="cuda", dtype=torch.float64)[None, None, :]
    kk = (kx * kx + ky * ky + kz * kz).sqrt()
    amp = torch.where((kk >= 1) & (kk <= k2), kk.clamp(min=1.0) ** ((p - 2.0) / 2.0), 0.0)
    re = torch.randn(kk.shape, generator=g, device="cuda", dtype=torch.float64)
    im = torch.randn(kk.shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.fft.irfftn(torch.complex(re * amp, im * amp), s=shape, dim=(0, 1, 2))


def _flow(shape, seed, nf=5, mach=0.1, lnrho_rms=1e-3, s_rms=1e-2):
    """Decaying-turbulence state: k^-2 velocity at the given rms Mach number,
    a small density perturbation, a passive scalar."""
    g = _gen(seed)
    k2 = min(8.0, min(shape) / 4.0)
    st = torch.zeros((nf,) + tuple(shape), device="cuda", dtype=torch.float64)
    for i in range(3):
        st[1 + i] = _shell_field(g, shape, k2)
    st[1:4] *= mach * CS / st[1:4].square().sum(0).mean().sqrt()
    for f, rms in ((0, lnrho_rms), (4, s_rms)):
        if f < nf and rms > 0:
            v = _shell_field(g, shape, k2)
            v = v - v.mean()
            st[f] = v * (rms / v.square().mean().sqrt())
    return st


def _wall_flow(shape, seed, lengths, nf, amp=0.05):
    """A state between two z walls: even in z for all fields but u_z, which
    vanishes on the walls."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx)]
    z = (ax[0] * (math.pi / (nz - 1)))[:, None, None]
    y = (ax[1] * (TWO_PI / ny))[None, :, None]
    x = (ax[2] * (TWO_PI / nx))[None, None, :]
    st = torch.zeros((nf,) + tuple(shape), device="cuda", dtype=torch.float64)
    for f in range(nf):
        for _ in range(4):
            m, ky, kx = (int(v) for v in rng.integers(0, 4, 3))
            ph, a = rng.uniform(0.0, TWO_PI), rng.standard_normal() * amp
            zz = torch.sin((m + 1) * z) if f == 3 else torch.cos(m * z)
            st[f] += a * zz * torch.cos(ky * y + kx * x + ph)
    if nf > 3:
        st[3, 0] = 0.0
        st[3, -1] = 0.0
    return st


def _forcing(seed, steps, kmin=1.0, kmax=2.0):
    """Per step: an integer wave vector of the isotropic set, a phase, a unit
    vector perpendicular to it."""
    rng = np.random.default_rng(seed)
    r = range(-int(kmax), int(kmax) + 1)
    pool = np.array([(a, b, c) for a in r for b in r for c in r
                     if kmin ** 2 <= a * a + b * b + c * c <= kmax ** 2], dtype=np.int64)
    k = pool[rng.integers(0, len(pool), steps)]
    phi = rng.uniform(0.0, TWO_PI, steps)
    e = rng.standard_normal((steps, 3))
    kh = k / np.linalg.norm(k, axis=1)[:, None]
    e -= (e * kh).sum(1)[:, None] * kh
    return k, phi, e / np.linalg.norm(e, axis=1)[:, None]


F0 = 0.02  # forcing amplitude


def _lengths(case):
    if not case["even"]:
        return (TWO_PI,) * 3
    h = TWO_PI / max(case["nx"], case["ny"], case["nz"])
    nz = case["nz"] - (1 if case["bc"] == "wall" else 0)
    return (h * case["nx"], h * case["ny"], h * nz)


def _spacings(case):
    lx, ly, lz = _lengths(case)
    nz = case["nz"] - (1 if case["bc"] == "wall" else 0)
    return lx / case["nx"], ly / case["ny"], lz / nz


def _dt(st, h, nu):
    """The binding's time step rule on a state, as a plain number."""
    umax = float(st[1:4].double().square().sum(0).max().sqrt())
    d = min(h)
    dt = CFL * d / (umax + CS)
    return min(dt, CNU * d * d / nu) if nu > 0 else dt


def _step_input(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    nf = 5 if case["entropy"] else 4
    if case["bc"] == "wall":
        st = _wall_flow(shape, seed, _lengths(case), nf)
    else:
        st = _flow(shape, seed, nf)
    return st if case["precision"] == "fp64" else st.float()


def _batch_boxes(case):
    return [n for n, c in (("na", "ca"), ("nb", "cb"), ("nc", "cc")) for n in [case[n]] * case[c]]


def _batch_input(case, seed):
    rng = np.random.default_rng(seed)
    ns = _batch_boxes(case)
    nus = rng.uniform(2e-3, 1e-2, len(ns))
    machs = rng.uniform(0.05, 0.3, len(ns))
    states = [_flow((n,) * 3, 1000 * seed + i, mach=m).float()
              for i, (n, m) in enumerate(zip(ns, machs))]
    dts = [_dt(s, (TWO_PI / n,) * 3, nu) for s, n, nu in zip(states, ns, nus)]
    return ns, nus, states, dts


def _net_params(seed):
    """He-style start with the last layer scaled down, as training begins."""
    rng = np.random.default_rng(seed)
    p = {}
    for i, (o, c) in enumerate(WIDTHS):
        p["W%d" % (i + 1)] = rng.standard_normal((o, c, 3, 3, 3)) * math.sqrt(2.0 / (27 * c))
        p["b%d" % (i + 1)] = 0.01 * rng.standard_normal(o)
    p["W3"] *= 0.1
    return {k: v.astype(np.float32) for k, v in p.items()}


def _norm(xs, ts):
    dims = (0, 2, 3, 4)
    out = [xs.mean(dim=dims), xs.std(dim=dims), (ts - xs).std(dim=dims)]
    out = [v.double().cpu().numpy() for v in out]
    for v in out[1:]:
        v[v < 1e-12] = 1.0
    return [v.astype(np.float32) for v in out]


def _train_input(case, seed):
    """Coarse states and the targets beside them: a residual with the shape of
    a truncation error (smaller scales, a small fraction of the state)."""
    n = case["n"]
    xs, ts = [], []
    for b in range(case["batch"]):
        x = _flow((n,) * 3, 100 * seed + b, mach=0.2)
        d = _flow((n,) * 3, 100 * seed + 50 + b, mach=0.002, lnrho_rms=1e-5, s_rms=1e-4)
        xs.append(x.float())
        ts.append((x + d).float())
    xs, ts = torch.stack(xs), torch.stack(ts)
    return xs, ts, _net_params(seed), _norm(xs, ts)


LR = 1e-5  # late in a decaying schedule


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        st = _step_input(case, seed)
        s = gbfd.Solver((case["nz"], case["ny"], case["nx"]), lengths=_lengths(case), cs=CS,
                        nu=case["nu"], precision=case["precision"], form=case["form"],
                        entropy_mode=case["entropy"], bc_z=case["bc"])
        return {"case": case, "solver": s, "in": st, "out": torch.empty_like(st),
                "dt": _dt(st, _spacings(case), case["nu"]),
                "forcing": _forcing(seed, case["steps"]) if case["forced"] else None}
    if kind == "batch":
        ns, nus, states, dts = _batch_input(case, seed)
        b = gbfd.Batch(ns, [TWO_PI] * len(ns), nus, cs=CS)
        out = torch.empty(sum(s.numel() for s in states), device="cuda", dtype=torch.float32)
        return {"case": case, "batch": b, "in": states, "out": out, "dt": dts,
                "views": list(out.split([s.numel() for s in states]))}
    if kind == "train":
        xs, ts, p, norm = _train_input(case, seed)
        net = gbfd.CNN(case["n"], batch=case["batch"])
        net.set_params(p)
        net.set_norm(*norm)
        return {"case": case, "net": net, "xs": xs, "ts": ts}
    if kind == "corrected":
        n = case["n"]
        tc = {"n": n, "batch": 1}
        xs, _, p, norm = _train_input(tc, seed)
        s = gbfd.Solver((n,) * 3, precision="fp32", nu=5e-3)
        net = gbfd.CNN(n, batch=1)
        net.set_params(p)
        net.set_norm(*norm)
        return {"case": case, "solver": s, "net": net, "in": xs[0], "out": torch.empty_like(xs[0]),
                "dt": _dt(xs[0], (TWO_PI / n,) * 3, 5e-3)}
    n, r = case["n"], case["ratio"]
    st = _flow((n,) * 3, seed, mach=0.2).float()
    fine = gbfd.Solver((n,) * 3, precision="fp32", nu=5e-3)
    coarse = gbfd.Solver((n // r,) * 3, precision="fp32", nu=5e-3)
    return {"case": case, "fine": fine, "coarse": coarse, "in": st,
            "dt": _dt(st, (TWO_PI / n,) * 3, 5e-3)}


# -------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        s = state["solver"]
        s.set_state(state["in"])
        if case["forced"]:
            s.rk3_step_forced(state["dt"], F0, *state["forcing"])
        elif case["adaptive"]:
            for _ in range(case["steps"]):
                s.rk3_step(s.cfl_dt(CFL, CNU), 1)
        else:
            s.rk3_step(state["dt"], case["steps"])
        return s.get_state(out=state["out"])
    if kind == "batch":
        b = state["batch"]
        for i, st in enumerate(state["in"]):
            b.set_state(i, st)
        b.step(state["dt"], case["steps"])
        get = gbfd.load().gbfd_batch_get_state  # into device memory
        for i, v in enumerate(state["views"]):
            if get(b.b, i, ctypes.c_void_p(v.data_ptr()), 1, 0) != gbfd.GBFD_OK:
                raise gbfd.GbfdError(3, "batch get_state")
        return state["out"]
    if kind == "train":
        net = state["net"]
        if case["entry"] == "gradients":
            g, loss = net.gradients(state["xs"], state["ts"], nf=case["nf"])
            return {"gradients": g, "loss": loss}
        loss = net.train_step(state["xs"], state["ts"], LR, nf=case["nf"])
        return {"params": net.get_params(), "loss": loss}
    if kind == "corrected":
        s = state["solver"]
        s.set_state(state["in"])
        state["net"].step_corrected(s, state["dt"], case["steps"])
        return s.get_state(out=state["out"])
    fine, coarse, r = state["fine"], state["coarse"], case["ratio"]
    fine.set_state(state["in"])
    c = gbfd.box_filter(fine, r)
    coarse.set_state(c)
    coarse.rk3_step(r * state["dt"], 1)
    x = torch.empty_like(c)
    coarse.get_state(out=x)
    fine.rk3_step(state["dt"], r)
    return {"x": x, "t": gbfd.box_filter(fine, r)}


# ------------------------------------------------- what a pass cannot do without

# floating-point operations of one point and substep, counted from the
# equations (central differences, right-hand sides, update; FMA = 2)
STEP_FLOPS = {("55p", 1): 418, ("55p", 0): 376, ("19p", 1): 340, ("19p", 0): 298}
NET_MACS = 27 * sum(o * c for o, c in WIDTHS)  # one forward pass, per point


def work(case):
    """States and parameters in and out once; the arithmetic of every step."""
    kind = case["kind"]
    if kind == "step":
        pts = case["nx"] * case["ny"] * case["nz"]
        nf, w = 4 + case["entropy"], 8 if case["precision"] == "fp64" else 4
        return {"bytes": 2 * nf * w * pts,
                "flops": 3 * STEP_FLOPS[case["form"], case["entropy"]] * pts * case["steps"]}
    if kind == "batch":
        pts = sum(n ** 3 for n in _batch_boxes(case))
        return {"bytes": 40 * pts, "flops": 3 * STEP_FLOPS["55p", 1] * pts * case["steps"]}
    if kind == "train":
        pts = case["n"] ** 3 * case["batch"]
        # forward, weight gradients, and the input gradients of layers 2 and 3
        macs = 2 * NET_MACS + 27 * sum(o * c for o, c in WIDTHS[1:])
        return {"bytes": 2 * case["nf"] * 4 * pts, "flops": 2 * macs * pts}
    if kind == "corrected":
        pts = case["n"] ** 3
        return {"bytes": 40 * pts,
                "flops": (3 * STEP_FLOPS["55p", 1] + 2 * NET_MACS) * pts * case["steps"]}
    pts, cpts = case["n"] ** 3, (case["n"] // case["ratio"]) ** 3
    return {"bytes": 20 * pts + 40 * cpts,
            "flops": 3 * STEP_FLOPS["55p", 1] * (case["ratio"] * pts + cpts)}


# --------------------------------------------------- the same in plain 64 bits

def _d1(f, ax, h):
    r = lambda k: torch.roll(f, -k, ax)
    return (45.0 * (r(1) - r(-1)) - 9.0 * (r(2) - r(-2)) + (r(3) - r(-3))) / (60.0 * h)


def _d2(f, ax, h):
    r = lambda k: torch.roll(f, -k, ax)
    return (270.0 * (r(1) + r(-1)) - 27.0 * (r(2) + r(-2)) + 2.0 * (r(3) + r(-3)) -
            490.0 * f) / (180.0 * h * h)


def _dmix(f, a, b, ha, hb):
    r = lambda i, j: torch.roll(f, (-i, -j), (a, b))
    acc = 0.0
    for k, c in ((1, 270.0), (2, -27.0), (3, 2.0)):
        acc = acc + c * (r(k, k) - r(-k, k) + r(-k, -k) - r(k, -k))
    return acc / (720.0 * ha * hb)


def _rhs(st, h, nu, form, force):
    """Right-hand sides of the continuity, momentum and passive-scalar
    equations; axes of a field are (z, y, x), components (x, y, z)."""
    ax, u = (2, 1, 0), [st[1], st[2], st[3]]
    D = lambda f, a: _d1(f, ax[a], h[a])
    g = [[D(u[i], a) for a in range(3)] for i in range(3)]
    div = g[0][0] + g[1][1] + g[2][2]
    gl = [D(st[0], a) for a in range(3)]
    adv = lambda gr: u[0] * gr[0] + u[1] * gr[1] + u[2] * gr[2]
    out = torch.empty_like(st)
    out[0] = -adv(gl) - div
    for i in range(3):
        lap, gd = 0.0, 0.0
        for a in range(3):
            d2 = _d2(u[i], ax[a], h[a])
            lap = lap + d2
            if a == i:
                same = d2
        if form == "19p":
            gd = D(div, i)
        else:
            gd = same
            for j in range(3):
                if j != i:
                    gd = gd + _dmix(u[j], ax[i], ax[j], h[i], h[j])
        sgl = -(2.0 / 3.0) * div * gl[i]
        for j in range(3):
            sgl = sgl + (g[i][j] + g[j][i]) * gl[j]
        out[1 + i] = -adv(g[i]) - CS * CS * gl[i] + nu * (lap + gd / 3.0 + sgl)
        if force is not None:
            out[1 + i] += force[i]
    if st.shape[0] == 5:
        out[4] = -adv([D(st[4], a) for a in range(3)])
    return out


def _rk3(st, dt, h, nu, form="55p", force=None):
    w = torch.zeros_like(st)
    for a, b in zip(ALPHA, BETA):
        w = a * w + dt * _rhs(st, h, nu, form, force)
        st = st + b * w
    return st


def _force(shape, lengths, dt, k, phi, e):
    kp = np.array([TWO_PI * ki / li for ki, li in zip(k, lengths)])
    kk, ke = float(kp @ kp), float(kp @ e)
    amp = F0 * CS * math.sqrt(math.sqrt(kk) * CS / dt) * np.cross(kp, e) / math.sqrt(kk - ke * ke)
    ph = 0.0
    for a, n in enumerate(reversed(shape)):
        i = torch.arange(n, device="cuda", dtype=torch.float64) * (TWO_PI * float(k[a]) / n)
        ph = ph + i.reshape([-1 if d == 2 - a else 1 for d in range(3)])
    c = torch.cos(ph + float(phi))
    return [float(v) * c for v in amp]


def _exact_step(case, seed):
    st = _step_input(case, seed)
    h, nu = _spacings(case), case["nu"]
    dt = _dt(st, h, nu)
    st = st.double()
    nz, wall = case["nz"], case["bc"] == "wall"
    if wall:  # the periodic run of the mirror-extended state
        ext = torch.cat([st, st[:, 1:nz - 1].flip(1)], 1)
        ext[3, nz:] *= -1.0
        st = ext
    fr = _forcing(seed, case["steps"]) if case["forced"] else None
    for n in range(case["steps"]):
        if case["adaptive"]:
            dt = _dt(st, h, nu)
        force = None
        if fr:
            force = _force(st.shape[1:], _lengths(case), dt, fr[0][n], fr[1][n], fr[2][n])
        st = _rk3(st, dt, h, nu, case["form"], force)
    return st[:, :nz].contiguous() if wall else st


def _conv(x, W, b):
    y = b[:, None].expand(-1, x[0].numel())
    for i, t in enumerate(TAPS):
        xs = torch.roll(x, [-v for v in t], (1, 2, 3)).reshape(x.shape[0], -1)
        y = y + W[:, :, t[0] + 1, t[1] + 1, t[2] + 1] @ xs
    return y.reshape((-1,) + tuple(x.shape[1:]))


def _net(x, p):
    gelu = torch.nn.functional.gelu
    a = gelu(_conv(x, p["W1"], p["b1"]))
    a = gelu(_conv(a, p["W2"], p["b2"]))
    return _conv(a, p["W3"], p["b3"])


def _params64(p, grad=False):
    return {k: torch.tensor(p[k], dtype=torch.float64, device="cuda", requires_grad=grad)
            for k in PARAMS}


def _norm64(norm):
    return [torch.tensor(v, dtype=torch.float64, device="cuda")[:, None, None, None] for v in norm]


def _exact_train(case, seed):
    xs, ts, p0, norm = _train_input(case, seed)
    mean, std, sout = _norm64(norm)
    p = _params64(p0, True)
    loss = 0.0
    for x, t in zip(xs.double(), ts.double()):
        x0 = (x - mean) / std
        r = (t - x) / sout
        if case["nf"] == 4:
            x0[4], r[4] = 0.0, 0.0
        part = (_net(x0, p) - r).square().sum() / xs.numel()
        part.backward()
        loss += float(part)
    flat = lambda f: np.concatenate([f(p[k]).detach().cpu().numpy().ravel() for k in PARAMS])
    g = flat(lambda v: v.grad)
    if case["entry"] == "gradients":
        return {"gradients": g, "loss": loss}
    # the first step of Adam: both moments' bias corrections cancel
    return {"params": flat(lambda v: v) - LR * g / (np.abs(g) + 1e-8), "loss": loss}


def _exact_corrected(case, seed):
    n = case["n"]
    xs, _, p, norm = _train_input({"n": n, "batch": 1}, seed)
    mean, std, sout = _norm64(norm)
    p = _params64(p)
    h = (TWO_PI / n,) * 3
    dt, st = _dt(xs[0], h, 5e-3), xs[0].double()
    with torch.no_grad():
        for _ in range(case["steps"]):
            st = _rk3(st, dt, h, 5e-3)
            st = st + sout * _net((st - mean) / std, p)
    return st


def _filter(st, r):
    """Centred box filter on every r-th point, weights (1/2, 1, .., 1, 1/2) / r."""
    for ax in (1, 2, 3):
        acc = 0.0
        for o in range(-(r // 2), r // 2 + 1):
            w = (0.5 if abs(o) == r // 2 else 1.0) / r
            acc = acc + w * torch.roll(st, -o, ax)
        st = acc.index_select(ax, torch.arange(0, st.shape[ax], r, device="cuda"))
    return st


def _exact_pairs(case, seed):
    n, r = case["n"], case["ratio"]
    st = _flow((n,) * 3, seed, mach=0.2).float()
    dt, st = _dt(st, (TWO_PI / n,) * 3, 5e-3), st.double()
    x = _rk3(_filter(st, r), r * dt, (r * TWO_PI / n,) * 3, 5e-3)
    for _ in range(r):
        st = _rk3(st, dt, (TWO_PI / n,) * 3, 5e-3)
    return {"x": x, "t": _filter(st, r)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ns, nus, states, dts = _batch_input(case, seed)
        out = []
        for n, nu, st, dt in zip(ns, nus, states, dts):
            st = st.double()
            for _ in range(case["steps"]):
                st = _rk3(st, dt, (TWO_PI / n,) * 3, nu)
            out.append(st.reshape(-1))
        return torch.cat(out)
    return {"step": _exact_step, "train": _exact_train, "corrected": _exact_corrected,
            "pairs": _exact_pairs}[kind](case, seed)
