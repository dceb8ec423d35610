"""The work this framework does for its users, as timed cases: time stepping in every
storage and arithmetic form, batches of uneven lattices, the adjoint and a whole gradient,
the observables, and a run from host memory and back.

States are Rayleigh-Taylor flows in motion (a hot layer under a cold one between thermal
walls, hydrostatic density, a few vortices of a few hundredths of the sound speed, and
populations a little off equilibrium), as a run holds them at any time after its start.
"""
import functools
import math

import numpy as np
import torch

# ------------------------------------------------------------------------------ the model
# D2Q37: 0 = rest, 18 representatives, then their opposites in the same order.
_REPS = [(1, 0), (0, 1), (1, 1), (1, -1), (2, 0), (0, 2), (2, 1), (1, 2), (2, -1), (1, -2), (2, 2), (2, -2),
         (3, 0), (0, 3), (3, 1), (1, 3), (3, -1), (1, -3)]
_V = [(0, 0)] + _REPS + [(-a, -b) for a, b in _REPS]
_C = 1.196979770393074358972388463853275434844
_W2 = {0: 0.2331506691323525022865067040668499509961, 1: 0.107306091542219002412464287183139935851,
       2: 0.05766785988879488203006921539333941471077, 4: 0.01420821615845075026469894234413445497343,
       5: 0.005353049000513775232731501662188493535094, 8: 0.001011937592673575475410908506639114714702,
       9: 0.0002453010277577173454659166432678444638839, 10: 0.0002834142529941982174005252941948802334792}
_W = [_W2[a * a + b * b] for a, b in _V]
_Q = 37
_G = 1e-4                       # gravity, in -y
_TB, _TT = 1.15, 0.85           # wall temperatures
_FORMS = {"fp64": 0, "fp32": 1, "fp64fix": 2, "fp32cons": 3}


def _f32(case):
    return case["form"] in ("fp32", "fp32cons")


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # a small lattice stepped a few times between two looks at it (parameter studies,
        # parity checks): latency and launches
        {"name": "run_small", "kind": "run", "form": "fp64", "lx": 64, "ly": 128, "steps": 10, "tau": 0.8},
        # one call of one step on a lattice of odd size, its result in the other buffer
        {"name": "step_odd", "kind": "run", "form": "fp64", "lx": 501, "ly": 1003, "steps": 1, "tau": 0.62},
        # the flagship: the default float64 form on the 4096 x 8192 lattice
        {"name": "run_large", "kind": "run", "form": "fp64", "lx": 4096, "ly": 8192, "steps": 2, "tau": 0.8},
        # the float64 form with the fixed-point relaxation on the paper's 2160 x 8192 lattice
        {"name": "run_fix", "kind": "run", "form": "fp64fix", "lx": 2160, "ly": 8192, "steps": 2, "tau": 0.8},
        # float32 storage, shifted: long runs of big lattices at half the memory
        {"name": "run_fp32", "kind": "run", "form": "fp32", "lx": 2048, "ly": 8192, "steps": 4, "tau": 0.8},
        # float32 storage with conserved moments, an ordinary and odd size
        {"name": "run_fp32cons", "kind": "run", "form": "fp32cons", "lx": 1021, "ly": 2050, "steps": 4, "tau": 1.1},
        # a parameter sweep: uneven lattices, each with its own tau, stepped together
        {"name": "batch_fp64", "kind": "batch", "form": "fp64", "n": 48, "lo": 128, "hi": 512, "steps": 2, "tau": 0.8},
        # many small lattices in float32, where launches would dominate
        {"name": "batch_fp32", "kind": "batch", "form": "fp32", "n": 256, "lo": 32, "hi": 128, "steps": 10, "tau": 0.8},
        # one adjoint step, the inner loop of every gradient
        {"name": "adjoint", "kind": "adjoint", "form": "fp64", "lx": 512, "ly": 1024, "steps": 1, "tau": 0.8},
        # a whole gradient of the final kinetic energy: forward run, checkpoints, backward
        {"name": "gradient", "kind": "gradient", "form": "fp64", "lx": 256, "ly": 512, "steps": 50, "tau": 0.8},
        # what a run reports every so often: the four fields and the total kinetic energy
        {"name": "observe", "kind": "observe", "form": "fp64", "lx": 2048, "ly": 4096, "steps": 0, "tau": 0.8},
        # from host fields to host fields: copies, initial state, steps, moments
        {"name": "host", "kind": "host", "form": "fp64", "lx": 1024, "ly": 2048, "steps": 20, "tau": 0.8},
    ]


def _size(rng, lo, hi):
    """Spread over the logarithm of [lo, hi]; about half of them odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, n | 1) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "batch", "adjoint", "gradient", "observe", "host"])
    form = "fp64"
    if kind == "run":
        form = rng.choice(["fp64", "fp64", "fp64fix", "fp32", "fp32cons"])
    elif kind == "batch":
        form = rng.choice(["fp64", "fp64fix", "fp32", "fp32cons"])
    elif kind == "host":
        form = rng.choice(["fp64", "fp64fix", "fp32cons"])
    case = {"kind": kind, "form": form, "tau": rng.uniform(0.6, 1.2)}
    if kind == "batch":
        lo = _size(rng, 32, 128)
        hi = _size(rng, lo + 16, 512)
        n = int(rng.uniform(8, 256))
        case.update(n=max(4, min(n, int(1.2e7 / (hi * hi)))), lo=lo, hi=hi, steps=rng.choice([2, 4, 10]))
        return case
    top = {"run": (4096, 8192), "adjoint": (1024, 2048), "gradient": (320, 640), "observe": (2048, 4096),
           "host": (1024, 2048)}[kind]
    case["lx"], case["ly"] = _size(rng, 24, top[0]), _size(rng, 40, top[1])
    sites = case["lx"] * case["ly"]
    steps = {"run": [1, 2, 4, 10, 20], "adjoint": [1], "gradient": [10, 24, 50], "observe": [0],
             "host": [1, 4, 20]}[kind]
    steps = [s for s in steps if s * sites <= 4.5e7] or [1]
    case["steps"] = rng.choice(steps)
    return case


def work(case):
    """Every time step reads and writes a state of 37 values per site and takes 512 operations
    per site (138 additions, 97 products, 138 multiply-adds counted twice, one division); an
    adjoint step reads two states and writes one, and takes about twice the operations."""
    val = 4 if _f32(case) else 8
    kind = case["kind"]
    sites = sum(a * b for a, b, _ in _lattices(case)) if kind == "batch" else case["lx"] * case["ly"]
    step_b, step_f = 2 * _Q * val * sites, 512 * sites
    n = case["steps"]
    if kind in ("run", "batch"):
        return {"bytes": n * step_b, "flops": n * step_f}
    if kind == "adjoint":
        return {"bytes": 3 * _Q * 8 * sites, "flops": 1024 * sites}
    if kind == "gradient":
        # the forward steps and the adjoint steps; the initial state, the energy's gradient
        # and the gradients of the four fields
        return {"bytes": n * (2 + 3) * _Q * 8 * sites + 2 * _Q * 8 * sites + (4 + _Q + 8) * 8 * sites,
                "flops": n * (512 + 1024) * sites}
    if kind == "observe":
        return {"bytes": (_Q * val + 4 * 8) * sites, "flops": 130 * sites}
    return {"bytes": n * step_b + (4 * 8 + _Q * val) * 2 * sites, "flops": (n + 1) * step_f}


# ------------------------------------------------------------------------------ inputs
def _equilibrium(rho, ux, uy, T, i):
    """Population i of the fourth-order Hermite equilibrium."""
    a, b = _V[i]
    q, t = _C * _C * (a * a + b * b), T - 1.0
    s = (_C * a) * ux + (_C * b) * uy
    U = ux * ux + uy * uy
    c0 = 1.0 - 0.5 * U + 0.5 * (q - 2.0) * t + 0.125 * U * U + 0.25 * (4.0 - q) * t * U \
        + 0.125 * (q * q - 8.0 * q + 8.0) * t * t
    c1 = 1.0 - 0.5 * U + 0.5 * (q - 4.0) * t
    c2 = 0.5 - 0.25 * U + 0.25 * (q - 6.0) * t
    return _W[i] * rho * (c0 + s * (c1 + s * (c2 + s * (1.0 / 6.0 + s * (1.0 / 24.0)))))


def _rng(seed, *more):
    return np.random.Generator(np.random.Philox([int(seed), *[int(m) for m in more]]))


def _fields(lx, ly, seed, still=False):
    """(rho, ux, uy, T) on the GPU: two layers with a wavy interface, hydrostatic pressure, and
    four vortices (no flow where `still`)."""
    r = _rng(seed, lx, ly)
    x = torch.arange(lx, dtype=torch.float64, device="cuda")[:, None]
    y = torch.arange(ly, dtype=torch.float64, device="cuda")[None, :]
    yc = torch.full_like(x, ly / 2.0)
    for k in range(1, 9):
        yc = yc + float(r.uniform(-1, 1)) * 0.003 * ly * torch.cos(2 * math.pi * k * x / lx + float(r.uniform(0, 2 * math.pi)))
    T = _TB + (_TT - _TB) * 0.5 * (1.0 + torch.tanh((y - yc) / 3.0))
    rho = torch.exp(-_G * (y - ly / 2.0) / T) / T
    ux, uy = torch.zeros_like(T), torch.zeros_like(T)
    if not still:
        for _ in range(4):
            kx, ky = int(r.integers(1, 4)), int(r.integers(1, 4))
            px, py, amp = float(r.uniform(0, 6.28)), float(r.uniform(0, 6.28)), float(r.uniform(0.002, 0.012))
            ax, ay = 2 * math.pi * kx / lx * x + px, 2 * math.pi * ky / ly * y + py
            ux += amp * torch.sin(ax) * torch.cos(ay)
            uy -= amp * torch.cos(ax) * torch.sin(ay)
    return rho, ux, uy, T


def _populations(lx, ly, seed):
    """[37, lx, ly] populations of a flow in motion, in float64, one plane after the other."""
    f = torch.empty((_Q, lx, ly), dtype=torch.float64, device="cuda")
    rho, ux, uy, T = _fields(lx, ly, seed)
    r = _rng(seed, lx, ly, 37)
    x = torch.arange(lx, dtype=torch.float64, device="cuda")[:, None]
    y = torch.arange(ly, dtype=torch.float64, device="cuda")[None, :]
    for i in range(_Q):
        ph = r.uniform(0, 2 * math.pi, 2)
        off = torch.cos(4 * math.pi * x / lx + ph[0]) * torch.cos(6 * math.pi * y / ly + ph[1])
        f[i] = _equilibrium(rho, ux, uy, T, i) * (1.0 + 2e-3 * off)
    return f


def _stored(f, case, out):
    """Writes populations into a state buffer of the case's form (padding: 0)."""
    ly = f.shape[2]
    out.zero_()
    for i in range(_Q):
        out[i, :, :ly] = f[i] - _W[i] if _f32(case) else f[i]
    return out


def _unstored(g, case):
    """The populations that a float32 or float64 state holds, in float64."""
    if not _f32(case):
        return g
    return g.double() + torch.tensor(_W, dtype=torch.float64, device="cuda")[:, None, None]


@functools.lru_cache(maxsize=8)
def _batch_of(n, lo, hi, tau):
    r = _rng(n, lo, hi)
    lx = np.exp(r.uniform(math.log(lo), math.log(hi), n)).astype(int)
    return [(int(a), int(2 * a) | int(r.integers(0, 2)), float(tau + r.uniform(-0.05, 0.2))) for a in lx]


def _lattices(case):
    return _batch_of(case["n"], case["lo"], case["hi"], case["tau"])


def _params(case, lx=None, ly=None, tau=None):
    from paper_1703_04594_gb300 import lbm
    return lbm.Params(lx or case["lx"], ly or case["ly"], tau=tau or case["tau"], gy=-_G, t_bottom=_TB, t_top=_TT,
                      precision=_FORMS[case["form"]])


def _pitch(ly):
    return (ly + 31) // 32 * 32


def _lam(case, seed):
    """An adjoint state of smooth values, the size that a sum over sites gives."""
    r = _rng(seed, 3)
    lx, ly = case["lx"], case["ly"]
    x = torch.arange(lx, dtype=torch.float64, device="cuda")[:, None]
    y = torch.arange(ly, dtype=torch.float64, device="cuda")[None, :]
    lam = torch.empty((_Q, lx, ly), dtype=torch.float64, device="cuda")
    for i in range(_Q):
        a, b, p, q = r.uniform(0.01, 0.05), r.uniform(-0.05, 0.05), r.uniform(0, 6.28), r.uniform(0, 6.28)
        lam[i] = b + a * torch.sin(2 * math.pi * x / lx + p) * torch.cos(4 * math.pi * y / ly + q)
    return lam


# ------------------------------------------------------------------------------ the passes
def prepare(case, seed):
    from paper_1703_04594_gb300 import lbm
    kind, s = case["kind"], {"case": case}
    if kind == "batch":
        dt = torch.float32 if _f32(case) else torch.float64
        sizes = _lattices(case)
        total = sum(_Q * a * _pitch(b) for a, b, _ in sizes)
        s["a"], s["b"] = torch.zeros(total, dtype=dt, device="cuda"), torch.zeros(total, dtype=dt, device="cuda")
        ps, fa, fb, at = [], [], [], 0
        for j, (a, b, tau) in enumerate(sizes):
            n = _Q * a * _pitch(b)
            fa.append(s["a"][at:at + n].view(_Q, a, _pitch(b)))
            fb.append(s["b"][at:at + n].view(_Q, a, _pitch(b)))
            ps.append(_params(case, a, b, tau))
            _stored(_populations(a, b, seed * 1000 + j), case, fa[-1])
            at += n
        s["batch"] = lbm.Batch(ps, fa, fb)
        return s
    p = s["p"] = _params(case)
    if kind == "host":
        s["in"] = [t.cpu().pin_memory() for t in _fields(p.lx, p.ly, seed)]
        s["out"] = [torch.empty_like(t).pin_memory() for t in s["in"]]
        s["a"], s["b"] = lbm.empty_state(p), lbm.empty_state(p)
        s["fields"] = torch.empty(4 * p.lx * p.ly, dtype=torch.float64, device="cuda")
        return s
    if kind == "gradient":
        s["fields"] = [t.requires_grad_() for t in _fields(p.lx, p.ly, seed)]
        s["tau"] = torch.tensor(case["tau"], dtype=torch.float64, requires_grad=True)
        return s
    s["a"] = _stored(_populations(p.lx, p.ly, seed), case, lbm.empty_state(p))
    if kind == "run":
        s["b"] = torch.zeros_like(s["a"])
    elif kind == "adjoint":
        s["next"] = _stored(_lam(case, seed), case, lbm.empty_state(p))
        s["lam"] = torch.zeros_like(s["next"])
        s["dtau"] = torch.zeros((), dtype=torch.float64, device="cuda")
        s["work"] = lbm.adjoint_work(p)
    else:
        s["out"] = [torch.empty((p.lx, p.ly), dtype=torch.float64, device="cuda") for _ in range(4)]
        s["e"] = torch.empty((), dtype=torch.float64, device="cuda")
        s["scratch"] = torch.empty(lbm.reduce_scratch_bytes(p) // 8, dtype=torch.float64, device="cuda")
    return s


def run(s):
    from paper_1703_04594_gb300 import lbm
    case, kind = s["case"], s["case"]["kind"]
    if kind == "run":
        if case["steps"] == 1:
            return lbm.step(s["p"], s["a"], s["b"])
        return lbm.run(s["p"], s["a"], s["b"], case["steps"])
    if kind == "batch":
        s["batch"].run(case["steps"])  # an even number of steps: the states are back in a
        return s["a"]
    if kind == "adjoint":
        s["dtau"].zero_()
        lbm.adjoint_step(s["p"], s["a"], s["next"], s["lam"], s["dtau"], s["work"])
        return [s["lam"], s["dtau"]]
    if kind == "gradient":
        from paper_1703_04594_gb300 import adjoint
        e = adjoint.kinetic_energy_after(*s["fields"], s["tau"], s["p"], case["steps"])
        return [e.detach(), *torch.autograd.grad(e, [*s["fields"], s["tau"]])]
    if kind == "observe":
        fields = lbm.moments(s["p"], s["a"], out=s["out"])
        return [*fields, lbm.kinetic_energy(s["p"], s["a"], out=s["e"], scratch=s["scratch"])]
    return lbm.simulate_host(s["p"], s["in"], case["steps"], s["out"], s["a"], s["b"], s["fields"])


# ------------------------------------------------------------------------------ in 64 bits
def _moments(f):
    rho = f.sum(0)
    jx = sum(a * f[i] for i, (a, _) in enumerate(_V) if a)
    jy = sum(b * f[i] for i, (_, b) in enumerate(_V) if b)
    e = sum((a * a + b * b) * f[i] for i, (a, b) in enumerate(_V) if a or b)
    ux, uy = _C * jx / rho, _C * jy / rho
    return rho, ux, uy, (_C * _C * e / rho - (ux * ux + uy * uy)) / 2.0


def _step_columns(f, tau, cols):
    """Columns `cols` of the state after one step of f [37, lx, ly]: pull, walls, BGK collision."""
    lx, ly = f.shape[1:]
    n = cols.numel()
    one = torch.ones((), dtype=torch.float64, device=f.device)
    rows = []
    for i, (a, b) in enumerate(_V):
        xs = (cols - a) % lx
        src = f[i][xs]
        if b > 0:
            wall = f[:, :, 0][:, xs].sum(0) * _equilibrium(one, 0 * one, 0 * one, _TB * one, i)
            src = torch.cat([wall[:, None].expand(n, b), src[:, :ly - b]], 1)
        elif b < 0:
            wall = f[:, :, ly - 1][:, xs].sum(0) * _equilibrium(one, 0 * one, 0 * one, _TT * one, i)
            src = torch.cat([src[:, -b:], wall[:, None].expand(n, -b)], 1)
        rows.append(src)
    ft = torch.stack(rows)
    rho, ux, uy, T = _moments(ft)
    uy = uy - tau * _G
    T = T + tau * (1.0 - tau) * (_G * _G) / 2.0
    return torch.stack([ft[i] + (_equilibrium(rho, ux, uy, T, i) - ft[i]) / tau for i in range(_Q)])


def _step(f, tau):
    lx, ly = f.shape[1:]
    cols = torch.arange(lx, device=f.device)
    width = max(1, int(4e6 // ly))
    if lx <= width:
        return _step_columns(f, tau, cols)
    out = torch.empty_like(f)
    for at in range(0, lx, width):
        out[:, at:at + width] = _step_columns(f, tau, cols[at:at + width])
    return out


def _advance(case, seed, lx, ly, tau):
    """The state a run starts from, as its form stores it, advanced in 64 bits; padded."""
    f = _populations(lx, ly, seed)
    if _f32(case):
        for i in range(_Q):
            f[i] = (f[i] - _W[i]).float().double() + _W[i]
    for _ in range(case["steps"]):
        f = _step(f, tau)
    out = torch.zeros((_Q, lx, _pitch(ly)), dtype=torch.float64, device="cuda")
    for i in range(_Q):
        out[i, :, :ly] = f[i] - _W[i] if _f32(case) else f[i]
    return out


def exact(case, seed):
    kind, tau = case["kind"], case["tau"]
    with torch.no_grad():
        if kind == "run":
            return _advance(case, seed, case["lx"], case["ly"], tau)
        if kind == "batch":
            return torch.cat([_advance(case, seed * 1000 + j, a, b, t).reshape(-1)
                              for j, (a, b, t) in enumerate(_lattices(case))])
        if kind == "observe":
            rho, ux, uy, T = _moments(_populations(case["lx"], case["ly"], seed))
            return [rho, ux, uy, T, (0.5 * rho * (ux * ux + uy * uy)).sum()]
        if kind == "host":
            fields = _fields(case["lx"], case["ly"], seed)
            f = torch.stack([_equilibrium(*fields, i) for i in range(_Q)])
            if _f32(case):
                return None  # the state is rounded to 32 bits at every step
            for _ in range(case["steps"]):
                f = _step(f, tau)
            return [t.cpu() for t in _moments(f)]
    if kind == "adjoint":
        f = _populations(case["lx"], case["ly"], seed).requires_grad_()
        t = torch.tensor(tau, dtype=torch.float64, device="cuda", requires_grad=True)
        out = _step_columns(f, t, torch.arange(case["lx"], device="cuda"))
        gf, gt = torch.autograd.grad(out, [f, t], grad_outputs=_lam(case, seed))
        lam = torch.zeros((_Q, case["lx"], _pitch(case["ly"])), dtype=torch.float64, device="cuda")
        lam[:, :, :case["ly"]] = gf
        return [lam, gt]
    # the gradient, one step at a time from the last: the states are kept, the graphs are not
    fields = [t.requires_grad_() for t in _fields(case["lx"], case["ly"], seed)]
    first = torch.stack([_equilibrium(*fields, i) for i in range(_Q)])
    cols = torch.arange(case["lx"], device="cuda")
    states = [first.detach()]
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(_step_columns(states[-1], tau, cols))
    last = states.pop().requires_grad_()
    rho, ux, uy, _ = _moments(last)
    e = (0.5 * rho * (ux * ux + uy * uy)).sum()
    (lam,) = torch.autograd.grad(e, [last])
    gtau = torch.zeros((), dtype=torch.float64, device="cuda")
    while states:
        f = states.pop().requires_grad_()
        t = torch.tensor(tau, dtype=torch.float64, device="cuda", requires_grad=True)
        lam, gt = torch.autograd.grad(_step_columns(f, t, cols), [f, t], grad_outputs=lam)
        gtau = gtau + gt
    return [e.detach(), *torch.autograd.grad(first, fields, grad_outputs=lam), gtau.cpu()]
