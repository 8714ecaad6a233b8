"""Performance cases of the droplet solver and of its proposal network.

Every case goes through the calls a user's program makes: ``lbfe.Solver``
(init, step, column blocks, observables), ``decomp.run`` and ``mlp.MLP``
(forward, fit).  Solvers keep the launch shape of a new handle.  A stepping
pass advances the lattice by ``steps`` time steps and takes the whole stored
state (populations, conformation and, in the reduced forms, the offset
densities) into a device buffer, as a program does that keeps snapshots.
The state is larger than the caches at the sizes of the paper's set-up.
"""
import math
import random

import numpy as np
import torch

from paper_1411_2181_gb300 import configs, decomp, lbfe, study
from paper_1411_2181_gb300 import mlp as proposal

Q = 19
CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0)
CY = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1)
WT = (1 / 3,) + (1 / 18,) * 6 + (1 / 36,) * 12
FP32, FP16, BF16 = 0, 1, 2
SYM = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}


# ---------------------------------------------------------------- the cases
def _box(name, kind, shape, R, Ca, De, lam, L2, phase, Uw, precision, advection, steps, parts=1):
    return {"name": name, "kind": kind, "Lx": shape[0], "Ly": shape[1], "Lz": shape[2], "R": R, "Ca": Ca, "De": De,
            "lam": lam, "L2": L2, "phase": phase, "Uw": Uw, "precision": precision, "advection": advection,
            "steps": steps, "parts": parts}


def listed():
    return [
        # smallest lattice: the 32^3 parity box, bound by launches and latency
        _box("box_32_fp32", "step", (32, 32, 32), 8.0, 0.1, 1.0, 1.0, 100.0, 1, 0.005, FP32, 0, 40),
        # the benchmark lattice: a matrix-viscoelastic droplet between moving walls
        _box("matrix_192_fp32", "step", (192, 96, 80), 16.0, 0.2, 1.0, 1.0, 100.0, 2, 0.02, FP32, 0, 20),
        # the strongly confined droplet-viscoelastic case in FP16 storage
        _box("droplet_256_fp16", "step", (256, 128, 64), 22.0, 0.2, 2.0, 3.0, 400.0, 1, 0.02, FP16, 0, 20),
        # the benchmark lattice in BF16 storage (stochastic rounding)
        _box("matrix_192_bf16", "step", (192, 96, 80), 16.0, 0.2, 1.0, 1.0, 100.0, 2, 0.02, BF16, 0, 20),
        # the second-order advection scheme
        _box("upwind2_192_fp32", "step", (192, 96, 80), 16.0, 0.2, 1.0, 1.0, 100.0, 2, 0.02, FP32, 1, 10),
        # an odd box: no extent divides a tile, rows are not 16-byte multiples
        _box("odd_141_fp32", "step", (141, 75, 53), 14.0, 0.15, 0.5, 3.0, 100.0, 1, 0.02, FP32, 0, 20),
        # one batch of the critical-Capillary search: equal boxes, many runs
        {"name": "study_16_fp32", "kind": "batch", "family": "study", "instances": 16, "shapes": 101,
         "precision": FP32, "steps": 10},
        # the uneven batch of the benchmark (ragged boxes) in FP16 storage
        {"name": "uneven_12_fp16", "kind": "batch", "family": "uneven", "instances": 12, "shapes": 4,
         "precision": FP16, "steps": 8},
        # the x-split domain decomposition: ghost exchange before every step
        _box("slabs_2_fp32", "slabs", (192, 96, 80), 16.0, 0.2, 1.0, 1.0, 100.0, 2, 0.02, FP32, 0, 4, parts=2),
        # the diagnostics taken between runs of steps
        {"name": "observe_192_fp32", "kind": "observe", "Lx": 192, "Ly": 96, "Lz": 80, "R": 16.0, "precision": FP32},
        # one epoch of the proposal network's training: seven mini-batches of 256 rows
        {"name": "mlp_fit_1792", "kind": "fit", "rows": 1792, "batch": 256},
        # one proposal: the network over the Capillary grid of a search
        {"name": "mlp_forward_341", "kind": "forward", "rows": 341},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "batch", "slabs", "observe", "fit", "forward"))
    if kind in ("fit", "forward"):
        rows = _log(rng, 64, 2048) if kind == "fit" else _log(rng, 1, 4096)
        c = {"kind": kind, "rows": rows}
        if kind == "fit":
            c["batch"] = rng.choice((128, 256, 256, 512))
        return c
    if kind == "batch":
        return {"kind": kind, "family": rng.choice(("study", "uneven")), "instances": rng.randrange(2, 11),
                "shapes": rng.randrange(1 << 16), "precision": rng.choice((FP32, FP16, BF16)),
                "steps": rng.randrange(3, 6)}
    Lx, Ly, Lz = _log(rng, 24, 256), _log(rng, 20, 128), _log(rng, 16, 96)
    R = round(rng.uniform(0.25, 0.4) * min(Ly, Lz, 0.5 * Lx + 8), 2)
    precision = rng.choice((FP32, FP32, FP16, BF16))
    if kind == "observe":
        return {"kind": kind, "Lx": Lx, "Ly": Ly, "Lz": Lz, "R": R, "precision": precision}
    lam, Uw = rng.choice((1.0, 3.0)), rng.choice((0.01, 0.02))
    # relaxation times stay below about 9, where the scheme is stable: lam * eta_M <= 3
    Ca = round(min(rng.uniform(0.1, 0.3), 3.0 / lam * (2.0 * Uw / Lz) * R / configs.SIGMA), 4)
    c = _box("", kind, (Lx, Ly, Lz), R, Ca, rng.choice((0.0, 0.5, 1.0, 2.0)), lam, rng.choice((100.0, 400.0)),
             rng.choice((1, 2)), Uw, precision, rng.choice((0, 0, 0, 1)) if kind == "step" else 0, 0)
    del c["name"]
    if kind == "slabs":
        c["parts"], c["steps"] = rng.choice((2, 2, 3)), rng.randrange(2, 7)
    else:
        c["steps"] = max(1, min(40, 20000000 // (Lx * Ly * Lz)))
    return c


# ---------------------------------------------------------------- inputs
def _params(c):
    p = configs.make_params(c["Lx"], c["Ly"], c["Lz"], c["R"], Ca=c["Ca"], De=c["De"], lam=c["lam"], L2=c["L2"],
                            phase=c["phase"], Uw=c["Uw"], precision=c["precision"])
    p.advection = c["advection"]
    return p


def _instances(c):
    """Parameters of every instance of a stepping case."""
    if c["kind"] != "batch":
        return [_params(c)]
    if c["family"] == "study":
        ps = [study.case_params(x) for x in study.sample_cases(c["instances"], c["shapes"])]
    else:
        ps = [p for p, _ in configs.config4(c["instances"], seed=c["shapes"])]
    for p in ps:
        p.precision = c["precision"]
    return ps


def _densities(p, seed, axes=(1.0, 1.0, 1.0), tilt=0.0):
    """Seeded densities [2][Lz][Ly][Lx] (float64, GPU) of a droplet near the
    middle of the box (an ellipsoid tilted in the x-z plane where asked for)
    with a little noise."""
    r = random.Random(seed)
    off = [r.uniform(-0.5, 0.5) for _ in range(3)]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def axis(n, o):
        return torch.arange(n, dtype=torch.float64, device="cuda") - ((n - 1) / 2 + o)

    x = axis(p.Lx, off[0])[None, None, :]
    y = axis(p.Ly, off[1])[None, :, None]
    z = axis(p.Lz, off[2])[:, None, None]
    ct, st = math.cos(tilt), math.sin(tilt)
    xa, za = ct * x + st * z, ct * z - st * x
    inside = (xa / axes[0]) ** 2 + (y / axes[1]) ** 2 + (za / axes[2]) ** 2 <= p.R * p.R
    hi = torch.full((), p.rho_in, dtype=torch.float64, device="cuda")
    lo = torch.full((), p.rho_out, dtype=torch.float64, device="cuda")
    rho = torch.stack([torch.where(inside, hi, lo), torch.where(inside, lo, hi)])
    noise = torch.rand(rho.shape, generator=g, dtype=torch.float64, device="cuda")
    return rho + configs.NOISE * (2.0 * noise - 1.0)


def _observe_densities(c, p, seed):
    return _densities(p, seed, axes=(1.25, 1.0, 0.85), tilt=random.Random(seed + 1).uniform(0.3, 0.7))


def _net_data(c, seed):
    """Scaled case descriptors, targets and shape masks of a training set."""
    r = np.random.default_rng(seed)
    n = c["rows"]
    x = r.uniform(-1.0, 1.0, (n, 6)).astype(np.float32)
    x[:, 5] = np.where(r.uniform(size=n) < 0.3, -1.0, 1.0)
    broken = (x[:, 0] + 0.5 * x[:, 1] - 0.3 * x[:, 3] + 0.2 * r.normal(size=n) > 0.2).astype(np.float32)
    t = np.stack([r.uniform(0.1, 0.8, n), r.uniform(0.1, 0.5, n), broken, r.integers(0, 3, n) / 4.0],
                 axis=1).astype(np.float32)
    return x, t, (1.0 - broken).astype(np.float32)


def _solver(ps, rhos):
    s = lbfe.Solver(ps)
    for k, rho in enumerate(rhos):
        s.init(k, rho.cpu().numpy())
    return s


def _observe_params(c):
    return configs.make_params(c["Lx"], c["Ly"], c["Lz"], c["R"], Ca=0.2, De=1.0, phase=2, Uw=0.02,
                               precision=c["precision"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("fit", "forward"):
        x, t, m = _net_data(case, seed)
        net = proposal.MLP(max_batch=4096)
        net.set_params(proposal.init_params(seed))
        return {"case": case, "net": net, "x": x, "t": t, "m": m}
    if kind == "observe":
        p = _observe_params(case)
        return {"case": case, "solver": _solver([p], [_observe_densities(case, p, seed)])}
    ps = _instances(case)
    if kind == "slabs":
        rho = _densities(ps[0], seed).cpu().numpy()
        slabs = []
        for x0, nx in decomp.partition(ps[0].Lx, case["parts"]):
            s = lbfe.Solver(decomp.local_params(ps[0], nx))
            s.init(0, decomp.slab_field(rho, x0, nx))
            slabs.append(decomp.Slab(x0, nx, decomp.CudaSlabStepper(s)))
        return {"case": case, "slabs": slabs}
    s = _solver(ps, [_densities(p, seed + 17 * k) for k, p in enumerate(ps)])
    blocks = [torch.empty(s.columns_bytes(k, p.Lx), dtype=torch.uint8, device="cuda") for k, p in enumerate(ps)]
    return {"case": case, "solver": s, "params": ps, "blocks": blocks}


def _views(block, precision, Lx, Ly, Lz):
    """A column block as its populations, conformation and offset densities."""
    cells = Lx * Ly * Lz
    eb = 4 if precision == FP32 else 2
    nf, nc = 2 * Q * cells * eb, 6 * cells * 4
    dtype = {FP32: torch.float32, FP16: torch.float16, BF16: torch.bfloat16}[precision]
    out = {"f": block[:nf].view(dtype).view(2, Q, Lz, Ly, Lx),
           "C": block[nf:nf + nc].view(torch.float32).view(6, Lz, Ly, Lx)}
    if precision != FP32:
        out["dens"] = block[nf + nc:].view(torch.float32).view(Lz, Ly, Lx, 2)
    return out


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "fit":
        # the last, small learning rate of the training's schedule
        hist = state["net"].fit(state["x"], state["t"], state["m"], epochs=1, lr=1e-4, lr_final=1e-4,
                                batch=c["batch"])
        return {"loss": hist[0], "params": state["net"].get_params()}
    if kind == "observe":
        return state["solver"].observables(0)
    if kind == "slabs":
        slabs = state["slabs"]
        decomp.run(slabs, decomp.LocalRing(slabs), c["steps"])
        return [_views(s.stepper.get_columns(decomp.GHOST, s.nx), c["precision"], s.nx, c["Ly"], c["Lz"])
                for s in slabs]
    s = state["solver"]
    s.step(c["steps"])
    out = []
    for k, (p, b) in enumerate(zip(state["params"], state["blocks"])):
        s.get_columns(k, 0, p.Lx, b.data_ptr())
        out.append(_views(b, c["precision"], p.Lx, p.Ly, p.Lz))
    return out


def work(case):
    kind = case["kind"]
    if kind in ("fit", "forward"):
        macs = 6 * 128 + 3 * 128 * 128 + 128 * 4
        rows, params = case["rows"], macs + 4 * 128 + 4
        if kind == "forward":
            return {"bytes": 4.0 * 10 * rows + 2.0 * params, "flops": 2.0 * macs * rows}
        # each mini-batch reads and updates weights and both moments
        n = -(-rows // case["batch"])
        return {"bytes": 4.0 * 11 * rows + 24.0 * params * n, "flops": 6.0 * macs * rows}
    if kind == "observe":
        cells = case["Lx"] * case["Ly"] * case["Lz"]
        return {"bytes": (152.0 if case["precision"] == FP32 else 84.0) * cells, "flops": 40.0 * cells}
    cells = sum(p.N for p in _instances(case))
    # state per cell: populations, conformation, offset densities; read and written once a step,
    # and read and written once more by the snapshot
    state = 176.0 if case["precision"] == FP32 else 108.0
    return {"bytes": 2.0 * state * cells * (case["steps"] + 1), "flops": 700.0 * cells * case["steps"]}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _at(a, dx, dy, dz):
    """a(x + d): periodic in x and y, the wall layer repeated beyond z."""
    if dx or dy:
        a = torch.roll(a, (-dy, -dx), (-2, -1))
    if dz:
        n = a.shape[-3]
        i = (torch.arange(n, device=a.device) + dz).clamp(0, n - 1)
        a = a.index_select(a.dim() - 3, i)
    return a


def _minmod(a, b):
    return torch.where(a * b <= 0, torch.zeros_like(a), torch.where(a.abs() < b.abs(), a, b))


def _constants(p):
    rr = p.rho_in + p.rho_out
    eta_a, eta_b = p.lambda_ * p.eta_M, p.eta_M
    if p.visco_phase == 1:
        eta_a -= p.eta_P
    elif p.visco_phase == 2:
        eta_b -= p.eta_P
    return eta_a / rr, eta_b / rr, (p.eta_P / p.tau_P if p.visco_phase else 0.0)


def _step64(f, C, p):
    """One time step; returns the new populations and conformation and the densities of the old state."""
    nu_a, nu_b, pi_coef = _constants(p)
    Lz = p.Lz
    rho = f.sum(1)
    tot = rho.sum(0)
    both = f.sum(0)
    j = [sum(e[i] * both[i] for i in range(Q) if e[i]) for e in (CX, CY, CZ)]
    grad = [[0.0] * 3, [0.0] * 3]
    for i in range(1, Q):
        r = _at(rho, CX[i], CY[i], CZ[i])
        for a, e in enumerate((CX, CY, CZ)):
            if e[i]:
                for s in range(2):
                    grad[s][a] = grad[s][a] + WT[i] * e[i] * r[1 - s]
    unit = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
    fp = (p.L2 - 3.0) / (p.L2 - (C[0] + C[1] + C[2]))
    poly = [0.0] * 3
    if p.visco_phase:
        chi = pi_coef * rho[p.visco_phase - 1] / tot
        for a in range(3):
            for b in range(3):
                pi = chi * (fp * C[SYM[min(a, b), max(a, b)]] - (1.0 if a == b else 0.0))
                m = [-d for d in unit[b]]
                poly[a] = poly[a] + 0.5 * (_at(pi, *unit[b]) - _at(pi, *m))
    F = [[-p.G * rho[s] * grad[s][a] + (rho[s] / tot) * poly[a] + rho[s] * p.g[a] for a in range(3)]
         for s in range(2)]
    u = [(j[a] + 0.5 * (F[0][a] + F[1][a])) / tot for a in range(3)]

    # conformation: central grad u with the wall velocity, upwind advection
    gu = [[None] * 3 for _ in range(3)]
    for b in range(3):
        wall = p.Uw if b == 0 else 0.0
        gu[0][b] = 0.5 * (_at(u[b], 1, 0, 0) - _at(u[b], -1, 0, 0))
        gu[1][b] = 0.5 * (_at(u[b], 0, 1, 0) - _at(u[b], 0, -1, 0))
        up, dn = _at(u[b], 0, 0, 1).clone(), _at(u[b], 0, 0, -1).clone()
        up[Lz - 1] = 2.0 * wall - u[b][Lz - 1]
        dn[0] = -2.0 * wall - u[b][0]
        gu[2][b] = 0.5 * (up - dn)
    adv = 0.0
    for a in range(3):
        e, m = unit[a], tuple(-d for d in unit[a])
        pos = u[a] > 0
        cm, cp = _at(C, *m), _at(C, *e)
        if p.advection:
            cmm, cpp = _at(C, *(2 * d for d in m)), _at(C, *(2 * d for d in e))
            s0, sm, sp = _minmod(cp - C, C - cm), _minmod(C - cm, cm - cmm), _minmod(cpp - cp, cp - C)
            d = torch.where(pos, (C + 0.5 * s0) - (cm + 0.5 * sm), (cp - 0.5 * sp) - (C - 0.5 * s0))
        else:
            d = torch.where(pos, C - cm, cp - C)
        adv = adv + u[a] * d
    Cn = torch.empty_like(C)
    for (a, b), k in SYM.items():
        st = 0.0
        for m in range(3):
            st = st + C[SYM[min(a, m), max(a, m)]] * gu[m][b] + gu[m][a] * C[SYM[min(m, b), max(m, b)]]
        Cn[k] = C[k] - adv[k] + st - (fp * C[k] - (1.0 if a == b else 0.0)) / p.tau_P

    # collision, streaming, halfway bounce-back on the moving walls
    tau = 3.0 * (rho[0] * nu_a + rho[1] * nu_b) / tot + 0.5
    om, pre = 1.0 / tau, 1.0 - 0.5 / tau
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    fn = torch.empty_like(f)
    back = (0,) + tuple(i + 1 if i % 2 else i - 1 for i in range(1, Q))
    for s in range(2):
        uF = u[0] * F[s][0] + u[1] * F[s][1] + u[2] * F[s][2]
        for i in range(Q):
            e = (CX[i], CY[i], CZ[i])
            cu = sum((e[a] * u[a] for a in range(3) if e[a]), torch.zeros_like(uu))
            cF = sum((e[a] * F[s][a] for a in range(3) if e[a]), torch.zeros_like(uu))
            eq = WT[i] * rho[s] * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
            post = f[s, i] - om * (f[s, i] - eq) + pre * WT[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
            moved = torch.roll(post, (e[1], e[0]), (-2, -1))
            if e[2] > 0:
                fn[s, i, 1:] = moved[:-1]
                fn[s, back[i], Lz - 1] = post[Lz - 1] - 6.0 * WT[i] * rho[s, Lz - 1] * e[0] * p.Uw
            elif e[2] < 0:
                fn[s, i, :-1] = moved[1:]
                fn[s, back[i], 0] = post[0] + 6.0 * WT[i] * rho[s, 0] * e[0] * p.Uw
            else:
                fn[s, i] = moved
    return fn, Cn, rho


def _state64(p, rho, steps):
    w = torch.tensor(WT, dtype=torch.float64, device=rho.device)
    f = rho[:, None] * w[None, :, None, None, None]
    C = torch.zeros((6, p.Lz, p.Ly, p.Lx), dtype=torch.float64, device=rho.device)
    C[:3] = 1.0
    old = rho
    for _ in range(steps):
        f, C, old = _step64(f, C, p)
    out = {"f": f, "C": C}
    if p.precision != FP32:
        out["f"] = f - old[:, None] * w[None, :, None, None, None]
        out["dens"] = old.permute(1, 2, 3, 0).contiguous()
    return out


def _observables64(p, rho):
    A = rho[0] > rho[1]
    V = int(A.sum())
    z, y, x = (t.double() for t in torch.nonzero(A, as_tuple=True))
    c = [float(t.mean()) for t in (x, y, z)]
    d = [t - m for t, m in zip((x, y, z), c)]
    M = [float((d[a] * d[b]).sum()) for a, b in SYM]
    ev, vec = np.linalg.eigh(np.array([[M[0], M[3], M[4]], [M[3], M[1], M[5]], [M[4], M[5], M[2]]]))
    a, b = math.sqrt(5.0 * ev[2] / V), math.sqrt(5.0 * ev[0] / V)
    th = math.degrees(math.atan2(vec[2, 2], vec[0, 2]))
    th += 180.0 if th <= -90.0 else (-180.0 if th > 90.0 else 0.0)
    lp = int(A.any(0).any(0).sum())
    return dict(step=0, mass=(float(rho[0].sum()), float(rho[1].sum())), volume=float(V), centroid=tuple(c),
                M=tuple(M), D=(a - b) / (a + b), theta_deg=th, Lp=float(lp), Lp_over_2R=lp / (2.0 * p.R),
                t_over_tem=0.0, necks=0, fragments=1, broken=0, flags=0)


def _layers64(params):
    dims, out, o = (6, 128, 128, 128, 128, 4), [], 0
    for i, j in zip(dims, dims[1:]):
        out.append((params[o:o + i * j].view(i, j), params[o + i * j:o + i * j + j]))
        o += i * j + j
    return out


def _forward64(params, x):
    h = x
    for l, (w, b) in enumerate(_layers64(params)):
        h = h @ w + b
        if l < 4:
            h = 0.5 * h * (1.0 + torch.erf(h * math.sqrt(0.5)))
    return h


def _loss64(y, t, m):
    sq = (y[:, 0] - t[:, 0]) ** 2 + (y[:, 1] - t[:, 1]) ** 2 + (y[:, 3] - t[:, 3]) ** 2
    bce = torch.nn.functional.binary_cross_entropy_with_logits(y[:, 2], t[:, 2], reduction="none")
    return (m * sq + bce).mean()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "forward"):
        x, t, m = (torch.from_numpy(a).cuda().double() for a in _net_data(case, seed))
        w = torch.from_numpy(proposal.init_params(seed)).cuda().double()
        if kind == "forward":
            return _forward64(w.bfloat16().double(), x)      # the network reads its weights in BF16
        perm = torch.from_numpy(np.random.default_rng(0).permutation(len(x))).cuda()
        ms, vs, total, n = torch.zeros_like(w), torch.zeros_like(w), 0.0, 0
        for s in range(0, len(x), case["batch"]):
            i = perm[s:s + case["batch"]]
            wr = w.float().bfloat16().double().requires_grad_(True)
            loss = _loss64(_forward64(wr, x[i]), t[i], m[i])
            loss.backward()
            n += 1
            ms = 0.9 * ms + 0.1 * wr.grad
            vs = 0.999 * vs + 0.001 * wr.grad ** 2
            w = w - 1e-4 * (ms / (1 - 0.9 ** n) / ((vs / (1 - 0.999 ** n)).sqrt() + 1e-8) + 1e-4 * w)
            total += float(loss) * len(i)
        return {"loss": total / len(x), "params": w}
    if kind == "observe":
        p = _observe_params(case)
        return _observables64(p, _observe_densities(case, p, seed))
    ps = _instances(case)
    if kind == "slabs":
        o = _state64(ps[0], _densities(ps[0], seed), case["steps"])
        out = []
        for x0, nx in decomp.partition(ps[0].Lx, case["parts"]):
            d = {"f": o["f"][..., x0:x0 + nx], "C": o["C"][..., x0:x0 + nx]}
            if "dens" in o:
                d["dens"] = o["dens"][:, :, x0:x0 + nx]
            out.append(d)
        return out
    return [_state64(p, _densities(p, seed + 17 * k), case["steps"]) for k, p in enumerate(ps)]
