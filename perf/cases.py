"""Timed cases of the library: what its users have it do, through its public entry points.

The library advances pseudo-potential lattice Boltzmann lattices.  Its users run small D2Q9
lattices for many steps (planar interfaces, Laplace droplets, channel flow), one large D3Q19
lattice on a whole GPU, many uneven lattices in one batch, or a caller-owned population array
without allocation; in between they read out moments and reductions.  The listed cases are one
of each, with the sizes of the repository's workloads, tests and benchmark; ``draw`` spreads
over the same ranges.

A pass is one call of the stepping entry point with ``steps`` time steps (even, so that the
in-place populations end in the natural layout), or one round of the readouts.  The output of a
stepping pass is the updated state: the stored populations, in place.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2504_15018_gb300 as plb

# Coexistence densities of the Peng-Robinson EOS (a = 2/49, b = 2/21, R = 1, omega = 0.327).
PR_DENSITIES = {0.7: (0.05792898641860934, 8.05920880114368), 0.75: (0.1120861713332112, 7.657021621261066),
                0.8: (0.20185142553734936, 7.182057676999079), 0.85: (0.34734637349576725, 6.608342999892656),
                0.9: (0.5872090599108848, 5.889068046737519)}
PR_A, PR_B, PR_R, PR_OMEGA = 2.0 / 49.0, 2.0 / 21.0, 1.0, 0.327
# The paper's EOS for R134a at 30 C, 100 cells per 10 micrometres (Sec. VI).
PAPER = dict(rho_v=0.0375, rho_l=1.187, P=0.0439932, tau=0.56, tau_v=0.62873, kappa=1.0257)
RATES = dict(s_e=1.19, s_eps=1.4, s_q=1.2, s_pi=1.4, s_m=1.98)
PRECISION = {"fp64": 0, "fp32": 1, "fp16s": 2, "fp16s_sr": 2}
POP_BYTES = {"fp64": 8, "fp32": 4, "fp16s": 2, "fp16s_sr": 2}
POP_DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16s": torch.float16, "fp16s_sr": torch.float16}
BATCH_SIDES = (64, 96, 128, 192, 256, 384, 512)


def _case(name, api, lattice, dims, precision, steps, **kw):
    c = dict(api=api, lattice=lattice, nx=dims[0], ny=dims[1], nz=dims[2] if len(dims) > 2 else 1,
             precision=precision, steps=steps, collision="bgk", streaming="aa", eos="pr", t_ratio=0.8, tau=1.0,
             tau_v=0.0, kappa=1.0, wall=False, wall_rho=0.0, shape="droplet", ux=0.0, uy=0.0, uz=0.0, fx=0.0,
             count=1)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    r134a = dict(eos="paper", tau=PAPER["tau"], tau_v=PAPER["tau_v"], kappa=PAPER["kappa"])
    return [
        # the smallest lattice in use: the D2Q9 planar-interface benchmark, 20,000 and more steps a run
        _case("planar_8x256_fp32", "step", "d2q9", (8, 256), "fp32", 100, shape="slab"),
        # a Laplace droplet, 40,000 steps a run
        _case("laplace_256_fp32", "step", "d2q9", (256, 256), "fp32", 100),
        # the paper's two-phase channel between walls in FP64, on an odd, ragged grid
        _case("channel_301x203_fp64", "step", "d2q9", (301, 203), "fp64", 20, shape="slab", wall=True, fx=1e-7, **r134a),
        # a batch of uneven D2Q9 lattices (Laplace sweeps, ladders) stepped together
        _case("batch60_fp32", "batch", "d2q9", (512, 512), "fp32", 50, count=60),
        # allocation-free stepping of a caller-owned array (a plugin): 64^3 droplet
        _case("static_64_fp32", "static", "d3q19", (64, 64, 64), "fp32", 10),
        # a D3Q19 droplet of the FP64 refinement ladder
        _case("droplet_96_fp64", "step", "d3q19", (96, 96, 96), "fp64", 4, collision="mrt"),
        # a box of odd extents with walls, FP32
        _case("box_127x95x63_fp32", "step", "d3q19", (127, 95, 63), "fp32", 10, collision="mrt", wall=True,
              shape="slab", fx=1e-6),
        # the benchmark workload, in place, FP32 and FP16 storage
        _case("plates_fp32", "step", "d3q19", (512, 256, 256), "fp32", 10, collision="mrt", wall=True, shape="film",
              fx=1e-7),
        _case("plates_fp16s", "step", "d3q19", (512, 256, 256), "fp16s", 10, collision="mrt", wall=True, shape="film",
              fx=1e-7),
        # a moving droplet with FP16 storage and stochastic rounding (the FP16 mode that keeps the
        # surface tension within 1 %)
        _case("droplet_160_fp16s_sr", "step", "d3q19", (160, 160, 160), "fp16s_sr", 10, ux=0.02, uy=-0.01, uz=0.015),
        # the single-pass stepping mode, on a ragged lattice
        _case("plates_single_pass_fp32", "step", "d3q19", (394, 250, 186), "fp32", 10, collision="mrt",
              streaming="fused", wall=True, shape="film", fx=1e-7),
        # readouts of a running lattice: mass, momentum, max |u|, and the fields into device arrays
        _case("monitor_256x128x128_fp32", "monitor", "d3q19", (256, 128, 128), "fp32", 0, ux=0.02, uy=-0.01, uz=0.015),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["step", "step", "step", "step", "step", "batch", "static", "monitor"])
    lattice = "d2q9" if api == "batch" else rng.choice(["d2q9", "d3q19", "d3q19"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16s", "fp16s_sr"])
    most = 1 << 18 if api == "static" else (1 << 20 if precision == "fp64" else 1 << 23)
    if lattice == "d2q9":
        dims = [_log_int(rng, 8, 1024), _log_int(rng, 16, 1024), 1]
    else:
        dims = [_log_int(rng, 10, 512), _log_int(rng, 10, 256), _log_int(rng, 6, 256)]
    while dims[0] * dims[1] * dims[2] > most:
        k = max(range(3), key=lambda a: dims[a])
        dims[k] = int(dims[k] * 0.8)
    cells = dims[0] * dims[1] * dims[2]
    streaming = "aa"
    if api in ("step", "monitor") and precision != "fp64" and rng.random() < 0.25:
        streaming = "fused"
        dims[0] += dims[0] % 2
    steps = 2 * _log_int(rng, 1, 50 if cells < 1 << 18 else 5)
    kw = dict(collision=rng.choice(["bgk", "mrt"]), streaming=streaming)
    count = 1
    if api == "batch":
        count, steps = _log_int(rng, 4, 60), 2 * _log_int(rng, 1, 25)
        precision = rng.choice(["fp32", "fp32", "fp16s", "fp64"])
        if precision == "fp64":
            count = min(count, 12)
        dims = [512, 512, 1]
    if api == "monitor":
        steps = 0
    if precision in ("fp64", "fp32") and api != "batch" and rng.random() < 0.3:
        kw.update(eos="paper", tau=PAPER["tau"], tau_v=PAPER["tau_v"], kappa=PAPER["kappa"])
    else:
        kw.update(t_ratio=rng.choice(sorted(PR_DENSITIES)))
        if rng.random() < 0.3:
            kw.update(tau=0.8, tau_v=1.1)
    if api != "batch" and rng.random() < 0.4:
        kw.update(wall=True, shape="slab", fx=1e-7)
        if api != "static" and kw.get("eos") != "paper" and rng.random() < 0.3:
            kw.update(wall_rho=1.0)
    elif api != "batch" and (api == "monitor" or rng.random() < 0.4):
        kw.update(ux=0.02, uy=-0.01, uz=0.015 if lattice == "d3q19" else 0.0)
    return _case(None, api, lattice, dims, precision, steps, count=count, **kw)


# ------------------------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _densities(case):
    if case["eos"] == "paper":
        return PAPER["rho_v"], PAPER["rho_l"]
    return PR_DENSITIES[case["t_ratio"]]


def _initial_density(case, seed, width=4.0):
    """rho0 [N] (float64, on the device): tanh interfaces and noise of 1e-4 of the densities."""
    dev = _device()
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rv, rl = _densities(case)
    ax = [torch.arange(n, device=dev, dtype=torch.float64) for n in (nz, ny, nx)]
    if case["shape"] == "droplet":
        dims = (nz, ny, nx) if case["lattice"] == "d3q19" else (ny, nx)
        r2 = torch.zeros((nz, ny, nx), device=dev, dtype=torch.float64)
        for a, n in enumerate((nz, ny, nx)):
            if n > 1:
                r2 += ((ax[a] - n / 2) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
        d = r2.sqrt() - case.get("radius", 0.25 * min(dims))
    else:
        # a liquid layer in the middle of y, or a film on each wall
        lo, hi = ny // 4 - 0.5, 3 * ny // 4 - 0.5
        d = torch.maximum(lo - ax[1], ax[1] - hi)
        if case["shape"] == "film":
            d = -d
        d = d.reshape(1, -1, 1).expand(nz, ny, nx)
    rho = rv + (rl - rv) * 0.5 * (1.0 - torch.tanh(2.0 * d / width))
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    noise = torch.rand(rho.shape, generator=g, device=dev, dtype=torch.float64) * 2.0 - 1.0
    return (rho * (1.0 + 1e-4 * noise)).reshape(-1).contiguous()


def _initial_velocity(case, n):
    d = 3 if case["lattice"] == "d3q19" else 2
    u = (case["ux"], case["uy"], case["uz"])[:d]
    if not any(u):
        return None
    return torch.tensor(u, device=_device(), dtype=torch.float64).reshape(d, 1).expand(d, n).contiguous()


def _instances(case):
    """The lattices of a batch: side, kind, temperature, radius and speed, the same for every seed."""
    if case["count"] == 1:
        return [case]
    r = np.random.RandomState(250415018 + case["count"])
    out = []
    for _ in range(case["count"]):
        side = int(r.choice(BATCH_SIDES))
        kind = r.choice(["static", "translating", "planar"])
        t = float(r.choice(sorted(PR_DENSITIES)))
        angle, speed, rfrac = r.uniform(0, 2 * math.pi), r.uniform(0.01, 0.05), r.uniform(0.1, 0.3)
        c = dict(case, nx=side, ny=side, t_ratio=t, shape="slab" if kind == "planar" else "droplet", radius=rfrac * side)
        if kind == "translating":
            c.update(ux=speed * math.cos(angle), uy=speed * math.sin(angle))
        out.append(c)
    return out


def _options(case):
    rv, rl = _densities(case)
    kw = dict(kappa=case["kappa"], precision=PRECISION[case["precision"]],
              collision=plb.PLB_MRT if case["collision"] == "mrt" else plb.PLB_BGK, wall_y=int(case["wall"]),
              wall_rho=case["wall_rho"], body_force=(case["fx"], 0.0, 0.0),
              streaming=plb.PLB_STREAM_FUSED if case["streaming"] == "fused" else plb.PLB_STREAM_AA,
              fp16_rounding=int(case["precision"] == "fp16s_sr"), tau_v=case["tau_v"], tau_rho_v=rv, tau_rho_l=rl,
              **RATES)
    if case["precision"].startswith("fp16s"):
        kw["rho_ref"] = rv
    return plb.make_opts(**kw)


def _eos(case):
    if case["eos"] == "paper":
        return plb.paper_eos(PAPER["rho_v"], PAPER["rho_l"], PAPER["P"])
    return plb.pr_eos(case["t_ratio"])


def _lattice_id(case):
    return plb.PLB_D3Q19 if case["lattice"] == "d3q19" else plb.PLB_D2Q9


def prepare(case, seed):
    """The lattice (or batch, or population array) with its initial state, ready to step."""
    lat_id, subs = _lattice_id(case), _instances(case)
    q = 19 if lat_id == plb.PLB_D3Q19 else 9
    state = dict(case=case, subs=subs, q=q)
    if case["api"] == "batch":
        insts = [plb.make_instance((c["nx"], c["ny"], c["nz"]), _eos(c), c["tau"], -1.0, 2.0, opts=_options(c))
                 for c in subs]
        state["batch"] = b = plb.Batch(lat_id, insts)
        for k, c in enumerate(subs):
            rho = _initial_density(c, seed * 1000 + k)
            u = _initial_velocity(c, rho.numel())
            torch.cuda.synchronize()                     # the batch has a stream of its own
            plb.plb_batch_init(b.b, k, rho, u)
        return state
    rho = _initial_density(case, seed)
    u = _initial_velocity(case, rho.numel())
    dims = (case["nx"], case["ny"], case["nz"])
    if case["api"] == "static":
        f = _equilibrium(case, rho, u)
        if case["precision"].startswith("fp16s"):
            f = f - _velocities(case)[1].reshape(-1, 1) * _densities(case)[0]
        state.update(pops=f.to(POP_DTYPE[case["precision"]]).contiguous(), t=0, dims=dims, eos=_eos(case),
                     opts=_options(case), lattice=lat_id)
        return state
    lat = plb.Lattice(lat_id, dims, _eos(case), tau=case["tau"], G=-1.0, eps=2.0, opts=_options(case))
    plb.plb_init(lat.h, rho, u)
    state["lat"] = lat
    if case["api"] == "monitor":
        n = rho.numel()
        state["fields"] = [torch.empty(m, device=rho.device, dtype=torch.float64) for m in (n, lat.D * n, n)]
    return state


def _stored(handle, ws, case, q):
    """The handle's population store as a (Q, N) view of the caller's workspace."""
    pops, _ = plb.plb_slab_regions(handle)
    size = POP_BYTES[case["precision"]]
    pitch = (plb.plb_state_bytes(handle) - 64) // (q * size)
    off = pops - ws.data_ptr()
    raw = ws[off:off + q * pitch * size].view(POP_DTYPE[case["precision"]])
    return raw.reshape(q, pitch)[:, :case["nx"] * case["ny"] * case["nz"]]


def run(state):
    case, q = state["case"], state["q"]
    if case["api"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        return [_stored(plb.plb_batch_instance(b.b, k), b.ws, c, q) for k, c in enumerate(state["subs"])]
    if case["api"] == "static":
        plb.plb_step_pairs_static(state["lattice"], state["dims"], state["eos"], case["tau"], -1.0, 2.0, state["opts"],
                                  state["pops"].data_ptr(), case["steps"] // 2, state["t"],
                                  torch.cuda.current_stream().cuda_stream)
        state["t"] += case["steps"]
        return state["pops"]
    lat = state["lat"]
    if case["api"] == "monitor":
        mass, mom, umax = (lat.reduce(w) for w in (plb.PLB_MASS, plb.PLB_MOMENTUM, plb.PLB_UMAX))
        rho, u, p = state["fields"]
        plb.plb_moments(lat.h, rho, u, p)
        return dict(mass=mass, momentum=mom, umax=umax, rho=rho, u=u, p=p)
    lat.step(case["steps"])
    return _stored(lat.h, lat.ws, case, q)


def work(case):
    """Every time step reads each stored population once and writes it once; a readout reads each
    once and writes its fields.  Operations: the arithmetic of one cell update, about."""
    q = 19 if case["lattice"] == "d3q19" else 9
    cells = sum(c["nx"] * c["ny"] * c["nz"] for c in _instances(case))
    size = POP_BYTES[case["precision"]]
    if case["api"] == "monitor":
        return {"bytes": cells * (3 * q * size + (q * size + 8 * (5 if q == 19 else 4))), "flops": cells * 10.0 * q}
    per_cell = {(9, "bgk"): 250, (9, "mrt"): 320, (19, "bgk"): 560, (19, "mrt"): 700}[q, case["collision"]]
    return {"bytes": cells * case["steps"] * 2 * q * size, "flops": float(cells) * case["steps"] * per_cell}


# ------------------------------------------------- the same step in 64 bits, plain torch

def _velocities(case):
    dev = _device()
    if case["lattice"] == "d2q9":
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
             (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
             (0, -1, 1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return c, torch.tensor(w, device=dev, dtype=torch.float64)


def _equilibrium(case, rho, u):
    """(Q, N) second-order equilibrium in float64; u (d, N) or None."""
    c, w = _velocities(case)
    out = torch.empty((len(c), rho.numel()), device=rho.device, dtype=torch.float64)
    usq = 0.0 if u is None else (u * u).sum(0)
    for i, ci in enumerate(c):
        cu = 0.0 if u is None else sum(ci[a] * u[a] for a in range(u.shape[0]))
        out[i] = w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
    return out


def _pressure(case, rho):
    if case["eos"] == "paper":
        rv, rl, s = PAPER["rho_v"], PAPER["rho_l"], rho.sqrt()
        sv = math.sqrt(rv)
        return PAPER["P"] * (2 * rho ** 3 + (rv - 2 * rl) * rho ** 2 - 3 * sv * rho ** 2 * s + 2 * sv * rl * rho * s
                             + sv * rl * rl * s)
    tc = 0.0778 * PR_A / (0.45724 * PR_B * PR_R)
    m = 0.37464 + 1.54226 * PR_OMEGA - 0.26992 * PR_OMEGA ** 2
    alpha = (1 + m * (1 - math.sqrt(case["t_ratio"]))) ** 2
    br = PR_B * rho
    return rho * PR_R * case["t_ratio"] * tc / (1 - br) - PR_A * alpha * rho * rho / (1 + 2 * br - br * br)


def _psi(case, rho):
    return (2.0 * (rho / 3.0 - _pressure(case, rho))).sqrt()          # G = -1


def _at(a, c, wall_rows=None):
    """a(x + c) on (nz, ny, nx), periodic; wall_rows: the rows beyond the y walls (below, above)."""
    if c[1] and wall_rows is not None:
        a = torch.cat([a[:, 1:], wall_rows[1]], 1) if c[1] > 0 else torch.cat([wall_rows[0], a[:, :-1]], 1)
        c = (c[0], 0, c[2])
    shifts = [(-c[2], 0), (-c[1], 1), (-c[0], 2)]
    shifts = [(s, d) for s, d in shifts if s]
    return torch.roll(a, [s for s, _ in shifts], [d for _, d in shifts]) if shifts else a


def _force(case, rho):
    """Total force density (d, nz, ny, nx): Shan-Chen force, eps and kappa terms, body force."""
    c, w = _velocities(case)
    d = 3 if case["lattice"] == "d3q19" else 2
    psi = _psi(case, rho)
    rows = None
    if case["wall"]:
        rows = (psi[:, :1], psi[:, -1:])
        if case["wall_rho"] > 0:
            v = _psi(case, torch.full_like(psi[:, :1], case["wall_rho"]))
            rows = (v, v)
    m1 = [torch.zeros_like(psi) for _ in range(d)]
    m2 = {(a, b): torch.zeros_like(psi) for a in range(d) for b in range(a, d)}
    for i, ci in enumerate(c):
        p = _at(psi, ci, rows) * float(w[i])
        for a in range(d):
            if ci[a]:
                m1[a] += 3.0 * ci[a] * p
            for b in range(a, d):
                k = 9.0 * (ci[a] * ci[b] - (1.0 / 3.0 if a == b else 0.0))
                if k:
                    m2[a, b] += k * p
    g, eps, kappa = -1.0, 2.0, case["kappa"]
    ka, kb = -(g / 12.0) * (2.0 * kappa - 2.0 - 3.0 * eps), (g / 6.0) * (kappa - 1.0)
    tr = sum(m2[a, a] for a in range(d))
    force = torch.empty((d,) + tuple(psi.shape), device=psi.device, dtype=torch.float64)
    for a in range(d):
        m21 = sum(m2[min(a, b), max(a, b)] * m1[b] for b in range(d))
        force[a] = -g * psi * m1[a] + ka * m21 + kb * m1[a] * tr + (case["fx"] if a == 0 else 0.0)
    return force


def _basis(case):
    """Orthogonal moment basis (Q, Q) and the rate of each row (None: 1 / tau)."""
    c, _ = _velocities(case)
    v = np.array(c, dtype=float)
    x, y, z = v.T
    s = x * x + y * y + z * z
    if case["lattice"] == "d2q9":
        rows = [(1 + 0 * x, None), (3 * s - 4, "s_e"), (4 - 10.5 * s + 4.5 * s * s, "s_eps"), (x, None),
                ((3 * s - 5) * x, "s_q"), (y, None), ((3 * s - 5) * y, "s_q"), (x * x - y * y, None), (x * y, None)]
    else:
        rows = [(1 + 0 * x, None), (19 * s - 30, "s_e"), ((21 * s * s - 53 * s + 24) / 2, "s_eps"),
                (3 * x * x - s, None), ((3 * s - 5) * (3 * x * x - s), "s_pi"), (y * y - z * z, None),
                ((3 * s - 5) * (y * y - z * z), "s_pi"), (x * y, None), (y * z, None), (x * z, None),
                ((y * y - z * z) * x, "s_m"), ((z * z - x * x) * y, "s_m"), ((x * x - y * y) * z, "s_m")]
        for e in (x, y, z):
            rows += [(e, None), ((5 * s - 9) * e, "s_q")]
    m = torch.tensor(np.array([r for r, _ in rows]), device=_device(), dtype=torch.float64)
    return m, [k if k is None else RATES[k] for _, k in rows]


def _macroscopic(case, f):
    c, _ = _velocities(case)
    d = 3 if case["lattice"] == "d3q19" else 2
    rho = f.sum(0)
    force = _force(case, rho)
    u = torch.stack([(sum(ci[a] * f[i] for i, ci in enumerate(c) if ci[a]) + 0.5 * force[a]) / rho for a in range(d)])
    return rho, u, force


def _one_step(case, f):
    c, w = _velocities(case)
    d = 3 if case["lattice"] == "d3q19" else 2
    rho, u, force = _macroscopic(case, f)
    om = torch.full_like(rho, 1.0 / case["tau"])
    if case["tau_v"] > 0:
        rv, rl = _densities(case)
        om = 1.0 / (case["tau_v"] + ((rho - rv) / (rl - rv)).clamp(0, 1) * (case["tau"] - case["tau_v"]))
    usq = (u * u).sum(0)
    uf = (u * force).sum(0)
    mrt = case["collision"] == "mrt"
    neq, guo = (torch.empty_like(f), torch.empty_like(f)) if mrt else (None, None)
    for i, ci in enumerate(c):
        cu = sum((ci[a] * u[a] for a in range(d) if ci[a]), torch.zeros_like(rho))
        cf = sum((ci[a] * force[a] for a in range(d) if ci[a]), torch.zeros_like(rho))
        ne = f[i] - w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
        gu = w[i] * (3.0 * cf + 9.0 * cu * cf - 3.0 * uf)
        if mrt:
            neq[i], guo[i] = ne, gu
        else:
            f[i] += (1.0 - 0.5 * om) * gu - om * ne
    if mrt:
        m, rates = _basis(case)
        q = f.shape[0]
        mom = (m @ neq.reshape(q, -1)).reshape(f.shape)
        del neq
        mg = (m @ guo.reshape(q, -1)).reshape(f.shape)
        del guo
        for k, r in enumerate(rates):
            s = om if r is None else r
            mom[k] = ((1.0 - 0.5 * s) * mg[k] - s * mom[k]) / (m[k] * m[k]).sum()
        del mg
        f += (m.T @ mom.reshape(q, -1)).reshape(f.shape)
        del mom
    out = torch.empty_like(f)
    opposite = [c.index((-a, -b, -e)) for a, b, e in c]
    for i, ci in enumerate(c):
        rows = None
        if case["wall"]:                     # f_i comes from y - c_y; beyond a wall: bounced f_opp(i)
            o = f[opposite[i]]
            rows = (o[:, :1], o[:, -1:])
            if ci[1]:
                moved = torch.roll(f[i], [ci[2], ci[0]], [0, 2])
                out[i] = _at(moved, (0, -ci[1], 0), rows)
                continue
        out[i] = _at(f[i], (-ci[0], -ci[1], -ci[2]), None)
    return out


def _evolved(case, seed):
    rho = _initial_density(case, seed)
    u = _initial_velocity(case, rho.numel())
    f = _equilibrium(case, rho, u).reshape(-1, case["nz"], case["ny"], case["nx"])
    del rho, u
    for _ in range(case["steps"]):
        f = _one_step(case, f)
    return f


def exact(case, seed):
    if case["api"] == "monitor":
        f = _evolved(case, seed)
        rho, u, _ = _macroscopic(case, f)
        d = u.shape[0]
        mom = torch.zeros(3, dtype=torch.float64, device=rho.device)
        mom[:d] = (rho * u).reshape(d, -1).sum(1)
        return dict(mass=rho.sum().reshape(1), momentum=mom, umax=(u * u).sum(0).sqrt().max().reshape(1),
                    rho=rho.reshape(-1), u=u.reshape(-1), p=_pressure(case, rho).reshape(-1))
    out = []
    for k, c in enumerate(_instances(case)):
        f = _evolved(c, seed * 1000 + k if case["api"] == "batch" else seed)
        f = f.reshape(f.shape[0], -1)
        if case["precision"].startswith("fp16s"):
            f = f - _velocities(c)[1].reshape(-1, 1) * _densities(c)[0]       # the stored deviation
        out.append(f)
    return out if case["api"] == "batch" else out[0]
