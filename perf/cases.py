"""Work that users of this library have it do, as cases that can be timed.

A case is a dict of plain values.  `op` says which public call it stands for:

* ``step``     ``Lattice.step(n)`` on one periodic lattice that holds a drop or a
  bubble: the inner loop of every study, at every box, storage, stencil, psi and
  tau that the library takes.  Returns the whole stored state (19 populations).
* ``group``    ``Group.step(n)`` on lattices of several sizes, the launches that a
  sweep over radii is made of.  Returns every lattice's stored state.
* ``relax``    a whole small run: initialise a drop, step it, copy the density
  field to the host and measure the observables.
* ``observe``  the convergence check: ``observables()`` and the two profiles.
* ``flat``     ``flat_interface()``: coexistence densities and tension of a strip,
  which every sweep runs first for each coupling.
"""
import math

import numpy as np
import torch

import paper_2105_08772_gb300 as lbm

# coexistence densities of the couplings that the sweeps and studies use:
# (psi, G, T, liquid, gas)
FLUIDS = {
    "G4.6": ("one_minus_exp", -4.6, 0.0, 1.5618, 0.2034),
    "G5.0": ("one_minus_exp", -5.0, 0.0, 1.8884, 0.1194),
    "G5.5": ("one_minus_exp", -5.5, 0.0, 2.2477, 0.0563),
    "exp.159": ("exp_inv", -8.563916018660622, 0.0, 2.0026, 0.5104),
    "exp.293": ("exp_inv", -9.55404953591733, 0.0, 2.5489, 0.4024),
    "cs.9": ("cs", -1.0, 0.9 * 0.09432870312373377, 0.2455, 0.0394),
}


def _step(name, box, prec, steps, fluid="G5.0", stencil="E4", tau=1.0, bubble=False):
    return {"name": name, "op": "step", "nx": box[0], "ny": box[1], "nz": box[2], "prec": prec, "steps": steps,
            "fluid": fluid, "stencil": stencil, "tau": tau, "bubble": bubble}


def listed():
    return [
        # the smallest whole call: the strip whose rest state starts a sweep (latency of 2048 tiny steps)
        {"name": "flat_100_f64", "op": "flat", "nx": 100, "steps": 2048, "prec": "f64", "fluid": "G5.0", "stencil": "E4"},
        # the small FP64 run that results are pinned on: 32^3, 2000 steps, field and observables read back
        {"name": "relax_32_f64", "op": "relax", "nx": 32, "ny": 32, "nz": 32, "prec": "f64", "steps": 2000,
         "fluid": "G5.0", "stencil": "E4", "tau": 1.0, "bubble": False},
        # the sweep's smallest box: the state stays in L2, launches and latency count
        _step("drop_64_f32", (64, 64, 64), "f32", 256, fluid="G4.6"),
        # the headline workload: a droplet in a 128^3 box, shifted FP32
        _step("drop_128_f32", (128, 128, 128), "f32", 128),
        # one of the paper's own boxes: odd side, psi = exp(-1/n), a bubble
        _step("bubble_157_f32", (157, 157, 157), "f32", 128, fluid="exp.159", bubble=True),
        # the largest ordinary box: 2.5 GB of state, HBM traffic counts
        _step("drop_256_f32", (256, 256, 256), "f32", 128),
        # the precision study's FP16 storage at its own size
        _step("drop_192_f16", (192, 192, 192), "f16", 128),
        # the FP64 plain path that every reduced precision is compared with
        _step("bubble_128_f64", (128, 128, 128), "f64", 24, bubble=True),
        # wider forcing stencil with the Carnahan-Starling psi, the study's 256^3 box
        _step("cs_e6_256_f32", (256, 256, 256), "f32", 32, fluid="cs.9", stencil="E6"),
        # another relaxation time (viscosity) in a ragged box
        _step("tau0.8_120x72x100_f32", (120, 72, 100), "f32", 128, tau=0.8),
        # a sweep's resident lattices advancing together, boxes of several sizes
        {"name": "group_sweep_f32", "op": "group", "sides": "64,72,80,96,112,128", "prec": "f32", "steps": 128,
         "fluid": "G5.0", "stencil": "E4", "tau": 1.0, "bubble": False},
        # the convergence check, once per 2048 steps and after every run
        {"name": "observe_128_f32", "op": "observe", "nx": 128, "ny": 128, "nz": 128, "prec": "f32",
         "fluid": "G5.0", "stencil": "E4", "tau": 1.0, "bubble": False},
    ]


# node updates that one pass may cost, by storage and stencil (below the largest listed case's time)
_BUDGET = {"f32": 1.2e9, "f16": 8e8, "f64": 4.5e7}


def draw(rng):
    op = rng.choice(["step"] * 8 + ["group", "relax", "observe", "flat"])
    fluid = rng.choice(["G4.6", "G5.0", "G5.5", "exp.159", "exp.293"])
    bubble = rng.random() < 0.4

    def side(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.4 else max(lo, n // 4 * 4)      # many boxes are multiples of 4

    if op == "flat":
        return {"op": "flat", "nx": side(40, 240), "steps": 2048, "prec": rng.choice(["f64", "f64", "f32"]),
                "fluid": rng.choice(["G4.6", "G5.0", "G5.5"]), "stencil": rng.choice(["E4", "E4", "E6"])}
    if op == "group":
        k = rng.randint(2, 8)
        sides = ",".join(str(side(40, 120)) for _ in range(k))
        return {"op": "group", "sides": sides, "prec": "f32", "steps": 2 * rng.randint(16, 64), "fluid": fluid,
                "stencil": "E4", "tau": 1.0, "bubble": bubble}
    if op == "observe":
        nx, ny, nz = side(40, 256), side(40, 256), side(40, 256)
        return {"op": "observe", "nx": nx, "ny": ny, "nz": nz, "prec": rng.choice(["f32", "f64", "f16"]),
                "fluid": fluid, "stencil": rng.choice(["E4", "E4", "E6"]), "tau": 1.0, "bubble": bubble}
    if op == "relax":
        nx, ny, nz = side(20, 40), side(20, 40), side(20, 40)
        return {"op": "relax", "nx": nx, "ny": ny, "nz": nz, "prec": "f64", "steps": 2 * rng.randint(100, 500),
                "fluid": fluid, "stencil": "E4", "tau": 1.0, "bubble": False}
    prec = rng.choice(["f32"] * 6 + ["f16"] * 2 + ["f64"] * 2)
    stencil = rng.choice(["E4"] * 6 + ["E6", "E8"])
    tau = rng.choice([1.0] * 5 + [0.8, 1.3])
    if stencil != "E4" and rng.random() < 0.7:
        fluid = "cs.9"
    if prec == "f16" and rng.random() < 0.8:   # FP16 runs are mostly the plain E4 ones, whole 8-node groups
        stencil, tau, fluid = "E4", 1.0, "G5.0"
    nx, ny, nz = side(32, 256), side(24, 256), side(24, 256)
    if prec == "f16" and stencil == "E4":
        nx = max(48, nx // 8 * 8)
    wide = {"E4": 1, "E6": 2, "E8": 3}[stencil]
    steps = int(_BUDGET[prec] / wide / (nx * ny * nz))
    return {"op": "step", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "steps": max(2, min(160, steps // 2 * 2)),
            "fluid": fluid, "stencil": stencil, "tau": tau, "bubble": bubble}


# ------------------------------------------------------------------ inputs and runs

def _drop(case, box, seed):
    """Centre, radius and the two densities of one drop: a quarter of the smallest side, densities near
    coexistence, all shifted a little by the seed."""
    rng = np.random.default_rng([seed, *box])
    psi, G, T, rho_l, rho_g = FLUIDS[case["fluid"]]
    centre = [n // 2 + float(rng.uniform(-0.5, 0.5)) for n in box]
    R = 0.25 * min(box) * (1.0 + float(rng.uniform(-0.04, 0.04)))
    rho_l *= 1.0 + float(rng.uniform(-0.004, 0.004))
    rho_g *= 1.0 + float(rng.uniform(-0.004, 0.004))
    inner, outer = (rho_g, rho_l) if case["bubble"] else (rho_l, rho_g)
    return centre, R, inner, outer


def _boxes(case):
    if case["op"] == "group":
        return [(int(s),) * 3 for s in case["sides"].split(",")]
    return [(case["nx"], case["ny"], case["nz"])]


def _lattice(case, box):
    psi, G, T, _, _ = FLUIDS[case["fluid"]]
    return lbm.Lattice(*box, tau=case["tau"], G=G, psi=psi, cs_T=T, stencil=case["stencil"], prec=case["prec"])


_TORCH = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}


def _state(lat):
    """The lattice's stored populations (19, nz, ny, nx), as they lie in its workspace."""
    addr, nbytes = lbm.lbm_state_plane(lat.ctx, 0, 0)
    off = addr - lat.workspace.data_ptr()
    flat = lat.workspace[off:off + 19 * lat.nz * nbytes].view(_TORCH[lat.prec])
    return flat.view(19, lat.nz, lat.ny, lat.nx)


def _flat_args(case, seed):
    psi, G, T, rho_l, rho_g = FLUIDS[case["fluid"]]
    rng = np.random.default_rng([seed, case["nx"]])
    return dict(G=G, psi=psi, cs_T=T, stencil=case["stencil"], prec=case["prec"], tau=1.0, Lx=case["nx"],
                rho_l0=rho_l * (1.0 + float(rng.uniform(-0.01, 0.01))),
                rho_g0=rho_g * (1.0 + float(rng.uniform(-0.01, 0.01))), max_steps=case["steps"], tol_du=1e-30)


def prepare(case, seed):
    if case["op"] == "flat":
        return {"case": case, "args": _flat_args(case, seed)}
    lats, drops = [], []
    for box in _boxes(case):
        lat = _lattice(case, box)
        drop = _drop(case, box, seed)
        lat.init_drop(*drop)
        lats.append(lat)
        drops.append(drop)
    st = {"case": case, "lats": lats, "drops": drops}
    if case["op"] == "group":
        st["group"] = lbm.Group(lats)
    return st


_OBS = ("n_in", "n_out", "P_in", "P_out", "dP", "mass", "R_e", "C", "D", "R_s", "sigma_s", "max_u")


def _measured(o):
    out = {k: getattr(o, k) for k in _OBS}
    out.update(com0=o.com[0], com1=o.com[1], com2=o.com[2], steps=int(o.steps), bits=int(o.status_bits))
    return out


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "flat":
        _, n_g, n_l, sigma0, steps = lbm.flat_interface(**state["args"])
        return {"n_g": n_g, "n_l": n_l, "sigma0": sigma0, "steps": int(steps)}
    lat = state["lats"][0]
    if op == "step":
        lat.step(case["steps"])
        return _state(lat)
    if op == "group":
        state["group"].step(case["steps"])
        return [_state(lat) for lat in state["lats"]]
    if op == "relax":
        lat.init_drop(*state["drops"][0])
        lat.step(case["steps"])
        return {"rho": lat.rho(), "obs": _measured(lat.observables())}
    obs = _measured(lat.observables())
    return {"obs": obs, "rho_r": lat.rho_profile(), "pt_r": lat.pt_profile()}


def work(case):
    """Bytes: every stored population of every node read and written once per time step (the observe call:
    read once).  Operations: pull sums, force, velocity and collision of one node, about 300 (the wider
    stencils: their extra links)."""
    es = {"f64": 8, "f32": 4, "f16": 2}[case["prec"]]
    links = {"E4": 18, "E6": 32, "E8": 92}[case["stencil"]]
    flops = 250.0 + 4.0 * links
    if case["op"] == "flat":
        m = 3 if case["stencil"] == "E4" else 5
        nodes, steps = case["nx"] * m * m, case["steps"]
    else:
        nodes, steps = sum(a * b * c for a, b, c in _boxes(case)), case.get("steps", 1)
    if case["op"] == "observe":
        return {"bytes": nodes * 19 * es, "flops": nodes * flops}
    return {"bytes": float(nodes) * steps * 38 * es, "flops": float(nodes) * steps * flops}


# ------------------------------------------------------------------ the same in 64 bits, by plain torch

_XI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
       (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_SHELL = {"E4": {1: 1 / 6, 2: 1 / 12},
          "E6": {1: 2 / 15, 2: 1 / 15, 3: 1 / 60, 4: 1 / 120},
          "E8": {1: 4 / 45, 2: 1 / 21, 3: 2 / 105, 4: 5 / 504, 5: 1 / 315, 6: 1 / 630, 8: 1 / 5040}}


def _links(stencil):
    sh = _SHELL[stencil]
    r = range(-2, 3)
    return [(x, y, z, sh[x * x + y * y + z * z]) for x in r for y in r for z in r if x * x + y * y + z * z in sh]


def _psi(n, fluid):
    psi, G, T, _, _ = FLUIDS[fluid]
    if psi == "one_minus_exp":
        return -torch.expm1(-n)
    if psi == "exp_inv":
        return torch.exp(-1.0 / n)
    p = n * T * (1 + n + n ** 2 - n ** 3) / (1 - n) ** 3 - n ** 2       # a = 1, b = 4, R = 1: b n / 4 = n
    return torch.sqrt(2.0 * (p - n / 3.0) / (G / 3.0))


def _at(a, x, y, z):
    """a(r + (x, y, z)) of a periodic field [z, y, x]."""
    return torch.roll(a, (-z, -y, -x), (-3, -2, -1))


def _force(psi, G, stencil):
    F = [torch.zeros_like(psi) for _ in range(3)]
    for x, y, z, w in _links(stencil):
        s = w * _at(psi, x, y, z)
        for a, c in enumerate((x, y, z)):
            if c:
                F[a] += c * s
    k = -G / 3.0 * psi
    return [k * f for f in F]


def _moments(g):
    """n and j of the populations that stream into each node."""
    n = torch.zeros_like(g[0])
    j = [torch.zeros_like(n) for _ in range(3)]
    for i, (x, y, z) in enumerate(_XI):
        f = _at(g[i], -x, -y, -z)
        n += f
        for a, c in enumerate((x, y, z)):
            if c:
                j[a] += c * f
    return n, j


def _advance(g, case, steps):
    psi_name, G, T, _, _ = FLUIDS[case["fluid"]]
    om = 1.0 / case.get("tau", 1.0)
    for _ in range(steps):
        n, j = _moments(g)
        F = _force(_psi(n, case["fluid"]), G, case["stencil"])
        u = [(ja + 0.5 * fa) / n for ja, fa in zip(j, F)]
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        new = torch.empty_like(g)
        for i, (x, y, z) in enumerate(_XI):
            eu = x * u[0] + y * u[1] + z * u[2]
            eF = x * F[0] + y * F[1] + z * F[2]
            eq = _W[i] * n * (1.0 + 3.0 * eu + 4.5 * eu ** 2 - 1.5 * uu)
            src = (1.0 - 0.5 * om) * _W[i] * (3.0 * eF + 9.0 * eu * eF - 3.0 * uF)
            if om == 1.0:
                new[i] = eq + src
            else:
                new[i] = (1.0 - om) * _at(g[i], -x, -y, -z) + om * eq + src
        g = new
    return g


def _profile(box, drop, dev):
    centre, R, inner, outer = drop
    d2 = 0.0
    for a, n in enumerate(box):
        d = torch.arange(n, dtype=torch.float64, device=dev) - centre[a]
        d = torch.remainder(d + 0.5 * n, n) - 0.5 * n
        d2 = d2 + (d * d).view([-1 if k == 2 - a else 1 for k in range(3)])
    return 0.5 * (inner + outer) - 0.5 * (inner - outer) * torch.tanh(torch.sqrt(d2) - R)


def _at_rest(n):
    """Stored state of a fluid at rest: slot i of a node is what streams to its neighbour along xi_i."""
    return torch.stack([w * _at(n, *xi) for w, xi in zip(_W, _XI)])


def _stored(g, case, box, drop):
    """As the storage holds it: (f_i - w_i n0) times a power of two for the shifted storages."""
    if case["prec"] == "f64":
        return g
    _, R, inner, outer = drop
    frac = min(1.0, 4.0 * math.pi * R ** 3 / (3.0 * box[0] * box[1] * box[2]))
    n0 = outer + (inner - outer) * frac
    scale = 1.0
    if case["prec"] == "f16":
        dev = max(abs(inner - n0), abs(outer - n0)) / 3.0
        scale = 2.0 ** min(24, max(-24, math.floor(math.log2(8192.0 / dev))))
    for i in range(19):
        g[i] = (g[i] - _W[i] * n0) * scale
    return g


def _pressure(n, case):
    """P^xx and P^yy of the lattice pressure tensor."""
    _, G, _, _, _ = FLUIDS[case["fluid"]]
    psi = _psi(n, case["fluid"])
    sxx, syy = torch.zeros_like(n), torch.zeros_like(n)
    for x, y, z, w in _links(case["stencil"]):
        s = w * _at(psi, x, y, z)
        sxx += x * x * s
        syy += y * y * s
    return n / 3.0 + G / 6.0 * psi * sxx, n / 3.0 + G / 6.0 * psi * syy


def _observed(g, case, box):
    """The observables, and n and P_T on the +x half axis."""
    n, j = _moments(g)
    _, G, _, _, _ = FLUIDS[case["fluid"]]
    F = _force(_psi(n, case["fluid"]), G, case["stencil"])
    u2 = sum(((ja + 0.5 * fa) / n) ** 2 for ja, fa in zip(j, F))
    pxx, pyy = _pressure(n, case)
    nx, ny, nz = box
    c = (nz // 2, ny // 2, nx // 2)
    far = tuple((a + b // 2) % b for a, b in zip(c, (nz, ny, nx)))
    o = {"n_in": float(n[c]), "n_out": float(n[far]), "P_in": float(pxx[c]), "P_out": float(pxx[far])}
    o["dP"] = o["P_in"] - o["P_out"]
    o["mass"] = float(n.sum())
    w = n - o["n_out"]
    for a, m in enumerate(box):
        d = torch.arange(m, dtype=torch.float64, device=n.device) - m // 2
        d[2 * d == -m] = 0.0
        d = d.view([-1 if k == 2 - a else 1 for k in range(3)])
        o["com%d" % a] = m // 2 + float((w * d).sum() / w.sum())
    ex = 3.0 * (o["mass"] - nx * ny * nz * o["n_out"]) / (4.0 * math.pi * (o["n_in"] - o["n_out"]))
    o["R_e"] = math.copysign(abs(ex) ** (1.0 / 3.0), ex)
    x = torch.remainder(torch.arange(nx // 2 + 1, device=n.device) + c[2], nx)
    n_r, pt = n[c[0], c[1], x].cpu().numpy(), pyy[c[0], c[1], x].cpu().numpy()
    r = np.arange(nx // 2 + 1, dtype=np.float64)
    wt = np.ones_like(r)
    wt[0] = wt[-1] = 0.5
    o["C"] = float((wt * r * r * (o["P_out"] - pt)).sum())
    o["D"] = float((wt * r * (o["P_out"] - pt)).sum())
    q = o["C"] / o["dP"] if o["dP"] else -1.0
    o["R_s"] = (6.0 * q) ** (1.0 / 3.0) if q > 0 else float("nan")
    o["sigma_s"] = 0.5 * o["dP"] * o["R_s"]
    o["max_u"] = float(u2.max().sqrt())
    return n, o, n_r, pt


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["op"] == "flat":
        a = _flat_args(case, seed)
        L, m = a["Lx"], 3 if case["stencil"] == "E4" else 5
        x = torch.arange(L, dtype=torch.float64, device=dev)
        h = 0.5 * (a["rho_l0"] - a["rho_g0"])
        n = 0.5 * (a["rho_l0"] + a["rho_g0"]) - h * torch.tanh(x - 0.25 * L) + h * (torch.tanh(x - 0.75 * L) + 1.0)
        g = _advance(_at_rest(n.expand(m, m, L).contiguous()), case, case["steps"])
        n, _ = _moments(g)
        pxx, pyy = _pressure(n, case)
        c = (m // 2, m // 2)
        xs = torch.remainder(torch.arange(L // 2 + 1, device=dev) + L // 2, L)
        s = (pxx[c] - pyy[c])[xs].cpu().numpy()
        return {"n_g": float(n[c][L // 2]), "n_l": float(n[c][(L // 2 + L // 2) % L]),
                "sigma0": float(s.sum() - 0.5 * (s[0] + s[-1])), "steps": None}
    out = []
    for box in _boxes(case):
        drop = _drop(case, box, seed)
        g = _at_rest(_profile(box, drop, dev))
        if case["op"] == "observe":
            _, o, n_r, pt = _observed(g, case, box)
            return {"obs": o, "rho_r": n_r, "pt_r": pt}
        g = _advance(g, case, case["steps"])
        if case["op"] == "relax":
            n, o, _, _ = _observed(g, case, box)
            return {"rho": n.cpu().numpy(), "obs": o}
        out.append(_stored(g, case, box, drop))
    return out if case["op"] == "group" else out[0]
