"""The work that users of this framework have it do, as measurable cases.

A case is one of three kinds:
  step    a simulation advanced a few PIC steps and read back (fields and
          particles by id), as a run with regular diagnostics does;
  serve   a batch of independent 2D requests through the request server;
  bin     caller-owned particles binned by box.
The recipes are those of ``paper_2104_11385_gb300.workloads`` (uniform plasma,
laser foil, boxes of uneven counts, the 2D laser-ion disk), drawn on the GPU,
with the fields of a run under way (a laser pulse near the foil, noise at the
plasma) instead of the zero fields of a run's first step.
"""
import math

import numpy as np
import torch

import paper_2104_11385_gb300 as pic
from paper_2104_11385_gb300.server import Server
from paper_2104_11385_gb300.sim import bin_particles

PROTON_MASS = 1836.15267343
F64 = torch.float64


def _step(name, layout, dim, order, n, box, ppc, steps, uth, precision=1, species=2, absorb=0, energy=False,
          sched="queue", ctas=2, rho=False, hot=False):
    return {"name": name, "kind": "step", "layout": layout, "dim": dim, "order": order, "nx": n[0], "ny": n[1],
            "nz": n[2], "bx": box[0], "by": box[1], "bz": box[2], "ppc": ppc, "steps": steps, "uth": uth,
            "precision": precision, "species": species, "absorb": absorb, "energy": energy, "sched": sched,
            "ctas": ctas, "rho": rho, "hot": hot}


def listed():
    return [
        # the smallest run anybody makes (a quick look, a unit of a scan): launches and gaps count
        _step("plasma16_linear", "plasma", 3, 1, (16, 16, 16), (8, 8, 8), 8, 20, 0.01, species=1, sched="none", ctas=1),
        # the 32^3 thermal plasma with a density diagnostic
        _step("plasma32_linear", "plasma", 3, 1, (32, 32, 32), (8, 8, 8), 8, 20, 0.01, species=1, sched="lists",
              rho=True),
        # a cubic, energy-conserving run on ragged boxes (60 x 36 x 50 cells)
        _step("plasma_cubic_energy", "plasma", 3, 3, (60, 36, 50), (12, 18, 10), 8, 4, 0.05, energy=True, sched="lists",
              ctas=1),
        # the laser foil at half extents, before the pulse arrives: a cold, dense slab in vacuum
        _step("foil128", "foil", 3, 1, (128, 128, 128), (16, 16, 16), 64, 4, 0.01, absorb=8),
        # the same foil with the pulse on it: hot electrons, most of them crossing cells every step
        _step("foil128_hot", "foil", 3, 1, (128, 128, 128), (16, 16, 16), 64, 4, 0.5, absorb=8, hot=True),
        # the foil in the float-float arithmetic
        _step("foil128_floatfloat", "foil", 3, 1, (128, 128, 128), (16, 16, 16), 64, 4, 0.01, precision=2, absorb=8),
        # the 256^3 foil, 67 M particles, in FP64 and in FP32
        _step("foil256", "foil", 3, 1, (256, 256, 256), (32, 32, 32), 64, 3, 0.01, absorb=16),
        _step("foil256_fp32", "foil", 3, 1, (256, 256, 256), (32, 32, 32), 64, 8, 0.01, precision=3, absorb=16),
        # boxes of log-normal particle counts, quadratic shapes
        _step("uneven512_quadratic", "uneven", 3, 2, (128, 128, 128), (16, 16, 16), 4, 3, 0.01, species=1, ctas=1),
        # the 2D3V laser-ion disk at 960^2 cells, cubic shapes
        _step("disk960_cubic", "disk", 2, 3, (960, 1, 960), (32, 1, 32), 32, 3, 0.01, absorb=32, hot=True),
        # a batch of 2D requests of mixed sizes through the server
        {"name": "serve6", "kind": "serve", "sides": "64,64,128,128,192,256", "ppcs": "4,16,8,32,4,16",
         "steps": "60,80,40,60,50,40"},
        # particles of a caller binned by box
        {"name": "bin16m", "kind": "bin", "dim": 3, "nx": 256, "ny": 256, "nz": 256, "box": 16, "np": 16777216,
         "shuffled": True},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plasma", "plasma", "plasma", "foil", "foil", "uneven", "disk", "serve", "bin"])
    if kind == "serve":
        k = rng.randint(2, 6)
        sides = [32 * rng.randint(2, 8) for _ in range(k)]
        ppcs = [_logint(rng, 1, 32) for _ in range(k)]
        steps = [rng.randint(20, 80) for _ in range(k)]
        return {"kind": "serve", "sides": ",".join(map(str, sides)), "ppcs": ",".join(map(str, ppcs)),
                "steps": ",".join(map(str, steps))}
    if kind == "bin":
        box = rng.choice([8, 16, 20, 32])
        dim = rng.choice([2, 3])
        n = [box * rng.randint(2, 256 // box) for _ in range(3)]
        return {"kind": "bin", "dim": dim, "nx": n[0], "ny": n[1], "nz": n[2], "box": box,
                "np": _logint(rng, 10001, 20000003), "shuffled": rng.random() < 0.7}
    precision = rng.choice([1, 1, 1, 1, 2, 3])
    if kind == "foil":
        m = rng.choice([1, 2, 3, 4])
        box = rng.choice([16, 32])
        n = (32 * rng.randint(m, 2 * m), 32 * rng.randint(m, 2 * m), 64 * rng.randint(1, 4))
        hot = rng.random() < 0.4
        order = rng.choice([1, 1, 1, 2])
        return _unnamed(_step("", "foil", 3, order, n, (box,) * 3, rng.choice([16, 33, 64]) if order == 1 else 8,
                              rng.randint(2, 4), 0.5 if hot else 0.01, precision=precision,
                              absorb=rng.choice([4, 8, 12]), hot=hot))
    if kind == "uneven":
        box = rng.choice([8, 12, 16])
        n = tuple(box * rng.randint(3, 8) for _ in range(3))
        return _unnamed(_step("", "uneven", 3, rng.choice([1, 2, 2, 3]), n, (box,) * 3, rng.choice([1, 2, 4]),
                              rng.randint(2, 4), 0.01, precision=precision, species=1,
                              sched=rng.choice(["queue", "lists"]), ctas=rng.choice([1, 2])))
    if kind == "disk":
        box = rng.choice([16, 32, 64])
        n = box * rng.randint(max(4, 256 // box), 960 // box)
        return _unnamed(_step("", "disk", 2, rng.choice([1, 2, 3, 3]), (n, 1, n), (box, 1, box), _logint(rng, 4, 32),
                              rng.randint(2, 6), 0.01, precision=precision, absorb=rng.choice([8, 16, 32]), hot=True))
    dim = rng.choice([2, 3, 3])
    box = tuple(2 * rng.randint(4, 12) for _ in range(3))
    cells = _logint(rng, 4096, 500000)
    edge = cells ** (1.0 / dim)
    n = tuple(b * max(1, int(round(edge * rng.uniform(0.6, 1.6) / b))) for b in box)
    if dim == 2:
        box, n = (box[0], 1, box[2]), (n[0], 1, n[2])
    order = rng.choice([1, 1, 2, 3])
    return _unnamed(_step("", "plasma", dim, order, n, box, _logint(rng, 1, 20), rng.randint(4, 20),
                          math.exp(rng.uniform(math.log(0.003), math.log(0.3))), precision=precision,
                          species=rng.randint(1, 2), energy=rng.random() < 0.3,
                          sched=rng.choice(["none", "queue", "lists"]), ctas=rng.choice([1, 2]),
                          rho=rng.random() < 0.3))


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _grid(case):
    """dx per direction, dt, laser"""
    dim, n = case["dim"], (case["nx"], case["ny"], case["nz"])
    lam = 2.0 * math.pi
    laser = None
    if case["layout"] == "foil":
        d = lam / 32.0
        laser = {"a0": 20.0, "w0": 2.0 * lam, "tau": 3.75 * lam, "t_peak": 3.0 * 3.75 * lam, "omega": 1.0,
                 "xc": 0.5 * n[0] * d, "yc": 0.5 * n[1] * d, "k_ant": case["absorb"] + 4}
    elif case["layout"] == "disk":
        um = lam / 0.8
        d = 30.0 * um / n[0]
        tau = 10.0 * lam * 0.299792458 / 0.8
        laser = {"a0": 25.0, "w0": 4.0 * um, "tau": tau, "t_peak": 2.5 * tau, "omega": 1.0, "xc": 15.0 * um, "yc": 0.0,
                 "k_ant": min(n[2] - 1, case["absorb"] + 2)}
    else:
        d = 0.25
    dx = (d, d if dim == 3 else 1.0, d)
    dt = 0.99 * d / math.sqrt(float(dim))
    return dx, dt, laser


def _uneven_counts(case):
    """log-normal particles per box; part of the layout, the same for every seed"""
    nb = [case["n" + a] // case["b" + a] for a in "xyz"]
    r = np.random.Generator(np.random.PCG64(17))
    c = np.exp(r.normal(0.0, 2.0, nb[0] * nb[1] * nb[2]))
    total = case["ppc"] * case["nx"] * case["ny"] * case["nz"]
    return np.floor(c * (total / c.sum())).astype(np.int64), nb


def _slab(case):
    """foil cell layers [z0, z1)"""
    z0 = case["nz"] // 2
    return z0, z0 + max(2, case["nz"] // 32)


def _disk_cells(case):
    n, um = case["nx"], 2.0 * math.pi / 0.8
    c = (np.arange(n) + 0.5) * (30.0 * um / n)
    cz, cx = np.meshgrid(c - 10.0 * um, c - 15.0 * um, indexing="ij")
    return np.nonzero(np.sqrt(cx * cx + cz * cz) < 7.0 * um)


def _particles(case):
    """particles per species"""
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["layout"] == "uneven":
        return int(_uneven_counts(case)[0].sum())
    if case["layout"] == "foil":
        z0, z1 = _slab(case)
        return case["nx"] * case["ny"] * (z1 - z0) * case["ppc"]
    if case["layout"] == "disk":
        return _disk_cells(case)[0].size * case["ppc"]
    return cells * case["ppc"]


def _species(case, seed):
    """(charge, mass, [x, y, z, ux, uy, uz, w]) per species, on the GPU"""
    g = _gen(seed)
    dx, _, _ = _grid(case)
    n = (case["nx"], case["ny"], case["nz"])
    L = [n[a] * dx[a] for a in range(3)]
    npart = _particles(case)
    uni = [torch.rand(npart, dtype=F64, device="cuda", generator=g) for _ in range(3)]
    dV = dx[0] * dx[1] * dx[2]
    if case["layout"] == "uneven":
        counts, nb = _uneven_counts(case)
        b = torch.repeat_interleave(torch.arange(counts.size, device="cuda"), torch.as_tensor(counts, device="cuda"))
        ijk = (b % nb[0], (b // nb[0]) % nb[1], b // (nb[0] * nb[1]))
        size = (case["bx"], case["by"], case["bz"])
        pos = [(ijk[a] + uni[a]) * (size[a] * dx[a]) for a in range(3)]
        w = torch.full((npart,), dV * n[0] * n[1] * n[2] / max(npart, 1), dtype=F64, device="cuda")
    elif case["layout"] == "foil":
        z0, z1 = _slab(case)
        pos = [uni[0] * L[0], uni[1] * L[1], (z0 + uni[2] * (z1 - z0)) * dx[2]]
        w = torch.full((npart,), 30.0 * dV / case["ppc"], dtype=F64, device="cuda")
    elif case["layout"] == "disk":
        kz, kx = _disk_cells(case)
        kz = torch.as_tensor(kz, device="cuda").repeat_interleave(case["ppc"])
        kx = torch.as_tensor(kx, device="cuda").repeat_interleave(case["ppc"])
        pos = [(kx + uni[0]) * dx[0], torch.zeros_like(uni[1]), (kz + uni[2]) * dx[2]]
        um = 2.0 * math.pi / 0.8
        rad = torch.sqrt((pos[0] - 15.0 * um) ** 2 + (pos[2] - 10.0 * um) ** 2)
        w = 5.0 * torch.where(rad <= 5.0 * um, 1.0, torch.exp(-(rad - 5.0 * um) / (0.05 * um))) * dV / case["ppc"]
    else:
        pos = [uni[a] * L[a] for a in range(3)]
        w = torch.full((npart,), dV / case["ppc"], dtype=F64, device="cuda")
    if case["dim"] == 2:
        pos[1] = torch.zeros_like(pos[0])
    del uni

    def momenta(s):
        return [torch.randn(npart, dtype=F64, device="cuda", generator=g) * s for _ in range(3)]

    out = [(-1.0, 1.0, pos + momenta(case["uth"]) + [w])]
    if case["species"] == 2:
        out.append((1.0, PROTON_MASS, [p.clone() for p in pos] + momenta(0.001) + [w.clone()]))
    return out


def _fields(case, seed):
    """six dense E, B arrays of a run under way"""
    g = _gen(seed + 7919)
    dx, _, laser = _grid(case)
    n = (case["nx"], case["ny"], case["nz"])
    k = torch.arange(n[2], dtype=F64, device="cuda").view(-1, 1, 1)
    j = torch.arange(n[1], dtype=F64, device="cuda").view(1, -1, 1)
    i = torch.arange(n[0], dtype=F64, device="cuda").view(1, 1, -1)
    out = []
    for _ in range(6):
        out.append(torch.randn(n[2], n[1], n[0], dtype=F64, device="cuda", generator=g) * 0.02)
    if case["layout"] in ("foil", "disk"):
        if case["layout"] == "foil":
            z0, z1 = _slab(case)
        else:
            z0, z1 = int(n[2] * 0.1), int(n[2] * 0.57)
        near = ((k >= z0 - 6) & (k < z1 + 6)).to(F64)  # plasma noise; vacuum elsewhere
        zc = (z0 - 4 if case["hot"] else z0 - n[2] // 4) * dx[2]
        half = n[2] * dx[2] / 12.0
        r2 = ((i + 0.5) * dx[0] - laser["xc"]) ** 2
        if case["dim"] == 3:
            r2 = r2 + (j * dx[1] - laser["yc"]) ** 2
        side = laser["a0"] * torch.exp(-r2 / laser["w0"] ** 2)
        for c in range(6):
            out[c] *= near
        for c, s in ((0, 0.0), (4, 0.5)):
            z = (k + s) * dx[2] - zc
            out[c] += side * (torch.exp(-(z / half) ** 2) * torch.sin(z))
    else:
        for c in range(6):
            ph = float(torch.rand(1, dtype=F64, device="cuda", generator=g)) * 2.0 * math.pi
            out[c] += 0.05 * torch.sin(2.0 * math.pi * ((c % 3 + 1) * i / n[0] + k / n[2]) + ph)
    return [f.reshape(-1) for f in out]


def _first_step(case):
    _, dt, laser = _grid(case)
    return int(laser["t_peak"] / dt) if laser and case["hot"] else 0


def _requests(case):
    z = zip(case["sides"].split(","), case["ppcs"].split(","), case["steps"].split(","))
    return [{"kind": "step", "layout": "plasma", "dim": 2, "order": 1, "nx": int(s), "ny": 1, "nz": int(s), "bx": 32,
             "by": 1, "bz": 32, "ppc": int(p), "steps": int(t), "uth": 0.01, "species": 1, "absorb": 0,
             "energy": False, "hot": False, "rho": False} for s, p, t in z]


# ---------------------------------------------------------------- the three calls

def prepare(case, seed):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        if case["kind"] == "serve":
            reqs = []
            for r, c in enumerate(_requests(case)):
                q, m, soa = _species(c, seed * 64 + r)[0]
                sp = {"q": q, "m": m, "id": np.arange(soa[0].numel())}
                sp.update({k: a.cpu().numpy() for k, a in zip(("x", "y", "z", "ux", "uy", "uz", "w"), soa)})
                dx, dt, _ = _grid(c)
                reqs.append((c, dx, dt, sp))
            return {"case": case, "server": Server(dim=2, max_active=16, hbm_budget_bytes=8 << 30), "requests": reqs}
        if case["kind"] == "bin":
            x, off, box = _bin_inputs(case, seed)
            np_ = case["np"]
            return {"case": case, "stream": stream, "x": x, "boxes": torch.arange(off.numel() - 1, device="cuda"),
                    "off": off, "perm": torch.empty(np_, dtype=torch.int64, device="cuda"), "box": box}
        dx, dt, laser = _grid(case)
        sim = pic.Simulation(case["dim"], (case["nx"], case["ny"], case["nz"]), (case["bx"], case["by"], case["bz"]),
                             dx, dt=dt, shape_order=case["order"], absorb_cells=case["absorb"],
                             stream=stream.cuda_stream)
        counts = []
        for q, m, soa in _species(case, seed):
            counts.append(soa[0].numel())
            sim.add_species(q, m, *soa, ids=torch.arange(counts[-1], device="cuda"))
            del soa
        if laser:
            sim.add_laser(**laser)
        for c, f in enumerate(_fields(case, seed)):
            sim.set_field(c, f)
        sim.set_step(_first_step(case))
        if case["energy"]:
            sim.set_gather(True)
        sim.set_launch(precision=case["precision"], ctas_per_sm=case["ctas"])
        if case["sched"] != "none":
            lb = dict(mode=pic.LB_DYNAMIC, interval=20, policy=pic.POLICY_KNAPSACK,
                      sched=pic.SCHED_QUEUE if case["sched"] == "queue" else pic.SCHED_LISTS)
            sim.rebalance(**lb, theta=0.0, cost=pic.COST_HEURISTIC)
            sim.set_lb_params(**lb, theta=0.10, cost=pic.COST_DEVICE_CLOCK)
        return {"case": case, "stream": stream, "sim": sim, "counts": counts}


def _bin_inputs(case, seed):
    g = _gen(seed)
    n = [case["nx"], case["ny"] if case["dim"] == 3 else 1, case["nz"]]
    box = [case["box"], case["box"] if case["dim"] == 3 else 1, case["box"]]
    x = [torch.rand(case["np"], dtype=F64, device="cuda", generator=g) * (n[a] * 0.25) for a in range(3)]
    if not case["shuffled"]:  # cell by cell along z, as a loader writes them
        x[2] = torch.sort(x[2])[0]
    nboxes = 1
    for a in range(3):
        nboxes *= n[a] // box[a]
    return x, torch.empty(nboxes + 1, dtype=torch.int64, device="cuda"), (n, box)


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        return _run_serve(state)
    with torch.cuda.stream(state["stream"]):
        if case["kind"] == "bin":
            x, (n, box) = state["x"], state["box"]
            bin_particles(case["dim"], n, box, (0.25, 0.25, 0.25), x[0], x[1] if case["dim"] == 3 else None, x[2],
                          state["off"], state["perm"], stream=state["stream"].cuda_stream)
            # the box of every particle (the order inside a box is free)
            counts = state["off"][1:] - state["off"][:-1]
            of = torch.empty_like(state["perm"])
            of[state["perm"]] = torch.repeat_interleave(state["boxes"], counts, output_size=case["np"])
            return {"offsets": state["off"], "box": of}
        sim = state["sim"]
        sim.step(case["steps"])
        cells = sim.ncells_total
        comps = list(range(pic.EX, pic.JZ + 1)) + ([pic.RHO] if case["rho"] else [])
        fields = [sim.read_field(c, torch.empty(cells, dtype=F64, device="cuda")) for c in comps]
        species = []
        for s, n in enumerate(state["counts"]):
            p = sim.particles(s, device=True)
            got = {}
            for k in ("x", "y", "z", "ux", "uy", "uz", "w"):
                if k == "y" and case["dim"] == 2:
                    continue
                got[k] = torch.zeros(n, dtype=F64, device="cuda")
                got[k][p["id"]] = p[k]
            species.append(got)
        return {"fields": fields, "species": species}


_SERVE_COMPS = (pic.EX, pic.EY, pic.EZ, pic.BY)
_SERVE_KEYS = ("x", "z", "ux", "uy", "uz", "w")


def _run_serve(state):
    srv = state["server"]
    rids = [srv.submit((c["nx"], 1, c["nz"]), (32, 1, 32), dx, c["steps"], dt=dt, species=[sp])
            for c, dx, dt, sp in state["requests"]]
    active, pending = 1, 1
    while active or pending:
        active, pending = srv.tick()
    out = []
    for rid, (c, _, _, _) in zip(rids, state["requests"]):
        fields = [srv.read_field(rid, f, (c["nx"], 1, c["nz"])) for f in _SERVE_COMPS]
        p = srv.particles(rid)
        got = {}
        for k in _SERVE_KEYS:
            got[k] = np.empty_like(p[k])
            got[k][p["id"]] = p[k]
        out.append({"fields": fields, "particles": got})
        srv.release(rid)
    return out


# ---------------------------------------------------------------- work

def _flops(dim, order):
    # gather, Boris push, Esirkepov deposit of one particle that keeps its support
    return {(3, 1): 275, (3, 2): 763, (3, 3): 1591, (2, 1): 168, (2, 2): 348, (2, 3): 546}[dim, order]


def _step_work(case):
    npart = _particles(case) * case["species"]
    cells = case["nx"] * case["ny"] * case["nz"]
    steps = case["steps"]
    # per step: a particle's seven values read and six written; a cell's E, B, J read and E, B written
    nbytes = steps * (npart * 104 + cells * 120) + npart * 56 + cells * 72
    return nbytes, steps * (npart * _flops(case["dim"], case["order"]) + cells * 39)


def work(case):
    if case["kind"] == "serve":
        w = [_step_work(c) for c in _requests(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    if case["kind"] == "bin":
        return {"bytes": case["np"] * (8 * case["dim"] + 16), "flops": case["np"] * 3 * case["dim"]}
    b, f = _step_work(case)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in plain torch, 64 bits

def _bspline(xi, order, half):
    """first node and weights at xi on the node or half-node grid"""
    t = xi - 0.5 if half else xi
    if order == 0:  # the half node whose cell holds xi
        s = torch.floor(xi)
        w = [torch.ones_like(xi)]
    elif order == 1:
        s = torch.floor(t)
        f = t - s
        w = [1.0 - f, f]
    elif order == 2:
        c = torch.floor(t + 0.5)
        d = t - c
        s = c - 1.0
        w = [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]
    else:
        fl = torch.floor(t)
        f = t - fl
        h = 1.0 - f
        s = fl - 1.0
        w = [h ** 3 / 6.0, 2.0 / 3.0 - f * f + 0.5 * f ** 3, 2.0 / 3.0 - h * h + 0.5 * h ** 3, f ** 3 / 6.0]
    return s.to(torch.int64), w


class _Plain:
    """The PIC cycle of one case: gather, Boris, Esirkepov, Yee, layers."""

    def __init__(self, case, seed, species, fields):
        self.c = case
        self.n = (case["nx"], case["ny"], case["nz"])
        self.dx, self.dt, self.laser = _grid(case)
        if case["dim"] == 2:
            self.axes = (0, 2)
        else:
            self.axes = (0, 1, 2)
        self.step_no = _first_step(case)
        shape = (self.n[2], self.n[1], self.n[0])
        self.E = [f.clone().view(shape) for f in fields[:3]]
        self.B = [f.clone().view(shape) for f in fields[3:]]
        self.J = [torch.zeros(shape, dtype=F64, device="cuda") for _ in range(3)]
        self.sp = []
        for q, m, soa in species:
            X = []
            for a in range(3):
                v = soa[a] / self.dx[a] if a in self.axes else torch.zeros_like(soa[a])
                X.append(v)
            self.sp.append([q, m, X, [u.clone() for u in soa[3:6]], soa[6],
                            torch.ones(soa[0].numel(), dtype=torch.bool, device="cuda")])

    def _flat(self, idx):
        nx, ny, nz = self.n
        return (torch.remainder(idx[2], nz) * ny + torch.remainder(idx[1], ny)) * nx + torch.remainder(idx[0], nx)

    def _gather(self, F, X, halves):
        order, ec = self.c["order"], self.c["energy"]
        S = []
        for a in range(3):
            if a not in self.axes:
                S.append((torch.zeros_like(X[a], dtype=torch.int64), [torch.ones_like(X[a])]))
            else:
                S.append(_bspline(X[a], order - 1 if ec and halves[a] else order, halves[a]))
        acc = torch.zeros_like(X[0])
        F = F.reshape(-1)
        for c, wz in enumerate(S[2][1]):
            for b, wy in enumerate(S[1][1]):
                wyz = wz * wy
                for a, wx in enumerate(S[0][1]):
                    acc += wx * wyz * F[self._flat((S[0][0] + a, S[1][0] + b, S[2][0] + c))]
        return acc

    def _deposit(self, q, X0, X1, w, vy):
        order, dim = self.c["order"], self.c["dim"]
        W = order + 3
        base, S0, S1 = [], [], []
        for a in range(3):
            if a not in self.axes:
                base.append(torch.zeros_like(X0[a], dtype=torch.int64))
                S0.append(None)
                S1.append(None)
                continue
            s0, w0 = _bspline(X0[a], order, False)
            s1, w1 = _bspline(X1[a], order, False)
            base.append(s0 - 1)
            z = torch.zeros_like(X0[a])
            S0.append([z] + w0 + [z])
            A = torch.zeros(X0[a].numel(), W, dtype=F64, device="cuda")
            A.scatter_(1, (s1 - s0 + 1).unsqueeze(1) + torch.arange(order + 1, device="cuda"), torch.stack(w1, 1))
            S1.append([A[:, l] for l in range(W)])
        dt, dx = self.dt, self.dx
        A = [None if S0[a] is None else [0.5 * (S0[a][l] + S1[a][l]) for l in range(W)] for a in range(3)]
        D = [None if S0[a] is None else [S1[a][l] - S0[a][l] for l in range(W)] for a in range(3)]
        qw = q * w
        for a in self.axes:  # the prefix currents
            o = [b for b in self.axes if b != a]
            area = 1.0
            for b in o:
                area *= dx[b]
            pre = torch.zeros_like(w)
            Ja = self.J[a].reshape(-1)
            for l in range(W - 1):
                pre = pre + D[a][l]
                pl = -qw / (area * dt) * pre
                for m in range(W):
                    if dim == 2:
                        idx = [base[0], base[1], base[2]]
                        idx[a] = base[a] + l
                        idx[o[0]] = base[o[0]] + m
                        Ja.index_add_(0, self._flat(idx), pl * A[o[0]][m])
                        continue
                    for r in range(W):
                        idx = [None, None, None]
                        idx[a], idx[o[0]], idx[o[1]] = base[a] + l, base[o[0]] + m, base[o[1]] + r
                        t = A[o[0]][m] * A[o[1]][r] + D[o[0]][m] * D[o[1]][r] / 12.0
                        Ja.index_add_(0, self._flat(idx), pl * t)
        if dim == 2:  # the current out of the plane
            Jy = self.J[1].reshape(-1)
            f = qw * vy / (dx[0] * dx[2])
            for m in range(W):
                for r in range(W):
                    t = A[0][m] * A[2][r] + D[0][m] * D[2][r] / 12.0
                    Jy.index_add_(0, self._flat((base[0] + m, base[1], base[2] + r)), f * t)

    def _push(self, sp, lo, hi):
        q, m, X, U, w, alive = sp
        sel = alive[lo:hi].nonzero().squeeze(1) + lo
        x = [X[a][sel] for a in range(3)]
        u = [U[a][sel] for a in range(3)]
        e = [self._gather(self.E[a], x, [b == a for b in range(3)]) for a in range(3)]
        b = [self._gather(self.B[a], x, [c != a for c in range(3)]) for a in range(3)]
        kq = q * self.dt / (2.0 * m)
        um = [u[a] + kq * e[a] for a in range(3)]
        t = [kq * b[a] / torch.sqrt(1.0 + um[0] ** 2 + um[1] ** 2 + um[2] ** 2) for a in range(3)]
        s = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)

        def cross(p, r):
            return [p[1] * r[2] - p[2] * r[1], p[2] * r[0] - p[0] * r[2], p[0] * r[1] - p[1] * r[0]]

        c1 = cross(um, t)
        up = [um[a] + c1[a] for a in range(3)]
        c2 = cross(up, t)
        u1 = [um[a] + s * c2[a] + kq * e[a] for a in range(3)]
        ig = 1.0 / torch.sqrt(1.0 + u1[0] ** 2 + u1[1] ** 2 + u1[2] ** 2)
        x1 = [x[a] + u1[a] * ig * (self.dt / self.dx[a]) if a in self.axes else x[a] for a in range(3)]
        self._deposit(q, x, x1, w[sel], u1[1] * ig)
        A = self.c["absorb"]
        for a in self.axes:
            if not (a == 2 and A > 0):
                v = x1[a]
                v = torch.where(v < 0.0, v + self.n[a], v)
                x1[a] = torch.where(v >= self.n[a], v - self.n[a], v)
        if A > 0:
            iz = torch.floor(x1[2])
            alive[sel] = ~((iz < A) | (iz >= self.n[2] - A))
        for a in range(3):
            X[a][sel] = x1[a]
            U[a][sel] = u1[a]

    def _curl(self, F, sgn):
        """curl by forward (sgn -1) or backward (+1) differences"""
        dims = (2, 1, 0)

        def d(f, a):
            if a not in self.axes:
                return 0.0
            g = torch.roll(f, sgn, dims[a])
            return (f - g if sgn > 0 else g - f) / self.dx[a]

        return [d(F[2], 1) - d(F[1], 2), d(F[0], 2) - d(F[2], 0), d(F[1], 0) - d(F[0], 1)]

    def step(self):
        for j in self.J:
            j.zero_()
        chunk = 1 << 22
        for sp in self.sp:
            for lo in range(0, sp[4].numel(), chunk):
                self._push(sp, lo, min(sp[4].numel(), lo + chunk))
        dt, L = self.dt, self.laser
        if L:
            t = (self.step_no + 0.5) * dt
            amp = 2.0 * L["a0"] / self.dx[2] * math.exp(-((t - L["t_peak"]) / L["tau"]) ** 2)
            amp *= math.sin(L["omega"] * (t - L["t_peak"]))
            i = (torch.arange(self.n[0], dtype=F64, device="cuda") + 0.5) * self.dx[0] - L["xc"]
            r2 = (i * i).view(1, -1)
            if self.c["dim"] == 3:
                j = torch.arange(self.n[1], dtype=F64, device="cuda") * self.dx[1] - L["yc"]
                r2 = r2 + (j * j).view(-1, 1)
            self.J[0][L["k_ant"]] += amp * torch.exp(-r2 / L["w0"] ** 2)
        for half in range(2):
            c = self._curl(self.E, -1)
            for a in range(3):
                self.B[a] = self.B[a] - 0.5 * dt * c[a]
            if half == 0:
                c = self._curl(self.B, 1)
                for a in range(3):
                    self.E[a] = self.E[a] + dt * (c[a] - self.J[a])
        A = self.c["absorb"]
        if A > 0:
            k = torch.arange(self.n[2], dtype=F64, device="cuda")
            p = torch.clamp(torch.maximum(A - k, k - (self.n[2] - 1 - A)), min=0.0)
            f = (1.0 - 0.5 * (p / A) ** 2).view(-1, 1, 1)
            for F in (self.E, self.B):
                for a in range(3):
                    F[a] = F[a] * f
        self.step_no += 1

    def rho(self):
        out = torch.zeros(self.n[0] * self.n[1] * self.n[2], dtype=F64, device="cuda")
        for q, _, X, _, w, alive in self.sp:
            S = []
            for a in range(3):
                if a not in self.axes:
                    S.append((torch.zeros_like(X[a], dtype=torch.int64), [torch.ones_like(X[a])]))
                else:
                    S.append(_bspline(X[a], self.c["order"], False))
            v = q * w / (self.dx[0] * self.dx[1] * self.dx[2]) * alive
            for c, wz in enumerate(S[2][1]):
                for b, wy in enumerate(S[1][1]):
                    for a, wx in enumerate(S[0][1]):
                        out.index_add_(0, self._flat((S[0][0] + a, S[1][0] + b, S[2][0] + c)), v * wx * wy * wz)
        return out

    def particles(self, i, keys):
        _, _, X, U, w, alive = self.sp[i]
        v = {"x": X[0] * self.dx[0], "y": X[1] * self.dx[1], "z": X[2] * self.dx[2], "ux": U[0], "uy": U[1],
             "uz": U[2], "w": w}
        return {k: v[k] * alive for k in keys}


def exact(case, seed):
    if case["kind"] == "bin":
        return None  # whole numbers
    if case["kind"] == "serve":
        out = []
        for r, c in enumerate(_requests(case)):
            sp = _species(c, seed * 64 + r)
            zero = [torch.zeros(c["nx"] * c["nz"], dtype=F64, device="cuda") for _ in range(6)]
            p = _Plain(c, seed, sp, zero)
            for _ in range(c["steps"]):
                p.step()
            F = p.E + p.B
            out.append({"fields": [F[f].reshape(c["nz"], 1, c["nx"]) for f in _SERVE_COMPS],
                        "particles": p.particles(0, _SERVE_KEYS)})
        return out
    p = _Plain(case, seed, _species(case, seed), _fields(case, seed))
    for _ in range(case["steps"]):
        p.step()
    keys = [k for k in ("x", "y", "z", "ux", "uy", "uz", "w") if not (k == "y" and case["dim"] == 2)]
    return {"fields": [f.reshape(-1) for f in p.E + p.B + p.J] + ([p.rho()] if case["rho"] else []),
            "species": [p.particles(i, keys) for i in range(case["species"])]}
