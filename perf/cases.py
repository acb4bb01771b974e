"""The calls by which this framework's speed is measured.

A case is one call, or one short chain of calls, through the public entry points,
as a program that simulates sputter depositions makes it.  What such a program
keeps (the scene resident on the GPU with its tables, the tally tensors, a captured
graph, the measurement patches) is made in ``prepare``; ``run`` is one pass and
returns every tally or map it writes.

Fields of a case:
  call      "run"       one transport launch into device tallies (Transport.run)
            "graph"     the same, replayed from a CUDA graph
            "host"      the same into host arrays (sput_run_host)
            "maps"      composition maps of several libraries (library.composition_maps)
            "gradient"  forward and backward of a composition map (adjoint.CompositionMap)
            "saved"     composition map and its backward pass from saved tallies
  scene     name of a builder of ``workloads``
  n         atoms per instance, or the upper end of the instances' range (sweep)
  pressure  Pa; the sweep's highest one
"""

import ctypes
import math

import numpy as np
import torch

import workloads
from paper_2411_14413_gb300 import Transport, _native, library, run_opts, sput_graph_create, sput_graph_destroy, \
    sput_graph_launch, sput_run_host
from paper_2411_14413_gb300.adjoint import MapSetup, composition_function
from workloads.measurement import calibration_points, measurement_patches, voltage_points

N_POINTS = 342
QUATERNARY = ("Ni", "Pd", "Pt", "Ru")
POWERS = {"Ni": 20.0, "Pd": 30.0, "Pt": 15.0, "Ru": 20.0}


def listed():
    return [
        # A first look at a new chamber: a few thousand atoms, all latency and launches.
        {"name": "single_ni_3e3", "call": "run", "scene": "single_ni", "n": 3001, "pressure": 0.5},
        # The single-cathode simulation at its usual size: 1e5 atoms, 50 x 50 int32 counts.
        {"name": "single_ni_1e5", "call": "run", "scene": "single_ni", "n": 100_000, "pressure": 0.5},
        # A control loop that replays a small co-sputter simulation from a CUDA graph.
        {"name": "quaternary_graph_1e5", "call": "graph", "scene": "quaternary", "n": 100_003, "pressure": 0.5},
        # The same from a program without device buffers: tallies come back into host arrays.
        {"name": "quaternary_host_1e6", "call": "host", "scene": "quaternary", "n": 1_000_000, "pressure": 0.3},
        # Co-sputtering from four cathodes at production statistics: the headline workload.
        {"name": "quaternary_1e7", "call": "run", "scene": "quaternary", "n": 10_000_000, "pressure": 0.5},
        # Pressure and temperature sensitivities (score tallies) in a warm gas.
        {"name": "quaternary_scores", "call": "run", "scene": "quaternary", "n": 250_001, "pressure": 1.0, "T": 500.0,
         "score": True, "score_T": True},
        # A process map: 512 conditions (4 cathodes, 16 pressures, 8 tilts) of uneven counts in one launch.
        {"name": "sweep_512", "call": "run", "scene": "sweep", "n": 200_000, "pressure": 2.0},
        # A shielded chamber at high pressure: hundreds of collisions per atom, 64 surfaces, histograms.
        {"name": "shielded_3pa", "call": "run", "scene": "large", "n": 1_000_000, "pressure": 3.0},
        # The same chamber with the diffusion shortcut for thermalised atoms.
        {"name": "shielded_diffusion", "call": "run", "scene": "large", "n": 4_000_000, "pressure": 3.0,
         "switch_eV": 0.1},
        # Launches from a tabulated angle-energy distribution, an odd grid.
        {"name": "launch_table_1e6", "call": "run", "scene": "single_ni_table", "n": 1_000_000, "pressure": 1.0,
         "nx": 127, "ny": 93, "energy": True},
        # One step of the inverse solve: map, loss gradient, boundary run, gradients in pressure and powers.
        {"name": "gradient_step", "call": "gradient", "scene": "quaternary", "n": 1_000_000, "pressure": 0.5},
        # Post-processing of saved tallies: the composition map and its gradients, no transport.
        {"name": "saved_map", "call": "saved", "scene": "quaternary", "n": 1_000_000, "pressure": 0.5},
    ]


# collisions per atom at these pressures (measured counts of the scenes at 300 K)
_PRESSURES = (0.2, 0.5, 1.0, 2.0, 3.0)
_COLLISIONS = {"single_ni": (5.6, 34.9, 165.0, 587.0, 1059.0), "single_ni_table": (4.8, 29.3, 152.0, 605.0, 1159.0),
               "quaternary": (4.9, 23.3, 106.0, 408.0, 784.0), "large": (3.7, 16.6, 72.4, 293.0, 567.0)}
_COLLISIONS["tilt_scan"] = _COLLISIONS["sweep"] = _COLLISIONS["quaternary"]
_PRIMS = {"single_ni": 7, "single_ni_table": 7, "quaternary": 16, "sweep": 16, "tilt_scan": 16, "large": 64}
_MOST_COLLISIONS = 9.0e8


def _instances(case):
    return {"quaternary": 4, "sweep": 512, "tilt_scan": 3 * int(case.get("tilts", 8))}.get(case["scene"], 1)


def _per_atom(scene, pressure):
    return math.exp(np.interp(math.log(pressure), np.log(_PRESSURES), np.log(_COLLISIONS[scene])))


def _collisions(case):
    """Estimate of a pass's collisions (steps of the walk for atoms under the diffusion shortcut)."""
    scene, p = case["scene"], case["pressure"] * 300.0 / case.get("T", 300.0)  # the density counts
    n = case["n"] * _instances(case)
    if scene == "sweep":  # counts uniform up to n; pressures log-spaced over the decade below p
        n, per = 0.5 * n, float(np.mean([_per_atom(scene, q) for q in np.geomspace(0.1 * p, p, 16)]))
    else:
        per = _per_atom(scene, p)
    if case.get("switch_eV", 0.0) > 0.0:
        per *= 0.25
    return n * per * (2.0 if case["call"] == "gradient" else 1.0)


def draw(rng):
    """One more case over the listed ones' ranges: any call and scene, sizes spread over their logarithm."""
    call, scene = rng.choice([("run", "single_ni"), ("run", "single_ni_table"), ("run", "quaternary"),
                              ("run", "quaternary"), ("run", "large"), ("run", "large"), ("run", "sweep"),
                              ("graph", "single_ni"), ("graph", "quaternary"), ("host", "quaternary"),
                              ("maps", "tilt_scan"), ("gradient", "quaternary"), ("saved", "quaternary")])
    case = {"call": call, "scene": scene}
    lo, hi = {"sweep": (2e3, 2e5), "tilt_scan": (2e4, 1e6)}.get(scene, (1e5, 1e8) if call == "saved" else (1e3, 1e7))
    case["n"] = int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1
    case["pressure"] = round(math.exp(rng.uniform(math.log(0.2), math.log(3.0))), 4)
    if scene == "sweep":
        case["pressure"] = round(rng.uniform(1.0, 2.5), 4)
    if call in ("run", "host", "graph") and scene != "sweep":
        case["nx"], case["ny"] = rng.randint(33, 400), rng.randint(33, 400)
        case["T"] = round(rng.uniform(280.0, 600.0), 1)
        case["E_i"] = round(rng.uniform(250.0, 500.0), 1)
        case["energy"] = rng.random() < 0.6
        case["score"] = rng.random() < 0.3
    if call == "run" and scene in ("single_ni", "large") and rng.random() < 0.4:
        case["switch_eV"] = round(rng.uniform(0.05, 0.15), 3)
    elif call == "run" and scene == "quaternary":
        case["tilt"] = round(rng.uniform(0.0, 40.0), 2)
        case["score_T"] = rng.random() < 0.3
    if call == "maps":
        case["tilts"] = rng.randint(2, 8)
    if call == "saved":
        case["nx"] = case["ny"] = rng.randrange(100, 600, 2)
    over = _collisions(case) / _MOST_COLLISIONS
    if over > 1.0 and call != "saved":
        case["n"] = max(1001, int(case["n"] / over)) | 1
    return case


def _scene(case, seed):
    name, n = case["scene"], int(case["n"])
    kw = {"T": float(case.get("T", 300.0)), "E_i": float(case.get("E_i", 400.0)), "seed": int(seed)}
    if "nx" in case:
        kw["nx"], kw["ny"] = int(case["nx"]), int(case["ny"])
    if case.get("switch_eV", 0.0) > 0.0:
        kw["physics"] = {"thermal_switch_eV": float(case["switch_eV"])}
    p = float(case["pressure"])
    if name == "sweep":
        return workloads.scene_by_name(name, n_range=(max(1, n // 100), n), p_range=(0.1 * p, p), counts_seed=seed, **kw)
    if name == "tilt_scan":
        tilts = np.linspace(27.0, 34.0, int(case["tilts"]))
        return workloads.scene_by_name(name, tilts=[float(t) for t in tilts], n_per_cathode=n, pressure=p, **kw)
    if name == "quaternary":
        return workloads.scene_by_name(name, n_per_cathode=n, pressure=p, tilt_deg=float(case.get("tilt", 30.0)), **kw)
    return workloads.scene_by_name(name, n=n, pressure=p, **kw)


def _calibration(elements):
    rows = []
    for e in elements:
        (pa, ra), (pb, rb) = calibration_points(e)
        el = workloads.element(e)
        rows.append([pa, ra, pb, rb, el.density, el.mass])
    return np.array(rows)


def _voltage(elements):
    return np.array([[pa, va, pb, vb] for (pa, va), (pb, vb) in map(voltage_points, elements)])


class _Graph:
    """A captured run of a Transport, released with it."""

    def __init__(self, tr):
        self.tr = tr
        stream = torch.cuda.current_stream().cuda_stream
        self.g = sput_graph_create(tr.h, run_opts(seed=tr.scene.seed), stream, tr._tal)

    def __del__(self):
        sput_graph_destroy(self.g)


def _saved_inputs(case, seed):
    """Tallies as an earlier deposition left them (about n atoms per cathode, peaked towards the
    cathode's side, noisy scores) and a loss gradient of the map, on the GPU."""
    nx, ny = int(case.get("nx", 200)), int(case.get("ny", 200))
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kw = {"device": "cuda", "dtype": torch.float64}
    y = torch.linspace(-1.0, 1.0, ny, **kw)[:, None]
    x = torch.linspace(-1.0, 1.0, nx, **kw)[None, :]
    az = torch.arange(4, **kw) * (math.pi / 2.0)
    shape = torch.exp(-0.8 * ((x - 0.4 * torch.cos(az)[:, None, None]) ** 2 + (y - 0.4 * torch.sin(az)[:, None, None]) ** 2))
    mean = 0.3 * case["n"] * shape / shape.sum(dim=(1, 2), keepdim=True)
    counts = torch.poisson(mean, generator=gen)
    score = torch.randn(mean.shape, generator=gen, **kw) * torch.sqrt(20.0 * counts) - 0.2 * counts
    grad = torch.randn((N_POINTS, 4), generator=gen, **kw)
    return counts.to(torch.int64), score, grad


def prepare(case, seed):
    call = case["call"]
    s = {"call": call, "seed": int(seed)}
    if call in ("maps", "gradient", "saved"):
        elements = ("Pd", "Pt", "Ru") if call == "maps" else QUATERNARY
        scene_case = dict(case, n=1000) if call == "saved" else case
        sc = _scene(scene_case, seed)
        g = sc.grid
        s["power"] = np.array([POWERS[e] for e in elements])
        cal = _calibration(elements)
        patch, _, ref = measurement_patches(nx=g["nx"], ny=g["ny"])
        if call == "maps":
            s.update(tr=Transport(sc, energy=False, prim_counts=False), patch=patch, ref=ref, cal=cal, n_el=len(elements))
        elif call == "saved":
            s["setup"] = setup = MapSetup(sc, patch, ref, cal)
            counts, score, s["grad"] = _saved_inputs(case, seed)
            setup.tr.t["counts"].copy_(counts)
            setup.tr.t["score"].copy_(score)
        else:
            s["setup"] = MapSetup(sc, patch, ref, cal, voltage=_voltage(elements))
            s["function"] = composition_function()
            s["log_p"] = torch.tensor(math.log(case["pressure"]), dtype=torch.float64, device="cuda", requires_grad=True)
            s["log_power"] = torch.tensor(np.log(s["power"]), device="cuda", requires_grad=True)
            gen = torch.Generator(device="cuda").manual_seed(int(seed))
            s["target"] = 25.0 + 3.0 * torch.randn((N_POINTS, 4), dtype=torch.float64, device="cuda", generator=gen)
        return s
    sc = _scene(case, seed)
    if call == "host":
        s["tr"] = tr = Transport(sc, energy=False, prim_counts=False)
        L = tr.layout
        ni = L.n_instances
        s["host"] = host = {"counts": np.zeros((ni, L.ny, L.nx), np.int64), "energy": np.zeros((ni, L.ny, L.nx)),
                            "prim_counts": np.zeros((ni, L.max_prims), np.int64), "timed_out": np.zeros(ni, np.int64)}
        if not case.get("energy", True):
            del host["energy"]
        if case.get("score", False):
            host["score"] = np.zeros((ni, L.ny, L.nx))
        s["tallies"] = t = _native.sput_tallies()
        for k, v in host.items():
            setattr(t, k, v.ctypes.data)
        return s
    s["tr"] = Transport(sc, energy=case.get("energy"), score=case.get("score", False),
                        score_T=case.get("score_T", False))
    if call == "graph":
        s["graph"] = _Graph(s["tr"])
    return s


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def run(s):
    call = s["call"]
    if call == "run":
        s["tr"].run(seed=s["seed"], want_stats=False)
        return s["tr"].t
    if call == "graph":
        sput_graph_launch(s["graph"].g, s["seed"], torch.cuda.current_stream().cuda_stream)
        return s["tr"].t
    if call == "host":
        sput_run_host(s["tr"].h, run_opts(seed=s["seed"]), s["tallies"])
        return s["host"]
    if call == "maps":
        return library.composition_maps(s["tr"], s["n_el"], s["patch"], s["ref"], s["cal"], s["power"], seed=s["seed"])
    if call == "saved":
        m = s["setup"]
        rc = _native.load().sput_composition(m.n_cath, m.n_cells, m.n_points, _ptr(m.tr.t["counts"]), _ptr(m.patch),
                                             m.ref, m.cal.ctypes.data_as(ctypes.c_void_p),
                                             s["power"].ctypes.data_as(ctypes.c_void_p), _ptr(m.patch_counts),
                                             _ptr(m.comp), ctypes.c_void_p(m.stream()))
        _native.check(rc, "sput_composition")
        grad_logp, grad_power = m.backward(s["grad"], s["power"])
        return {"composition": m.comp, "patch_counts": m.patch_counts, "grad_counts": m.grad_counts,
                "grad_logp": grad_logp, "grad_power": grad_power}
    s["log_p"].grad = s["log_power"].grad = None
    comp = s["function"].apply(s["log_p"], torch.exp(s["log_power"]), s["setup"], s["seed"])
    loss = ((comp - s["target"]) ** 2).mean()
    loss.backward()
    m = s["setup"]
    return {"composition": comp.detach(), "loss": loss.detach(), "grad_log_p": s["log_p"].grad,
            "grad_log_power": s["log_power"].grad, "grad_ion_energy": m.grad_Ei, "counts": m.tr.t["counts"],
            "score": m.tr.t["score"]}


def work(case):
    """Lane operations of the method (as the benchmark counts them: random words, flights, surface tests,
    partner draws, collisions, launches) and the bytes of the tallies, each written once."""
    sc_cells = {"single_ni": 2500, "single_ni_table": 2500, "sweep": 10000, "large": 512 * 512}.get(case["scene"], 40000)
    cells = int(case["nx"]) * int(case["ny"]) if "nx" in case else sc_cells
    ni = _instances(case)
    if case["call"] == "saved":
        # counts, scores, patch ids and the map's gradient in; map, patch counts and gradients out
        return {"bytes": ni * cells * 24 + cells * 4 + N_POINTS * ni * 24, "flops": ni * cells * 3 + N_POINTS * ni * 20}
    n = case["n"] * ni * (0.5 if case["scene"] == "sweep" else 1.0) * (2.0 if case["call"] == "gradient" else 1.0)
    coll = _collisions(case)
    flights = coll + n
    ops = flights * (116 + 25 * _PRIMS[case["scene"]]) + 1.25 * coll * 135 + coll * 78 + n * 280
    tallies = 1 + int(bool(case.get("energy", case["scene"] in ("quaternary", "large")))) + int(bool(case.get("score")))
    return {"bytes": ni * cells * 8 * tallies, "flops": ops}


def exact(case, seed):
    """The map and gradients of saved tallies in 64 bits.  A transport has no such value: its counts
    are whole numbers, and its sums follow each atom's own random path."""
    if case["call"] != "saved":
        return None
    counts, score, grad = (t.cpu().numpy() for t in _saved_inputs(case, seed))
    elements = QUATERNARY
    nx, ny = int(case.get("nx", 200)), int(case.get("ny", 200))
    patch, _, ref = measurement_patches(nx=nx, ny=ny)
    n_points = int(patch.max()) + 1
    cal = _calibration(elements)
    power = np.array([POWERS[e] for e in elements])
    inside = patch >= 0
    N = np.stack([np.bincount(patch[inside], weights=c.reshape(-1)[inside], minlength=n_points) for c in counts])
    slope = (cal[:, 3] - cal[:, 1]) / (cal[:, 2] - cal[:, 0])
    R = cal[:, 1] + slope * (power - cal[:, 0])
    w = cal[:, 4] / cal[:, 5]
    nref = N[:, ref]
    a = R[:, None] * N / nref[:, None] * w[:, None]
    A = a.sum(axis=0)
    comp = 100.0 * a / A
    g = grad.T
    ga = 100.0 / A * (g - (g * comp).sum(axis=0) / 100.0)
    gN = ga * (R * w / nref)[:, None]
    gN[:, ref] -= (ga * a).sum(axis=1) / nref
    g_power = (ga * a).sum(axis=1) / R * slope
    g_counts = np.where(inside, gN[:, np.where(inside, patch, 0)], 0.0)
    g_logp = (g_counts * score.reshape(len(elements), -1)).sum(axis=1)
    return {"composition": comp.T.copy(), "patch_counts": N, "grad_counts": g_counts, "grad_logp": g_logp,
            "grad_power": g_power}
