"""The work that users of the library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` one more of the same
ranges, `prepare(case, seed)` what a program holds before the call (inputs, context, resident
population), `run(state)` one pass through the public entry points, `work(case)` the bytes and
operations no implementation can do without, and `exact(case, seed)` the result in float64 from plain
numpy and torch (None where that would take too long).

Kinds of case:
  eval        tnep_eval on a trajectory: water (2 types) or the BaZrO3 perovskite (3 types)
  requests    tnep_eval_batch on a mix of open anions and periodic water boxes (6 types), host buffers
  clusters    tnep_eval_batch on open water clusters with per-atom contributions, device buffers
  cells       tnep_eval_batch_cell on small triclinic cells, host buffers
  population  tnep_population_eval: one generation of parameter vectors on resident structures
  snes        tnep_snes_run: generations of the training loop on resident structures
  spectrum    tnep_spectrum: infrared or Raman spectrum of a tensor series
  polarized   tnep_raman_tensor, then tnep_raman_porto_map on its result
"""

import math

import numpy as np
import torch

from paper_2312_05233_gb300 import tnep

RC_R, RC_A = 6.0, 4.0
N_MAX, BASIS, L_MAX, HIDDEN = 4, 8, 4, 30
DIM = (N_MAX + 1) * (L_MAX + 2)
WATER_PER_A3 = 0.033428  # molecules per cubic Angstrom at 1 g/cm^3
ANION_P = (0.4, 0.3, 0.1, 0.1, 0.05, 0.05)  # H, C, N, O, F, S
KINDS = {"ir": tnep.TNEP_SPECTRUM_IR, "iso": tnep.TNEP_SPECTRUM_RAMAN_ISO, "aniso": tnep.TNEP_SPECTRUM_RAMAN_ANISO}
CM_PER_INV_FS = 1.0 / 2.99792458e-5


def listed():
    return [
        # one step of an MD run that asks for dipole and polarizability of a small box as it goes
        {"name": "water step", "kind": "eval", "system": "water", "size": 64, "frames": 1, "ranks": "12",
         "precision": 0, "host": False},
        # the small water trajectory: many small frames in one call
        {"name": "water trajectory", "kind": "eval", "system": "water", "size": 64, "frames": 100, "ranks": "12",
         "precision": 0, "host": True},
        # bulk water, the workload of the benchmark: both tensors, split-BF16 network, frames from pinned memory
        {"name": "bulk water", "kind": "eval", "system": "water", "size": 13824, "frames": 60, "ranks": "12",
         "precision": 2, "host": True},
        # susceptibility along a perovskite trajectory: three types, frames on the device
        {"name": "perovskite", "kind": "eval", "system": "perovskite", "size": 12, "frames": 20, "ranks": "2",
         "precision": 0, "host": False},
        # what a server collects into one batch: anions and water boxes of uneven size
        {"name": "requests", "kind": "requests", "structs": 96, "max_mol": 1000, "ranks": "12", "precision": 0},
        # open clusters with per-atom contributions
        {"name": "clusters", "kind": "clusters", "structs": 61, "max_mol": 100, "ranks": "12", "precision": 0},
        # crystals in small skewed cells
        {"name": "triclinic cells", "kind": "cells", "structs": 24, "max_mol": 48, "ranks": "12", "precision": 0},
        # one generation handed over by a trainer of its own, polarizability, odd population
        {"name": "population", "kind": "population", "structs": 80, "pop": 37, "rank": 2},
        # the training loop: two generations of fifty individuals
        {"name": "training", "kind": "snes", "structs": 120, "pop": 50, "rank": 1, "generations": 2},
        # infrared spectrum of a short run
        {"name": "infrared", "kind": "spectrum", "spectrum": "ir", "steps": 2000, "max_lag": 1000, "host": False},
        # anisotropic Raman spectrum of a production run
        {"name": "raman", "kind": "spectrum", "spectrum": "aniso", "steps": 100000, "max_lag": 10000, "host": True},
        # lineshape tensor of a production run and the map over crystal orientations
        {"name": "polarized raman", "kind": "polarized", "steps": 100000, "max_lag": 2000, "angles": 181},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "requests", "clusters", "cells", "population", "snes", "spectrum",
                       "spectrum", "polarized"])
    if kind == "eval":
        system = rng.choice(["water", "water", "perovskite"])
        size = _log_int(rng, 64, 13824) if system == "water" else rng.randint(3, 12)
        ranks = rng.choice(["1", "2", "12"])
        most = 2_400_000 // _atoms(system, size)
        return {"kind": kind, "system": system, "size": size, "frames": min(_log_int(rng, 1, 500), most),
                "ranks": ranks, "precision": rng.choice([0, 1, 2]), "host": rng.random() < 0.5}
    if kind == "requests":
        return {"kind": kind, "structs": _log_int(rng, 2, 256), "max_mol": _log_int(rng, 70, 2000),
                "ranks": rng.choice(["1", "2", "12"]), "precision": rng.choice([0, 2])}
    if kind == "clusters":
        return {"kind": kind, "structs": _log_int(rng, 1, 512), "max_mol": rng.randint(10, 100),
                "ranks": rng.choice(["1", "2", "12"]), "precision": rng.choice([0, 2])}
    if kind == "cells":
        return {"kind": kind, "structs": _log_int(rng, 1, 48), "max_mol": rng.randint(6, 64),
                "ranks": rng.choice(["1", "2", "12"]), "precision": rng.choice([0, 2])}
    if kind == "population":
        return {"kind": kind, "structs": _log_int(rng, 10, 120), "pop": rng.randint(11, 60), "rank": rng.choice([1, 2])}
    if kind == "snes":
        return {"kind": kind, "structs": _log_int(rng, 10, 120), "pop": rng.randint(11, 60),
                "rank": rng.choice([1, 2]), "generations": rng.randint(1, 3)}
    if kind == "spectrum":
        steps = _log_int(rng, 200, 100000)
        return {"kind": kind, "spectrum": rng.choice(["ir", "iso", "aniso"]), "steps": steps,
                "max_lag": _log_int(rng, max(20, steps // 20), min(steps // 2, 12000)), "host": rng.random() < 0.5}
    steps = _log_int(rng, 1000, 100000)
    return {"kind": kind, "steps": steps, "max_lag": _log_int(rng, 200, min(steps // 2, 2000)),
            "angles": rng.randint(5, 181)}


# ---------------------------------------------------------------- inputs
def _atoms(system, size):
    return 3 * size if system == "water" else 5 * size ** 3


def _rotations(n, rng):
    q = rng.standard_normal((n, 4))
    q /= np.linalg.norm(q, axis=1)[:, None]
    w, x, y, z = q.T
    return np.stack([np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)], -1),
                     np.stack([2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)], -1),
                     np.stack([2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1)], 1)


def _molecules(centres, rng):
    """Randomly turned water molecules (O, H, H; 0.96 A, 104.5 degrees) at the centres."""
    half = math.radians(104.5) / 2
    mol = np.array([[0.0, 0.0, 0.0], [0.96 * math.sin(half), 0.0, 0.96 * math.cos(half)],
                    [-0.96 * math.sin(half), 0.0, 0.96 * math.cos(half)]])
    return (centres[:, None, :] + np.einsum("ka,mba->mkb", mol, _rotations(len(centres), rng))).reshape(-1, 3)


def _grid_sites(n, rng):
    """n of the sites of the smallest cubic grid that holds them, as fractions of the edge."""
    side = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    g = (np.arange(side) + 0.5) / side
    sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    return sites[np.sort(rng.choice(len(sites), size=n, replace=False))]


def _water_box(n_mol, rng):
    edge = (n_mol / WATER_PER_A3) ** (1.0 / 3.0)
    pos = _molecules(_grid_sites(n_mol, rng) * edge, rng) + 0.05 * rng.standard_normal((3 * n_mol, 3))
    pos = np.mod(pos, edge).astype(np.float32)
    return np.where(pos >= np.float32(edge), np.float32(0), pos), np.full(3, edge, np.float32)


def _water_cluster(n_mol, rng):
    side = int(math.ceil(n_mol ** (1.0 / 3.0))) + 2
    g = (np.arange(side) - (side - 1) / 2) * WATER_PER_A3 ** (-1.0 / 3.0)
    sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    order = np.argsort(np.linalg.norm(sites, axis=1) + 1e-9 * np.arange(len(sites)), kind="stable")
    pos = _molecules(sites[order[:n_mol]], rng) + 0.05 * rng.standard_normal((3 * n_mol, 3))
    return pos.astype(np.float32), np.zeros(3, np.float32)


def _anions(n, rng):
    """n open molecules of 20 to 60 atoms: bonded trees, bonds 1.0-1.5 A, no two atoms closer than 0.9 A."""
    size = rng.integers(20, 61, n)
    pos = np.full((n, 60, 3), 1e6)
    pos[:, 0] = 0.0
    have = np.ones(n, np.int64)
    while (have < size).any():
        s = np.flatnonzero(have < size)
        v = rng.standard_normal((len(s), 3))
        parent = pos[s, (rng.random(len(s)) * have[s]).astype(np.int64)]
        cand = parent + rng.uniform(1.0, 1.5, (len(s), 1)) * v / np.linalg.norm(v, axis=1, keepdims=True)
        fits = np.linalg.norm(pos[s] - cand[:, None], axis=2).min(axis=1) >= 0.9
        pos[s[fits], have[s[fits]]] = cand[fits]
        have[s[fits]] += 1
    return [(pos[k, :size[k]].astype(np.float32), rng.choice(6, size=size[k], p=ANION_P).astype(np.int32))
            for k in range(n)]


def _batch(structs):
    """(offsets, pos, box, types) of a list of (pos, types, box)."""
    offsets = np.zeros(len(structs) + 1, np.int32)
    offsets[1:] = np.cumsum([len(s[1]) for s in structs])
    return (offsets, np.concatenate([s[0] for s in structs]).astype(np.float32),
            np.stack([s[2] for s in structs]).astype(np.float32),
            np.concatenate([s[1] for s in structs]).astype(np.int32))


def _water_types(n_mol):
    return np.tile(np.array([0, 1, 1], np.int32), n_mol)


def _requests(case, rng):
    n = case["structs"]
    out = [(p, t, np.zeros(3, np.float32)) for p, t in _anions((n + 1) // 2, rng)]
    for _ in range(n // 2):
        n_mol = int(round(math.exp(rng.uniform(math.log(64), math.log(case["max_mol"])))))
        p, b = _water_box(n_mol, rng)
        out.append((p, np.where(_water_types(n_mol) == 0, 3, 0).astype(np.int32), b))
    return _batch([out[k] for k in rng.permutation(len(out))])


def _clusters(case, rng):
    out = []
    sizes = np.random.default_rng(case["structs"]).integers(1, case["max_mol"] + 1, case["structs"])
    for n_mol in sizes.tolist():  # a set of its own, whatever the seed: the per-atom results keep their shape
        p, b = _water_cluster(n_mol, rng)
        out.append((p, _water_types(n_mol), b))
    return _batch(out)


def _cells(case, rng):
    out = []
    for _ in range(case["structs"]):
        n_mol = int(rng.integers(4, case["max_mol"] + 1))
        shape = np.eye(3) * rng.uniform(0.85, 1.15, 3) + np.tril(rng.uniform(-0.25, 0.25, (3, 3)), -1)
        cell = shape * (n_mol / WATER_PER_A3 / abs(np.linalg.det(shape))) ** (1.0 / 3.0)
        out.append((_molecules(_grid_sites(n_mol, rng) @ cell, rng), _water_types(n_mol), cell.reshape(9)))
    return _batch(out)


def _training_set(case, rng):
    """Open clusters of 1 to 100 molecules and periodic boxes of 64 to 512, half of each."""
    out = []
    for k in range(case["structs"]):
        n_mol = int(rng.integers(1, 101)) if k % 2 == 0 else int(rng.choice([64, 128, 256, 512]))
        p, b = _water_cluster(n_mol, rng) if k % 2 == 0 else _water_box(n_mol, rng)
        out.append((p, _water_types(n_mol), b))
    return _batch(out)


def _trajectory(case, seed):
    """(frames [F][N][3] on the device, types, box): a random walk (water) or thermal displacements (perovskite)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["system"] == "water":
        edge = (case["size"] / WATER_PER_A3) ** (1.0 / 3.0)
        base = _molecules(_grid_sites(case["size"], rng) * edge, rng)
        types, sigma = _water_types(case["size"]), 0.01
    else:
        n, a = case["size"], 4.19
        g = np.arange(n)
        cells = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        basis = np.array([[0, 0, 0], [.5, .5, .5], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]])
        base, edge = ((cells[:, None, :] + basis[None]) * a).reshape(-1, 3), n * a
        types, sigma = np.tile(np.array([0, 1, 2, 2, 2], np.int32), len(cells)), 0.08
    step = sigma * torch.randn((case["frames"],) + base.shape, generator=gen, device="cuda")
    if case["system"] == "water":
        step = torch.cumsum(step, 0)
    edge = float(np.float32(edge))
    pos = torch.remainder(torch.as_tensor(base, dtype=torch.float32, device="cuda") + step, edge)
    pos = torch.where(pos >= edge, torch.zeros_like(pos), pos)
    return pos, types, np.full(3, edge, np.float32)


def _series(case, seed):
    """[T][3 or 9] float64: a constant tensor, damped modes with drifting phases and noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    steps, width = case["steps"], 3 if case.get("spectrum") == "ir" else 9

    def rand(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    t = torch.arange(steps, device="cuda", dtype=torch.float64)
    out = rand(1, width) + 0.01 * rand(steps, width)
    for _ in range(4):
        freq = 0.02 + 0.3 * torch.rand((), generator=gen, device="cuda", dtype=torch.float64)
        phase = torch.cumsum(0.05 * rand(steps), 0)
        out += 0.05 * torch.cos(freq * t + phase)[:, None] * rand(1, width)
    if width == 9:
        out = 0.5 * (out + out.reshape(-1, 3, 3).transpose(1, 2).reshape(-1, 9))
    return out.contiguous()


def _n_params(n_types):
    return n_types * (HIDDEN * DIM + 2 * HIDDEN + 1) + n_types ** 2 * 2 * (N_MAX + 1) * (BASIS + 1)


def _params(n_types, rng, shape=()):
    return (0.1 * rng.standard_normal(shape + (_n_params(n_types),))).astype(np.float32)


def _scaler():
    """Scales the descriptor so that the hidden layer is not saturated (radial, angular, 4-body)."""
    n = N_MAX + 1
    return np.array([0.5] * n + [5.0] * (n * L_MAX) + [100.0] * n, np.float32)


def _n_types(case):
    return {"requests": 6}.get(case["kind"], 3 if case.get("system") == "perovskite" else 2)


def _models(case, seed):
    rng = np.random.default_rng(seed + 7)
    ranks = [int(r) for r in case.get("ranks", str(case.get("rank", "")))]
    return [tnep.Model(rank=r, params=_params(_n_types(case), rng), q_scaler=_scaler(),
                       mlp_precision=case.get("precision", 0)) for r in ranks]


def _host_inputs(case, seed):
    make = {"requests": _requests, "clusters": _clusters, "cells": _cells, "population": _training_set,
            "snes": _training_set}[case["kind"]]
    return make(case, np.random.default_rng(seed))


def _individuals(case, seed):
    return _params(2, np.random.default_rng(seed + 3), (case["pop"],))


def _targets(case, seed):
    width = 3 if case["rank"] == 1 else 9
    return np.random.default_rng(seed + 5).standard_normal((case["structs"], width))


def prepare(case, seed):
    kind, state = case["kind"], {"case": case}
    if kind in ("spectrum", "polarized"):
        series = _series(case, seed)
        state["series"] = series.cpu().numpy() if case.get("host", True) else series
        if kind == "polarized":
            state["angles"] = np.linspace(0.0, math.pi, case["angles"])
        return state
    ctx = tnep.tnep_create(_models(case, seed), _n_types(case), cutoffs=(RC_R, RC_A))
    if kind == "eval":
        pos, types, box = _trajectory(case, seed)
        if case["host"]:
            state["pos"], state["types"] = pos.cpu().pin_memory(), types
        else:
            state["pos"], state["types"] = pos, torch.from_numpy(types).cuda()
        state["box"] = np.tile(box, (case["frames"], 1))
        state["ctx"] = ctx
        return state
    offsets, pos, box, types = _host_inputs(case, seed)
    if kind in ("population", "snes"):
        # a fixed form makes the training reproducible from run to run
        tnep.tnep_set_option(ctx, tnep.TNEP_OPT_POPULATION_FORM, 3)
        if kind == "population":
            state["params"] = _individuals(case, seed)
            state["population"] = tnep.tnep_population_create(ctx, 0, state["params"], offsets, pos, box, types,
                                                              _targets(case, seed))
        else:
            d = _n_params(2)
            mu0 = 0.1 * np.random.default_rng(seed + 9).standard_normal(d)
            state["snes"] = tnep.tnep_snes_create(ctx, 0, case["pop"], mu0, 0.1, offsets, pos, box, types,
                                                  _targets(case, seed), seed=seed, lambda1=0.01, lambda2=0.01)
        state["ctx"] = ctx  # after what is built on it: a dict gives its entries up in their order
        return state
    if kind == "clusters":
        pos, box, types = (torch.from_numpy(x).cuda() for x in (pos, box, types))
    state.update(offsets=offsets, pos=pos, box=box, types=types, ctx=ctx)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "eval":
        return tnep.tnep_eval(state["ctx"], state["pos"], state["box"], state["types"])
    if kind == "requests":
        return tnep.tnep_eval_batch(state["ctx"], state["offsets"], state["pos"], state["box"], state["types"])[0]
    if kind == "clusters":
        return list(tnep.tnep_eval_batch(state["ctx"], state["offsets"], state["pos"], state["box"], state["types"],
                                         per_atom=True))
    if kind == "cells":
        return tnep.tnep_eval_batch_cell(state["ctx"], state["offsets"], state["pos"], state["box"], state["types"])
    if kind == "population":
        return list(state["population"].eval(state["params"], want_out=True))
    if kind == "snes":
        history = state["snes"].run(case["generations"])
        mu, sigma, _ = state["snes"].state()
        return [history, mu, sigma]
    if kind == "spectrum":
        return list(tnep.tnep_spectrum(state["series"], 0.5, KINDS[case["spectrum"]], case["max_lag"], want_acf=True))
    freq, L = tnep.tnep_raman_tensor(state["series"], 5.0, case["max_lag"])
    return [freq, L, *tnep.tnep_raman_porto_map(L, state["angles"])]


# ---------------------------------------------------------------- work
def work(case):
    """Operations: 235 per radial pair for the moments all models share, then per model 1380 per angular
    pair and 4500 per atom (descriptor products and the network, forward and backward); transforms 5 N log2 N."""
    kind = case["kind"]
    if kind in ("spectrum", "polarized"):
        width = 3 if case.get("spectrum") == "ir" else 9
        T, M = case["steps"], case["max_lag"]
        transforms = {"ir": 4, "iso": 2, "aniso": 10}.get(case.get("spectrum"), 54)
        n_out = 3 * (M + 1) if kind == "spectrum" else (M + 1) * (82 + 2 * case["angles"])
        flops = transforms * 2.5 * (T + M) * math.log2(T + M)
        if kind == "polarized":
            flops += 2.0 * 2 * 81 * case["angles"] * (M + 1)
        return {"bytes": 8.0 * (T * width + n_out), "flops": flops}
    if kind == "eval":
        n, structs = _atoms(case["system"], case["size"]) * case["frames"], case["frames"]
        radial, angular = (100.0, 26.0) if case["system"] == "water" else (75.0, 20.0)
    else:
        mean = {"requests": lambda: 20 + 1.5 * (case["max_mol"] - 64) / math.log(case["max_mol"] / 64.0),
                "clusters": lambda: 1.5 * case["max_mol"], "cells": lambda: 1.5 * (case["max_mol"] + 4)}
        n = case["structs"] * mean.get(kind, lambda: 450.0)()
        structs = case["structs"]
        radial, angular = (100.0, 26.0) if kind in ("cells",) else (75.0, 22.0)
    ranks = case.get("ranks", str(case.get("rank", "")))
    models = len(ranks) * case.get("pop", 1) * case.get("generations", 1)
    width = sum(3 if r == "1" else 9 for r in ranks)
    shared = 0.0 if kind in ("population", "snes") else 235.0 * radial  # resident structures keep the moments
    flops = n * (shared + models * (1380.0 * angular + 4500.0))
    out = 8.0 * structs * width * case.get("pop", 1) + (4.0 * n * width if kind == "clusters" else 0.0)
    return {"bytes": 12.0 * n + 4.0 * n / (case.get("frames", 1)) + out, "flops": flops}


# ---------------------------------------------------------------- results in 64 bits
def _pairs(pos, H, offsets):
    """Centre, neighbour and r_ij of every pair within RC_R, structure by structure: all images for a cell
    (rows of H, zeros = open)."""
    ci, cj, cr = [], [], []
    for s in range(len(offsets) - 1):
        a, b = int(offsets[s]), int(offsets[s + 1])
        p, cell = pos[a:b], H[s]
        shifts = np.zeros((1, 3))
        if np.abs(cell).sum() > 0:
            inv = np.linalg.inv(cell)
            f = p @ torch.as_tensor(inv, device=p.device)
            p = (f - torch.floor(f)) @ torch.as_tensor(cell, device=p.device)
            k = [int(math.ceil(RC_R * np.linalg.norm(inv[:, d]))) for d in range(3)]
            shifts = np.stack(np.meshgrid(*[np.arange(-m, m + 1) for m in k], indexing="ij"), -1).reshape(-1, 3) @ cell
        for sh in shifts:
            q = p + torch.as_tensor(sh, device=p.device)
            rows = max(1, 20_000_000 // max(len(p), 1))
            for c0 in range(0, len(p), rows):
                d = q[None] - p[c0:c0 + rows, None]
                r2 = (d * d).sum(-1)
                i, j = torch.nonzero((r2 < RC_R ** 2) & (r2 > 1e-12), as_tuple=True)
                ci.append(a + c0 + i), cj.append(a + j), cr.append(d[i, j])
    order = torch.argsort(torch.cat(ci), stable=True)
    return torch.cat(ci)[order], torch.cat(cj)[order], torch.cat(cr)[order]


def _basis(r, rc):
    x = 2 * (r / rc - 1) ** 2 - 1
    fc = 0.5 * (1 + torch.cos(math.pi * r / rc))
    t = [torch.ones_like(x), x]
    for _ in range(2, BASIS + 1):
        t.append(2 * x * t[-1] - t[-2])
    return torch.stack([(v + 1) * 0.5 * fc for v in t], -1)


def _per_atom(rank, params, n_types, types, pairs):
    """[N][3 or 9] contributions of every atom.  Sums over pairs of neighbours of P_l(cos) come from the
    Cartesian moments of the unit vectors, the 4-body term from the trace of the traceless second moment."""
    dev, n = types.device, N_MAX + 1
    w = torch.as_tensor(params, dtype=torch.float64, device=dev)
    per = HIDDEN * DIM + 2 * HIDDEN + 1
    nets = w[:n_types * per].reshape(n_types, per)
    W0, b0 = nets[:, :HIDDEN * DIM].reshape(-1, HIDDEN, DIM), nets[:, HIDDEN * DIM:HIDDEN * (DIM + 1)]
    w1, b1 = nets[:, HIDDEN * (DIM + 1):HIDDEN * (DIM + 2)], nets[:, -1]
    cR, cA = w[n_types * per:].reshape(2, n_types, n_types, n, BASIS + 1)
    scaler = torch.as_tensor(_scaler(), dtype=torch.float64, device=dev)
    c4 = -math.sqrt(2.0 / 35.0) * (5.0 / (4.0 * math.pi)) ** 1.5 * 4.5
    pi, pj, pr = pairs
    N = len(types)
    out = torch.empty((N, 3 if rank == 1 else 9), dtype=torch.float64, device=dev)
    start = torch.searchsorted(pi, torch.arange(N + 1, device=dev))
    for a in range(0, N, 20000):
        b = min(N, a + 20000)
        lo, hi = int(start[a]), int(start[b])
        r = pr[lo:hi].clone().requires_grad_(True)
        i, m = pi[lo:hi] - a, b - a
        ti, tj = types[pi[lo:hi]], types[pj[lo:hi]]
        dist = r.norm(dim=1)
        q = [torch.zeros((m, n), dtype=torch.float64, device=dev).index_add(
            0, i, torch.einsum("pnk,pk->pn", cR[ti, tj], _basis(dist, RC_R)))]
        near = dist.detach() < RC_A
        i, ti, tj, dn = i[near], ti[near], tj[near], dist[near]
        u = r[near] / dn[:, None]
        g = torch.einsum("pnk,pk->pn", cA[ti, tj], _basis(dn, RC_A))
        power, moments = torch.ones((len(dn), 1), dtype=torch.float64, device=dev), []
        for _ in range(5):
            terms = (g[:, :, None] * power[:, None, :])
            moments.append(torch.zeros((m, n, power.shape[1]), dtype=torch.float64, device=dev).index_add(0, i, terms))
            power = (power[:, :, None] * u[:, None, :]).flatten(1)
        s = [(v * v).sum(-1) for v in moments]
        q += [s[1], (3 * s[2] - s[0]) / 2, (5 * s[3] - 3 * s[1]) / 2, (35 * s[4] - 30 * s[2] + 3 * s[0]) / 8]
        M = moments[2].reshape(m, n, 3, 3) - moments[0][..., None] * torch.eye(3, dtype=torch.float64, device=dev) / 3
        q.append(c4 * torch.einsum("inab,inbc,inca->in", M, M, M))
        t = types[a:b]
        U = torch.zeros(m, dtype=torch.float64, device=dev)
        x = torch.cat(q, 1) * scaler
        for k in range(n_types):
            U = U + (t == k) * ((torch.tanh(x @ W0[k].T - b0[k]) * w1[k]).sum(1) - b1[k])
        (f,) = torch.autograd.grad(U.sum(), r)
        rr, i = r.detach(), pi[lo:hi] - a
        if rank == 1:
            c = -(rr * rr).sum(1, keepdim=True) * f
        else:
            c = -(rr[:, :, None] * f[:, None, :]).flatten(1)
        acc = torch.zeros((m, c.shape[1]), dtype=torch.float64, device=dev).index_add(0, i, c)
        if rank == 2:
            acc = acc + U.detach()[:, None] * torch.eye(3, dtype=torch.float64, device=dev).flatten()
        out[a:b] = acc
    return out


def _sums(per_atom, offsets):
    S = len(offsets) - 1
    sizes = torch.as_tensor(np.diff(offsets), device=per_atom.device)
    which = torch.repeat_interleave(torch.arange(S, device=per_atom.device), sizes)
    return torch.zeros((S, per_atom.shape[1]), dtype=torch.float64, device=per_atom.device).index_add(0, which, per_atom)


def _exact_tensors(case, seed):
    if case["kind"] == "eval":
        pos, types, box = _trajectory(case, seed)
        F, N = pos.shape[:2]
        offsets, types = np.arange(F + 1) * N, np.tile(types, F)
        pos, boxes = pos.reshape(-1, 3), np.tile(box, (F, 1))
    else:
        offsets, pos, boxes, types = _host_inputs(case, seed)
    pos = torch.as_tensor(pos, device="cuda").double()
    types = torch.as_tensor(types, device="cuda").long()
    H = boxes.astype(np.float64)
    H = H.reshape(-1, 3, 3) if H.shape[1] == 9 else np.stack([np.diag(b) for b in H])
    pairs = _pairs(pos, H, offsets)
    if case["kind"] == "population":
        pred = torch.stack([_sums(_per_atom(case["rank"], p, 2, types, pairs), offsets)
                            for p in _individuals(case, seed)])
        diff = pred - torch.as_tensor(_targets(case, seed), device="cuda")
        return [diff.square().mean((1, 2)).sqrt(), pred]
    atoms = [_per_atom(m.rank, m.params, _n_types(case), types, pairs) for m in _models(case, seed)]
    sums = [_sums(a, offsets) for a in atoms]
    return [sums, atoms] if case["kind"] == "clusters" else sums


def _cosine(c, dt):
    """dt [c(0) + 2 sum_tau c(tau) cos(pi k tau / M)] along the last axis (tau = 0..M)."""
    y = torch.cat([c[..., :-1], 2 * c[..., -1:], c[..., 1:-1].flip(-1)], -1)
    return dt * torch.fft.rfft(y).real


def _correlations(x, y, M):
    """Sum over t of x(t) y(t + tau), tau = 0..M, along the last axis."""
    N = 1 << (x.shape[-1] + M).bit_length()
    return torch.fft.irfft(torch.fft.rfft(x, N).conj() * torch.fft.rfft(y, N), N)[..., :M + 1]


def _exact_spectra(case, seed):
    x = _series(case, seed)
    T, M = x.shape[0], case["max_lag"]
    count = T - torch.arange(M + 1, device="cuda", dtype=torch.float64)
    if case["kind"] == "spectrum":
        dt, kind = 0.5, case["spectrum"]
        freq = torch.arange(M + 1, device="cuda", dtype=torch.float64) / (2 * M * dt)
        if kind != "ir":
            gamma = (x[:, 0] + x[:, 4] + x[:, 8])[:, None] / 3
            x = gamma if kind == "iso" else x - gamma * torch.eye(3, dtype=torch.float64, device="cuda").flatten()
        x = (x - x.mean(0)).T
        y = x.reshape(3, 3, T).transpose(0, 1).reshape(9, T) if kind == "aniso" else x
        acf = _correlations(x, y, M).sum(0) / count / (3 if kind == "ir" else 1)
        spec = _cosine(acf, dt)
        if kind == "ir":
            spec = spec * (2 * math.pi * freq) ** 2
        return [freq * CM_PER_INV_FS, spec, acf]
    dt = 5.0
    x = (x - x.mean(0)).T
    L = torch.empty((M + 1, 9, 9), dtype=torch.float64, device="cuda")
    for p in range(9):
        C = (_correlations(x[p:p + 1], x, M) + _correlations(x, x[p:p + 1], M)) / (2 * count)
        L[:, p] = _cosine(C, dt).T
    freq = torch.arange(M + 1, device="cuda", dtype=torch.float64) / (2 * M * dt) * CM_PER_INV_FS
    th = torch.as_tensor(np.linspace(0.0, math.pi, case["angles"]), device="cuda")
    zero = torch.zeros_like(th)
    e, y = torch.stack([th.cos(), -th.sin(), zero], 1), torch.stack([th.sin(), th.cos(), zero], 1)
    maps = []
    for seen in (e, y):
        wv = (seen[:, :, None] * e[:, None, :]).flatten(1)
        maps.append(torch.einsum("op,kpq,oq->ok", wv, L, wv))
    return [freq, L, *maps]


def exact(case, seed):
    kind = case["kind"]
    if kind == "snes":
        return None  # the run depends on its own stream of normals
    if kind in ("spectrum", "polarized"):
        return _exact_spectra(case, seed)
    atoms = _atoms(case["system"], case["size"]) * case["frames"] if kind == "eval" else 0
    if atoms > 600_000:
        return None
    return _exact_tensors(case, seed)
