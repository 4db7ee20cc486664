"""Performance cases: the calls users of the potential make, over their sizes.

    listed()             the cases, dicts of plain values
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  a user's inputs, buffers and Potential handle on the GPU
    run(state)           one pass through the public entry points
    work(case)           bytes and FLOPs one pass cannot do without
    exact(case, seed)    run's outputs in 64 bits, from plain torch

Energies and virials are returned as float32: they are sums of FP32 atomic terms
(the double that carries the sum has no more information than that), and float32
is what a training loss or an integrator of float32 coordinates takes them as.
"""
from __future__ import annotations

import functools
import math
import types

import numpy as np
import torch

# ---------------------------------------------------------------- models
SPECIES = {"ani4": (1, 6, 7, 8), "ani7": (1, 6, 7, 8, 16, 9, 17), "ani7x8": (1, 6, 7, 8, 16, 9, 17)}
HIDDEN = {"ani4": (160, 128, 96), "ani7": (256, 192, 160), "ani7x8": (256, 192, 160)}
ENSEMBLE = {"ani4": 1, "ani7": 1, "ani7x8": 8}
RC_R, RC_A, ETA_R, ETA_A, ZETA, ALPHA = 5.2, 3.5, 16.0, 8.0, 32.0, 0.1
SHF_R = tuple(0.9 + r * (5.2 - 0.9) / 16.0 for r in range(16))
SHF_A = tuple(0.9 + a * (3.5 - 0.9) / 4.0 for a in range(4))
SHF_Z = tuple((2 * z + 1) * math.pi / 16.0 for z in range(8))
H, C, N, O, S, F, CL = range(7)
# how often a species occurs: small organic molecules, and the solutes of boxes
ORGANIC = {H: 12, C: 7, N: 3, O: 2}
SOLUTE = {C: 0.35, H: 0.45, N: 0.07, O: 0.08, S: 0.02, F: 0.015, CL: 0.015}
WATER_VOLUME = 44.77 ** 3 / 3000   # A^3 per molecule at 1 g/cm^3


def _dim(model):
    s = len(SPECIES[model])
    return 16 * s + 32 * (s * (s + 1) // 2)


def _widths(model):
    return (_dim(model),) + HIDDEN[model] + (1,)


def _spec(model):
    aev = types.SimpleNamespace(n_species=len(SPECIES[model]), rc_r=RC_R, eta_r=ETA_R, shf_r=SHF_R, rc_a=RC_A,
                                eta_a=ETA_A, zeta=ZETA, shf_a=SHF_A, shf_z=SHF_Z, cos_scale=1.0)
    return types.SimpleNamespace(aev=aev, widths=_widths(model), n_ensemble=ENSEMBLE[model], celu_alpha=ALPHA,
                                 atomic_numbers=SPECIES[model])


@functools.lru_cache(maxsize=4)
def _weights(model):
    """The model's parameters (a user loads one trained model: the same for every seed),
    U(-1/sqrt(fan_in), 1/sqrt(fan_in)) per layer, flat [member][species][layer] (W, b)."""
    rng = np.random.Generator(np.random.PCG64(1))
    w, out = _widths(model), []
    for _ in range(ENSEMBLE[model] * len(SPECIES[model])):
        for l in range(4):
            b = 1.0 / math.sqrt(w[l])
            out.append(rng.uniform(-b, b, size=w[l + 1] * w[l] + w[l + 1]))
    return np.concatenate(out).astype(np.float32)


# ---------------------------------------------------------------- geometries
def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _species_counts(fractions, n, rng):
    k = np.array(list(fractions), dtype=np.uint8)
    raw = np.array([fractions[i] for i in fractions], dtype=float)
    raw *= n / raw.sum()
    cnt = np.floor(raw).astype(int)
    cnt[np.argsort(cnt - raw, kind="stable")[:n - cnt.sum()]] += 1
    sp = np.repeat(k, cnt)
    rng.shuffle(sp)
    return sp


def _molecule(rng, n, fractions):
    """n atoms uniform in a cube at 0.024 atoms/A^3, no pair closer than 0.9 A."""
    edge, pts, k = (n / 0.024) ** (1 / 3), np.empty((n, 3)), 0
    while k < n:
        p = rng.uniform(0.0, edge, size=3)
        if k == 0 or np.min(np.sum((pts[:k] - p) ** 2, axis=1)) >= 0.81:
            pts[k] = p
            k += 1
    return pts.astype(np.float32), _species_counts(fractions, n, rng)


def _rotations(rng, n):
    q = rng.normal(size=(n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=1).reshape(n, 3, 3)


def _waters(rng, centres):
    """Rigid waters (O-H 0.96 A, 104.5 deg) in random orientations, atoms O, H, H."""
    a = math.radians(104.5) / 2
    t = 0.96 * np.array([[0, 0, 0], [math.sin(a), 0, math.cos(a)], [-math.sin(a), 0, math.cos(a)]])
    xyz = centres[:, None, :] + np.einsum("mij,kj->mki", _rotations(rng, len(centres)), t)
    return xyz.reshape(-1, 3), np.tile(np.array([O, H, H], dtype=np.uint8), len(centres))


@functools.lru_cache(maxsize=8)
def _solute(n):
    """A branched solute of n atoms grown from the origin: bonds of 1.0-1.5 A to an atom
    with fewer than four, no other atom closer than 1.0 A (one molecule; a seed turns and
    perturbs it)."""
    rng = _rng(n)
    pts, bonds, k = np.zeros((n, 3)), np.zeros(n, dtype=int), 1
    while k < n:
        parent = rng.choice(np.flatnonzero(bonds[:k] < 4))
        d = rng.normal(size=3)
        p = pts[parent] + d / np.linalg.norm(d) * rng.uniform(1.0, 1.5)
        d2 = np.sum((pts[:k] - p) ** 2, axis=1)
        d2[parent] = np.inf
        if np.min(d2) >= 1.0:
            pts[k], bonds[k] = p, 1
            bonds[parent] += 1
            k += 1
    return pts, _species_counts(SOLUTE, n, rng)


def _box(rng, waters, solute):
    """A periodic cube at 1 g/cm^3: `waters` on sites of a jittered lattice that are
    farther than 2.5 A from the solute (atoms 0 .. solute - 1) at the centre."""
    edge = (waters * WATER_VOLUME + 12.0 * solute) ** (1 / 3)
    if solute:
        sx, ssp = _solute(solute)
        sx = sx @ _rotations(rng, 1)[0].T + rng.normal(0, 0.02, size=sx.shape) + edge / 2
    side = max(2, math.ceil((1.1 * waters) ** (1 / 3)))
    while True:
        g = (np.arange(side) + 0.5) * (edge / side)
        sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), axis=-1).reshape(-1, 3)
        if solute:
            near = np.flatnonzero(np.all(np.abs(sites - edge / 2) < np.abs(sx - edge / 2).max() + 2.5, axis=1))
            keep = np.ones(len(sites), dtype=bool)
            d = torch.cdist(torch.from_numpy(sites[near]).to(_device()), torch.from_numpy(sx).to(_device()))
            keep[near] = (d.amin(1) > 2.5).cpu().numpy() if len(near) else True
            sites = sites[keep]
        if len(sites) >= waters:
            break
        side += 1
    sites = sites[np.sort(rng.choice(len(sites), size=waters, replace=False))]
    wx, wsp = _waters(rng, sites + rng.uniform(-0.25, 0.25, size=sites.shape))
    x, sp = (np.concatenate([sx, wx]), np.concatenate([ssp, wsp])) if solute else (wx, wsp)
    return np.mod(x, edge).astype(np.float32), sp.astype(np.uint8), [edge] * 3


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _inputs(case, seed):
    """The systems of a case as host arrays: a list of (coords, species, box or None)."""
    rng, how = _rng(seed), case["how"]
    if how in ("molecules", "train_molecules"):
        # sizes vary within a batch, as the molecules of a data set or a queue do
        lo, hi = case["atoms_min"], case["atoms_max"]
        n = [int(round(lo + (hi - lo) * k / max(1, case["molecules"] - 1))) for k in range(case["molecules"])]
        rng.shuffle(n)
        return [_molecule(rng, m, ORGANIC if case["model"] == "ani4" else SOLUTE) + (None,) for m in n]
    if how == "snapshots":
        x, sp, box = _box(rng, case["waters"], case["solute"])
        return [(x + rng.normal(0, 0.05, size=x.shape).astype(np.float32), sp, box) for _ in range(case["snapshots"])]
    x, sp, box = _box(rng, case["waters"], case["solute"])
    if how == "md":
        # two successive frames of a trajectory: every atom moves by about 0.01 A
        return [(x, sp, box), (x + rng.normal(0, 0.01, size=x.shape).astype(np.float32), sp, box)]
    return [(x, sp, box)]


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one small molecule per call: an interactive energy, a Monte Carlo or geometry
        # step (latency and launches)
        {"name": "molecule24", "how": "molecules", "molecules": 1, "atoms_min": 24, "atoms_max": 24, "model": "ani4", "precision": "fp32"},
        # a queue of drug-like molecules scored in one call: screening, replicas, the
        # batches the server forms
        {"name": "molecules64", "how": "molecules", "molecules": 64, "atoms_min": 10, "atoms_max": 120, "model": "ani7", "precision": "fp32"},
        # a force-matching training step on a batch of molecules (forward and backward)
        {"name": "train64", "how": "train_molecules", "molecules": 64, "atoms_min": 20, "atoms_max": 60, "model": "ani4"},
        # a training step on one periodic frame, energy and forces in the loss
        {"name": "train_water1500", "how": "train_box", "waters": 500, "solute": 0, "model": "ani4"},
        # a water box, the unit of condensed-phase molecular dynamics, at FP32 accuracy and
        # constant pressure (virial)
        {"name": "water9000_virial", "how": "box", "waters": 3000, "solute": 0, "model": "ani4", "precision": "fp32", "virial": True},
        # the same at constant volume with BF16 networks
        {"name": "water9000_bf16", "how": "box", "waters": 3000, "solute": 0, "model": "ani4", "precision": "bf16", "virial": False},
        # a solvated macromolecule with an eight-network ensemble: the largest box
        {"name": "solvated100k", "how": "box", "waters": 33000, "solute": 1000, "model": "ani7x8", "precision": "fp32", "virial": False},
        # a mid-sized solvated box, ensemble, BF16 networks
        {"name": "solvated20k_bf16", "how": "box", "waters": 6667, "solute": 50, "model": "ani7x8", "precision": "bf16", "virial": False},
        # a small solvated box on the FP32 FMA networks (the option for hosts that want
        # no split operands), ensemble
        {"name": "solvated3k_simt", "how": "box", "waters": 999, "solute": 75, "model": "ani7x8", "precision": "fp32_simt", "virial": False},
        # two steps of hybrid dynamics: only the solute is in the ML region (mask), the
        # neighbour lists persist with a skin, asynchronous calls
        {"name": "hybrid20k_md", "how": "md", "waters": 6667, "solute": 50, "model": "ani7", "precision": "fp32"},
        # energies of stored snapshots for reweighting: no forces, one batch
        {"name": "snapshots8", "how": "snapshots", "snapshots": 8, "waters": 3000, "solute": 0, "model": "ani4", "precision": "fp32"},
        # an engine that holds host buffers: copies in and out around the call
        {"name": "host_solvated6k", "how": "host", "waters": 2001, "solute": 137, "model": "ani7", "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    how = rng.choice(["molecules", "molecules", "train_molecules", "train_box", "box", "box", "box", "md", "snapshots", "host"])
    precision = rng.choice(["fp32", "fp32", "bf16"])
    if how in ("molecules", "train_molecules"):
        lo = rng.randint(6, 60)
        case = {"how": how, "molecules": _log(rng, 1, 200 if how == "molecules" else 96), "atoms_min": lo,
                "atoms_max": lo + rng.randint(0, 60), "model": rng.choice(["ani4", "ani7"])}
        return case if how == "train_molecules" else dict(case, precision=precision)
    if how == "train_box":
        return {"how": how, "waters": _log(rng, 60, 1000), "solute": 0, "model": "ani4"}
    model = rng.choice(["ani4", "ani7", "ani7x8"])
    solute = 0 if model == "ani4" else _log(rng, 10, 400)
    if how == "md":
        return {"how": how, "waters": _log(rng, 400, 8000), "solute": _log(rng, 20, 120), "model": rng.choice(["ani7", "ani7x8"]),
                "precision": precision}
    if how == "snapshots":
        return {"how": how, "snapshots": rng.randint(2, 12), "waters": _log(rng, 200, 3000), "solute": solute, "model": model,
                "precision": precision}
    if how == "host":
        return {"how": how, "waters": _log(rng, 300, 12000), "solute": solute, "model": model, "precision": precision}
    if rng.random() < 0.2:
        return {"how": how, "waters": _log(rng, 200, 1500), "solute": solute, "model": model, "precision": "fp32_simt", "virial": False}
    return {"how": how, "waters": _log(rng, 200, 30000), "solute": solute, "model": model, "precision": precision,
            "virial": precision == "fp32" and rng.random() < 0.4}


# ---------------------------------------------------------------- preparation and passes
def prepare(case, seed):
    from paper_2207_14276_gb300 import Potential

    dev, how, systems = _device(), case["how"], _inputs(case, seed)
    pot = Potential(_spec(case["model"]), _weights(case["model"]), precision=case.get("precision", "fp32"))
    sizes = [len(x) for x, _, _ in systems]
    if how == "md":
        pot.set_skin(0.5)
    # a program reserves for the batches it will send; the solute's core is denser than water
    pot.reserve(max(sizes) if how == "md" else sum(sizes), len(sizes), 288 if case.get("solute") else 128,
                96 if case.get("solute") else 48)
    st = {"how": how, "pot": pot, "sizes": sizes, "virial": case.get("virial", False)}
    if how == "host":
        x, sp, box = systems[0]
        pin = (lambda a: torch.from_numpy(a).pin_memory().numpy())
        return dict(st, x=pin(x), sp=pin(sp), box=box, out=pin(np.empty((len(x), 3), dtype=np.float32)))
    if how == "md":
        n = sizes[0]
        mask = torch.zeros(n, dtype=torch.uint8, device=dev)
        mask[:case["solute"]] = 1
        return dict(st, frames=[torch.from_numpy(x).to(dev) for x, _, _ in systems], mask=mask, box=systems[0][2],
                    sp=torch.from_numpy(systems[0][1]).to(dev), x=torch.from_numpy(systems[0][0]).to(dev),
                    E=torch.zeros(2, dtype=torch.float64, device=dev),
                    F=torch.zeros((2, n, 3), dtype=torch.float32, device=dev))
    x = torch.from_numpy(np.concatenate([s[0] for s in systems])).to(dev)
    sp = torch.from_numpy(np.concatenate([s[1] for s in systems])).to(dev)
    if how in ("train_molecules", "train_box"):
        g = torch.Generator(device=dev).manual_seed(int(seed))
        return dict(st, x=x.requires_grad_(True), sp=sp, box=systems[0][2],
                    w=torch.from_numpy(_weights(case["model"])).to(dev).requires_grad_(True),
                    target=torch.randn(x.shape, generator=g, device=dev))
    if how == "box":
        return dict(st, x=x, sp=sp, box=systems[0][2])
    # batched calls write into buffers that the program keeps
    at = np.cumsum([0] + sizes)
    energy = torch.empty(len(sizes), dtype=torch.float64, device=dev)
    per_atom = torch.empty((len(x), 3) if how == "molecules" else len(x), dtype=torch.float32, device=dev)
    name = "forces" if how == "molecules" else "atom_energies"
    return dict(st, energy=energy, per_atom=per_atom,
                batch=[{"coords": x[a:b], "species": sp[a:b], "box": s[2]} for a, b, s in zip(at, at[1:], systems)],
                outs=[{"energy": energy[k:k + 1], name: per_atom[a:b]} for k, (a, b) in enumerate(zip(at, at[1:]))])


def run(st):
    from paper_2207_14276_gb300.autograd import NNPBatchFunction, NNPFunction

    how, pot = st["how"], st["pot"]
    if how == "box":
        out = pot.energy_forces(st["x"], st["sp"], st["box"], virial=st["virial"])
        return [out[0].float(), out[1]] + [v.float() for v in out[2:]]
    if how == "molecules":
        pot.energy_forces_batch(st["batch"], outputs=st["outs"])
        return [st["energy"].float(), st["per_atom"]]
    if how == "snapshots":
        pot.energy_forces_batch(st["batch"], outputs=st["outs"], forces=False, atom_energies=True)
        return [st["energy"].float(), st["per_atom"]]
    if how == "train_molecules":
        _, f = NNPBatchFunction.apply(st["x"], st["w"], pot, st["sp"], st["sizes"])
        loss = ((f - st["target"]) ** 2).sum()
        return [loss.detach(), f.detach()] + list(torch.autograd.grad(loss, (st["x"], st["w"])))
    if how == "train_box":
        e, f = NNPFunction.apply(st["x"], st["w"], pot, st["sp"], st["box"])
        loss = ((f - st["target"]) ** 2).sum() + e.float().square().sum() / len(f)
        return [loss.detach(), f.detach()] + list(torch.autograd.grad(loss, (st["x"], st["w"])))
    if how == "md":
        for k in range(2):
            st["x"].copy_(st["frames"][k])
            pot.energy_forces_into(st["x"], st["sp"], st["box"], st["mask"], st["E"][k:k + 1], st["F"][k])
        return [st["E"].float(), st["F"]]
    e, f = pot.energy_forces_host_into(st["x"], st["sp"], st["box"], None, out_forces=st["out"])
    return [np.float32(e), f]


def work(case):
    """Inputs, weights and outputs once; per atom the radial terms (16 shells of about 5
    FLOP forward, 8 backward), the angular pairs (200 and 330) and the networks' 2 K N
    over the features that are not zero by the atom's surroundings (water: 128)."""
    how, model = case["how"], case["model"]
    d, e, (h1, h2, h3) = _dim(model), ENSEMBLE[model], HIDDEN[model]
    if how in ("molecules", "train_molecules"):
        m, size = case["molecules"], (case["atoms_min"] + case["atoms_max"]) / 2
        n, nr, na, dense = m * size, min(size - 1, 11), 4, m * size
    else:
        dense = case["solute"]
        n, nr, na = 3 * case["waters"] + dense, 59, 17
        if how == "md":
            n, nr, na = dense, 30, 15
        n *= case.get("snapshots", 1)
        dense *= case.get("snapshots", 1)
    live = dense * d + (n - dense) * min(d, 128)
    nets = 2.0 * e * (live * h1 + n * (h1 * h2 + h2 * h3 + h3))
    aev_f, aev_b = n * (nr * 80 + na * (na - 1) / 2 * 200), n * (nr * 128 + na * (na - 1) / 2 * 330)
    weights = 4.0 * len(SPECIES[model]) * e * (d * h1 + h1 * h2 + h2 * h3 + h3)
    if how.startswith("train"):
        # the forces, then along their gradient: forward tangent, the backward of both, and
        # two products per weight
        return {"bytes": n * 61 + 3 * weights, "flops": (2 + 1 + 2 + 2) * nets + 3 * (aev_f + aev_b)}
    if how == "snapshots":
        return {"bytes": n * 17 + weights, "flops": nets + aev_f}
    once = {"bytes": n * 25 + weights, "flops": 2 * nets + aev_f + aev_b}
    return {k: v * (2 if how == "md" else 1) for k, v in once.items()}


# ---------------------------------------------------------------- 64 bits
def _f32(v):
    """The value as the library's FP32 parameters hold it."""
    return torch.tensor(v, dtype=torch.float32, device=_device()).double()


def _nets(model, flat):
    """Per species the four layers (W [E, out, in], b [E, 1, out]) of a flat vector."""
    w, e, s = _widths(model), ENSEMBLE[model], len(SPECIES[model])
    flat, out, at = flat.reshape(e, s, -1), [], 0
    for l in range(4):
        n = w[l + 1] * w[l]
        out.append((flat[:, :, at:at + n].reshape(e, s, w[l + 1], w[l]), flat[:, :, at + n:at + n + w[l + 1]]))
        at += n + w[l + 1]
    return [[(a[:, k], b[:, k].unsqueeze(1)) for a, b in out] for k in range(s)]


def _pairs(x, box, centres, rc):
    """(row of `centres`, j, periodic shift) of every pair within rc, rows ascending."""
    d = x.unsqueeze(0) - x[centres].unsqueeze(1)
    if box is not None:
        d = d - torch.round(d / box) * box
    r2 = d.square().sum(-1)
    i, j = torch.nonzero((r2 < rc * rc) & (r2 > 1e-12), as_tuple=True)
    return i, j, d[i, j] - (x[j] - x[centres[i]])


def _atom_energies(model, nets, x, sp, box, centres, strain=None):
    """Energies of the atoms `centres`, differentiable in x and nets (Eqs. 2-5)."""
    s, b = len(SPECIES[model]), len(centres)
    rc_r, rc_a = _f32(RC_R), _f32(RC_A)
    with torch.no_grad():
        i, j, shift = _pairs(x, box, centres, RC_R)
    v = x[j] - x[centres[i]] + shift
    v = v if strain is None else v + v @ strain
    r = v.square().sum(-1).sqrt()
    fc = 0.5 * torch.cos(math.pi * r / rc_r) + 0.5
    feat = torch.exp(-ETA_R * (r[:, None] - _f32(SHF_R)) ** 2) * fc[:, None]
    radial = torch.zeros(b * s, 16, dtype=x.dtype, device=x.device).index_add(0, i * s + sp[j], feat).reshape(b, -1)
    near = torch.nonzero(r.detach() < rc_a).flatten()
    ia, ra, sa, ua = i[near], r[near], sp[j[near]], v[near] / r[near, None]
    fa = 0.5 * torch.cos(math.pi * ra / rc_a) + 0.5
    cnt = torch.bincount(ia, minlength=b)
    end = torch.cumsum(cnt, 0)
    p = torch.arange(len(ia), device=x.device)
    more = end[ia] - p - 1                             # later neighbours of the same centre
    t1 = torch.repeat_interleave(p, more)
    t2 = t1 + 1 + torch.arange(len(t1), device=x.device) - torch.repeat_interleave(torch.cumsum(more, 0) - more, more)
    c = (ua[t1] * ua[t2]).sum(-1)
    sn = torch.linalg.cross(ua[t1], ua[t2]).square().sum(-1).clamp_min(1e-30).sqrt()
    z = _f32(SHF_Z)
    ang = (1 + c[:, None] * torch.cos(z) + sn[:, None] * torch.sin(z)) ** int(ZETA) * 2.0 ** (1 - ZETA)
    rad = torch.exp(-ETA_A * (0.5 * (ra[t1] + ra[t2])[:, None] - _f32(SHF_A)) ** 2) * (fa[t1] * fa[t2])[:, None]
    lo, hi = torch.minimum(sa[t1], sa[t2]), torch.maximum(sa[t1], sa[t2])
    q = lo * s - lo * (lo - 1) // 2 + hi - lo
    n_q = s * (s + 1) // 2
    angular = torch.zeros(b * n_q, 32, dtype=x.dtype, device=x.device).index_add(
        0, ia[t1] * n_q + q, (rad[:, :, None] * ang[:, None, :]).reshape(-1, 32)).reshape(b, -1)
    g = torch.cat([radial, angular], dim=1)
    out = torch.zeros(b, dtype=x.dtype, device=x.device)
    for k in range(s):
        rows = torch.nonzero(sp[centres] == k).flatten()
        if len(rows):
            h = g[rows].expand(ENSEMBLE[model], -1, -1)
            for l, (w, bias) in enumerate(nets[k]):
                h = h @ w.transpose(1, 2) + bias
                h = torch.nn.functional.celu(h, ALPHA) if l < 3 else h
            out = out.index_add(0, rows, h.mean(0).squeeze(-1))
    return out


def _energy_forces(model, nets, x, sp, box, forces=True):
    """(energy, atomic energies, forces, virial) of one system, its centres in chunks."""
    x = x.clone().requires_grad_(forces)
    step = max(64, min(2048, int(2e8 / max(1, len(x)))))
    ae, f = [], torch.zeros_like(x)
    virial = torch.zeros(3, 3, dtype=x.dtype, device=x.device)
    for a in range(0, len(x), step):
        centres = torch.arange(a, min(a + step, len(x)), device=x.device)
        if forces:
            # the derivative along a strain of every displacement: sum v (x) dE/dv
            strain = torch.zeros(3, 3, dtype=x.dtype, device=x.device, requires_grad=True)
            e = _atom_energies(model, nets, x, sp, box, centres, strain)
            gx, gs = torch.autograd.grad(e.sum(), (x, strain))
            f, virial = f - gx, virial - gs
        else:
            e = _atom_energies(model, nets, x, sp, box, centres)
        ae.append(e.detach())
    ae = torch.cat(ae)
    return ae.sum(), ae, f, virial


def exact(case, seed):
    dev, how, model, systems = _device(), case["how"], case["model"], _inputs(case, seed)
    flat = torch.from_numpy(_weights(model)).to(dev).double()
    sys64 = [(torch.from_numpy(x).to(dev).double(), torch.from_numpy(sp).to(dev).long(),
              None if box is None else torch.tensor(box, dtype=torch.float64, device=dev)) for x, sp, box in systems]
    if how.startswith("train"):
        flat.requires_grad_(True)
        nets = _nets(model, flat)
        g = torch.Generator(device=dev).manual_seed(int(seed))
        n = sum(len(x) for x, _, _ in sys64)
        target = torch.randn((n, 3), generator=g, device=dev).double()
        loss, fs, gxs, gw, at = 0.0, [], [], torch.zeros_like(flat), 0
        for x, sp, box in sys64:
            x = x.requires_grad_(True)
            e = _atom_energies(model, nets, x, sp, box, torch.arange(len(x), device=dev)).sum()
            f = -torch.autograd.grad(e, x, create_graph=True)[0]
            part = (f - target[at:at + len(x)]).square().sum()
            if how == "train_box":
                part = part + e.square() / n
            gx, gwk = torch.autograd.grad(part, (x, flat), retain_graph=True)
            at += len(x)
            loss += float(part.detach())
            fs.append(f.detach())
            gxs.append(gx)
            gw += gwk
        return [torch.tensor(loss, dtype=torch.float64), torch.cat(fs), torch.cat(gxs), gw]
    nets = _nets(model, flat)
    if how == "md":
        e, f = [], []
        for x, sp, box in sys64:
            m = case["solute"]
            ek, _, fk, _ = _energy_forces(model, nets, x[:m], sp[:m], box)
            e.append(ek)
            f.append(torch.cat([fk, torch.zeros(len(x) - m, 3, dtype=fk.dtype, device=dev)]))
        return [torch.stack(e), torch.stack(f)]
    got = [_energy_forces(model, nets, *s, forces=how != "snapshots") for s in sys64]
    if how == "molecules":
        return [torch.stack([e for e, _, _, _ in got]), torch.cat([f for _, _, f, _ in got])]
    if how == "snapshots":
        return [torch.stack([e for e, _, _, _ in got]), torch.cat([a for _, a, _, _ in got])]
    e, _, f, v = got[0]
    if how == "host":
        return [e, f]
    return [e.reshape(1), f] + ([v] if case["virial"] else [])
