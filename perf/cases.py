"""Performance cases of the ANN-potential library, through its public entry points.

Each case is one piece of work that a user's program gives the library:

* ``frames`` -- energies, forces, virials and atomic energies of stored
  configurations, one ``AenetGPU.compute`` call per frame (re-evaluating a
  trajectory, a screening or Monte-Carlo loop);
* ``md`` -- a segment of velocity-Verlet MD from a stored start
  (``AenetGPU.md_nve``), with the energy records of every frame;
* ``batch`` -- many independent structures of ragged sizes, water and solid,
  through the prepared batch (``batch_prepare`` / ``batch_run``);
* ``train`` -- one training pass over small frames of ragged sizes: the energies
  and the loss gradient with respect to the network weights, through the
  autograd function;
* ``descriptors`` -- the fingerprints of one structure (featurising a data set).

Structures are liquid water (the paper's 52-descriptor basis) and a 4-species
solid at 0.07 atoms/A^3 on a jittered lattice with no two atoms closer than
1.6 A. ``exact`` restates the potential in 64-bit torch operations.
"""
import math

import numpy as np
import torch

from paper_2107_11311_gb300 import inputs
from paper_2107_11311_gb300.aenet import AenetGPU, energy_function

DEV = "cuda"
F64 = torch.float64
DT = 2.5e-4  # ps: a 0.25 fs step, for hydrogen in a hot start


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: a DFT-sized water cell handed over in host arrays, as an MD engine's pair
        # style does it; latency, staging and launches count
        {"name": "frames_water_192_host", "kind": "frames", "family": "water", "atoms": 192, "hidden": 15,
         "precision": "fp32", "frames": 32, "host": True, "tilt": 0.0},
        # the ordinary evaluation: a mid-sized liquid box on device buffers
        {"name": "frames_water_12288", "kind": "frames", "family": "water", "atoms": 12288, "hidden": 15,
         "precision": "fp32", "frames": 8, "host": False, "tilt": 0.0},
        # the largest box with the widest fused network
        {"name": "frames_water_331776", "kind": "frames", "family": "water", "atoms": 331776, "hidden": 32,
         "precision": "fp32", "frames": 2, "host": False, "tilt": 0.0},
        # the second basis (long cutoffs, angular order 6, four species)
        {"name": "frames_solid_27000", "kind": "frames", "family": "amorphous", "atoms": 27000, "hidden": 30,
         "precision": "fp32", "frames": 4, "host": False, "tilt": 0.0},
        # the accurate tensor-core form of the networks
        {"name": "frames_water_98304_bf16x3", "kind": "frames", "family": "water", "atoms": 98304, "hidden": 32,
         "precision": "bf16x3", "frames": 2, "host": False, "tilt": 0.0},
        # MD of the paper's own water system (1,536 atoms, 52-25-25-1): the step's latency
        {"name": "md_water_1536", "kind": "md", "family": "water", "atoms": 1536, "hidden": 25, "steps": 20,
         "skin": 0.0},
        # MD of an ordinary box
        {"name": "md_water_12288", "kind": "md", "family": "water", "atoms": 12288, "hidden": 15, "steps": 20,
         "skin": 0.0},
        # MD of the largest box (the benchmark's headline system)
        {"name": "md_water_331776", "kind": "md", "family": "water", "atoms": 331776, "hidden": 32, "steps": 4,
         "skin": 0.0},
        # MD of the solid
        {"name": "md_solid_27000", "kind": "md", "family": "amorphous", "atoms": 27000, "hidden": 30, "steps": 10,
         "skin": 0.0},
        # screening: 512 structures of 32 ... 2,048 atoms, half water, half solid
        {"name": "batch_512", "kind": "batch", "structures": 512, "layout": 30, "lo": 32, "hi": 2048},
        # training on DFT-sized frames of ragged sizes
        {"name": "train_water", "kind": "train", "frames": 16, "lo": 90, "hi": 390, "layout": 7, "hidden": 15},
        # featurising a structure
        {"name": "descriptors_water_12288", "kind": "descriptors", "family": "water", "atoms": 12288},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _atoms(rng, family, lo, hi):
    n = _log_uniform(rng, lo, hi)
    return 3 * max(1, n // 3) if family == "water" else n


def draw(rng):
    kind = rng.choice(["frames", "frames", "frames", "md", "md", "md", "batch", "train", "descriptors"])
    family = rng.choice(["water", "water", "amorphous"])
    top = 331776 if family == "water" else 60000
    hidden = rng.choice([15, 25, 32]) if family == "water" else 30
    if kind == "frames":
        n = _atoms(rng, family, 150, top)
        return {"kind": kind, "family": family, "atoms": n, "hidden": hidden,
                "precision": rng.choice(["fp32", "fp32", "fp32", "bf16x3"]),
                "frames": max(2, min(32, 40000 // n)), "host": n < 2000 and rng.random() < 0.5,
                "tilt": rng.choice([0.0, 0.0, round(rng.uniform(0.05, 0.3), 3)])}
    if kind == "md":
        n = _atoms(rng, family, 300, top)
        return {"kind": kind, "family": family, "atoms": n, "hidden": hidden, "steps": max(4, min(20, 200000 // n)),
                "skin": rng.choice([0.0, 0.0, 0.5])}
    if kind == "batch":
        return {"kind": kind, "structures": 2 * _log_uniform(rng, 16, 256), "layout": rng.randrange(1000),
                "lo": rng.randrange(24, 64), "hi": _log_uniform(rng, 256, 2048)}
    if kind == "train":
        lo = rng.randrange(60, 200)
        return {"kind": kind, "frames": rng.randrange(4, 24), "lo": lo, "hi": lo * rng.randrange(2, 6),
                "layout": rng.randrange(1000), "hidden": hidden if family == "water" else 15}
    return {"kind": kind, "family": family, "atoms": _atoms(rng, family, 150, 60000)}


# --------------------------------------------------------------- their inputs

def _solid(n, rng):
    """n atoms of four species on the sites of a jittered simple cubic lattice."""
    box = (n / 0.07) ** (1.0 / 3.0)
    m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    a = box / m
    site = rng.permutation(m ** 3)[:n]
    pos = (np.stack([site // (m * m), site // m % m, site % m], 1) + 0.5) * a
    pos += rng.uniform(-0.5, 0.5, size=(n, 3)) * max(0.0, a - 1.6)
    return pos, rng.choice(4, size=n, p=[0.4, 0.3, 0.2, 0.1]).astype(np.int32), np.full(3, box)


def _structure(family, n, seed):
    """(positions [n, 3], species [n], box edges [3]) of one structure."""
    if family == "water":
        st = inputs.water(n // 3, None, seed)
        return st.pos, st.types, st.box
    return _solid(n, np.random.default_rng(seed))


def _sizes(case, count):
    rng = np.random.default_rng(case["layout"])
    return np.rint(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=count))).astype(int)


def _model(case, family=None):
    family = family or case["family"]
    hidden = case.get("hidden")
    return inputs.make_model(family, hidden=None if hidden is None else (hidden, hidden))


def _frames(case, seed):
    """Frames of a frames case: positions [F, n, 3], species, box, tilts."""
    n = case["atoms"]
    got = [_structure(case["family"], n, 1000 * seed + f) for f in range(case["frames"])]
    pos, types, box = np.stack([g[0] for g in got]), got[0][1], got[0][2]
    tilt = case["tilt"] * box[0] * np.array([1.0, -0.5, 0.7])
    # the tilted cell holds the same fractional coordinates
    y, z = pos[..., 1] / box[1], pos[..., 2] / box[2]
    pos[..., 0] += y * tilt[0] + z * tilt[1]
    pos[..., 1] += z * tilt[2]
    return pos, types, box, tilt


def _md_start(case, seed):
    m = _model(case)
    pos, types, box = _structure(case["family"], case["atoms"], 1000 * seed)
    return m, pos, inputs.maxwell_boltzmann(m.masses[types], 300.0, seed=seed + 1), types, box


def _batch(case, seed):
    """The two families' structures of a batch case."""
    half = case["structures"] // 2
    sizes = _sizes(case, 2 * half)
    for family, part in (("water", sizes[:half]), ("amorphous", sizes[half:])):
        sts = [_structure(family, 3 * max(1, n // 3) if family == "water" else int(n), 1000 * seed + k)
               for k, n in enumerate(part)]
        off = np.concatenate([[0], np.cumsum([len(s[0]) for s in sts])]).astype(np.int64)
        yield (family, off, np.concatenate([s[0] for s in sts]), np.concatenate([s[1] for s in sts]),
               np.stack([s[2] for s in sts]))


def _train_frames(case, seed):
    """Frames and their reference energies (labels spread over the model's energy scale)."""
    rng = np.random.default_rng(seed + 5)
    for k, n in enumerate(_sizes(case, case["frames"])):
        pos, types, box = _structure("water", 3 * max(1, n // 3), 1000 * seed + k)
        yield pos, types, box, len(pos) * rng.uniform(0.5, 1.0)


def _gpu(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frames":
        pos, types, box, tilt = _frames(case, seed)
        F, n = pos.shape[:2]
        gpu = AenetGPU(_model(case), case["precision"])
        if tilt.any():
            gpu.set_box_tilt(*tilt)
        shapes = {"energy": (F,), "forces": (F, n, 3), "virial": (F, 3, 3), "e_atom": (F, n)}
        if case["host"]:
            out = {k: np.zeros(s) for k, s in shapes.items()}
        else:
            pos, types = _gpu(pos), _gpu(types)
            out = {k: torch.zeros(s, dtype=F64, device=DEV) for k, s in shapes.items()}
        return {"kind": kind, "gpu": gpu, "pos": pos, "types": types, "box": box, "out": out}
    if kind == "md":
        m, pos, vel, types, box = _md_start(case, seed)
        gpu = AenetGPU(m, "fp32")
        gpu.set_skin(case["skin"])
        start = (_gpu(pos), _gpu(vel))
        K = case["steps"]
        return {"kind": kind, "gpu": gpu, "start": start, "types": _gpu(types), "box": box, "steps": K,
                "out": {"pos": torch.empty_like(start[0]), "vel": torch.empty_like(start[1]),
                        "e_pot": torch.zeros(K + 1, dtype=F64, device=DEV),
                        "e_kin": torch.zeros(K + 1, dtype=F64, device=DEV)}}
    if kind == "batch":
        gpus, out = [], {}
        for family, off, pos, types, boxes in _batch(case, seed):
            gpu = AenetGPU(_model({}, family), "fp32")
            S = len(boxes)
            o = {"energies": torch.zeros(S, dtype=F64, device=DEV),
                 "forces": torch.zeros((len(pos), 3), dtype=F64, device=DEV),
                 "virials": torch.zeros((S, 3, 3), dtype=F64, device=DEV)}
            gpu.batch_prepare(off, boxes, _gpu(pos), _gpu(types), **o)
            gpus.append(gpu)
            out[family] = o
        return {"kind": kind, "gpus": gpus, "out": out}
    if kind == "train":
        m = _model(case, "water")
        frames = [(_gpu(p), _gpu(t), b, e) for p, t, b, e in _train_frames(case, seed)]
        return {"kind": kind, "gpu": AenetGPU(m, "fp32"), "frames": frames,
                "params": _gpu(m.params).requires_grad_(True)}
    pos, types, box = _structure(case["family"], case["atoms"], 1000 * seed)
    m = _model(case)
    return {"kind": kind, "gpu": AenetGPU(m, "fp32"), "pos": _gpu(pos), "types": _gpu(types), "box": box,
            "out": torch.zeros((len(pos), m.D), dtype=torch.float32, device=DEV)}


# ------------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "frames":
        o = state["out"]
        for f in range(len(state["pos"])):
            state["gpu"].compute(state["pos"][f], state["types"], state["box"], energy=o["energy"][f:f + 1],
                                 forces=o["forces"][f], virial=o["virial"][f], e_atom=o["e_atom"][f])
        return {"forces": o["forces"], "virial": o["virial"], "e_atom": o["e_atom"]}
    if kind == "md":
        o = state["out"]
        o["pos"].copy_(state["start"][0])
        o["vel"].copy_(state["start"][1])
        state["gpu"].md_nve(o["pos"], o["vel"], state["types"], state["box"], DT, state["steps"], o["e_pot"],
                            o["e_kin"])
        return o
    if kind == "batch":
        for gpu in state["gpus"]:
            gpu.batch_run()
        return state["out"]
    if kind == "train":
        energy = energy_function().apply
        params = state["params"]
        params.grad = None
        energies = [energy(p, params, state["gpu"], t, b) for p, t, b, _ in state["frames"]]
        loss = sum(((e - ref) / len(p)) ** 2 for e, (p, _, _, ref) in zip(energies, state["frames"]))
        loss.backward()
        return {"energies": torch.stack(energies).detach(), "dloss_dparams": params.grad}
    return state["gpu"].descriptors(state["pos"], state["types"], state["box"], out=state["out"])


def _unit_work(m, family):
    """Flops of one atom in one energy + force evaluation (FMA = 2): per neighbour
    within the cutoff, per unordered angular pair and per network weight."""
    rho = 0.07 if family == "amorphous" else 3.0 * 6.02214076e23 / 18.015 / 1e24
    nb, na = (rho * 4.0 / 3.0 * math.pi * r ** 3 for r in (m.rc_rad, m.rc_ang))
    pairs, Kr, Ka = na * na / 2, m.order_rad + 1, m.order_ang + 1
    forward = (12 + 4 * Kr) * nb + (10 + 4 * Ka) * pairs
    backward = (20 + 6 * Kr) * nb + (40 + 6 * Ka) * pairs
    net = 4 * sum(m.widths[k] * m.widths[k - 1] for k in range(1, len(m.widths)))
    return forward, forward + backward + net


def work(case):
    kind = case["kind"]
    if kind == "batch":
        half = case["structures"] // 2
        sizes = _sizes(case, 2 * half)
        flops = sum(float(s.sum()) * _unit_work(_model({}, f), f)[1]
                    for f, s in (("water", sizes[:half]), ("amorphous", sizes[half:])))
        return {"bytes": float(sizes.sum()) * 52 + 80.0 * len(sizes), "flops": flops}
    if kind == "train":
        n, m = float(_sizes(case, case["frames"]).sum()), _model(case, "water")
        return {"bytes": n * 28 + 16.0 * m.params.size, "flops": n * _unit_work(m, "water")[1]}
    m = _model(case)
    forward, both = _unit_work(m, case["family"])
    n = float(case["atoms"])
    if kind == "descriptors":
        return {"bytes": n * (28 + 4 * m.D), "flops": n * forward}
    if kind == "md":  # positions and velocities in and out, types in
        return {"bytes": n * 100 + 16.0 * (case["steps"] + 1), "flops": n * (case["steps"] + 1) * both}
    return {"bytes": case["frames"] * n * 60, "flops": case["frames"] * n * both}


# ------------------------------------------------- the same in 64-bit numbers

def _neighbours(pos, cell, rc):
    """(i, j, d) of every image-atom j within rc of atom i, sorted by i. cell:
    the lattice vectors as rows."""
    inv = torch.linalg.inv(cell)
    frac = pos @ inv
    frac = frac - torch.floor(frac)
    frac = torch.where(frac >= 1.0, frac - 1.0, frac)
    width = 1.0 / inv.norm(dim=0)  # distances between opposite faces
    nc = torch.clamp((width / rc).floor().long(), min=1)
    m = torch.ceil(rc * nc / width).long().tolist()
    ci = torch.minimum((frac * nc).long(), nc - 1)
    flat = (ci[:, 0] * nc[1] + ci[:, 1]) * nc[2] + ci[:, 2]
    count = torch.bincount(flat, minlength=int(nc.prod()))
    order = torch.argsort(flat, stable=True)
    first = torch.cumsum(count, 0) - count
    table = torch.full((len(count), int(count.max())), -1, dtype=torch.long, device=pos.device)
    s = flat[order]
    table[s, torch.arange(len(pos), device=pos.device) - first[s]] = order
    x = frac @ cell
    found = []
    for ox in range(-m[0], m[0] + 1):
        for oy in range(-m[1], m[1] + 1):
            for oz in range(-m[2], m[2] + 1):
                u = ci + torch.tensor([ox, oy, oz], device=pos.device)
                wrap = torch.div(u, nc, rounding_mode="floor")
                v = u - wrap * nc
                shift = wrap.to(F64) @ cell
                j = table[(v[:, 0] * nc[1] + v[:, 1]) * nc[2] + v[:, 2]]
                d = x[j.clamp(min=0)] + (shift - x)[:, None, :]
                keep = (j >= 0) & (d.square().sum(-1) <= rc * rc)
                if not (ox or oy or oz):  # the atom itself; its images count
                    keep &= j != torch.arange(len(pos), device=pos.device)[:, None]
                i, c = torch.nonzero(keep, as_tuple=True)
                found.append((i, j[i, c], d[i, c]))
    i = torch.cat([f[0] for f in found])
    by = torch.argsort(i, stable=True)
    return i[by], torch.cat([f[1] for f in found])[by], torch.cat([f[2] for f in found])[by]


def _cutoff(r, rc):
    return torch.where(r <= rc, 0.5 * (torch.cos(math.pi * r / rc) + 1.0), torch.zeros_like(r))


def _fingerprints(m, n, i, d, s):
    """Descriptor rows [n, D] of n atoms from their neighbours' displacements d
    (sorted by atom index i) and species weights s."""
    r = d.norm(dim=1)
    cols = {}

    def sums(name, order, x, w, ww, at):
        t0, t1 = torch.ones_like(x), x
        for q in range(order + 1):
            for copy, f in ((name, w), (name + "_w", ww)):
                cols.setdefault(copy, []).append(torch.zeros(n, dtype=F64, device=d.device).index_add(0, at, t0 * f))
            t0, t1 = t1, 2.0 * x * t1 - t0

    fr = _cutoff(r, m.rc_rad)
    sums("rad", m.order_rad, 2.0 * r / m.rc_rad - 1.0, fr, fr * s, i)
    near = torch.nonzero(r <= m.rc_ang)[:, 0]
    ia, ra, sa = i[near], r[near], s[near]
    ua, fa = d[near] / ra[:, None], _cutoff(ra, m.rc_ang)
    count = torch.bincount(ia, minlength=n)
    last = torch.cumsum(count, 0)[ia]  # one past the atom's last entry
    here = torch.arange(len(ia), device=d.device)
    left = last - 1 - here
    a = torch.repeat_interleave(here, left)
    b = a + 1 + torch.arange(len(a), device=d.device) - torch.repeat_interleave(torch.cumsum(left, 0) - left, left)
    w = 2.0 * fa[a] * fa[b]  # every unordered pair stands for two ordered ones
    sums("ang", m.order_ang, (ua[a] * ua[b]).sum(1), w, w * sa[a] * sa[b], ia[a])
    return torch.stack(cols["rad"] + cols["ang"] + cols["rad_w"] + cols["ang_w"], 1)


def _network(m, params, G, types):
    """Atomic energies from descriptor rows."""
    E = torch.zeros(len(G), dtype=F64, device=G.device)
    shift, scale = _gpu(m.in_shift, F64), _gpu(m.in_scale, F64)
    for t in range(m.n_species):
        at = torch.nonzero(types == t)[:, 0]
        x, p = (G[at] - shift[t]) * scale[t], 0
        for k in range(1, len(m.widths)):
            o, c = m.widths[k], m.widths[k - 1]
            x = x @ params[t, p:p + o * c].reshape(o, c).T + params[t, p + o * c:p + o * c + o]
            p += o * c + o
            if k < len(m.widths) - 1:
                x = torch.tanh(x)
        E = E.index_put((at,), x[:, 0])
    return E


def _exact_eval(m, pos, types, cell, params=None, descriptors=False):
    """Energy per atom, forces, virial (and the energy's weight gradient when
    params is given), or the descriptor rows."""
    n, dev = len(pos), pos.device
    weights = _gpu(m.type_weights, F64)
    i, j, d = _neighbours(pos, cell, max(m.rc_rad, m.rc_ang))
    par = (_gpu(m.params, F64) if params is None else params).requires_grad_(params is not None)
    starts = torch.searchsorted(i, torch.arange(n + 1, device=dev))
    e_atom, F, W = torch.zeros(n, dtype=F64, device=dev), torch.zeros_like(pos), torch.zeros((3, 3), dtype=F64, device=dev)
    dW, rows = torch.zeros_like(par), []
    step = 16384 if m.rc_ang < 5.0 else 2048
    for c0 in range(0, n, step):
        c1 = min(n, c0 + step)
        lo, hi = int(starts[c0]), int(starts[c1])
        ic, jc, dc = i[lo:hi], j[lo:hi], d[lo:hi].clone().requires_grad_(not descriptors)
        G = _fingerprints(m, c1 - c0, ic - c0, dc, weights[types[jc].long()])
        if descriptors:
            rows.append(G)
            continue
        E = _network(m, par, G, types[c0:c1])
        g = torch.autograd.grad(E.sum(), [dc] + ([par] if params is not None else []))
        e_atom[c0:c1] = E.detach()
        F.index_add_(0, ic, g[0])
        F.index_add_(0, jc, -g[0])
        W -= d[lo:hi].T @ g[0]
        if params is not None:
            dW += g[1]
    return torch.cat(rows) if descriptors else (e_atom, F, W, dW)


def _cell(box, tilt=(0.0, 0.0, 0.0)):
    return torch.tensor([[box[0], 0.0, 0.0], [tilt[0], box[1], 0.0], [tilt[1], tilt[2], box[2]]], dtype=F64, device=DEV)


def exact(case, seed):
    kind = case["kind"]
    if kind == "frames":
        pos, types, box, tilt = _frames(case, seed)
        m, t = _model(case), _gpu(types)
        got = [_exact_eval(m, _gpu(p), t, _cell(box, tilt)) for p in pos]
        return {"forces": torch.stack([g[1] for g in got]), "virial": torch.stack([g[2] for g in got]),
                "e_atom": torch.stack([g[0] for g in got])}
    if kind == "md":
        m, pos, vel, types, box = _md_start(case, seed)
        x, v, t, cell = _gpu(pos), _gpu(vel), _gpu(types), _cell(box)
        mass = _gpu(m.masses, F64)[t.long()][:, None]
        e_pot, e_kin = [], []
        for k in range(case["steps"] + 1):
            if k:
                v = v + 0.5 * DT * inputs.EV_PER_AMU * F / mass
                x = x + DT * v
            e, F = _exact_eval(m, x, t, cell)[:2]
            if k:
                v = v + 0.5 * DT * inputs.EV_PER_AMU * F / mass
            e_pot.append(e.sum())
            e_kin.append(0.5 * (mass * v * v).sum() / inputs.EV_PER_AMU)
        return {"pos": x, "vel": v, "e_pot": torch.stack(e_pot), "e_kin": torch.stack(e_kin)}
    if kind == "batch":
        out = {}
        for family, off, pos, types, boxes in _batch(case, seed):
            m, x, t = _model({}, family), _gpu(pos), _gpu(types)
            got = [_exact_eval(m, x[a:b], t[a:b], _cell(box)) for a, b, box in zip(off[:-1], off[1:], boxes)]
            out[family] = {"energies": torch.stack([g[0].sum() for g in got]),
                           "forces": torch.cat([g[1] for g in got]), "virials": torch.stack([g[2] for g in got])}
        return out
    if kind == "train":
        m = _model(case, "water")
        energies, grad = [], 0.0
        for pos, types, box, ref in _train_frames(case, seed):
            e, _, _, dW = _exact_eval(m, _gpu(pos), _gpu(types), _cell(box), params=_gpu(m.params, F64))
            grad = grad + 2.0 * (e.sum() - ref) / len(pos) ** 2 * dW
            energies.append(e.sum())
        return {"energies": torch.stack(energies), "dloss_dparams": grad}
    pos, types, box = _structure(case["family"], case["atoms"], 1000 * seed)
    return _exact_eval(_model(case), _gpu(pos), _gpu(types), _cell(box), descriptors=True)
