"""Cases for timing the ionising-MD library through its public entry points.

Three kinds of pass, each what a user's program does with the library:

* ``run``: a segment of a simulation.  The state (positions, velocities,
  charges, K holes, free-electron gas, step) is restored, ``steps`` timesteps
  are taken in one call, and the whole state is read back.
* ``forces``: one allocation-free force evaluation on device buffers, as a
  plug-in of another program calls it.
* ``analysis``: what is computed from one frame: pair-distance histograms of
  every species pair, fragments and their ion yields, energies.

Samples have the compositions and densities of ``workloads``: water boxes and
droplets, methane clusters (alone and as a batch of replicas), protein
globules in water.  ``phase`` says where in a run the segment sits: "start"
(neutral, room temperature) or "peak" (ionised and heated by the pulse, where
lists are short-lived and every atom has a charge state).

On the mixed path the pair forces are FP32 arithmetic, so positions,
velocities, forces and potential energies come back as the single-precision
frames that trajectory files hold; on the FP64 path they stay FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

R_CUT = 1.2
SKIN = 0.12          # the Verlet buffer of the benchmark
TE_EV = 40.0         # electron temperature at the pulse peak
PULSE = {"methane": (8.0, 10.0, 1e12), "batch": (8.0, 10.0, 1e12), "water": (6.0, 25.0, 5e12),
         "protein": (9.0, 10.0, 1e13), "droplet": (8.0, 20.0, 1e13)}   # keV, fs, photons/um^2
EV_KJ = 96.48533212


def _run(name, sample, atoms, steps, **kw):
    c = {"name": name, "kind": "run", "sample": sample, "atoms": atoms, "steps": steps, "phase": "peak",
         "precision": "mixed", "skin": SKIN, "screening": "debye", "bonded": False, "langevin": 0.0,
         "autotune": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest single sample: one methane cluster, bound by latency and launches
        _run("methane_1500", "methane", 1500, 64),
        # a small cluster with the constructor's defaults: lists rebuilt at every step
        _run("methane_8k_defaults", "methane", 8005, 48, skin=0.0, phase="start"),
        # bulk water, the ordinary size of a single-molecule-imaging run
        _run("water_30k", "water", 30000, 48, autotune=True),
        # solvated protein lattice: all five species, the largest table of charge states
        _run("protein_200k", "protein", 199773, 32, autotune=True),
        # 256 realisations of clusters of 500 to 20,000 atoms in one handle
        _run("methane_batch", "batch", 1400000, 32, autotune=True),
        # the largest single sample
        _run("droplet_2m", "droplet", 1999998, 32, autotune=True),
        # ion-sphere electrostatics, an odd number of molecules
        _run("water_12k_hybrid", "water", 12003, 48, screening="hybrid"),
        # bonded terms and electron-ion coupling on a cluster of the paper's largest size
        _run("methane_45k_bonded_langevin", "methane", 45005, 32, bonded=True, langevin=0.003, phase="start"),
        # the reference-quality path
        _run("water_30k_fp64", "water", 30000, 8, precision="fp64"),
        # forces alone, from device buffers
        {"name": "forces_12k", "kind": "forces", "sample": "water", "atoms": 12297, "phase": "peak",
         "precision": "mixed"},
        # one frame's analysis: a small cluster and a large droplet
        {"name": "analysis_20k", "kind": "analysis", "sample": "methane", "atoms": 20005, "phase": "peak",
         "precision": "mixed"},
        {"name": "analysis_1m", "kind": "analysis", "sample": "droplet", "atoms": 999999, "phase": "peak",
         "precision": "mixed"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["forces", "analysis"])
    phase = rng.choice(["peak", "start"])
    fp64 = rng.random() < 0.15
    prec = "fp64" if fp64 else "mixed"
    if kind == "forces":
        return {"kind": kind, "sample": rng.choice(["water", "methane"]), "atoms": _log(rng, 6600, 16000),
                "phase": phase, "precision": prec}
    sample = rng.choice(["methane", "water", "droplet", "protein", "batch"])
    lo, hi = {"methane": (500, 60000), "water": (6600, 600000), "droplet": (3000, 1200000),
              "protein": (20000, 400000), "batch": (10000, 800000)}[sample]
    if fp64:
        hi = 40000
    n = _log(rng, lo, hi)
    if kind == "analysis":
        return {"kind": kind, "sample": sample, "atoms": n, "phase": phase, "precision": prec}
    steps = 8 if fp64 else (rng.randrange(33, 65) if n < 60000 else rng.randrange(17, 33))
    c = _run("", sample, n, steps, phase=phase, precision=prec, skin=rng.choice([SKIN, SKIN, 0.08, 0.0]),
             screening=rng.choice(["debye", "debye", "debye", "hybrid"]), bonded=rng.random() < 0.25,
             langevin=0.003 if rng.random() < 0.2 else 0.0, autotune=rng.random() < 0.3)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _tile(s, edge, m):
    """m^3 copies of a periodic sample side by side."""
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = (s.x[None] + (g * edge)[:, None, :]).reshape(-1, 3)
    frag = (s.fragment[None] + np.arange(len(g))[:, None] * (int(s.fragment.max()) + 1)).reshape(-1)
    return x, np.tile(s.species, len(g)), frag.astype(np.int32)


def _water_block(n_mol, seed):
    """A periodic water block of about n_mol molecules or fewer, and the copies per edge that make n_mol."""
    m = max(1, math.ceil((n_mol / 4500) ** (1 / 3)))
    per = max(1, round(n_mol / m ** 3))
    edge = 6.7 * (per / 10000) ** (1 / 3)
    return W.water_box(per, edge, seed), edge, m


def _one(kind, atoms, seed):
    """(positions, species, fragments, box edge or 0, electron-gas volume) of one sample."""
    if kind == "methane":
        s = W.methane_cluster(max(2, atoms // 5), seed)
        return s.x, s.species, s.fragment, 0.0, float(s.volume[0])
    if kind == "water":
        s, edge, m = _water_block(atoms // 3, seed)
        return (*_tile(s, edge, m), edge * m, (edge * m) ** 3)
    if kind == "protein":
        m = 3 if atoms > 100000 else 2 if atoms > 40000 else 1
        s = W.protein_crystal(round(atoms / m ** 3), seed, n_cells=1)
        edge = float(s.box[0, 0])
        return (*_tile(s, edge, m), edge * m, (edge * m) ** 3)
    n_mol = atoms // 3
    radius = (3 * n_mol / (4 * math.pi * 33.25)) ** (1 / 3)
    edge = 6.7 * 0.1728 ** (1 / 3)
    m = math.ceil(2 * (radius + 0.3) / edge)
    x, sp, fr = _tile(W.water_box(1728, edge, seed), edge, m)
    o = x.reshape(-1, 3, 3)[:, 0] - 0.5 * m * edge          # a molecule goes by its oxygen
    keep = np.argpartition((o * o).sum(1), n_mol - 1)[:n_mol] if n_mol < len(o) else np.arange(len(o))
    keep.sort()
    mol = x.reshape(-1, 3, 3)[keep] - 0.5 * m * edge
    wrap = mol - mol[:, :1]                                 # molecules cut by a block's face are made whole
    mol = mol - edge * m * np.round(wrap / (edge * m))
    near = mol - mol[:, :1]
    mol = mol - edge * np.round(near / edge)
    return mol.reshape(-1, 3), np.tile(sp[:3], len(keep)), np.repeat(np.arange(len(keep), dtype=np.int32), 3), 0.0, \
        4 / 3 * math.pi * radius ** 3


def _inputs(case, seed):
    """The sample and the state to restore, from the seed alone."""
    rng = np.random.default_rng([int(seed), 2401])
    kind = case["sample"]
    if kind == "batch":
        # 16 cluster sizes over the range, each of them several replicas: the sizes are the case's, the rest the seed's
        sizes = np.exp(np.random.default_rng(case["atoms"]).uniform(np.log(500), np.log(20000), 16)).astype(int) // 5
        shapes = [_one("methane", 5 * int(n), int(rng.integers(1 << 30))) for n in sizes]
        order, total = [], 0
        while total < case["atoms"] and len(order) < 256:
            order.append((7 * len(order)) % 16)
            total += len(shapes[order[-1]][0])
        parts = [shapes[k] for k in order]
    else:
        parts = [_one(kind, case["atoms"], int(rng.integers(1 << 30)))]
    off = np.concatenate([[0], np.cumsum([len(p[0]) for p in parts])]).astype(np.int32)
    fbase = np.concatenate([[0], np.cumsum([int(p[2].max()) + 1 for p in parts])])
    x = np.concatenate([p[0] for p in parts])
    sp = np.concatenate([p[1] for p in parts]).astype(np.uint8)
    frag = np.concatenate([p[2] + b for p, b in zip(parts, fbase)]).astype(np.int32)
    n, R = len(x), len(parts)
    box = np.array([[p[3]] * 3 for p in parts])
    vol = np.array([p[4] for p in parts])
    peak = case["phase"] == "peak"
    # room temperature, or ions heated to a few eV
    v = rng.standard_normal((n, 3)) * np.sqrt((EV_KJ * 4.0 if peak else W.KB_KJ * 300.0) / W.MASS[sp])[:, None]
    q = rng.binomial(W.Z[sp], np.where(sp == W.H, 0.4, 0.15)).astype(np.uint8) if peak else np.zeros(n, np.uint8)
    h = ((rng.random(n) < 0.01) & (W.Z[sp] - q >= 3)).astype(np.uint8) if peak else np.zeros(n, np.uint8)
    n_e = np.add.reduceat(q.astype(np.int64), off[:-1])
    state = {"x": x, "v": v, "q": q, "h": h, "n_e": n_e, "step": 0,
             "e_gas_mev": np.rint(n_e * 1500.0 * TE_EV).astype(np.int64)}
    s = W.Sample(x=x, v=v, species=sp, fragment=frag, q0=np.zeros(n, np.uint8), replica_offset=off,
                 seed=rng.integers(1, 1 << 62, R).astype(np.uint64), box=box, volume=vol)
    if case.get("bonded"):
        s = W.with_topology(s)
    return s, state


def _pulse(case):
    kev, fwhm, flu = PULSE[case["sample"]]
    return kev, W.Pulse(kev, fwhm, flu, 0.0)


def _t_start(case):
    dt = 1000.0 * W.DT_PS
    return (-0.5 * case.get("steps", 1) * dt) if case["phase"] == "peak" else -_pulse(case)[1].fwhm_fs


RESTORE = M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_PLASMA | M.MD_FIELD_STEP
READ = M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_PLASMA | M.MD_FIELD_COUNTS


def prepare(case, seed):
    s, state = _inputs(case, seed)
    if case["kind"] == "forces":
        dev = {"x": torch.from_numpy(s.x).cuda(), "species": torch.from_numpy(s.species).cuda(),
               "q": torch.from_numpy(state["q"]).cuda(), "fragment": torch.from_numpy(s.fragment).cuda()}
        f = torch.empty((s.n_atoms, 3), dtype=torch.float64, device="cuda")
        inp = M.MDForcesInput()
        inp.n_atoms = s.n_atoms
        inp.d_x, inp.d_species = dev["x"].data_ptr(), dev["species"].data_ptr()
        inp.d_q, inp.d_fragment = dev["q"].data_ptr(), dev["fragment"].data_ptr()
        inp.kappa, inp.r_cut, inp.coulomb_f = float(_kappa(state, s)[0][0]), R_CUT, M.COULOMB_F
        inp.precision = M.MD_PREC_FP64 if case["precision"] == "fp64" else M.MD_PREC_MIXED
        inp.n_species = len(W.Z)
        for k in range(len(W.Z)):
            inp.z[k], inp.lj_sigma0[k], inp.lj_eps0[k] = int(W.Z[k]), float(W.LJ_SIGMA0[k]), float(W.LJ_EPS0[k])
        for d in range(3):
            inp.box[d] = float(s.box[0, d])
        return {"case": case, "inp": inp, "dev": dev, "f": f}
    kev, pulse = _pulse(case)
    g = M.IonisingMD(s, W.atomic_data(kev), precision=case["precision"], r_cut=R_CUT, dt_ps=W.DT_PS,
                     max_steps=case.get("steps", 1) + 1, t_start_fs=_t_start(case),
                     autotune=case.get("autotune", False), list_skin_nm=case.get("skin", SKIN),
                     screening=case.get("screening", "debye"), langevin_g=case.get("langevin") or None)
    g.set_pulse([pulse])
    if case["kind"] == "analysis":
        g.set_state(RESTORE, **state)
    return {"case": case, "md": g, "state": state}


def _out(case, a):
    return a if case["precision"] == "fp64" else a.astype(np.float32)


def run(state):
    case = state["case"]
    if case["kind"] == "forces":
        M.md_forces_noalloc(state["inp"], state["f"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["f"] if case["precision"] == "fp64" else state["f"].float()
    g = state["md"]
    if case["kind"] == "analysis":
        rdf = g.rdf(R_CUT, 240)
        label, yields = g.fragments(0.16)
        e_kin, e_pot, pairs = g.energies()
        return {"rdf": rdf, "label": label, "yields": yields, "e_kin": e_kin, "e_pot": _out(case, e_pot),
                "pairs": pairs}
    g.set_state(RESTORE, **state["state"])
    g.step(case["steps"])
    r = g.get_state(READ)
    r["x"], r["v"] = _out(case, r["x"]), _out(case, r["v"])
    return r


# ---------------------------------------------------------------------------
# work: 41 operations per pair within the cutoff (once per pair), ~120 per atom
# ---------------------------------------------------------------------------
def _pairs(case):
    n, rho = case["atoms"], {"water": 99.75, "droplet": 99.75, "protein": 102.0, "methane": 78.8, "batch": 78.8}[case["sample"]]
    if case["sample"] in ("water", "protein"):
        return 0.5 * n * rho * 4 / 3 * math.pi * R_CUT ** 3
    one = min(n, 5500) if case["sample"] == "batch" else n
    u = R_CUT / (3 * one / (4 * math.pi * rho)) ** (1 / 3)       # the part of an atom's cutoff sphere inside the sample
    return min(0.5 * n * one, 0.5 * n * rho * 4 / 3 * math.pi * R_CUT ** 3 * max(0.2, 1 - 9 / 16 * u + u ** 3 / 32))


def work(case):
    n, k, wide = case["atoms"], case.get("steps", 1), 8 if case["precision"] == "fp64" else 4
    evals = {"run": k + 1, "forces": 1, "analysis": 2}[case["kind"]]
    # per evaluation: position, charge, type in, force out; per step: x, v in and out, charge state in and out;
    # per pass: the state in and out
    per_atom = evals * (3 * 8 + 2 + 4 + 3 * 8) + (k * (12 * 8 + 4) if case["kind"] == "run" else 0) + 2 * (6 * wide + 2)
    return {"bytes": float(n * per_atom), "flops": evals * 41.0 * _pairs(case) + 120.0 * n * k}


# ---------------------------------------------------------------------------
# the same in 64 bits, all pairs
# ---------------------------------------------------------------------------
def _kappa(st, s):
    """Inverse Debye length and electron density per replica from the gas's count and energy."""
    ne = st["n_e"] / s.volume
    te = np.where(st["n_e"] > 0, st["e_gas_mev"] / np.maximum(1500.0 * st["n_e"], 1.0), 0.0)
    return np.where(ne > 0, np.sqrt(4 * math.pi * M.COULOMB_F * ne / (np.maximum(te, 1.0) * EV_KJ)), 0.0), ne, te


def _cuda(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda").to(dtype)


def _ion(q, ne, kap):
    """Transition radius, constants and outer amplitude of an ion of charge q (uniform electron density ne)."""
    q = np.asarray(q, float)
    rp, c1, G = np.zeros_like(q), np.zeros_like(q), q.copy()
    if ne > 0 and kap > 0:
        sr = kap * np.cbrt(3 * q / (4 * math.pi * ne))
        t = np.cbrt(1 + sr ** 3)
        rp = sr ** 3 / (kap * (t * t + t + 1))
        y = kap * rp
        D = 3 + 3 * y + y * y
        c1, G = -q * kap * (3 + 1.5 * y) / D, 3 * q * np.exp(y) / D
    return rp, c1, G, -2 * math.pi * ne / 3


def _replica_forces(x, q, sp, frag, box, kap, ne, hybrid, topo):
    """Forces [n,3], potential energy and pairs within the cutoff of one replica."""
    f0, rc = M.COULOMB_F, R_CUT
    n = len(q)
    X, Q = _cuda(x), _cuda(q)
    sg = _cuda(W.LJ_SIGMA0[sp] * (1 - q / W.Z[sp]))
    ep, fr = _cuda(np.sqrt(W.LJ_EPS0[sp])), _cuda(frag, torch.int64)
    F = torch.zeros_like(X)
    U, pairs = 0.0, 0
    ion = [_cuda(a) for a in _ion(q, ne, kap)[:3]] if hybrid else None
    c2 = -2 * math.pi * ne / 3
    ids = torch.arange(n, device="cuda")
    step = max(1, int(3e7 // n))
    for a in range(0, n, step):
        r2 = torch.zeros((min(step, n - a), n - a), dtype=torch.float64, device="cuda")
        for d in range(3):
            e = X[a:a + step, None, d] - X[None, a:, d]
            if box > 0:
                e = e - box * torch.round(e / box)
            r2 += e * e
        i, j = torch.nonzero((r2 < rc * rc) & (ids[a:a + step, None] < ids[None, a:]), as_tuple=True)
        i, j = i + a, j + a
        d = X[i] - X[j]
        if box > 0:
            d = d - box * torch.round(d / box)
        rr = (d * d).sum(1)
        r = rr.sqrt()
        on = (fr[i] != fr[j]).double()
        s6 = (0.5 * (sg[i] + sg[j])) ** 6
        c6 = 4 * ep[i] * ep[j] * s6 * on
        c12 = c6 * s6
        e = torch.exp(-kap * r)
        lj = c12 / rr ** 6 - c6 / rr ** 3
        fs = e * ((12 * c12 / rr ** 6 - 6 * c6 / rr ** 3) / rr + kap / r * lj)
        erc = math.exp(-kap * rc)
        u = e * lj - erc * (c12 / rc ** 12 - c6 / rc ** 6)
        if hybrid:
            for p, o in ((i, j), (j, i)):
                rp, c1, G = (t[p] for t in ion)
                inside = r < rp
                phi = torch.where(inside, Q[p] / r + c1 - c2 * rr, G * e / r)
                dphi = torch.where(inside, Q[p] / rr + 2 * c2 * r, G * e * (1 + kap * r) / rr)
                cut = torch.where(rp > rc, Q[p] / rc + c1 - c2 * rc * rc, G * erc / rc)
                fs = fs + 0.5 * f0 * Q[o] * dphi / r
                u = u + 0.5 * f0 * Q[o] * (phi - cut)
        else:
            qq = f0 * Q[i] * Q[j]
            fs = fs + qq * e * (1 / r + kap) / rr
            u = u + qq * (e / r - erc / rc)
        F.index_add_(0, i, fs[:, None] * d)
        F.index_add_(0, j, -fs[:, None] * d)
        U += float(u.sum())
        pairs += len(r)
    if topo is not None:
        Xg = X.clone().requires_grad_(True)
        b, t = _cuda(topo.bonds, torch.int64), _cuda(topo.angles, torch.int64)
        bp, tp = _cuda(topo.bond_params)[b[:, 2]], _cuda(topo.angle_params)[t[:, 3]]
        r = (Xg[b[:, 0]] - Xg[b[:, 1]]).norm(dim=1)
        ub = (1 - Q[b[:, :2]].sum(1) / 2).clamp(0, 1) * bp[:, 0] * (1 - torch.exp(-bp[:, 2] * (r - bp[:, 1]))) ** 2
        p, w = Xg[t[:, 0]] - Xg[t[:, 1]], Xg[t[:, 2]] - Xg[t[:, 1]]
        th = torch.atan2(torch.linalg.cross(p, w).norm(dim=1), (p * w).sum(1))
        ut = (1 - Q[t[:, :3]].sum(1) / 3).clamp(0, 1) * 0.5 * tp[:, 0] * (th - tp[:, 1]) ** 2
        (ub.sum() + ut.sum()).backward()
        F, U = F - Xg.grad, U + float(ub.sum() + ut.sum())
    return F.cpu().numpy(), U, pairs


def _own_terms(topo, a, b):
    """The bonded terms of the replica of atoms a .. b - 1, by that replica's own atom indices."""
    if topo is None:
        return None
    bonds, angles = (t[(t[:, 0] >= a) & (t[:, 0] < b)] for t in (topo.bonds, topo.angles))
    return W.Topology(bonds=bonds - np.array([a, a, 0], bonds.dtype), bond_params=topo.bond_params,
                      angles=angles - np.array([a, a, a, 0], angles.dtype), angle_params=topo.angle_params)


def _forces(case, s, st):
    kap, ne, _ = _kappa(st, s)
    F, U, pairs = np.empty((s.n_atoms, 3)), np.zeros(s.n_replicas), 0
    for r in range(s.n_replicas):
        a, b = int(s.replica_offset[r]), int(s.replica_offset[r + 1])
        F[a:b], U[r], k = _replica_forces(st["x"][a:b], st["q"][a:b], s.species[a:b], s.fragment[a:b],
                                          float(s.box[r, 0]), float(kap[r]), float(ne[r]),
                                          case.get("screening") == "hybrid", _own_terms(s.topology, a, b))
        pairs += k
    return F, U, pairs


def _philox(key, c0, c1, c2):
    """Philox4x32-10 (Salmon et al., SC'11) for counters (c0, c1, c2, 0)."""
    m32 = np.uint64(0xffffffff)
    c = [np.asarray(c0, np.uint64), np.full(len(c0), c1, np.uint64), np.full(len(c0), c2, np.uint64),
         np.zeros(len(c0), np.uint64)]
    k = [np.asarray(key, np.uint64) & m32, np.asarray(key, np.uint64) >> np.uint64(32)]
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k[0], p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k[1], p0 & m32]
        k = [(k[0] + np.uint64(0x9E3779B9)) & m32, (k[1] + np.uint64(0xBB67AE85)) & m32]
    return c


def _fluence(p, t0, dt):
    """Photons per nm^2 of a Gaussian pulse between t0 and t0 + dt (fs)."""
    z0, z1 = ((t - p.t_center_fs) * 2 * math.sqrt(math.log(2)) / p.fwhm_fs for t in (t0, t0 + dt))
    if z0 >= 0:
        part = 0.5 * (math.erfc(z0) - math.erfc(z1))
    elif z1 <= 0:
        part = 0.5 * (math.erfc(-z1) - math.erfc(-z0))
    else:
        part = 1 - 0.5 * (math.erfc(-z0) + math.erfc(z1))
    return p.fluence_ph_um2 * 1e-6 * part


def _charges(case, s, st, atom, rep, loc, step, counts):
    """One stochastic charge update: at most one event per atom."""
    dt = W.DT_PS
    dF = _fluence(_pulse(case)[1], _t_start(case) + 1000 * dt * step, 1000 * dt)
    _, ne, te = _kappa(st, s)
    xt = np.clip(te / atom.dte_ev, 0, atom.n_te - 1)
    i0 = np.minimum(xt.astype(int), atom.n_te - 2)[rep]
    wt = (xt[rep] - i0)
    q, h, sp = st["q"].astype(int), st["h"].astype(int), s.species
    Z, ts = W.Z[sp], atom.ts_offset[sp] + q
    interp = lambda K: K[ts, i0] + wt * (K[ts, i0 + 1] - K[ts, i0])  # noqa: E731
    tau = np.where(atom.tau_auger_ps > 0, dt / np.where(atom.tau_auger_ps > 0, atom.tau_auger_ps, 1), 0)[sp]
    c0 = atom.sigma_pi[ts, h] * dF
    c1 = c0 + np.where(h == 1, tau, 0)
    c2 = c1 + np.where(q < Z, (ne * dt)[rep] * interp(atom.k_ci), 0)
    lam = c2 + np.where((q > 0) & (h == 0), (ne * dt)[rep] * interp(atom.k_rec), 0)
    w = _philox(s.seed[rep], loc, step, 0)
    u = [((w[k] >> np.uint64(5)) * np.uint64(1 << 26) + (w[k + 1] >> np.uint64(6))).astype(float) * 2.0 ** -53 for k in (0, 2)]
    t = u[1] * lam
    ch = np.where(u[0] < -np.expm1(-lam), (t >= c0).astype(int) + (t >= c1) + (t >= c2), -1)
    qn, hn = q + np.where(ch < 0, 0, np.where(ch == 3, -1, 1)), h.copy()
    opens = (ch == 0) & (Z >= 3) & (h == 0) & (Z - qn >= 2)
    hn[opens] = 1
    hn[(ch == 1) | (((ch == 0) | (ch == 2)) & (qn == Z))] = 0
    de = np.select([ch == 0, ch == 1, ch == 2, ch == 3],
                   [atom.e_pi_mev[ts, h], atom.e_auger_mev[sp], -atom.ip_mev[ts], atom.ip_mev[ts - 1]], 0)
    off = s.replica_offset[:-1]
    st["n_e"] = st["n_e"] + np.add.reduceat(qn - q, off)
    st["e_gas_mev"] = np.maximum(st["e_gas_mev"] + np.add.reduceat(de, off), 0)
    for k in range(4):
        counts[:, k] += np.add.reduceat((ch == k).astype(np.int64), off)
    st["q"], st["h"] = qn.astype(np.uint8), hn.astype(np.uint8)


def exact(case, seed):
    n, k = case["atoms"], case.get("steps", 1)
    one = min(n, 20000) if case["sample"] == "batch" else n
    if float(n) * one * (k if case["kind"] == "run" else 1) > 5e10:
        return None      # all pairs would take too long
    s, st = _inputs(case, seed)
    F, U, pairs = _forces(case, s, st)
    if case["kind"] == "forces":
        return F
    m = W.MASS[s.species][:, None]
    off = s.replica_offset[:-1]
    if case["kind"] == "analysis":
        return {"rdf": None, "label": None, "yields": None, "pairs": pairs, "e_pot": U,
                "e_kin": np.add.reduceat(0.5 * (m * st["v"] ** 2).sum(1), off)}
    dt, atom = W.DT_PS, W.atomic_data(_pulse(case)[0])
    rep = np.repeat(np.arange(s.n_replicas), np.diff(s.replica_offset))
    loc = np.arange(s.n_atoms) - off[rep]
    counts = np.zeros((s.n_replicas, 4), np.int64)
    L = s.box[rep]
    for step in range(k):
        v = st["v"] + 0.5 * dt * F / m
        if case["langevin"]:
            _, ne, te = _kappa(st, s)
            c = np.exp(-ne * case["langevin"] * dt)[rep][:, None]
            w = [(a.astype(float) + 0.5) * 2.0 ** -32 for a in _philox(s.seed[rep], loc, step, 1)]
            ra, rb = np.sqrt(-2 * np.log(w[0])), np.sqrt(-2 * np.log(w[2]))
            xi = np.stack([ra * np.cos(2 * np.pi * w[1]), ra * np.sin(2 * np.pi * w[1]), rb * np.cos(2 * np.pi * w[3])], 1)
            v = c * v + np.sqrt((1 - c * c) * (te * EV_KJ)[rep][:, None] / m) * xi
        x = st["x"] + dt * v
        st["x"] = np.where(L > 0, x - L * np.floor(x / np.where(L > 0, L, 1)), x)
        _charges(case, s, st, atom, rep, loc, step, counts)
        F, _, _ = _forces(case, s, st)
        st["v"] = v + 0.5 * dt * F / m
    kap, _, te = _kappa(st, s)
    return {"x": st["x"], "v": st["v"], "q": None, "h": None, "n_e": None, "e_gas_mev": None, "te_ev": te,
            "kappa": kap, "event_counts": None}
