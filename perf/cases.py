"""The calls whose speed this repository follows, as its users make them.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (a
batch on the device, parameters, a context, a captured graph, a descriptor store), ``run`` makes
the call through the public entry points and returns its outputs, ``work`` counts what the call
cannot do without, and ``exact`` evaluates the same outputs in 64 bits with plain torch.

Energies, losses, charges and trajectories leave the library as FP64 sums of FP32 terms; they are
handed on here in FP32, the precision that they carry (forces, gradients, descriptors and atomic
energies are FP32 already).
"""
import math

import numpy as np
import torch

from paper_2305_11805_gb300 import panna as P
from paper_2305_11805_gb300 import workloads as W

PRECISION = {"fp32": P.PANNA_MLP_FP32, "bf16": P.PANNA_MLP_BF16}


def listed():
    return [
        # Langevin dynamics of one 16-atom carbon cell: the smallest step a simulation takes, where
        # launches and latency are everything
        dict(name="md_carbon16", kind="md", structure="carbon", n=1, precision="fp32", steps=10, skin=0.5),
        # one call on a small periodic box: a geometry optimiser or a plugin asking for forces
        dict(name="infer_diamond64", kind="infer", structure="diamond", n=2, precision="fp32", virial=True,
             graph=False),
        # a training step on a small minibatch of molecules
        dict(name="train_molecules50", kind="train", structure="molecules", n=50, precision="fp32"),
        # a training step on a large minibatch of molecules (the benchmark's training workload)
        dict(name="train_molecules1024", kind="train", structure="molecules", n=1024, precision="fp32"),
        # the same step with precomputed descriptors and Jacobians
        dict(name="store_molecules1024", kind="store", structure="molecules", n=1024, precision="fp32"),
        # FP32 inference with the virial: a mid-sized liquid box under a barostat
        dict(name="infer_water3999_fp32", kind="infer", structure="water", n=3999, precision="fp32", virial=True,
             graph=False),
        # a BF16 evaluation of a large liquid box (the benchmark's precision workload)
        dict(name="infer_water32768", kind="infer", structure="water", n=32768, precision="bf16", virial=False,
             graph=False),
        # many boxes of uneven sizes through one captured graph (the headline workload, fewer boxes)
        dict(name="infer_ragged256", kind="infer", structure="ragged", n=256, precision="bf16", virial=True,
             graph=True),
        # the largest single box (the benchmark's scale workload)
        dict(name="infer_fcc1048576", kind="infer", structure="fcc", n=64, precision="bf16", virial=False,
             graph=False),
        # descriptors of a dataset, for analysis or selection
        dict(name="descriptors_ragged48", kind="descriptors", structure="ragged", n=48, precision="fp32"),
        # charge equilibration: energies, charges and forces of charged clusters
        dict(name="qeq_nacl1024", kind="qeq", structure="nacl", n=1024, precision="fp32"),
        # the standard Behler-Parrinello angular term
        dict(name="infer_bp_water4096", kind="infer", structure="water_bp", n=4096, precision="bf16", virial=False,
             graph=False),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["md", "infer", "infer", "infer", "infer", "infer", "train", "train", "store", "descriptors",
                       "qeq", "bp"])
    if what == "md":
        return dict(kind="md", structure="carbon", n=_log_int(rng, 1, 64), precision=rng.choice(["fp32", "bf16"]),
                    steps=rng.randint(4, 10), skin=rng.choice([0.0, 0.4, 0.6]))
    if what in ("train", "store"):
        return dict(kind=what, structure="molecules", n=_log_int(rng, 8, 1024), precision="fp32")
    if what == "descriptors":
        return dict(kind="descriptors", structure=rng.choice(["ragged", "water", "fcc", "molecules"]),
                    n=0, precision="fp32", scale=rng.random())
    if what == "qeq":
        return dict(kind="qeq", structure="nacl", n=_log_int(rng, 16, 2048), precision="fp32")
    if what == "bp":
        return dict(kind="infer", structure="water_bp", n=_log_int(rng, 400, 8192),
                    precision=rng.choice(["fp32", "bf16"]), virial=rng.random() < 0.5, graph=False)
    structure = rng.choice(["diamond", "water", "ragged", "fcc", "molecules", "carbon"])
    lo, hi = RANGE[structure]
    precision = rng.choice(["bf16", "fp32"])
    if precision == "fp32":
        lo, hi = RANGE_FP32[structure]
    return dict(kind="infer", structure=structure, n=_log_int(rng, lo, hi), precision=precision,
                virial=rng.random() < 0.5, graph=rng.random() < 0.4)


# sizes per structure: cells per edge (diamond, fcc), atoms (water), configurations (the others)
RANGE = {"diamond": (2, 16), "water": (500, 32768), "ragged": (1, 256), "fcc": (4, 64), "molecules": (8, 2048),
         "carbon": (1, 2048), "nacl": (16, 2048), "water_bp": (400, 8192)}
RANGE_FP32 = {"diamond": (2, 16), "water": (500, 16384), "ragged": (1, 128), "fcc": (4, 40), "molecules": (8, 2048),
              "carbon": (1, 1024)}


def _size(case):
    """The case's n; cases that give a place in their structure's range instead have it from there."""
    if case["n"]:
        return int(case["n"])
    lo, hi = RANGE_FP32[case["structure"]]
    return max(lo, int(round(lo * (hi / lo) ** float(case["scale"]))))


# ------------------------------------------------------------------------------------ inputs

def _box_positions(rng, n, L, dmin=0.9, spacing=1.45):
    """n random positions in a periodic cube, at least dmin apart: random sites of a fine grid, each
    displaced at random inside its site."""
    k = max(1, int(L / spacing))
    while k ** 3 < n:
        k += 1
    h = L / k
    site = rng.permutation(k ** 3)[:n]
    x = np.stack([site // (k * k), site // k % k, site % k], 1).astype(np.float64)
    x += 0.5 + rng.uniform(-0.5, 0.5, size=x.shape) * max(0.0, 1.0 - dmin / h)
    return x * h


def _lattice(rng, basis, ncell, a, sigma):
    g = np.arange(ncell)
    cells = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 1, 3)
    x = ((cells + basis[None]) * a).reshape(-1, 3)
    return np.mod(x + rng.normal(0.0, sigma, size=x.shape), ncell * a)


def _one_box(pos, spec, L, n_species):
    return W.System(np.array([0, len(pos)], np.int64), pos, spec.astype(np.int32), (np.eye(3) * L).reshape(1, 9),
                    np.ones((1, 3), np.uint8), n_species)


def _ragged_sizes(n_cfg):
    """Box sizes spread evenly over the logarithm of 32..4096, ends included in the middle of bins."""
    q = (np.arange(n_cfg) + 0.5) / n_cfg
    return np.rint(32.0 * 128.0 ** q).astype(np.int64)


def _molecule_sizes(n_mol):
    return 5 + (np.arange(n_mol, dtype=np.int64) * 25 // n_mol if n_mol >= 25 else np.arange(n_mol) * 7 % 25)


def _chains(rng, sizes, dmin=0.9):
    """Random bonded chains (bonds of 1.0 to 1.5 A, every two atoms at least dmin apart), grown side
    by side."""
    m, top = len(sizes), int(sizes.max())
    pos = np.full((m, top, 3), 1e9)
    pos[:, 0] = 0.0
    at = np.ones(m, np.int64)
    tries = np.zeros(m, np.int64)
    while True:
        todo = np.nonzero(at < sizes)[0]
        if len(todo) == 0:
            return np.concatenate([pos[c, :s] for c, s in enumerate(sizes)])
        v = rng.normal(size=(len(todo), 3))
        v *= (rng.uniform(1.0, 1.5, size=len(todo)) / np.sqrt((v * v).sum(1)))[:, None]
        p = pos[todo, at[todo] - 1] + v
        d2 = ((pos[todo] - p[:, None]) ** 2).sum(-1)
        d2[np.arange(top)[None] >= at[todo][:, None]] = np.inf
        ok = d2.min(1) >= dmin * dmin
        pos[todo[ok], at[todo[ok]]] = p[ok]
        at[todo[ok]] += 1
        tries[todo[ok]] = 0
        tries[todo[~ok]] += 1
        stuck = tries > 200
        at[stuck], tries[stuck] = 1, 0


def _inputs(case, seed):
    """The batch, descriptor, networks and parameters of a case (host arrays), from the seed alone."""
    rng = np.random.default_rng(1000003 * int(seed) + 17)
    s, n = case["structure"], _size(case)
    extra = {}
    if s == "diamond":
        a, gains = 5.43, W.GAINS["diamond64"]
        pos = _lattice(rng, W.DIAMOND_BASIS, n, a, 0.1)
        system = _one_box(pos, np.zeros(len(pos)), n * a, 1)
        desc, hidden = W.descriptor_params(1, 4.6, 32, 8, 8), (256, 128, 32)
    elif s in ("water", "water_bp"):
        L, gains = (n / 0.1003) ** (1.0 / 3.0), W.GAINS["water32k"]
        spec = np.ones(n)
        spec[rng.permutation(n)[:int(round(n / 3))]] = 0
        system = _one_box(_box_positions(rng, n, L), spec, L, 2)
        desc, hidden = W.descriptor_params(2, 6.0, 32, 8, 8), (256, 128)
        if s == "water_bp":
            gains = (1.0, 0.05)
            desc.angular = "bp"
            desc.bp_lambda, desc.bp_zeta = np.array([1.0, -1.0, 1.0, -1.0]), np.array([1.0, 1.0, 4.0, 4.0])
            desc.bp_eta = np.array([0.005, 0.05])
    elif s == "fcc":
        a, gains = 4.05, W.GAINS["fcc1m"]
        pos = _lattice(rng, W.FCC_BASIS, n, a, 0.05)
        system = _one_box(pos, np.zeros(len(pos)), n * a, 1)
        desc, hidden = W.descriptor_params(1, 5.0, 64, 16, 8), (128, 64)
    elif s == "ragged":
        gains = W.GAINS["ragged4096"]
        sizes = rng.permutation(_ragged_sizes(n))
        pos, spec, cell = [], [], []
        for m in sizes:
            L = (m / 0.05) ** (1.0 / 3.0)
            pos.append(_box_positions(rng, int(m), L))
            spec.append(rng.choice(3, size=int(m), p=rng.dirichlet([1.0, 1.0, 1.0])))
            cell.append((np.eye(3) * L).ravel())
        system = W.System(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), np.concatenate(pos),
                          np.concatenate(spec).astype(np.int32), np.asarray(cell), np.ones((n, 3), np.uint8), 3)
        desc, hidden = W.descriptor_params(3, 5.5, 32, 8, 8), (128, 32)
    elif s == "molecules":
        gains = W.GAINS["molecules1024"]
        sizes = rng.permutation(_molecule_sizes(n))
        pos = _chains(rng, sizes)
        spec = rng.choice(4, size=len(pos), p=[0.5, 0.3, 0.1, 0.1])
        system = W.System(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), pos, spec.astype(np.int32),
                          np.zeros((n, 9)), np.zeros((n, 3), np.uint8), 4)
        desc, hidden = W.descriptor_params(4, 5.2, 32, 8, 8), (128, 32)
        extra["e_ref"] = rng.normal(0.0, 1.0, size=n) * np.sqrt(sizes)
        extra["f_ref"] = rng.normal(0.0, 0.5, size=(len(pos), 3)).astype(np.float32)
    elif s == "carbon":
        a, gains = 3.567, W.GAINS["carbon16"]
        L = np.array([2 * a, a, a])
        ideal = np.concatenate([(W.DIAMOND_BASIS + np.array([c, 0, 0])) * a for c in range(2)])
        pos = np.mod(ideal[None] + rng.normal(0.0, 0.05, size=(n, 16, 3)), L).reshape(-1, 3)
        system = W.System(np.arange(n + 1, dtype=np.int64) * 16, pos, np.zeros(16 * n, np.int32),
                          np.tile(np.diag(L).reshape(1, 9), (n, 1)), np.ones((n, 3), np.uint8), 1)
        desc, hidden = W.descriptor_params(1, 5.0, 24, 16, 8), (64, 32)
        extra["vel"] = rng.normal(0.0, 0.0045, size=(16 * n, 3))   # 300 K, A/fs
    elif s == "nacl":
        wl = W.nacl(int(seed), n)
        return dict(system=wl.system, desc=wl.desc, archs=wl.archs, theta=wl.theta.astype(np.float32), qeq=wl.qeq,
                    charge=wl.charge)
    else:
        raise ValueError(s)
    acts = (W.ACT_GAUSSIAN,) * len(hidden) + (W.ACT_LINEAR,)
    archs = [W.MLPArch((desc.D,) + hidden + (1,), acts) for _ in range(desc.n_species)]
    theta = W.init_weights(rng, desc, archs, *gains).astype(np.float32)
    return dict(system=system, desc=desc, archs=archs, theta=theta, **extra)


# ------------------------------------------------------------------------------------ the calls

MD = dict(dt=0.5, temperature=300.0, friction=0.01, mass=[12.011])


def prepare(case, seed):
    x = _inputs(case, seed)
    st = dict(case=case, pot=P.Potential(x["desc"], x["archs"]), sys=P.DeviceSystem(x["system"]),
              theta=torch.as_tensor(x["theta"], device="cuda"))
    kind, N, C = case["kind"], x["system"].n_atoms, x["system"].n_cfg
    if kind == "md":
        st.update(pos0=st["sys"].pos.clone(), vel0=torch.as_tensor(x["vel"], device="cuda"),
                  vel=torch.empty((N, 3), dtype=torch.float64, device="cuda"), seed=int(seed),
                  F=torch.empty((N, 3), dtype=torch.float32, device="cuda"),
                  E=torch.empty(C, dtype=torch.float64, device="cuda"))
    if kind in ("train", "store"):
        st.update(e_ref=torch.as_tensor(x["e_ref"], device="cuda"), f_ref=torch.as_tensor(x["f_ref"], device="cuda"))
    if kind == "store":
        st["store"] = P.Store(st["pot"], st["sys"])
    if kind == "qeq":
        P.panna_set_qeq(st["pot"].ctx, x["qeq"]["sigma"], x["qeq"]["chi0"], x["qeq"]["hard0"])
        st["charge"] = torch.as_tensor(x["charge"], device="cuda")
    if kind == "infer" and case["graph"]:
        st.update(E=torch.empty(C, dtype=torch.float64, device="cuda"),
                  Ea=torch.empty(N, dtype=torch.float32, device="cuda"),
                  F=torch.empty((N, 3), dtype=torch.float32, device="cuda"),
                  V=torch.empty((C, 3, 3), dtype=torch.float64, device="cuda") if case["virial"] else None)
        P.panna_capture(st["pot"].ctx, st["sys"], st["theta"], PRECISION[case["precision"]], st["E"], st["Ea"],
                        st["F"], st["V"])
    return st


def run(st):
    case, pot, sysd, theta = st["case"], st["pot"], st["sys"], st["theta"]
    kind, prec = case["kind"], PRECISION[case["precision"]]
    if kind == "infer":
        if case["graph"]:
            P.panna_replay(pot.ctx)
            E, Ea, F, V = st["E"], st["Ea"], st["F"], st["V"]
        else:
            E, Ea, F, V = pot.energy_forces(sysd, theta, prec, virial=case["virial"])
        return {"E": E.float(), "E_atom": Ea, "F": F, "V": None if V is None else V.float()}
    if kind == "train":
        loss, g, E, F = pot.loss_grad(sysd, theta, st["e_ref"], st["f_ref"], 0.1)
        return {"loss": loss.float(), "dtheta": g, "E": E.float(), "F": F}
    if kind == "store":
        loss, g, E, F = st["store"].loss_grad(sysd, theta, st["e_ref"], st["f_ref"], 0.1)
        return {"loss": loss.float(), "dtheta": g, "E": E.float(), "F": F}
    if kind == "descriptors":
        return {"G": pot.descriptors(sysd)}
    if kind == "qeq":
        E, Ea, q, F = pot.qeq_energy_forces(sysd, theta, st["charge"])
        return {"E": E.float(), "E_atom": Ea, "q": q.float(), "F": F}
    # a stretch of dynamics from the saved state; the frame it ends with
    sysd.pos.copy_(st["pos0"])
    st["vel"].copy_(st["vel0"])
    P.panna_md_run(pot.ctx, sysd, st["vel"], theta, prec, MD["dt"], MD["temperature"], MD["friction"], case["skin"],
                   MD["mass"], st["seed"], 0, case["steps"], st["F"], False, st["E"])
    return {"pos": sysd.pos.float(), "vel": st["vel"].float(), "F": st["F"], "E": st["E"].float()}


# ------------------------------------------------------------------------------------ work

def _counts(case):
    """(atoms, configurations, neighbour entries, angular pairs) expected for the case."""
    s, n = case["structure"], _size(case)
    if s == "molecules":
        m = _molecule_sizes(n).astype(np.float64)
        nb = 0.84 * (m - 1)
        return int(m.sum()), n, float((m * nb).sum()), float((m * nb * (nb - 1) / 2).sum())
    if s == "nacl":
        N = 17 * (n - n // 2) + 16 * (n // 2)
        return N, n, 11.0 * N, 55.0 * N
    N, C, nb = {"diamond": (8 * n ** 3, 1, 24.6), "fcc": (4 * n ** 3, 1, 42), "water": (n, 1, 90.7),
                "water_bp": (n, 1, 90.7), "ragged": (0, n, 34.8), "carbon": (16 * n, n, 88.4)}[s]
    if s == "ragged":
        N = int(_ragged_sizes(n).sum())
    lattice = s in ("diamond", "fcc", "carbon")
    return N, C, float(N * nb), float(N * nb * (nb - (1 if lattice else 0)) / 2)


def work(case):
    N, C, entries, pairs = _counts(case)
    s, kind = case["structure"], case["kind"]
    S, n_rad, n_th, n_r, hidden, n_out = {
        "diamond": (1, 32, 8, 8, (256, 128, 32), 1), "water": (2, 32, 8, 8, (256, 128), 1),
        "water_bp": (2, 32, 4, 2, (256, 128), 1), "fcc": (1, 64, 16, 8, (128, 64), 1),
        "ragged": (3, 32, 8, 8, (128, 32), 1), "molecules": (4, 32, 8, 8, (128, 32), 1),
        "carbon": (1, 24, 16, 8, (64, 32), 1), "nacl": (2, 9, 3, 3, (15, 15), 3)}[s]
    D = S * n_rad + S * (S + 1) // 2 * n_th * n_r
    widths = (D,) + hidden + (n_out,)
    params = S * sum(b * a + b for a, b in zip(widths, widths[1:]))
    layer = 2.0 * sum(a * b for a, b in zip(widths, widths[1:]))
    # per pair: geometry, n_th powers, n_r Gaussians and the n_th x n_r products
    d_desc = pairs * (57 + 10 * n_th + 2 * n_th * n_r) + 6.0 * n_rad * entries
    d_adj = pairs * (111 + 16 * n_th + 4 * n_th * n_r) + 8.0 * n_rad * entries
    d_jvp = pairs * (66 + 16 * n_th + 4 * n_th * n_r) + 8.0 * n_rad * entries
    batch = N * (24 + 4) + C * (72 + 3 + 8)
    out = 12.0 * N + 4.0 * N + 8.0 * C
    if kind == "descriptors":
        return {"bytes": batch + 4.0 * N * D, "flops": d_desc}
    if kind == "train":
        return {"bytes": batch + 8.0 * params + 12.0 * N + out, "flops": d_desc + d_adj + d_jvp + 6.0 * N * layer}
    if kind == "store":
        width = 4 * -(-n_rad // 4) + S * 4 * -(-n_th * n_r // 4)
        # the stored Jacobians enter the forces and, once those are known, the gradient
        stored = entries * (12.0 * width + 24) + 4.0 * N * D
        return {"bytes": 2 * stored + 8.0 * params + 12.0 * N + out,
                "flops": 12.0 * width * entries + 6.0 * N * layer}
    once = {"bytes": batch + 4.0 * params + out + (72.0 * C if case.get("virial") else 0.0),
            "flops": d_desc + d_adj + 2.0 * N * layer}
    if kind == "md":
        return {k: v * (case["steps"] + 1) for k, v in once.items()}
    return once


# ------------------------------------------------------------------------------------ 64 bits

F64 = dict(dtype=torch.float64, device="cuda")


def _entries(system, rc, pos=None):
    """All neighbour entries (i, j, vector) with 0 < r < rc, sorted by i; every periodic image."""
    x = torch.as_tensor(system.pos, **F64) if pos is None else pos
    out = []
    for c in range(system.n_cfg):
        a, b = int(system.atom_off[c]), int(system.atom_off[c + 1])
        p, n = x[a:b], b - a
        if n == 0:
            continue
        per = bool(system.pbc[c].any())
        L = torch.as_tensor(np.diag(system.cell[c].reshape(3, 3)).copy(), **F64) if per else None
        if per and float(L.min()) > 2 * rc:
            shifts = None
        elif per:
            k = [int(math.ceil(rc / float(v))) + 1 for v in L]
            shifts = torch.cartesian_prod(*[torch.arange(-m, m + 1) for m in k]).to(**F64) * L
        else:
            shifts = torch.zeros((1, 3), **F64)
        step = max(1, int(3e7 // (n * (1 if shifts is None else len(shifts)))))
        for r0 in range(0, n, step):
            d = p[None, :] - p[r0:r0 + step, None]
            if shifts is None:
                d = d - L * torch.round(d / L)
                d = d[:, :, None]
            else:
                d = d[:, :, None] + shifts
            r2 = (d * d).sum(-1)
            hit = ((r2 < rc * rc) & (r2 > 1e-12)).nonzero()
            out.append((hit[:, 0] + (a + r0), hit[:, 1] + a, d[hit[:, 0], hit[:, 1], hit[:, 2]]))
    if not out:
        z = torch.zeros(0, dtype=torch.int64, device="cuda")
        return z, z, torch.zeros((0, 3), **F64)
    return tuple(torch.cat([o[k] for o in out]) for k in range(3))


class _Reference:
    """Descriptors, their products with vectors, networks, energies and forces in 64 bits."""

    def __init__(self, x, pos=None):
        self.x, self.desc, self.archs = x, x["desc"], x["archs"]
        system = x["system"]
        self.N, self.S, self.D = system.n_atoms, self.desc.n_species, self.desc.D
        self.species = torch.as_tensor(system.species, device="cuda").long()
        self.cfg = torch.repeat_interleave(torch.arange(system.n_cfg, device="cuda"),
                                           torch.as_tensor(np.diff(system.atom_off), device="cuda"))
        self.i, self.j, self.vec = _entries(system, self.desc.rc, pos)
        n = torch.bincount(self.i, minlength=self.N)
        self.start = torch.cumsum(n, 0) - n
        self.count = n
        self.theta = torch.as_tensor(x["theta"], device="cuda").double()

    def chunks(self):
        """Ranges of centres whose padded pair lists take a few GB."""
        d, a = self.desc, 0
        top = int(self.count.max()) if self.N else 0
        per = 8.0 * max(1, top * (top - 1) // 2) * (8 * (d.n_theta + d.n_ang_r) + 60) + 64.0 * top * d.n_rad
        step = max(1, int(12e9 / per))
        while a < self.N:
            yield a, min(self.N, a + step)
            a += step

    def rows(self, a, b):
        """Padded neighbour entries of the centres a..b-1: entry indices [n, K] and a mask."""
        K = max(1, int(self.count[a:b].max()))
        k = torch.arange(K, device="cuda")
        mask = k[None] < self.count[a:b, None]
        idx = torch.where(mask, self.start[a:b, None] + k, torch.zeros((), dtype=torch.int64, device="cuda"))
        return idx, mask

    def G(self, vec, spec, mask):
        """Descriptor rows from padded vectors [n, K, 3], neighbour species and mask [n, K]."""
        d, S = self.desc, self.S
        r = torch.sqrt((vec * vec).sum(-1))
        fc = 0.5 * (1 + torch.cos(math.pi * r / d.rc)) * mask
        rs = torch.as_tensor(d.rs_rad, **F64)
        g = torch.exp(-d.eta_rad * (r[..., None] - rs) ** 2) * fc[..., None]
        out = [(g * (spec == s)[..., None]).sum(1) for s in range(S)]
        K = r.shape[1]
        p, q = torch.triu_indices(K, K, 1, device="cuda")
        c = ((vec[:, p] * vec[:, q]).sum(-1) / (r[:, p] * r[:, q]))
        f = fc[:, p] * fc[:, q]
        if d.angular == "bp":
            lam, zeta, eta = (torch.as_tensor(v, **F64) for v in (d.bp_lambda, d.bp_zeta, d.bp_eta))
            e = vec[:, p] - vec[:, q]
            e2 = (e * e).sum(-1)
            live = mask[:, p] & mask[:, q] & (e2 < d.rc ** 2) & (e2 > 0)
            r3 = torch.sqrt(torch.where(live, e2, torch.ones((), **F64)))
            f = f * torch.where(live, 0.5 * (1 + torch.cos(math.pi * r3 / d.rc)), torch.zeros((), **F64))
            A = 2.0 ** (1 - zeta) * torch.clamp(1 + lam * c[..., None], min=0) ** zeta
            B = torch.exp(-eta * (r[:, p] ** 2 + r[:, q] ** 2 + r3 ** 2)[..., None])
        else:
            th = torch.as_tensor(d.theta_s, **F64)
            sn = torch.sqrt(torch.clamp(1 - c * c, min=0) + d.eps_theta)
            y = torch.clamp((1 + c[..., None] * torch.cos(th) + sn[..., None] * torch.sin(th)) / 2, min=0)
            A = 2.0 * y ** d.zeta
            x = (0.5 * (r[:, p] + r[:, q]))[..., None] - torch.as_tensor(d.rs_ang, **F64)
            B = torch.exp(-d.eta_ang * x * x)
        B = B * f[..., None]
        lo, hi = torch.minimum(spec[:, p], spec[:, q]), torch.maximum(spec[:, p], spec[:, q])
        for s in range(S):
            for t in range(s, S):
                m = ((lo == s) & (hi == t))[..., None]
                out.append(torch.bmm((A * m).transpose(1, 2), B).flatten(1))
        return torch.cat(out, 1)

    def padded(self, a, b):
        idx, mask = self.rows(a, b)
        if len(self.vec) == 0:
            return idx, torch.ones(idx.shape + (3,), **F64), torch.zeros_like(idx), mask
        far = torch.tensor([1.0, 0.5, 0.25], **F64)   # any vector: masked entries have weight zero
        # padding entries of one row get different directions, so that no angle is exactly 0
        far = far * (1 + torch.arange(idx.shape[1], device="cuda", dtype=torch.float64)[:, None] %
                     torch.tensor([2.0, 3.0, 5.0], **F64))
        vec = torch.where(mask[..., None], self.vec[idx], far)
        return idx, vec, self.species[self.j[idx]], mask

    def descriptors(self):
        out = torch.zeros((self.N, self.D), **F64)
        for a, b in self.chunks():
            _, vec, spec, mask = self.padded(a, b)
            out[a:b] = self.G(vec, spec, mask)
        return out

    def adjoint(self, g):
        """Per-entry gradients q = g_i . dG_i/dvec."""
        q = torch.zeros_like(self.vec)
        for a, b in self.chunks():
            idx, vec, spec, mask = self.padded(a, b)
            vec = vec.detach().requires_grad_(True)
            got, = torch.autograd.grad(self.G(vec, spec, mask), vec, g[a:b])
            q[idx[mask]] = got[mask]
        return q

    def tangent(self, ue):
        """w_i = sum over entries of dG_i/dvec . ue."""
        out = torch.zeros((self.N, self.D), **F64)
        for a, b in self.chunks():
            idx, vec, spec, mask = self.padded(a, b)
            vec = vec.detach().requires_grad_(True)
            v = torch.zeros((b - a, self.D), **F64, requires_grad=True)
            gv, = torch.autograd.grad(self.G(vec, spec, mask), vec, v, create_graph=True)
            u = torch.where(mask[..., None], ue[idx] if len(ue) else torch.zeros_like(vec), torch.zeros((), **F64))
            out[a:b], = torch.autograd.grad(gv, v, u)
        return out

    def net(self, G, theta):
        """Network outputs per atom."""
        n_out = self.archs[0].widths[-1]
        out = torch.zeros((self.N, n_out), **F64)
        off = 0
        for s, arch in enumerate(self.archs):
            rows = (self.species == s).nonzero()[:, 0]
            h = G[rows]
            for l in range(arch.n_layers):
                fi, fo = arch.widths[l], arch.widths[l + 1]
                w = theta[off:off + fi * fo].view(fo, fi)
                off += fi * fo
                h = h @ w.T + theta[off:off + fo]
                off += fo
                if arch.acts[l] == W.ACT_GAUSSIAN:
                    h = torch.exp(-h * h)
            out = out.index_copy(0, rows, h)
        return out

    def per_cfg(self, v):
        return torch.zeros(self.x["system"].n_cfg, **F64).index_add(0, self.cfg, v)

    def forces(self, q):
        return torch.zeros((self.N, 3), **F64).index_add(0, self.i, q).index_add(0, self.j, -q)

    def energy_forces(self):
        G = self.descriptors().requires_grad_(True)
        e = self.net(G, self.theta)[:, 0]
        g, = torch.autograd.grad(e.sum(), G)
        q = self.adjoint(g)
        vir = torch.zeros((self.x["system"].n_cfg, 3, 3), **F64)
        vir.index_add_(0, self.cfg[self.i], -q[:, :, None] * self.vec[:, None, :])
        return self.per_cfg(e.detach()), e.detach(), self.forces(q), vir, G.detach()

    def loss_grad(self, w_force):
        E, _, F, _, G = self.energy_forces()
        C = self.x["system"].n_cfg
        dE = E - torch.as_tensor(self.x["e_ref"], **F64)
        dF = F - torch.as_tensor(self.x["f_ref"], device="cuda").double()
        loss = (dE ** 2).sum() / C + w_force / (3 * self.N) * (dF ** 2).sum()
        u = 2 * w_force / (3 * self.N) * dF
        w = self.tangent(u[self.j] - u[self.i])
        theta = self.theta.clone().requires_grad_(True)
        G = G.requires_grad_(True)
        e = self.net(G, theta)[:, 0]
        g, = torch.autograd.grad(e.sum(), G, create_graph=True)
        # sum F . u = sum over centres of g . w, up to the sign of F = -dE/dx with dvec = dx_j - dx_i
        dtheta, = torch.autograd.grad(((2 * dE / C)[self.cfg] * e).sum() - (g * w).sum(), theta)
        return loss.reshape(1), dtheta, E, F


def _exact_qeq(x):
    ref = _Reference(x)
    system, q_tot = x["system"], torch.as_tensor(x["charge"], **F64)
    sigma, chi0, hard0 = (torch.as_tensor(x["qeq"][k], **F64) for k in ("sigma", "chi0", "hard0"))
    ke = 14.399645478425668
    C, off = system.n_cfg, np.asarray(system.atom_off)
    M = int(np.diff(off).max())
    slot = torch.arange(ref.N, device="cuda") - torch.as_tensor(off[:-1], device="cuda")[ref.cfg]
    G = ref.descriptors().requires_grad_(True)
    out = ref.net(G, ref.theta)
    pos = torch.as_tensor(system.pos, **F64).requires_grad_(True)

    def dense(v, fill):
        return torch.full((C, M) + v.shape[1:], fill, **F64).index_put((ref.cfg, slot), v)
    live = dense(torch.ones(ref.N, **F64), 0.0)
    X, s = dense(pos, 0.0), dense(sigma[ref.species], 1.0)
    eye = torch.eye(M, **F64)
    pair = live[:, :, None] * live[:, None, :] * (1 - eye)
    d2 = ((X[:, :, None] - X[:, None]) ** 2).sum(-1)
    r = torch.sqrt(torch.where(pair > 0, d2, torch.ones((), **F64)))
    K = ke * pair * torch.erf(r / torch.sqrt(2 * (s[:, :, None] ** 2 + s[:, None] ** 2))) / r
    K = K + torch.diag_embed(ke * live / (s * math.sqrt(math.pi)))
    chi, hard = dense(chi0[ref.species] + out[:, 1], 0.0), dense(hard0[ref.species] + out[:, 2], 1.0)
    with torch.no_grad():
        A = torch.zeros((C, M + 1, M + 1), **F64)
        A[:, :M, :M] = K + torch.diag_embed(hard)
        A[:, :M, M] = A[:, M, :M] = live
        q = torch.linalg.solve(A, torch.cat([-chi, q_tot[:, None]], 1))[:, :M] * live
    e = out[:, 0] + ((chi + 0.5 * hard * q + 0.5 * (K @ q[..., None])[..., 0]) * q)[ref.cfg, slot]
    g, gx = torch.autograd.grad(e.sum(), (G, pos))
    e = e.detach()
    return {"E": ref.per_cfg(e), "E_atom": e, "q": q[ref.cfg, slot], "F": ref.forces(ref.adjoint(g)) - gx}


def _philox_normals(seed, n, step):
    """Three normals for each of n atoms: Philox4x32-10 (Salmon et al., SC'11) and Box-Muller."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.zeros(n, np.uint64), np.full(n, step, np.uint64), np.zeros(n, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [(v.astype(np.float64) + 0.5) / 4294967296.0 for v in c]
    a, b = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    return np.stack([a * np.cos(2 * np.pi * u[1]), a * np.sin(2 * np.pi * u[1]), b * np.cos(2 * np.pi * u[3])], 1)


def _exact_md(x, case, seed):
    acc, kb = 9.648533212e-3 / MD["mass"][0], 8.617333262e-5
    dt, c1 = MD["dt"], math.exp(-MD["friction"] * MD["dt"])
    c2, sig = math.sqrt(1 - c1 * c1), math.sqrt(kb * MD["temperature"] * acc)
    pos, vel = torch.as_tensor(x["system"].pos, **F64), torch.as_tensor(x["vel"], **F64)
    E, _, F, _, _ = _Reference(x, pos).energy_forces()
    for t in range(case["steps"]):
        vel = vel + 0.5 * dt * acc * F
        pos = pos + 0.5 * dt * vel
        vel = c1 * vel + c2 * sig * torch.as_tensor(_philox_normals(int(seed), len(pos), t), **F64)
        pos = pos + 0.5 * dt * vel
        E, _, F, _, _ = _Reference(x, pos).energy_forces()
        vel = vel + 0.5 * dt * acc * F
    return {"pos": pos, "vel": vel, "F": F, "E": E}


def exact(case, seed):
    N, _, _, pairs = _counts(case)
    # the largest boxes would take minutes
    if pairs > 2e8 or (case["structure"] == "fcc" and N > 40000) or (case["kind"] == "md" and N > 512):
        return None
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "md":
        return _exact_md(x, case, seed)
    if kind == "qeq":
        return _exact_qeq(x)
    ref = _Reference(x)
    if kind == "descriptors":
        return {"G": ref.descriptors()}
    if kind == "infer":
        E, e, F, V, _ = ref.energy_forces()
        return {"E": E, "E_atom": e, "F": F, "V": V if case["virial"] else None}
    loss, dtheta, E, F = ref.loss_grad(0.1)
    return {"loss": loss, "dtheta": dtheta, "E": E, "F": F}
