"""Performance cases of the library's public entry points.

Each case is one call (or the short sequence of calls) that a program makes
through ``paper_1803_07491_gb300.bop``: energy, forces and virial of one
structure, the neighbour list and bond blocks of a structure, the moments
that training data is made from, one training step of the network.

Kinds:
  evaluate   Context.evaluate: structure, energy (with its SCF), forces, virial
             (torques of a non-collinear model);
  structure  Context.build, then the neighbour list and the bond blocks;
  moments    Context.build, bop_moments (FP64, 17 moments: the training data
             of the learned terminator);
  train      bop_mlp_gradient and bop_mlp_adam on one batch.

A program that runs the FP32-products mode keeps single-precision results,
so those cases hand their energies, forces and virials on in float32.  What
they are off by is measured against ``exact``: the same quantities in plain
64-bit torch, written from the formulas of the method (arXiv:1803.07491).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1803_07491_gb300 import bop
from paper_1803_07491_gb300 import inputs as I

MODELS = {"s": I.MODEL_S, "d": I.MODEL_D, "sd": I.MODEL_SD}
ELECTRONS = {"s": 0.7, "d": 6.8, "sd": 8.0}
SCF_TOL_FP32 = 3e-5  # the SCF tolerance that the benchmark takes with FP32 products

EVAL = {"kind": "evaluate", "lattice": "bcc", "model": "d", "n_mom": 9, "scf": "none", "precision": "fp32",
        "sigma": 0.05, "form": "plain"}


def listed():
    return [
        # a molecule-sized s-band cell in the default precision: what one call costs at the least
        {**EVAL, "name": "s128_fp64", "n1": 4, "n2": 4, "n3": 4, "model": "s", "precision": "fp64"},
        # a small d-band cell with local charge neutrality in the default precision (a defect or alloy cell)
        {**EVAL, "name": "d250_lcn_fp64", "n1": 5, "n2": 5, "n3": 5, "scf": "lcn", "precision": "fp64"},
        # the ordinary production call: 2,000 atoms, local charge neutrality, forces with the SCF response
        {**EVAL, "name": "d2000_lcn_fp32", "n1": 10, "n2": 10, "n3": 10, "scf": "lcn"},
        # close-packed lattice (18 neighbours), odd sizes
        {**EVAL, "name": "fcc1372_fp32", "lattice": "fcc", "n1": 7, "n2": 7, "n3": 7},
        # sd-valent blocks (6 x 6) with local charge neutrality
        {**EVAL, "name": "sd2000_lcn_fp32", "n1": 10, "n2": 10, "n3": 10, "model": "sd", "scf": "lcn"},
        # a slab with vacancies and free surfaces at 13 moments: large clusters, ragged levels
        {**EVAL, "name": "slab2000_13mom_fp64", "lattice": "slab", "n1": 8, "n2": 8, "n3": 16, "n_mom": 13,
         "precision": "fp64", "sigma": 0.08},
        # collinear magnetism: two spin channels, Stoner self-consistency
        {**EVAL, "name": "mag432_stoner_fp64", "n1": 6, "n2": 6, "n3": 6, "scf": "stoner", "precision": "fp64"},
        # non-collinear magnetism: a spin spiral at fixed magnitudes, forces and torques
        {**EVAL, "name": "nc2000_fp32", "n1": 10, "n2": 10, "n3": 10, "form": "spiral"},
        # the largest: 131,072 atoms with the learned terminator (the benchmark's default workload)
        {**EVAL, "name": "learned131k_fp32", "n1": 32, "n2": 32, "n3": 64, "form": "learned"},
        # structure only, at a size of its own: neighbour list and bond blocks of 65,536 atoms
        {"kind": "structure", "name": "structure65k", "lattice": "bcc", "n1": 32, "n2": 32, "n3": 32, "model": "d",
         "n_mom": 9, "sigma": 0.05, "precision": "fp32"},
        # training data of the learned terminator: 17 moments of a strained 2,000-atom cell in FP64
        {"kind": "moments", "name": "train_moments2000_fp64", "lattice": "bcc", "n1": 10, "n2": 10, "n3": 10,
         "model": "d", "n_mom": 17, "sigma": 0.08, "precision": "fp64"},
        # one step of the network's training at the benchmark's batch
        {"kind": "train", "name": "train_step4096", "rows": 200000, "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evaluate"] * 7 + ["structure", "moments", "train"])
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 20000, 400000), "batch": _log_int(rng, 256, 16384)}
    if kind == "structure":
        n = [_log_int(rng, 4, 40) for _ in range(3)]
        # bcc: its shells lie clear of the cutoff, so that every seed has the same number of pairs
        return {"kind": "structure", "lattice": "bcc", "n1": n[0], "n2": n[1], "n3": n[2],
                "model": rng.choice(["s", "d", "sd"]), "n_mom": rng.choice([5, 7, 9]),
                "sigma": round(rng.uniform(0.02, 0.06), 4), "precision": "fp32"}
    if kind == "moments":
        n = [rng.randint(4, 10) for _ in range(3)]
        return {"kind": "moments", "lattice": "bcc", "n1": n[0], "n2": n[1], "n3": n[2], "model": "d",
                "n_mom": rng.choice([9, 13, 17]), "sigma": round(rng.uniform(0.02, 0.12), 4), "precision": "fp64"}
    sigma = round(rng.uniform(0.03, 0.08), 4)
    form = rng.choice(["plain"] * 5 + ["learned", "spiral", "cut"])
    if form != "plain":
        n = [_log_int(rng, 4, 24 if form == "learned" else 11) for _ in range(3)]
        return {**EVAL, "n1": n[0], "n2": n[1], "n3": n[2], "sigma": sigma, "form": form}
    scf = rng.choice(["none", "none", "lcn", "lcn", "stoner"])
    model = "d" if scf == "stoner" else rng.choice(["d", "d", "d", "sd"] + (["s"] if scf == "none" else []))
    lattice = rng.choice(["bcc", "bcc", "fcc"] + (["slab"] if scf == "none" and model == "d" else []))
    fp64 = scf == "stoner" or lattice == "slab" or rng.random() < 0.35
    # the self-consistent loops of these models converge at 9 moments, not at 7
    n_mom = 9 if scf != "none" else rng.choice([7, 9, 11] if fp64 else [7, 9])
    top = (6 if scf == "stoner" else 7) if fp64 else (10 if lattice == "fcc" else 14)
    if scf == "stoner":  # near the magnetic crystal, where the plain iteration converges
        lattice, sigma = "bcc", round(0.7 * sigma, 4)
    n = [_log_int(rng, 3, top) for _ in range(3)]
    return {**EVAL, "lattice": lattice, "n1": n[0], "n2": n[1], "n3": n[2] + (4 if lattice == "slab" else 0),
            "model": model, "scf": scf, "precision": "fp64" if fp64 else "fp32", "n_mom": n_mom, "sigma": sigma}


# ------------------------------------------------------------ inputs

def _cell(case, seed):
    """Positions, cell and periodicity of a case's structure."""
    n1, n2, n3, sigma = case["n1"], case["n2"], case["n3"], case["sigma"]
    if case["lattice"] == "slab":
        return I.slab_with_vacancies(n1, n2, n3, max(1, n1 * n2 * n3 // 128), sigma, seed)
    if case["lattice"] == "fcc":
        return (*I.fcc_jittered(n1, n2, n3, sigma, seed), (1, 1, 1))
    if case["kind"] == "moments":  # a training cell: homogeneous strain, then the jitter
        rng = np.random.default_rng(seed)
        e = rng.uniform(-0.03, 0.03, size=6)
        strain = np.eye(3) + np.array([[e[0], e[5], e[4]], [e[5], e[1], e[3]], [e[4], e[3], e[2]]])
        pos, cell = I.bcc_cell(n1, n2, n3)
        pos, cell = pos @ strain.T, cell @ strain.T
        return I.jittered(pos, cell, (1, 1, 1), sigma, rng), cell, (1, 1, 1)
    return (*I.bcc_jittered(n1, n2, n3, sigma, seed), (1, 1, 1))


def _run_params(case):
    kw = {}
    scf, form = case.get("scf", "none"), case.get("form", "plain")
    if scf != "none":
        kw.update(scf=scf, **I.ANDERSON_STEP)
        if case["precision"] == "fp32":
            kw["scf_tol"] = SCF_TOL_FP32
    if scf == "stoner":
        kw.update(n_spin=2, stoner_I=0.8, m_mix=1.0)
    if form == "spiral":
        kw.update(n_spin=2, stoner_I=0.8, noncollinear=True)
    if form == "learned":
        kw.update(terminator="mlp")
    if form == "cut":
        kw.update(r_path=5.5)
    return I.RunParams(n_e=ELECTRONS[case["model"]], n_mom=case["n_mom"], **kw)


def _batch(case, seed):
    rng = np.random.default_rng(seed)
    rows = case["rows"]
    x = rng.standard_normal((rows, bop.MLP_NIN), dtype=np.float32)
    t = rng.standard_normal((rows, bop.MLP_NOUT), dtype=np.float32)
    mask = (rng.random(rows) > 0.02).astype(np.float32)
    idx = rng.permutation(rows)[:case["batch"]].astype(np.int32)
    return x, t, mask, idx


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "train":
        s["x"], s["t"], s["mask"], s["idx"] = (torch.as_tensor(a, device="cuda") for a in _batch(case, seed))
        s["net"] = bop.Network(I.mlp_init_params(seed))
        s["net"].set_norm(I.mlp_fixed_norm())
        s["grad"] = torch.empty(bop.MLP_NPARAM, dtype=torch.float32, device="cuda")
        s["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
        return s
    pos, s["cell"], s["pbc"] = _cell(case, seed)
    s["pos"] = torch.as_tensor(pos, dtype=torch.float64, device="cuda")
    net = None
    if case.get("form") == "learned":
        net = bop.Network(I.mlp_init_params(seed, 0.3))
        net.set_norm(I.mlp_fixed_norm())
    s["ctx"] = bop.Context(MODELS[case["model"]], _run_params(case), case["precision"], net=net)
    if case.get("form") == "spiral":
        s["spin_dir"] = torch.as_tensor(I.spiral_directions(pos, s["cell"][0, 0], np.pi / 3), dtype=torch.float64,
                                        device="cuda")
        s["m"] = torch.full((len(pos),), 2.0, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "train":
        bop.bop_mlp_gradient(s["net"].h, s["x"], s["t"], s["mask"], s["idx"], s["grad"], s["loss"])
        bop.bop_mlp_adam(s["net"].h, 1e-3)
        return {"grad": s["grad"], "loss": s["loss"]}
    ctx = s["ctx"]
    if case["kind"] == "structure":
        ctx.build(s["pos"], s["cell"], s["pbc"])
        row, col, img = bop.bop_get_neighbors(ctx.h)
        atoms, d, blocks = bop.bop_get_bonds(ctx.h, MODELS[case["model"]].norb)
        return {"row": row, "col": col, "img": img, "atoms": atoms, "d": d, "blocks": blocks}
    if case["kind"] == "moments":
        ctx.build(s["pos"], s["cell"], s["pbc"])
        return {"mu": bop.bop_moments(ctx.h, 1, ctx.n, MODELS[case["model"]].norb, case["n_mom"])}
    r = ctx.evaluate(s["pos"], s["cell"], s["pbc"], spin_dir=s.get("spin_dir"), m=s.get("m"))
    out = {"e_atom": r.e_atom, "forces": r.forces, "virial": r.virial}
    if r.torques is not None:
        out["torques"] = r.torques
    if case["precision"] == "fp32":
        out = {k: v.float() for k, v in out.items()}
    return out


# ------------------------------------------------------------ work

def _atoms(case):
    return case["n1"] * case["n2"] * case["n3"] * (4 if case["lattice"] == "fcc" else 2)


def _products(lattice, K):
    """Block products of one moments pass per atom of the perfect crystal:
    neighbours x the sites within 0 .. K-1 hops."""
    half = {"fcc": ((1, 1, 0), (2, 0, 0))}.get(lattice, ((1, 1, 1), (2, 0, 0)))
    steps = set()
    for v in half:
        for perm in {(v[i], v[j], v[3 - i - j]) for i in range(3) for j in range(3) if i != j}:
            for sx in (1, -1):
                for sy in (1, -1):
                    for sz in (1, -1):
                        steps.add((sx * perm[0], sy * perm[1], sz * perm[2]))
    sites, total = {(0, 0, 0)}, 0
    for _ in range(K):
        total += len(sites) * len(steps)
        sites |= {(x + u, y + v, z + w) for x, y, z in sites for u, v, w in steps}
    return total, len(steps)


def work(case):
    if case["kind"] == "train":
        macs = bop.MLP_NPARAM  # per row: one forward, and the reverse for inputs and weights
        return {"bytes": case["batch"] * 4.0 * (bop.MLP_NIN + bop.MLP_NOUT + 2) + 4.0 * 7 * bop.MLP_NPARAM,
                "flops": 6.0 * macs * case["batch"]}
    n = _atoms(case)
    norb = MODELS[case["model"]].norb
    prod, deg = _products(case["lattice"], (case["n_mom"] - 1) // 2)
    pair = norb * (norb + 1) // 2
    if case["kind"] == "structure":
        return {"bytes": n * (24.0 + 8 + deg * 7 + deg / 2 * (8 + 24 + 8 * pair)), "flops": n * deg * 100.0}
    spins = 2 if case.get("scf") == "stoner" or case.get("form") == "spiral" else 1
    columns = norb * (8 if case.get("form") == "spiral" else spins)
    one = 2.0 * prod * norb * norb * columns * n
    if case["kind"] == "moments":
        return {"bytes": n * (24.0 + 8.0 * norb * case["n_mom"]), "flops": one}
    # one moments pass, one reverse sweep with the bond cotangents, and the
    # sums over the expansion (forward recurrence, N and U, their reverse)
    scalar = n * norb * spins * 201.0 * (10.0 * case["n_mom"] + 40.0)
    out = 4.0 if case["precision"] == "fp32" else 8.0
    return {"bytes": n * (24.0 + out * (4 + (3 if case.get("form") == "spiral" else 0))), "flops": 3.0 * one + scalar}


# ------------------------------------------------------------ the same in 64 bits

_F64 = torch.float64
_MAX_ROWS, _MAX_STARTS = 90000, 12500  # orbitals of the (replicated) cell, starting orbitals


def _edges(pos, cell, pbc, rc, dev):
    """All directed pairs (i, j, image) with 0 < |r_j + S cell - r_i| < rc."""
    n = len(pos)
    p = torch.as_tensor(pos, dtype=_F64, device=dev)
    c = torch.as_tensor(np.asarray(cell), dtype=_F64, device=dev)
    width = 1.0 / np.linalg.norm(np.linalg.inv(np.asarray(cell)), axis=0)
    reach = [int(math.ceil(rc / width[a])) if pbc[a] else 0 for a in range(3)]
    ii, jj, ss = [], [], []
    for sx in range(-reach[0], reach[0] + 1):
        for sy in range(-reach[1], reach[1] + 1):
            for sz in range(-reach[2], reach[2] + 1):
                shift = torch.tensor([sx, sy, sz], dtype=_F64, device=dev) @ c
                for i0 in range(0, n, 2048):
                    d2 = torch.zeros((min(2048, n - i0), n), dtype=_F64, device=dev)
                    for a in range(3):
                        d2 += (p[None, :, a] + shift[a] - p[i0:i0 + 2048, None, a]) ** 2
                    hit = d2 < rc * rc
                    if sx == sy == sz == 0:
                        hit &= d2 > 0
                    i, j = torch.nonzero(hit, as_tuple=True)
                    ii.append(i + i0)
                    jj.append(j)
                    ss.append(torch.tensor([sx, sy, sz], device=dev).repeat(len(i), 1))
    return torch.cat(ii), torch.cat(jj), torch.cat(ss), p, c


def _blocks(m, d):
    """Two-centre blocks [E, norb, norb] of the bond vectors d [E, 3]."""
    r = d.norm(dim=1)
    taper = torch.where(r < m.rc - m.dc, torch.ones_like(r),
                        0.5 * (torch.cos(math.pi * (r - (m.rc - m.dc)) / m.dc) + 1.0))
    radial = torch.exp(-m.lam * (r - m.r0)) * taper
    if m.norb == 1:
        return (m.b0[0] * radial)[:, None, None]
    # the d orbitals 3z^2-r^2, zx, yz, x^2-y^2, xy as symmetric traceless
    # tensors Q_a; the bond direction u splits them into sigma, pi, delta
    q = math.sqrt(0.5)
    basis = torch.zeros((5, 3, 3), dtype=d.dtype, device=d.device)
    basis[0] = torch.diag(torch.tensor([-1.0, -1.0, 2.0], dtype=d.dtype)).to(d.device) / math.sqrt(6.0)
    basis[1, 0, 2] = basis[1, 2, 0] = q
    basis[2, 1, 2] = basis[2, 2, 1] = q
    basis[3, 0, 0], basis[3, 1, 1] = q, -q
    basis[4, 0, 1] = basis[4, 1, 0] = q
    u = d / r[:, None]
    qu = torch.einsum("aij,ej->eai", basis, u)       # Q_a u
    sg = torch.einsum("eai,ei->ea", qu, u) * math.sqrt(1.5)   # sigma component (m = 0)
    # sum over the two pi components: 2 (Q_a u . Q_b u - (u Q_a u)(u Q_b u))
    pi2 = 2.0 * (qu @ qu.transpose(1, 2) - (2.0 / 3.0) * sg[:, :, None] * sg[:, None, :])
    sg2 = sg[:, :, None] * sg[:, None, :]
    dl2 = torch.eye(5, dtype=d.dtype, device=d.device) - sg2 - pi2
    dd = (m.b0[0] * sg2 + m.b0[1] * pi2 + m.b0[2] * dl2) * radial[:, None, None]
    if m.norb == 5:
        return dd
    top = torch.cat([(m.b0[3] * radial)[:, None, None], (m.b0[4] * radial[:, None] * sg)[:, None, :]], 2)
    return torch.cat([top, torch.cat([(m.b0[4] * radial[:, None] * sg)[:, :, None], dd], 2)], 1)


class _Lattice:
    """H of a structure as blocks padded to the largest degree, on enough
    replicas of the cell that no path of 2K hops closes around it."""

    def __init__(self, case, seed):
        pos, cell, pbc = _cell(case, seed)
        self.m = MODELS[case["model"]]
        self.K = (case["n_mom"] - 1) // 2
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.n, self.norb = len(pos), self.m.norb
        i, j, S, p, c = _edges(pos, cell, pbc, self.m.rc, self.dev)
        self.i, self.j = i, j
        self.d = p[j] + S.to(_F64) @ c - p[i]
        inv = torch.linalg.inv(c)
        span = (self.d @ inv).abs().max(0).values * 2 * self.K  # in cells along each axis
        self.R = [int(math.floor(float(span[a]))) + 1 if pbc[a] else 1 for a in range(3)]
        self.reps = self.R[0] * self.R[1] * self.R[2]
        deg = torch.bincount(i, minlength=self.n)
        self.D = int(deg.max())
        order = torch.argsort(i, stable=True)
        slot = torch.empty_like(i)
        start = torch.cumsum(deg, 0) - deg
        slot[order] = torch.arange(len(i), device=self.dev) - start[i[order]]
        self.flat = i * self.D + slot
        g = torch.stack(torch.meshgrid(*[torch.arange(r, device=self.dev) for r in self.R], indexing="ij"),
                        -1).reshape(-1, 3)
        R = torch.tensor(self.R, device=self.dev)
        to = (g[:, None, :] + S[None]) % R
        rep = (to[..., 0] * self.R[1] + to[..., 1]) * self.R[2] + to[..., 2]
        idx = torch.zeros((self.reps, self.n * self.D), dtype=torch.int64, device=self.dev)
        idx[:, self.flat] = rep * self.n + j[None]
        self.idx = idx.reshape(self.reps * self.n, self.D)

    def fits(self):
        return self.reps * self.n * self.norb <= _MAX_ROWS and self.n * self.norb <= _MAX_STARTS

    def pad(self, B):
        Bp = torch.zeros((self.n * self.D, self.norb, self.norb), dtype=_F64, device=self.dev)
        Bp = Bp.index_put((self.flat,), B).reshape(self.n, self.D, self.norb, self.norb)
        return Bp.permute(0, 2, 1, 3).reshape(self.n, self.norb, self.D * self.norb)

    def chunk(self, Bp, onsite, lo, hi):
        """Moments [hi-lo, norb, 2K+1] of the atoms lo .. hi-1 of the first replica."""
        cols = (hi - lo) * self.norb
        x = torch.zeros((self.reps * self.n, self.norb, cols), dtype=_F64, device=self.dev)
        q = torch.arange(cols, device=self.dev)
        x[lo + q // self.norb, q % self.norb, q] = 1.0
        A, E = Bp.repeat(self.reps, 1, 1), onsite.repeat(self.reps, 1)
        mu = [torch.ones(cols, dtype=_F64, device=self.dev)]
        for _ in range(self.K):
            y = E[:, :, None] * x + torch.bmm(A, x[self.idx].reshape(len(A), self.D * self.norb, cols))
            mu += [(x * y).sum((0, 1)), (y * y).sum((0, 1))]
            x = y
        return torch.stack(mu, 1).reshape(hi - lo, self.norb, 2 * self.K + 1)

    def chunks(self):
        per = max(1, int(2.0e9 / (8.0 * self.reps * self.n * self.D * self.norb * self.norb)))
        return [(a, min(self.n, a + per)) for a in range(0, self.n, per)]

    def moments(self, Bp, onsite):
        with torch.no_grad():
            return torch.cat([self.chunk(Bp, onsite, a, b) for a, b in self.chunks()])

    def reverse(self, Bp, onsite, w, blocks=False):
        """Cotangents of sum w mu: of the onsite levels, and of the padded blocks when asked for."""
        Bp = Bp.detach().requires_grad_(blocks)
        e = onsite.detach().requires_grad_(True)
        ge = torch.zeros_like(e)
        gb = torch.zeros_like(Bp)
        for a, b in self.chunks():
            v = (self.chunk(Bp, e, a, b) * w[a:b]).sum()
            g = torch.autograd.grad(v, [e, Bp] if blocks else [e])
            ge += g[0]
            if blocks:
                gb += g[1]
        return ge, gb


def _chain(mu):
    """Recursion coefficients a_0 .. a_{K-1}, b_1 .. b_K of moments [M, 2K+1]."""
    K = (mu.shape[1] - 1) // 2
    zero = torch.zeros_like(mu[:, 0])
    prev, cur = [zero] * (K + 2), [torch.ones_like(zero)] + [zero] * (K + 1)
    a, b = [], [zero]
    for n in range(K):
        an = sum(cur[p] * cur[q] * mu[:, p + q + 1] for p in range(n + 1) for q in range(n + 1))
        nxt = [(cur[p - 1] if p else zero) - an * cur[p] - b[n] * prev[p] for p in range(n + 2)]
        bn = torch.sqrt(sum(nxt[p] * nxt[q] * mu[:, p + q] for p in range(n + 2) for q in range(n + 2)))
        a.append(an)
        b.append(bn)
        prev, cur = cur, [v / bn for v in nxt] + [zero] * (K - n)
    return a, b


def _expand(mu, n_exp):
    """Damped expansion coefficients [M, n_exp+1], band centre and half-width / 2."""
    a, b = _chain(mu)
    K = len(a)
    top = torch.stack([a[k] + b[k] + b[k + 1] for k in range(K)]).max(0).values
    bot = torch.stack([a[k] - b[k] - b[k + 1] for k in range(K)]).min(0).values
    A, B = 0.5 * (top + bot), 0.25 * (top - bot)
    # sum_m sigma_m t^m = D_1(t) / D_0(t) for the terminated chain
    hi = [torch.ones_like(A)]
    lo = [torch.ones_like(A)]
    for k in range(K - 1, -1, -1):
        a2, bb = (a[k] - A) / B, (b[k + 1] / B) ** 2
        new = []
        for q in range(max(len(lo) + 2, len(hi) + 2)):
            v = torch.zeros_like(A)
            if q < len(lo):
                v = v + lo[q]
            if 1 <= q <= len(lo):
                v = v - a2 * lo[q - 1]
            if 2 <= q < len(lo) + 2:
                v = v + lo[q - 2]
            if 2 <= q < len(hi) + 2:
                v = v - bb * hi[q - 2]
            new.append(v)
        hi, lo = lo, new
    sig = []
    for q in range(n_exp + 1):
        v = hi[q] if q < len(hi) else torch.zeros_like(A)
        for p in range(1, min(q, len(lo) - 1) + 1):
            v = v - lo[p] * sig[q - p]
        sig.append(v)
    N = n_exp
    k = torch.arange(1, N + 2, dtype=_F64, device=mu.device)
    x = math.pi / (N + 1)
    g = ((N - k + 1) * torch.cos(k * x) + torch.sin(k * x) / math.tan(x)) / (N + 1)
    return torch.stack(sig, 1) * (g / g[0])[None], A, B


def _count(gs, A, B, E, ef):
    """Electron count and bond energy of every orbital at the Fermi level ef."""
    n = gs.shape[1]
    phi = torch.acos(((ef - A) / (2.0 * B)).clamp(-1.0, 1.0))[:, None]
    k = torch.arange(1, n + 2, dtype=_F64, device=gs.device)[None]
    s = torch.cat([phi - math.pi, torch.sin(k * phi) / k], 1)   # s_0 = phi - pi, s_k = sin(k phi) / k
    chi = torch.cat([torch.zeros_like(phi), (s[:, 2:] - s[:, :-2]) / math.pi], 1)  # chi_0 .. chi_n
    chi2 = (torch.sin((n + 2) * phi) / (n + 2) - torch.sin(n * phi) / n) / math.pi
    chi = torch.cat([chi, chi2], 1)                              # chi_0 .. chi_{n+1}
    N = (gs * chi[:, 1:n + 1]).sum(1)
    P = (gs * (chi[:, 2:n + 2] + chi[:, 0:n])).sum(1)
    return N, B * P - (E - A) * N


def _fermi(gs, A, B, target):
    lo, hi = float((A - 2 * B).min()) - 1e-3, float((A + 2 * B).max()) + 1e-3
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 2.0 * float(_count(gs, A, B, A, mid)[0].sum()) < target else (lo, mid)
    return 0.5 * (lo + hi)


def _scalar(mu, E, target, n_exp, ef=None):
    """Counts and energies with what their derivatives need, at fixed ef."""
    M = mu.reshape(-1, mu.shape[-1]).detach().requires_grad_(True)
    gs, A, B = _expand(M, n_exp)
    if ef is None:
        ef = _fermi(gs.detach(), A.detach(), B.detach(), target)
    level = torch.tensor(ef, dtype=_F64, device=M.device, requires_grad=True)
    N, U = _count(gs, A, B, E.reshape(-1), level)
    return M, N, U, level


def _neutral(L, Bp, E0, target, n_e, n_exp):
    """Per-atom onsite shifts with N_i = n_e (Anderson mixing of the residual over the local DOS)."""
    shift = torch.zeros(L.n, dtype=_F64, device=L.dev)
    xs, fs = [], []
    for _ in range(60):
        E = E0 + shift[:, None]
        mu = L.moments(Bp, E)
        with torch.no_grad():
            gs, A, B = _expand(mu.reshape(-1, mu.shape[-1]), n_exp)
            ef = _fermi(gs, A, B, target)
            N = 2.0 * _count(gs, A, B, A, ef)[0].reshape(L.n, -1).sum(1)
            h = 1e-4
            dos = 2.0 * (_count(gs, A, B, A, ef + h)[0] - _count(gs, A, B, A, ef - h)[0]).reshape(L.n, -1).sum(1)
            dos = (dos / (2 * h)).clamp(min=0.1)
        res = N - n_e
        if float(res.abs().max()) < 1e-11:
            break
        f = res / dos
        xs, fs = (xs + [shift])[-9:], (fs + [f - f.mean()])[-9:]
        x, g = xs[-1], fs[-1]
        if len(xs) > 1:
            dF = torch.stack([g - q for q in fs[:-1]], 1)
            dX = torch.stack([x - q for q in xs[:-1]], 1)
            gamma = torch.linalg.lstsq(dF, g[:, None]).solution[:, 0]
            x, g = x - dX @ gamma, g - dF @ gamma
        shift = x + g
    return shift, E0 + shift[:, None], mu, ef, dos


def _gmres(apply, rhs, scale, rtol=1e-9, most=60):
    """x with apply(x) = rhs, right-preconditioned by scale."""
    beta = float(rhs.norm())
    V, H = [rhs / beta], np.zeros((most + 1, most))
    for k in range(most):
        w = apply(scale * V[k])
        for _ in range(2):
            for q in range(k + 1):
                h = float(V[q] @ w)
                H[q, k] += h
                w = w - h * V[q]
        H[k + 1, k] = float(w.norm())
        V.append(w / H[k + 1, k])
        e = np.zeros(k + 2)
        e[0] = beta
        y, *_ = np.linalg.lstsq(H[:k + 2, :k + 1], e, rcond=None)
        if np.linalg.norm(e - H[:k + 2, :k + 1] @ y) < rtol * beta:
            break
    return scale * sum(float(c) * v for c, v in zip(y, V))


def _exact_energy(case, seed):
    L = _Lattice(case, seed)
    if not L.fits():
        return None
    rp = _run_params(case)
    B = _blocks(L.m, L.d)
    Bp = L.pad(B)
    E0 = torch.full((L.n, L.norb), L.m.onsite0, dtype=_F64, device=L.dev)
    if L.norb == 6:
        E0[:, 0] = L.m.onsite_s
    target = rp.n_e * L.n
    if case["scf"] == "lcn":
        _, E, mu, ef, dos = _neutral(L, Bp, E0, target, rp.n_e, rp.n_exp)
        M, N, U, level = _scalar(mu, E, target, rp.n_exp, ef)
        wU = 2.0 * torch.autograd.grad(U.sum(), M, retain_graph=True)[0].reshape(L.n, L.norb, -1)
        wN = 2.0 * torch.autograd.grad(N.sum(), M, retain_graph=True)[0].reshape(L.n, L.norb, -1)
        N, U = N.detach(), U.detach()
        rhs = (L.reverse(Bp, E, wU)[0] - 2.0 * N.reshape(L.n, -1)).sum(1)
        y = _gmres(lambda v: L.reverse(Bp, E, wN * v[:, None, None])[0].sum(1), rhs, 1.0 / dos)
        w = wU - y[:, None, None] * wN
    else:
        mu = L.moments(Bp, E0)
        E = E0
        M, N, U, level = _scalar(mu, E, target, rp.n_exp)
        wU, uf = torch.autograd.grad(U.sum(), [M, level], retain_graph=True)
        wN, nf = torch.autograd.grad(N.sum(), [M, level])
        w = 2.0 * (wU - (uf / nf) * wN).reshape(L.n, L.norb, -1)
        U = U.detach()
    gb = L.reverse(Bp, E, w, blocks=True)[1]
    d = L.d.detach().requires_grad_(True)
    g = torch.autograd.grad((L.pad(_blocks(L.m, d)) * gb).sum(), d)[0]  # of every directed pair
    F = torch.zeros((L.n, 3), dtype=_F64, device=L.dev)
    F.index_add_(0, L.i, g)
    F.index_add_(0, L.j, -g)
    return {"e_atom": 2.0 * U.reshape(L.n, L.norb).sum(1), "forces": F, "virial": g.T @ L.d}


def _exact_structure(case, seed):
    """Bond vectors and unique block elements in the order of the bond list:
    by the lower atom (a self bond: the positive image), then as the rows of
    the neighbour list."""
    pos, cell, pbc = _cell(case, seed)
    if len(pos) > 20000 or min(case["n1"], case["n2"], case["n3"]) < 3:
        return None
    m = MODELS[case["model"]]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    i, j, S, p, c = _edges(pos, cell, pbc, m.rc, dev)
    keep = i < j
    i, j, S = i[keep], j[keep], S[keep]
    key = (((i * len(pos) + j) * 64 + (S[:, 0] + 32)) * 64 + (S[:, 1] + 32)) * 64 + (S[:, 2] + 32)
    order = torch.argsort(key)
    i, j, S = i[order], j[order], S[order]
    d = p[j] + S.to(_F64) @ c - p[i]
    r, q = np.triu_indices(m.norb)
    return {"row": None, "col": None, "img": None, "atoms": None, "d": d, "blocks": _blocks(m, d)[:, r, q]}


def _exact_train(case, seed):
    x, t, mask, idx = (torch.as_tensor(a) for a in _batch(case, seed))
    norm = torch.as_tensor(I.mlp_fixed_norm())
    nin, nout = bop.MLP_NIN, bop.MLP_NOUT
    row = idx.long()
    xs = (x[row].double() - norm[:nin]) / norm[nin:2 * nin]
    ts = (t[row].double() - norm[4 * nin:4 * nin + nout]) / norm[4 * nin + nout:]
    p = torch.as_tensor(I.mlp_init_params(seed), dtype=_F64).requires_grad_(True)
    parts, at = [], 0
    for shape in I.MLP_SHAPES:
        size = int(np.prod(shape))
        parts.append(p[at:at + size].reshape(shape))
        at += size
    h = torch.nn.functional.gelu(xs @ parts[0].T + parts[1])
    h = torch.nn.functional.gelu(h @ parts[2].T + parts[3])
    r = (h @ parts[4].T + parts[5] - ts) * mask[row].double()[:, None]
    loss = (r * r).sum() / (nout * mask[row].double().sum().clamp(min=1.0))
    return {"grad": torch.autograd.grad(loss, p)[0], "loss": loss.detach().reshape(1)}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "structure":
        return _exact_structure(case, seed)
    if _atoms(case) > 3000:
        return None
    if case["kind"] == "moments":
        L = _Lattice(case, seed)
        if not L.fits():
            return None
        E = torch.full((L.n, L.norb), L.m.onsite0, dtype=_F64, device=L.dev)
        return {"mu": L.moments(L.pad(_blocks(L.m, L.d)), E)[None]}
    # learned, magnetic and path-cut forms have no plain 64-bit form here
    if case["form"] != "plain" or case["scf"] == "stoner":
        return None
    return _exact_energy(case, seed)
