"""The work that users of this library have it do, as measurable cases.

Each case is one call (or one short sequence of calls) of the public Python binding on an
atom-centred grid of a random molecule: what a quantum-chemistry code does with the library in a
self-consistent-field iteration, a response iteration, a nuclear-derivative step or a sweep over
many small molecules.  Grids, densities and trial densities follow the recipes of
paper_2208_14639_gb300.synth (Becke partition, three s-Gaussians per atom, nuclear-displacement
trials, an uncontracted s/p basis), evaluated with torch on the GPU.

listed() names the cases, draw() samples the same ranges, prepare() builds what a program has in
hand before the call, run() makes the call, work() counts what it cannot do without, and exact()
evaluates the printed formulas in plain FP64 torch, without the library.
"""
import math

import numpy as np
import torch

from paper_2208_14639_gb300 import synth, vv10

DEV = torch.device("cuda", 0)
F64 = dict(dtype=torch.float64, device=DEV)
B_VV, C_VV, RHO_CUT = 6.0, 0.01, 1e-10
PREC = {"fp64": vv10.VV10_FP64, "tf32x3": vv10.VV10_MIXED_TF32X3, "f16x3": vv10.VV10_MIXED_F16X3,
        "fp64tc": vv10.VV10_FP64_TC}
KEPT = 0.77  # share of a grid's points above the density cutoff, near enough for counting work


def listed():
    case = lambda name, call, mol, atoms, n_rad, n_ang, prec, trials=0: dict(
        name=name, call=call, mol=mol, atoms=atoms, n_rad=n_rad, n_ang=n_ang, prec=prec, trials=trials)
    return [
        # One SCF iteration: new density in, energy and potential out.  936 points in the default
        # precision is the smallest call (latency); 9,900 and 174,600 points are the water and
        # water-hexamer grids in mixed precision; 100,080 points the 24-atom cluster in FP64.
        case("scf_water_936_fp64", "scf", "water", 3, 12, 26, "fp64"),
        case("scf_water_9900_mixed", "scf", "water", 3, 30, 110, "tf32x3"),
        case("scf_hexamer_174600_mixed", "scf", "waters", 18, 50, 194, "tf32x3"),
        case("scf_cluster_100080_fp64", "scf", "chon", 24, 30, 139, "fp64"),
        # The whole derivative step of a large molecule (energy, potential, response to 180
        # nuclear-displacement trials, point gradient) in split FP16, on a coarse grid of a
        # 60-atom molecule.
        case("step_chon60_105600_f16", "step", "chon", 60, 40, 44, "f16x3", 180),
        # One iteration of a response solver: the contraction with the trials, point set and
        # energy sums kept.  Split TF32 on the hexamer; the FP64 default on four atoms; the FP64
        # tensor-core option on twelve.
        case("response_hexamer_174600_tf32", "response", "waters", 18, 50, 194, "tf32x3", 54),
        case("response_chon4_26400_fp64", "response", "chon", 4, 60, 110, "fp64", 12),
        case("response_chon12_52800_fp64tc", "response", "chon", 12, 40, 110, "fp64tc", 36),
        # Nuclear-derivative sums: grid-position terms with the atom-resolved sums and the
        # grid-grid Hessian blocks; the weight-derivative sums along 3 N_atom directions.
        case("coords_hexamer_87300_mixed", "coords", "waters", 18, 50, 97, "tf32x3"),
        case("weights_chon12_52800_mixed", "weights", "chon", 12, 40, 110, "tf32x3", 36),
        # AO-side assembly: the Fock matrix and the contracted orbital Hessian of 54 trials.
        case("ao_hexamer_174600", "ao", "waters", 18, 50, 194, "fp64", 54),
        # A sweep over small molecules of 3 to 14 atoms (each with 3 N_atom trials) in one batch.
        case("batch_12_molecules_mixed", "batch", "mixture", 12, 30, 110, "tf32x3"),
    ]


# What one draw may ask for: call -> (precisions, most points, trial range).  The most points are
# those of the largest listed case of that call and precision.
_RANGE = {
    "scf": {"fp64": (600, 100_000), "tf32x3": (600, 174_600), "f16x3": (600, 174_600)},
    "step": {"f16x3": (8_000, 105_600), "tf32x3": (8_000, 105_600)},
    "response": {"tf32x3": (8_000, 174_600), "f16x3": (8_000, 174_600), "fp64": (3_000, 26_400),
                 "fp64tc": (6_000, 52_800)},
    "coords": {"tf32x3": (6_000, 87_300), "fp64": (2_000, 12_000)},
    "weights": {"tf32x3": (6_000, 52_800), "fp64": (2_000, 12_000)},
    "ao": {"fp64": (6_000, 174_600)},
    "batch": {"tf32x3": (2_000, 5_000), "f16x3": (2_000, 5_000)},
}
_MOST_ATOMS = {"scf": 30, "step": 60, "response": 18, "coords": 18, "weights": 12, "ao": 18}
_MOST_TRIALS = {"step": {"f16x3": 180, "tf32x3": 180},
                "response": {"tf32x3": 54, "f16x3": 54, "fp64": 12, "fp64tc": 36},
                "weights": {"tf32x3": 36, "fp64": 12}, "ao": {"fp64": 54}}


def draw(rng):
    call = rng.choice(["scf", "scf", "step", "response", "response", "coords", "weights", "ao", "batch"])
    prec = rng.choice(sorted(_RANGE[call]))
    lo, hi = _RANGE[call][prec]
    points = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if call == "batch":  # points per molecule
        atoms, mol = rng.randint(2, 12), "mixture"
        n_ang = rng.randint(26, 110)
        n_rad = max(8, int(points / (3 * n_ang)))
        return dict(call=call, mol=mol, atoms=atoms, n_rad=min(n_rad, 30), n_ang=n_ang, prec=prec, trials=0)
    least = 2 if call in ("coords", "weights", "step") else 1
    atoms = rng.randint(least, max(least, min(_MOST_ATOMS[call], int(points / 1200))))
    mol = "waters" if atoms % 3 == 0 and rng.random() < 0.5 else "chon"
    if mol == "chon" and call == "ao":  # at most the hexamer's 78 basis functions
        atoms = min(atoms, 7)
    n_ang = rng.randint(26, 194)
    n_rad = max(10, min(90, int(points / (atoms * n_ang))))
    n_ang = max(14, min(302, int(points / (atoms * n_rad))))
    most = _MOST_TRIALS.get(call, {}).get(prec, 0)
    trials = min(rng.randint(1, max(1, most)), 3 * atoms) if most else 0
    return dict(call=call, mol=mol, atoms=atoms, n_rad=n_rad, n_ang=n_ang, prec=prec, trials=trials)


# ------------------------------------------------------------------ inputs

def _molecule(kind, atoms, rng):
    """A molecule whose geometry depends on the seed alone."""
    if kind == "water":
        w = synth.water()
        return synth.Molecule(list(w.symbols), w.coords * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, (3, 1))))
    if kind == "waters":
        if atoms == 3:
            return _molecule("water", 3, rng)
        return synth.water_cluster(rng, atoms // 3)
    mol = synth.random_chon(rng, atoms)  # the elements go with the size, the geometry with the seed
    return synth.Molecule(synth.random_chon(np.random.default_rng(atoms), atoms).symbols, mol.coords)


def _becke(points, owner, atoms):
    """Becke cell weight of each point's owner over the owner and its 8 nearest other atoms."""
    d = torch.cdist(points, atoms, compute_mode="donot_use_mm_for_euclid_dist")
    k = min(9, atoms.shape[0])
    first = d.clone()
    first.scatter_(1, owner[:, None], -1.0)
    idx = first.topk(k, dim=1, largest=False).indices             # the owner comes first
    dm = d.gather(1, idx)
    rab = torch.cdist(atoms, atoms, compute_mode="donot_use_mm_for_euclid_dist")
    rab = rab[idx[:, :, None], idx[:, None, :]]
    eye = torch.eye(k, dtype=torch.bool, device=points.device)
    mu = torch.where(eye, 0.0, (dm[:, :, None] - dm[:, None, :]) / torch.where(eye, 1.0, rab)).clamp(-1.0, 1.0)
    for _ in range(3):
        mu = 1.5 * mu - 0.5 * mu ** 3
    cell = torch.where(eye, 1.0, 0.5 * (1.0 - mu)).prod(2)
    return cell[:, 0] / cell.sum(1)


def _grid(mol, n_rad, n_ang, shift=None):
    """(points, weights, owner) of the atom-centred grid; `shift` moves atom shift[0] along
    shift[1] by shift[2] with its points."""
    coords = mol.coords.copy()
    if shift is not None:
        coords[shift[0], shift[1]] += shift[2]
    u, wa = synth.fibonacci_sphere(n_ang)
    rad = [synth.radial_grid(n_rad, synth.RADIAL_SCALE[s]) for s in mol.symbols]
    r = torch.tensor(np.stack([x[0] for x in rad]), **F64)
    wr = torch.tensor(np.stack([x[1] for x in rad]), **F64)
    u, wa, at = (torch.tensor(x, **F64) for x in (u, wa, coords))
    pts = (r[:, :, None, None] * u + at[:, None, None, :]).reshape(-1, 3)
    own = torch.arange(mol.n_atom, device=DEV).repeat_interleave(n_rad * n_ang)
    w = (wr[:, :, None] * wa).reshape(-1)
    frac = torch.cat([_becke(p, o, at) for p, o in zip(pts.split(65536), own.split(65536))])
    return pts.contiguous(), w * frac, own


def _density(mol, pts):
    rho, grad = torch.zeros(pts.shape[0], **F64), torch.zeros_like(pts)
    for z, c in zip(mol.charges, mol.coords):
        d = pts - torch.tensor(c, **F64)
        r2 = (d * d).sum(1)
        for a in synth.GAUSS_EXPONENTS:
            e = float(z) / 3.0 * (a / math.pi) ** 1.5 * torch.exp(-a * r2)
            rho += e
            grad -= (2.0 * a * e)[:, None] * d
    return rho, grad


def _system(kind, atoms, n_rad, n_ang, rng):
    mol = _molecule(kind, atoms, rng)
    xyz, w, own = _grid(mol, n_rad, n_ang)
    rho, grad = _density(mol, xyz)
    return dict(molecule=mol, xyz=xyz, w=w, rho=rho, grad=grad, own=own.to(torch.int32), atoms=mol.n_atom)


def _trials(g, P):
    """The first P nuclear-displacement trial densities."""
    rt, gt = synth.trial_densities_torch(g["molecule"], g["xyz"], atoms=range(-(-P // 3)))
    return rt[:P].contiguous(), gt[:P].contiguous()


def _weight_directions(g, P, n_rad, n_ang, h=1e-4):
    """Central differences of the Becke weights along the first P nuclear displacements."""
    out = torch.empty(P, g["w"].shape[0], **F64)
    for t in range(P):
        lo, hi = (_grid(g["molecule"], n_rad, n_ang, (t // 3, t % 3, s * h))[1] for s in (-1.0, 1.0))
        out[t] = (hi - lo) / (2.0 * h)
    return out


def _basis(g):
    """Values and gradients of the s/p basis on the grid."""
    bs = synth.ao_basis(g["molecule"])
    phi = torch.empty(g["xyz"].shape[0], bs.nbf, **F64)
    dphi = torch.empty(g["xyz"].shape[0], bs.nbf, 3, **F64)
    for m in range(bs.nbf):
        d = g["xyz"] - torch.tensor(bs.centers[m], **F64)
        e = float(bs.norm[m]) * torch.exp(-float(bs.alpha[m]) * (d * d).sum(1))
        c = int(bs.comp[m])
        phi[:, m] = e if c < 0 else e * d[:, c]
        dphi[:, m] = -2.0 * float(bs.alpha[m]) * d * phi[:, m, None]
        if c >= 0:
            dphi[:, m, c] += e
    return phi, dphi


def _inputs(case, seed):
    """Everything of a case that does not come from the library."""
    rng = np.random.default_rng(20220830 + int(seed))
    call, size = case["call"], (case["n_rad"], case["n_ang"])
    if call == "batch":
        mols = [_system("chon", 3 + 5 * k % 12, *size, rng) for k in range(case["atoms"])]
        tr = [_trials(m, 3 * m["atoms"]) for m in mols]
        return dict(mols=mols, trials=tr)
    g = _system(case["mol"], case["atoms"], *size, rng)
    if call in ("step", "response"):
        g["rt"], g["gt"] = _trials(g, case["trials"])
    if call == "weights":
        g["wt"] = _weight_directions(g, case["trials"], *size)
    if call == "ao":
        # potential and response of a local functional of the right size, per point
        g["rt"], g["gt"] = _trials(g, case["trials"])
        g["phi"], g["dphi"] = _basis(g)
        keep = (g["rho"] >= RHO_CUT).to(torch.float64)
        third = g["rho"].clamp_min(RHO_CUT) ** (1.0 / 3.0)
        g["vrho"] = keep * (0.005 - 0.04 * third)
        g["vgamma"] = keep * 1e-3 / (0.1 + third ** 4)
        g["frt"] = keep * (-0.04 / 3.0) / third ** 2 * g["rt"]
        g["fgt"] = keep * (-4e-3 / 3.0) * third / (0.1 + third ** 4) ** 2 * g["rt"]
    return g


def _prepare_points(eng, g):
    return eng.prepare(g["xyz"], g["w"], g["rho"], g["grad"], g["own"], g["atoms"], B_VV, C_VV, RHO_CUT)


def prepare(case, seed):
    g = _inputs(case, seed)
    call, prec = case["call"], PREC[case["prec"]]
    eng = vv10.VV10(0)
    state = dict(call=call, prec=prec, eng=eng, g=g)
    if call == "batch":
        mols = g["mols"]
        cat = lambda k: torch.cat([m[k] for m in mols]).contiguous()
        off = np.concatenate([[0], np.cumsum([m["w"].shape[0] for m in mols])])
        state.update(off=off, P=[3 * m["atoms"] for m in mols], atoms=[m["atoms"] for m in mols],
                     pts={k: cat(k) for k in ("xyz", "w", "rho", "grad", "own")},
                     rt=torch.cat([t[0].reshape(-1) for t in g["trials"]]),
                     gt=torch.cat([t[1].reshape(-1, 3) for t in g["trials"]]))
        n, tot = int(off[-1]), state["rt"].shape[0]
        state.update(E=torch.empty(len(mols), **F64), vr=torch.empty(n, **F64), vg=torch.empty(n, **F64),
                     fr=torch.empty(tot, **F64), fg=torch.empty(tot, **F64))
        g.clear()
    elif call in ("response", "coords", "weights", "ao"):
        _prepare_points(eng, g)
        if call == "response":
            eng.energy_potential(prec)
    elif call == "step":
        vv10.vv10_set_options(eng.h, vv10.VV10_OPT_FUSE_HESSIAN_SUMS)
    return state


# ------------------------------------------------------------------ the calls

def run(state):
    eng, g, prec = state["eng"], state["g"], state["prec"]
    call = state["call"]
    if call == "scf":
        _prepare_points(eng, g)
        return eng.energy_potential(prec)
    if call == "step":
        _prepare_points(eng, g)
        e, vr, vg, fr, fg, gp, ga, _ = eng.evaluate(prec, g["rt"], g["gt"])
        return e, vr, vg, fr, fg, gp, ga
    if call == "response":
        return eng.hessian_contract(g["rt"], g["gt"], prec)
    if call == "coords":
        gp, ga, euw = eng.coord_grad(prec, resolved=True)
        blocks, _ = eng.coord_hessian(prec)
        return gp, ga, euw, blocks
    if call == "weights":
        return eng.weight_response(g["wt"], prec)
    if call == "ao":
        return (eng.fock_matrix(g["phi"], g["dphi"], g["vrho"], g["vgamma"]),
                eng.orbital_hessian(g["phi"], g["dphi"], g["frt"], g["fgt"], g["gt"], g["vgamma"]))
    p = state["pts"]
    vv10.vv10_batch_prepare(eng.h, state["off"], p["xyz"], p["w"], p["rho"], p["grad"], p["own"],
                            state["atoms"], B_VV, C_VV, RHO_CUT)
    vv10.vv10_batch_run(eng.h, prec, state["P"], state["rt"], state["gt"], state["E"], state["vr"],
                        state["vg"], state["fr"], state["fg"])
    return state["E"], state["vr"], state["vg"], state["fr"], state["fg"]


def work(case):
    """Bytes of the caller's arrays read and written once; flops of the sums over unordered pairs
    (what two points share is evaluated once, each adds its own terms)."""
    call, P = case["call"], case["trials"]
    if call == "batch":  # on average 8.5 atoms a molecule
        n = 8.5 * case["n_rad"] * case["n_ang"]
        k = KEPT * n
        one = (8 * n * (8.5 + 2) + 26 * n * 48, k * k * (20 + 8 * 26))
        return {"bytes": case["atoms"] * one[0], "flops": case["atoms"] * one[1]}
    n = case["atoms"] * case["n_rad"] * case["n_ang"]
    k = KEPT * n
    pts = 8 * n * 8.5
    if call == "scf":
        return {"bytes": pts + 16 * n, "flops": 15 * k * k}
    if call == "step":
        return {"bytes": pts + 16 * n + 24 * n + 48 * P * n, "flops": k * k * (29 + 8 * P)}
    if call == "response":
        return {"bytes": 48 * P * n, "flops": 8 * P * k * k}
    if call == "coords":
        return {"bytes": pts + 24 * n + 72 * n * case["atoms"], "flops": 50 * k * k}
    if call == "weights":
        return {"bytes": 32 * P * n, "flops": (15 + 6 * P) * k * k}
    nbf = 13 * case["atoms"] / 3
    return {"bytes": 8 * n * (4 * nbf + 2 + 5 * P) + 8 * nbf * nbf * (P + 1),
            "flops": 2 * nbf * nbf * k * (P + 1)}


# ------------------------------------------------------------------ plain FP64 values

class _Points:
    """The kept points with omega, kappa and their derivatives (Sec. II.A)."""

    def __init__(self, g):
        keep = (g["rho"] >= RHO_CUT).nonzero()[:, 0]
        self.keep, self.n = keep, g["w"].shape[0]
        self.r, self.w, rho, self.grad = (g[k][keep] for k in ("xyz", "w", "rho", "grad"))
        gam = (self.grad ** 2).sum(1)
        self.rho, self.c = rho, self.w * rho
        self.own = g["own"][keep].long()
        om = (C_VV * gam ** 2 / rho ** 4 + 4.0 * math.pi / 3.0 * rho).sqrt()
        ka = B_VV * 1.5 * math.pi * (rho / (9.0 * math.pi)) ** (1.0 / 6.0)
        self.om, self.ka, self.ka_r, self.ka_rr = om, ka, ka / (6.0 * rho), -5.0 / 36.0 * ka / rho ** 2
        self.om_r = (-2.0 * C_VV * gam ** 2 / rho ** 5 + 2.0 * math.pi / 3.0) / om
        self.om_g = C_VV * gam / rho ** 4 / om
        self.om_rr = (10.0 * C_VV * gam ** 2 / rho ** 6 - self.om_r ** 2) / om
        self.om_rg = (-4.0 * C_VV * gam / rho ** 5 - self.om_r * self.om_g) / om
        self.om_gg = (C_VV / rho ** 4 - self.om_g ** 2) / om
        self.beta = (3.0 / B_VV ** 2) ** 0.75 / 32.0

    def full(self, v):
        """Values of the kept points (last index, or last but one) in the caller's order."""
        out = torch.zeros(*v.shape[:-1], self.n, **F64)
        out[..., self.keep] = v
        return out

    def chunks(self, elements=1 << 26):
        return torch.arange(self.r.shape[0], device=DEV).split(max(1, elements // max(1, self.r.shape[0])))

    def pairs(self, i, j=slice(None)):
        """R^2, Phi, 1/s, 1/g, 1/g' for rows i and columns j (no terms left out)."""
        d = self.r[i][:, None, :] - self.r[j][None, :, :]
        r2 = (d * d).sum(2)
        g = self.om[i][:, None] * r2 + self.ka[i][:, None]
        gp = self.om[j] * r2 + self.ka[j]
        s = g + gp
        return d, r2, -1.5 / (g * gp * s), 1.0 / s, 1.0 / g, 1.0 / gp


def _row_sums(p):
    """E, U, W, A, B, C of every kept point and the point-gradient sums."""
    out = [torch.empty_like(p.rho) for _ in range(6)]
    G = torch.empty_like(p.r)
    for i in p.chunks(1 << 24):
        d, r2, phi, L, Gi, Gj = p.pairs(i)
        f = phi * p.c
        t = L + Gi
        D = p.om[i][:, None] * Gi + p.om * Gj + (p.om[i][:, None] + p.om) * L
        G[i] = torch.einsum("ij,ijk->ik", f * D, d)
        m = 2.0 * f * (L * t + Gi * Gi)
        for q, v in enumerate((f, -f * t, -f * t * r2, m, m * r2, m * r2 * r2)):
            out[q][i] = v.sum(1)
    return out + [G]


def _potential(p, s):
    E, U, W = s[:3]
    return (p.c * (p.beta + 0.5 * E)).sum(), p.beta + E + p.rho * (p.ka_r * U + p.om_r * W), p.rho * p.om_g * W


def _response(p, s, rt, gt):
    """f^{rho,t}, f^{gamma,t}: the directional derivatives of f^rho, f^gamma."""
    E, U, W, A, B, C = s[:6]
    dr = rt[:, p.keep].T
    dg = 2.0 * torch.einsum("kc,tkc->kt", p.grad, gt[:, p.keep])
    u, y = p.w[:, None] * dr, (p.w * p.rho * p.om_g)[:, None] * dg
    fr, fg = torch.empty_like(u), torch.empty_like(u)
    a, b = p.rho * p.ka_r, p.rho * p.om_r
    for i in p.chunks(1 << 25):
        _, r2, phi, L, Gi, Gj = p.pairs(i)
        ni, nj = a[i][:, None] + b[i][:, None] * r2, a + b * r2
        M, t, tj = 2.0 * (L * L + Gi * Gj), L + Gi, L + Gj
        X = phi * (ni * M - tj)
        fr[i] = (phi * (1.0 - ni * t) + X * nj) @ u + (X * r2) @ y
        phi = phi * r2
        fg[i] = (phi * (nj * M - t)) @ u + (phi * r2 * M) @ y
    col = lambda v: v[:, None]
    dk, do = col(p.ka_r) * dr, col(p.om_r) * dr + col(p.om_g) * dg
    dU, dW = col(A) * dk + col(B) * do, col(B) * dk + col(C) * do
    fr += col(U) * dk + col(W) * do + dr * col(p.ka_r * U + p.om_r * W) + col(p.rho) * (
        col(p.ka_rr * U) * dr + (col(p.om_rr) * dr + col(p.om_rg) * dg) * col(W) + col(p.ka_r) * dU + col(p.om_r) * dW)
    fg = col(p.rho * p.om_g) * (fg + dW) + dr * col(p.om_g * W) + col(p.rho * W) * (col(p.om_rg) * dr + col(p.om_gg) * dg)
    return p.full(fr.T), p.full(fg.T)


def _coords(p, n_atom):
    """Point and atom gradients, the atom-resolved sums and the grid-grid blocks."""
    nk = p.r.shape[0]
    euw = torch.zeros(3, nk, n_atom, 3, **F64)
    G = torch.zeros(nk, 3, **F64)
    H = torch.zeros(n_atom, n_atom, 3, 3, **F64)
    eye = torch.eye(3, **F64)
    for B in range(n_atom):
        j = (p.own == B).nonzero()[:, 0]
        if not len(j):
            continue
        for i in torch.arange(nk, device=DEV).split(max(1, (1 << 24) // len(j))):
            d, r2, phi, L, Gi, Gj = p.pairs(i, j)
            f, oi, so = phi * p.c[j], p.om[i][:, None], p.om[i][:, None] + p.om[j]
            D, t = oi * Gi + p.om[j] * Gj + so * L, L + Gi
            X = D * t + oi * Gi * Gi + so * L * L
            for q, v in enumerate((2.0 * f * D, -2.0 * f * X, -2.0 * f * (r2 * X - t))):
                euw[q, i, B] = torch.einsum("ij,ijk->ik", v, d)
            G[i] += 0.5 * euw[0, i, B]
            h = 2.0 * f * (D * D + (oi * Gi) ** 2 + (p.om[j] * Gj) ** 2 + (so * L) ** 2)
            Dij = -2.0 * (torch.einsum("ijk,ij,ijl->ikl", d, h, d) - (f * D).sum(1)[:, None, None] * eye)
            Dij *= p.c[i][:, None, None]
            H[:, B].index_add_(0, p.own[i], Dij)
    at = torch.arange(nk, device=DEV)
    euw[:, at, p.own] = 0.0
    euw[:, at, p.own] = -euw.sum(2)
    a = torch.arange(n_atom, device=DEV)
    H[a, a] = 0.0
    H[a, a] = -H.sum(1)
    gp = torch.zeros(p.n, 3, **F64)
    gp[p.keep] = -2.0 * p.c[:, None] * G
    ga = torch.zeros(n_atom, 3, **F64).index_add_(0, p.own, gp[p.keep])
    out = torch.zeros(3, p.n, n_atom, 3, **F64)
    out[:, p.keep] = euw
    return gp, ga, out, H


def _weights(p, wt):
    v = (wt[:, p.keep] * p.rho).T.contiguous()
    out = [torch.empty_like(v) for _ in range(3)]
    for i in p.chunks(1 << 25):
        _, r2, phi, L, Gi, _ = p.pairs(i)
        t = -phi * (L + Gi)
        for q, f in enumerate((phi, t, t * r2)):
            out[q][i] = f @ v
    return tuple(p.full(x.T) for x in out)


def _assemble(p, g):
    phi, dphi = g["phi"][p.keep], g["dphi"][p.keep]

    def matrix(s, v):
        z = 0.5 * s[:, None] * phi + 2.0 * torch.einsum("kc,kmc->km", v, dphi)
        m = phi.T @ (p.w[:, None] * z)
        return m + m.T

    k = lambda name: g[name][..., p.keep]
    fock = matrix(k("vrho"), k("vgamma")[:, None] * p.grad)
    gt = [matrix(s, f[:, None] * p.grad + k("vgamma")[:, None] * d)
          for s, f, d in zip(k("frt"), k("fgt"), g["gt"][:, p.keep])]
    return fock, torch.stack(gt)


def exact(case, seed):
    g = _inputs(case, seed)
    call = case["call"]
    if call == "batch":
        parts = []
        for m, (rt, gt) in zip(g["mols"], g["trials"]):
            p = _Points(m)
            s = _row_sums(p)
            e, vr, vg = _potential(p, s)
            fr, fg = _response(p, s, rt, gt)
            parts.append((e[None], p.full(vr), p.full(vg), fr.reshape(-1), fg.reshape(-1)))
        return tuple(torch.cat(x) for x in zip(*parts))
    p = _Points(g)
    if call == "coords":
        return _coords(p, g["atoms"])
    if call == "weights":
        return _weights(p, g["wt"])
    if call == "ao":
        return _assemble(p, g)
    s = _row_sums(p)
    e, vr, vg = _potential(p, s)
    if call == "scf":
        return float(e), p.full(vr), p.full(vg)
    fr, fg = _response(p, s, g["rt"], g["gt"])
    if call == "response":
        return fr, fg
    gp = torch.zeros(p.n, 3, **F64)
    gp[p.keep] = -2.0 * p.c[:, None] * s[6]
    ga = torch.zeros(g["atoms"], 3, **F64).index_add_(0, p.own, gp[p.keep])
    return float(e), p.full(vr), p.full(vg), fr, fg, gp, ga
