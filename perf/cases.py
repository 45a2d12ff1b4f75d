"""Workloads that time this library: what each stands for, its inputs and its work.

Every case is one pass of a program that uses the library through its Python
binding: a single-point energy and forces (`Surface`), the orthonormalisation
of a new geometry's guess, one sweep over a caller-built Fock matrix, forces at
given MOs, the density of given MOs, one SCC iteration of a restarted SCF, the
grouping of a geometry. Systems are the seeded water lattices of `synth`.

Two kinds of MOs are used. The SCC cases restart from MOs that the SCF itself
reached (guess, loose orthonormalisation, three iterations), held in
page-locked host memory as a restarting program holds them. The single layers
(sweep, forces, density) take MOs drawn here: every MO is spread over the
molecules within `reach` bohr of its group, decaying with the distance down to
the sparse threshold, as MOs are in the middle of an SCF; their results can
then be checked against plain 64-bit arithmetic (`exact`).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1402_2880_gb300 import SSCF_FP64, SSCF_MIXED, SSCF_ORTHO_ALL, Context
from paper_1402_2880_gb300._lib import group_molecules
from paper_1402_2880_gb300.dynamics import Surface
from synth import concat_clusters, default_params, lattice_water

PREC = {"fp64": SSCF_FP64, "mixed": SSCF_MIXED}
DECAY = 3.4   # bohr: from 0.3 at the MO's own molecule to the threshold 1e-5 at 35 bohr
REACH = 35.0  # bohr: fills an MO of a 4096-molecule lattice as the SCF does after a few iterations


def listed():
    return [
        # the smallest whole call: energy and forces of a few molecules, all launch latency
        {"name": "point_8_mixed", "kind": "point", "n": 8, "precision": "mixed"},
        # the converged 32-molecule cluster (the accuracy workload), one step of an MD or an optimisation
        {"name": "point_32_fp64", "kind": "point", "n": 32, "precision": "fp64"},
        # the start of an SCF at a new geometry off the lattice: guess, loose orthonormalisation, charges; k-means groups, some not full
        {"name": "ortho_512_mixed", "kind": "ortho", "n": 512, "precision": "mixed", "sigma": 0.1, "groups": "kmeans"},
        # a caller's own Fock matrix (another method's step IV) through transform, selection and sweep
        {"name": "sweep_216_fp64", "kind": "sweep", "n": 216, "precision": "fp64", "eps": 1e-5},
        # forces of a small system in FP64 and of a large one in mixed precision
        {"name": "forces_216_fp64", "kind": "forces", "n": 216, "precision": "fp64"},
        {"name": "forces_2000_mixed", "kind": "forces", "n": 2000, "precision": "mixed"},
        # charges, energy and P on the pattern for given MOs; 997 leaves the last cells partly filled
        {"name": "density_997_mixed", "kind": "density", "n": 997, "precision": "mixed"},
        # one SCC iteration in FP64; 7 x 7 x 7 leaves a face of half-filled groups
        {"name": "scc_343_fp64", "kind": "scc", "sizes": "343", "precision": "fp64", "eps": 1e-5, "graph": False},
        # one SCC iteration, ordinary size, ragged
        {"name": "scc_997_mixed", "kind": "scc", "sizes": "997", "precision": "mixed", "eps": 1e-5, "graph": False},
        # the benchmark's cluster, one SCC iteration
        {"name": "scc_4096_mixed", "kind": "scc", "sizes": "4096", "precision": "mixed", "eps": 1e-5, "graph": False},
        # a batch of independent clusters in one context, each iteration one CUDA-graph replay
        {"name": "scc_batch_mixed", "kind": "scc", "sizes": "211,640,1500,333,2222", "precision": "mixed", "eps": 1e-5,
         "graph": True},
        # step I for a disordered geometry: constrained k-means
        {"name": "group_1000", "kind": "group", "n": 1000, "sigma": 0.5, "n_link": 7},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["point", "ortho", "sweep", "forces", "density", "scc", "scc", "scc", "group"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if kind == "point":
        return {"kind": kind, "n": rng.randint(2, 16), "precision": precision}
    if kind == "ortho":
        return {"kind": kind, "n": _log_int(rng, 20, 1000 if precision == "mixed" else 300), "precision": precision,
                "sigma": round(rng.uniform(0.0, 0.1), 3), "groups": rng.choice(["cells", "kmeans"])}
    if kind == "sweep":
        return {"kind": kind, "n": _log_int(rng, 20, 350), "precision": precision, "eps": rng.choice([1e-4, 1e-5, 1e-6])}
    if kind == "forces":
        return {"kind": kind, "n": _log_int(rng, 20, 1600 if precision == "mixed" else 250), "precision": precision}
    if kind == "density":
        return {"kind": kind, "n": _log_int(rng, 20, 1600 if precision == "mixed" else 400), "precision": precision}
    if kind == "group":
        return {"kind": kind, "n": _log_int(rng, 50, 1000), "sigma": round(rng.uniform(0.3, 0.6), 3),
                "n_link": rng.randint(4, 8)}
    eps = rng.choice([1e-4, 1e-5, 1e-6])
    if rng.random() < 0.3:
        sizes = ",".join(str(_log_int(rng, 60, 900 if precision == "mixed" else 150)) for _ in range(rng.randint(2, 4)))
    else:
        sizes = str(_log_int(rng, 27, 2500 if precision == "mixed" else 340))
    return {"kind": "scc", "sizes": sizes, "precision": precision, "eps": eps, "graph": rng.random() < 0.4}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _system(case, seed):
    if "sizes" in case:
        return concat_clusters([lattice_water(int(n), seed=seed + 1000 * k)
                                for k, n in enumerate(case["sizes"].split(","))])
    if case["kind"] == "density":
        seed = 0   # one geometry, whose block pattern shapes P; the MOs differ
    if case["kind"] == "point":   # the points of one trajectory, around a cluster that converges
        return lattice_water(case["n"], seed=0, displace_sigma_A=0.01, displace_seed=seed)
    s = lattice_water(case["n"], seed=seed, displace_sigma_A=case.get("sigma", 0.0), displace_seed=seed + 5)
    if case.get("groups") == "kmeans":
        s.group_of_mol, s.n_groups, _ = group_molecules(s.xyz)
    return s


def _tiles(s):
    """Tiles of 16 MOs as sscf_get_C_tiles numbers them: (group, virtual?, first MO inside the group, MOs) each."""
    n_mol = np.bincount(s.group_of_mol, minlength=s.n_groups)
    out = []
    for virt, per in ((0, 4), (1, 2)):
        for g in range(s.n_groups):
            out += [(g, virt, k, min(16, per * n_mol[g] - k)) for k in range(0, per * n_mol[g], 16)]
    return np.array(out, dtype=np.int64)


def _drawn_mos(s, seed, eps):
    """MOs in the stored form of sscf_set_C_tiles: (nt, tiles, vals on the GPU). Values fit FP32."""
    tl = _tiles(s)
    o = torch.as_tensor(s.xyz.reshape(-1, 3, 3)[:, 0], device="cuda")
    grp = torch.as_tensor(s.group_of_mol, dtype=torch.int64, device="cuda")
    cen = torch.zeros(s.n_groups, 3, dtype=torch.float64, device="cuda").index_add_(0, grp, o)
    cen /= torch.bincount(grp, minlength=s.n_groups)[:, None]
    t_grp = torch.as_tensor(tl[:, 0], device="cuda")
    d = torch.cdist(o, cen)                              # molecule x group
    row, tile = torch.nonzero(d[:, t_grp] < REACH, as_tuple=True)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(row.numel(), 6, 16, generator=gen, device="cuda")
    v *= (0.05 * torch.exp(-d[row, t_grp[tile]] / DECAY)).float()[:, None, None]
    # an MO's own molecule: orthonormal coefficients, as the guess gives them
    Q = torch.linalg.qr(torch.randn(s.n_mol, 6, 6, generator=gen, device="cuda", dtype=torch.float64))[0].float()
    order = np.argsort(s.group_of_mol, kind="stable")    # molecules group by group
    local = np.empty(s.n_mol, dtype=np.int64)
    first = np.concatenate([[0], np.cumsum(np.bincount(s.group_of_mol, minlength=s.n_groups))])[:-1]
    local[order] = np.arange(s.n_mol) - first[s.group_of_mol[order]]
    loc = torch.as_tensor(local, device="cuda")
    t_virt, t_k = (torch.as_tensor(tl[:, i], device="cuda") for i in (1, 2))
    per = torch.where(t_virt[tile] == 1, 2, 4)
    col0 = per * loc[row] - t_k[tile]                    # column of the molecule's first MO of this kind
    own = (grp[row] == t_grp[tile]) & (col0 >= 0) & (col0 < 16)
    for virt, cols in ((0, range(4)), (1, range(2))):
        k = torch.nonzero(own & (t_virt[tile] == virt))[:, 0]
        for c in cols:
            v[k, :, col0[k] + c] = Q[row[k], :, (4 if virt else 0) + c]
    v[v.abs() < eps] = 0.0
    n_mo = torch.as_tensor(tl[:, 3], device="cuda")
    v *= torch.arange(16, device="cuda")[None, None, :] < n_mo[tile][:, None, None]
    nt = torch.bincount(row, minlength=s.n_mol)
    return nt, tile, v.double()


def _drawn_fock(s, mn, seed):
    """A symmetric one-electron matrix on the molecule-pair blocks mn, decaying with the distance."""
    n = mn.shape[0]
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    ij = torch.as_tensor(mn, dtype=torch.int64, device="cuda")
    o = torch.as_tensor(s.xyz.reshape(-1, 3, 3)[:, 0], device="cuda")
    X = torch.randn(n, 6, 6, generator=gen, device="cuda", dtype=torch.float64)
    X *= (0.2 * torch.exp(-(o[ij[:, 0]] - o[ij[:, 1]]).norm(dim=1) / 2.0))[:, None, None]
    diag = ij[:, 0] == ij[:, 1]
    X[diag] += torch.diag(torch.tensor([-0.9, -0.6, -0.5, -0.4, 0.2, 0.3], dtype=torch.float64, device="cuda"))
    key = ij[:, 0] * s.n_mol + ij[:, 1]                  # blocks come sorted by it
    rev = torch.searchsorted(key, ij[:, 1] * s.n_mol + ij[:, 0])
    return 0.5 * (X + X[rev].transpose(1, 2))


def _pinned(a):
    a = torch.as_tensor(a)
    t = torch.empty(a.shape, dtype=a.dtype, pin_memory=True)
    t.copy_(a)
    return t.numpy()


def prepare(case, seed):
    p = default_params()
    kind = case["kind"]
    s = _system(case, seed)
    if kind == "group":
        return {"kind": kind, "xyz": s.xyz, "n_link": case["n_link"]}
    prec = PREC[case["precision"]]
    if kind == "point":
        return {"kind": kind, "surface": Surface(s, p, precision=prec, restart=False), "xyz": s.xyz}
    eps = case.get("eps", 1e-5)
    st = {"kind": kind}
    stream = None
    if case.get("graph"):
        st["stream"] = torch.cuda.Stream()
        stream = st["stream"].cuda_stream
    ctx = st["ctx"] = Context.from_system(s, p, precision=prec, stream=stream)
    if kind == "ortho":
        ctx.set_thresholds(1e-3, 1e-1, 1e-8)   # the loose stage
        return st
    if kind == "scc":
        ctx.set_thresholds(1e-3, 1e-1, 1e-8)
        ctx.guess()
        ctx.orthonormalise(SSCF_ORTHO_ALL)
        ctx.set_thresholds(eps, 10 * eps, 1e-6)
        ctx.reset_charges()
        for _ in range(3):
            ctx.step()
        st["C"] = tuple(_pinned(a) for a in ctx.get_C_tiles())
        st["q"] = tuple(_pinned(a) for a in ctx.get_charges())
        if case["graph"]:
            ctx.enable_graph(True)
        return st
    ctx.set_thresholds(eps, 10 * eps, 1e-6)
    nt, tiles, vals = _drawn_mos(s, seed, eps)
    st["C"] = (_pinned(nt.int()), _pinned(tiles.int()), _pinned(vals))
    if kind == "sweep":
        mn = ctx.get_blocks()[0]
        st["X"] = _pinned(_drawn_fock(s, mn, seed))
    else:
        ctx.set_C_tiles(*st.pop("C"))
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "point":
        pt = st["surface"](st["xyz"])
        return {"energy": pt.energy, "forces": pt.forces, "converged": pt.converged}
    if kind == "group":
        groups, n_groups, iters = group_molecules(st["xyz"], n_link=st["n_link"])
        return {"group_of_mol": groups, "n_groups": n_groups, "iters": iters}
    ctx = st["ctx"]
    if kind == "ortho":
        ctx.guess()
        passes, eta = ctx.orthonormalise(SSCF_ORTHO_ALL)
        energy = ctx.reset_charges()
        q, dq_in, Q_in = ctx.get_charges()
        return {"passes": passes, "eta": eta, "energy": energy, "q": q, "dq_in": dq_in, "Q_in": Q_in}
    if kind == "sweep":
        ctx.set_C_tiles(*st["C"])
        ctx.set_fock_blocks(st["X"])
        n_rot, max_fov = ctx.rotate_sweep()
        F_ov, F_diag = ctx.get_F()
        return {"n_rot": n_rot, "max_fov": max_fov, "F_ov": F_ov, "F_diag": F_diag, "C": ctx.get_C()}
    if kind == "forces":
        dx, dp = ctx.gradients()
        return {"dE_dxyz": dx, "dE_dparams": dp}
    if kind == "density":
        q, energy, _ = ctx.density()
        return {"q": q, "energy": energy, "P": ctx.density_blocks()}
    ctx.set_C_tiles(*st["C"])
    ctx.set_charges(*st["q"])
    info = ctx.step()
    q, dq_in, Q_in = ctx.get_charges()
    cl_energy, cl_dq = ctx.cluster_results()
    return {"energy": info["energy"], "dq_max": info["dq_max"], "max_fov": info["max_fov"], "eta": info["eta"],
            "n_rot": info["n_rot"], "n_combo": info["n_combo"], "q": q, "dq_in": dq_in, "Q_in": Q_in,
            "cluster_energy": cl_energy, "cluster_dq": cl_dq}


# ---------------------------------------------------------------------------
# bytes and operations of one pass
# ---------------------------------------------------------------------------
def _within(radius_bohr, n):
    """Molecules of an n-molecule lattice cluster within a radius of one of them."""
    r = radius_bohr * 0.529177 / 3.1
    return min(float(n), 4.0 / 3.0 * math.pi * r ** 3)


def work(case):
    kind = case["kind"]
    if kind == "group":
        n = case["n"]
        c = math.ceil(n / case["n_link"])
        return {"bytes": 24.0 * n + 24.0 * c + 4.0 * n, "flops": 2 * 8.0 * n * c}
    b = 4 if case["precision"] == "mixed" else 8
    total = {"bytes": 0.0, "flops": 0.0}
    for n in [int(x) for x in case.get("sizes", str(case.get("n"))).split(",")]:
        held = _within(33.0, n)            # molecules an MO is spread over (all of them in a small cluster)
        pattern = _within(11.5, n)         # molecules that one molecule has matrix blocks with
        near = _within(26.0, n)            # molecules in the neighbouring groups of one molecule's group
        c_occ, c_all = 24.0 * n * held, 36.0 * n * held          # stored values
        blocks = 36.0 * n * pattern
        charges = 8.0 * 3 * n * 6
        f_density = 2 * 4.0 * blocks / 2 * held
        f_xc = 2 * 6.0 * pattern * c_all                          # X C
        f_ov = 2 * 8.0 * n * near * 6 * held                      # C^T (X C) on neighbouring blocks
        f_oo = 2 * 16.0 * n * near / 2 * 6 * held
        f_combo = 4 * 16.0 * n * near / 2 * 0.65 * 6 * held       # 2x2 updates of an occupied pass
        f_rot = 6 * 40.0 * n * 6 * held                           # at most 10 N_occ rotations
        f_gamma = 10.0 * 9 * n * n
        if kind == "density":
            total["bytes"] += b * c_occ + 3 * 8 * blocks + charges
            total["flops"] += f_density + f_gamma
        elif kind == "forces":
            total["bytes"] += b * c_occ + 8 * 2 * blocks + charges
            total["flops"] += 2 * f_density + f_xc + f_oo + 2 * 16.0 * n * near * 6 * held + 2 * f_gamma
        elif kind == "sweep":
            total["bytes"] += 8 * (c_all + 36.0 * n * n + blocks + 8.0 * n * n + 6 * n)
            total["flops"] += f_xc + f_ov + f_rot
        elif kind == "ortho":
            total["bytes"] += 8 * 2 * blocks + charges
            total["flops"] += 3 * (f_xc + 2.25 * (f_oo + f_combo)) + f_density + f_gamma
        else:
            rounds = 30 if kind == "point" else 1
            total["bytes"] += 8 * c_all + 8 * 2 * blocks + charges
            total["flops"] += rounds * (2 * f_xc + f_ov + f_oo + f_combo + f_rot + f_density + f_gamma)
    return total


# ---------------------------------------------------------------------------
# the same results in plain 64-bit arithmetic
# ---------------------------------------------------------------------------
def _sk(x, p, tab):
    """Slater-Koster matrix (H0 or S) of the atoms x: AOs O s, px, py, pz, H s, H s per molecule."""
    n_at = x.shape[0]
    dev = x.device
    V = tab
    R = x[None, :, :] - x[:, None, :]
    d2 = (R * R).sum(-1)
    eye = torch.eye(n_at, dtype=torch.bool, device=dev)
    on = (d2 <= p["r_cut"] ** 2) & ~eye
    r = torch.sqrt(torch.where(eye, torch.ones_like(d2), d2))
    e = R / r[:, :, None]
    f = torch.where(on, torch.exp(-r / p["r_decay"]), torch.zeros_like(r))
    at = torch.arange(n_at, device=dev)
    ao_at = torch.stack([at[0::3], at[0::3], at[0::3], at[0::3], at[1::3], at[2::3]], 1).reshape(-1)
    comp = torch.tensor([-1, 0, 1, 2, -1, -1], device=dev).repeat(n_at // 3)   # p component, or -1 for s
    f, e = f[ao_at][:, ao_at], e[ao_at][:, ao_at]
    pi, pj = (comp >= 0)[:, None], (comp >= 0)[None, :]
    c = comp.clamp(min=0)
    ei = torch.gather(e, 2, c[:, None, None].expand(-1, e.shape[1], 1))[:, :, 0]
    ej = torch.gather(e, 2, c[None, :, None].expand(e.shape[0], -1, 1))[:, :, 0]
    same = (comp[:, None] == comp[None, :]).double()
    pp = ei * ej * (V[2] - V[3]) + same * V[3]
    m = torch.where(pi & pj, pp, torch.where(pj & ~pi, ej * V[1], torch.where(pi & ~pj, -ei * V[1], V[0] * torch.ones_like(f))))
    return m * f


def _dense_mos(s, nt, tile, vals):
    """The drawn MOs as a dense matrix, occupied columns first, and the group of every column."""
    tl = torch.as_tensor(_tiles(s), device="cuda")
    mo0 = torch.cumsum(tl[:, 3], 0) - tl[:, 3]            # tiles in order hold the MOs in order
    C = torch.zeros(s.n_mol, 6, 6 * s.n_mol, dtype=torch.float64, device="cuda")
    row = torch.repeat_interleave(torch.arange(s.n_mol, device="cuda"), nt)
    for c in range(16):
        k = torch.nonzero(tl[tile, 3] > c)[:, 0]
        C[row[k], :, mo0[tile[k]] + c] = vals[k, :, c]
    return C.reshape(6 * s.n_mol, 6 * s.n_mol), torch.repeat_interleave(tl[:, 0], tl[:, 3])


def _neighbours(s, p):
    """Groups with an atom pair closer than group_cut."""
    x = torch.as_tensor(s.xyz.reshape(-1, 3), device="cuda")
    g = torch.as_tensor(np.repeat(s.group_of_mol, 3), dtype=torch.int64, device="cuda")
    near = torch.zeros(s.n_groups, s.n_groups, dtype=torch.bool, device="cuda")
    for k in range(0, x.shape[0], 1024):
        d2 = (x[k:k + 1024, None] - x[None]).square().sum(-1)
        a, b = torch.nonzero(d2 < p["group_cut"] ** 2, as_tuple=True)
        near[g[a + k], g[b]] = True
    return near


def _gamma(x, U):
    d2 = (x[:, None] - x[None]).square().sum(-1)
    h = 0.5 * (1 / U[:, None] + 1 / U[None])
    return 1 / torch.sqrt(d2 + h * h)


def exact(case, seed):
    kind = case["kind"]
    # the others give whole numbers, or the product of millions of ordered 2x2 updates: no plain form under 20 seconds
    if kind not in ("sweep", "forces", "density"):
        return None
    p = default_params()
    s = _system(case, seed)
    eps = case.get("eps", 1e-5)
    nt, tile, vals = _drawn_mos(s, seed, eps)
    C, mo_grp = _dense_mos(s, nt, tile, vals)
    n_mol, n_occ = s.n_mol, 4 * s.n_mol
    x = torch.as_tensor(s.xyz.reshape(-1, 3), device="cuda")
    onsite = torch.tensor([p["onsite_O_s"]] + 3 * [p["onsite_O_p"]] + 2 * [p["onsite_H_s"]], dtype=torch.float64,
                          device="cuda").repeat(n_mol)
    eye = torch.eye(6 * n_mol, dtype=torch.float64, device="cuda")
    near = _neighbours(s, p)
    d2 = (x[:, None] - x[None]).square().sum(-1).reshape(n_mol, 3, n_mol, 3).amin((1, 3))
    ij = torch.nonzero(d2 <= p["r_cut"] ** 2)             # the molecule-pair pattern, sorted
    if kind == "sweep":
        X = _drawn_fock(s, ij.cpu().numpy(), seed)
        diag = (ij[:, 0] == ij[:, 1])[:, None, None] & torch.eye(6, dtype=torch.bool, device="cuda")
        X = torch.where((X.abs() < eps) & ~diag, torch.zeros_like(X), X)
        H = torch.zeros(n_mol, n_mol, 6, 6, dtype=torch.float64, device="cuda")
        H[ij[:, 0], ij[:, 1]] = X
        F = C.T @ H.permute(0, 2, 1, 3).reshape(6 * n_mol, 6 * n_mol) @ C
        F_ov = F[:n_occ, n_occ:] * near[mo_grp[:n_occ]][:, mo_grp[n_occ:]]
        return {"n_rot": None, "max_fov": float(F_ov.abs().max()), "F_ov": F_ov.cpu().numpy(),
                "F_diag": F.diagonal().cpu().numpy(), "C": None}
    ao_at = torch.arange(3 * n_mol, device="cuda").reshape(-1, 3)[:, [0, 0, 0, 0, 1, 2]].reshape(-1)
    U = torch.tensor([p["U_O"], p["U_H"], p["U_H"]], dtype=torch.float64, device="cuda").repeat(n_mol)
    q0 = torch.tensor([p["q0_O"], p["q0_H"], p["q0_H"]], dtype=torch.float64, device="cuda").repeat(n_mol)
    V0 = torch.tensor(p["V0"], dtype=torch.float64, device="cuda")
    S0 = torch.tensor(p["S0"], dtype=torch.float64, device="cuda")
    H0, S = _sk(x, p, V0) + torch.diag(onsite), _sk(x, p, S0) + eye
    Co = C[:, :n_occ]
    P = 2 * Co @ Co.T
    q = torch.zeros(3 * n_mol, dtype=torch.float64, device="cuda").index_add_(0, ao_at, (P * S).sum(1))
    dq = q - q0
    Q = _gamma(x, U) @ dq
    if kind == "density":
        e = (P * H0).sum() + 0.5 * (dq * Q).sum()
        blocks = P.reshape(n_mol, 6, n_mol, 6).permute(0, 2, 1, 3)[ij[:, 0], ij[:, 1]]
        return {"q": q.cpu().numpy(), "energy": float(e), "P": blocks.cpu().numpy()}
    half = 0.5 * (Q[ao_at][:, None] + Q[ao_at][None])
    H = H0 + S * half
    F_oo = (Co.T @ H @ Co) * near[mo_grp[:n_occ]][:, mo_grp[:n_occ]]
    G = P * half - 2 * Co @ F_oo @ Co.T                   # what dS is contracted with
    del H, F_oo, half
    x.requires_grad_(True)
    V0.requires_grad_(True)
    S0.requires_grad_(True)
    e = (P * _sk(x, p, V0)).sum() + (G * _sk(x, p, S0)).sum() + 0.5 * (dq * (_gamma(x, U) @ dq)).sum()
    gx, gv, gs = torch.autograd.grad(e, (x, V0, S0))
    return {"dE_dxyz": gx.cpu().numpy(), "dE_dparams": torch.cat([gv, gs]).cpu().numpy()}
