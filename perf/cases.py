"""Timed cases of the library's main paths, each through the ctypes binding of the C ABI.

A case is a dict of plain values. `listed()` names the cases, `draw(rng)` gives further ones of the same
ranges, `prepare(case, seed)` builds what a program holds before the call (system, plan, sweep, network,
output buffers), `run(state)` makes one pass, `work(case)` counts the bytes and operations of a pass and
`exact(case, seed)` gives the same outputs in plain FP64 torch, from dense matrices.

The FP64 form's results are handed on in FP64. The mixed form does its column arithmetic in FP32 (and FP32
pairs), and its results are handed on in FP32.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1202_0098_gb300 import mka

DIAMOND = SimpleNamespace(Es=-5.0, Ep=1.0, V=(-4.0, 4.5, 5.5, -1.8), Sv=(0.10, -0.12, -0.15, 0.05), d0=1.54, rc=2.6)
FCC = SimpleNamespace(Es=-2.0, Ep=0.5, V=(-4.0, 4.5, 5.5, -1.8), Sv=(0.10, -0.12, -0.15, 0.05), d0=1.54, rc=3.4)
BASIS = {"diamond": [[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
                     [.25, .25, .25], [.25, .75, .75], [.75, .25, .75], [.75, .75, .25]],
         "fcc": [[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]]}
# the materials of the repository's workloads: lattice constant, vacancies, parameters, kT, blocks per row of H
LATTICE = {"diamond": (3.567, 0.0, DIAMOND, 0.1, 13.3), "fcc": (4.0, 0.05, FCC, 0.05, 12.4)}
STORED = {"fp64": 8, "fp32": 4, "bf16": 2}
MLP_IN, MLP_HID, MLP_OUT, PATCH = 132, 128, 68, 17


def _solve(name, kind, lattice, cells, sigma, R, p, q, storage, arith, n, **more):
    return dict(name=name, kind=kind, lattice=lattice, cells=cells, sigma=sigma, R=R, p=p, q=q, storage=storage,
                arith=arith, n=n, **more)


def listed():
    return [
        # the smallest call: the levels of one atom's four columns, as a program probing one site asks for them
        _solve("one_atom", "levels", "diamond", 4, 0.05, 6.0, 15, 15, "fp64", "fp64", 1),
        # density of states wants large subspaces on a few sites: levels of 37 atoms at nu = 100, then the curve
        _solve("dos_nu100", "levels", "diamond", 4, 0.05, 6.0, 50, 50, "fp64", "fp64", 37, energies=201),
        # the 512-atom system in full: every column, mu, rho, band energy, plain FP64, one direct call each
        _solve("density_512", "density", "diamond", 4, 0.05, 6.0, 15, 15, "fp64", "fp64", 512),
        # production batches through a plan: BF16-stored values, mixed form (the step of the whole-system runs)
        _solve("batch_bf16", "batch", "diamond", 13, 0.1, 6.0, 15, 15, "bf16", "mixed", 8192),
        # uneven clusters (fcc, vacancies), FP64, work ordered by cluster size, an odd number of atoms
        _solve("batch_fcc_fp64", "batch", "fcc", 16, 0.08, 7.0, 15, 15, "fp64", "fp64", 2999, order=True),
        # amorphous-like disorder, larger clusters and subspaces, FP32-stored values, an odd number of atoms
        _solve("batch_fp32_nu40", "batch", "diamond", 13, 0.15, 7.0, 20, 20, "fp32", "mixed", 2501),
        # the whole work flow over a system: learned CG start, sweep, one mu, rho everywhere, forces (an MD step)
        _solve("system_learned", "system", "diamond", 12, 0.1, 6.0, 15, 15, "bf16", "mixed", 13824, batch=4096, kp=8),
        # the training set of the learned start: features and FP64 CG solutions on each atom's patch
        _solve("targets_1500", "targets", "diamond", 8, 0.15, 7.0, 1, 0, "fp32", "fp64", 1500),
        # response of a solved batch: Green's function at one complex energy, energy density matrix and forces
        _solve("response_2048", "response", "diamond", 8, 0.1, 6.0, 15, 15, "fp64", "fp64", 2048),
        # the global products, at memory size and at the smallest system (one launch)
        dict(name="spmv_262k", kind="spmv", cells=32, sigma=0.1, storage="fp32", x="fp32", k=1, which=0),
        dict(name="spmv_512", kind="spmv", cells=4, sigma=0.05, storage="fp64", x="fp64", k=4, which=1),
        # loss and gradients of one training batch of the learned start's network
        dict(name="gradients_1024", kind="gradients", rows=1024),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["levels", "levels", "density", "batch", "batch", "batch", "system", "targets", "response",
                       "spmv", "spmv", "gradients"])
    if kind == "spmv":
        return dict(kind=kind, cells=_log(rng, 4, 30), sigma=round(rng.uniform(0.03, 0.15), 3),
                    storage=rng.choice(list(STORED)), x=rng.choice(["fp64", "fp32"]), k=rng.choice([1, 2, 4]),
                    which=rng.choice([0, 1]))
    if kind == "gradients":
        return dict(kind=kind, rows=_log(rng, 64, 4096))
    lattice = "diamond" if kind == "system" else rng.choice(["diamond", "diamond", "fcc"])
    sigma = round(rng.uniform(0.05, 0.15), 3) if lattice == "diamond" else round(rng.uniform(0.05, 0.1), 3)
    if kind == "system":
        sigma = round(rng.uniform(0.07, 0.12), 3)
    arith = "mixed" if kind == "system" else "fp64" if kind == "targets" else rng.choice(["fp64", "mixed"])
    storage = rng.choice(["fp32", "bf16"]) if arith == "mixed" else rng.choice(list(STORED))
    p = rng.choice([10, 12, 15, 15, 18, 20])
    q = rng.choice([p, p, p - 3, p // 2])
    c = dict(kind=kind, lattice=lattice, cells=rng.choice([5, 6, 7, 8, 9]), sigma=sigma,
             R=round(rng.uniform(5.0 if lattice == "diamond" else 5.7, 7.0), 2), p=p, q=q, storage=storage, arith=arith)
    if kind == "targets":
        c.update(p=1, q=0)
    most = 4 * c["cells"] ** 3 * (2 if lattice == "diamond" else 0.9)
    top = {"levels": 300, "density": 512, "batch": 3000 if arith == "mixed" else 1000, "system": 0, "targets": 1000,
           "response": 1500}[kind]
    if kind == "levels" and rng.random() < 0.3:
        c.update(lattice="diamond", R=round(rng.uniform(5.8, 6.5), 2), p=rng.choice([25, 40, 50]), energies=rng.choice([41, 100, 300]))
        c.update(q=c["p"])
        top = 40
    c["n"] = _log(rng, 1 if kind == "levels" else 60, int(min(top or most, most)))
    if kind == "batch":
        c["order"] = rng.random() < 0.5
    if kind == "system":
        c.update(n=8 * c["cells"] ** 3, batch=rng.choice([500, 1024, 2000]), kp=9, R=round(rng.uniform(5.5, 6.0), 2), p=15, q=15)
    return c


class Owner:
    """The library objects of one state, freed in reverse order when the state goes."""

    def __init__(self):
        self._free = []

    def keep(self, handle, free):
        self._free.append((handle, free))
        return handle

    def __del__(self):
        while self._free:
            h, f = self._free.pop()
            f(h)


def _positions(lattice, cells, sigma, seed):
    """Sites in (ix, iy, iz, basis) order, vacancies, normal displacements; wrapped into the box."""
    a, vacancy = LATTICE[lattice][:2]
    rng = np.random.default_rng(seed)
    g = np.arange(cells, dtype=np.float64)
    cell = np.stack(np.meshgrid(g, g, g, indexing="ij"), axis=-1).reshape(-1, 1, 3)
    pos = ((cell + np.array(BASIS[lattice])[None]) * a).reshape(-1, 3)
    if vacancy:
        pos = pos[rng.random(len(pos)) >= vacancy]
    pos = pos + rng.normal(0.0, sigma, pos.shape)
    box = np.full(3, a * cells)
    pos = np.mod(pos, box)
    pos[pos >= box] -= a * cells
    return np.ascontiguousarray(pos), box


def _selection(case, n_atoms, seed):
    n = min(case["n"], n_atoms)
    if n == n_atoms:
        return np.arange(n, dtype=np.int64)
    return np.sort(np.random.default_rng(seed + 1).choice(n_atoms, n, replace=False)).astype(np.int64)


def _capacity(lattice, n):
    """Pattern blocks a buffer for n atoms holds (more than any configuration's; the rest stays zero)."""
    return n * (19 if lattice == "diamond" else 14) + 16


def _network(seed):
    """Weights of a usable start: each orbital's one-hot passed through to its own entry of s_j, and small noise."""
    rng = np.random.default_rng(seed + 2)
    w1, w2 = rng.normal(0, 0.02, (MLP_HID, MLP_IN)), rng.normal(0, 0.02, (MLP_HID, MLP_HID))
    w3 = rng.normal(0, 0.02, (MLP_OUT, MLP_HID))
    for o in range(4):
        w1[o, 128 + o], w2[o, o], w3[o, o] = 4.0, 1.0, 0.27
    z = np.zeros
    return np.concatenate([w1.ravel(), z(MLP_HID), w2.ravel(), z(MLP_HID), w3.ravel(), z(MLP_OUT)]).astype(np.float32)


def _cg_tol(case):
    return 1e-12 if case["arith"] == "fp64" else 1e-7


def prepare(case, seed):
    s = SimpleNamespace(case=case, own=Owner())
    kind = case["kind"]
    if kind == "gradients":
        g = torch.Generator(device="cuda").manual_seed(seed)
        B = case["rows"]
        s.X = torch.randn((B, MLP_IN), generator=g, device="cuda")
        s.T = torch.randn((B, MLP_OUT), generator=g, device="cuda") * 0.3
        s.net = s.own.keep(mka.mka_mlp_create(seed), mka.mka_mlp_destroy)
        s.grad = torch.empty(mka.mka_mlp_num_params(), dtype=torch.float32, device="cuda")
        s.loss = torch.empty(1, dtype=torch.float32, device="cuda")
        return s
    lattice = case.get("lattice", "diamond")
    pos, box = _positions(lattice, case["cells"], case["sigma"], seed)
    sk, kT = LATTICE[lattice][2:4]
    s.N, s.kT = len(pos), kT
    s.sys = s.own.keep(mka.mka_build_system(pos, box, sk, case["storage"], cluster_radius=case.get("R", 5.0)),
                       mka.mka_system_destroy)
    if kind == "spmv":
        dt = torch.float64 if case["x"] == "fp64" else torch.float32
        g = torch.Generator(device="cuda").manual_seed(seed)
        s.x = torch.randn((4 * s.N, case["k"]), generator=g, device="cuda", dtype=dt)
        s.y = torch.empty_like(s.x)
        return s
    s.atoms = _selection(case, s.N, seed)
    n = len(s.atoms)
    s.mu = 1.98 if lattice == "diamond" else 0.9
    if kind == "targets":
        s.X = torch.empty((4 * n, MLP_IN), dtype=torch.float32, device="cuda")
        s.Y = torch.empty((4 * n, MLP_OUT), dtype=torch.float32, device="cuda")
        s.patch = torch.empty((n, PATCH), dtype=torch.int32, device="cuda")
        return s
    s.prm = mka.solve_params(case["p"], case["q"], arith=case["arith"], cg_tol=_cg_tol(case),
                             keep_vectors=kind != "levels", use_warm_start=kind == "system")
    if kind == "levels":
        e = case.get("energies", 0)
        s.energies = np.linspace(s.mu - 4.0, s.mu + 4.0, e) if e else None
        return s
    blocks = _capacity(lattice, n)
    s.rho = torch.zeros(blocks * 16, dtype=torch.float64, device="cuda")
    if kind == "response":
        s.res = s.own.keep(mka.mka_solve_columns(s.sys, s.atoms, s.prm), mka.mka_result_destroy)
        s.G = torch.zeros((blocks * 16, 2), dtype=torch.float64, device="cuda")
        s.forces = torch.empty((s.N, 3), dtype=torch.float64, device="cuda")
    elif kind == "batch":
        s.plan = s.own.keep(mka.mka_plan_create(s.sys, n, s.prm, mka.tuning(256, 0, case.get("order", False))),
                            mka.mka_plan_destroy)
        mka.mka_plan_run(s.plan, s.atoms, 4.0 * n, kT, s.rho.data_ptr())          # a plan captures its graph once
    elif kind == "system":
        s.net = s.own.keep(mka.mka_mlp_create(0), mka.mka_mlp_destroy)
        mka.mka_mlp_set_params(s.net, _network(seed))
        mka.mka_system_set_warm_start(s.sys, s.net)
        s.plan = s.own.keep(mka.mka_plan_create(s.sys, case["batch"], s.prm), mka.mka_plan_destroy)
        s.sweep = s.own.keep(mka.mka_sweep_create(s.sys, 0, s.N, case["p"] + case["q"], s.mu - 1.0 - 40 * kT,
                                                  s.mu + 1.0 + 40 * kT, case["kp"], 4096, with_forces=True),
                             mka.mka_sweep_destroy)
        s.forces = torch.empty((s.N, 3), dtype=torch.float64, device="cuda")
        for size in {min(case["batch"], s.N), s.N % case["batch"] or case["batch"]}:    # one graph per batch size
            mka.mka_plan_run_sweep(s.plan, s.sweep, s.atoms[:size])
    return s


def _typed(case, v):
    """Results in the type of the form's column arithmetic."""
    if case["arith"] == "fp64":
        return v
    return v.to(torch.float32) if isinstance(v, torch.Tensor) else v.astype(np.float32)


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "spmv":
        mka.mka_spmv(s.sys, c["which"], mka.MKA_FP64 if c["x"] == "fp64" else mka.MKA_MIXED_FP32, s.x.data_ptr(),
                     s.y.data_ptr(), c["k"])
        return s.y
    if kind == "gradients":
        mka.mka_mlp_gradients(s.net, s.X.data_ptr(), s.T.data_ptr(), c["rows"], s.grad.data_ptr(), s.loss.data_ptr())
        return {"grad": s.grad, "loss": s.loss}
    if kind == "targets":
        mka.mka_warm_start_features(s.sys, s.atoms, s.X.data_ptr(), s.patch.data_ptr())
        mka.mka_cg_patch_targets(s.sys, s.atoms, c["arith"], _cg_tol(c), s.patch.data_ptr(), s.Y.data_ptr())
        return {"X": s.X, "Y": s.Y, "patch": s.patch}
    n_el = 4.0 * len(s.atoms)
    if kind == "levels":
        res = mka.mka_solve_columns(s.sys, s.atoms, s.prm)
        lv = mka.mka_result_copy_levels(res)
        out = {"eps": _typed(c, lv["eps"]), "w": _typed(c, lv["w"]), "nu_eff": lv["nu_eff"], "status": lv["status"]}
        if s.energies is not None:
            eps, w = mka.mka_result_device_levels(res)
            out["dos"] = _typed(c, mka.mka_dos(eps, w, lv["eps"].size, s.energies, 0.1))
        mka.mka_result_destroy(res)
        return out
    if kind == "density":
        res = mka.mka_solve_columns(s.sys, s.atoms, s.prm)
        mu = mka.mka_find_mu(res, n_el, s.kT)
        e, n = mka.mka_density_energy(s.sys, res, mu, s.kT, s.rho.data_ptr())
        mka.mka_result_destroy(res)
        return {"rho": _typed(c, s.rho), "mu": mu, "e_band": e, "n_electrons": n}
    if kind == "response":
        mka.mka_greens(s.sys, s.res, complex(s.mu, 0.2), s.G.data_ptr())
        s.forces.zero_()
        mka.mka_forces(s.sys, s.res, s.mu, s.kT, s.rho.data_ptr(), s.forces.data_ptr())
        return {"G": _typed(c, s.G), "pi": _typed(c, s.rho), "forces": _typed(c, s.forces)}
    if kind == "batch":
        mka.mka_plan_run(s.plan, s.atoms, n_el, s.kT, s.rho.data_ptr())
        mu, e, n = mka.mka_plan_scalars(s.plan)
        return {"rho": _typed(c, s.rho), "mu": mu, "e_band": e, "n_electrons": n}
    for a in range(0, s.N, c["batch"]):          # the whole system: every column, one mu, rho, energy, forces
        mka.mka_plan_run_sweep(s.plan, s.sweep, s.atoms[a:a + c["batch"]])
    mu = mka.mka_sweep_find_mu(s.sweep, n_el, s.kT)
    mka.mka_sweep_density(s.sweep, s.plan, mu, s.kT, s.rho.data_ptr())
    e = float(mka.mka_sweep_chunk_sums(s.sweep, mu, s.kT, levels=False, rho=True)["e_rho"].sum())
    mka.mka_sweep_forces(s.sweep, s.plan, mu, s.kT, s.forces.data_ptr())
    return {"rho": _typed(c, s.rho), "mu": mu, "e_band": e, "forces": _typed(c, s.forces)}


def work(case):
    """What a pass cannot do without: the stored values it needs and its results once; the operations of the
    inner CG, the products with H and S, the subspace's overlaps and the reduced eigenproblems."""
    kind = case["kind"]
    if kind == "gradients":
        macs = MLP_IN * MLP_HID + MLP_HID * MLP_HID + MLP_HID * MLP_OUT
        return {"bytes": 4 * case["rows"] * (MLP_IN + MLP_OUT) + 6 * macs,
                "flops": 2 * case["rows"] * (3 * macs - MLP_IN * MLP_HID)}
    lattice = case.get("lattice", "diamond")
    a, vacancy, _, _, per_row = LATTICE[lattice]
    per_cell = len(BASIS[lattice]) * (1 - vacancy)
    N = per_cell * case["cells"] ** 3
    if kind == "spmv":
        t = 8 if case["x"] == "fp64" else 4
        return {"bytes": N * (per_row * (16 * STORED[case["storage"]] + 4) + 8 * t * case["k"]),
                "flops": 32 * N * per_row * case["k"]}
    n, nu = min(case["n"], N), case["p"] + case["q"]
    ncl = per_cell / a ** 3 * 4 / 3 * math.pi * case["R"] ** 3
    blocks, m = 0.8 * per_row * ncl, 4 * ncl
    n_cg = 30 if case["arith"] == "fp64" else 22
    read = 2 * min(N, n * ncl) * per_row * (16 * STORED[case["storage"]] + 4)
    out = 8 * 16 * n * per_row
    if kind == "targets":
        return {"bytes": read / 2 + 16 * n * (MLP_IN + MLP_OUT), "flops": 4 * n * (32 * blocks + 10 * m) * n_cg}
    if kind == "response":
        return {"bytes": 4 * out + 8 * 4 * n * (nu * nu + 4 * per_row * nu), "flops": 4 * n * (6 * nu * nu + 32 * per_row * nu)}
    if kind == "levels":
        out = 8 * 2 * 4 * n * nu
    flops = 4 * n * (32 * blocks * (n_cg + 2 * nu) + 10 * m * n_cg + m * nu * nu + 17 / 3 * nu ** 3)
    return {"bytes": read + out, "flops": flops + 4 * n * nu * 4 * case.get("energies", 0)}


# ---- the same outputs in FP64 from dense matrices -------------------------------------------------

def _image(d, box):
    return d - box * torch.round(d / box)


def _blocks(d, r2, P, d0):
    """Two-centre blocks [..., 4, 4] of displacements d[..., 3]."""
    r = torch.sqrt(r2)
    f = torch.exp(-2.0 * (r / d0 - 1.0))
    l = d / r[..., None]
    row0 = torch.cat([(P[0] * f)[..., None], l * (P[1] * f)[..., None]], -1)[..., None, :]
    pp = l[..., :, None] * l[..., None, :] * ((P[2] - P[3]) * f)[..., None, None]
    pp = pp + torch.eye(3, dtype=d.dtype, device=d.device) * (P[3] * f)[..., None, None]
    rest = torch.cat([-l[..., None] * (P[1] * f)[..., None, None], pp], -1)
    return torch.cat([row0, rest], -2)


def _stored(v, storage):
    return v if storage == "fp64" else v.float().double() if storage == "fp32" else v.float().bfloat16().double()


def _pair_blocks(d, same, sk, storage=None):
    """H and S blocks of pairs at displacements d, the on-site blocks where `same`, zero beyond the cutoff."""
    r2 = (d * d).sum(-1)
    near = (r2 <= sk.rc ** 2)[..., None, None]
    r2 = torch.where(same, torch.ones_like(r2), r2)
    on = torch.diag(torch.tensor([sk.Es, sk.Ep, sk.Ep, sk.Ep], dtype=d.dtype, device=d.device))
    H = torch.where(same[..., None, None], on, _blocks(d, r2, sk.V, sk.d0)) * near
    S = torch.where(same[..., None, None], torch.eye(4, dtype=d.dtype, device=d.device), _blocks(d, r2, sk.Sv, sk.d0)) * near
    return (H, S) if storage is None else (_stored(H, storage), _stored(S, storage))


def _padded(mask):
    """Column indices of the set entries of each row, ascending, padded; and which are real."""
    n = mask.sum(1)
    M = int(n.max())
    idx = torch.sort(mask.to(torch.int8), dim=1, descending=True, stable=True).indices[:, :M]
    return idx, torch.arange(M, device=mask.device)[None] < n[:, None]


def _columns(case, pos, box, atoms, s_only=False):
    """Yields per chunk of atoms: levels, weights, V on the pattern rows and row j of V (or s_j), and the pattern."""
    sk = LATTICE[case["lattice"]][2]
    p, nu = case["p"], case["p"] + case["q"]
    B = max(4, int(64 * (160.0 / (4.2 * case["R"] ** 3 * 0.1763)) ** 2 * min(1.0, 40.0 / nu)))
    for c0 in range(0, len(atoms), B):
        at = atoms[c0:c0 + B]
        d = _image(pos[None] - pos[at][:, None], box)
        r2 = (d * d).sum(-1)
        near = r2 <= sk.rc ** 2
        cl, real = _padded(r2 <= case["R"] ** 2)
        b, M = cl.shape
        X = pos[cl]
        same = torch.eye(M, dtype=torch.bool, device=pos.device)[None].expand(b, M, M)
        H, S = _pair_blocks(_image(X[:, None] - X[:, :, None], box), same, sk, case["storage"])
        on = (real[:, :, None] & real[:, None, :])[..., None, None]
        eye = torch.eye(4, dtype=H.dtype, device=H.device) * (same & ~real[:, :, None])[..., None, None]
        H = (H * on).transpose(2, 3).reshape(b, 4 * M, 4 * M)
        S = (S * on + eye).transpose(2, 3).reshape(b, 4 * M, 4 * M)
        t0 = (cl == at[:, None]).int().argmax(1)
        j = 4 * t0[:, None] + torch.arange(4, device=pos.device)[None]                     # [b, 4] row of column c
        e = torch.zeros((b, 4 * M, 4), dtype=H.dtype, device=H.device).scatter_(1, j[:, None], 1.0)
        x, r = torch.zeros_like(e), e.clone()                                              # CG, to rounding
        g, rr = r.clone(), (r * r).sum(1, keepdim=True)
        for _ in range(200):
            Sg = S @ g
            al = rr / (g * Sg).sum(1, keepdim=True).clamp_min(1e-300)
            x, r = x + al * g, r - al * Sg
            new = (r * r).sum(1, keepdim=True)
            if float(new.max()) < 1e-31:
                break
            g, rr = r + new / rr.clamp_min(1e-300) * g, new
        if s_only:
            yield SimpleNamespace(at=at, s=x, cl=cl, real=real)
            continue
        U, SU, HU = (torch.empty((b, nu, 4 * M, 4), dtype=H.dtype, device=H.device) for _ in range(3))
        l = e
        for n in range(nu):
            for _ in range(3):
                if n:
                    l = l - torch.einsum("bnmc,bnc->bmc", U[:, :n], torch.einsum("bnmc,bmc->bnc", SU[:, :n], l))
            Sl = S @ l
            inv = 1.0 / torch.sqrt((l * Sl).sum(1, keepdim=True))
            U[:, n], SU[:, n] = l * inv, Sl * inv
            HU[:, n] = H @ U[:, n]
            l = x if n + 1 == p else HU[:, n]
        Hr, Sr = (torch.einsum("bnmc,bkmc->bcnk", U, V) for V in (HU, SU))
        L = torch.linalg.cholesky(0.5 * (Sr + Sr.mT))
        A = torch.linalg.solve_triangular(L, 0.5 * (Hr + Hr.mT), upper=False)
        A = torch.linalg.solve_triangular(L, A.mT, upper=False)
        A = 0.5 * (A + A.mT)
        eps, Y = torch.linalg.eigh(A.cpu() if nu > 32 else A)
        eps, Y = eps.to(A.device), Y.to(A.device)
        C = torch.linalg.solve_triangular(L.mT, Y, upper=True)                             # [b, c, nu, alpha]
        row = lambda T: torch.gather(T, 2, j[:, None, None].expand(b, nu, 1, 4))[:, :, 0]   # noqa: E731  [b, nu, c]
        vj = torch.einsum("bnc,bcna->bca", row(U), C)
        w = vj * torch.einsum("bnc,bcna->bca", row(SU), C)
        nb, ok = _padded(near)                                                             # pattern atoms
        hit = (nb[:, :, None] == cl[:, None]) & real[:, None]
        loc, inside = hit.int().argmax(2), hit.any(2) & ok
        rows = (4 * loc[:, :, None] + torch.arange(4, device=pos.device)).reshape(b, 1, -1, 1).expand(b, nu, -1, 4)
        Ur = torch.gather(U, 2, rows).reshape(b, nu, nb.shape[1], 4, 4)                    # [b, n, k, r, c]
        V = torch.einsum("bnkrc,bcna->bkcra", Ur, C) * inside[:, :, None, None, None]
        Hrow = _pair_blocks(_image(pos[nb] - pos[at][:, None], box), nb == at[:, None], sk, case["storage"])[0]
        yield SimpleNamespace(at=at, eps=eps, w=w, V=V, vj=vj, nb=nb, ok=ok, H=Hrow)


def _fermi(x, mu, kT):
    return 0.5 * (1.0 - torch.tanh((x - mu) / (2.0 * kT)))


def _filled(case, n, v):
    """The pattern's blocks [blocks, 4, 4, ...] of n atoms in a zeroed buffer as prepare() makes it."""
    out = v.new_zeros((_capacity(case["lattice"], n) * 16,) + tuple(v.shape[3:]))
    out[:v.shape[0] * 16] = v.reshape((-1,) + tuple(v.shape[3:]))
    return out


def _weighted(cols, f):
    """sum_alpha f(eps_alpha) V_i V_j on the pattern, [blocks, 4, 4] in order."""
    return torch.cat([torch.einsum("bkcra,bca->bkcr", c.V, f(c.eps) * c.vj)[c.ok] for c in cols])


def _chemical_potential(cols, n_el, kT):
    eps, w = (torch.cat([getattr(c, k).reshape(-1) for c in cols]) for k in ("eps", "w"))
    lo, hi = float(eps.min()) - 40 * kT, float(eps.max()) + 40 * kT
    while hi - lo > 1e-12:
        mid = 0.5 * (lo + hi)
        if 2.0 * float((_fermi(eps, mid, kT) * w).sum()) < n_el:
            lo = mid
        else:
            hi = mid
    mu = 0.5 * (lo + hi)
    return mu, 2.0 * float((_fermi(eps, mu, kT) * w).sum())


def _exact_forces(cols, pos, box, sk, rho, pi):
    """-d/dR of 2 Tr[rho H(R)] - 2 Tr[pi S(R)] with rho and pi held fixed, over the columns' pattern entries."""
    a = torch.cat([c.at[:, None].expand_as(c.nb)[c.ok] for c in cols])
    b = torch.cat([c.nb[c.ok] for c in cols])
    off = a != b
    a, b, rho, pi = a[off], b[off], rho[off], pi[off]
    R = pos.clone().requires_grad_(True)
    d = _image(R[b] - R[a], box)
    r2 = (d * d).sum(-1)
    e = 2.0 * ((rho * _blocks(d, r2, sk.V, sk.d0)).sum() - (pi * _blocks(d, r2, sk.Sv, sk.d0)).sum())
    return -torch.autograd.grad(e, R)[0]


def _exact_features(at, pos, box):
    """Inputs and patch of the learned start: neighbours by (distance, id)."""
    n = len(at)
    X = torch.zeros((n, 4, MLP_IN), dtype=torch.float64, device=pos.device)
    patch = torch.empty((n, PATCH), dtype=torch.int64, device=pos.device)
    for c0 in range(0, n, 512):
        a = at[c0:c0 + 512]
        d = _image(pos[None] - pos[a][:, None], box)
        r = torch.sqrt((d * d).sum(-1)).scatter_(1, a[:, None], -1.0)
        r, idx = torch.sort(r, dim=1, stable=True)
        patch[c0:c0 + 512] = idx[:, :PATCH]
        r, idx = r[:, 1:33], idx[:, 1:33]
        d = torch.gather(d, 1, idx[:, :, None].expand(-1, -1, 3))
        g = torch.cat([r[..., None], d / r[..., None]], -1) * (r <= 3.0)[..., None]
        X[c0:c0 + 512, :, :128] = g.reshape(len(a), 1, 128)
    X[:, :, 128:] = torch.eye(4, dtype=torch.float64, device=pos.device)
    return X.reshape(4 * n, MLP_IN), patch


def _exact_spmv(case, pos, box, x):
    """Row by row from the lattice's own cells: a site's neighbours lie in the 27 cells around it."""
    n = case["cells"]
    y = torch.empty_like(x)
    k = x.shape[1]
    ids = torch.arange(len(pos), device=pos.device)
    if len(torch.unique(torch.arange(-1, 2) % n)) < 3:
        raise ValueError("needs three cells per edge")
    o = torch.arange(-1, 2, device=pos.device)
    off = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    sk = DIAMOND
    for c0 in range(0, len(pos), 8192):
        a = ids[c0:c0 + 8192]
        cell = torch.stack([a // 8 // n // n, a // 8 // n % n, a // 8 % n], -1)
        nc = (cell[:, None] + off[None]) % n
        cand = (((nc[..., 0] * n + nc[..., 1]) * n + nc[..., 2]) * 8)[..., None] + torch.arange(8, device=pos.device)
        cand = cand.reshape(len(a), -1)
        d = _image(pos[cand] - pos[a][:, None], box)
        keep, ok = _padded((d * d).sum(-1) <= sk.rc ** 2)
        nb = torch.gather(cand, 1, keep)
        d = torch.gather(d, 1, keep[:, :, None].expand(-1, -1, 3))
        A = _pair_blocks(d, nb == a[:, None], sk, case["storage"])[case["which"]] * ok[..., None, None]
        y[4 * c0:4 * (c0 + len(a))] = torch.einsum("abij,abjk->aik", A, x.reshape(-1, 4, k)[nb]).reshape(-1, k)
    return y


def _exact_gradients(case, seed):
    """The network in FP64 on its BF16-rounded weights (the library's own initial values)."""
    s = prepare(case, seed)
    theta = torch.from_numpy(mka.mka_mlp_get_params(s.net, bf16_rounded=True)).double().cuda().requires_grad_(True)
    o, shapes = 0, []
    for rows, cols in ((MLP_HID, MLP_IN), (MLP_HID, MLP_HID), (MLP_OUT, MLP_HID)):
        shapes.append((theta[o:o + rows * cols].reshape(rows, cols), theta[o + rows * cols:o + rows * cols + rows]))
        o += rows * cols + rows
    h = s.X.double()
    for i, (W, b) in enumerate(shapes):
        h = h @ W.T + b
        h = torch.nn.functional.silu(h) if i < 2 else h
    loss = ((h - s.T.double()) ** 2).mean()
    return {"grad": torch.autograd.grad(loss, theta)[0], "loss": loss.detach().reshape(1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradients":
        return _exact_gradients(case, seed)
    lattice = case.get("lattice", "diamond")
    hpos, hbox = _positions(lattice, case["cells"], case["sigma"], seed)
    pos, box = torch.from_numpy(hpos).cuda(), torch.from_numpy(hbox).cuda()
    sk, kT = LATTICE[lattice][2:4]
    if kind == "spmv":
        dt = torch.float64 if case["x"] == "fp64" else torch.float32
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((4 * len(pos), case["k"]), generator=g, device="cuda", dtype=dt)
        return _exact_spmv(case, pos, box, x.double())
    atoms = torch.from_numpy(_selection(case, len(pos), seed)).cuda()
    if kind == "targets":
        X, patch = _exact_features(atoms, pos, box)
        Y, c0 = [], 0
        for c in _columns(case, pos, box, atoms, s_only=True):
            at = patch[c0:c0 + len(c.at)]
            c0 += len(c.at)
            hit = (at[:, :, None] == c.cl[:, None]) & c.real[:, None]
            rows = (4 * hit.int().argmax(2)[:, :, None] + torch.arange(4, device=pos.device)).reshape(len(at), -1, 1)
            y = torch.gather(c.s, 1, rows.expand(-1, -1, 4)) * hit.any(2).repeat_interleave(4, 1)[..., None]
            Y.append(y.transpose(1, 2).reshape(-1, MLP_OUT))
        return {"X": X, "Y": torch.cat(Y), "patch": patch.int()}
    mu0 = 1.98 if lattice == "diamond" else 0.9
    cols = list(_columns(case, pos, box, atoms))
    if kind == "levels":
        nu = case["p"] + case["q"]
        eps, w = (torch.cat([getattr(c, k) for c in cols]).reshape(-1, nu) for k in ("eps", "w"))
        out = {"eps": eps, "w": w, "nu_eff": None, "status": None}
        if case.get("energies"):
            E = torch.linspace(mu0 - 4.0, mu0 + 4.0, case["energies"], dtype=torch.float64, device="cuda")
            e, ww = eps.reshape(-1), w.reshape(-1)
            out["dos"] = torch.stack([(ww * 0.1 / ((x - e) ** 2 + 0.01)).sum() / math.pi for x in E])
        return out
    if kind == "response":
        z = complex(mu0, 0.2)
        G = torch.cat([torch.einsum("bkcra,bca->bkcr", c.V.to(torch.complex128), c.vj / (z - c.eps))[c.ok] for c in cols])
        rho = _weighted(cols, lambda x: _fermi(x, mu0, kT))
        pi = _weighted(cols, lambda x: _fermi(x, mu0, kT) * x)
        return {"G": _filled(case, len(atoms), torch.view_as_real(G)), "pi": _filled(case, len(atoms), pi),
                "forces": _exact_forces(cols, pos, box, sk, rho, pi)}
    mu, n_el = _chemical_potential(cols, 4.0 * len(atoms), kT)
    rho = _weighted(cols, lambda x: _fermi(x, mu, kT))
    e = 2.0 * float((rho * torch.cat([c.H[c.ok] for c in cols])).sum())
    out = {"rho": _filled(case, len(atoms), rho), "mu": mu, "e_band": e}
    if kind == "system":
        out["forces"] = _exact_forces(cols, pos, box, sk, rho, _weighted(cols, lambda x: _fermi(x, mu, kT) * x))
    else:
        out["n_electrons"] = n_el
    return out
