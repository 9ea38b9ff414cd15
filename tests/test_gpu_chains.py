"""The short-recurrence kernel (chains.cu) against the general one and the oracle, at the edges of its rule.

mka_solve_columns takes the short recurrences for subspaces up to nu = 48 on clusters of at least 6 nu rows;
mka_solve_columns_static always takes the general kernel. Both run the same inner CG and form the same
subspace, so levels and weights agree to the tolerance of the other FP64 parity tests (1e-10; the recurrences'
rounding enters like the Gram-Schmidt's). Sizes: both sides of nu = 48 and of m = 6 nu, odd nu, q = 0 and
p = 1, S = I (s_j drops out and the first chain continues), a cluster whose Krylov space closes early
(left to the general kernel), uneven clusters of which some are left over, CTA sizes of a plan.
The mixed form is held to the bars of the mixed parity test: 1e-6 in rho, 1e-5 eV/atom.
"""
from dataclasses import replace

import numpy as np
import pytest

from oracle import system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_CARBON_LIKE, SK_FCC_METAL, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
I_S = replace(SK_CARBON_LIKE, Sv=(0.0, 0.0, 0.0, 0.0))


@pytest.fixture(scope="module")
def lib():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    mka.load()
    return mka


def general_levels(mka, s, atoms, p, q):
    n, nu = 4 * len(atoms), p + q
    eps, w = (torch.full((n, nu), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    ib = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for _ in range(3)]
    cap = int(mka.mka_cluster_sizes(s, atoms).max())
    mka.mka_solve_columns_static(s, atoms, p, q, 1e-13, 500, cap, eps.data_ptr(), w.data_ptr(), ib[0].data_ptr(),
                                 ib[1].data_ptr(), ib[2].data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return eps.cpu().numpy(), w.cpu().numpy(), ib[0].cpu().numpy(), ib[1].cpu().numpy()


# (lattice, cells, sigma, vacancy, sk, R, p, q, storage)
FORMS = [
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.3, 24, 24, "fp64"),     # nu = 48, the largest
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.3, 25, 24, "fp64"),     # nu = 49: the general kernel on both sides
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 12, 7, "fp32"),
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 7, 12, "bf16"),
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 19, 0, "fp64"),      # one chain, odd
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 1, 1, "fp64"),
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 1, 0, "fp64"),
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 5.0, 1, 9, "fp64"),
    ("diamond", 3, 0.07, 0.0, I_S, 5.0, 8, 8, "fp64"),                  # S = I
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 2.8, 6, 5, "fp64"),       # m = 68, 6 nu = 66: some atoms on each side
    ("diamond", 3, 0.08, 0.0, SK_CARBON_LIKE, 2.0, 2, 1, "fp64"),       # five-atom clusters
    ("fcc", 4, 0.08, 0.2, SK_FCC_METAL, 6.0, 10, 10, "fp64"),           # uneven, 6 nu = 120 amid the sizes
]


@pytest.mark.parametrize("form", FORMS, ids=lambda f: f"{f[0]}-R{f[5]}-p{f[6]}q{f[7]}-{f[8]}")
def test_chains_match_the_general_kernel(lib, form):
    mka = lib
    lat, cells, sig, vac, sk, R, p, q, storage = form
    pos, box = lattice_positions(lat, 3.567 if lat == "diamond" else 4.0, cells, sig, vac, 31)
    atoms = np.arange(0, len(pos), 7, dtype=np.int64)
    s = mka.mka_build_system(pos, box, sk, storage, cluster_radius=R)
    try:
        eps, w, nu_eff, it = general_levels(mka, s, atoms, p, q)
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, cg_tol=1e-13, keep_vectors=True))
        lv = mka.mka_result_copy_levels(res)
        mka.mka_result_destroy(res)
        np.testing.assert_array_equal(lv["nu_eff"], nu_eff)
        np.testing.assert_array_equal(lv["cg_iters"], it)
        np.testing.assert_allclose(lv["eps"], eps, rtol=0, atol=TOL)
        np.testing.assert_allclose(lv["w"], w, rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)


@pytest.mark.parametrize("threads", [128, 256, 512])
@pytest.mark.parametrize("storage,R,p,q", [("bf16", 5.0, 11, 8), ("fp32", 5.3, 20, 17), ("fp64", 5.0, 13, 0)])
def test_chains_mixed_form(lib, storage, R, p, q, threads):
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 17)
    atoms = np.array([0, 31, 77, 150, 215], dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, SK_CARBON_LIKE, R, atoms, p, q, storage="fp32" if storage == "fp64" else storage)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, storage, cluster_radius=R)
    try:
        plan = mka.mka_plan_create(s, 8, mka.solve_params(p, q, arith="mixed", cg_tol=1e-7), mka.tuning(threads, 0, True))
        nb = sum(len(r.neigh) for r in ores)
        rho = torch.zeros(nb * 16, dtype=torch.float64, device="cuda")
        mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1, rho.data_ptr())
        mu, e, _ = mka.mka_plan_scalars(plan)
        mka.mka_plan_destroy(plan)
        orho, oe, _ = osys.density(ores, mu, 0.1)
        assert np.abs(rho.cpu().numpy().reshape(-1, 4, 4) - np.concatenate(orho)).max() <= 1e-6
        assert abs(e - oe) / len(atoms) <= 1e-5
    finally:
        mka.mka_system_destroy(s)


def test_two_plans_of_different_cluster_sizes(lib):
    """Plans of two systems captured in turn: the second one's smaller clusters leave the first one's launches valid."""
    mka = lib
    systems, plans = [], []
    atoms = np.arange(24, dtype=np.int64)
    for R in (6.0, 5.0):
        pos, box = lattice_positions("diamond", 3.567, 4, 0.08, 0.0, 9)
        systems.append(mka.mka_build_system(pos, box, SK_CARBON_LIKE, "bf16", cluster_radius=R))
        plans.append(mka.mka_plan_create(systems[-1], len(atoms), mka.solve_params(8, 8, arith="mixed", cg_tol=1e-7)))
    for plan in plans:
        mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1)
        mu, _, n = mka.mka_plan_scalars(plan)
        assert abs(n - 4.0 * len(atoms)) < 1e-6
    for plan in plans:
        mka.mka_plan_destroy(plan)
    for s in systems:
        mka.mka_system_destroy(s)
