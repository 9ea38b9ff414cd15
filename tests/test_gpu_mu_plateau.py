"""mu where the electron count stands still over a range of mu: mka_find_mu and plans return the lowest mu with the asked
count, as the oracle's bisection does. Atoms without neighbours have one level a column (Es, Ep, Ep, Ep with weight 1),
so that the plateaus' counts are whole numbers: the gap's, full and empty bands. The lower edge is where the missing
electrons D = N exp(-(mu - e) / kT) round away. All f are 1 once D / N <= 2^-54, and a sum of depth d cannot be N before
D / N <= (d + 2) 2^-53: two orders of the sum, of depth 25 or less, put it up to kT ln(2 * 27) = 4 kT apart. And in a band,
where mu is unique: 1e-10."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import mka as om
from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    mka.load()
    return mka


def both(mka, s, atoms, p, q, n_electrons, kT):
    """mu of the result's levels and of a plan's, and the oracle's on the same levels."""
    res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, cg_tol=1e-13))
    lv = mka.mka_result_copy_levels(res, check=False)
    direct = mka.mka_find_mu(res, n_electrons, kT)
    mka.mka_result_destroy(res)
    plan = mka.mka_plan_create(s, len(atoms), mka.solve_params(p, q, cg_tol=1e-13))
    mka.mka_plan_run(plan, atoms, n_electrons, kT)
    planned = mka.mka_plan_scalars(plan)[0]
    mka.mka_plan_destroy(plan)
    return direct, planned, om.find_mu(lv["eps"], lv["w"], n_electrons, kT)


@pytest.mark.parametrize("kT", [0.01, 0.1])
@pytest.mark.parametrize("electrons", ["gap", "full", "empty"])
@pytest.mark.parametrize("n", [1, 300])
def test_lowest_mu_on_a_plateau(lib, n, electrons, kT):
    mka = lib
    pos = np.stack(np.unravel_index(np.arange(n), (8, 8, 8)), 1) * 5.0
    sk = replace(SK_CARBON_LIKE, rc=2.0)
    s = mka.mka_build_system(pos, np.full(3, 40.0), sk, "fp64", cluster_radius=2.0)
    try:
        atoms = np.arange(n, dtype=np.int64)
        ne = {"gap": 2.0 * n, "full": 8.0 * n, "empty": 0.0}[electrons]     # Es < Ep
        direct, planned, ref = both(mka, s, atoms, 1, 0, ne, kT)
        tol = 1e-10 if electrons == "empty" else 4 * kT  # the empty plateau's lower end is the bracket's
        assert abs(direct - ref) <= tol
        assert abs(planned - ref) <= tol
    finally:
        mka.mka_system_destroy(s)


def test_mu_inside_a_band(lib):
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 5)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=5.0)
    try:
        atoms = np.arange(40, dtype=np.int64)
        for per in (0.1, 2.3, 4.0, 7.9):
            direct, planned, ref = both(mka, s, atoms, 8, 8, per * len(atoms), 0.1)
            assert abs(direct - ref) <= 1e-10 and abs(planned - ref) <= 1e-10
    finally:
        mka.mka_system_destroy(s)
