"""The forms of the batched reduced problems against the oracle: a warp per column, teams of 8, 16 and 32 lanes, one
lane per column, on both sides of the subspace sizes and column counts between them (nu = 4, 5, 32, 33, 64, 65 and
nu = 160, 161; 2,048 columns; columns of several sizes in one warp). FP64 tolerance of the other parity tests."""
import numpy as np
import pytest

from oracle import system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_CARBON_LIKE, SK_FCC_METAL, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def lib():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    mka.load()
    return mka


def levels(mka, s, atoms, p, q):
    res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, cg_tol=1e-13))
    try:
        return mka.mka_result_copy_levels(res)
    finally:
        mka.mka_result_destroy(res)


@pytest.mark.parametrize("p,q", [(2, 2), (3, 2), (16, 16), (17, 16), (32, 32), (33, 32), (80, 80), (81, 80)])
def test_subspace_sizes(lib, p, q):
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 4, 0.08, 0.0, 19)
    R = 6.0 if p > 40 else 5.0
    atoms = np.array([3, 200, 401], dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, SK_CARBON_LIKE, R, atoms, p, q)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=R)
    try:
        lv = levels(mka, s, atoms, p, q)
        oe, ow = osys.stack_eps_w(ores)
        np.testing.assert_array_equal(lv["nu_eff"], [c.nu_eff for r in ores for c in r.data])
        np.testing.assert_allclose(lv["eps"], oe, rtol=0, atol=TOL)
        np.testing.assert_allclose(lv["w"], ow, rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)


def test_column_counts_agree(lib):
    """The same atoms within selections of 3 atoms, 513 (just above 2,048 columns) and 10,241 (just above 40,960)."""
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 11, 0.1, 0.0, 23)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=4.0)
    try:
        few = levels(mka, s, np.array([5, 300, 512], dtype=np.int64), 8, 7)
        for n in (513, 10241):
            lv = levels(mka, s, np.arange(n, dtype=np.int64), 8, 7)
            rows = np.concatenate([np.arange(4 * a, 4 * a + 4) for a in (5, 300, 512)])
            np.testing.assert_allclose(lv["eps"][rows], few["eps"], rtol=0, atol=TOL)
            np.testing.assert_allclose(lv["w"][rows], few["w"], rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)


def test_subspaces_of_several_sizes(lib):
    """Clusters of 1 to about 13 atoms, many smaller than nu, so that the columns of a warp end their bases at
    different sizes: a warp per column (few columns) against teams of 8 and 16 lanes (the same columns in a selection
    above 2,048). Both run the same basis kernel, so nu_eff and status are equal and the levels agree to rounding."""
    mka = lib
    pos, box = lattice_positions("fcc", 4.0, 6, 0.05, 0.55, 4)
    p, q = 9, 8
    atoms = np.arange(len(pos), dtype=np.int64)
    pick = atoms[:: max(1, len(atoms) // 40)]
    s = mka.mka_build_system(pos, box, SK_FCC_METAL, "fp64", cluster_radius=3.2)
    try:
        few = levels(mka, s, pick, p, q)
        ne = few["nu_eff"]
        assert len(set(ne)) > 3
        copies = 2 + 2100 // (4 * len(atoms))
        many = levels(mka, s, np.concatenate([atoms] * copies), p, q)
        rows = np.concatenate([np.arange(4 * a, 4 * a + 4) for a in pick])
        np.testing.assert_array_equal(many["nu_eff"][rows], ne)
        np.testing.assert_array_equal(many["status"][rows], few["status"])
        np.testing.assert_allclose(many["eps"][rows], few["eps"], rtol=0, atol=TOL)
        # weights of levels closer than 1e-8 eV are not unique one by one: summed over each group
        for c in range(len(ne)):
            a = 0
            while a < ne[c]:
                b = a + 1
                while b < ne[c] and few["eps"][c, b] - few["eps"][c, b - 1] < 1e-8:
                    b += 1
                assert abs(many["w"][rows[c], a:b].sum() - few["w"][c, a:b].sum()) <= TOL
                a = b
    finally:
        mka.mka_system_destroy(s)


@pytest.mark.parametrize("p,q", [(8, 7), (10, 10)])
def test_degenerate_levels(lib, p, q):
    """A perfect crystal: the three p columns of an atom have the same levels, and a column's own come close together.
    Few columns (bisection) against the same in a selection above 2,048 (QL)."""
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 5, 0.0, 0.0, 1)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=5.0)
    try:
        few = levels(mka, s, np.array([7], dtype=np.int64), p, q)
        many = levels(mka, s, np.arange(600, dtype=np.int64), p, q)
        np.testing.assert_array_equal(many["nu_eff"][28:32], few["nu_eff"])
        np.testing.assert_allclose(many["eps"][28:32], few["eps"], rtol=0, atol=TOL)
        for c in range(4):      # weights of levels closer than the tolerance may mix: compare their running sums
            a, b = np.cumsum(many["w"][28 + c]), np.cumsum(few["w"][c])
            apart = np.append(np.diff(few["eps"][c]) > 1e-6, True)
            np.testing.assert_allclose(a[apart], b[apart], rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)
