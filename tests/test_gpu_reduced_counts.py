"""Every change of form of the batched reduced problems with the number of columns (reduced_rule.cuh), one atom on either
side of it: the same atoms' levels and weights as in a selection of three atoms, FP64 tolerance of the parity tests."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
PICK = np.array([5, 100, 177], dtype=np.int64)


@pytest.fixture(scope="module")
def system():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, 11, 0.1, 0.0, 23)
    out = {R: mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=R) for R in (4.0, 5.0)}
    yield mka, out
    for s in out.values():
        mka.mka_system_destroy(s)


@pytest.mark.parametrize("p,q,edges", [(3, 2, (192, 1024)), (4, 4, (192, 1536)), (8, 8, (512, 3072)), (13, 11, (6144,)),
                                       (17, 16, (512, 4096)), (21, 20, (512, 4096)), (33, 32, (512, 3072)),
                                       (57, 56, (2560,)), (65, 64, (2048,))])
def test_columns_on_both_sides(system, p, q, edges):
    mka, systems = system
    s = systems[4.0 if p + q <= 41 else 5.0]
    prm = mka.solve_params(p, q, cg_tol=1e-13, keep_vectors=False)

    def levels(atoms):
        res = mka.mka_solve_columns(s, atoms, prm)
        try:
            return mka.mka_result_copy_levels(res)
        finally:
            mka.mka_result_destroy(res)

    few = levels(PICK)
    rows = np.concatenate([np.arange(4 * a, 4 * a + 4) for a in PICK])
    for n in [m for e in edges for m in (e, e + 1)]:
        lv = levels(np.arange(n, dtype=np.int64))
        np.testing.assert_array_equal(lv["status"][rows], few["status"])
        np.testing.assert_allclose(lv["eps"][rows], few["eps"], rtol=0, atol=TOL)
        np.testing.assert_allclose(lv["w"][rows], few["w"], rtol=0, atol=TOL)
