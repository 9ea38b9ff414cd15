"""Selections that the short recurrences mostly leave over (a perfect crystal, whose Krylov spaces close by symmetry): a
plan drops them after its trial, and a direct solve of many atoms after its first wave; with disorder both go on with
them. Which kernels ran is seen by their number; levels against the general kernel's, FP64 tolerance."""
import numpy as np
import pytest

from synth import SK_FCC_METAL, lattice_positions
from tests.test_gpu_chains import general_levels, lib  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [0.0, 0.08])
def test_plans_and_large_selections(lib, sigma):  # noqa: F811
    mka = lib
    p, q = 8, 8
    pos, box = lattice_positions("fcc", 4.0, 5, sigma, 0.0, 31)
    s = mka.mka_build_system(pos, box, SK_FCC_METAL, "fp64", cluster_radius=7.0)
    try:
        sample = np.arange(0, len(pos), 50, dtype=np.int64)
        eps, _, nu_eff, _ = general_levels(mka, s, sample, p, q)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        prm = mka.solve_params(p, q, cg_tol=1e-13)

        def check(lv):
            k = len(lv["eps"]) // len(eps)
            np.testing.assert_array_equal(lv["nu_eff"], np.tile(nu_eff, k))
            np.testing.assert_allclose(lv["eps"], np.tile(eps, (k, 1)), rtol=0, atol=1e-10)

        # beyond two waves at the most CTAs an SM holds (16): the first by itself, the judgement, the rest, the general kernel
        atoms = np.tile(sample, 2 * 16 * sms // len(sample) + 1)
        n0 = mka.mka_kernel_launches()
        res = mka.mka_solve_columns(s, atoms, prm)
        assert mka.mka_kernel_launches() - n0 in (1 + 4 + 3, 1 + 4 + 1)
        check(mka.mka_result_copy_levels(res))
        mka.mka_result_destroy(res)
        # a plan of 200 atoms: beyond the CTA-per-column form
        atoms = np.tile(sample, 200 // len(sample))
        plan = mka.mka_plan_create(s, len(atoms), prm)
        n0 = mka.mka_kernel_launches()
        mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1)
        kernels = mka.mka_kernel_launches() - n0
        check(mka.mka_result_copy_levels(mka.mka_plan_result(plan)))
        mka.mka_plan_destroy(plan)
        # the column kernels, three of the reduced problems, 68 of mu, four of the density
        assert kernels == (1 if sigma == 0.0 else 2) + 3 + 68 + 4
    finally:
        mka.mka_system_destroy(s)
