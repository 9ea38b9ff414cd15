"""The short-recurrence kernel itself, in selections too large for a CTA per column, at the edges of its rule (the forms of
test_gpu_chains.py: both sides of nu = 48 and of m = 6 nu, q = 0, p = 1, S = I, uneven clusters): FP64 levels and
weights against the general kernel's within 1e-10, and the kernels that ran, by their number. And the mixed form with
one chain shorter than eight vectors, whose staged S_r products end in a part of the lanes' vectors (gram_s): rho
within 1e-6 of the oracle's and the band energy within 1e-5 eV an atom, as in the mixed parity test."""
import numpy as np
import pytest

from oracle import system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_CARBON_LIKE, lattice_positions
from tests.test_gpu_chains import FORMS, general_levels, lib  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("form", FORMS, ids=lambda f: f"{f[0]}-R{f[5]}-p{f[6]}q{f[7]}-{f[8]}")
def test_chains_in_large_selections(lib, form):  # noqa: F811
    mka = lib
    lat, cells, sig, vac, sk, R, p, q, storage = form
    nu = p + q
    pos, box = lattice_positions(lat, 3.567 if lat == "diamond" else 4.0, cells, sig, vac, 31)
    atoms = np.arange(0, len(pos), 7, dtype=np.int64)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = 2 * sms // len(atoms) + 1
    s = mka.mka_build_system(pos, box, sk, storage, cluster_radius=R)
    try:
        eps, w, nu_eff, it = general_levels(mka, s, atoms, p, q)
        recurrences = nu <= 48 and 4 * int(mka.mka_cluster_sizes(s, atoms).max()) >= 6 * nu
        n0 = mka.mka_kernel_launches()
        res = mka.mka_solve_columns(s, np.tile(atoms, copies), mka.solve_params(p, q, cg_tol=1e-13, keep_vectors=True))
        # cluster sizes, the column kernels, the reduced problems (teams from nu = 5 on)
        assert mka.mka_kernel_launches() - n0 == 1 + (2 if recurrences else 1) + (3 if nu >= 5 else 1)
        lv = mka.mka_result_copy_levels(res)
        mka.mka_result_destroy(res)
        np.testing.assert_array_equal(lv["nu_eff"], np.tile(nu_eff, copies))
        np.testing.assert_array_equal(lv["cg_iters"], np.tile(it, copies))
        np.testing.assert_allclose(lv["eps"], np.tile(eps, (copies, 1)), rtol=0, atol=TOL)
        np.testing.assert_allclose(lv["w"], np.tile(w, (copies, 1)), rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)


@pytest.mark.parametrize("R,p,q", [(6.0, 24, 1), (6.0, 20, 5), (5.0, 15, 2), (4.4, 8, 1), (4.4, 1, 1), (4.4, 2, 7), (5.0, 1, 0),
                                   (5.0, 3, 14), (5.4, 41, 1)])
def test_mixed_form_with_a_short_chain(lib, R, p, q):  # noqa: F811
    mka = lib
    pos, box = lattice_positions("diamond", 3.567, 4, 0.1, 0.0, 17)
    atoms = np.array([0, 31, 77, 150, 215, 402], dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, SK_CARBON_LIKE, R, atoms, p, q, storage="bf16")
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "bf16", cluster_radius=R)
    try:
        assert 4 * int(mka.mka_cluster_sizes(s, atoms).min()) >= 6 * (p + q)
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, arith="mixed", cg_tol=1e-7))
        nb = mka.mka_result_info(res)["n_blocks"]
        rho = torch.full((nb * 16,), float("nan"), dtype=torch.float64, device="cuda")
        mu, kT = 1.9, 0.1
        e, _ = mka.mka_density_energy(s, res, mu, kT, rho.data_ptr())
        mka.mka_result_destroy(res)
        orho, oe, _ = osys.density(ores, mu, kT)
        assert np.abs(rho.cpu().numpy().reshape(-1, 4, 4) - np.concatenate(orho)).max() <= 1e-6
        assert abs(e - oe) / len(atoms) <= 1e-5
    finally:
        mka.mka_system_destroy(s)
