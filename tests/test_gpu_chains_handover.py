"""Atoms the short recurrences hand over, and those they just keep (chains.cu).

An atom whose recurrence vectors overlap the start vector e_j by more than 1e-3 goes to the general kernel; below that
the Gram matrices have to make good the lost orthogonality. fcc clusters of m >= 6 nu rows with a short first chain
have many of both, which the recurrences in numpy show here before the call. The selection is beyond the size that
runs a CTA per column, so that the short recurrences see every atom, and a CTA meets kept and handed-over atoms in turn.
Levels and weights against the general kernel's (mka_solve_columns_static) with the FP64 parity tolerance, 1e-10;
the mixed form's rho against the oracle's with its own, 1e-6."""
import numpy as np
import pytest

from oracle import mka as om, sk as osk, system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_FCC_METAL, lattice_positions
from tests.test_chains_math import chains
from tests.test_gpu_chains import general_levels, lib  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


def overlaps(pos, box, R, atoms, p, q):
    """Largest overlap of an atom's recurrence vectors with their column's e_j, and the cluster's rows."""
    out = []
    for a in atoms:
        cl = osk.cluster_atoms(pos, box, int(a), R)
        H, S = osk.cluster_matrices(pos, box, cl, SK_FCC_METAL)
        t = int(np.searchsorted(cl, a))
        x = 0.0
        for j in range(4 * t, 4 * t + 4):
            s, _ = om.cg(S, np.eye(len(H))[j])
            x = max(x, np.abs(chains(H, S, j, s, p, q)[0][j, 1:]).max())
        out.append((len(H), x))
    return np.array(out)


@pytest.mark.parametrize("R,p,q", [(7.0, 10, 34), (7.6, 10, 38)])
def test_kept_and_handed_over_atoms(lib, R, p, q):  # noqa: F811
    mka = lib
    pos, box = lattice_positions("fcc", 4.0, 4, 0.08, 0.2, 31)
    atoms = np.arange(0, len(pos), 7, dtype=np.int64)
    ov = overlaps(pos, box, R, atoms, p, q)
    ov = ov[ov[:, 0] >= 6 * (p + q)][:, 1]
    assert (ov > 2e-3).sum() >= 2 and ((ov > 1e-5) & (ov < 5e-4)).sum() >= 5
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = 2 * sms // len(atoms) + 1
    s = mka.mka_build_system(pos, box, SK_FCC_METAL, "fp64", cluster_radius=R)
    try:
        eps, w, nu_eff, it = general_levels(mka, s, atoms, p, q)
        n0 = mka.mka_kernel_launches()
        res = mka.mka_solve_columns(s, np.tile(atoms, copies), mka.solve_params(p, q, cg_tol=1e-13))
        assert mka.mka_kernel_launches() - n0 == 1 + 2 + 3     # cluster sizes, both column kernels, reduced problems
        lv = mka.mka_result_copy_levels(res)
        mka.mka_result_destroy(res)
        np.testing.assert_array_equal(lv["nu_eff"], np.tile(nu_eff, copies))
        np.testing.assert_array_equal(lv["cg_iters"], np.tile(it, copies))
        np.testing.assert_allclose(lv["eps"], np.tile(eps, (copies, 1)), rtol=0, atol=TOL)
        np.testing.assert_allclose(lv["w"], np.tile(w, (copies, 1)), rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)


@pytest.mark.parametrize("threads", [128, 256, 512])
def test_kept_and_handed_over_atoms_in_the_mixed_form(lib, threads):  # noqa: F811
    mka = lib
    R, p, q = 7.0, 10, 34
    pos, box = lattice_positions("fcc", 4.0, 4, 0.08, 0.2, 31)
    pick = np.arange(0, len(pos), 14, dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, SK_FCC_METAL, R, pick, p, q, storage="fp32")
    atoms = np.tile(pick, 40)
    s = mka.mka_build_system(pos, box, SK_FCC_METAL, "fp32", cluster_radius=R)
    try:
        plan = mka.mka_plan_create(s, len(atoms), mka.solve_params(p, q, arith="mixed", cg_tol=1e-7),
                                   mka.tuning(threads, 0, True))
        nb = sum(len(r.neigh) for r in ores)
        rho = torch.zeros(40, nb * 16, dtype=torch.float64, device="cuda")
        mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1, rho.data_ptr())
        mu, _, _ = mka.mka_plan_scalars(plan)
        mka.mka_plan_destroy(plan)
        orho = np.concatenate(osys.density(ores, mu, 0.1)[0])
        assert np.abs(rho.cpu().numpy().reshape(40, -1, 4, 4) - orho).max() <= 1e-6
    finally:
        mka.mka_system_destroy(s)
