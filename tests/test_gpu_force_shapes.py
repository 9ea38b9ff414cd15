"""Forces, pi and G where the kernels for kept vectors change form: odd subspaces (rows of U read one entry at a time),
the smallest, and the largest there is (shared memory), against the oracle with the FP64 tolerances of the force and
parity tests. mka_forces needs rows of up to 32 blocks for one pass: the dense lattice has more."""
import numpy as np
import pytest

from oracle import forces as ofo, system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_CARBON_LIKE, SK_FCC_METAL, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("lattice,a,cells,R,p,q", [("diamond", 3.567, 4, 5.0, 1, 1), ("diamond", 3.567, 4, 5.0, 4, 3),
                                                   ("diamond", 3.567, 4, 6.5, 160, 160), ("fcc", 2.6, 5, 4.0, 5, 5)])
def test_forces_and_pi(lattice, a, cells, R, p, q):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    sk = SK_CARBON_LIKE if lattice == "diamond" else SK_FCC_METAL
    pos, box = lattice_positions(lattice, a, cells, 0.06, 0.0, 13)
    atoms = np.array([9, 100], dtype=np.int64)
    mu, kT = 1.9, 0.1
    ores = solve_atoms_parallel(pos, box, sk, R, atoms, p, q)
    orho, _, _ = osys.density(ores, mu, kT)
    opi = ofo.energy_density(ores, mu, kT)
    oF = ofo.forces(pos, box, sk, ores, orho, opi)
    s = mka.mka_build_system(pos, box, sk, "fp64", cluster_radius=R)
    try:
        if lattice == "fcc":
            assert np.diff(mka.mka_system_copy_bsr(s, values=False)["row_ptr"]).max() > 32
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, cg_tol=1e-13))
        nb = mka.mka_result_info(res)["n_blocks"]
        pi = torch.empty(nb * 16, dtype=torch.float64, device="cuda")
        F = torch.zeros(pos.shape[0] * 3, dtype=torch.float64, device="cuda")
        mka.mka_forces(s, res, mu, kT, pi.data_ptr(), F.data_ptr())
        rho = torch.empty(nb * 16, dtype=torch.float64, device="cuda")
        mka.mka_density_energy(s, res, mu, kT, rho.data_ptr())
        G = torch.zeros(nb * 16, 2, dtype=torch.float64, device="cuda")
        mka.mka_greens(s, res, complex(mu, 0.2), G.data_ptr())
        torch.cuda.synchronize()
        np.testing.assert_allclose(rho.cpu().numpy().reshape(nb, 4, 4), np.concatenate(orho), rtol=0, atol=TOL)
        np.testing.assert_allclose(pi.cpu().numpy().reshape(nb, 4, 4), np.concatenate(opi), rtol=0, atol=TOL)
        np.testing.assert_allclose(F.cpu().numpy().reshape(-1, 3), oF, rtol=0, atol=TOL)
        assert torch.isfinite(G).all()
        mka.mka_result_destroy(res)
    finally:
        mka.mka_system_destroy(s)
