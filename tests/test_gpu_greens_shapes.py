"""The Green's function at the subspace sizes where the products with kept vectors change form (odd, smallest, largest, rows
of more than 32 blocks) against the oracle, every entry written; the tolerance of the parity test."""
import numpy as np
import pytest

from oracle import system as osys
from oracle.parallel import solve_atoms_parallel
from synth import SK_CARBON_LIKE, SK_FCC_METAL, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,a,cells,R,p,q", [("diamond", 3.567, 4, 5.0, 1, 0), ("diamond", 3.567, 4, 5.0, 1, 1),
                                                   ("diamond", 3.567, 4, 5.0, 4, 3), ("diamond", 3.567, 4, 5.0, 15, 15),
                                                   ("diamond", 3.567, 4, 6.5, 160, 160), ("fcc", 2.6, 5, 4.0, 5, 5)])
def test_greens(lattice, a, cells, R, p, q):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    sk = SK_CARBON_LIKE if lattice == "diamond" else SK_FCC_METAL
    pos, box = lattice_positions(lattice, a, cells, 0.06, 0.0, 13)
    atoms = np.array([9, 100], dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, sk, R, atoms, p, q)
    s = mka.mka_build_system(pos, box, sk, "fp64", cluster_radius=R)
    try:
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, cg_tol=1e-13))
        nb = mka.mka_result_info(res)["n_blocks"]
        G = torch.full((nb * 16, 2), float("nan"), dtype=torch.float64, device="cuda")
        z = complex(1.9, 0.2)
        mka.mka_greens(s, res, z, G.data_ptr())
        got = torch.view_as_complex(G).cpu().numpy().reshape(nb, 4, 4)
        mka.mka_result_destroy(res)
        np.testing.assert_allclose(got, np.concatenate(osys.greens(ores, z)), rtol=0, atol=1e-9)
    finally:
        mka.mka_system_destroy(s)
