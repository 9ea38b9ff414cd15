"""A CTA per column (few atoms) against the kernels that take an atom's four columns together (the same atoms within a
selection beyond the change at 3/4 or 3/2 of the chip's SMs): levels, weights and rho of the FP64 form, over subspaces
below and above the short recurrences' limit, without a second chain, all value types; and against the oracle through
the parity tests, whose selections are small. FP64 tolerance of those tests."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("p,q,storage", [(15, 15, "fp64"), (15, 15, "bf16"), (9, 0, "fp32"), (1, 1, "fp64"), (24, 25, "fp64"),
                                         (40, 30, "fp32")])
def test_few_atoms_agree_with_many(p, q, storage):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, 5, 0.08, 0.0, 31)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, storage, cluster_radius=5.0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prm = mka.solve_params(p, q, cg_tol=1e-13)
    got = []
    try:
        few = np.array([700, 3, 41], dtype=np.int64)
        many = np.concatenate([few, np.arange(100, 100 + 2 * sms, dtype=np.int64)])
        info = mka.mka_system_copy_bsr(s, values=False)
        blocks = np.diff(info["row_ptr"])
        for atoms in (few, many):
            res = mka.mka_solve_columns(s, atoms, prm)
            try:
                lv = mka.mka_result_copy_levels(res)
                rho = torch.zeros(int(blocks[atoms].sum()) * 16, dtype=torch.float64, device="cuda")
                mka.mka_density_energy(s, res, 1.9, 0.1, rho.data_ptr())
                got.append((lv, rho.cpu().numpy()))
            finally:
                mka.mka_result_destroy(res)
        (a, ra), (b, rb) = got
        np.testing.assert_array_equal(a["nu_eff"], b["nu_eff"][:12])
        np.testing.assert_array_equal(a["status"], b["status"][:12])
        np.testing.assert_allclose(a["eps"], b["eps"][:12], rtol=0, atol=TOL)
        np.testing.assert_allclose(a["w"], b["w"][:12], rtol=0, atol=TOL)
        np.testing.assert_allclose(ra, rb[:len(ra)], rtol=0, atol=TOL)
    finally:
        mka.mka_system_destroy(s)
