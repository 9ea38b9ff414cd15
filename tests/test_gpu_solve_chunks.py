"""A direct solve that runs in several chunks (the reduced problems' buffer stays within 2 GiB): an atom listed in a full
chunk and again in the short last one, which by itself would take other kernels, has the same bits in both."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith,storage", [("fp64", "fp64"), ("mixed", "bf16")])
def test_copies_in_different_chunks(arith, storage):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    p, q = 50, 50
    per = 8 * (3 * 100 * 100 + 2 * 100) * 4                # bytes of an atom's reduced problems
    chunk = (2 << 30) // per // 8 * 8
    pos, box = lattice_positions("diamond", 3.567, 3, 0.08, 0.0, 23)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, storage, cluster_radius=5.0)
    try:
        n = chunk + 5
        atoms = np.arange(n, dtype=np.int64) % 8
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(p, q, arith=arith, cg_tol=1e-12 if arith == "fp64" else 1e-7,
                                                               keep_vectors=False))
        lv = mka.mka_result_copy_levels(res)
        mka.mka_result_destroy(res)
        for k in ("eps", "w", "nu_eff", "status"):
            x = lv[k].reshape(n, 4, -1)
            for a in range(8):
                assert (x[atoms == a] == x[a]).all(), (k, a)
    finally:
        mka.mka_system_destroy(s)


def test_copies_in_different_chunks_without_allocation():
    """The same for the allocation-free entry point, whose chunks follow from its fixed scratch."""
    from paper_1202_0098_gb300 import build, mka
    build.build()
    p, q = 5, 5
    pos, box = lattice_positions("diamond", 3.567, 3, 0.08, 0.0, 23)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=4.0)
    try:
        per = 8 + 8 * (3 * 100 + 20) * 4
        n = (64 << 20) // 2 // per + 40                     # more than the scratch's half holds, which a chunk fills
        atoms = np.arange(n, dtype=np.int64) % 8
        eps, w = (torch.full((4 * n, p + q), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
        ib = [torch.full((4 * n,), -1, dtype=torch.int32, device="cuda") for _ in range(3)]
        cap = int(mka.mka_cluster_sizes(s, atoms[:8]).max())
        mka.mka_solve_columns_static(s, atoms, p, q, 1e-13, 500, cap, eps.data_ptr(), w.data_ptr(), ib[0].data_ptr(),
                                     ib[1].data_ptr(), ib[2].data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        for k in (eps, w, *ib):
            x = k.cpu().numpy().reshape(n, 4, -1)
            for a in range(8):
                assert (x[atoms == a] == x[a]).all(), a
    finally:
        mka.mka_system_destroy(s)
