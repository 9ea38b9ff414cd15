"""A sweep's levels do not depend on how its atoms are batched: batches of a few atoms (which by themselves would take a CTA
per column and a warp per reduced problem), a middle size and the whole system at once give the same chunk sums, bit for
bit, and so do two processes' ranges with plans of their own sizes. Systems of up to 2,048 columns, up to 40,960 and of
subspaces on either side of nu = 32 and 64, FP64 and mixed form; rho of atoms solved again at mu likewise."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def sweep_sums(mka, s, prm, nu, a0, a1, sizes, window, kT):
    sw = mka.mka_sweep_create(s, a0, a1, nu, *window, 6, 1)
    plan = mka.mka_plan_create(s, max(sizes), prm)
    try:
        a, i = a0, 0
        while a < a1:
            n = min(sizes[i % len(sizes)], a1 - a)
            mka.mka_plan_run_sweep(plan, sw, np.arange(a, a + n, dtype=np.int64))
            a, i = a + n, i + 1
        nb = mka.mka_sweep_info(sw)["n_blocks"]
        rho = torch.full((nb * 16,), float("nan"), dtype=torch.float64, device="cuda")
        mka.mka_sweep_density(sw, plan, 1.9, kT, rho.data_ptr())
        torch.cuda.synchronize()
        return {**mka.mka_sweep_chunk_sums(sw, 1.9, kT, True, True), "rho": rho.cpu().numpy()}
    finally:
        mka.mka_plan_destroy(plan)
        mka.mka_sweep_destroy(sw)


@pytest.mark.parametrize("cells,p,q,arith,storage", [(3, 8, 7, "fp64", "fp64"), (4, 15, 15, "mixed", "bf16"),
                                                     (4, 20, 21, "fp64", "fp32"), (4, 33, 33, "fp64", "fp64"),
                                                     (6, 4, 4, "mixed", "fp32")])
@pytest.mark.parametrize("window", [(-4.5, 8.5), (30.0, 40.0)])     # kT = 0.05: mu inside it, and outside (all again)
def test_batches(cells, p, q, arith, storage, window):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, cells, 0.1, 0.0, 23)
    n, kT = len(pos), 0.05
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, storage, cluster_radius=5.0)
    prm = mka.solve_params(p, q, arith=arith, cg_tol=1e-13 if arith == "fp64" else 1e-7)
    try:
        whole = sweep_sums(mka, s, prm, p + q, 0, n, (n,), window, kT)
        assert np.isfinite(whole["rho"]).all()
        mixed = sweep_sums(mka, s, prm, p + q, 0, n, (1, 7, 50, 150), window, kT)
        half = n // 2
        lo = sweep_sums(mka, s, prm, p + q, 0, half, (60,), window, kT)
        hi = sweep_sums(mka, s, prm, p + q, half, n, (n,), window, kT)
        for k in ("count", "e_levels", "e_rho", "rho"):
            np.testing.assert_array_equal(mixed[k], whole[k])
            np.testing.assert_array_equal(np.concatenate([lo[k], hi[k]]), whole[k])
    finally:
        mka.mka_system_destroy(s)
