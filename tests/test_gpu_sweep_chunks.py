"""Chunk sums of a sweep for chunks of one atom up to the whole range (threads share a column in short ones): each chunk's
electron count and level energy against the sums of the sweep's own levels in numpy, and a range sweep whose chunks start
inside against the whole one's, bit for bit. Sums of n terms differ by n roundings of the magnitudes' sum."""
import numpy as np
import pytest

from oracle import mka as om
from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [1, 2, 3, 16, 17, 32, 33, 64, 65, 200, 1 << 61])
def test_chunk_sums(chunk):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 23)
    n, nu, mu, kT = 150, 15, 1.9, 0.1
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=5.0)
    try:
        plan = mka.mka_plan_create(s, n, mka.solve_params(8, 7, cg_tol=1e-13))
        sums = []
        for a0 in (0, 100):
            sw = mka.mka_sweep_create(s, a0, n, nu, 0.0, 4.0, 8, chunk)
            mka.mka_plan_run_sweep(plan, sw, np.arange(a0, n, dtype=np.int64))
            sums.append(mka.mka_sweep_chunk_sums(sw, mu, kT))
            alone = mka.mka_sweep_chunk_sums(sw, mu, kT, levels=False)["count"]
            np.testing.assert_array_equal(alone, sums[-1]["count"])
            if a0 == 0:
                res = mka.mka_plan_result(plan)
                lv = mka.mka_result_copy_levels(res)
                first = mka.mka_sweep_info(sw)["chunk0"]
            mka.mka_sweep_destroy(sw)
        mka.mka_plan_destroy(plan)
        assert first == 0
        f = 2.0 * om.fermi(lv["eps"], mu, kT) * lv["w"]
        per = min(chunk, n)
        for name, x in (("count", f), ("e_levels", f * lv["eps"])):
            want = [x[4 * g:4 * (g + per)].sum() for g in range(0, n, per)]
            mag = [np.abs(x[4 * g:4 * (g + per)]).sum() for g in range(0, n, per)]
            assert len(sums[0][name]) == len(want)
            assert (np.abs(sums[0][name] - want) <= 4 * per * nu * 2.0 ** -53 * np.array(mag) + 1e-300).all()
            if 100 % per == 0:
                np.testing.assert_array_equal(sums[1][name], sums[0][name][100 // per:])
    finally:
        mka.mka_system_destroy(s)
