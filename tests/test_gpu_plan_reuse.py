"""A plan outlives the objects its graphs were captured with: sweeps made and destroyed one after the other (which may lie
at the same address) with the same batches through one plan each get their own levels."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 23)
    s = mka.mka_build_system(pos, box, SK_CARBON_LIKE, "fp64", cluster_radius=5.0)
    yield mka, s, len(pos)
    mka.mka_system_destroy(s)


def test_sweeps_one_after_the_other(system):
    mka, s, n = system
    plan = mka.mka_plan_create(s, n, mka.solve_params(4, 4, cg_tol=1e-13))
    want = None
    for i in range(8):
        sw = mka.mka_sweep_create(s, 0, n, 8, -2.0, 6.0, 6, 10 + i)
        mka.mka_plan_run_sweep(plan, sw, np.arange(n, dtype=np.int64))
        assert mka.mka_sweep_status(sw)[0] == n
        total = mka.mka_sweep_chunk_sums(sw, 1.9, 0.05)["count"].sum()
        mka.mka_sweep_destroy(sw)
        want = total if want is None else want
        assert abs(total - want) <= 1e-10 * abs(want)
    mka.mka_plan_destroy(plan)


def test_networks_one_after_the_other(system):
    """The learned start's network replaced between runs: every run starts from the one attached then, as a direct solve
    does; with none attached a plan refuses, as a direct solve does."""
    mka, s, n = system
    atoms = np.arange(40, dtype=np.int64)
    prm = mka.solve_params(4, 4, arith="mixed", cg_tol=1e-7, use_warm_start=True)
    plan, seen = None, []
    for i in range(6):
        net = mka.mka_mlp_create(i)
        mka.mka_mlp_set_params(net, mka.mka_mlp_get_params(net) * np.float32(0.02 + 0.1 * (i % 3)))
        mka.mka_system_set_warm_start(s, net)
        plan = plan or mka.mka_plan_create(s, len(atoms), prm)
        res = mka.mka_solve_columns(s, atoms, prm)
        want = mka.mka_result_copy_levels(res)["cg_iters"], mka.mka_result_copy_warm_start(res)
        mka.mka_result_destroy(res)
        mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1)
        pres = mka.mka_plan_result(plan)
        np.testing.assert_array_equal(mka.mka_result_copy_levels(pres)["cg_iters"], want[0])
        np.testing.assert_array_equal(mka.mka_result_copy_warm_start(pres), want[1])
        seen.append((want[0].sum(), want[1].sum()))
        mka.mka_system_set_warm_start(s, None)
        with pytest.raises(mka.MkaError) as e:
            mka.mka_plan_run(plan, atoms, 4.0 * len(atoms), 0.1)
        assert e.value.status == mka.MKA_ERR_INVALID_ARG
        mka.mka_mlp_destroy(net)
    mka.mka_plan_destroy(plan)
    assert len(set(seen)) > 1
