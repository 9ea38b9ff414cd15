"""The mixed form's worst columns. In a few of 10^5 columns the second chain's span is some hundred times more sensitive to
the seam's vectors than in most; their atoms in the 262,144-atom diamond system (found by comparing the mixed form with
FP64 over all of it) against the oracle. An emulation of the form's roundings gives rho errors below 3e-8 there with the
projection vector z held to 48 bits (FP32 S_r and kept rows: 1e-8; z: 2e-8), and 1e-7 to 3e-7 with an FP32 z: 1e-7."""
import numpy as np
import pytest

from oracle import system as osys
from oracle.parallel import solve_atoms_parallel
from synth import WORKLOADS, workload_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_sensitive_columns():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    w = WORKLOADS["diamond262k"]
    pos, box = workload_positions(w)
    atoms = np.array([245197, 78245, 202130, 244691, 79683, 56093], dtype=np.int64)
    ores = solve_atoms_parallel(pos, box, w.sk, w.R, atoms, w.p, w.q, storage="bf16")
    s = mka.mka_build_system(pos, box, w.sk, "bf16", cluster_radius=w.R)
    try:
        res = mka.mka_solve_columns(s, atoms, mka.solve_params(w.p, w.q, arith="mixed", cg_tol=1e-7))
        nb = mka.mka_result_info(res)["n_blocks"]
        rho = torch.full((nb * 16,), float("nan"), dtype=torch.float64, device="cuda")
        mka.mka_density_energy(s, res, 1.983, w.kT, rho.data_ptr())
        mka.mka_result_destroy(res)
        orho = np.concatenate(osys.density(ores, 1.983, w.kT)[0])
        assert np.abs(rho.cpu().numpy().reshape(-1, 4, 4) - orho).max() <= 1e-7
    finally:
        mka.mka_system_destroy(s)
