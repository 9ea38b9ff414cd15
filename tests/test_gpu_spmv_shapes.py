"""The global products at the edges of their kernels: systems below and above the change from eight to four slots, row
counts that are no multiple of a warp's atoms, the change to rows for BF16 on large systems, rows of 1 to about 55 blocks
(more than a batch of 8 and of 16), all value and vector types. Against a row-by-row product of the stored values in FP64: sums of n products differ by at most
(n + 2) roundings of the vector's type times the sum of the magnitudes."""
import numpy as np
import pytest

from synth import SK_CARBON_LIKE, SK_FCC_METAL, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


SMALL = [("diamond", 3.567, 0.0, 4), ("fcc", 4.0, 0.55, 5), ("fcc", 2.3, 0.03, 5), ("diamond", 3.567, 0.01, 11)]


@pytest.mark.parametrize("lattice,a,vac,cells,storage", [(*c, t) for c in SMALL for t in ("fp64", "fp32", "bf16")] +
                         [("diamond", 3.567, 0.01, 26, "bf16")])    # above 131,072 atoms: rows, not slots
def test_products(lattice, a, vac, cells, storage):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions(lattice, a, cells, 0.05, vac, 3)
    sk = SK_CARBON_LIKE if lattice == "diamond" else SK_FCC_METAL
    s = mka.mka_build_system(pos, box, sk, storage, cluster_radius=4.0)
    try:
        n = len(pos)
        b = mka.mka_system_copy_bsr(s)
        row_ptr, col, H, S = b["row_ptr"], b["col"], b["H"].reshape(-1, 4, 4), b["S"].reshape(-1, 4, 4)
        rows = np.repeat(np.arange(n), np.diff(row_ptr))
        for which, val in ((0, H), (1, S)):
            for dt, eps in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
                for k in (1, 2, 4):
                    x = torch.randn((4 * n, k), device="cuda", dtype=dt, generator=torch.Generator("cuda").manual_seed(k))
                    y = torch.full((4 * n + 8, k), 7.0, device="cuda", dtype=dt)
                    mka.mka_spmv(s, which, mka.MKA_FP64 if dt == torch.float64 else mka.MKA_MIXED_FP32, x.data_ptr(),
                                 y.data_ptr(), k)
                    xb = x.double().cpu().numpy().reshape(n, 4, k)[col]
                    want, mag = np.zeros((n, 4, k)), np.zeros((n, 4, k))
                    np.add.at(want, rows, np.einsum("bij,bjk->bik", val, xb))
                    np.add.at(mag, rows, np.einsum("bij,bjk->bik", np.abs(val), np.abs(xb)))
                    got = y.double().cpu().numpy()
                    assert (got[4 * n:] == 7.0).all()
                    bound = (4 * np.diff(row_ptr).max() + 2) * eps * mag.reshape(4 * n, k)
                    assert (np.abs(got[:4 * n] - want.reshape(4 * n, k)) <= bound).all()
    finally:
        mka.mka_system_destroy(s)
