"""The global products where a thread per row takes over (spmv_rule.cuh): one block a row at any size, few blocks, and
FP64 values on large systems; all value and vector types, against the bound of test_gpu_spmv_shapes.py."""
from dataclasses import replace

import numpy as np
import pytest

from synth import SK_CARBON_LIKE, lattice_positions

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# cells, neighbour radius: about 1, 2, 4.4 and 8.4 blocks a row; 64 to 110,592 atoms
@pytest.mark.parametrize("cells,rc", [(2, 1.2), (8, 1.2), (15, 1.2), (15, 1.45), (10, 1.7), (15, 1.7), (10, 2.45), (24, 2.45)])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16"])
def test_products(cells, rc, storage):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    pos, box = lattice_positions("diamond", 3.567, cells, 0.1, 0.01, 3)
    s = mka.mka_build_system(pos, box, replace(SK_CARBON_LIKE, rc=rc), storage, cluster_radius=1.5)
    try:
        n = len(pos)
        b = mka.mka_system_copy_bsr(s)
        row_ptr, col, H = b["row_ptr"], b["col"], b["H"].reshape(-1, 4, 4)
        start = row_ptr[:-1]
        for dt, eps in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
            for k in (1, 2, 4):
                x = torch.randn((4 * n, k), device="cuda", dtype=dt, generator=torch.Generator("cuda").manual_seed(k))
                y = torch.full((4 * n + 8, k), 7.0, device="cuda", dtype=dt)
                mka.mka_spmv(s, 0, mka.MKA_FP64 if dt == torch.float64 else mka.MKA_MIXED_FP32, x.data_ptr(), y.data_ptr(), k)
                xb = x.double().cpu().numpy().reshape(n, 4, k)[col]
                want = np.add.reduceat(np.einsum("bij,bjk->bik", H, xb), start).reshape(4 * n, k)
                mag = np.add.reduceat(np.einsum("bij,bjk->bik", np.abs(H), np.abs(xb)), start).reshape(4 * n, k)
                got = y.double().cpu().numpy()
                assert (got[4 * n:] == 7.0).all()
                assert (np.abs(got[:4 * n] - want) <= (4 * np.diff(row_ptr).max() + 2) * eps * mag).all()
    finally:
        mka.mka_system_destroy(s)
