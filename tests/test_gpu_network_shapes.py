"""The learned start's network at the edges of its row tiles (8), gradient slices (32 rows) and row chunks (2,048),
against the FP64 oracle on the same BF16-rounded parameters, with the tolerances of the FP32 network test; rows
beyond the batch change nothing, and the sums do not depend on timing."""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_batch_sizes():
    from paper_1202_0098_gb300 import build, mka
    build.build()
    net = mka.mka_mlp_create(11)
    try:
        theta = mka.mka_mlp_get_params(net, bf16_rounded=True).astype(np.float64)
        for B in (33, 1, 7, 8, 9, 2049, 2048, 32, 5000):
            rng = np.random.default_rng(B)
            X = rng.normal(size=(B, 132)).astype(np.float32)
            T = (rng.normal(size=(B, 68)) * 0.1).astype(np.float32)
            Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
            Y = torch.full((B + 8, 68), 7.0, dtype=torch.float32, device="cuda")
            mka.mka_mlp_forward(net, Xd.data_ptr(), Y.data_ptr(), B)
            Yo, _ = omlp.forward(theta, X.astype(np.float64))
            np.testing.assert_allclose(Y[:B].cpu().numpy(), Yo, rtol=0, atol=1e-4 * (1 + np.abs(Yo).max()))
            assert (Y[B:] == 7.0).all()
            out = []
            for _ in range(2):
                g = torch.empty(mka.mka_mlp_num_params(), dtype=torch.float32, device="cuda")
                loss = torch.empty(1, dtype=torch.float32, device="cuda")
                mka.mka_mlp_gradients(net, Xd.data_ptr(), Td.data_ptr(), B, g.data_ptr(), loss.data_ptr())
                out.append((g.cpu().numpy(), loss.item()))
            Lo, go = omlp.loss_and_grad(theta, X.astype(np.float64), T.astype(np.float64))
            gg, L = out[0]
            assert abs(L - Lo) <= 1e-4 * Lo
            assert np.linalg.norm(gg - go) <= 1e-4 * np.linalg.norm(go)
            np.testing.assert_allclose(gg, go, rtol=1e-3, atol=1e-5 * np.abs(go).max())
            np.testing.assert_array_equal(gg, out[1][0])
            assert L == out[1][1]
    finally:
        mka.mka_mlp_destroy(net)
