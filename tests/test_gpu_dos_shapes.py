"""The density of states at the edges of its grid: level counts around the staged 256 and the chunks, energy counts
around a warp and around the groups that share a CTA's warps. All terms are positive, so n + 8 roundings of 2^-53 bound
the relative difference of any two summation orders."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 65, 257, 14800, 700001])
@pytest.mark.parametrize("n_e", [1, 32, 33, 129, 257])
def test_level_and_energy_counts(n, n_e):
    from paper_1202_0098_gb300 import build, mka
    build.build()
    rng = np.random.default_rng(100 * n + n_e)
    eps, w = rng.uniform(-3, 3, n), rng.uniform(0.1, 1, n)
    w[rng.random(n) < 0.2] = 0.0            # levels without weight count for nothing, whatever their energy
    eps[w == 0.0] = np.nan
    grid, eta = np.linspace(-3.5, 3.5, n_e), 0.1
    want = np.array([(w[w > 0] / ((e - eps[w > 0]) ** 2 + eta ** 2)).sum() for e in grid]) * eta / np.pi
    de, dw = torch.from_numpy(eps).cuda(), torch.from_numpy(w).cuda()
    got = mka.mka_dos(de.data_ptr(), dw.data_ptr(), n, grid, eta)
    np.testing.assert_allclose(got, want, rtol=(n + 8) * 2.0 ** -53, atol=0)
