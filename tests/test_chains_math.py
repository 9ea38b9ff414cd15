"""The short recurrences of the two chains (the identity behind chains.cu) in plain numpy against the oracle's
Gram-Schmidt basis: the same levels and density matrix from a 2-orthonormal basis, z = S Q (Q^T S Q)^{-1} e_p standing
in for the S-orthogonal projection, and H_r given by the recurrence coefficients as far as orthogonality is kept."""
import numpy as np
import pytest
import scipy.linalg

from oracle import mka as om
from oracle import sk as osk
from synth import SK_CARBON_LIKE, lattice_positions


def chains(H, S, j, s, p, q):
    nu = p + q
    W, T = np.zeros((H.shape[0], nu)), np.zeros((nu, nu))
    x, last, beta = np.eye(H.shape[0])[j], 0.0, 0.0
    r = s.copy()
    for n in range(p):
        W[:, n] = x
        h = H @ x - beta * last
        T[n, n] = x @ h
        h -= T[n, n] * x
        r -= (x @ r) * x
        beta, last = np.linalg.norm(h), x
        x = h / beta
        if n + 1 < nu:
            T[n, n + 1] = beta if n + 1 < p else 0.0
    Q, bp, qn = W[:, :p], beta, x
    z = S @ (Q @ np.linalg.solve(Q.T @ S @ Q, np.eye(p)[:, -1]))
    a, b, v, last, eta = Q[:, -1].copy(), qn.copy(), r / np.linalg.norm(r), 0.0, 0.0
    zs = np.zeros(nu)
    for n in range(p, nu):
        W[:, n] = v
        zv, qv = z @ v, qn @ v
        zs[n] = zv
        h = H @ v - bp * qv * a - bp * zv * b - eta * last
        hk = v @ h
        h -= hk * v
        a, b = a + zv * v, b - qv * v
        T[p - 1, n] = bp * qv
        T[p:n + 1, n] += bp * qv * zs[p:n + 1]
        T[n, n] += hk
        if n > p:
            T[n - 1, n] += eta
        eta, last = np.linalg.norm(h), v
        v = h / eta
    T = np.triu(T) + np.triu(T, 1).T
    return W, T, W.T @ S @ W


@pytest.mark.parametrize("p,q", [(1, 1), (1, 6), (6, 1), (9, 0), (8, 8), (15, 15)])
def test_chains_span_the_oracles_subspace(p, q):
    pos, box = lattice_positions("diamond", 3.567, 3, 0.1, 0.0, 11)
    cl = osk.cluster_atoms(pos, box, 40, 5.0)
    H, S = osk.cluster_matrices(pos, box, cl, SK_CARBON_LIKE)
    t = int(np.searchsorted(cl, 40))
    for o in range(4):
        j = 4 * t + o
        ref = om.solve_column(H, S, j, p, q)
        W, Hr, Sr = chains(H, S, j, ref.s, p, q)
        # H W = W K + (a rest along the next vector) holds to rounding with the coefficients K, so that the
        # coefficients differ from the projection by (W^T W - I) K and its like: ||H|| times the lost orthogonality,
        # from either side
        Hg = W.T @ H @ W
        lost = np.linalg.norm(W.T @ W - np.eye(p + q), 2)
        assert np.linalg.norm(Hr - Hg, 2) <= np.linalg.norm(H, 2) * (2 * lost + 1e-13)
        eps, C = scipy.linalg.eigh(0.5 * (Hg + Hg.T), Sr)      # as the FP64 form takes it
        V = W @ C
        np.testing.assert_allclose(eps, ref.eps, rtol=0, atol=1e-10)
        f = om.fermi(eps, 0.4, 0.1)
        np.testing.assert_allclose(V @ (f * V[j]), om.rho_column(ref, om.fermi(ref.eps, 0.4, 0.1), np.arange(len(H))),
                                   rtol=0, atol=1e-10)
