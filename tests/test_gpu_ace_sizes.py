"""xk_ace's K_ij, Cholesky and vectors over its block sizes (64-column blocks,
32-wide row registers, the 512-column limit), against NumPy on the same K and C."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 128, 130, 257, 513])
def test_sizes(n):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2207_04636_gb300 as xk
    N, Ng = n + 5, 1200
    rng = np.random.default_rng(n)
    phi = rng.standard_normal((Ng, N)) / np.sqrt(Ng)
    C = np.linalg.qr(rng.standard_normal((N, n)))[0]
    # every grid point an interpolation point, a positive diagonal V and no W: K_ij is
    # 2 sum_R V(R, R) rho(R) psi_i(R) psi_j(R), positive definite
    idx = np.arange(Ng)
    V, W = np.diag(rng.uniform(5.0, 15.0, Ng)), np.zeros((Ng, Ng))
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, _ = h.build(C)
    Kij, xi, sg, br = h.ace()
    h.release()
    Kij0, xi0, s0, br0 = oracle.ace_factor(K, C)
    assert br == br0 == "cholesky" and np.array_equal(sg, np.ones(n))
    # N-term FP64 sums
    assert np.abs(Kij - Kij0).max() <= 4 * N * 2.0 ** -53 * (np.abs(C).T @ np.abs(K)).max()
    # xi xi^T gives K back on the occupied space: n-term sums, times K_ij's conditioning
    err = np.abs((xi @ xi.T) @ C - K).max()
    assert err <= 16 * n * 2.0 ** -53 * np.linalg.cond(Kij0) * np.abs(K).max()


def test_graded_basis():
    """Basis functions scaled by 2^k and the rows of C by 2^-k: K_ij and the vectors follow
    to the last bit, with K_ij from 2e7 multiply-adds on (n = 280) formed from digits."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2207_04636_gb300 as xk
    N = n = 280
    Ng = 300
    rng = np.random.default_rng(1)
    phi = rng.standard_normal((Ng, N)) / np.sqrt(Ng)
    C = np.linalg.qr(rng.standard_normal((N, n)))[0]
    V, W = np.diag(rng.uniform(5.0, 15.0, Ng)), np.zeros((Ng, Ng))

    def run(k):
        s = np.exp2(k)[:, None]
        h = xk.Handle(phi * s.T, np.arange(Ng), V, W, 1.0, n, mode="fp64")
        h.build(C / s)
        Kij, xi, _, br = h.ace()
        h.release()
        return Kij, xi / s, br == "cholesky"

    for a, b in zip(run(np.zeros(N)), run(rng.integers(-40, 41, size=N).astype(np.float64))):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("top", [2.0 ** 1023, 2.0 ** -1010])
def test_pivots_at_the_ends_of_the_range(top):
    """K_ij whose pivots lie just below 2^1023, or below 2^-1010: its vectors still give K back."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2207_04636_gb300 as xk
    n, N, Ng = 4, 9, 1200
    rng = np.random.default_rng(4)
    phi = rng.standard_normal((Ng, N)) / np.sqrt(Ng)
    C = np.linalg.qr(rng.standard_normal((N, n)))[0]
    V, W = np.diag(rng.uniform(5.0, 15.0, Ng)) * 2.0 ** 10, np.zeros((Ng, Ng))  # a dV in range

    def run(dV):
        h = xk.Handle(phi, np.arange(Ng), V, W, dV, n, mode="fp64")
        K, _ = h.build(C)
        Kij, xi, _, br = h.ace()
        h.release()
        assert br == "cholesky"
        return K, Kij, xi

    Kij = run(1.0)[1]
    assert np.diag(Kij).max() < 1.8 * np.diag(Kij).min()
    K, Kij, xi = run(0.95 * top / np.diag(Kij).max())
    assert np.diag(Kij).min() > 0.5 * top or top < 1.0
    K, Kij = K / top, Kij / top
    xi = xi / 2.0 ** (np.log2(top) // 2)
    err = np.abs((xi @ xi.T) @ C / (top / 4.0 ** (np.log2(top) // 2)) - K).max()
    assert err <= 16 * n * 2.0 ** -53 * np.linalg.cond(Kij) * np.abs(K).max()
