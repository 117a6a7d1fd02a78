"""FP64 products split into digits on the tensor cores (large products of an
XK_FP64 handle): exact where FP64 is exact, no further from a wider reference
than FP64 rounding, and the general path for operands that cannot be split."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xk():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2207_04636_gb300 as m
    return m


def _ints(rng, shape, m):
    return rng.integers(-m, m + 1, size=shape).astype(np.float64)


def _case(Ng, N, n, na, seed, m=3):
    rng = np.random.default_rng(seed)
    phi, C, V = _ints(rng, (Ng, N), m), _ints(rng, (N, n), m), _ints(rng, (na, Ng), m)
    W = _ints(rng, (na, na), m)
    return phi, np.sort(rng.permutation(Ng)[:na]), V, W + W.T, C


def _lines(phi, idx, V, W, C):
    psi = phi @ C
    psig, phig = psi[idx], phi[idx]
    V2 = V * (psig @ psi.T)
    return ((psig.T @ V2) @ phi, (V2 @ psi).T @ phig, ((W * (psig @ psig.T)) @ psig).T @ phig)


# Rows, columns and depths on both sides of the 128 x 64 tiles, the 32-deep
# blocks and the 256-term groups; odd row lengths (unaligned rows) and even.
SHAPES = [(4992, 24, 16, 400), (4993, 127, 33, 128), (5119, 129, 64, 129), (4097, 66, 65, 255),
          (6145, 40, 8, 641), (2048, 257, 128, 256), (90001, 33, 31, 65)]


@pytest.mark.parametrize("Ng,N,n,na", SHAPES)
def test_integers_exact(xk, Ng, N, n, na):
    """Small integers: every sum is an integer below 2^53, so K and the full K
    equal the host's bit for bit."""
    phi, idx, V, W, C = _case(Ng, N, n, na, Ng + n, m=1 if Ng > 50000 else 2)
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, E = h.build(C)
    Kf = h.build_full(C)
    h.release()
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    assert max(np.abs(l).max() for l in (l1, l2, l3)) < 2.0 ** 52
    assert np.array_equal(K, (l1 + l2 - l3).T)
    psi = phi @ C
    psig, phig = psi[idx], phi[idx]
    Y = phig.T @ ((V * (psig @ psi.T)) @ phi)
    assert np.array_equal(Kf, Y + Y.T - phig.T @ ((W * (psig @ psig.T)) @ phig))


@pytest.mark.parametrize("spread", [0, 40])
def test_against_wider(xk, spread):
    """Reals (rows scaled by up to 2^spread) against extended precision: eight
    roundings of 2^-53 in the 2-norm of the three lines."""
    Ng, N, n, na = 4096, 24, 20, 400
    rng = np.random.default_rng(5)
    phi, C = rng.standard_normal((Ng, N)), rng.standard_normal((N, n))
    phi *= np.exp2(-rng.uniform(0, spread, size=(Ng, 1)))
    V, W = rng.standard_normal((na, Ng)), rng.standard_normal((na, na))
    W = W + W.T
    idx = np.sort(rng.permutation(Ng)[:na])
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, _ = h.build(C)
    h.release()
    x = _lines(*(a.astype(np.longdouble) if a.dtype.kind == "f" else a for a in (phi, idx, V, W, C)))
    err = np.linalg.norm((K - (x[0] + x[1] - x[2]).T).astype(np.float64))
    assert err <= 8 * 2.0 ** -53 * sum(np.linalg.norm(l.astype(np.float64)) for l in x)


def test_not_finite(xk):
    """A NaN or an infinity in C reaches K as FP64 arithmetic has it, and the
    handle's next build is exact again."""
    phi, idx, V, W, C = _case(4993, 40, 16, 400, 3)
    phi[phi == 0] = 1.0
    h = xk.Handle(phi, idx, V, W, 1.0, 16, mode="fp64")
    for bad in (np.nan, np.inf):
        Cb = C.copy()
        Cb[5, 3] = bad
        K, E = h.build(Cb)
        assert np.all(np.isnan(K)) and np.isnan(E)
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    assert np.array_equal(h.build(C)[0], (l1 + l2 - l3).T)
    h.release()


def test_tiny_rows(xk):
    """Rows whose largest entry is below 2^-900 keep the general path: a basis
    scaled by 2^-950 with C scaled back gives K scaled by 2^-950 exactly."""
    phi, idx, V, W, C = _case(4993, 40, 16, 400, 4)
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    h = xk.Handle(phi * 2.0 ** -950, idx, V, W, 1.0, 16, mode="fp64")
    K, _ = h.build(C * 2.0 ** 950)
    h.release()
    assert np.array_equal(K, (l1 + l2 - l3).T * 2.0 ** -950)


@pytest.mark.parametrize("N", [64, 65, 129, 200, 257])
def test_symmetric_product(xk, N):
    """J forms one half of a symmetric product: every tile on or below the diagonal,
    mirrored; the Poisson solve's even and odd grids."""
    import oracle

    grid = 24 if N % 2 else 21
    rng = np.random.default_rng(N)
    phi, C = rng.standard_normal((grid ** 3, N)), rng.standard_normal((N, 5)) / N
    idx, V, W = np.arange(8), np.zeros((8, grid ** 3)), np.zeros((8, 8))
    dV = 6.0 ** 3 / grid ** 3
    h = xk.Handle(phi, idx, V, W, dV, 5, mode="fp64")
    J, EJ = h.coulomb(C, grid, 6.0)
    h.release()
    J0, EJ0 = oracle.coulomb_j(phi, C, 6.0, grid, dV)
    assert np.array_equal(J, J.T)
    # sums of grid^3 products in FP64 on the host, the potential's rounding alike
    tol = 2.0 ** -53 * np.sqrt(grid ** 3) * 16
    assert np.linalg.norm(J - J0) <= tol * np.linalg.norm(J0)
    assert abs(EJ - EJ0) <= tol * abs(EJ0)


@pytest.mark.parametrize("n", [32, 33, 48, 64, 65])
def test_kept_rows(xk, n):
    """Products of 33 to 64 terms keep the digits of Y rows that successive tiles
    share: more than 152 tiles along X (tiles t and t + 152 share them or not), three
    along Y, and the depths beside the two that fit."""
    phi, idx, V, W, C = _case(25001, 72, n, 130, n, m=1)
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, _ = h.build(C)
    h.release()
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    assert max(np.abs(l).max() for l in (l1, l2, l3)) < 2.0 ** 52
    assert np.array_equal(K, (l1 + l2 - l3).T)


@pytest.mark.parametrize("Ng,N,n,na", [(6145, 40, 32, 130), (5000, 70, 64, 641), (4100, 300, 257, 129)])
@pytest.mark.parametrize("bad", [None, np.nan])
def test_maxima_of_a_product(xk, Ng, N, n, na, bad):
    """The largest entries of V2 come with it (up to 256 terms; 257 are read again):
    exact results from rows of different size, and after a NaN, whose products go the
    general way."""
    phi, idx, V, W, C = _case(Ng, N, n, na, n, m=1)
    V = V * 2.0 ** np.random.default_rng(1).integers(-3, 4, size=na)[:, None]
    bound = _lines(*(np.abs(a) if a is not idx else a for a in (phi, idx, V, W, C)))
    assert 8 * sum(l.max() for l in bound) < 2.0 ** 53
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    if bad is not None:
        Cb = C.copy()
        Cb[0, 0] = bad
        assert np.isnan(h.build(Cb)[1])
    K, _ = h.build(C)
    h.release()
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    assert np.array_equal(K, (l1 + l2 - l3).T)


@pytest.mark.parametrize("n", [16, 31, 32])
def test_one_block_tiles(xk, n):
    """Products of up to 32 terms: one block a tile and several tiles a CTA, so the
    exponents of a tile's rows are replaced as soon as its block is stored; rows of
    different size, so that a wrong exponent shows."""
    phi, idx, V, W, C = _case(6145, 40, n, 641, n, m=1)
    phi *= np.exp2(np.random.default_rng(2).integers(0, 4, size=phi.shape[0]))[:, None]
    bound = _lines(*(np.abs(a) if a is not idx else a for a in (phi, idx, V, W, C)))
    assert sum(l.max() for l in bound) < 2.0 ** 53
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, _ = h.build(C)
    h.release()
    l1, l2, l3 = _lines(phi, idx, V, W, C)
    assert np.array_equal(K, (l1 + l2 - l3).T)


def test_graded_basis(xk):
    """Basis functions scaled by 2^k and the rows of C by 2^-k are the same calculation:
    every result of an FP64 handle follows to the last bit."""
    grid, N, n, na = 17, 129, 64, 129
    rng = np.random.default_rng(8)
    Ng = grid ** 3
    phi, C = rng.standard_normal((Ng, N)), rng.standard_normal((N, n)) / N
    V, W = rng.standard_normal((na, Ng)), rng.standard_normal((na, na))
    idx = np.sort(rng.permutation(Ng)[:na])

    def run(k):
        s = np.exp2(k)
        h = xk.Handle(phi * s, idx, V, W + W.T, 0.25, n, mode="fp64")
        c = C / s[:, None]
        K, E = h.build(c)
        Kij, xi, _, _ = h.ace()
        J, EJ = h.coulomb(c, grid, 6.0)
        out = (K / s[:, None], E, Kij, xi / s[:, None], h.energy(c), J / s[:, None] / s, EJ,
               h.build_full(c) / s[:, None] / s)
        h.release()
        return out

    for a, b in zip(run(np.zeros(N)), run(rng.integers(-40, 41, size=N).astype(np.float64))):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("r", [0, 10, 30])
def test_small_points(xk, r):
    """Interpolation points where the basis is 2^-r of its usual size, with potentials that
    make up for it, against extended precision: eight roundings of 2^-53 in the 2-norm of
    the three lines, as for points of one size.  V and W are returned as they came."""
    Ng, N, n, na = 4096, 24, 20, 400
    rng = np.random.default_rng(9)
    phi, C = rng.standard_normal((Ng, N)), rng.standard_normal((N, n))
    idx = np.sort(rng.permutation(Ng)[:na])
    s = np.exp2(-rng.integers(0, r + 1, size=na).astype(np.float64))
    phi[idx] *= s[:, None]
    V, W = rng.standard_normal((na, Ng)) / s[:, None] ** 2, rng.standard_normal((na, na))
    W = (W + W.T) / s[:, None] ** 2 / s ** 2
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    K, _ = h.build(C)
    W1, V1, _ = h.tables([0, na - 1])
    h.release()
    assert np.array_equal(W1, W) and np.array_equal(V1, V[[0, na - 1]])
    x = _lines(*(a.astype(np.longdouble) if a.dtype.kind == "f" else a for a in (phi, idx, V, W, C)))
    err = np.linalg.norm((K - (x[0] + x[1] - x[2]).T).astype(np.float64))
    assert err <= 8 * 2.0 ** -53 * sum(np.linalg.norm(l.astype(np.float64)) for l in x)


def test_graded_basis_tensor_path(xk):
    """The tensor path's Q = L^T C, from 6e7 multiply-adds on formed from digits: a graded
    basis gives the same energy to the last bit."""
    Ng, N, n, na = 2000, 832, 100, 150
    rng = np.random.default_rng(11)
    phi, C = rng.standard_normal((Ng, N)) / np.sqrt(Ng), rng.standard_normal((N, n)) / np.sqrt(N)
    V, W = rng.standard_normal((na, Ng)), rng.standard_normal((na, na))
    idx = np.sort(rng.permutation(Ng)[:na])
    E = []
    for k in (np.zeros(N), rng.integers(-20, 21, size=N).astype(np.float64)):
        h = xk.Handle(phi * np.exp2(k), idx, V, W + W.T, 0.25, n, mode="f16x3")
        E.append(h.energy(C * np.exp2(-k)[:, None]))
        h.release()
    assert E[0] == E[1] and np.isfinite(E[0])


@pytest.mark.parametrize("Ng,N,n,na", [(27000, 16, 16, 64), (25001, 72, 48, 130), (90001, 33, 31, 65),
                                       (6145, 40, 32, 130)])
def test_few_points_on_a_fine_grid(xk, Ng, N, n, na):
    """A product is formed from digits by its size alone, also where the handle's other
    buffers are small: a sum 1 + 15 2^-54 is rounded once, to 1 + 2^-50, where FMAs in the
    order of the terms give 1."""
    phi, V, W = np.zeros((Ng, N)), np.zeros((na, Ng)), np.zeros((na, na))
    idx = np.arange(na)
    phi[0, :16] = phi[Ng - 1, :16] = [1.0] + [2.0 ** -27] * 15
    V[0, Ng - 1] = 1.0
    h = xk.Handle(phi, idx, V, W, 1.0, n, mode="fp64")
    C = np.eye(N, n)
    K, _ = h.build(C)
    E = h.energy(C)
    h.release()
    assert K[0, 0] == 2 * (1 + 2.0 ** -50) and E == -2 * (1 + 2.0 ** -50) ** 2


def test_digits_at_their_limit(xk):
    """Operands whose digits are as large as they get (126, then 127 and 124 at the end, as an
    element is below 127/128 of its grid): levels 4 to 7 of a group's 256 terms pass 2^24
    in their accumulators, where an addition may lose a unit (some 20 of level 4, 2^-50 of the
    sum).  E_x = -2 P^2 doubles that and adds its own roundings."""
    Ng, n, na = 4000, 256, 40
    x = 0x7e7f7f7f7f7f7c  # of 2^-55
    assert int(float(x)) == x
    phi, V, W = np.full((Ng, n), x * 2.0 ** -55), np.zeros((na, Ng)), np.zeros((na, na))
    V[3, Ng - 5] = 1.0
    h = xk.Handle(phi, np.arange(na), V, W, 1.0, n, mode="fp64")
    E = h.energy(np.eye(n))
    h.release()
    exact = 2 * (n * x * x) ** 2  # of 2^-220
    got = int(-E * 2.0 ** 60) << 160
    assert abs(got - exact) <= exact >> 48


def test_large_coefficients_that_cancel(xk):
    """Two equal basis functions with coefficients 2^14 and -2^14 beside others below one,
    multiples of 2^-48, which a grid of 2^-55 of the largest would round to 2^-40 (2^-39 in Psi,
    at every grid point alike).  Read from K = Psi_0(R) Psi_i(R); eight digits hold the
    coefficients, and taking the sums out rounds to 2^-58 of the largest product, twice."""
    Ng, N, n, na = 20001, 66, 24, 130
    rng = np.random.default_rng(13)
    phi, V, W = _ints(rng, (Ng, N), 1), np.zeros((na, Ng)), np.zeros((na, na))
    phi[:, 1] = phi[:, 0]
    phi[:, 65] = phi[0] = 0.0
    phi[0, 65] = V[0, Ng - 1] = 1.0
    c = rng.integers(-2 ** 47, 2 ** 47, size=(N, n))  # of 2^-48
    c[0], c[1], c[65] = 2 ** 62, -2 ** 62, 0
    c[65, 0] = 2 ** 48
    h = xk.Handle(phi, np.arange(na), V, W, 1.0, n, mode="fp64")
    K = h.build(c * 2.0 ** -48)[0][65]
    h.release()
    psi = (phi[Ng - 1].astype(np.int64) @ c) * 2.0 ** -48  # below 64, exact
    err = np.abs(K - psi[0] * psi)
    assert np.all(err <= (np.abs(psi[0]) + np.abs(psi)) * 2.0 ** -42 + 2.0 ** -46)


def test_ties_of_one_sign(xk):
    """A row whose elements with coefficients +2^10 lie half-way between two values of the
    row's grid, those with -2^10 on it: Psi there is a small difference (a multiple of
    2^-45) that ties rounded all one way would move by 2^-40.  E_x = -2 Psi^2."""
    Ng, N, n, na = 20001, 66, 16, 64
    rng = np.random.default_rng(17)
    plus = np.arange(64) % 4 < 2
    x = 2 ** 52 + 2 * rng.integers(0, 2 ** 39, size=64) + plus  # of 2^-55
    phi, C = np.zeros((Ng, N)), np.zeros((N, n))
    phi[0, 65] = phi[Ng - 1, 64] = 1.0
    phi[1 + np.arange(64), np.arange(64)] = 1.0  # columns of one size
    phi[Ng - 1, :64] = x * 2.0 ** -55
    C[:64, 0], C[65, 0] = np.where(plus, 2.0 ** 10, -2.0 ** 10), 1.0
    V, W = np.zeros((na, Ng)), np.zeros((na, na))
    V[0, Ng - 1] = 1.0
    h = xk.Handle(phi, np.arange(na), V, W, 1.0, n, mode="fp64")
    E = h.energy(C)
    h.release()
    psi = float(np.where(plus, x, -x).sum()) * 2.0 ** -45
    assert abs(E + 2 * psi ** 2) <= 2.0 ** -51 * 2 * psi ** 2
