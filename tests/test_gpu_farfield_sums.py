"""The far field's sums over spheres: their rounding (runs of a bounded number of spheres, the order in which k.r is
added up) and the shapes that large problems take: tiles of 64 directions with a ragged last one, several sphere chunks,
runs added up in the scratch, and more directions than one pass holds."""

import math

import numpy as np
import pytest

from oracle import farfield

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_02145_gb300 import binding as B  # noqa: E402

K = 2.0 * np.pi / 550.0
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    B.load()


def far_field(pos, b, dirs, L):
    N = len(pos)
    ctx = B.celes_create(pos, np.full(N, 50.0), np.full(N, 1.5 + 0j), 1.0, K, L)
    try:
        B.celes_set_incident(ctx, [B.make_incident("plane")])
        B.celes_set_initial_guess(ctx, b[None])
        B.celes_solve(ctx, 1e30, mode=B.CELES_SOLVE_FP64, x0=B.CELES_X0_USER, use_precond=False)
        return B.celes_farfield(ctx, dirs)
    finally:
        B.celes_destroy(ctx)


def lattice(N, seed, jitter=20.0):
    """Sites of a cube, centred in x and y, z from 0."""
    rng = np.random.default_rng(seed)
    n = math.ceil(N ** (1.0 / 3.0))
    grid = np.stack(np.unravel_index(rng.permutation(n ** 3)[:N], (n, n, n)), axis=1) * 150.0
    grid[:, :2] -= 75.0 * n
    return grid + rng.uniform(-jitter, jitter, (N, 3)), rng


def directions(rng, n):
    return np.stack([np.arccos(rng.uniform(-1.0, 1.0, n)), rng.uniform(0.0, 2 * np.pi, n)], axis=1)


@pytest.mark.parametrize("N,Nd,run", [(250, 1200, 63), (2000, 60100, 256)])
def test_runs_are_short(N, Nd, run):
    # in phase (z = 0, beta = 0): a sum of 1 and terms of 0.9 half-ulps of it, each of which a running sum would lose
    # (0.9 N U in all).  A sum of run spheres loses at most run U, adding those up N / run U, the rest of the evaluation
    # about 20 U.  At lmax 5 these numbers of directions leave one sphere chunk, in four interleaved sums (few directions)
    # or sums of 256.
    L = 5
    side = math.ceil(math.sqrt(N))
    pos = np.stack([150.0 * (np.arange(N) % side), 150.0 * (np.arange(N) // side), np.zeros(N)], axis=1)
    row = 2  # tau = 1, l = 1, m = 1
    b = np.zeros((N, 2 * L * (L + 2)), complex)
    b[:, row] = 0.9 * U
    b[0, row] = 1.0
    one = np.zeros((1, b.shape[1]), complex)
    one[0, row] = math.fsum(b[:, row].real)
    want = farfield.farfield_amplitude(L, K, np.zeros((1, 3)), one, np.zeros((1, 2)))
    got = far_field(pos, b, np.zeros((Nd, 2)), L)
    err = np.linalg.norm(got - want, axis=-1) / np.linalg.norm(want)
    assert err.max() <= (run + N / run + 20) * U


def two_prod(a, b):
    def split(v):
        t = v * 134217729.0
        h = t - (t - v)
        return h, v - h
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def test_error_is_that_of_the_phases():
    # against phases in twice the precision, no more than 1.1 times the error of correctly summed phases that are
    # rounded like x and y first, then z, each addition once (z first, whose range is the largest, has 1.2 times)
    L, N, Nd = 2, 2400, 400
    pos, rng = lattice(N, 3)
    dirs = directions(rng, Nd)
    b = rng.normal(size=(N, 16)) + 1j * rng.normal(size=(N, 16))
    ld = dirs.astype(np.longdouble)
    ex = [np.longdouble(K) * np.sin(ld[:, 0]) * np.cos(ld[:, 1]), np.longdouble(K) * np.sin(ld[:, 0]) * np.sin(ld[:, 1]),
          np.longdouble(K) * np.cos(ld[:, 0])]
    s, e = np.zeros((Nd, N)), np.zeros((Nd, N))
    for q in range(3):
        hi = ex[q].astype(float)
        p, pe = two_prod(hi[:, None], pos[None, :, q])
        s, se = two_sum(s, p)
        e += pe + se + (ex[q] - hi).astype(float)[:, None] * pos[None, :, q]
    true = np.exp(-1j * s) * (1.0 - 1j * e)
    sb, cb, sa, ca = np.sin(dirs[:, 0]), np.cos(dirs[:, 0]), np.sin(dirs[:, 1]), np.cos(dirs[:, 1])
    kx, ky, kz = K * sb * ca, K * sb * sa, K * cb

    def fma(a, v, c):
        p, pe = two_prod(a[:, None], v[None, :])
        t, te = two_sum(p, c)
        return t + (te + pe)
    rounded = np.exp(-1j * fma(kz, pos[:, 2], fma(kx, pos[:, 0], ky[:, None] * pos[None, :, 1])))

    def amplitude(phase):
        # the sum over spheres, then the angular factors: one sphere in the origin per direction
        F = phase @ b
        return np.stack([farfield.farfield_amplitude(L, K, np.zeros((1, 3)), F[d:d + 1], dirs[d:d + 1])[0]
                         for d in range(Nd)])
    want = amplitude(true)
    allowed = np.linalg.norm(amplitude(rounded) - want)
    assert np.linalg.norm(far_field(pos, b, dirs, L) - want) <= 1.1 * allowed


@pytest.mark.parametrize("N,L,Nd", [(1001, 1, 321), (1001, 2, 321), (1001, 3, 321), (1001, 5, 321), (9, 5, 60100)])
def test_large_shapes(N, L, Nd):
    # parity bar 1e-10 at sampled directions: the edges of tiles and passes among them
    pos, rng = lattice(N, 5 + L)
    dirs = directions(rng, Nd)
    dirs[0], dirs[-1, 0] = 0.0, np.pi
    b = rng.normal(size=(N, 2 * L * (L + 2))) + 1j * rng.normal(size=(N, 2 * L * (L + 2)))
    some = np.unique(np.concatenate([[0, 63, 64, 319, 320, Nd - 1], np.clip([59903, 59904, 59967, 60000], 0, Nd - 1),
                                     rng.integers(0, Nd, 30)]))
    got = far_field(pos, b, dirs, L)
    want = farfield.farfield_amplitude(L, K, pos, b, dirs[some])
    assert np.isfinite(got).all()
    assert np.linalg.norm(got[some] - want) <= 1e-10 * np.linalg.norm(want)
