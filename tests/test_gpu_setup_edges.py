"""Context set-up where its kernels change shape: Gaussian-beam coefficients for sphere counts around the 32 of a CTA
(and the cluster that shares the nodes of few spheres), node counts that are no multiple of its step, every degree, and
every branch of the Bessel functions (on the axis, next to it, below and above the switch at 8); the overlap test around
its tile of 256 spheres, far from the origin, for spheres that just touch and that just overlap.

Tolerance of the coefficients: the parity bar 1e-10; both sides use the same Gauss-Legendre rule, whose sum of at most
129 terms and Bessel values of 1e-15 leave about 1e-14."""

import numpy as np
import pytest

from oracle import incident

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_02145_gb300 import binding as B  # noqa: E402

K = 2.0 * np.pi / 550.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    B.load()


@pytest.mark.parametrize("N,L,nb", [(1, 1, 128), (31, 2, 129), (32, 3, 40), (33, 4, 128), (70, 5, 61)])
def test_gaussian_coefficients_edges(N, L, nb):
    rng = np.random.default_rng(N + L)
    focus = (30.0, -20.0, 10.0)
    # a line of spheres from the axis outwards: k rho sin(beta) from 0 through 1e-6, 1 and 8 to about 80
    rho = np.concatenate([[0.0, 1e-5, 1.0, 200.0], np.linspace(300.0, 9000.0, 70)])[:N]
    phi = rng.uniform(0.0, 2 * np.pi, N)
    pos = np.stack([focus[0] + rho * np.cos(phi), focus[1] + rho * np.sin(phi), 300.0 * np.arange(N) - 500.0], axis=1)
    ctx = B.celes_create(pos, np.full(N, 50.0), np.full(N, 1.5 + 0j), 1.0, K, L)
    try:
        B.celes_set_incident(ctx, [B.make_incident("gaussian", waist=1000.0, focus=focus, n_beta=nb)])
        want = incident.gaussian_beam_coeffs(L, K, pos, 1000.0, focus, -np.pi / 2, n_beta=nb)
        got = B.celes_get_incident_coefficients(ctx)[0]
        assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
    finally:
        B.celes_destroy(ctx)


@pytest.mark.parametrize("N", [2, 255, 256, 257, 600])
@pytest.mark.parametrize("offset", [0.0, 3.0e7])
def test_overlap_check_edges(N, offset):
    pos = np.stack([100.0 * np.arange(N), np.zeros(N), np.zeros(N)], axis=1) + offset
    rad = np.full(N, 50.0)  # neighbours touch: distance exactly R_i + R_j, no overlap

    def create(p):
        ctx = B.celes_create(p, rad, np.full(N, 1.5 + 0j), 1.0, K, 1)
        B.celes_destroy(ctx)

    create(pos)
    for a in sorted({0, N // 2 - 1, N - 2}):
        near = pos.copy()
        near[a + 1:, 0] -= 1e-6  # the pair (a, a + 1) overlaps by 1e-8 of the distance
        with pytest.raises(B.CelesError) as err:
            create(near)
        assert err.value.code == B.CELES_EOVERLAP
