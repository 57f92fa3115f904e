"""Gaussian-beam coefficients of a sphere next to the beam's axis: what the first steps off the axis change, J_0 and J_2 by
x^2 of their arguments x = k rho sin(beta) and J_1 by x, around the limit of the leading terms; and beams of fewer nodes
than the coefficient kernel takes at a time.

Tolerance of the change: the coefficients on and off the axis are sums of the same 128 terms with Bessel functions right
to 2e-16, so that their difference is right to a few 1e-16 of them; the oracle's likewise.  5e-15 leaves a factor of
ten, and x^2 / 4 is 2e-13 at the largest distance."""

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


def coefficients(pos, L, waist, n_beta):
    N = len(pos)
    ctx = B.celes_create(pos, np.full(N, 50.0), np.full(N, 1.5 + 0j), 1.0, K, L)
    try:
        B.celes_set_incident(ctx, [B.make_incident("gaussian", waist=waist, n_beta=n_beta)])
        return B.celes_get_incident_coefficients(ctx)[0]
    finally:
        B.celes_destroy(ctx)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("krho", [9e-7, 1.1e-6, 1e-7, 9e-9, 1.1e-8])
def test_first_step_off_the_axis(krho, L):
    rho = krho / K
    pos = np.array([[0.0, 0.0, 40.0]]), np.array([[0.6 * rho, 0.8 * rho, 40.0]])
    got = [coefficients(p, L, 300.0, 128) for p in pos]
    want = [incident.gaussian_beam_coeffs(L, K, p, 300.0, (0.0, 0.0, 0.0), -np.pi / 2, n_beta=128) for p in pos]
    err = np.linalg.norm((got[1] - got[0]) - (want[1] - want[0]))
    assert err <= 5e-15 * np.linalg.norm(want[0])


@pytest.mark.parametrize("n_beta", [1, 2, 7, 8, 9])
@pytest.mark.parametrize("N", [1, 40])
def test_few_nodes(N, n_beta):
    rng = np.random.default_rng(n_beta)
    pos = np.stack([150.0 * np.arange(N), rng.uniform(-2000.0, 2000.0, N), rng.uniform(-500.0, 500.0, N)], axis=1)
    want = incident.gaussian_beam_coeffs(3, K, pos, 900.0, (0.0, 0.0, 0.0), -np.pi / 2, n_beta=n_beta)
    got = coefficients(pos, 3, 900.0, n_beta)
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
