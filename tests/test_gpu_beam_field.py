"""The Gaussian beam's field far from its axis, where it is a small difference of large Bessel terms: their arguments
reach every form in which J_0, J_1 and J_2 are evaluated.  Against the oracle's angular spectrum (trapezoid in alpha,
exact to rounding above 2 (k rho + 40) nodes).

Tolerance, of E_0: an argument z = k rho sin(beta) rounds by 2 z 2^-53 and moves J by at most sqrt(2 / (pi z)) of that,
6e-15 at z = 1 000; the values and sums add about 1e-15 on either side."""

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


@pytest.mark.parametrize("waist", [500.0, 2000.0])
def test_far_from_the_axis(waist):
    rng = np.random.default_rng(int(waist))
    rho, phi = rng.uniform(100.0, 1000.0, 150) / K, rng.uniform(0.0, 2 * np.pi, 150)
    p = np.stack([rho * np.cos(phi), rho * np.sin(phi), rng.uniform(-500.0, 500.0, 150)], axis=1)
    ctx = B.celes_create(np.zeros((1, 3)), np.full(1, 50.0), np.full(1, 1.5 + 0j), 1.0, K, 1)
    try:
        B.celes_set_incident(ctx, [B.make_incident("gaussian", waist=waist, focus=(0.0, 0.0, 0.0))])
        got = B.celes_nearfield(ctx, p, 0, 1)
    finally:
        B.celes_destroy(ctx)
    want = incident.gaussian_beam_field(K, waist, (0.0, 0.0, 0.0), -np.pi / 2, p, n_beta=128, n_alpha=2560)
    assert np.abs(got - want).max() <= 1e-14
