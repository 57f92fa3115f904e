"""Near and far fields where their kernels change shape: sphere counts around the staged tiles (8 and 16), points and
directions around the CTA tiles (64), every degree; points on the beam axis, near it (the Bessel series) and far from
it, above and below a sphere, inside one; directions at the poles.  Against the oracle's field expansion, angular
spectrum and amplitudes.

Tolerance: the FP64 parity bar 1e-10 (both sides sum at most 1e5 terms of rounding 1e-16)."""

import numpy as np
import pytest

from oracle import farfield, incident, svwf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_02145_gb300 import binding as B  # noqa: E402

K = 2.0 * np.pi / 550.0
R = 60.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    B.load()


def solved_context(N, L, inc):
    """A context whose stored solution is the random b returned with it."""
    rng = np.random.default_rng(100 * L + N)
    sites = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    pos = sites[rng.permutation(64)[:N]] * 200.0 + rng.uniform(-30.0, 30.0, (N, 3)) - 300.0
    ctx = B.celes_create(pos, np.full(N, R), np.full(N, 1.5 + 0j), 1.0, K, L)
    B.celes_set_incident(ctx, [inc])
    b = rng.normal(size=(1, N, 2 * L * (L + 2))) + 1j * rng.normal(size=(1, N, 2 * L * (L + 2)))
    B.celes_set_initial_guess(ctx, b)
    B.celes_solve(ctx, 1e30, mode=B.CELES_SOLVE_FP64, x0=B.CELES_X0_USER, use_precond=False)
    assert np.array_equal(B.celes_get_coefficients(ctx), b)
    return ctx, pos, b[0], rng


@pytest.mark.parametrize("N,L,Np", [(1, 1, 1), (15, 2, 63), (16, 3, 64), (17, 4, 65), (33, 5, 7)])
def test_near_field_edges(N, L, Np):
    focus = (20.0, -10.0, 30.0)
    inc = B.make_incident("gaussian", waist=900.0, focus=focus)
    ctx, pos, b, rng = solved_context(N, L, inc)
    try:
        p = rng.uniform(-2500.0, 2500.0, (Np, 3))
        special = np.array([[focus[0], focus[1], 700.0], [focus[0] + 1e-3, focus[1], -800.0],
                            [focus[0] + 30.0, focus[1] - 10.0, 900.0], [pos[0, 0], pos[0, 1], pos[0, 2] + 5 * R],
                            [pos[0, 0], pos[0, 1], pos[0, 2] - 1.5 * R]])[:Np]
        p[:len(special)] = special
        dist = np.linalg.norm(p[:, None] - pos[None], axis=2)
        out = (dist >= R).all(axis=1)
        scat = sum(svwf.field_expansion(3, b[i], L, K, p[out], pos[i]) for i in range(N))
        beam = incident.gaussian_beam_field(K, 900.0, focus, -np.pi / 2, p, n_beta=128, n_alpha=256)
        for what, want, rows in ((0, scat, out), (1, beam, np.ones(Np, bool)), (2, scat + beam[out], out)):
            got = B.celes_nearfield(ctx, p, 0, what)
            assert np.linalg.norm(got[rows] - want) <= 1e-10 * np.linalg.norm(want)
            assert np.isnan(got[~rows]).all()
        centre = B.celes_nearfield(ctx, pos[:1] + np.array([0.3 * R, 0.0, 0.0]), 0, 2)
        assert np.isnan(centre).all()
    finally:
        B.celes_destroy(ctx)


@pytest.mark.parametrize("N,L,Nd", [(1, 1, 1), (7, 2, 63), (8, 3, 64), (9, 4, 65), (40, 5, 130)])
def test_far_field_edges(N, L, Nd):
    ctx, pos, b, rng = solved_context(N, L, B.make_incident("plane"))
    try:
        d = np.stack([np.arccos(rng.uniform(-1.0, 1.0, Nd)), rng.uniform(-7.0, 7.0, Nd)], axis=1)
        d[0] = 0.0
        d[-1, 0] = np.pi
        want = farfield.farfield_amplitude(L, K, pos, b, d)
        got = B.celes_farfield(ctx, d)
        assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
    finally:
        B.celes_destroy(ctx)
