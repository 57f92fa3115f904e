"""Solves whose Arnoldi steps take each form of the orthogonalisation: one cluster of 1, 2, 4 or 8 blocks, the
cooperative launch with and without its extra barrier, and the separate kernels (long vectors, more than 128 basis
vectors), in FP64 and mixed precision, against the dense LU solution.

Unknowns of one right-hand side are N nmax: a block holds 256 elements, a cluster 8 192, the cooperative form 65 536.
Tolerance: residuals of 1e-11 at a condition below 1e2 leave less than 1e-8."""

import numpy as np
import pytest

import synth
from oracle import incident, mie, solve, translation

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_02145_gb300 import binding as B  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    B.load()


@pytest.mark.parametrize("mode", [B.CELES_SOLVE_FP64, B.CELES_SOLVE_MIXED])
@pytest.mark.parametrize("N,L,restart", [(1, 1, 100), (43, 1, 100), (86, 1, 5), (20, 3, 100), (70, 3, 128),
                                         (70, 3, 129), (52, 4, 7)])
def test_solution_of_every_form(N, L, restart, mode):
    sc = synth.random_cluster(41, N + L, N, L, radius=80.0, fill=0.15, n=1.5 + 0.01j)
    ctx = B.celes_create(sc.positions, sc.radii, sc.n_sphere, sc.n0, sc.k0, L)
    try:
        B.celes_set_incident(ctx, [B.make_incident("plane", beta=0.4, alpha=0.9, pol=1)])
        for _ in range(2):  # the second solve finds the first one's buffers
            B.celes_solve(ctx, 1e-11, mode=mode, restart=restart)
            b = B.celes_get_coefficients(ctx)[0]
        a = incident.plane_wave_coeffs(L, sc.k, sc.positions, 0.4, 0.9, 1)
        t = mie.t_diagonal(L, sc.k, sc.radii, sc.n_rel)
        M = solve.master_matrix(t.reshape(-1), translation.coupling_matrix(sc.positions, sc.k, L))
        want = np.linalg.solve(M, (t * a).reshape(-1)).reshape(b.shape)
        assert np.linalg.norm(b - want) <= 1e-8 * np.linalg.norm(want)
    finally:
        B.celes_destroy(ctx)


@pytest.mark.parametrize("N", [300, 700, 2300])
def test_longer_vectors_reach_the_residual(N):
    # 9 000, 21 000 and 69 000 unknowns: cooperative launch, and the separate kernels beyond 65 536
    rng = np.random.default_rng(N)
    side = int(np.ceil(N ** (1.0 / 3.0)))
    grid = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:N]
    pos = grid * 330.0 + rng.uniform(-30.0, 30.0, (N, 3))
    ctx = B.celes_create(pos, np.full(N, 100.0), np.full(N, 1.45 + 0.01j), 1.0, 2.0 * np.pi / 550.0, 3)
    try:
        B.celes_set_incident(ctx, [B.make_incident("plane")])
        info = B.celes_solve(ctx, 1e-6)
        assert info["residual"] <= 1e-6
        x = torch.from_numpy(B.celes_get_coefficients(ctx)).cuda()
        y = torch.empty_like(x)
        B.celes_master_matvec(ctx, x, y, precision=B.CELES_FP64)
        torch.cuda.synchronize()
        t, a = B.celes_get_tmatrix(ctx), B.celes_get_incident_coefficients(ctx)[0]
        r = y.cpu().numpy()[0] - t * a
        assert np.linalg.norm(r) <= 1.01e-6 * np.linalg.norm(t * a)
    finally:
        B.celes_destroy(ctx)
