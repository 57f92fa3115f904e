"""Solves on either side of the lengths where the orthogonalisation changes form: 8 192 unknowns (one cluster, then a
cooperative launch that deals the dots out) and 65 536 (then separate kernels).  The residual of the solution, from a
product in FP64, reaches the tolerance asked for (with 1 % for its own rounding)."""

import numpy as np
import pytest

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
@pytest.mark.parametrize("N", [273, 274, 2184, 2185])  # 8 190, 8 220, 65 520 and 65 550 unknowns
def test_residual_at_the_edges(N, mode):
    rng = np.random.default_rng(N)
    side = int(np.ceil(N ** (1.0 / 3.0)))
    grid = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:N]
    pos = grid * 330.0 + rng.uniform(-30.0, 30.0, (N, 3))
    ctx = B.celes_create(pos, np.full(N, 100.0), np.full(N, 1.45 + 0.01j), 1.0, 2.0 * np.pi / 550.0, 3)
    try:
        B.celes_set_incident(ctx, [B.make_incident("plane")])
        tol = 1e-5 if mode == B.CELES_SOLVE_FP64 else 1e-8
        assert B.celes_solve(ctx, tol, mode=mode, restart=40)["residual"] <= tol
        x = torch.from_numpy(B.celes_get_coefficients(ctx)).cuda()
        y = torch.empty_like(x)
        B.celes_master_matvec(ctx, x, y, precision=B.CELES_FP64)
        torch.cuda.synchronize()
        rhs = B.celes_get_tmatrix(ctx) * B.celes_get_incident_coefficients(ctx)[0]
        assert np.linalg.norm(y.cpu().numpy()[0] - rhs) <= 1.01 * tol * np.linalg.norm(rhs)
    finally:
        B.celes_destroy(ctx)
