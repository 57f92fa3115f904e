"""The blocked preconditioner build where its steps change shape: blocks of one partial tile, of exactly one tile, one
row more, and on both sides of every panel class (128, 256, 512, 1024 rows and 2048 rows), all in one build, against
the oracle's dense block solves.

Tolerance: the FP64 bar of the parity tests, 1e-10 (both sides solve systems of condition below 1e3 with backward
error about n eps < 1e-12)."""

import numpy as np
import pytest

from oracle import mie, precond

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


@pytest.mark.parametrize("lmax,counts", [
    (1, [1, 5, 6, 21, 22, 42, 43]),       # 6, 30, 36, 126, 132, 252, 258 unknowns
    (2, [2, 1, 3, 16, 17, 32, 33]),       # 32, 16, 48, 256, 272, 512, 528
    (3, [35, 34, 4, 69, 68]),             # 1050, 1020, 120, 2070 (above every cluster), 2040
])
def test_mixed_block_sizes_in_one_build(lmax, counts):
    edge, R, lam = 2000.0, 60.0, 550.0
    rng = np.random.default_rng(7 + lmax)
    # the counts[b] spheres of cuboid b on a jittered 5 x 5 x 5 grid inside it; a sphere at the origin anchors the grid
    sites = np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    pos = []
    for b, n in enumerate(counts):
        cell = sites[rng.permutation(len(sites))[:n]] * 380.0 + 200.0 + rng.uniform(-60.0, 60.0, (n, 3))
        if b == 0:
            cell[0] = 0.0
        pos.append(cell + np.array([edge * b, 0.0, 0.0]))
    pos = np.concatenate(pos)
    pos = pos[rng.permutation(len(pos))]
    N, nmax = len(pos), 2 * lmax * (lmax + 2)
    radii, index = np.full(N, R), np.full(N, 1.6 + 0.01j)
    k0 = 2.0 * np.pi / lam
    ctx = B.celes_create(pos, radii, index, 1.0, k0, lmax)
    try:
        B.celes_precond_build(ctx, edge)
        nb, maxd, _ = B.celes_precond_stats(ctx)
        assert nb == len(counts) and maxd == max(counts) * nmax
        P = precond.BlockPreconditioner(pos, k0, lmax, mie.t_diagonal(lmax, k0, radii, index), edge)
        y = rng.normal(size=(1, N, nmax)) + 1j * rng.normal(size=(1, N, nmax))
        ref = P.apply(y[0])
        yd = torch.from_numpy(y).cuda()
        xd = torch.full_like(yd, float("nan"))
        B.celes_precond_apply(ctx, yd, xd, precision=B.CELES_FP64)
        torch.cuda.synchronize()
        got = xd.cpu().numpy()[0]
        assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
    finally:
        B.celes_destroy(ctx)
