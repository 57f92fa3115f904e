"""Several right-hand sides in one coupling launch, short source chunks, and the slice that the in-L2 reduction leaves
zeroed between products: products of 1, 3 and 8 right-hand sides, in alternation and repeated, at sphere counts around
the receiver blocks (64 and 128) and down to one chunk per source, against the dense coupling matrix.

Tolerances: the parity bars, 1e-10 (FP64) and 1e-5 (FP32)."""

import numpy as np
import pytest

import synth
from oracle import mie, translation

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


@pytest.mark.parametrize("variant", [-1, 0, 4, 5])
@pytest.mark.parametrize("N,L", [(1, 3), (3, 5), (64, 1), (65, 2), (129, 1), (40, 4), (33, 5)])
def test_grouped_products_in_alternation(N, L, variant):
    sc = synth.random_cluster(31, N + 7 * L, N, L, radius=90.0, fill=0.2, n=1.6 + 0.01j)
    ctx = B.celes_create(sc.positions, sc.radii, sc.n_sphere, sc.n0, sc.k0, L, variant=variant)
    try:
        W = translation.coupling_matrix(sc.positions, sc.k, L)
        t = mie.t_diagonal(L, sc.k, sc.radii, sc.n_rel)
        x = synth.random_vector(31, N, (8, N, sc.nmax))
        wx = (W @ x.reshape(8, -1).T).T.reshape(x.shape)
        mx = x - t[None] * wx
        for nrhs in (1, 8, 3, 8, 1):
            for prec, dt, tol in ((B.CELES_FP32, np.complex64, 1e-5), (B.CELES_FP64, np.complex128, 1e-10)):
                xd = torch.from_numpy(x[:nrhs].astype(dt)).cuda()
                for fn, ref in ((B.celes_coupling_matvec, wx), (B.celes_master_matvec, mx)):
                    yd = torch.full_like(xd, float("nan"))
                    fn(ctx, xd, yd, nrhs=nrhs, precision=prec)
                    torch.cuda.synchronize()
                    got, want = yd.cpu().numpy().astype(np.complex128), ref[:nrhs]
                    assert np.linalg.norm(got - want) <= tol * max(np.linalg.norm(want), 1e-300)
    finally:
        B.celes_destroy(ctx)
