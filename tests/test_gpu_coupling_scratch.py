"""The scratch of a context's products: fixed by its first product, so that captured products stay valid whatever number
of right-hand sides follows; launches over more right-hand sides than it holds; several launches of one product.

Tolerances against the dense coupling matrix: the parity bars, 1e-10 (FP64) and 1e-5 (FP32)."""

import numpy as np
import pytest

import synth
from oracle import mie, translation

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1706_02145_gb300 import binding as B  # noqa: E402

PRECISIONS = ((B.CELES_FP32, np.complex64, 1e-5), (B.CELES_FP64, np.complex128, 1e-10))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    B.load()


class Scene:
    def __init__(self, N, L, nrhs, **options):
        sc = synth.random_cluster(57, N + L, N, L, radius=90.0, fill=0.2, n=1.6 + 0.01j)
        self.ctx = B.celes_create(sc.positions, sc.radii, sc.n_sphere, sc.n0, sc.k0, L, **options)
        W = translation.coupling_matrix(sc.positions, sc.k, L)
        t = mie.t_diagonal(L, sc.k, sc.radii, sc.n_rel)
        self.x = synth.random_vector(57, N, (nrhs, N, sc.nmax))
        self.want = self.x - t[None] * (W @ self.x.reshape(nrhs, -1).T).T.reshape(self.x.shape)

    def vectors(self, nrhs, dtype):
        x = torch.from_numpy(self.x[:nrhs].astype(dtype)).cuda()
        return x, torch.full_like(x, float("nan"))

    def check(self, y, tol):
        torch.cuda.synchronize()
        got, want = y.cpu().numpy().astype(np.complex128), self.want[:len(y)]
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)

    def product(self, nrhs, precision, dtype, tol):
        x, y = self.vectors(nrhs, dtype)
        B.celes_master_matvec(self.ctx, x, y, nrhs, precision)
        self.check(y, tol)


def captured(scene, nrhs, precision, dtype):
    x, y = scene.vectors(nrhs, dtype)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        B.celes_master_matvec(scene.ctx, x, y, nrhs, precision, stream=stream)
    graph.x = x  # read by every replay
    return graph, y


@pytest.mark.parametrize("variant", [-1, 0, 4, 6])
@pytest.mark.parametrize("N,L", [(3, 5), (70, 3)])
def test_captured_product_survives_more_right_hand_sides(N, L, variant):
    s = Scene(N, L, 40, variant=variant)
    try:
        for precision, dtype, tol in PRECISIONS:
            s.product(1, precision, dtype, tol)
            one, y1 = captured(s, 1, precision, dtype)
            eight, y8 = captured(s, 8, precision, dtype)  # more than any product before it
            held = [torch.full((1 << 20,), float("nan"), device="cuda") for _ in range(8)]
            for nrhs in (8, 40, 1):
                s.product(nrhs, precision, dtype, tol)
                for graph, y in ((one, y1), (eight, y8), (one, y1)):
                    y.fill_(float("nan"))
                    graph.replay()
                    s.check(y, tol)
            assert all(bool(torch.isnan(h).all()) for h in held)
    finally:
        torch.cuda.synchronize()
        B.celes_destroy(s.ctx)


def test_first_product_of_a_precision_under_capture():
    s = Scene(33, 3, 9)
    try:
        s.product(1, B.CELES_FP32, np.complex64, 1e-5)
        graph, y = captured(s, 8, B.CELES_FP64, np.complex128)
        for _ in range(2):
            y.fill_(float("nan"))
            graph.replay()
            s.check(y, 1e-10)
            s.product(9, B.CELES_FP64, np.complex128, 1e-10)
        del graph
    finally:
        torch.cuda.synchronize()
        B.celes_destroy(s.ctx)


@pytest.mark.parametrize("variant", [-1, 0, 4, 6])
@pytest.mark.parametrize("N,L,nrhs", [(3, 1, 257), (3, 1, 600), (130, 4, 70)])
def test_products_of_several_launches(N, L, nrhs, variant):
    # 256 right-hand sides a launch at most; 70 of 130 spheres at lmax 4 need more than the scratch
    s = Scene(N, L, nrhs, variant=variant)
    try:
        for precision, dtype, tol in PRECISIONS:
            for n in (nrhs, 1, nrhs):
                s.product(n, precision, dtype, tol)
    finally:
        B.celes_destroy(s.ctx)


@pytest.mark.parametrize("variant", [-1, 0, 4, 5])
def test_products_and_replays_on_several_streams(variant):
    # ordered by events; the scratch is cleared by the epilogues, by the products or by the graph
    s = Scene(300, 3, 8, variant=variant)
    streams = [torch.cuda.Stream() for _ in range(3)]
    try:
        for precision, dtype, tol in PRECISIONS:
            s.product(1, precision, dtype, tol)
            graph, yg = captured(s, 3, precision, dtype)
            work = [(streams[q % 3], nrhs, *s.vectors(nrhs, dtype)) for q, nrhs in enumerate((1, 8, 1, 8, 8, 1, 1, 3))]
            torch.cuda.synchronize()
            last = None
            for q in range(40):
                stream, nrhs, x, y = work[q % len(work)]
                if last is not None:
                    stream.wait_stream(last)
                if q % 5 == 4:
                    with torch.cuda.stream(stream):
                        graph.replay()
                B.celes_master_matvec(s.ctx, x, y, nrhs, precision, stream=stream)
                last = stream
            for y in [w[3] for w in work] + [yg]:
                s.check(y, tol)
            s.product(8, precision, dtype, tol)
    finally:
        torch.cuda.synchronize()
        B.celes_destroy(s.ctx)
