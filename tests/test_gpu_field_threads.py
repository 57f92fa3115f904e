"""Field evaluations of one context from several host threads at once: each needs another size of the context's
workspace, which they take in turn.  Equal to the same calls one after another, bit by bit."""

import threading

import numpy as np
import pytest

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


def test_concurrent_field_evaluations():
    rng = np.random.default_rng(8)
    N, L = 60, 3
    pos = np.stack(np.unravel_index(rng.permutation(64)[:N], (4, 4, 4)), axis=1) * 200.0
    ctx = B.celes_create(pos, np.full(N, 60.0), np.full(N, 1.5 + 0j), 1.0, K, L)
    try:
        B.celes_set_incident(ctx, [B.make_incident("gaussian", waist=900.0), B.make_incident("gaussian", waist=900.0)])
        b = rng.normal(size=(2, N, 30)) + 1j * rng.normal(size=(2, N, 30))
        B.celes_set_initial_guess(ctx, b)
        B.celes_solve(ctx, 1e30, mode=B.CELES_SOLVE_FP64, x0=B.CELES_X0_USER, use_precond=False)
        calls = []
        for n in (3, 900, 40, 5000, 200, 20000):
            d = np.stack([rng.uniform(0.0, np.pi, n), rng.uniform(0.0, 2 * np.pi, n)], axis=1)
            p = rng.uniform(-3000.0, 3000.0, (n, 3))
            calls += [lambda d=d: B.celes_farfield(ctx, d), lambda p=p: B.celes_nearfield(ctx, p, 1, 2),
                      lambda n=n: B.celes_s11(ctx, np.linspace(0.1, 3.0, 8), 0, 1, n_alpha=n // 8 + 1)]
        want = [call() for call in calls]
        wrong = []

        def work(k):
            for q in range(len(calls)):
                i = (5 * q + 3 * k) % len(calls)
                if not np.array_equal(calls[i](), want[i], equal_nan=True):
                    wrong.append(i)

        threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not wrong
    finally:
        B.celes_destroy(ctx)
