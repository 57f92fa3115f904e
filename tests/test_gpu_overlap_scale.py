"""The overlap test at lengths whose squares leave FP32's range, in either direction: a pair that overlaps by 1e-4 of its
distance is refused, one that is as far apart is not, in any unit of length."""

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


@pytest.mark.parametrize("unit", [1e-60, 1e-30, 1e-24, 3e-23, 1e-22, 1e-21, 1e-19, 1e-10, 1.0, 1e10, 1e18, 1e30])
def test_overlap_in_any_unit(unit):
    rng = np.random.default_rng(5)
    for trial in range(20):
        v = rng.normal(size=3)
        v /= np.linalg.norm(v)
        radii = rng.uniform(0.3, 1.0, 3)
        for sign in (-1.0, 1.0):
            pos = np.array([[4.0, -3.0, 2.0], [0.0, 0.0, 0.0], v * (radii[1] + radii[2]) * (1.0 + sign * 1e-4)])

            def create():
                B.celes_destroy(B.celes_create(pos * unit, radii * unit, np.full(3, 1.5 + 0j), 1.0, 1.0 / unit, 1))

            if sign > 0.0:
                create()
            else:
                with pytest.raises(B.CelesError) as err:
                    create()
                assert err.value.code == B.CELES_EOVERLAP
