"""Shared memory of the launches: a kernel's limit is not that of the handle made
last, and the kernels' static arrays fit beside a dynamic part of just 48 KB."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_09605_gb300 import workloads as W
from tests import test_gpu_standard as std

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def test_standard_scheme_with_48_kb_of_tables_and_tile():
    prob = W.landau(n=1000, nc=1024, order=2, dt=0.05, seed=3)
    std._compare(prob, std._oracle(prob, 0, 3), std._gpu(prob, 0, 3))


def _makers():
    from paper_2411_09605_gb300 import pic

    def es(nc, **kw):
        return lambda: pic.Simulation(W.landau(n=1000, nc=nc, order=2, seed=1), **kw)

    def em(n, precision):
        prob = W.weibel_1d2v(n=n, ppc=4, order=2, seed=1)
        return lambda: pic.Simulation1D2V(prob, solver=O.PSATD, precision=precision)

    return [
        (es(512, precision=1), es(64, precision=1)),
        (es(512, precision=1, scheme=1), es(64, precision=1, scheme=1)),
        (es(8192, precision=1, sort_period=1), es(64, precision=1, sort_period=1)),
        (es(8192), es(2000)), (es(1792), es(8)),
        (es(4096, solver=pic.PIC_SOLVER_STANDARD_LEAPFROG),
         es(2048, solver=pic.PIC_SOLVER_STANDARD_LEAPFROG)),
        (em(1024, 0), em(512, 0)), (em(1024, 1), em(512, 1)),
    ]


@pytest.mark.parametrize("k", range(8))
def test_a_large_grid_steps_after_a_smaller_one_was_made(k):
    """The same steps with and without another handle made in between."""
    large, small = _makers()[k]
    alone, sim = large(), large()
    other = small()
    try:
        fb, te = alone.step(2)
        fb2, te2 = sim.step(2)
        assert np.array_equal(fb, fb2) and np.allclose(te, te2, rtol=1e-12)
        other.step(1)
    finally:
        for s in (alone, sim, other):
            s.close()
