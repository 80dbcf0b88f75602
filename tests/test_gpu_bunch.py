"""Time of a dense bunch that drifts through an empty grid: about that of the same markers
spread over the grid.  Nodes that it reaches have had no amounts; scales that they
would get only with them sent the bunch's deposits to global memory, one addition at
a time (60 times as long)."""
import time

import numpy as np
import pytest

from paper_2411_09605_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def _step_seconds(cells, cells_a_step, weighted, **kw):
    from paper_2411_09605_gb300 import pic
    n, nc, L = 300_000, 256, 2 * np.pi
    x = L / nc * (3 + cells * np.random.default_rng(1).random(n))
    w = np.full(n, 1e-9 * L / n)
    prob = W.Problem1D("bunch", L, nc, 2, cells_a_step * L / nc, 0,
                       [W.Markers1D(-1.0, 1.0, x, np.ones(n), w if weighted else None, w[0])])
    sim = pic.Simulation(prob, **kw)
    try:
        sim.step(20)
        best = np.inf
        for _ in range(5):
            t = time.perf_counter()
            sim.step(64)
            best = min(best, time.perf_counter() - t)
    finally:
        sim.close()
    return best


@pytest.mark.parametrize("solver", ["ampere", "standard"])
@pytest.mark.parametrize("cells,cells_a_step", [(10, 4.0), (2, 1.3), (40, 30.0)])
def test_a_bunch_takes_no_longer(cells, cells_a_step, solver):
    from paper_2411_09605_gb300 import pic
    kw = {"solver": pic.PIC_SOLVER_STANDARD_LEAPFROG} if solver == "standard" else {}
    spread = _step_seconds(250, cells_a_step, True, **kw)
    assert _step_seconds(cells, cells_a_step, True, **kw) <= 2.0 * spread
