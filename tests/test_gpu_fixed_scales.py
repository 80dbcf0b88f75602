"""Deposits of the FP64 forms where amounts span twelve decades: markers with large
amounts (weights, speeds, a species' weight, adjoints) fill one part of the domain,
with small ones another, and the fields of the nodes that only the small ones reach
are judged by themselves.  A deposit that rounds every amount to a unit of the
largest is good to 1e-4 there.

Bar: the 1e-11 (fields) and 1e-9 (gradients) of these forms' other tests, relative to
the largest value of that part: there the sums of both sides are those of a run that
has the small amounts alone, of which those bars were taken.  E^0 = 0 and the mean
current stays in, so that the nodes have nothing but their own deposits."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_09605_gb300 import workloads as W
from tests import test_gpu_standard as std
from tests.parity_util import gpu_run, oracle_run
from tests.test_gpu_em1d import _gpu_run

pytestmark = pytest.mark.gpu
SMALL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def _part(nc):
    i = np.arange(nc) / nc
    return (i > 0.56) & (i < 0.95)


def _problem(kind, n, nc, order):
    rng = np.random.default_rng(n + nc + order)
    L = 2 * np.pi
    x = L * np.where(np.arange(n) % 2, rng.uniform(0.1, 0.4, n), rng.uniform(0.6, 0.9, n))
    small = x > L / 2
    v, w = 0.3 * rng.standard_normal(n), np.full(n, L / n)
    if kind == "speeds":
        v = np.where(small, SMALL * v, v)
        sp = [W.Markers1D(-1.0, 1.0, x, v, None, L / n)]
    elif kind == "weights":
        sp = [W.Markers1D(-1.0, 1.0, x, v, np.where(small, SMALL * w, w), 0.0)]
    elif kind == "species":
        sp = [W.Markers1D(-1.0, 1.0, x[~small], v[~small], None, L / n),
              W.Markers1D(1.0, 20.0, x[small], 0.3 * v[small], None, SMALL * L / n)]
    else:
        sp = [W.Markers1D(-1.0, 1.0, x, v, w, 0.0)]
    return W.Problem1D("scales", L, nc, order, 0.05 if nc < 500 else 0.005, 0, sp)


@pytest.mark.parametrize("n,nc", [(601, 64), (200_001, 300), (20_001, 1792)])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("kind", ["speeds", "weights", "species"])
def test_1d1v(kind, scheme, order, n, nc):
    prob = _problem(kind, n, nc, order)
    E0, at = np.zeros(nc), _part(nc)
    ref = oracle_run(prob, scheme, 3, remove_mean=False, E0=E0)["E"]
    got = gpu_run(prob, scheme, 3, remove_mean=False, E0=E0)["E"]
    assert 0.0 < np.abs(ref[at]).max() < 1e-9
    assert np.abs(got - ref)[at].max() <= 1e-11 * np.abs(ref[at]).max()
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
def test_heavy_marker_on_its_way(scheme, order):
    """One heavy marker crosses nodes of light ones: what it adds to a node comes above
    the node's scale, and the scale it leaves there falls again.  Each node's field is
    judged by itself: what the heavy marker left is exact to its own rounding, the nodes
    ahead of it hold the light markers' currents."""
    rng = np.random.default_rng(5)
    n, nc, L = 40_001, 100, 2 * np.pi
    x, v, w = rng.uniform(0, L, n), 0.1 * rng.standard_normal(n), np.full(n, SMALL * L / n)
    x[0], v[0], w[0] = 0.105 * L, 10.0, L
    prob = W.Problem1D("heavy", L, nc, order, 0.01, 0, [W.Markers1D(-1.0, 1.0, x, v, w, 0.0)])
    ref = oracle_run(prob, scheme, 8, remove_mean=False, E0=np.zeros(nc))["E"]
    got = gpu_run(prob, scheme, 8, remove_mean=False, E0=np.zeros(nc))["E"]
    ahead = np.arange(nc) > 40
    assert np.abs(got - ref)[ahead].max() <= 1e-11 * np.abs(ref[ahead]).max()
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
def test_fast_marker_among_slow_ones(scheme, order):
    """One marker crosses a fifth of the domain in a step: the nodes that it does not
    deposit to (its cells and their neighbours in every pass) hold the slow markers'
    currents alone."""
    rng = np.random.default_rng(6)
    n, nc, L, dt, steps = 40_001, 400, 2 * np.pi, 0.01, 3
    x, v = rng.uniform(0, L, n), SMALL * rng.standard_normal(n)
    x[0], v[0] = 0.1013 * L, 0.2 * L / dt
    prob = W.Problem1D("fast", L, nc, order, dt, 0, [W.Markers1D(-1.0, 1.0, x, v, None, 1e-9 * L / n)])
    ref = oracle_run(prob, scheme, steps, remove_mean=False, E0=np.zeros(nc))["E"]
    got = gpu_run(prob, scheme, steps, remove_mean=False, E0=np.zeros(nc))["E"]
    there = (0.1013 + 0.1 * np.arange(2 * steps + 3)) * nc     # x^n and x^{n+1/2}
    away = np.abs((np.arange(nc)[:, None] - there + nc / 2) % nc - nc / 2).min(axis=1) > 3
    assert 0.0 < np.abs(ref[away]).max() < 1e-20
    assert np.abs(got - ref)[away].max() <= 1e-11 * np.abs(ref[away]).max()


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("n,cells", [(30_001, 64), (30_001, 256)])
def test_1d2v(n, cells, scheme, order):
    """Ey, whose update is the node's own jy (the oracle transforms it with the rest, so
    the deposit is numpy's): without fields v* = v^n to 1e-12 of it (weights of 1e-9)
    and Ey after one step is -dt times the deposit at y + dt/2 vy.  The small half has
    small vy only, so that the two components' scales differ."""
    rng = np.random.default_rng(n + cells)
    L, dt, w0 = 10.0, 0.02, 1e-9 * 10.0 / n
    y = L * np.where(np.arange(n) % 2, rng.uniform(0.1, 0.4, n), rng.uniform(0.6, 0.9, n))
    small = y > L / 2
    vx, vy = 0.3 * rng.standard_normal(n), 0.1 * rng.standard_normal(n)
    vy = np.where(small, SMALL * vy, vy)
    prob = W.Problem1D2V("scales", L, cells, order, dt, 1.0, 0, np.zeros((2, cells)),
                         np.zeros(cells), [W.Markers1D2V(-1.0, 1.0, y, vx, vy, None, w0)])
    h = L / cells
    xi = (y + 0.5 * dt * vy) / h
    jy = np.zeros(cells)
    if order == 1:
        i = np.floor(xi).astype(int)
        d = xi - i
        shape = ((0, 1 - d), (1, d))
    else:
        i = np.floor(xi + 0.5).astype(int)
        d = xi - i
        shape = ((-1, 0.5 * (0.5 - d) ** 2), (0, 0.75 - d * d), (1, 0.5 * (0.5 + d) ** 2))
    for k, s in shape:
        np.add.at(jy, (i + k) % cells, -w0 / h * vy * s)
    ref, got, at = -dt * jy, _gpu_run(prob, O.CN, scheme, 1)[1][1], _part(cells)
    assert 0.0 < np.abs(ref[at]).max() < 1e-20
    assert np.abs(got - ref)[at].max() <= 1e-11 * np.abs(ref[at]).max()
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n,nc", [(601, 64), (60_001, 256)])
def test_standard(n, nc, order):
    prob = _problem("weights", n, nc, order)
    std._compare(prob, std._oracle(prob, 1, 4), std._gpu(prob, 1, 4))


@pytest.mark.parametrize("n,nc", [(601, 64), (60_001, 300), (9_001, 1792)])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("kind", ["adjoints", "species"])
def test_reverse(kind, scheme, order, n, nc):
    prob = _problem(kind, n, nc, order)
    at, N = _part(nc), prob.n_markers
    rng = np.random.default_rng(2)
    x = np.concatenate([s.x for s in prob.species])
    seed = np.where(x > prob.L / 2, SMALL, 1.0)
    xb, vb = seed * rng.standard_normal(N), seed * rng.standard_normal(N)
    Eb = np.where((np.arange(nc) > 0.05 * nc) & (np.arange(nc) < 0.48 * nc), 1.0, SMALL)
    Eb = Eb * rng.standard_normal(nc)
    cfg = O.ES1DConfig(nc=nc, L=prob.L, order=order, dt=prob.dt, scheme=scheme, remove_mean=False)
    cut = np.cumsum([len(s.x) for s in prob.species])[:-1]
    ref = O.es1d_grad(cfg, [O.Species(s.q, s.m, s.x, s.v, s.w, s.w0) for s in prob.species],
                      np.zeros(nc), 3, Eb, np.split(xb, cut), np.split(vb, cut))[0]
    from paper_2411_09605_gb300 import pic
    sim = pic.Simulation(prob, scheme=scheme, E0=np.zeros(nc), remove_mean=False)
    try:
        pic.pic_grad_forward(sim.h, 3, 2)
        got = np.zeros(nc)
        pic.pic_grad_backward(sim.h, Eb, xb, vb, got, None, None, None)
    finally:
        sim.close()
    assert 0.0 < np.abs(ref[at]).max() < 1e-9
    assert np.abs(got - ref)[at].max() <= 1e-9 * np.abs(ref[at]).max()
    assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()
