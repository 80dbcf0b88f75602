"""The FP64 moment passes (gather by polynomials, deposit by moments; 1D1V, then
1D2V, the standard scheme and 2D3V)
against the oracle at the edges of their ranges: the smallest grid, the last
grid they take and the first that runs the general passes; one marker, a ragged
warp, the marker counts where the block size changes (128, 256 and 512 threads),
several trips; one uniform species, weighted markers and two species.

Bar: the FP64 form's 1e-11 after a few steps (double arithmetic on both sides,
differences of order 1e-16 per operation and marker, amplified at most by the
few steps), fallback counts equal."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_09605_gb300 import workloads as W
from tests import test_gpu_em2d as yee, test_gpu_standard as std
from tests.parity_util import compare, gpu_run, oracle_run
from tests.test_gpu_em1d import _compare, _gpu_run, _oracle_run

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def _check(prob, scheme, steps=4):
    ref, got = oracle_run(prob, scheme, steps), gpu_run(prob, scheme, steps)
    d = compare(prob, ref, got)
    assert max(d.values()) <= TOL, d
    assert np.array_equal(ref["nfb"], got["nfb"])


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("n,nc", [(1, 4), (33, 5), (1000, 1792), (1000, 1793), (303 * 128, 33),
                                  (303 * 128 + 1, 64), (303 * 256 + 1, 300), (400_003, 100)])
def test_sizes(n, nc, order, scheme):
    _check(W.landau(n=n, nc=nc, order=order, seed=n + nc), scheme)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
def test_weighted_and_two_species(order, scheme):
    _check(W.bump_on_tail(n=50_001, nc=96, order=order, seed=8), scheme)
    prob = W.landau(n=20_001, nc=48, order=order, seed=9)
    ions = W.landau(n=7_000, nc=48, order=order, seed=10, vth=0.1).species[0]
    ions.q, ions.m = 1.0, 100.0
    prob.species.append(ions)
    _check(prob, scheme)


@pytest.mark.parametrize("order", [1, 2])
def test_every_marker_in_one_cell(order):
    """One node's sums take every marker of a block (one tile copy on this grid): the
    high words of the fixed-point sums fill and are emptied on the way."""
    prob = W.landau(n=1_200_000, nc=1792, order=order, seed=11)
    s = prob.species[0]
    h = prob.L / prob.nc
    s.x = (7.0 + 0.9 * np.random.default_rng(1).random(len(s.x))) * h
    s.v = 3.0 + 0.1 * s.v
    s.w0 *= 1e-4
    _check(prob, 2, steps=2)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
def test_cold_start_and_one_fast_marker(order, scheme):
    """Amounts above the previous pass's largest: markers that start at rest (every
    amount of the first pass), and a marker that a strong field accelerates."""
    prob = W.landau(n=30_000, nc=64, order=order, seed=12, vth=0.0, alpha=0.3)
    _check(prob, scheme)
    prob = W.landau(n=30_000, nc=64, order=order, seed=13, vth=1e-9, alpha=0.3)
    prob.species[0].v[17] = 2.0
    _check(prob, scheme)


@pytest.mark.parametrize("solver", [O.CN, O.PSATD])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n,ppc,scheme", [(4, 7, 2), (4, 40_000, 1), (64, 33, 2), (64, 2_500, 1),
                                          (128, 33, 2), (1024, 11, 2)])
def test_spectral_sizes(n, ppc, scheme, order, solver):
    """1D2V: the smallest grid (a block of one warp; a response sum that fills part of
    a warp), the last grid of the direct field solve and the first of the transforms,
    the largest; one block, one and two blocks per SM."""
    prob = W.weibel_1d2v(n=n, ppc=ppc, k0=0.5, b=0.02, order=order, seed=n + ppc)
    _compare(prob, _oracle_run(prob, solver, scheme, 3), _gpu_run(prob, solver, scheme, 3))


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n,nc,passes", [(1, 4, 0), (33, 4, 1), (20_001, 64, 2), (152 * 512 + 1, 512, 0),
                                         (30_000, 4096, 1)])
def test_standard_sizes(n, nc, passes, order):
    """The standard scheme's passes and field solve: the smallest grid (nodes fill part of a
    block's warps) and the largest, one marker, the marker count where a second block per SM
    starts."""
    prob = W.landau(n=n, nc=nc, order=order, dt=0.05, seed=n + nc)
    std._compare(prob, std._oracle(prob, passes, 4), std._gpu(prob, passes, 4))


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("nx,ny,n", [(4, 5, 40), (33, 9, 45), (64, 40, 30_001), (31, 8, 120_000)])
def test_yee_sizes(nx, ny, n, scheme, order):
    """2D3V: grids that leave the tiles of the grid kernels ragged in both directions, part
    of a warp, one and several trips a block."""
    prob = W.weibel(nx=nx, ny=ny, ppc=-(-n // (nx * ny)), order=order, seed=n)
    s = prob.species[0]
    for k in ("x", "y", "vx", "vy", "vz"):
        setattr(s, k, np.ascontiguousarray(getattr(s, k)[:n]))
    s.w0 = prob.Lx * prob.Ly / n
    yee._check(prob, scheme, steps=3)


@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("order,nx,ny,n", [(1, 150, 130, 5552), (1, 150, 130, 5553),
                                           (2, 65, 64, 65_799), (2, 65, 64, 65_800)])
def test_yee_line_between_the_passes(order, nx, ny, n, scheme):
    """2D3V: the most markers that the general passes take on a grid and the fewest
    of the moment passes."""
    test_yee_sizes(nx, ny, n, scheme, order)
