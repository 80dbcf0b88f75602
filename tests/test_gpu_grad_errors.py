"""Errors of the steps that pic_grad_forward takes: the handle is left at the last step
that was reached, as by pic_step, and pic_grad_backward refuses it."""
import numpy as np
import pytest

from paper_2411_09605_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def _raises(f, *a):
    from paper_2411_09605_gb300 import pic
    with pytest.raises(pic.PicError):
        f(*a)


@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("every", [1, 100, 2000])
def test_forward_error_leaves_a_consistent_state(every, scheme):
    """A marker that crosses several periods a step is reported when the step counters
    are full (1024 steps); its steps are defined all the same."""
    from paper_2411_09605_gb300 import pic
    prob = W.landau(n=300, nc=16, order=2, dt=1e-3, seed=3)
    prob.species[0].v[7] = 2.5 * prob.L / prob.dt
    sims = [pic.Simulation(prob, scheme=scheme) for _ in range(2)]
    try:
        _raises(pic.pic_grad_forward, sims[0].h, 1500, every)
        _raises(sims[1].step, 1024)
        for more in (0, 3):
            if more:
                for s in sims:
                    _raises(s.step, more)
            assert pic.pic_step_count(sims[0].h) == pic.pic_step_count(sims[1].h) == 1024 + more
            for a, b in zip((*sims[0].particles(), sims[0].field()),
                            (*sims[1].particles(), sims[1].field())):
                # (1e3 steps of a smooth problem; the sums' order is free)
                assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
        out = np.zeros(prob.nc)
        _raises(pic.pic_grad_backward, sims[0].h, None, None, np.ones(300), out, None, None, None)
        assert not out.any()
    finally:
        for s in sims:
            s.close()


@pytest.mark.parametrize("device", [False, True])
def test_backward_reports_the_last_step(device):
    """An energy that overflows in the last forward step, whose stats were not read: the
    reverse reports it and leaves the outputs as they are."""
    import torch
    from paper_2411_09605_gb300 import pic
    prob = W.landau(n=50, nc=8, dt=1e-6, seed=4)
    prob.species[0].w0 = 1e300
    sim = pic.Simulation(prob, scheme=1, E0=np.zeros(8))
    out = [torch.full((k,), 7.0, dtype=torch.float64, device="cuda" if device else "cpu")
           for k in (8, 50, 50, 50)]
    try:
        pic.pic_grad_forward(sim.h, 1, 1)
        torch.cuda.synchronize()
        with pytest.raises(pic.PicError) as e:
            pic.pic_grad_backward(sim.h, None, None, np.ones(50), *out)
        assert pic.ERRORS[e.value.code] == "PIC_ERR_NONFINITE"
        assert all(bool((t == 7.0).all()) for t in out)
    finally:
        sim.close()
