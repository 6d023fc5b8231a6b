"""The checkpoints of AdjointRunner.forward and the steps its reverse sweep
recomputes from them are the same states, bit for bit: at tau = 1 the steps of
a call that does not record keep moments instead of populations between them,
which rounds differently."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("particles", [0, 1])
@pytest.mark.parametrize("tau", [1.0, 0.9])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_recomputed_steps_meet_the_checkpoints(prec, tau, particles):
    from paper_2004_04080_gb300 import lbgb
    from paper_2004_04080_gb300.adjoint import AdjointRunner
    from paper_2004_04080_gb300.lbgb import LBLattice

    shape = (20, 14, 12)
    lat = LBLattice(shape, prec, max_colloids=1)
    run = AdjointRunner(lat, 11, checkpoint_every=4)
    col = dict(pos=[[9.3, 6.2, 5.1]], radius=[2.6]) if particles else None
    run.forward(dict(G=0.9, tau=(tau, tau)), *mixture_densities(shape, seed=13, amp=0.05), col)
    assert sorted(run.checkpoints) == [0, 4, 8, 11]
    for start, end in ((0, 4), (4, 8), (8, 11)):
        lbgb.lb_set_state(lat.h, run.checkpoints[start].data_ptr())
        lbgb.lb_record(lat.h, run.stack.data_ptr(), None, end - start)
        lat.step(end - start)
        f = [lat.populations(k) for k in (0, 1)]  # (a state has padding too)
        lbgb.lb_set_state(lat.h, run.checkpoints[end].data_ptr())
        assert all(np.array_equal(f[k], lat.populations(k)) for k in (0, 1))


def test_gradient_is_that_of_the_recomputed_run():
    """Without particles at tau = 1: the objective of the forward run equals,
    bit for bit, that of the same steps taken one call each."""
    from paper_2004_04080_gb300 import lbgb
    from paper_2004_04080_gb300.adjoint import AdjointRunner
    from paper_2004_04080_gb300.lbgb import LBLattice

    shape = (20, 14, 12)
    a, b = mixture_densities(shape, seed=13, amp=0.05)
    lat = LBLattice(shape, "fp32")
    run = AdjointRunner(lat, 10)
    _, value = run.forward(dict(G=0.9), a, b, None)
    one = LBLattice(shape, "fp32")
    one.set_params(G=0.9)
    one.init_fields(a, b)
    for _ in range(10):
        one.step(1)
    assert value == lbgb.lb_adjoint_seed(one.h, 0.0, run.adj[0].data_ptr(), run.scratch.data_ptr())
    assert np.isfinite(value)
