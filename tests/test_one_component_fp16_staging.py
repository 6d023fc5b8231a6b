"""The read-out and the initial fields pass through the population buffer that
is free, five FP64 values a site, whichever of the two it is: after an odd
number of steps it is the first one.  The smallest form, one component in FP16,
holds 38 bytes of populations a site in a buffer."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities

SHAPE = (44, 21, 19)


def test_both_buffers_hold_the_staged_values():
    from paper_2004_04080_gb300 import lbgb

    for n in (32, 64, 200):
        size = lbgb.lb_workspace_bytes(n, n, n, lbgb.LB_FP16 | lbgb.LB_ONE_COMPONENT, 0)
        assert size >= 2 * 5 * 8 * n ** 3
    # the other forms hold more than that in their populations already
    n = 64
    for prec in (lbgb.LB_FP16, lbgb.LB_FP32, lbgb.LB_FP32 | lbgb.LB_ONE_COMPONENT):
        assert lbgb.lb_workspace_bytes(n, n, n, prec, 0) >= 2 * 5 * 8 * n ** 3


def lattice(prec, fields):
    from paper_2004_04080_gb300.lbgb import LBLattice

    g = LBLattice(SHAPE, prec, components=1)
    g.set_params(rho0=(1.0, 0.0), bc=(1, 1, 0), wall_u_lo=(0.01, 0.0, 0.0))
    g.init_fields(*fields)
    return g


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp16", "fp32"])
@pytest.mark.parametrize("steps", [1, 2, 3])
def test_reading_leaves_the_state(steps, prec):
    rng = np.random.Generator(np.random.PCG64(3))
    n = int(np.prod(SHAPE))
    fields = (mixture_densities(SHAPE, seed=5, amp=0.02)[0], None, 0.02 * (rng.random((3, n)) - 0.5))
    g, h = lattice(prec, fields), lattice(prec, fields)
    for _ in range(3):
        g.step(steps)
        h.step(steps)
        first = g.get_fields()
        again = g.get_fields()
        assert all(np.array_equal(a, b) for a, b in zip(first, again))
    assert np.array_equal(g.populations(0), h.populations(0))
    g.init_fields(*fields)
    h = lattice(prec, fields)
    assert np.array_equal(g.populations(0), h.populations(0))
