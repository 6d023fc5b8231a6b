"""A particle may move less than 1/2 along each axis in a step, so up to
sqrt(3)/2 along a diagonal: the node map follows it (against the oracle) however
the steps are split into calls, also where a node changes side further than 0.65
from the surface."""
import numpy as np
import pytest

from oracle import Oracle
from paper_2004_04080_gb300.workloads import mixture_densities

SHAPE = (32, 24, 20)
STEPS = 4
# one heavy particle: velocity, radius, position
CASES = [((0.4, 0.4, 0.4), 2.1, (16.67, 12.75, 10.94)), ((0.48, -0.47, 0.0), 3.1, (16.27, 12.96, 10.54)), ((-0.45, 0.2, -0.45), 2.3, (16.68, 12.21, 10.05))]


def far_changes(velocity, radius, pos):
    """Nodes that change side further than 0.65 from the surface after a move."""
    far = 0
    for t in range(1, STEPS):
        old, new = np.array(pos) + (t - 1) * np.array(velocity), np.array(pos) + t * np.array(velocity)
        g = np.stack(np.meshgrid(*[np.arange(np.floor(c - 6), c + 6) for c in new], indexing="ij"), -1).reshape(-1, 3)
        d0, d1 = np.linalg.norm(g - old, axis=1), np.linalg.norm(g - new, axis=1)
        far += int(np.sum(((d0 < radius) != (d1 < radius)) & (np.abs(d1 - radius) > 0.65)))
    return far


@pytest.mark.parametrize("velocity,radius,pos", CASES)
def test_cases_reach_beyond(velocity, radius, pos):
    assert all(abs(v) < 0.5 for v in velocity) and np.linalg.norm(velocity) > 0.65
    assert far_changes(velocity, radius, pos) >= 1


@pytest.mark.gpu
@pytest.mark.parametrize("calls", [(STEPS,), (1,) * STEPS, (2, 2)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("velocity,radius,pos", CASES)
def test_node_map(velocity, radius, pos, prec, calls):
    from paper_2004_04080_gb300.lbgb import LBLattice

    dens = mixture_densities(SHAPE, seed=5, amp=0.02)
    g, o = LBLattice(SHAPE, prec, max_colloids=1), Oracle(*SHAPE, 1)
    for x in (g, o):
        x.set_params(G=0.3)
        x.init_fields(*dens)
        x.add_colloids(pos=[pos], radius=[radius], mass=[1e9], vel=[velocity])
    for n in calls:
        g.step(n)
        o.step(n)
        assert np.array_equal(g.owner(), o.owner())
