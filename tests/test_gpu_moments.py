"""Calls of several steps at tau = 1, which keep rho^k and j between the steps
(lbgb_moment.cu), against the oracle at the sizes where the march can go
wrong: a row of 28 sites and one more or fewer, rows that close on themselves
(nx = 32), the smallest sides, blocks of 8 rows with an odd or a single row
left, one to a few planes per block, walls, and particles across the edges of
the blocks, in contact (sites next to two particles).  Bounds: those of the
forms (FP32 1e-5, FP16 1e-3), velocities relative to the lattice speed."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities
from test_gpu_parity import compare_colloids, compare_fields, run_both

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp16": 1e-3}
WALLS = dict(bc=(1, 1, 0), wall_u_lo=(-0.03, 0.01, 0.0), wall_u_hi=(0.04, 0.0, 0.0))


def velocity(shape, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return 0.02 * (rng.random((3, int(np.prod(shape)))) - 0.5)


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(4, 4, 4), (28, 8, 5), (32, 9, 6), (36, 7, 12), (56, 17, 4), (60, 5, 33)])
def test_fluid(shape, walls, prec):
    params = dict(G=0.6, body_force=(2e-5, 0.0, -1e-5), **(WALLS if walls else {}))
    g, o = run_both(shape, params, 9, prec, dens=mixture_densities(shape, seed=17, amp=0.05),
                    u=velocity(shape, 3))
    compare_fields(g, o, TOL[prec])


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("shape,tau", [((4, 4, 4), 1.0), ((28, 9, 5), 1.0), ((32, 8, 7), 1.0), ((60, 17, 6), 1.0)])
def test_one_component(shape, tau, prec):
    from test_gpu_single import _run, rel

    params = dict(tau=(tau, tau), rho0=(1.0, 0.0), body_force=(2e-5, 0, -1e-5), **WALLS)
    g, o = _run(shape, params, 9, prec)
    (ga, _, gu), (ra, _, ru) = g.get_fields(), o.get_fields()
    assert rel(ga, ra) < TOL[prec]
    assert rel(gu, ru, floor=1.0) < TOL[prec]


@pytest.mark.parametrize("walls", [False, True])
def test_particles_across_block_edges(walls):
    """Particles at the column edge x = 28 and the row edge y = 8 of the
    blocks and across the periodic faces, two of them closer than two sites."""
    shape = (60, 21, 27)
    params = dict(G=0.5, zeta=(0.1, -0.1), hertz_K=20, hertz_sigma=8.0, hertz_rcap=7.0, **(WALLS if walls else {}))
    col = dict(pos=[[27.6, 7.8, 9.3], [34.9, 8.1, 9.6], [59.4, 20.3, 17.2], [14.2, 15.4, 12.9]],
               radius=[3.5, 3.4, 3.5, 3.1], mass=[400.0, 380.0, 400.0, 300.0],
               vel=[[0.03, 0.02, -0.01], [-0.02, 0.0, 0.02], [0.01, 0.03, 0.02], [0.0, -0.02, 0.01]],
               omega=[[0.0, 0.01, 0.0], [0.01, 0.0, 0.0], [0.0, 0.0, 0.02], [0.01, 0.01, 0.0]])
    g, o = run_both(shape, params, 15, "fp32", col, mixture_densities(shape, seed=19, amp=0.05), velocity(shape, 5))
    compare_fields(g, o, 1e-5)
    compare_colloids(g, o, 1e-5)


def test_one_call_or_many():
    """The state a call leaves is the populations: reading it out between
    calls and splitting a run into calls changes the rounding only, and the
    mass stays."""
    from paper_2004_04080_gb300.lbgb import LBLattice

    shape = (44, 19, 23)
    a, b = mixture_densities(shape, seed=23, amp=0.05)
    runs = []
    for calls in ([12], [1] * 12, [5, 1, 6]):
        g = LBLattice(shape, "fp32")
        g.set_params(G=0.6)
        g.init_fields(a, b, velocity(shape, 7))
        m0 = g.totals()
        for n in calls:
            g.step(n)
        f = g.populations(0)
        ga, _, gu = g.get_fields()
        assert np.abs(f.sum(axis=0) - ga).max() < 1e-6
        assert np.all(np.abs(g.totals()[:2] - m0[:2]) < 1e-6 * m0[:2])
        runs.append((f, gu))
    for f, u in runs[1:]:
        assert np.abs(f - runs[0][0]).max() < 1e-5 and np.abs(u - runs[0][1]).max() < 1e-5
