"""The particle kernels at the edges of their ranges, against the oracle."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities
from test_gpu_parity import compare_colloids, compare_fields, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33])
@pytest.mark.parametrize("spin", [0.0, 1e-9, 0.1, 0.8])
def test_orientation_closed_form(spin, n):
    """The closed form of the implicit mid-step (Eqs. 33-34) against the
    oracle's iteration, which stops when the rate changes by 1e-14 or less; the
    iteration contracts by |omega| / 4, so its rest is below 0.8 / 4 / (1 - 0.8 / 4)
    x 1e-14 a step, and 1e-13 covers three steps and their rounding.  Heavy
    particles keep their spin; one block of 32 particles, one less and one more."""
    rng = np.random.Generator(np.random.PCG64(7))
    shape = (24, 24, 16)
    cells = np.stack(np.meshgrid(range(6), range(6), range(4), indexing="ij"), -1).reshape(-1, 3)[:n]
    axis = rng.standard_normal((n, 3))
    quat = rng.standard_normal((n, 4))
    col = dict(pos=4.0 * cells + 1.37, radius=np.full(n, 1.2), mass=np.full(n, 1e15),
               omega=spin * axis / np.linalg.norm(axis, axis=1)[:, None],
               quat=quat / np.linalg.norm(quat, axis=1)[:, None])
    g, o = run_both(shape, dict(G=0.3), 3, "fp64", col, mixture_densities(shape, seed=3, amp=0.02))
    gc, rc = g.get_colloids(), o.get_colloids()
    assert np.abs(gc["quat"] - rc["quat"]).max() < 1e-13
    assert np.abs(np.linalg.norm(gc["quat"], axis=1) - 1.0).max() < 1e-15


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("calls", [(8,), (1,) * 8])
@pytest.mark.parametrize("speed", [0.0, 0.02, 0.45])
def test_remap_shell(speed, calls, prec, tol):
    """Only nodes within |v| of a surface are looked at after the first step of
    a call: slow and nearly fastest particles, across the periodic edges and
    next to a wall, in one call and in calls of one step.  Bounds of the forms;
    the node maps are equal."""
    shape = (28, 19, 23)
    vel = speed * np.array([[1.0, 0.0, 0.0], [-0.6, 0.0, 0.8], [0.0, -0.8, 0.6], [0.577, 0.577, -0.577]])
    col = dict(pos=[[26.9, 3.2, 4.6], [8.3, 4.1, 6.2], [7.7, 14.2, 17.3], [20.4, 12.9, 15.1]],
               radius=[3.1, 2.5, 3.4, 2.9], mass=[1e6] * 4, vel=vel, omega=[[0.0, 0.02, 0.01]] * 4)
    params = dict(G=0.3, zeta=(0.05, -0.05), bc=(1, 1, 0))
    dens = mixture_densities(shape, seed=5, amp=0.02)
    g, o = run_both(shape, params, calls[0], prec, col, dens)
    for n in calls[1:]:
        g.step(n)
        o.step(n)
    compare_fields(g, o, tol)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_overlap_is_reported_by_every_call(prec):
    """Particles that have run into each other are reported by the call in
    which they meet and by the ones after it."""
    from paper_2004_04080_gb300.lbgb import LBError, LBLattice

    g = LBLattice((24, 16, 16), prec, max_colloids=2)
    g.set_params(G=0.0)
    g.init_fields(*mixture_densities((24, 16, 16), seed=5, amp=0.0))
    g.add_colloids(pos=[[7.5, 8.1, 8.2], [14.9, 8.1, 8.2]], radius=[3.5, 3.5], mass=[1e6, 1e6],
                   vel=[[0.1, 0.0, 0.0], [0.0, 0.0, 0.0]])
    with pytest.raises(LBError):
        g.step(12)
    for _ in range(2):
        with pytest.raises(LBError):
            g.step(1)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(12, 12, 11), (32, 13, 12), (36, 12, 13), (32, 40, 33)])
def test_lean_short_marches(shape, walls, prec, tol):
    """Calls of one step on lattices whose lean kernel takes marches of two or
    a few planes, of which the last may be shorter, with a particle across
    several of them.  Bounds of the forms."""
    col = dict(pos=[[s / 2 + 0.3 for s in shape]], radius=[2.7], mass=[300.0], vel=[[0.03, -0.02, 0.01]],
               omega=[[0.0, 0.01, 0.02]])
    params = dict(G=0.4, zeta=(0.05, -0.05), bc=(1, 1, 0 if walls else 1))
    g, o = run_both(shape, params, 1, prec, col, mixture_densities(shape, seed=9, amp=0.05))
    for _ in range(5):
        g.step(1)
        o.step(1)
    compare_fields(g, o, tol)
    compare_colloids(g, o, tol)
