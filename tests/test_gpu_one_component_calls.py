"""Which calls on the one-component lattice keep moments between their steps
(those that advance enough sites to gain by it): the others are the same bits
as calls of one step; those that do, at sides where the march can go wrong,
against the oracle."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities
from test_gpu_single import _run, rel

pytestmark = pytest.mark.gpu

ENOUGH = 3 << 18


def lattice(shape, prec):
    from paper_2004_04080_gb300.lbgb import LBLattice

    g = LBLattice(shape, prec, components=1)
    g.set_params(rho0=(1.0, 0.0), bc=(1, 1, 0), wall_u_lo=(0.01, 0.0, 0.0))
    g.init_fields(mixture_densities(shape, seed=5, amp=0.02)[0], None)
    return g


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("shape,steps", [((32, 32, 32), 2), ((36, 16, 16), 20), ((4, 4, 512), 30), ((64, 64, 64), 3)])
def test_small_calls_keep_populations(shape, steps, prec):
    assert (steps - 1) * np.prod(shape) < ENOUGH
    g, o = lattice(shape, prec), lattice(shape, prec)
    g.step(steps)
    for _ in range(steps):
        o.step(1)
    assert np.array_equal(g.populations(0), o.populations(0))


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp16", 1e-3)])
@pytest.mark.parametrize("shape", [(4, 9, 400), (28, 9, 70), (32, 8, 66), (36, 12, 43), (60, 17, 18), (56, 33, 9)])
def test_large_calls(shape, prec, tol):
    """As test_gpu_single's runs: walls, a body force, a random velocity."""
    steps = 60
    assert (steps - 1) * np.prod(shape) >= ENOUGH
    params = dict(tau=(1.0, 1.0), rho0=(1.0, 0.0), bc=(1, 1, 0), wall_u_lo=(-0.03, 0.01, 0), wall_u_hi=(0.02, 0, 0),
                  body_force=(2e-5, 0, -1e-5))
    g, o = _run(shape, params, steps, prec)
    (ga, _, gu), (ra, _, ru) = g.get_fields(), o.get_fields()
    assert rel(ga, ra) < tol
    assert rel(gu, ru, floor=1.0 if prec == "fp16" else 0.03) < tol


@pytest.mark.parametrize("gravity,steps", [(0.1, 20)])
def test_atmosphere(gravity, steps):
    """rho ~ exp(-3 g z) between walls, a tenth of a per cent to 1, in a call
    that keeps moments: the error relative to each site's own density stays
    below the form's bound."""
    from oracle import Oracle
    from paper_2004_04080_gb300.lbgb import LBLattice

    shape = (60, 36, 20)
    assert (steps - 1) * np.prod(shape) >= ENOUGH
    z = np.repeat(np.arange(shape[2]), shape[0] * shape[1])
    a = np.exp(-3.0 * gravity * z) * (1.0 + 0.05 * np.random.default_rng(1).random(z.size))
    params = dict(tau=(1.0, 1.0), rho0=(1.0, 0.0), bc=(1, 1, 0), body_force=(0.0, 0.0, -gravity))
    g, o = LBLattice(shape, "fp32", components=1), Oracle(*shape, 0)
    g.set_params(**params)
    o.set_params(**params)
    g.init_fields(a, None)
    o.init_fields(a, np.zeros_like(a))
    g.step(steps)
    o.step(steps)
    (ga, _, gu), (ra, _, ru) = g.get_fields(), o.get_fields()
    assert np.abs(ga / ra - 1.0).max() < 1e-5
    assert np.abs(gu - ru).max() < 1e-5


@pytest.mark.parametrize("face", [0, 1])
def test_drained_site_is_reported(face):
    from paper_2004_04080_gb300.lbgb import LBError, LBLattice

    shape = (128, 64, 100)
    g = LBLattice(shape, "fp32", components=1)
    walls = dict(wall_u_lo=(0.0, 0.0, -2.0)) if face == 0 else dict(wall_u_hi=(0.0, 0.0, 2.0))
    g.set_params(bc=(1, 1, 0), open=(2, 0) if face == 0 else (0, 2), **walls)
    g.init_fields(mixture_densities(shape, seed=5, amp=0.01)[0], None)
    with pytest.raises(LBError, match="negative density"):
        g.step(2)
