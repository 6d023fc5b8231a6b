"""Calls of one step at tau = 1: density pass, lean kernel and the kernel of the
z faces in every step, with every kind of face, with and without
extrapolation, with moving particles, in each storage form, against the
oracle at the bounds of the forms.  (A call of several steps runs these kernels
in its first and last step only.)"""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities
from test_gpu_parity import compare_colloids, compare_fields, run_both

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp16": 1e-3}
SHAPE = (36, 13, 11)
FACES = {
    "periodic": dict(),
    "walls": dict(bc=(1, 1, 0), wall_u_lo=(-0.03, 0.01, 0.0), wall_u_hi=(0.04, 0.0, 0.0)),
    "pressure_equilibrium": dict(bc=(1, 1, 0), open=(1, 3), open_rho=(0.52, 0.5, 0.5, 0.48)),
    "velocity_pressure": dict(bc=(1, 1, 0), open=(2, 1), wall_u_lo=(0.0, 0.0, 0.01), open_rho=(0.5, 0.5, 0.5, 0.49)),
    "velocity_pressure_extrapolated": dict(bc=(1, 1, 0), open=(2, 1), wall_u_lo=(0.0, 0.0, 0.01),
                                           open_rho=(0.5, 0.5, 0.5, 0.49), open_extrap=1),
}


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("particles", [False, True])
@pytest.mark.parametrize("faces", sorted(FACES))
def test_calls_of_one_step(faces, particles, prec):
    col = None
    if particles:
        col = dict(pos=[[9.3, 6.2, 5.1], [25.6, 7.4, 6.3]], radius=[2.6, 2.4], mass=[400.0, 300.0],
                   vel=[[0.02, 0.01, 0.01], [-0.02, 0.0, 0.01]], omega=[[0.0, 0.01, 0.0], [0.01, 0.0, 0.02]])
    rng = np.random.Generator(np.random.PCG64(3))
    u = 0.02 * (rng.random((3, int(np.prod(SHAPE)))) - 0.5)
    params = dict(G=0.5, zeta=(0.1, -0.1), body_force=(1e-5, 0.0, -1e-5), **FACES[faces])
    g, o = run_both(SHAPE, params, 1, prec, col, mixture_densities(SHAPE, seed=17, amp=0.03), u)
    assert g.fused_kernel() == "k_lean"
    for _ in range(14):
        g.step(1)
        o.step(1)
    compare_fields(g, o, TOL[prec])
    if particles:
        compare_colloids(g, o, TOL[prec])
