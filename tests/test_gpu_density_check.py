"""A density that turns negative in any step of a call is reported by that
call (LB_ERR_NONFINITE), however the steps are split into calls: at a z face
whose links carry more out of a site than it holds (Eq. 9 with an outward
normal velocity u: rho' = rho (1 - u) + what streams in), and at a particle
whose surface moves faster than the fluid can follow (Eq. 17).  A call of two
steps at tau = 1 forms the densities of its first step by the moment kernels
and reads none of them back from populations."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities

pytestmark = pytest.mark.gpu

SHAPE = (32, 13, 12)


def raises(g, calls):
    from paper_2004_04080_gb300.lbgb import LBError

    with pytest.raises(LBError, match="negative density"):
        for n in calls:
            g.step(n)


@pytest.mark.parametrize("calls", [(2,), (1, 1), (3,)])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("components,face", [(2, 0), (2, 1), (1, 0), (1, 1)])
def test_z_face(components, face, prec, calls):
    from paper_2004_04080_gb300.lbgb import LBLattice

    g = LBLattice(SHAPE, prec, components=components)
    walls = dict(wall_u_lo=(0.0, 0.0, -2.0)) if face == 0 else dict(wall_u_hi=(0.0, 0.0, 2.0))
    g.set_params(G=0.1, bc=(1, 1, 0), open=(2, 0) if face == 0 else (0, 2), **walls)
    a, b = mixture_densities(SHAPE, seed=5, amp=0.01)
    g.init_fields(a, b if components == 2 else None)
    raises(g, calls)


@pytest.mark.parametrize("calls", [(2,), (1, 1), (3,)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_particle_surface(prec, walls, calls):
    from paper_2004_04080_gb300.lbgb import LBLattice

    g = LBLattice(SHAPE, prec, max_colloids=1)
    g.set_params(G=0.1, **(dict(bc=(1, 1, 0)) if walls else {}))
    g.init_fields(*mixture_densities(SHAPE, seed=5, amp=0.01))
    # surface speed 3 R: a link takes up to 6 w_i rho |c_i . u_w| out of a site
    g.add_colloids(pos=[[16.3, 6.2, 3.6]], radius=[3.3], mass=[1e15], omega=[[0.0, 0.0, 3.0]])
    raises(g, calls)


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
def test_full_sums_are_judged(prec):
    """A site at a wall that hands back all it takes holds its density: the
    sum without the returned links is not judged."""
    from paper_2004_04080_gb300.lbgb import LBLattice

    g = LBLattice(SHAPE, prec, max_colloids=1)
    g.set_params(G=0.1, bc=(1, 1, 0))
    a, b = mixture_densities(SHAPE, seed=5, amp=0.01)
    g.init_fields(a, b)
    g.add_colloids(pos=[[16.3, 6.2, 3.6]], radius=[3.3], mass=[1e15])
    g.step(20)
    ga, gb, _ = g.get_fields()
    fluid = g.owner() < 0
    assert np.all(ga[fluid] > 0.0) and np.all(gb[fluid] > 0.0)
