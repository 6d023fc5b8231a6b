"""The particle kernels at the edges of their ranges, against the oracle."""
import numpy as np
import pytest

from paper_2004_04080_gb300.workloads import mixture_densities
from test_gpu_parity import run_both

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
