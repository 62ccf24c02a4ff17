"""Gridded A^T where the trajectory dwells: thousands of spreading units in one
tile of the node grid, with terms of one sign, so that the order and precision
of their sum decide.

Tolerances: 2e-7 where the terms differ (a unit's chains are off by 1.1e-7 in
the mean square, independently from unit to unit; the transforms leave up to
1.5e-7 of so concentrated an image; the units are added in pairs of floats),
1e-6 where they are all equal (a chain of 112 equal terms is off by 8e-7 in the
mean square over their sizes, the same in every unit; pair sums: 1.6e-6)."""
import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded

pytestmark = pytest.mark.gpu
F32 = torch.float32


@pytest.mark.parametrize("T", [1 << 16, 1 << 20])
@pytest.mark.parametrize("rest", [False, True])
def test_dwelling_samples_of_one_sign(orc, T, rest):
    """All samples within a node's width of one point, or resting on it, with
    positive data and a common direction of motion."""
    rng = np.random.default_rng(T + rest)
    m, g = syn.default_model(n_ch=1), syn.square_grid(40, 24.0, 36)
    r = np.array([1.7, -2.3]) + (0.0 if rest else 0.02) * rng.uniform(-1, 1, size=(T, 2))
    v = np.tile([3.0e3, 1.0e3], (T, 1))
    s = np.ones((1, T)) if rest else rng.uniform(0.5, 1.5, size=(1, T))
    r, v, s = (rounded(x, F32) for x in (r, v, s))
    n0 = api.mpi_kernel_launches()
    got = api.mpi_adjoint(m, g, dev(r, F32), dev(v, F32), dev(s, F32))
    assert api.mpi_kernel_launches() - n0 >= 8  # gridded (pair sums: five at most)
    assert rel_l2(host(got), orc.adjoint(m, g, r, v, s)) <= (1e-6 if rest else 2e-7)
