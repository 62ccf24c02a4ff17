"""Shapes that only the gridded FP32 operators' less common code reaches, with
the route stated: both calls must have run on the grid (six and eight launches;
the pair sums take five at most).

Tolerance 1e-6, as derived in test_gpu_field.py."""
import pytest
import torch

from paper_2505_22797_gb300 import api
from tests.gpu_util import dev, host, rel_l2
from tests.test_gpu_field import TOL, _case

pytestmark = pytest.mark.gpu
F32 = torch.float32

CASES = [
    dict(nx=1, ny=700, T=400001),                        # one column of voxels
    dict(nx=16, ny=12, T=1200001),                       # few voxels, thousands of samples per run of the order
    dict(nx=300, ny=280, T=6001, fov=48.0),              # 1536 nodes per axis
    dict(nx=3, ny=1200, T=50001),                        # y box beyond 2048 voxels: columns in pairs
    dict(nx=40, ny=40, T=250001, aspect=4.0),            # y axis beyond 2048 nodes
    dict(nx=40, ny=40, T=250001, aspect=4.0, flip=True, G=[[2.1e-3, 2e-4], [1e-4, 2.6e-3]]),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c.values() if not isinstance(x, list)))
def test_gridded_shapes(orc, case):
    m, g, r, v, c, s = _case(seed=4, **case)
    R, V = dev(r, F32), dev(v, F32)
    n0 = api.mpi_kernel_launches()
    got = api.mpi_forward(m, g, R, V, dev(c, F32))
    n1 = api.mpi_kernel_launches()
    a = api.mpi_adjoint(m, g, R, V, dev(s, F32))
    assert (n1 - n0, api.mpi_kernel_launches() - n1) == (6, 8)
    assert rel_l2(host(got), orc.forward(m, g, r, v, c)) <= TOL
    assert rel_l2(host(a), orc.adjoint(m, g, r, v, s)) <= TOL
    assert torch.equal(a, api.mpi_adjoint(m, g, R, V, dev(s, F32)))
