"""The one-launch Core Stage solve of small problems (FP32) against the FP64
oracle at its edges: one node, one row, node counts around a block's 256,
grids just within and just beyond what one launch holds on this device, no
samples, one channel, a step count of one, stop tests that hold at once."""
import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded, tol

pytestmark = pytest.mark.gpu
DT = torch.float32


def _data(nx, ny, T, seed=1, rows=2):
    g = syn.square_grid(nx, 24.0, ny)
    rng = np.random.default_rng(seed + nx + T)
    r, v = syn.lissajous(max(T, 1), 17, 16, amp=12.5)
    s = rng.normal(size=(rows, T))
    return g, rounded(r[:T], DT), rounded(v[:T], DT), rounded(s, DT)


def _edge():
    """Side of the largest square one launch holds (2 blocks of 256 per SM)."""
    return int(np.sqrt(2 * 256 * torch.cuda.get_device_properties(0).multi_processor_count))


@pytest.mark.parametrize("nx, ny, T", [(1, 1, 5), (1, 257, 900), (255, 1, 900), (16, 16, 1000), (257, 3, 3001),
                                       (0, 0, 20000), (0, 1, 20000)])
def test_resident_core_stage(orc, nx, ny, T):
    """gamma = 1e-2 keeps the system well conditioned, so a fixed number of
    steps agrees to the FP32 bar (one node: two distinct eigenvalues, so CG is
    done after two steps and only the first is compared)."""
    if nx == 0:
        nx, ny = _edge(), _edge() + ny
    g, r, v, s = _data(nx, ny, T)
    for steps in (1, 9) if nx * ny > 1 else (1,):
        want, want_u, hist = orc.core_stage(g, r, v, s, 1e-2, max_iter=steps)
        A, u, n = api.mpi_grid(g, dev(r, DT), dev(v, DT), dev(s, DT), gamma=1e-2, max_iter=steps, rel_tol=0.0,
                               return_iters=True)
        assert n == len(hist) - 1
        assert rel_l2(host(A), want) <= tol(DT)
        assert rel_l2(host(u), want_u) <= tol(DT)


@pytest.mark.parametrize("k", [0, 1])
def test_resident_core_stage_channel(orc, k):
    g, r, v, s = _data(33, 21, 2001, rows=1)
    want, want_kk, hist = orc.core_stage_channel(g, r, v, s[0], k, 1e-2, 8)
    A, akk, n = api.mpi_grid(g, dev(r, DT), dev(v, DT), dev(s[0], DT), gamma=1e-2, max_iter=8, rel_tol=0.0,
                             return_iters=True, channel=k)
    assert n == len(hist) - 1
    assert rel_l2(host(A), want) <= tol(DT)
    assert rel_l2(host(akk), want_kk) <= tol(DT)


def test_resident_core_stage_stops_at_once():
    """Zero data, no samples, and a tolerance that the start meets: no step, a
    zero field."""
    g, r, v, s = _data(20, 30, 500)
    for rr, vv, ss, tolerance in ((r, v, 0 * s, 0.0), (r[:0], v[:0], s[:, :0], 0.0), (r, v, s, 1.0)):
        A, u, n = api.mpi_grid(g, dev(rr, DT), dev(vv, DT), dev(ss, DT), gamma=1e-2, max_iter=50, rel_tol=tolerance,
                               return_iters=True)
        assert n == 0
        assert not host(A).any() and not host(u).any()


@pytest.mark.parametrize("shape", [(1, 1, 1), (17, 5, 3), (48, 30, 48), (48, 31, 48)])
def test_resident_core_stage3(orc, shape):
    """Within (69 120 nodes) and beyond (71 424) one launch on 152 SMs."""
    g = syn.box_grid3(*shape)
    T = 5001
    r, v = syn.lissajous3(T, 17, 16, 15)
    r, v = rounded(r, DT), rounded(v, DT)
    s = rounded(np.random.default_rng(4).normal(size=(3, T)), DT)
    steps = 5 if shape[0] > 1 else 2  # (one node: three distinct eigenvalues)
    want, want_u, hist = orc.core_stage3(g, r, v, s, 1e-2, max_iter=steps)
    A, u, n = api.mpi_grid3(g, dev(r, DT), dev(v, DT), dev(s, DT), gamma=1e-2, max_iter=steps, rel_tol=0.0,
                            return_iters=True)
    assert n == len(hist) - 1
    assert rel_l2(host(A), want) <= tol(DT)
    assert rel_l2(host(u), want_u) <= tol(DT)
