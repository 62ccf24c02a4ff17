"""Host time of a call that plans for the grid and then takes the pair sums:
not more than a few microseconds above a call that goes to the pair sums
straight (factoring every candidate length took 12 us here)."""
import time

import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu
F32 = torch.float32


def _enqueue_us(call, args, out):
    best = 1e30
    for _ in range(7):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(100):
            call(*args, s=out)
        best = min(best, (time.perf_counter() - t0) * 1e4)
    torch.cuda.synchronize()
    return best


def test_planning_costs_little():
    m, g = syn.default_model(), syn.square_grid(512, 48.0)
    r, v = syn.lissajous(80, 3, 2, amp=24.0)
    args = (m, g, dev(r, F32), dev(v, F32), torch.rand((512, 512), dtype=F32, device="cuda"))
    out = torch.empty((2, 80), dtype=F32, device="cuda")
    n0 = api.mpi_kernel_launches()
    api.mpi_forward(*args, s=out)
    planned = api.mpi_kernel_launches() - n0
    api.mpi_forward_sums(*args, s=out)
    assert api.mpi_kernel_launches() - n0 == 2 * planned and planned <= 5  # both by pair sums
    sums = _enqueue_us(api.mpi_forward_sums, args, out)
    assert _enqueue_us(api.mpi_forward, args, out) <= sums + 10.0
