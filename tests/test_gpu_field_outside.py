"""The gridded FP32 operators on samples beyond the node window, which are
summed directly beside the transforms: bursts and whole scans outside, both
kinds of G, odd sizes, and how long they take.

Tolerance 1e-6 as for the gridded operators (the direct sums, rows of at most
128 terms and then compensated, are below that: 128 x 2^-24 / 2 if every
rounding had the same sign)."""
import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded

pytestmark = pytest.mark.gpu
F32 = torch.float32
TOL = 1e-6
TILTED = [[2.1e-3, 4e-4], [3e-4, 2.6e-3]]


def _case(nx, ny, T, out, G=None, n_ch=2, seed=1):
    """out samples in a row outside (to one side), the others within."""
    rng = np.random.default_rng(seed)
    m, g = syn.default_model(n_ch=n_ch), syn.square_grid(nx, 24.0, ny)
    if G:
        m["G"] = G
    r, v = syn.lissajous(T, 17, 16, amp=11.5)
    r, v = np.array(r), np.array(v)
    k = (T - out) // 3
    r[k:k + out] += [9.0, 31.0]
    r, v = rounded(r, F32), rounded(v, F32)
    c = rounded(rng.uniform(size=(ny, nx)) * (rng.uniform(size=(ny, nx)) < 0.3), F32)
    s = rounded(rng.normal(size=(n_ch, T)), F32)
    return m, g, r, v, c, s


# one sample, a block's share and one more, all of them; the widest rows and a
# single one, a tall grid
CASES = [(128, 128, 20000, 1), (128, 128, 20000, 769), (131, 97, 20011, 20011), (1025, 9, 20000, 700),
         (1700, 1, 90001, 333), (40, 300, 20001, 65)]


@pytest.mark.parametrize("G", [None, TILTED], ids=["diagonal", "tilted"])
@pytest.mark.parametrize("nx,ny,T,out", CASES)
def test_outside_samples(orc, nx, ny, T, out, G):
    m, g, r, v, c, s = _case(nx, ny, T, out, G, n_ch=1 + out % 2)
    R, V, C, S = (dev(x, F32) for x in (r, v, c, s))
    n0 = api.mpi_kernel_launches()
    got = api.mpi_forward(m, g, R, V, C)
    n1 = api.mpi_kernel_launches()
    a = api.mpi_adjoint(m, g, R, V, S)
    assert n1 - n0 == 6 and api.mpi_kernel_launches() - n1 == 8  # the gridded route
    want = orc.forward(m, g, r, v, c)
    assert rel_l2(host(got), want) <= TOL
    # the outside samples by themselves: their signal is the smaller one
    k = (T - out) // 3
    assert rel_l2(host(got)[:, k:k + out], want[:, k:k + out]) <= TOL
    assert rel_l2(host(a), orc.adjoint(m, g, r, v, s)) <= TOL
    assert torch.equal(got, api.mpi_forward(m, g, R, V, C))
    assert torch.equal(a, api.mpi_adjoint(m, g, R, V, S))


@pytest.mark.parametrize("G", [None, TILTED], ids=["diagonal", "tilted"])
def test_solve_with_outside_samples(orc, G):
    """A quarter of the samples outside, several products on one plan (the
    counters of the outside sums start each of them anew)."""
    m, g, r, v, c, _ = _case(64, 60, 40001, 10000, G)
    s = rounded(orc.forward(m, g, r, v, c), F32)
    nu0 = orc.nu0_from_frob2(orc.frob2(m, g, r, v), 64 * 60)
    want = orc.pnp(lambda x: orc.forward(m, g, r, v, x), lambda y: orc.adjoint(m, g, r, v, y), s, (60, 64), 3, 4, nu0)
    got = host(api.mpi_pnp_solve(m, g, dev(r, F32), dev(v, F32), dev(s, F32), 3, 4, nu0))
    assert rel_l2(got, want) <= 1e-5


def _us(f, n=20):
    for _ in range(3):
        f()
    best = 1e30
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


@pytest.mark.parametrize("amp", [18.0, 48.0])
def test_scan_beyond_the_grid_costs_no_more_than_pair_sums(amp):
    """50 and 94 % of the samples outside: the gridded A may take the pair sums'
    time and its own transforms' (three times the pair sums is what summing the
    samples of a block one after another took, and more)."""
    m, g = syn.default_model(), syn.square_grid(128, 24.0)
    r, v = syn.lissajous(65536, 17, 16, amp=amp)
    R, V = dev(r, F32), dev(v, F32)
    C = torch.rand((128, 128), dtype=F32, device="cuda")
    field = _us(lambda: api.mpi_forward(m, g, R, V, C))
    sums = _us(lambda: api.mpi_forward_sums(m, g, R, V, C))
    assert field <= 1.5 * sums
