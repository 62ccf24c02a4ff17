"""The gridded FP32 route of the 2-D pair operators (large problems) against
the FP64 oracle: odd sizes, thin and one-column grids, general and negative
axes, one channel, dwelling and repeated positions, samples beyond the node
window, non-finite positions, and the calls that stay with the direct sums.

Tolerance 1e-6: the transforms have about 25 butterfly levels and the
interpolation 6 more, each rounding by 2^-24; if all of them added up the
relative error would be 31 x 2^-24 = 1.8e-6, and they add in the root mean
square (below 4e-7).  The window's own error is 4e-9."""
import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded

pytestmark = pytest.mark.gpu
F32 = torch.float32
TOL = 1e-6


def _case(nx, ny, T, seed, G=None, p=None, fov=24.0, flip=False, aspect=1.0, spread=1.0):
    rng = np.random.default_rng(seed)
    g = syn.square_grid(nx, fov, ny)
    g["y0"], g["dy"] = g["y0"] * aspect, g["dy"] * aspect
    if flip:
        g["x0"], g["dx"] = -g["x0"], -g["dx"]
    m = dict(syn.default_model(), **({"G": G} if G else {}), **({"p": p} if p else {}))
    t = np.arange(T)
    w = 2 * np.pi * np.array([17.0, 16.0]) / T
    ph = rng.uniform(0, 6, 2)
    amp = spread * fov / 2 * np.array([1.0, aspect])
    r = rounded(amp * np.sin(t[:, None] * w + ph), F32)
    v = rounded(amp * w * np.cos(t[:, None] * w + ph), F32)
    c = rounded(rng.uniform(size=(ny, nx)) * (rng.uniform(size=(ny, nx)) < 0.3), F32)
    s = rounded(rng.normal(size=(len(m["p"]), T)), F32)
    return m, g, r, v, c, s


CASES = [
    dict(nx=131, ny=97, T=20011),
    dict(nx=128, ny=128, T=16385, G=[[2.1e-3, 4e-4], [3e-4, -2.6e-3]], p=[[0.6, 0.8]]),
    dict(nx=150, ny=60, T=30001, flip=True, aspect=0.4),
    dict(nx=1200, ny=3, T=50001),
    dict(nx=1, ny=700, T=230001),
    dict(nx=9, ny=7, T=2500001),
    dict(nx=300, ny=280, T=4097, fov=48.0),
    dict(nx=101, ny=99, T=20001, spread=1.15),                     # beyond the grid, mostly inside the window
    dict(nx=90, ny=110, T=20001, spread=4.0),                      # most samples beyond the window
    dict(nx=90, ny=110, T=20001, spread=4.0, G=[[2.1e-3, 4e-4], [3e-4, 2.6e-3]]),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(str(c[k]) for k in ("nx", "ny", "T")))
def test_field_operators(orc, case):
    m, g, r, v, c, s = _case(seed=3, **case)
    R, V = dev(r, F32), dev(v, F32)
    got = host(api.mpi_forward(m, g, R, V, dev(c, F32)))
    assert rel_l2(got, orc.forward(m, g, r, v, c)) <= TOL
    a = api.mpi_adjoint(m, g, R, V, dev(s, F32))
    assert rel_l2(host(a), orc.adjoint(m, g, r, v, s)) <= TOL
    assert torch.equal(a, api.mpi_adjoint(m, g, R, V, dev(s, F32)))


def test_field_dwelling_samples(orc):
    """All samples within two nodes of one point (one tile, many units), and
    exactly on it."""
    m, g, r, v, c, s = _case(130, 128, 20000, 5)
    rng = np.random.default_rng(6)
    r = rounded(np.array([1.7, -2.3]) + 0.05 * rng.normal(size=r.shape), F32)
    r[5000:9000] = r[0]
    R, V = dev(r, F32), dev(v, F32)
    assert rel_l2(host(api.mpi_forward(m, g, R, V, dev(c, F32))), orc.forward(m, g, r, v, c)) <= TOL
    assert rel_l2(host(api.mpi_adjoint(m, g, R, V, dev(s, F32))), orc.adjoint(m, g, r, v, s)) <= TOL


def test_field_non_finite_positions(orc):
    """A sample at NaN or infinity makes its own outputs NaN (as in the direct
    sums) and no others; in A^T it reaches every voxel."""
    m, g, r, v, c, s = _case(128, 128, 16384, 7)
    want = orc.forward(m, g, r, v, c)
    bad = r.copy()
    bad[17, 0], bad[9000, 1] = np.nan, np.inf
    got = host(api.mpi_forward(m, g, dev(bad, F32), dev(v, F32), dev(c, F32)))
    assert np.isnan(got[:, [17, 9000]]).all()
    keep = np.ones(r.shape[0], bool)
    keep[[17, 9000]] = False
    assert rel_l2(got[:, keep], want[:, keep]) <= TOL
    assert np.isnan(host(api.mpi_adjoint(m, g, dev(bad, F32), dev(v, F32), dev(s, F32)))).all()


def test_field_and_direct_routes_agree_on_alignment(orc):
    """A trajectory that is not 8-byte aligned runs the direct sums."""
    m, g, r, v, c, s = _case(128, 128, 16384, 8)
    buf = torch.empty(2 * r.size + 2, dtype=F32, device="cuda")
    R = buf[1:1 + r.size].view(-1, 2)
    R.copy_(dev(r, F32))
    assert R.data_ptr() % 8 == 4
    got = host(api.mpi_forward(m, g, R, dev(v, F32), dev(c, F32)))
    assert rel_l2(got, orc.forward(m, g, r, v, c)) <= TOL
