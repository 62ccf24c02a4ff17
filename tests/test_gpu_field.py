"""The gridded FP32 route of the 2-D pair operators (large problems) against
the FP64 oracle: odd sizes, thin and one-column grids, general and negative
axes, one channel, dwelling and repeated positions, samples beyond the node
window, non-finite positions, unaligned arrays.

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


def test_field_unaligned_trajectory(orc):
    """Arrays that are aligned to single floats only."""
    m, g, r, v, c, s = _case(128, 128, 16384, 8)
    buf = torch.empty((2, 2 * r.size + 2), dtype=F32, device="cuda")
    R, V = (buf[k, 1:1 + r.size].view(-1, 2) for k in range(2))
    R.copy_(dev(r, F32))
    V.copy_(dev(v, F32))
    assert R.data_ptr() % 8 == 4 and V.data_ptr() % 8 == 4
    assert rel_l2(host(api.mpi_forward(m, g, R, V, dev(c, F32))), orc.forward(m, g, r, v, c)) <= TOL
    assert rel_l2(host(api.mpi_adjoint(m, g, R, V, dev(s, F32))), orc.adjoint(m, g, r, v, s)) <= TOL


def test_field_solve_single_batch_and_sharded(orc):
    """Algorithm 1 on the gridded operators (64 x 60, 40 001 samples) against the oracle, held to the FP32 bar
    of the well-posed solves; the matched batch (beside a frame that keeps the
    pair sums) bit for bit, and the sharded solve."""
    big, small = _case(64, 60, 40001, 11), _case(20, 24, 900, 12)
    nu0 = []
    for m, g, r, v, c, s in (big, small):
        nu0.append(orc.nu0_from_frob2(orc.frob2(m, g, r, v), g["nx"] * g["ny"]))
    data = [rounded(orc.forward(m, g, r, v, c), F32) for m, g, r, v, c, _ in (big, small)]
    single = []
    for (m, g, r, v, c, _), s, nu in zip((big, small), data, nu0):
        single.append(host(api.mpi_pnp_solve(m, g, dev(r, F32), dev(v, F32), dev(s, F32), 3, 4, nu)))
    m, g, r, v = big[:4]
    want = orc.pnp(lambda x: orc.forward(m, g, r, v, x), lambda y: orc.adjoint(m, g, r, v, y), data[0],
                   (g["ny"], g["nx"]), 3, 4, nu0[0])
    assert rel_l2(single[0], want) <= 1e-5
    plan = api.BatchPlan([(q[0], q[1], q[2].shape[0]) for q in (big, small)], nu0, 3, 4,
                         flags=api.MPI_BATCH_MATCH_SINGLE)
    assert plan.info()["forward_items"] > 0  # the small frame's pair items
    arrays = [[dev(x, F32) for x in xs] for xs in ([big[2], small[2]], [big[3], small[3]], data)]
    for _ in range(2):
        got = [host(x) for x in plan.run(*arrays)]
        for a, b in zip(got, single):
            assert np.array_equal(a, b)
    sharded = host(api.mpi_pnp_solve_sharded(m, g, dev(r, F32), dev(v, F32), dev(data[0], F32), 3, 4, nu0[0],
                                             lambda t: None))
    assert rel_l2(sharded, want) <= 1e-5
