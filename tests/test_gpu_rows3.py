"""The row forms of the 3-D operators (diagonal G) against the FP64 oracle and
against the form for a general G, which an off-diagonal entry too small to
change any sum selects: ragged boxes, rows and sample groups, both axis
directions, near samples, grids far off the origin (where the row forms step
aside) and non-finite positions.

Tolerance: the bar of the pair operators (FP32: sums of up to 4e4 terms, each
pair to 3e-7, in blocks of at most 512; FP64: 1e-12)."""
import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded, tol

pytestmark = pytest.mark.gpu

CASES = [
    dict(nx=1, ny=1, nz=1, T=1),
    dict(nx=1, ny=9, nz=5, T=257),
    dict(nx=37, ny=1, nz=1, T=63),
    dict(nx=8, ny=8, nz=4, T=256),                                     # one box, one staged batch
    dict(nx=9, ny=17, nz=5, T=289),                                    # one voxel, row, layer and sample over
    dict(nx=31, ny=33, nz=7, T=1025, flip=True),
    dict(nx=24, ny=20, nz=12, T=4100, fov=3.0),                        # every pair near or in the closed form
    dict(nx=12, ny=10, nz=6, T=700, G=(2.5e-3, -1.2e-3, -1.3e-3), n_ch=2),
    dict(nx=16, ny=12, nz=6, T=600, far=3e6),                          # columns not resolved evenly in FP32
    dict(nx=16, ny=12, nz=6, T=600, far=20.0),
]


def _case(cs, dt):
    rng = np.random.default_rng(cs["nx"] + cs["T"])
    fov, far = cs.get("fov", 24.0), cs.get("far", 0.0)
    g = syn.box_grid3(cs["nx"], cs["ny"], cs["nz"], fov, fov / 2)
    r, v = syn.lissajous3(cs["T"], 5, 4, 3, amp=(fov / 2, fov / 2, fov / 4))
    if cs.get("flip"):
        g["x0"], g["dx"] = -g["x0"], -g["dx"]
        g["z0"], g["dz"] = -g["z0"], -g["dz"]
    g["x0"] += far
    r = r + np.array([far, 0.0, 0.0])
    m = syn.default_model3(n_ch=cs.get("n_ch", 3))
    if "G" in cs:
        m = dict(m, G=np.diag(cs["G"]).tolist())
    c = rounded(rng.uniform(size=(cs["nz"], cs["ny"], cs["nx"])), dt)
    s = rounded(rng.normal(size=(len(m["p"]), cs["T"])), dt)
    return m, g, rounded(r, dt), rounded(v, dt), c, s


def _both(m, g, r, v, c, s, dt):
    R, V = dev(r, dt), dev(v, dt)
    return (host(api.mpi_forward3(m, g, R, V, dev(c, dt))), host(api.mpi_adjoint3(m, g, R, V, dev(s, dt))))


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("cs", CASES, ids=lambda c: f"{c['nx']}x{c['ny']}x{c['nz']}_{c['T']}")
def test_row_forms(orc, dt, cs):
    m, g, r, v, c, s = _case(cs, dt)
    got = _both(m, g, r, v, c, s, dt)
    G = np.array(m["G"])
    G[0, 1] = 1e-300
    general = _both(dict(m, G=G.tolist()), g, r, v, c, s, dt)
    want = orc.forward3(m, g, r, v, c), orc.adjoint3(m, g, r, v, s)
    for a, b, w in zip(got, general, want):
        assert rel_l2(a, b) <= 2 * tol(dt)
        if cs.get("far", 0.0) < 1e3:  # (far off, rounding the positions themselves decides)
            assert rel_l2(a, w) <= tol(dt)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_row_forms_non_finite_positions(orc, dt):
    """A sample at NaN or infinity makes its own outputs NaN and no others;
    in A^T it reaches every voxel."""
    m, g, r, v, c, s = _case(dict(nx=20, ny=18, nz=9, T=900), dt)
    bad = r.copy()
    bad[17, 0], bad[600, 1], bad[700, 2] = np.nan, np.inf, np.nan
    fwd, adj = _both(m, g, bad, v, c, s, dt)
    keep = np.ones(r.shape[0], bool)
    keep[[17, 600, 700]] = False
    assert np.isnan(fwd[:, ~keep]).all() and np.isnan(adj).all()
    assert rel_l2(fwd[:, keep], orc.forward3(m, g, r, v, c)[:, keep]) <= tol(dt)
