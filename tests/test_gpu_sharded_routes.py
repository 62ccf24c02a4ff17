"""Sample-sharded solves whose processes evaluate their sums by different
routes (a long slice on the gridded operators, short and empty ones pair by
pair): every process makes the same reductions and ends with the same image,
that of the whole problem."""
import threading

import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api, sharded
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rel_l2, rounded, tol

pytestmark = pytest.mark.gpu
F32 = torch.float32
N_ITER, N_CG = 3, 4
PRODUCTS = N_ITER * (N_CG + 1)


def _case(orc, nx, ny, T):
    g = syn.square_grid(nx, 24.0, ny)
    m = syn.default_model()
    rng = np.random.default_rng(T)
    t = np.arange(T)
    w = 2 * np.pi * np.array([17.0, 16.0]) / T
    r = rounded(12.0 * np.sin(t[:, None] * w + [0.3, 1.1]), F32)
    v = rounded(12.0 * w * np.cos(t[:, None] * w + [0.3, 1.1]), F32)
    c = rng.uniform(size=(ny, nx)) * (rng.uniform(size=(ny, nx)) < 0.3)
    s = rounded(orc.forward(m, g, r, v, c), F32)
    nu0 = orc.nu0_from_frob2(orc.frob2(m, g, r, v), nx * ny)
    return m, g, r, v, s, nu0


def _launches(m, g, r, v, s, nu0):
    """Kernel launches of one process's solve on its slice alone."""
    n0 = api.mpi_kernel_launches()
    api.mpi_pnp_solve_sharded(m, g, dev(r, F32), dev(v, F32), dev(s, F32), N_ITER, N_CG, nu0, lambda t: None)
    return api.mpi_kernel_launches() - n0


@pytest.mark.parametrize("lengths", [(40000, 2000, 0), (300, 41700)])
def test_sharded_routes_agree(orc, lengths):
    m, g, r, v, s, nu0 = _case(orc, 64, 60, sum(lengths))
    ends = np.cumsum((0,) + lengths)
    parts = [(r[a:b], v[a:b], s[:, a:b]) for a, b in zip(ends[:-1], ends[1:])]
    # a gridded product A^T A is eight launches, one by pair sums four
    gridded = [_launches(m, g, *q, nu0) > 8 * PRODUCTS for q in parts]
    assert gridded == [n > 10000 for n in lengths]
    world = len(parts)
    ar = sharded.ThreadAllreduce(world, timeout=60)
    out, err, calls = [None] * world, [None] * world, [0] * world

    def run(k):
        fn = ar.for_rank(k)

        def counted(t):
            calls[k] += 1
            fn(t)
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                q = [dev(x, F32) for x in parts[k]]
                rho = api.mpi_pnp_solve_sharded(m, g, *q, N_ITER, N_CG, nu0, counted)
                st.synchronize()
                out[k] = rho.double().cpu().numpy()
        except BaseException as e:  # noqa: BLE001 - reported below
            err[k] = e
            ar.abort()
    threads = [threading.Thread(target=run, args=(k,)) for k in range(world)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert all(e is None for e in err), err
    assert calls == [1 + PRODUCTS] * world
    for k in range(world):
        assert np.array_equal(out[k], out[0])
    want = orc.pnp(lambda x: orc.forward(m, g, r, v, x), lambda y: orc.adjoint(m, g, r, v, y), s,
                   (g["ny"], g["nx"]), N_ITER, N_CG, nu0)
    assert rel_l2(out[0], want) <= tol(F32)


def test_sharded_one_gridded_process_is_the_plain_solve(orc):
    """One process: the residual goes through the reduction as A^T A v and
    comes back; only FP64 rounding and the order of the inner products differ
    from the plain solve."""
    m, g, r, v, s, nu0 = _case(orc, 64, 60, 40000)
    args = (m, g, dev(r, F32), dev(v, F32), dev(s, F32), N_ITER, N_CG, nu0)
    calls = []
    got = host(api.mpi_pnp_solve_sharded(*args, lambda t: calls.append(t.numel())))
    assert calls == [64 * 60] * (1 + PRODUCTS)
    assert rel_l2(got, host(api.mpi_pnp_solve(*args))) <= tol(F32)
