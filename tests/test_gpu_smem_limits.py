"""Plans whose kernels need different amounts of dynamic shared memory (more
than the default 48 KB), prepared one after another or by several threads: the
smaller one must not take from the larger what it was granted."""
import threading

import numpy as np
import pytest
import torch

from paper_2505_22797_gb300 import api
from paper_2505_22797_gb300 import synthetic as syn
from tests.gpu_util import dev, host, rounded

pytestmark = pytest.mark.gpu
F32 = torch.float32
SIZES = [(100, 100), (128, 128), (84, 97)]  # 57.5, 55.2 KB and less in the column launches


def _frame(nx, ny, T=16000):
    rng = np.random.default_rng(nx)
    m, g = syn.default_model(), syn.square_grid(nx, 24.0, ny)
    r, v = syn.lissajous(T, 17, 16, amp=12.0)
    c = rng.uniform(size=(ny, nx)) * (rng.uniform(size=(ny, nx)) < 0.3)
    R, V, C = dev(rounded(r, F32), F32), dev(rounded(v, F32), F32), dev(rounded(c, F32), F32)
    return m, g, R, V, api.mpi_forward(m, g, R, V, C)


@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0)])
def test_batch_of_gridded_frames_of_several_sizes(order):
    frames = [_frame(*SIZES[k]) for k in order]
    nu0 = [1e-3] * len(frames)
    plan = api.BatchPlan([(m, g, R.shape[0]) for m, g, R, _, _ in frames], nu0, 2, 3,
                         flags=api.MPI_BATCH_MATCH_SINGLE)
    assert plan.info()["forward_items"] == 0  # every frame gridded
    got = plan.run(*([f[k] for f in frames] for k in (2, 3, 4)))
    for a, (m, g, R, V, s) in zip(got, frames):
        assert np.array_equal(host(a), host(api.mpi_pnp_solve(m, g, R, V, s, 2, 3, 1e-3)))


def test_threads_of_several_sizes():
    frames = [_frame(*size) for size in SIZES]
    want = [api.mpi_adjoint(*f) for f in frames]
    torch.cuda.synchronize()
    err, equal = [None] * len(frames), [False] * len(frames)

    def run(k):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                got = [api.mpi_adjoint(*frames[k]) for _ in range(50)]
                st.synchronize()
                equal[k] = all(torch.equal(a, want[k]) for a in got)
        except BaseException as e:  # noqa: BLE001 - reported below
            err[k] = e
    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(frames))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert err == [None] * len(frames)
    assert all(equal)
