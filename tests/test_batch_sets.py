"""Batches of more jobs than a launch set holds (64): the workspace of the two sets in flight, and
the results, which do not depend on the sets."""
import ctypes

import numpy as np
import pytest

from paper_1810_11359_gb300 import build as libbuild
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")

FS, T, L, BETA = 16000.0, 0.6, [6.0, 5.0, 3.0], [0.85] * 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


def _size(n, n_rcv):
    j = ism.ism_job()
    j.room.L[:], j.room.beta[:], j.room.c = L, BETA, 343.0
    j.n_src, j.n_rcv, j.Tmax, j.fs, j.Tw = 1, n_rcv, T, FS, 32 / FS
    j.nb_img[:] = ism.ism_nb_img_from_t(T, L, 343.0, 32 / FS)
    arr, b = (ism.ism_job * n)(*[j] * n), ctypes.c_size_t()
    ism._check(ism.load().ism_batch_workspace_size(arr, n, 0, ctypes.byref(b)))
    return b.value


@pytest.mark.parametrize("n", [65, 100, 127, 128, 129, 300, 1000])
def test_two_sets_in_flight_take_one_full_sets_workspace(n):
    """Up to rounding: each of the two holds ceil(n / 2 ceil(n / 64)) <= 32 jobs."""
    assert _size(n, 16) <= 1.01 * _size(64, 16)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [65, 130])
def test_results_do_not_depend_on_the_sets(n):
    torch.cuda.set_device(0)
    rng = np.random.default_rng(n)
    jobs, keep = [], []
    for i in range(n):   # ~3.5e7 images in reach together; dense and sparse rooms, tails, other windows
        k = 1.0 if i % 5 else 2.5
        Li = [k * v for v in (3.3 + 0.01 * i, 3.9, 2.6)]
        kw = dict(Tdiff=0.25 if i % 3 else 0.0, Tw=32 / FS if i % 4 else 0.0, seed=i)
        nb = ism.ism_nb_img_from_t(kw["Tdiff"] or 0.4, Li, 343.0, kw["Tw"] or 4e-3)
        ps, pr = (torch.from_numpy(rng.uniform(0.4, 2.4, (m, 3)).astype(np.float32)).cuda() for m in (1, 1 + i % 6))
        out = torch.full((1, pr.shape[0], ism.ism_rir_length(0.4, FS)), float("nan"), device="cuda")
        jobs.append(ism.make_job(Li, BETA, ps, pr, nb, 0.4, FS, out, **kw))
        keep.append((Li, ps, pr, nb, kw, out))
    ism.ism_simulate_batch(jobs)
    for Li, ps, pr, nb, kw, out in keep:
        assert torch.equal(out, ism.ism_simulate(Li, BETA, ps, pr, nb, 0.4, FS, **kw))
