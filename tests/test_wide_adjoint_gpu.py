"""The fused Chebyshev adjoint for windows of other than 32 taps, and the per-tap adjoint that
keeps the short masked ones, against the oracle's analytic gradient, at the lengths where the
choice and the slots of 32 taps change.  Bound: 1e-4 of each group's largest
(test_adjoint_gpu.py); a batch of several windows is bitwise the same as each alone.
"""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, T = 16000.0, 0.09
L, BETA = [3.7, 2.9, 2.3], np.array([0.9, 0.8, 0.85, -0.7, 0.95, 0.6], np.float32)
PS = np.array([[1.0, 1.1, 0.7], [2.9, 2.2, 1.5]], np.float32)
PR = np.array([[2.0, 1.4, 1.2], [0.6, 0.5, 2.0]], np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _inputs(taps):
    Tw = float(np.float32(taps / FS))
    n = oracle.n_samples(np.float32(T), FS)
    g = np.random.default_rng(int(10 * taps)).standard_normal((2, 2, n)).astype(np.float32)
    return Tw, oracle.nb_img_from_t(T, L, 343.0, Tw), n, g


@pytest.mark.parametrize("taps", [15.0, 16.0, 17.5, 34.0, 64.0, 64.5, 79.3, 80.5, 96.0, 110.25, 176.4, 192.0, 256.0])
def test_gradients(taps):
    Tw, N, n, g = _inputs(taps)
    got = [v.cpu().numpy().astype(np.float64) for v in
           ism.ism_simulate_backward(L, BETA, PS, PR, N, T, FS, torch.from_numpy(g), Tw=Tw)]
    ref = [np.zeros(6), np.zeros((2, 3)), np.zeros((2, 3))]
    for i in range(2):
        for j in range(2):
            b, s, r = oracle.rir_grad(L, BETA.astype(np.float64), 343.0, FS, Tw, PS[i].astype(np.float64),
                                      PR[j].astype(np.float64), N, n, g[i, j].astype(np.float64))
            ref[0] += b
            ref[1][i] += s
            ref[2][j] += r
    for a, b in zip(got, ref):
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))


def test_windows_of_several_lengths_in_one_batch():
    jobs, keep, alone = [], [], []
    ps, pr = torch.from_numpy(PS).cuda(), torch.from_numpy(PR).cuda()
    for taps in (64.0, 32.0, 176.4, 20.5, 64.0):
        Tw, N, n, g = _inputs(taps)
        gd = torch.from_numpy(g).cuda()
        alone.append(ism.ism_simulate_backward(L, BETA, PS, PR, N, T, FS, gd, Tw=Tw))
        out = [torch.empty_like(v) for v in alone[-1]]
        jobs.append(ism.make_grad_job(ism.make_job(L, BETA, ps, pr, N, T, FS, gd, Tw=Tw), gd, *out))
        keep.append((gd, out))
    ism.ism_simulate_backward_batch(jobs)
    torch.cuda.synchronize()
    for (_, out), ref in zip(keep, alone):
        for a, b in zip(out, ref):
            assert torch.equal(a, b)
