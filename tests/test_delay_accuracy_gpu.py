"""Delays of sources 5 to 60 samples from the receiver in long RIRs.  All walls absorb (beta =
0), so a RIR is the direct path alone, whatever the number of images in its grid (66 a side make
its bins dense, 3 sparse), and its delay can be read from the samples: a least-squares fit of
amplitude and delay to the exact pulse.

Bounds: the fraction of a delay is rounded to 2^-25 sample, 3e-8.  What the taps' own errors add
is their norm over that of the pulse's derivative, 1.81: 2e-7 / 1.81 for taps at FP32 rounding
(test_window_accuracy_gpu.py), for the 8-term series of 32 taps another 3.8e-7 (its error along
the derivative, in 64 bits).  Squared offsets held in too few bits: 1e-6 sample and more.
"""
import numpy as np
import pytest

from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, C = 16000.0, 343.0
ROOM, PR = [6.0, 5.0, 3.0], np.array([3.03, 2.52, 1.49], np.float32)
N_SRC = 96
K = FS / float(np.float32(C))
ROUNDED = 3e-8 + 2e-7 / 1.81
# on both sides of the length from which the offsets are no longer split, and the longest
LENGTHS = [9600, 15900, 16000, 22500, 22700, 57600, 131000]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _sources(seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((N_SRC, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    return (PR + u * rng.uniform(5.0, 60.0, (N_SRC, 1)) / K).astype(np.float32)


def _pulse(x, taps):
    return np.where(np.abs(x) < taps / 2, 0.5 * (1 + np.cos(2 * np.pi * x / taps)) * np.sinc(x), 0.0)


def _case(n, taps, seed):
    ps = _sources(seed)
    s = np.linalg.norm(ps.astype(np.float64) - PR.astype(np.float64), axis=1) * K
    k = np.arange(0, 60 + int(taps) // 2 + 2)
    return ps, s, k[None, :] - s[:, None], dict(Tmax=n / FS, fs=FS, Tw=taps / FS)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("prec,taps,nb", [("fp32", 32, 66), ("fp32", 64, 66), ("fp32", 32, 3), ("fp32_direct", 32, 66)])
def test_forward(n, prec, taps, nb):
    ps, s, x, kw = _case(n, taps, n)
    h = ism.ism_simulate(ROOM, [0.0] * 6, ps, PR[None], [nb] * 3, prec=prec, **kw)
    h = h[:, 0, :x.shape[1]].cpu().numpy().astype(np.float64)
    eps = 1e-4
    g, d = _pulse(x, taps), (_pulse(x - eps, taps) - _pulse(x + eps, taps)) / (2 * eps)   # d/ds, x = k - s
    off = [np.linalg.lstsq(np.stack([g[i], d[i]], 1), h[i], rcond=None)[0] for i in range(N_SRC)]
    delta = np.array([b / a for a, b in off])
    tol = ROUNDED + (3.8e-7 if (prec, taps, nb) == ("fp32", 32, 66) else 0.0)
    assert np.max(np.abs(delta)) <= tol


@pytest.mark.parametrize("n", LENGTHS)
def test_gradient(n):
    """The direct path's gradient does not depend on the RIR's length beyond it.  dLoss/dh lies
    along the pulse's second derivative, where a delay's error enters in full; the two lengths'
    delays each have the bound above."""
    taps = 64
    ps, s, x, _ = _case(n, taps, n + 1)
    eps = 1e-3
    d2 = (_pulse(x - eps, taps) - 2 * _pulse(x, taps) + _pulse(x + eps, taps)) / eps ** 2
    norm2 = np.linalg.norm(d2, axis=1)
    go = torch.from_numpy((d2 / norm2[:, None]).astype(np.float32)).cuda()
    u = ps.astype(np.float64) - PR.astype(np.float64)
    r = np.linalg.norm(u, axis=1)

    def along(length):
        grad_out = torch.zeros((N_SRC, 1, length), device="cuda")
        grad_out[:, 0, :x.shape[1]] = go
        _, gs, _ = ism.ism_simulate_backward(ROOM, [0.0] * 6, ps, PR[None], [3] * 3, length / FS, FS, grad_out, Tw=taps / FS)
        return np.sum(gs.cpu().numpy().astype(np.float64) * u, axis=1) / r

    assert np.max(np.abs(along(n) - along(1600)) * (4 * np.pi * r) / (K * norm2)) <= 2 * ROUNDED
