"""The shell walk of the fused kernels where a warp's 32 columns hold more candidates than
one pass takes (a very flat room), and at the shortest delays, where the split of the
squared offsets is coarsest against them: against the FP64 oracle.

Bounds: those of the forms they exercise (FP32 1e-5 of the peak; gradients 1e-4 of each
group's largest, see test_parity_gpu.py and test_adjoint_gpu.py).
"""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, TW = 16000.0, 32 / 16000


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


# a 31 cm ceiling: ~35 images of a column fall in a 256-sample shell, 32 columns above 1023 candidates
FLAT = dict(L=[4.1, 3.6, 0.31], beta=[0.9, 0.85, 0.8, 0.9, 0.97, 0.95], ps=[1.3, 2.1, 0.12], pr=[2.9, 0.8, 0.2], T=0.12)
# source and receiver 5 mm, 9 cm apart in a long room: s^2 well below one step of the split
NEAR = dict(L=[9.0, 7.0, 3.0], beta=[0.8, 0.75, 0.9, 0.7, 0.85, 0.65], ps=[4.0, 3.0, 1.5], pr=[4.003, 3.004, 1.5], T=0.35)
CLOSE = dict(NEAR, pr=[4.05, 3.06, 1.54])


def _case(c):
    T = np.float32(c["T"])
    N = oracle.nb_img_from_t(float(T), c["L"], 343.0, TW)
    return np.asarray(c["beta"], np.float32), np.asarray([c["ps"]], np.float32), np.asarray([c["pr"]], np.float32), T, N


@pytest.mark.parametrize("c", [FLAT, NEAR, CLOSE], ids=["flat", "near", "close"])
@pytest.mark.parametrize("prec", ["fp32", "fp32_direct"])
def test_forward(c, prec):
    beta, ps, pr, T, N = _case(c)
    h = ism.ism_simulate(c["L"], beta, torch.from_numpy(ps).cuda(), torch.from_numpy(pr).cuda(), N, float(T), FS, Tw=TW, prec=prec)
    got = h.cpu().numpy().astype(np.float64)[0, 0]
    ref = oracle.rir(c["L"], beta.astype(np.float64), 343.0, FS, float(np.float32(TW)), ps[0], pr[0], N, got.size)
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("c", [FLAT, CLOSE], ids=["flat", "close"])
def test_adjoint(c):
    beta, ps, pr, T, N = _case(c)
    n = oracle.n_samples(T, FS)
    g = np.random.default_rng(3).standard_normal(n).astype(np.float32)
    got = ism.ism_simulate_backward(c["L"], beta, ps, pr, N, float(T), FS, torch.from_numpy(g[None, None]), Tw=TW)
    ref = oracle.rir_grad(c["L"], beta.astype(np.float64), 343.0, FS, float(np.float32(TW)), ps[0].astype(np.float64),
                          pr[0].astype(np.float64), N, n, g.astype(np.float64))
    for a, b in zip(got, ref):
        a = a.cpu().numpy().astype(np.float64).reshape(-1)
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))


@pytest.mark.parametrize("eps", [0.0, 1e-12, 1e-10, 1e-9, 5e-9, 1e-8, 3e-8, 5e-8, -1e-9, -3e-8])
@pytest.mark.parametrize("prec", ["fp32", "fp32_direct"])
def test_delays_next_to_an_integer(eps, prec):
    """Direct paths of 10 - eps samples (k = 1 sample per metre): a fraction that rounds to 1."""
    fs, c, Tw = 343.0, 343.0, 32 / 343.0
    dx = np.float64(np.float32(10.0) - np.float32(2.0 ** -18))   # the FP32 grid of y sets s to ~1e-12
    dy = np.float32(np.sqrt((10.0 - eps) ** 2 - dx * dx))
    L, beta, N = [40.0, 38.0, 36.0], np.full(6, 0.5, np.float32), [5, 5, 5]
    ps = np.array([[8.0, 2.0 ** -7, 16.0]], np.float32)
    pr = np.array([[8.0 + dx, 2.0 ** -7 + dy, 16.0]], np.float32)
    h = ism.ism_simulate(L, beta, torch.from_numpy(ps).cuda(), torch.from_numpy(pr).cuda(), N, 0.25, fs, Tw=Tw, c=c, prec=prec)
    got = h.cpu().numpy().astype(np.float64)[0, 0]
    assert np.all(np.isfinite(got))
    ref = oracle.rir(L, beta.astype(np.float64), c, fs, float(np.float32(Tw)), ps[0].astype(np.float64),
                     pr[0].astype(np.float64), N, got.size)
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))
