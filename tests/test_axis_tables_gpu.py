"""The tables of one axis, at the numbers of images where the powers of the reflection
coefficients leave their table (exponents of 32 and more) and where its bits change, against
the FP64 oracle: walls that reflect nearly everything, so that the highest powers count, and
walls of 0.  Bounds: 1e-5 of the peak (test_parity_gpu.py), 1e-4 of each gradient group's
largest (test_adjoint_gpu.py).
"""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, T, TW = 16000.0, 0.15, 0.002
SIDES = [0.5, 3.7, 2.9]
BETAS = {"high": [0.99, -0.985, 0.8, 0.7, -0.6, 0.9], "zero": [0.0, 0.99, 0.9, 0.0, 0.0, 0.0]}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [1, 2, 3, 11, 12, 13, 28, 60, 61, 123, 124, 125, 127, 129, 200, 253])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("beta", ["high", "zero"])
def test_against_the_oracle(n, axis, beta):
    L, b6 = np.roll(SIDES, axis), np.roll(np.float32(BETAS[beta]), 2 * axis)
    N = [5, 5, 5]
    N[axis] = n
    ps = np.roll([[0.2, 1.1, 0.7], [0.4, 2.2, 1.5]], axis, axis=1).astype(np.float32)
    pr = np.roll([[0.15, 1.4, 1.2]], axis, axis=1).astype(np.float32)
    n_s = oracle.n_samples(np.float32(T), FS)
    h = ism.ism_simulate(L, b6, ps, pr, N, T, FS, Tw=TW).cpu().numpy().astype(np.float64)
    g = np.random.default_rng(n).standard_normal((2, 1, n_s)).astype(np.float32)
    got = [v.cpu().numpy().astype(np.float64) for v in
           ism.ism_simulate_backward(L, b6, ps, pr, N, T, FS, torch.from_numpy(g), Tw=TW)]
    ref = [np.zeros(6), np.zeros((2, 3)), np.zeros((1, 3))]
    for i in range(2):
        args = (L, b6.astype(np.float64), 343.0, FS, float(np.float32(TW)), ps[i].astype(np.float64),
                pr[0].astype(np.float64), N, n_s)
        want = oracle.rir(*args)
        assert np.max(np.abs(h[i, 0] - want)) <= 1e-5 * np.max(np.abs(want))
        d = oracle.rir_grad(*args, g[i, 0].astype(np.float64))
        ref[0] += d[0]
        ref[1][i] += d[1]
        ref[2][0] += d[2]
    for a, b in zip(got, ref):
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))
