"""The Chebyshev form's shells are as thick as the launch asks; an RIR is bitwise the same at
any thickness: calls of few RIRs (thin shells, one wave) against the same RIRs out of one call
of many (8 bins).
"""
import numpy as np
import pytest

from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 16000.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("L,T,taps", [([6.0, 5.0, 3.0], 0.6, 32), ([3.0, 4.0, 2.5], 0.35, 64), ([8.0, 6.0, 3.0], 0.3, 32)])
def test_calls_of_few_rirs(L, T, taps):
    beta = ism.ism_beta_sabine(L, T)
    Tw = taps / FS
    N = ism.ism_nb_img_from_t(T, L, 343.0, Tw)
    rng = np.random.default_rng(11)
    ps = rng.uniform(0.5, np.array(L) - 0.5, (1, 3)).astype(np.float32)
    pr = rng.uniform(0.5, np.array(L) - 0.5, (96, 3)).astype(np.float32)
    many = ism.ism_simulate(L, beta, ps, pr, N, T, FS, Tw=Tw)
    for n in (1, 2, 4, 7, 8, 9, 10, 11, 16, 19, 20, 21, 34, 40):
        few = ism.ism_simulate(L, beta, ps, pr[:n], N, T, FS, Tw=Tw)
        assert torch.equal(few, many[:, :n])
