"""The overlap-save form of the moving-source filtering (many short segments): against the
definition in FP64, at sizes where its blocks, pieces and groups of pieces end, with segments
longer than a piece, of unequal length, empty, and with samples before the first.

Bound: that of the FFT form, 1e-5 of the largest sum |x| |h| (test_auralize_gpu.py).
"""
import numpy as np
import pytest

from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _check(n_x, n_points, n_mics, n_s, starts=None):
    rng = np.random.default_rng(n_x + n_points + n_s)
    x = rng.normal(size=n_x).astype(np.float32)
    h = (rng.normal(size=(n_points, n_mics, n_s)) * np.exp(-np.arange(n_s) / (n_s / 3.0))).astype(np.float32)
    xd, hd = torch.from_numpy(x).cuda(), torch.from_numpy(h).cuda()
    y = ism.ism_auralize(xd, hd, starts=starts, method="fft")
    assert torch.equal(y, ism.ism_auralize(xd, hd, starts=starts, method="fft"))
    cut = [p * n_x // n_points for p in range(n_points)] if starts is None else list(starts)
    cut = [min(max(c, 0), n_x) for c in cut] + [n_x]
    ref = torch.zeros((n_mics, n_x + n_s - 1), dtype=torch.float64, device="cuda")
    mag = torch.zeros_like(ref)
    N = 1 << (n_x + n_s).bit_length()
    for p in range(n_points):
        a, b = cut[p], cut[p + 1]
        if b > a:
            seg, hp = xd[a:b].double(), hd[p].double()
            for acc, u, v in ((ref, seg, hp), (mag, seg.abs(), hp.abs())):
                z = torch.fft.irfft(torch.fft.rfft(u, n=N) * torch.fft.rfft(v, n=N), n=N)
                acc[:, a:a + n_s + b - a - 1] += z[:, :n_s + b - a - 1]
    assert float((y.double() - ref).abs().max()) <= 1e-5 * float(mag.max())


@pytest.mark.parametrize("n_x,n_points,n_mics,n_s", [
    (57600, 64, 8, 57600),     # the 48 kHz array
    (30000, 40, 3, 20011),     # an odd microphone count
    (2048 * 7, 7, 2, 40000),   # segments of exactly half the DFT length
    (2049 * 7, 7, 2, 40000),   # and one sample more: two pieces each
    (40001, 9, 1, 30000),      # three pieces each
    (3000, 3000, 1, 9000),     # one sample each
    (70000, 300, 2, 3197),     # more pieces than a stretch of the scan
    (5000, 50, 4, 100)])       # RIRs shorter than a block
def test_uniform_segments(n_x, n_points, n_mics, n_s):
    _check(n_x, n_points, n_mics, n_s)


@pytest.mark.parametrize("starts", [[0, 1, 1, 5, 9000, 9000, 30000, 49999], [700, 800, 20000, 20001, 33333, 45000, 50000, 50000],
                                    [-5, 0, 0, 0, 4096, 8192, 12288, 60000]], ids=["short", "late", "clamped"])
def test_given_segments(starts):
    _check(50000, 8, 4, 25000, starts)
