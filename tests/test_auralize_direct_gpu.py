"""The direct filtering at the edges of its chunks of 128 taps, tiles of 128 outputs and groups of
microphones, with few and with many chunks and tiles, against FP64.

Bound per output: an FP32 sum of n products in any order is within n 2^-24 of the sum of their
magnitudes (n: the RIR's length, and 32 for the sums of the warps and the products' own rounding).
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


def _reference(x, h, starts):
    P, n = h.shape[0], x.shape[0] + h.shape[2] - 1
    cut = [min(max(int(s), 0), x.shape[0]) for s in starts] + [x.shape[0]]
    y = torch.zeros((h.shape[1], n), dtype=torch.float64, device="cuda")
    for p in range(P):
        a, b = cut[p], cut[p + 1]
        if b > a:
            seg = x[a:b].flip(0)[None, None]
            y[:, a:b + h.shape[2] - 1] += torch.nn.functional.conv1d(h[p][:, None], seg, padding=b - a - 1)[:, 0]
    return y


@pytest.mark.parametrize("n_s", [1, 51, 128, 129, 142, 256, 1000])
@pytest.mark.parametrize("n_x,P,given", [(260, 1, False), (997, 7, True), (2100, 150, False), (2100, 150, True), (70001, 3, True)])
@pytest.mark.parametrize("n_mics", [1, 2, 3, 9])
def test_edges(n_x, P, given, n_mics, n_s):
    g = torch.Generator(device="cuda").manual_seed(n_x + n_s)
    x = torch.randn(n_x, generator=g, device="cuda")
    h = torch.randn((P, n_mics, n_s), generator=g, device="cuda")
    starts = [p * n_x // P for p in range(P)]
    if given:   # some equal, the first after sample 0
        starts = np.sort(np.random.default_rng(n_s).integers(0, n_x, P)).tolist()
    got = ism.ism_auralize(x, h, starts=starts if given else None)
    ref, mag = _reference(x.double(), h.double(), starts), _reference(x.double().abs(), h.double().abs(), starts)
    assert bool(((got.double() - ref).abs() <= (n_s + 32) * 2.0 ** -24 * mag).all())
