"""Accuracy of the FP32 forms of windows of other than 32 taps against the FP64 oracle, in dense
rooms, where a Chebyshev series stands in for the taps of the windows that it follows.

Bound: an image's taps pass about eight roundings of 2^-24 (reciprocals, the amplitude's
products, the window's), 1e-7 of their norm together; a RIR's relative error stays below twice
that, 2e-7, unless something but rounding adds to it (a series over the cut taps of 17.5, 20.8
or 24.8 taps: 2.4e-7 to 3.7e-7).
"""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 16000.0
ROOM, T = [3.3, 4.1, 2.6], 0.3
BETA = np.array([0.8, -0.75, 0.9, 0.7, 0.85, 0.65], np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _errors(taps, prec, n_rir=6):
    """Relative errors (norms) of n_rir RIRs."""
    rng = np.random.default_rng(int(10 * taps))
    ps, pr = (rng.uniform(0.4, np.array(ROOM) - 0.4, (n, 3)).astype(np.float32) for n in (n_rir, 1))
    Tw = float(np.float32(taps / FS))
    N = oracle.nb_img_from_t(T, ROOM, 343.0, Tw)
    got = ism.ism_simulate(ROOM, BETA, ps, pr, N, T, FS, Tw=Tw, prec=prec).cpu().numpy().astype(np.float64)[:, 0]
    ref = oracle.rir_list(ROOM, BETA.astype(np.float64), 343.0, FS, Tw, ps.astype(np.float64),
                          np.broadcast_to(pr[0].astype(np.float64), ps.shape), N, got.shape[-1])
    return np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)


# ends in the middle of a sample interval, close to its ends, and on a sample; both sides of the
# length from which any window goes through the series
@pytest.mark.parametrize("taps", [16.0, 16.8, 17.5, 18.0, 18.8, 20.8, 24.8, 28.8, 33.3, 40.5, 44.1, 50.7, 63.2, 64.0, 79.0, 81.0])
def test_dense_windows(taps):
    assert np.sqrt(np.mean(_errors(taps, "fp32") ** 2)) <= 2e-7


def test_cut_windows_have_no_more_error_than_the_taps_one_by_one():
    """The shortest windows that end inside a sample interval and go through the series."""
    taps = [46.5, 47.0, 47.7, 48.6, 49.0, 50.7, 51.3, 53.0, 55.5, 57.4, 60.3, 61.0, 63.2, 65.0, 67.7, 70.4, 73.0, 75.1, 77.0, 79.0]
    series, direct = (np.concatenate([_errors(t, p, 8) for t in taps]) for p in ("fp32", "fp32_direct"))
    assert np.mean(series ** 2) <= np.mean(direct ** 2)


def test_series_has_no_more_error_than_the_taps_one_by_one():
    """Windows that go through the series, over lengths whose rounded coefficients differ."""
    taps = [16.0, 18.0, 24.0, 36.0, 44.0, 50.0, 64.0, 82.5, 88.2, 96.7, 110.25, 128.0, 150.3, 176.4, 192.0, 224.5]
    series, direct = (np.concatenate([_errors(t, p) for t in taps]) for p in ("fp32", "fp32_direct"))
    assert np.mean(series ** 2) <= np.mean(direct ** 2)
