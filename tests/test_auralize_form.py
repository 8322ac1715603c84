"""Which form of the moving-source filtering a call gets (host only), and the overlap-save form
at sizes whose pieces fill several stretches of its scan, with given starts too.

The automatic choice has to go by the form that will run: sizes whose piece spectra do not fit
the overlap-save form's workspace would otherwise run the four-step form, which its estimate
never saw (892 points x 2 microphones: 4370 us against 206 us direct).
"""
import ctypes

import numpy as np
import pytest

from paper_1810_11359_gb300 import build as libbuild
from paper_1810_11359_gb300 import ism
from test_auralize_ols_gpu import _check

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


# n_x, points, microphones, n_S -> the automatic choice for the uniform cut and for given starts
FORMS = [((57600, 64, 8, 57600), "overlap_save", "overlap_save"),    # the 48 kHz array
         ((57600, 64, 2, 4800), "overlap_save", "overlap_save"),
         ((120217, 941, 8, 4858), "overlap_save", "overlap_save"),
         ((121813, 504, 1, 10101), "overlap_save", "overlap_save"),
         ((144000, 500, 2, 19200), "overlap_save", "overlap_save"),
         ((151061, 892, 2, 4875), "direct", "direct"),               # the piece spectra do not fit
         ((48000, 256, 2, 9600), "overlap_save", "direct"),          # those of given starts do not
         ((100000, 2000, 4, 8000), "direct", "direct"),
         ((4099, 64, 8, 517), "direct", "direct"),                   # too small for three launches
         ((30000, 3, 8, 20000), "four_step", "overlap_save"),        # few long segments
         ((900000, 40, 2, 300000), "direct", "direct")]              # longer than the FFT form takes


@pytest.mark.parametrize("size,uniform,given", FORMS, ids=["x".join(map(str, f[0])) for f in FORMS])
def test_automatic_choice(size, uniform, given):
    assert (ism.ism_auralize_workspace_size(*size, "auto") == 0) == (uniform == given == "direct")
    assert ism.ism_auralize_form(*size) == uniform
    assert ism.ism_auralize_form(*size, given_starts=True) == given
    assert ism.ism_auralize_form(*size, method="direct") == "direct"


def test_automatic_choice_never_takes_the_four_step_form_for_overlap_saves_time():
    """Over random sizes: four-step only where its own operations say so (2.55 of its lane
    operations a multiply-add of the direct form), whatever the overlap-save form would take."""
    rng = np.random.default_rng(4)
    for _ in range(3000):
        n_x, n_s = (int(v) for v in np.exp(rng.uniform(np.log(1000), np.log(2e5), 2)))
        P, M = int(min(n_x, np.exp(rng.uniform(0.0, np.log(3000))))), int(rng.integers(1, 17))
        for given in (False, True):
            if ism.ism_auralize_form(n_x, P, M, n_s, given_starts=given) != "four_step":
                continue
            logN = max(4, (n_x + n_s - 2).bit_length())
            N, pairs = 1 << logN, (M + 1) // 2
            ops = (P * (1 + pairs) + pairs) * 4 * N * logN + P * pairs * 4 * N
            assert M * n_x * n_s > 2.55 * ops, (n_x, P, M, n_s, given)


@pytest.mark.parametrize("size,given,form", [
    ((270, 99, 2, 16285), True, "direct"),         # its 99 pieces would follow one another on 5 CTAs
    ((541, 510, 9, 26015), True, "overlap_save"),  # 510 on 35, and the direct form slower still
    ((3438, 1, 1, 1000), True, "direct"),          # less than three launches
    ((4963, 88, 8, 9000), False, "overlap_save")])
def test_automatic_choice_counts_the_pieces_that_follow_one_another(size, given, form):
    assert ism.ism_auralize_form(*size, given_starts=given) == form


@pytest.mark.parametrize("size,given,form", [
    ((312, 44, 3, 6720), True, "four_step"),       # 44 pieces in turn take longer than its passes
    ((387, 107, 15, 2477), False, "four_step"),
    ((100, 100, 8, 9000), False, "overlap_save"),  # the passes longer still
    ((57600, 64, 8, 57600), False, "overlap_save")])
def test_fft_method_takes_the_faster_form(size, given, form):
    assert ism.ism_auralize_form(*size, method="fft", given_starts=given) == form


@pytest.mark.parametrize("size", [(57600, 64, 8, 57600), (57600, 64, 2, 4800), (30000, 64, 4, 3200), (144000, 500, 2, 19200)])
def test_workspace_of_the_overlap_save_form(size):
    """The automatic choice asks for the overlap-save form's piece spectra (18 KB each; of given
    starts up to 1.5 a point) and block sums (32 KB each; groups up to 562 CTAs more than the
    blocks of 2049 outputs or more), not for the four-step form's 64 to 96 MB of chunk."""
    n_x, P, M, n_s = size
    pieces = 1.5 * P + n_x / 2048 + 2
    sums = 562 + ((n_x + n_s - 1) // 2049 + 1) * ((M + 1) // 2)
    b = ism.ism_auralize_workspace_size(*size, "auto")
    assert 0 < b <= pieces * (18432 + 16) + sums * 32768 + 32768 + 1024
    assert b < ism.ism_auralize_workspace_size(*size, "fft") / 2


def test_form_arguments():
    with pytest.raises(ism.IsmError):
        ism.ism_auralize_form(0, 1, 1, 1)
    with pytest.raises(ism.IsmError):
        ism.ism_auralize_form(900000, 40, 2, 300000, method="fft")


@pytest.mark.gpu
@pytest.mark.parametrize("n_x,n_points,n_mics,n_s,given", [
    (70000, 300, 8, 20000, False),       # 300 pieces: two stretches of the scan
    (70000, 300, 8, 20000, True),        # up to 449
    (60000, 800, 8, 20000, False),       # four stretches
    (280000, 130, 8, 20000, False),      # two pieces a segment, 260
    (100, 100, 8, 9000, False),          # one sample each
    (70000, 300, 2, 3197, False),        # RIRs shorter than a block
    (5000, 50, 16, 100, True)])          # and than a segment
def test_overlap_save_over_many_pieces(n_x, n_points, n_mics, n_s, given):
    assert ism.ism_auralize_form(n_x, n_points, n_mics, n_s, "fft", given) == "overlap_save"
    starts = None
    if given:   # sorted, some equal, the first after sample 0
        starts = np.sort(np.random.default_rng(n_x).integers(0, n_x, n_points)).tolist()
        starts[n_points // 2] = starts[n_points // 2 - 1]
    _check(n_x, n_points, n_mics, n_s, starts)


@pytest.mark.gpu
@pytest.mark.parametrize("n_x,n_points,n_mics,n_s", [(15000, 300, 2, 1500), (57600, 64, 2, 4800)])
def test_automatic_call_runs_the_chosen_form(n_x, n_points, n_mics, n_s):
    torch.cuda.set_device(0)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(n_x, generator=g, device="cuda")
    h = torch.randn((n_points, n_mics, n_s), generator=g, device="cuda")
    starts = torch.arange(n_points, dtype=torch.int32, device="cuda") * (n_x // n_points)
    for s in (None, starts):
        form = ism.ism_auralize_form(n_x, n_points, n_mics, n_s, given_starts=s is not None)
        want = ism.ism_auralize(x, h, starts=s, method="direct" if form == "direct" else "fft")
        assert torch.equal(ism.ism_auralize(x, h, starts=s, method="auto"), want)


@pytest.mark.gpu
def test_automatic_call_with_less_workspace_runs_directly():
    """One byte below the least that any form takes, and none: the direct form."""
    torch.cuda.set_device(0)
    n_x, P, M, n_s = 57600, 64, 2, 4800
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(n_x, generator=g, device="cuda")
    h = torch.randn((P, M, n_s), generator=g, device="cuda")
    direct = ism.ism_auralize(x, h, method="direct")
    out = torch.empty_like(direct)
    ws = torch.empty(1 << 23, dtype=torch.uint8, device="cuda")
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    for w, n in ((ws, 1 << 20), (None, 0)):
        ism._check(ism.load().ism_auralize_ex(ptr(x), n_x, ptr(h), P, M, n_s, None, ptr(out), ism.AURALIZE_METHODS["auto"],
                                              None if w is None else ptr(w), n, ism._stream_ptr(None)))
        assert torch.equal(out, direct)


@pytest.mark.gpu
def test_fft_method_refuses_a_workspace_of_no_bytes():
    torch.cuda.set_device(0)
    x, h, out = torch.ones(3000, device="cuda"), torch.ones((3, 2, 900), device="cuda"), torch.empty((2, 3899), device="cuda")
    ws = torch.empty(1 << 23, dtype=torch.uint8, device="cuda")   # (so that even an accepting call stays inside)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    for n_mics in (1, 2):
        st = ism.load().ism_auralize_ex(ptr(x), 3000, ptr(h), 3, n_mics, 900, None, ptr(out), ism.AURALIZE_METHODS["fft"], ptr(ws),
                                        0, ism._stream_ptr(None))
        assert st == 3   # ISM_ERR_WORKSPACE_TOO_SMALL
