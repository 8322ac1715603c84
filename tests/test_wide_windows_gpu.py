"""Windows of other than 32 taps: FP32 through Chebyshev moments (dense rooms), per tap over
binned ids (sparse rooms, FP32_DIRECT, short windows), against the FP64 oracle, at the
lengths where the slots of 32 taps, the mask of the last taps and the choice of form change.  Bound: that of FP32, 1e-5 of the peak (test_parity_gpu.py); the same call twice and
a call inside a batch of other windows are bitwise the same.
"""
import numpy as np
import pytest

import oracle
from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS = 16000.0
# ~200 images per 32-sample delay bin, and ~2
DENSE = dict(L=[3.3, 4.1, 2.6], T=0.15, ps=[[1.1, 0.9, 1.3], [2.9, 3.5, 0.4]], pr=[[2.2, 2.8, 1.9]])
SPARSE = dict(L=[17.3, 14.1, 7.6], T=0.1, ps=[[5.1, 2.9, 3.3], [12.9, 11.5, 1.4]], pr=[[9.2, 7.8, 1.9]])
BETA = np.array([0.8, -0.75, 0.9, 0.7, 0.85, 0.65], np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _run(c, taps, prec, mic="omni", orient=None):
    Tw = float(np.float32(taps / FS))
    N = oracle.nb_img_from_t(c["T"], c["L"], 343.0, Tw)
    kw = dict(mic_pattern=mic, orient_rcv=orient) if mic != "omni" else {}
    return ism.ism_simulate(c["L"], BETA, np.asarray(c["ps"], np.float32), np.asarray(c["pr"], np.float32), N, c["T"], FS,
                            Tw=Tw, prec=prec, **kw), N, Tw


@pytest.mark.parametrize("taps", [2.0, 5.3, 15.9, 16.0, 17.5, 31.0, 33.0, 40.0, 63.2, 64.0, 64.3, 95.7, 110.25, 128.0,
                                  176.4, 192.0, 224.5, 256.0])
@pytest.mark.parametrize("room", [DENSE, SPARSE], ids=["dense", "sparse"])
@pytest.mark.parametrize("prec", ["fp32", "fp32_direct"])
def test_forward(taps, room, prec):
    h, N, Tw = _run(room, taps, prec)
    again, _, _ = _run(room, taps, prec)
    assert torch.equal(h, again)
    got = h.cpu().numpy().astype(np.float64)
    for i, ps in enumerate(np.asarray(room["ps"], np.float32).astype(np.float64)):
        ref = oracle.rir(room["L"], BETA.astype(np.float64), 343.0, FS, Tw, ps,
                         np.asarray(room["pr"], np.float32)[0].astype(np.float64), N, got.shape[-1])
        assert np.max(np.abs(got[i, 0] - ref)) <= 1e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("room", [DENSE, SPARSE], ids=["dense", "sparse"])
def test_polar_pattern(room):
    """A cardioid is half the omnidirectional RIR plus half the figure of eight (linear in alpha)."""
    o = np.array([[0.3, -0.8, 0.4]], np.float32)
    a, b, c = (_run(room, 64.0, "fp32", m, o)[0].double() for m in ("cardioid", "omni", "bidirectional"))
    assert float((a - 0.5 * (b + c)).abs().max()) <= 1e-5 * float(b.abs().max())


def test_windows_of_several_lengths_in_one_batch():
    jobs, outs, alone, keep = [], [], [], []
    for room in (DENSE, SPARSE):
        for taps in (32.0, 64.0, 20.5, 176.4, 64.0, 6.0):
            Tw = float(np.float32(taps / FS))
            N = oracle.nb_img_from_t(room["T"], room["L"], 343.0, Tw)
            ps, pr = (torch.as_tensor(np.asarray(room[k], np.float32)).cuda() for k in ("ps", "pr"))
            h = _run(room, taps, "fp32")[0]
            out = torch.empty_like(h)
            jobs.append(ism.make_job(room["L"], BETA, ps, pr, N, room["T"], FS, out, Tw=Tw))
            outs.append(out)
            alone.append(h)
            keep.append((ps, pr))
    ism.ism_simulate_batch(jobs)
    torch.cuda.synchronize()
    for a, b in zip(outs, alone):
        assert torch.equal(a, b)
