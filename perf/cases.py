"""The calls whose speed counts, as a user's program makes them, and what they return in 64 bits.

Four kinds of call cover the public entry points:

  rir     ism.ism_simulate (or ism_simulate_host): the RIRs of one room
  rooms   ism.ism_simulate_batch: a ragged batch of rooms in one call
  fit     torch_ism.rir, a squared error against measured RIRs, and its gradients
  filter  ism.ism_auralize: a signal through the RIRs of a moving source

Sizes are those of the package's synthetic workloads (workloads.py), of the tests, or
generic.  Room sizes and reverberation times come from the case, positions, signals and
noise seeds from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1810_11359_gb300 import ism, torch_ism

C = 343.0


# --------------------------------------------------------------------------- #
# The cases
# --------------------------------------------------------------------------- #
def _rir(name, L, rt60, fs, Tmax, n_src, n_rcv, taps=32, Tdiff=0.0, nb=0, beta=0.0, prec="fp32", mic="omni",
         envelope="sabine", host=False):
    case = dict(kind="rir", Lx=L[0], Ly=L[1], Lz=L[2], rt60=rt60, fs=fs, Tmax=Tmax, Tdiff=Tdiff, n_src=n_src,
                n_rcv=n_rcv, taps=taps, nb=nb, beta=beta, prec=prec, mic=mic, envelope=envelope, host=host)
    return dict(case, name=name) if name else case


def _rooms_case(name, n_rooms, rooms, fs=16000.0, taps=32, max_rcv=16):
    case = dict(kind="rooms", n_rooms=n_rooms, rooms=rooms, fs=fs, taps=taps, max_rcv=max_rcv)
    return dict(case, name=name) if name else case


def _fit(name, n_rooms, rooms, n_src, n_rcv, Tmax, taps=32, fs=16000.0):
    case = dict(kind="fit", n_rooms=n_rooms, rooms=rooms, n_src=n_src, n_rcv=n_rcv, Tmax=Tmax, taps=taps, fs=fs)
    return dict(case, name=name) if name else case


def _filter(name, n_x, n_points, n_mics, n_s, fs, method, ragged=False):
    case = dict(kind="filter", n_x=n_x, n_points=n_points, n_mics=n_mics, n_s=n_s, fs=fs, method=method, ragged=ragged)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call: one RIR of a small room, where launches and latency count
        _rir("one_rir_16k", (3.0, 4.0, 2.5), 0.0, 16000.0, 0.3, 1, 1, nb=22, beta=0.7),
        # host positions in, host RIRs out: one request of a program without device memory
        _rir("host_4rir_tail_16k", (5.2, 3.7, 2.9), 0.45, 16000.0, 0.45, 1, 4, Tdiff=0.2, host=True),
        # no window given (taps 0: 4 ms, 64 taps at 16 kHz): the paper's small room, one source, a microphone set
        _rir("default_window_16rir_16k", (3.0, 4.0, 2.5), 0.7, 16000.0, 0.7, 1, 16, taps=0),
        # no window given at 44.1 kHz (176.4 taps), cardioid microphones, the Lehmann-Johansson tail
        _rir("default_window_15rir_44k_tail", (7.1, 5.3, 2.8), 0.6, 44100.0, 0.6, 5, 3, taps=0, Tdiff=0.15,
             mic="cardioid", envelope="lj"),
        # data generation: every source-microphone pair of a room, full image-source RIRs
        _rir("batched_128rir_16k", (6.0, 5.0, 3.0), 0.6, 16000.0, 0.6, 4, 32),
        # a moving source over a microphone array: many RIRs at 48 kHz, images early, tail late
        _rir("array_512rir_48k_tail", (10.0, 8.0, 3.5), 1.2, 48000.0, 1.2, 64, 8, Tdiff=0.3),
        # the reduced tap arithmetic, on half of the data-generation call
        _rir("fp16x2_64rir_16k", (6.0, 5.0, 3.0), 0.6, 16000.0, 0.6, 4, 16, prec="fp16x2"),
        # a batch of a simulation service: rooms of all sizes, 1 to 16 microphones each
        _rooms_case("rooms_32_16k_tail", 32, 4),
        # a training step: 256 rooms, the gradients of walls and positions
        _fit("fit_256rooms_16k", 256, 5, 1, 1, 0.4),
        # fitting one room to measurements with the default window
        _fit("fit_default_window_8rir_16k", 1, 7, 1, 8, 0.3, taps=0),
        # the array's RIRs applied to a signal
        _filter("filter_64x8_48k", 57600, 64, 8, 57600, 48000.0, "auto"),
        # a short clip through a few RIRs, segments of unequal length, the call without a method
        _filter("filter_10x2_16k", 12001, 10, 2, 4801, 16000.0, "none", ragged=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the listed cases' ranges (in their logarithm), cut to the cost of the largest ones."""
    kind = rng.choice(["rir", "rir", "rir", "rooms", "fit", "filter"])
    if kind == "rir":
        while True:
            L = tuple(round(rng.uniform(lo, hi), 2) for lo, hi in ((3.0, 10.0), (3.0, 8.0), (2.4, 4.0)))
            rt60 = round(rng.uniform(0.2, 1.2), 3)
            if not _feasible(L, rt60):
                continue
            fs = rng.choice([8000.0, 16000.0, 16000.0, 44100.0, 48000.0])
            tail = rng.random() < 0.5
            Tdiff = round(min(rng.uniform(0.1, 0.3), 0.7 * rt60), 3) if tail else 0.0
            prec = rng.choice(["fp32"] * 6 + ["fp32_direct", "fp16x2"])
            c = _rir(None, L, rt60, fs, rt60, _log_int(rng, 1, 64), _log_int(rng, 1, 32),
                     taps=rng.choice([32, 32, 0]), Tdiff=Tdiff, prec=prec,
                     mic=rng.choice(["omni", "omni", "cardioid", "hypercardioid"]),
                     envelope=rng.choice(["sabine", "lj"]) if tail else "sabine")
            n_rir = c["n_src"] * c["n_rcv"]
            if _images(c) * n_rir * max(1.0, _taps(c) / 32) <= 5.0e7 and n_rir * _len(c["Tmax"], fs) <= 2.9e7:
                return c
    if kind == "rooms":
        return _rooms_case(None, _log_int(rng, 2, 32), rng.randrange(1 << 20), fs=rng.choice([8000.0, 16000.0]),
                           taps=rng.choice([32, 32, 0]), max_rcv=rng.choice([4, 9, 16]))
    if kind == "fit":
        while True:
            c = _fit(None, _log_int(rng, 1, 256), rng.randrange(1 << 20), _log_int(rng, 1, 3), _log_int(rng, 1, 12),
                     round(rng.uniform(0.1, 0.4), 3), taps=rng.choice([32, 32, 0]))
            if sum(_images(r) for r in _room_list(c)) * c["n_src"] * c["n_rcv"] * max(1.0, _taps(c) / 32) <= 1.2e7:
                return c
    while True:
        fs = rng.choice([16000.0, 16000.0, 48000.0])
        n_x, n_s = _log_int(rng, 0.3 * fs, 3.0 * fs), _log_int(rng, 0.2 * fs, 1.2 * fs)
        c = _filter(None, n_x, _log_int(rng, 4, 64), _log_int(rng, 1, 8), n_s, fs,
                    rng.choice(["none", "auto", "auto"]), ragged=rng.random() < 0.4)
        if n_x * n_s * c["n_mics"] <= (2.6e10 if c["method"] == "auto" else 1.0e10):
            return c


# --------------------------------------------------------------------------- #
# Sizes
# --------------------------------------------------------------------------- #
def _len(T, fs):
    return int(math.ceil(float(np.float32(T)) * fs * (1.0 - 1e-6)))


def _n_ism(c):
    n = _len(c["Tmax"], c["fs"])
    return min(n, _len(c["Tdiff"], c["fs"])) if 0.0 < c["Tdiff"] < c["Tmax"] else n


def _taps(c):
    return float(c["taps"]) if c["taps"] else 4e-3 * c["fs"]


def _window(c):
    """The window length argument of the call, in seconds (0: the default)."""
    return c["taps"] / c["fs"] if c["taps"] else 0.0


def _feasible(L, rt60):
    """Whether every wall's absorption is below 1 for this reverberation time."""
    S = 2.0 * (L[0] * L[1] + L[0] * L[2] + L[1] * L[2])
    return 0.161 * L[0] * L[1] * L[2] / (rt60 * S) < 0.999


def _room_list(c):
    """The rooms of a "rooms" or "fit" case."""
    rng = np.random.default_rng(c["rooms"])
    out = []
    while len(out) < c["n_rooms"]:
        if c["kind"] == "rooms":
            L, rt60, n_rcv = rng.uniform(3.0, 10.0, 3), float(rng.uniform(0.2, 1.0)), int(rng.integers(1, c["max_rcv"] + 1))
            if not _feasible(L, rt60):
                continue
            out.append(dict(Lx=L[0], Ly=L[1], Lz=L[2], rt60=rt60, fs=c["fs"], Tmax=rt60, Tdiff=min(0.25, rt60), nb=0,
                            taps=c["taps"], n_src=1, n_rcv=n_rcv, beta=0.0))
        else:
            L, rt60 = rng.uniform(4.0, 8.0, 3), float(rng.uniform(0.3, 0.8))
            if not _feasible(L, rt60):
                continue
            out.append(dict(Lx=L[0], Ly=L[1], Lz=L[2], rt60=rt60, fs=c["fs"], Tmax=c["Tmax"], Tdiff=0.0, nb=0,
                            taps=c["taps"], n_src=c["n_src"], n_rcv=c["n_rcv"], beta=0.0))
    return out


def _images(c):
    """Image sources of one RIR whose pulse reaches its image-source samples: the sphere of reach, or the whole grid."""
    reach = (_n_ism(c) + _taps(c) / 2) * C / c["fs"]
    sphere = 4.0 / 3.0 * math.pi * reach ** 3 / (c["Lx"] * c["Ly"] * c["Lz"])
    return min(sphere, float(c["nb"]) ** 3) if c["nb"] else sphere


def work(case):
    """Per image: its delay and amplitude (42 operations) and a sum over its pulse (16); per tail sample 12; an FFT
    filter's 5 n log2 n per RIR.  Bytes: positions and signals read, results written, RIRs of a filter read."""
    if case["kind"] == "filter":
        n = case["n_s"] + case["n_x"] // case["n_points"]
        rirs = case["n_points"] * case["n_mics"]
        return {"bytes": 4 * (case["n_x"] + rirs * case["n_s"] + case["n_mics"] * (case["n_x"] + case["n_s"] - 1)),
                "flops": rirs * 2.5 * n * math.log2(n)}
    rooms = [case] if case["kind"] == "rir" else _room_list(case)
    nbytes = flops = 0.0
    for r in rooms:
        n_rir, n = r["n_src"] * r["n_rcv"], _len(r["Tmax"], r["fs"])
        nbytes += 4 * n_rir * n + 12 * (r["n_src"] + r["n_rcv"])
        flops += n_rir * (58.0 * _images(r) + 12.0 * (n - _n_ism(r)))
    if case["kind"] == "fit":   # the gradient reads dLoss/dh again; an image's adjoint costs about as much as itself
        nbytes, flops = 3 * nbytes, 2 * flops
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------- #
# What a program holds before the call, and the call
# --------------------------------------------------------------------------- #
def _inside(rng, r, n, margin=0.5):
    L = np.array([r["Lx"], r["Ly"], r["Lz"]])
    return (margin + (L - 2 * margin) * rng.random((n, 3))).astype(np.float32)


def _positions(rng, r):
    """Sources and microphones of one room: many sources are points of a path, with microphones on a circle."""
    if r["n_src"] < 16:
        return _inside(rng, r, r["n_src"]), _inside(rng, r, r["n_rcv"])
    a, b = _inside(rng, r, 2).astype(np.float64)
    t = np.linspace(0.0, 1.0, r["n_src"])[:, None]
    centre = _inside(rng, r, 1, margin=0.6)[0].astype(np.float64)
    ang = 2 * np.pi * np.arange(r["n_rcv"]) / r["n_rcv"]
    ring = np.stack([0.05 * np.cos(ang), 0.05 * np.sin(ang), 0.0 * ang], axis=1)
    return (a * (1 - t) + b * t).astype(np.float32), (centre + ring).astype(np.float32)


def _walls(r):
    return [r["beta"]] * 6 if r["beta"] else list(ism.ism_beta_sabine([r["Lx"], r["Ly"], r["Lz"]], r["rt60"]))


def _grid(r):
    if r["nb"]:
        return [r["nb"]] * 3
    T = r["Tdiff"] if 0.0 < r["Tdiff"] < r["Tmax"] else r["Tmax"]
    return ism.ism_nb_img_from_t(T, [r["Lx"], r["Ly"], r["Lz"]], C, _window(r) or 4e-3)


def _filter_inputs(case, seed):
    """A speech-like signal (noise under a slow envelope), RIRs with a decay, and the segment starts."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n_x, P, M, n_s = case["n_x"], case["n_points"], case["n_mics"], case["n_s"]
    t = torch.arange(n_x, device="cuda") / case["fs"]
    x = torch.randn(n_x, generator=g, device="cuda") * (0.55 + 0.45 * torch.sin(2 * math.pi * 3.0 * t))
    decay = torch.exp(-6.9 * torch.arange(n_s, device="cuda") / n_s)
    h = torch.randn((P, M, n_s), generator=g, device="cuda") * (0.1 * decay)
    starts = None
    if case["ragged"]:
        cuts = np.sort(np.random.default_rng(seed).integers(0, n_x, P - 1))
        starts = torch.tensor([0, *cuts], dtype=torch.int32, device="cuda")
    return x, h, starts


def _target(case, seed):
    """Measured RIRs to fit: decaying noise."""
    n = _len(case["Tmax"], case["fs"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    decay = torch.exp(-6.9 * torch.arange(n, device="cuda") / n)
    return 0.02 * torch.randn((case["n_rooms"], case["n_src"], case["n_rcv"], n), generator=g, device="cuda") * decay


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    if case["kind"] == "filter":
        x, h, starts = _filter_inputs(case, seed)
        return dict(case=case, x=x, h=h, starts=starts)
    if case["kind"] == "rir":
        ps, pr = _positions(rng, case)
        kw = dict(Tdiff=case["Tdiff"], Tw=_window(case), c=C, prec=case["prec"], seed=seed)
        if case["mic"] != "omni":
            kw.update(mic_pattern=case["mic"], orient_rcv=dev(rng.standard_normal((case["n_rcv"], 3)).astype(np.float32)))
        if case["envelope"] != "sabine":
            kw.update(envelope=case["envelope"])
        if not case["host"]:
            ps, pr = dev(ps), dev(pr)
        return dict(case=case, L=[case["Lx"], case["Ly"], case["Lz"]], beta=_walls(case), ps=ps, pr=pr, nb=_grid(case), kw=kw)
    rooms = _room_list(case)
    L = np.array([[r["Lx"], r["Ly"], r["Lz"]] for r in rooms])
    beta = np.array([_walls(r) for r in rooms])
    nb = np.array([_grid(r) for r in rooms], np.int32)
    pos = [_positions(rng, r) for r in rooms]
    if case["kind"] == "rooms":   # the jobs of rooms whose positions a program updates in place
        pos = [(dev(a), dev(b)) for a, b in pos]
        outs = [torch.empty((1, r["n_rcv"], _len(r["Tmax"], r["fs"])), device="cuda") for r in rooms]
        jobs = [ism.make_job(L[i], beta[i], pos[i][0], pos[i][1], nb[i], r["Tmax"], r["fs"], outs[i], Tdiff=r["Tdiff"],
                             Tw=_window(r), c=C, seed=seed + i) for i, r in enumerate(rooms)]
        return dict(case=case, jobs=jobs, outs=outs, pos=pos)
    leaf = lambda a: dev(a.astype(np.float32)).requires_grad_()  # noqa: E731
    return dict(case=case, L=L, nb=nb, target=_target(case, seed), beta=leaf(beta), ps=leaf(np.stack([p[0] for p in pos])),
                pr=leaf(np.stack([p[1] for p in pos])))


def run(state):
    case, s = state["case"], state
    if case["kind"] == "rir":
        call = ism.ism_simulate_host if case["host"] else ism.ism_simulate
        return call(s["L"], s["beta"], s["ps"], s["pr"], s["nb"], case["Tmax"], case["fs"], **s["kw"])
    if case["kind"] == "rooms":
        ism.ism_simulate_batch(s["jobs"])
        return s["outs"]
    if case["kind"] == "fit":
        h = torch_ism.rir(s["L"], s["beta"], s["ps"], s["pr"], case["Tmax"], case["fs"], Tw=_window(case), nb_img=s["nb"], c=C)
        loss = ((h - s["target"]) ** 2).sum()
        grads = torch.autograd.grad(loss, (s["beta"], s["ps"], s["pr"]))
        return {"h": h.detach(), "loss": loss.detach(), "grads": grads}
    return ism.ism_auralize(s["x"], s["h"], starts=s["starts"], method=None if case["method"] == "none" else case["method"])


# --------------------------------------------------------------------------- #
# The same in 64 bits, from the equations
# --------------------------------------------------------------------------- #
_F64 = torch.float64


def _axis(L, xs, xr, beta0, beta1, n):
    """Image offsets x_n - x_r and reflection products of one axis, for image indices n."""
    even = n % 2 == 0
    m = n.to(_F64)
    d = torch.where(even, m * L + xs, (m + 1) * L - xs) - xr
    e0 = torch.where(even, n.abs() // 2, (n - 1).abs() // 2)
    e1 = torch.where(even, n.abs() // 2, (n + 1).abs() // 2)
    return d, beta0 ** e0 * beta1 ** e1


def _exact_images(r, beta, ps, pr, orient=None, alpha=1.0):
    """The image-source samples of one source-microphone pair (beta, ps, pr: 64-bit tensors, differentiable)."""
    fs, n_ism, taps = r["fs"], _n_ism(r), _taps(r)
    H = math.ceil(taps / 2 - 1e-9)
    reach = (n_ism + H + 1) * C / fs
    L = [float(r["Lx"]), float(r["Ly"]), float(r["Lz"])]
    axes = []
    for a in range(3):
        M = int(math.ceil(reach / L[a])) + 1
        n = torch.arange(-(r["nb"] // 2), (r["nb"] + 1) // 2) if r["nb"] else torch.arange(-M, M + 1)
        axes.append(_axis(L[a], ps[a], pr[a], beta[2 * a], beta[2 * a + 1], n.to(ps.device)))
    with torch.no_grad():   # the images within reach
        sq = [d * d for d, _ in axes]
        keep = (sq[0][:, None, None] + sq[1][None, :, None] + sq[2][None, None, :] < reach * reach).nonzero()
    h = torch.zeros(n_ism, dtype=_F64, device=ps.device)
    j = torch.arange(-H, H + 2, device=ps.device)
    step = max(1, int(2.5e7 / j.numel()))
    for i in range(0, keep.shape[0], step):
        ix, iy, iz = keep[i:i + step].T
        dx, dy, dz = axes[0][0][ix], axes[1][0][iy], axes[2][0][iz]
        d = torch.sqrt(dx * dx + dy * dy + dz * dz)
        amp = axes[0][1][ix] * axes[1][1][iy] * axes[2][1][iz] / (4 * math.pi * d)
        if alpha != 1.0:
            amp = amp * (alpha + (1 - alpha) * (orient[0] * dx + orient[1] * dy + orient[2] * dz) / d)
        delay = d * (fs / C)
        k = torch.floor(delay.detach()).long()[:, None] + j
        x = k - delay[:, None]
        w = torch.where(x.abs() < taps / 2, 0.5 * (1 + torch.cos(2 * math.pi * x / taps)), 0.0)
        v = amp[:, None] * w * torch.sinc(x)
        ok = (k >= 0) & (k < n_ism)
        h = h.index_add(0, k.clamp(0, n_ism - 1).reshape(-1), torch.where(ok, v, 0.0).reshape(-1))
    return h


def _noise(seed, rir, n, device):
    """Unit-variance logistic noise from Philox4x32-10, counter (k / 4, rir, 0, 0)."""
    mask = 0xFFFFFFFF

    def mul(m, a):   # 32 x 32 -> high and low words, in 64-bit signed arithmetic
        lo, hi = m * (a & 0xFFFF), m * (a >> 16)
        top = hi + (lo >> 16)
        return top >> 16, ((top & 0xFFFF) << 16) | (lo & 0xFFFF)

    nb = (n + 3) // 4
    c = [torch.arange(nb, device=device), torch.full((nb,), rir, device=device), torch.zeros(nb, dtype=torch.int64, device=device),
         torch.zeros(nb, dtype=torch.int64, device=device)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u = ((torch.stack(c, 1).reshape(-1)[:n] >> 9).to(_F64) + 0.5) * 2.0 ** -23
    return math.sqrt(3.0) / math.pi * torch.log(u / (1 - u))


def _decay(r, beta, n, device):
    """Power envelope E(t_k) of the diffuse tail, k < n."""
    L, fs = [r["Lx"], r["Ly"], r["Lz"]], r["fs"]
    k = torch.arange(n, dtype=_F64, device=device)
    if r["envelope"] == "sabine":
        S = [L[1] * L[2], L[1] * L[2], L[0] * L[2], L[0] * L[2], L[0] * L[1], L[0] * L[1]]
        T60 = 0.161 * L[0] * L[1] * L[2] / sum(s * (1 - b * b) for s, b in zip(S, beta))
        return 10.0 ** (-6.0 * k / fs / T60)
    x, w = np.polynomial.legendre.leggauss(80)   # the average over an octant of directions
    ang, w = (x + 1) * math.pi / 4, w * math.pi / 4
    st, ct = np.sin(ang), np.cos(ang)
    gam = [-math.log(abs(beta[2 * a] * beta[2 * a + 1])) * C / (fs * L[a]) for a in range(3)]
    rate = st[:, None] * (ct[None, :] * gam[0] + st[None, :] * gam[1]) + ct[:, None] * gam[2]
    wt = torch.from_numpy((w[:, None] * w[None, :] * st[:, None] * 2 / math.pi).reshape(-1)).to(device)
    rate = torch.from_numpy(rate.reshape(-1)).to(device)
    return torch.cat([torch.exp(-kk[:, None] * rate) @ wt for kk in k.split(4096)])


def _exact_rir(r, beta, ps, pr, orient, seed):
    """[n_src, n_rcv, n] with the tail."""
    dev = ps.device
    n, n_ism, fs = _len(r["Tmax"], r["fs"]), _n_ism(r), r["fs"]
    alpha = {"omni": 1.0, "cardioid": 0.5, "hypercardioid": 0.25}[r["mic"]]
    out = torch.zeros((r["n_src"], r["n_rcv"], n), dtype=_F64, device=dev)
    if n_ism < n:
        E = _decay(r, beta.tolist(), n, dev)
        W = min(n_ism, math.ceil(0.02 * fs - 1e-9))
    for i in range(r["n_src"]):
        for m in range(r["n_rcv"]):
            o = None
            if alpha != 1.0:
                o = orient[m] / orient[m].norm()
            h = _exact_images(r, beta, ps[i], pr[m], o, alpha)
            out[i, m, :n_ism] = h
            if n_ism < n:
                A = (h[n_ism - W:] ** 2 * E[n_ism] / E[n_ism - W:n_ism]).mean()
                z = _noise(seed, i * r["n_rcv"] + m, n, dev)
                out[i, m, n_ism:] = (z * torch.sqrt(A * E / E[n_ism]))[n_ism:]
    return out


def exact(case, seed):
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    f64 = lambda a: torch.as_tensor(np.asarray(a, np.float32)).to(dev, _F64)  # noqa: E731
    if case["kind"] == "filter":
        x, h, starts = _filter_inputs(case, seed)
        n_x, P, M, n_s = case["n_x"], case["n_points"], case["n_mics"], case["n_s"]
        cut = starts.tolist() if starts is not None else [p * n_x // P for p in range(P)]
        cut.append(n_x)
        y = torch.zeros((M, n_x + n_s - 1), dtype=_F64, device=dev)
        for p in range(P):
            a, b = cut[p], cut[p + 1]
            if b > a:
                N = n_s + b - a - 1
                seg = torch.fft.rfft(x[a:b].to(_F64), n=N)
                y[:, a:a + N] += torch.fft.irfft(seg * torch.fft.rfft(h[p].to(_F64), n=N), n=N)
        return y
    rng = np.random.default_rng(seed)
    if case["kind"] == "rir":
        if _images(case) * case["n_src"] * case["n_rcv"] * _taps(case) > 4.0e9:   # too long in 64 bits
            return None
        ps, pr = _positions(rng, case)
        orient = rng.standard_normal((case["n_rcv"], 3)) if case["mic"] != "omni" else None
        h = _exact_rir(case, f64(_walls_64(case)), f64(ps), f64(pr), None if orient is None else f64(orient), seed)
        return h.cpu().numpy() if case["host"] else h
    rooms = _room_list(case)
    pos = [_positions(rng, r) for r in rooms]
    if case["kind"] == "rooms":
        return [_exact_rir(dict(r, mic="omni", envelope="sabine"), f64(_walls_64(r)), f64(pos[i][0]), f64(pos[i][1]), None,
                           seed + i) for i, r in enumerate(rooms)]
    target = _target(case, seed).to(_F64)
    h, loss, grads = torch.zeros_like(target), 0.0, [[], [], []]
    for b, r in enumerate(rooms):
        leaves = [f64(v).requires_grad_() for v in (_walls_64(r), pos[b][0], pos[b][1])]
        g = [torch.zeros_like(v) for v in leaves]
        for i in range(r["n_src"]):
            for m in range(r["n_rcv"]):
                hp = _exact_images(r, leaves[0], leaves[1][i], leaves[2][m])
                part = ((hp - target[b, i, m]) ** 2).sum()
                for acc, v in zip(g, torch.autograd.grad(part, leaves)):
                    acc += v
                h[b, i, m] = hp.detach()
                loss = loss + part.detach()
        for k in range(3):
            grads[k].append(g[k])
    return {"h": h, "loss": loss, "grads": tuple(torch.stack(g) for g in grads)}


def _walls_64(r):
    """Reflection coefficients: given, or equal ones whose Sabine reverberation time is the room's."""
    if r["beta"]:
        return [r["beta"]] * 6
    L = [r["Lx"], r["Ly"], r["Lz"]]
    S = 2.0 * (L[0] * L[1] + L[0] * L[2] + L[1] * L[2])
    return [math.sqrt(1.0 - 0.161 * L[0] * L[1] * L[2] / (r["rt60"] * S))] * 6
