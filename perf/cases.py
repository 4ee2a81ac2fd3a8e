"""The work this framework is measured on: RM synthesis calls of the sizes its users make.

Every case goes through the package's public entry points on inputs that are on
the GPU before the call.  Bands and grids are those of the repository's own
workloads (package module `inputs`): channels uniform in frequency (or in
lambda^2), a phi grid symmetric about zero, one to three Faraday-thin or
Burn-slab sources per line of sight (LOS) with noise on Q and U, flagged
channels holding interference that must not reach the result.
"""
import math

import numpy as np
import torch

import paper_1810_06250_gb300 as rms
from paper_1810_06250_gb300 import learned

C_LIGHT = 299792458.0

# first and last channel centre (Hz), largest |phi| of the grid and of the sources (rad m^-2)
BANDS = {
    "narrow": (120e6, 168e6, 50.0, 40.0),
    "lofar": (115e6, 178e6, 100.0, 40.0),
    "lofar_hr": (120.238e6, 166.087e6, 350.0, 300.0),
    "precision": (110e6, 190e6, 500.0, 450.0),
    "mwa": (72e6, 231e6, 2000.0, 1800.0),
}
CHUNK_VALUES = 1 << 25      # values of one temporary while inputs or 64-bit results are made


def listed():
    return [
        # the smallest cube of the tests: a postage stamp around one source, where latency counts
        dict(name="stamp", kind="synth", band="narrow", precision="bf16x3", layout="chan", nlos=256, nchan=64,
             nphi=101, flagged=0.0, uniform_l2=False),
        # a cut-out around one extended source, LOS-major as a rotated cube is stored, an odd number of LOS
        dict(name="cutout", kind="synth", band="lofar", precision="bf16x3", layout="los", nlos=5001, nchan=400,
             nphi=401, flagged=0.1, uniform_l2=False),
        # one LOFAR-HBA-like field, FITS plane order, the benchmark's second cube: F and the peak map
        dict(name="field", kind="synth", band="lofar", precision="bf16x3", layout="chan", nlos=512 * 512, nchan=400,
             nphi=401, flagged=0.1, uniform_l2=False),
        # the same band as a rotated cube at the tighter split precision, with an odd channel count (rows that
        # are not 16-byte aligned) and an odd number of LOS
        dict(name="field_rotated", kind="synth", band="lofar", precision="fp16x3", layout="los", nlos=200003,
             nchan=397, nphi=401, flagged=0.1, uniform_l2=False),
        # a quick look over a wide survey field in one BF16 product, no channel flagged
        dict(name="quicklook", kind="synth", band="precision", precision="bf16", layout="chan", nlos=400000,
             nchan=800, nphi=1001, flagged=0.0, uniform_l2=False),
        # the benchmark's MWA-like band and grid on 400 x 400 LOS: the largest contraction
        dict(name="wideband", kind="synth", band="mwa", precision="bf16x3", layout="chan", nlos=400 * 400, nchan=1536,
             nphi=4001, flagged=0.0, uniform_l2=False),
        # LOFAR high-resolution map: every peak output and no F (F of such a field does not fit the card)
        dict(name="peak_map", kind="map", band="lofar_hr", precision="bf16x3", layout="chan", nlos=200000, nchan=856,
             nphi=7000, flagged=0.0, uniform_l2=False),
        # the FP32 CUDA-core path that results are compared with
        dict(name="fp32_field", kind="synth", band="lofar", precision="fp32_table", layout="chan", nlos=100000,
             nchan=400, nphi=401, flagged=0.1, uniform_l2=False),
        # channels uniform in lambda^2: FFT synthesis of a whole field
        dict(name="fft_field", kind="synth", band="lofar", precision="fp32_czt", layout="chan", nlos=512 * 512,
             nchan=400, nphi=401, flagged=0.1, uniform_l2=True),
        # RM-CLEAN of the dirty spectra of a field's brighter part
        dict(name="clean", kind="clean", band="lofar", precision="bf16x3", layout="chan", nlos=20000, nchan=400,
             nphi=401, flagged=0.1, uniform_l2=False),
        # inference of the learned proposal: network, window centres, window synthesis
        dict(name="proposal", kind="proposal", band="lofar", precision="bf16x3", layout="los", nlos=512 * 512,
             nchan=400, nphi=401, flagged=0.1, uniform_l2=False),
        # the gradient of one training batch of the network
        dict(name="gradient", kind="gradient", band="lofar", precision="bf16x3", layout="los", nlos=4096, nchan=400,
             nphi=401, flagged=0.1, uniform_l2=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["synth"] * 6 + ["map", "clean", "proposal", "gradient"])
    precision = "bf16x3"
    uniform = False
    if kind == "synth":
        precision = rng.choice(["bf16x3"] * 4 + ["fp16x3"] * 2 + ["bf16", "fp32_table", "fp32_fly", "fp32_czt"])
    if precision == "fp32_czt":
        uniform = True
        band, nchan, nphi = "lofar", _log_int(rng, 64, 1000), _log_int(rng, 101, 1001)
        most = 1e11
    elif kind in ("clean", "proposal", "gradient"):
        band, nchan, nphi = "lofar", _log_int(rng, 128, 480), rng.randint(201, 501)
        most = 8e10
    else:
        band = rng.choice(sorted(BANDS))
        nchan = _log_int(rng, 48, 1536)
        top = {"narrow": 401, "lofar": 801, "lofar_hr": 7000, "precision": 2001, "mwa": 4001}[band]
        nphi = _log_int(rng, 101, top)
        most = 2e10 if precision.startswith("fp32") else 9e11
    nlos = _log_int(rng, 200, 300000)
    if kind == "clean":
        nlos = _log_int(rng, 200, 20000)
    if kind == "gradient":
        nlos = _log_int(rng, 500, 8192)
    nlos = max(200, min(nlos, int(most / (nchan * nphi))))
    flagged = rng.choice([0.0, 0.1])
    layout = "los" if kind == "gradient" else rng.choice(["chan", "los"])
    return dict(kind=kind, band=band, precision=precision, layout=layout, nlos=nlos, nchan=nchan, nphi=nphi,
                flagged=flagged, uniform_l2=uniform)


# ----------------------------------------------------------------------------- inputs
def _axes(case):
    """Frequencies (Hz), weights (0 for flagged channels), phi grid; FP64 on the host."""
    nu0, nu1, phi_max, _ = BANDS[case["band"]]
    n = case["nchan"]
    if case["uniform_l2"]:
        freq = C_LIGHT / np.sqrt(np.linspace((C_LIGHT / nu0) ** 2, (C_LIGHT / nu1) ** 2, n))
    else:
        freq = np.linspace(nu0, nu1, n)
    w = np.ones(n)
    bad = int(round(case["flagged"] * n))
    w[np.random.RandomState(n).permutation(n)[:bad]] = 0.0
    phi = -phi_max + (2.0 * phi_max / (case["nphi"] - 1)) * np.arange(case["nphi"])
    return freq, w, phi


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)


def _sources(case, seed):
    """Per LOS: three components' phi0, p0, chi0 and slab width (FP64, [nlos][3])."""
    g = _generator(seed, 1)
    n = case["nlos"]
    u = torch.rand(6, n, 3, generator=g, device="cuda", dtype=torch.float64)
    _, _, phi_max, src_max = BANDS[case["band"]]
    phi0 = src_max * (2.0 * u[0] - 1.0)
    if case["kind"] == "map":
        # A map holds indices: which of two samples is the larger has to be decided by the source and not by the
        # last bit of a sum, so its one thin, bright source lies within a tenth of a step, and of a beam, of a sample.
        step = 2.0 * phi_max / (case["nphi"] - 1)
        nu0, nu1 = BANDS[case["band"]][:2]
        beam = 2.0 * math.sqrt(3.0) / ((C_LIGHT / nu0) ** 2 - (C_LIGHT / nu1) ** 2)
        k = torch.round((phi0 + phi_max) / step)
        phi0 = -phi_max + step * k + 0.2 * min(step, beam) * (u[5] - 0.5)
        p0 = 0.5 + 0.5 * u[1]
        p0[:, 1:] = 0.0
        chi0 = 0.8 + 1.2 * u[2]         # away from 0 and pi, where the angle wraps
        width = torch.zeros_like(p0)
        return phi0, p0, chi0, width
    count = 1 + torch.floor(3.0 * u[5][:, :1])
    p0 = torch.where(torch.arange(3, device="cuda")[None, :] < count, u[1], torch.zeros_like(u[1]))
    slab = u[3] < 0.5 if case["band"].startswith("lofar") else torch.zeros_like(u[3], dtype=torch.bool)
    width = torch.where(slab, 10.0 * u[4], torch.zeros_like(u[4]))
    return phi0, p0, math.pi * u[2], width


def _cube(case, seed):
    """Q, U: FP32 CUDA tensors in the case's layout."""
    freq, w, _ = _axes(case)
    n, nchan = case["nlos"], case["nchan"]
    l2 = torch.from_numpy((C_LIGHT / freq) ** 2).cuda()
    rfi = torch.from_numpy(np.where(w == 0.0, 50.0, 0.0).astype(np.float32)).cuda()
    phi0, p0, chi0, width = _sources(case, seed)
    g = _generator(seed, 2)
    los = case["layout"] == "los"
    Q = torch.empty((n, nchan) if los else (nchan, n), device="cuda")
    U = torch.empty_like(Q)
    rows = max(1, CHUNK_VALUES // nchan)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        noise = torch.randn(2, b - a, nchan, generator=g, device="cuda")
        q, u = noise[0] * (0.005 + rfi), noise[1] * (0.005 + rfi)
        for c in range(3):
            if not bool((p0[a:b, c] != 0).any()):
                continue
            turns = (phi0[a:b, c, None] * l2 + chi0[a:b, c, None]) / math.pi
            angle = ((turns - torch.floor(turns)) * (2.0 * math.pi)).float()
            amp = (p0[a:b, c, None] * torch.sinc(width[a:b, c, None] * l2 / math.pi)).float()
            q += amp * torch.cos(angle)
            u += amp * torch.sin(angle)
        if los:
            Q[a:b], U[a:b] = q, u
        else:
            Q[:, a:b], U[:, a:b] = q.T, u.T
    return Q, U


def _spectra(case, Q, U):
    """F in 64 bits for consecutive LOS ranges: yields (first, last, complex128 [rows][nphi])."""
    freq, w, phi = _axes(case)
    l2 = (C_LIGHT / freq) ** 2
    x = torch.from_numpy(l2 - np.sum(w * l2) / np.sum(w)).cuda()
    live = torch.from_numpy(np.flatnonzero(w)).cuda()
    angle = 2.0 * x[live, None] * torch.from_numpy(phi).cuda()[None, :]
    wk = torch.from_numpy(w / np.sum(w)).cuda()[live, None]
    E = torch.complex(wk * torch.cos(angle), -wk * torch.sin(angle))
    if case["layout"] == "chan":
        Q, U = Q.T, U.T
    rows = max(1, CHUNK_VALUES // max(case["nchan"], case["nphi"]))
    for a in range(0, case["nlos"], rows):
        b = min(case["nlos"], a + rows)
        P = torch.complex(Q[a:b].index_select(1, live).double(), U[a:b].index_select(1, live).double())
        yield a, b, P @ E


def _dirty(case, seed):
    """The dirty spectra RM-CLEAN starts from (complex64 as FP32 pairs)."""
    Q, U = _cube(case, seed)
    F = torch.empty(case["nlos"], case["nphi"], 2, device="cuda")
    for a, b, f in _spectra(case, Q, U):
        F[a:b] = torch.view_as_real(f)
    return F


CLEAN_GAIN, CLEAN_ITER, HIDDEN = 0.1, 400, 256


def _clean_threshold(case):
    return float(np.float32(5.0 * 0.005 / math.sqrt((1.0 - case["flagged"]) * case["nchan"])))


def _weights(case, seed):
    """Network parameters: fan-in scaled normal weights, small biases, a strong linear response."""
    _, w, _ = _axes(case)
    nin, nb = 2 * int(np.count_nonzero(w)), case["nphi"]
    g = _generator(seed, 3)
    W1 = torch.randn(HIDDEN, nin, generator=g, device="cuda") * math.sqrt(2.0 / nin)
    b1 = torch.randn(HIDDEN, generator=g, device="cuda") * 0.05
    W2 = torch.randn(nb, HIDDEN, generator=g, device="cuda") * (3.0 / math.sqrt(HIDDEN))
    b2 = torch.randn(nb, generator=g, device="cuda") * 0.05
    return W1, b1, W2, b2


def _labels(case, seed):
    phi0, p0, _, _ = _sources(case, seed)
    phi_max = BANDS[case["band"]][2]
    main = phi0.gather(1, p0.argmax(1, keepdim=True))[:, 0]
    k = torch.round((main + phi_max) / (2.0 * phi_max) * (case["nphi"] - 1))
    return k.clamp(0, case["nphi"] - 1).to(torch.int32)


# ----------------------------------------------------------------------------- the calls
def prepare(case, seed):
    freq, w, phi = _axes(case)
    n, kind = case["nlos"], case["kind"]
    s = dict(kind=kind, n=n, layout=case["layout"], plan=rms.Plan(freq, phi, case["precision"], weights=w))
    if kind == "clean":
        s["clean"] = rms.rms_clean_create(s["plan"].handle)
        s["F"] = _dirty(case, seed)
        s["threshold"] = _clean_threshold(case)
        s["out"] = [torch.empty_like(s["F"]) for _ in range(3)] + [torch.empty(n, dtype=torch.int32, device="cuda")]
        s["release"] = _Release(s["clean"])
        return s
    s["Q"], s["U"] = _cube(case, seed)
    f32 = lambda: torch.empty(n, device="cuda")                               # noqa: E731
    i32 = lambda: torch.empty(n, dtype=torch.int32, device="cuda")            # noqa: E731
    if kind == "synth":
        s["F"] = torch.empty(n, case["nphi"], 2, device="cuda")
        s["idx"], s["abs"], s["phi"] = i32(), f32(), f32()
    elif kind == "map":
        s["out"] = [i32()] + [f32() for _ in range(5)]
    else:
        s["net"] = learned.Net(s["plan"], hidden=HIDDEN, max_batch=max(128, min(n, 8192)))
        s["net"].set_params(torch.cat([t.reshape(-1) for t in _weights(case, seed)]).cpu().numpy())
        if kind == "gradient":
            s["label"], s["loss"] = _labels(case, seed), torch.empty(1, device="cuda")
        else:
            s["win"] = learned.Window(s["plan"], 64)
            s["bin"], s["conf"], s["centre"], s["idx"] = i32(), f32(), i32(), i32()
            s["abs"], s["phi"] = f32(), f32()
    return s


class _Release:
    """Destroys an RM-CLEAN object when its state goes."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        try:
            rms.rms_clean_destroy(self.handle)
        except Exception:
            pass


def run(s):
    kind, n = s["kind"], s["n"]
    if kind == "synth":
        # the whole peak map is asked for, as a user does; |F| at the peak is returned of it, since the index of
        # a near-tie between two samples is decided by the last bit of either
        s["plan"].synth(s["Q"], s["U"], n, s["layout"], s["F"], s["idx"], s["abs"], s["phi"])
        return [s["F"], s["abs"]]
    if kind == "map":
        rms.rms_synth_peaks(s["plan"].handle, s["Q"], s["U"], n, s["layout"], None, *s["out"])
        return s["out"]
    if kind == "clean":
        rms.rms_clean(s["clean"], s["F"], n, CLEAN_GAIN, CLEAN_ITER, s["threshold"], *s["out"])
        return s["out"]
    if kind == "gradient":
        rms.rms_net_grad(s["net"].handle, s["Q"], s["U"], n, s["layout"], s["label"], s["loss"])
        return [s["loss"], s["net"].grads()]
    rms.rms_propose(s["net"].handle, s["Q"], s["U"], n, s["layout"], s["win"].conf_halfwidth, None, s["bin"],
                    s["conf"])
    rms.rms_window_centres(s["win"].handle, s["bin"], n, s["centre"])
    rms.rms_synth_window(s["win"].handle, s["Q"], s["U"], n, s["layout"], s["centre"], None, s["idx"], s["abs"],
                         s["phi"])
    return [s["bin"], s["conf"], s["abs"]]


def work(case):
    """One multiply-add of complex numbers (8 flops) per (LOS, active channel, phi); inputs and outputs once."""
    n, nphi = case["nlos"], case["nphi"]
    _, w, _ = _axes(case)
    nact = int(np.count_nonzero(w))
    data, kind = 8.0 * n * nact, case["kind"]
    if case["precision"] == "fp32_czt":         # one FFT's worth of work on twice the grid, and the chirps
        m = 2.0 ** math.ceil(math.log2(nphi + case["nchan"]))
        return dict(bytes=data + 8.0 * n * nphi + 12.0 * n, flops=n * (10.0 * m * math.log2(m) + 6.0 * m))
    if kind == "synth":
        return dict(bytes=data + 8.0 * n * nphi + 12.0 * n, flops=8.0 * n * nact * nphi)
    if kind == "map":
        return dict(bytes=data + 24.0 * n, flops=8.0 * n * nact * nphi)
    if kind == "clean":                         # about a hundred steps a LOS, each an update and a search
        return dict(bytes=n * (32.0 * nphi + 4.0), flops=100.0 * n * nphi * 11.0)
    params = HIDDEN * (2.0 * nact + 1.0) + nphi * (HIDDEN + 1.0)
    if kind == "gradient":
        return dict(bytes=data + 4.0 * n + 8.0 * params, flops=6.0 * n * params)
    return dict(bytes=data + 24.0 * n + 4.0 * params, flops=2.0 * n * params + 8.0 * n * nact * 64)


# ----------------------------------------------------------------------------- 64-bit results
def _exact_clean(case, F32):
    freq, w, phi = _axes(case)
    n, nphi = case["nlos"], case["nphi"]
    l2 = (C_LIGHT / freq) ** 2
    l2, wl = l2[w > 0], w[w > 0]
    l0 = np.sum(wl * l2) / np.sum(wl)
    step = (phi[-1] - phi[0]) / (nphi - 1)

    def response(offset):
        return np.exp(-2j * np.outer(offset, l2 - l0)) @ wl / np.sum(wl)

    lo, hi = 0.0, 2.0 * math.sqrt(3.0) / (l2.max() - l2.min()) / 4.0
    while abs(response(np.array([hi]))[0]) > 0.5:
        lo, hi = hi, hi * 1.1
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if abs(response(np.array([mid]))[0]) > 0.5 else (lo, mid)
    fwhm = 2.0 * lo
    R = torch.from_numpy(response((np.arange(2 * nphi - 1) - (nphi - 1)) * step)).cuda()
    gain, threshold = float(np.float32(CLEAN_GAIN)), _clean_threshold(case)
    res = torch.view_as_complex(F32.double())
    comp, count = torch.zeros_like(res), torch.zeros(n, dtype=torch.int32, device="cuda")
    live = torch.arange(n, device="cuda")
    k = torch.arange(nphi, device="cuda")
    r = res.clone()
    for _ in range(CLEAN_ITER):
        m2 = r.real * r.real + r.imag * r.imag
        best, j = m2.max(1)
        go = best >= threshold * threshold
        if not bool(go.all()):
            res[live[~go]] = r[~go]
            r, live, j = r[go], live[go], j[go]
        if not len(live):
            break
        c = gain * r.gather(1, j[:, None])
        comp[live, j] += c[:, 0]
        r = r - c * R[k[None, :] - j[:, None] + nphi - 1]
        count[live] += 1
    res[live] = r
    W = min(nphi - 1, math.ceil(3.0 * fwhm / step))
    d = torch.arange(-W, W + 1, device="cuda", dtype=torch.float64)
    beam = torch.exp(-4.0 * math.log(2.0) * (d * step) ** 2 / fwhm ** 2)
    pad = torch.view_as_real(comp).permute(0, 2, 1).reshape(2 * n, 1, nphi)
    smooth = torch.nn.functional.conv1d(pad, beam[None, None, :], padding=W).reshape(n, 2, nphi).permute(0, 2, 1)
    full = torch.view_as_real(res)
    return [full + smooth, full, torch.view_as_real(comp), count]


def _exact_gradient(case, seed, Q, U):
    _, w, _ = _axes(case)
    live = torch.from_numpy(np.flatnonzero(w)).cuda()
    x = torch.stack([Q[:, live], U[:, live]], dim=2).double()
    rms_p = torch.sqrt((x * x).sum((1, 2), keepdim=True) / len(live))
    x = (x / rms_p).reshape(case["nlos"], -1)
    p = [t.double().requires_grad_() for t in _weights(case, seed)]
    z = torch.relu(x @ p[0].T + p[1]) @ p[2].T + p[3]
    loss = torch.nn.functional.cross_entropy(z, _labels(case, seed).long())
    loss.backward()
    return [loss.detach().reshape(1), torch.cat([t.grad.reshape(-1) for t in p])]


def exact(case, seed):
    kind = case["kind"]
    if kind == "clean":
        return _exact_clean(case, _dirty(case, seed))
    if kind == "proposal":
        return None         # the windows hang on the network's choice of a bin
    Q, U = _cube(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed, Q, U)
    n, nphi = case["nlos"], case["nphi"]
    best = torch.empty(n, dtype=torch.float64, device="cuda")
    if kind == "synth":
        F = torch.empty(n, nphi, 2, dtype=torch.float64, device="cuda")
        for a, b, f in _spectra(case, Q, U):
            F[a:b] = torch.view_as_real(f)
            best[a:b] = f.abs().amax(1)
        return [F, best]
    freq, w, phi = _axes(case)
    l2 = (C_LIGHT / freq) ** 2
    l0 = float(np.sum(w * l2) / np.sum(w))
    grid = torch.from_numpy(phi).cuda()
    idx = torch.empty(n, dtype=torch.int32, device="cuda")
    peak = torch.empty(n, dtype=torch.complex128, device="cuda")
    for a, b, f in _spectra(case, Q, U):
        best[a:b], k = f.abs().max(1)
        idx[a:b], peak[a:b] = k.to(torch.int32), f.gather(1, k[:, None])[:, 0]
    at = grid[idx.long()]
    chi = 0.5 * torch.atan2(peak.imag, peak.real) - at * l0
    return [idx, best, at, peak.real.contiguous(), peak.imag.contiguous(), chi - math.pi * torch.floor(chi / math.pi)]
