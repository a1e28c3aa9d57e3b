"""Performance cases: the calls a user of the streaming time->energy library has it make.

A case is one pass of a program that owns a plan: reset, the segment's pushes, finalize (or the
differentiable spectrum and its backward), through the Python binding.  Inputs are synthetic exit
waves (an elastic part of Gaussian envelope, a few phonon lines, noise) drawn on the GPU from the
seed.  Pushed buffers hold either the whole sequence or a ring of frames that is cycled over, as a
multislice run that reuses its output buffers does.

`exact` restates the result in FP64: mean removal, window, transform to the energy grid (an FFT, a
chirp-z transform or a matrix product in complex128), |Psi|^2, Bose factor, detector sums, gradient.
"""
import math
import random

import numpy as np
import torch

from paper_2607_02236_gb300.autograd import spectrum
from paper_2607_02236_gb300.tacaw import DetectorConfig, StreamConfig, TacawPlan

H = 4.135667696          # Planck constant, meV ps
DT = 5.0                 # frame interval, fs
KB = 0.08617333262       # Boltzmann constant, meV / K

# One stream.  grid: "roi" nw energies from emin, end point excluded; "fft" the first nw FFT bins;
# "list" nw unevenly spaced energies.  gx, gy: the multislice grid the centred kx x ky ROI is cropped
# from.  ring: frames held (0: all of them).  segs/stride/skip: Welch averaging.  batches: segments
# (probe batches) one pass runs through the plan.
BASE = dict(kind="stream", P=1, kx=64, ky=64, gx=64, gy=64, T=256, Tc=256, nw=128, grid="roi", emin=0.0, emax=120.0,
            window="hann", wparam=0.0, mean=True, bose=0.0, prec="split_bf16", segs=0, stride=0, skip=0, dets=1,
            psi=False, host=False, pipelined=False, batches=1, ring=0, wait=False)


def _stream(name=None, **kw):
    c = dict(BASE, **kw)
    if name:
        c["name"] = name
    for k in ("x", "y"):
        if "g" + k not in kw:
            c["g" + k] = c["k" + k]
    return c


def listed():
    return [
        # the smallest call: one push of a short segment, first FFT bins, FP32, waits for its spectra
        _stream("tiny-fp32", P=4, T=256, Tc=256, nw=128, grid="fft", prec="fp32", wait=True),
        # a quick look at a scan position or two: ragged ROI, odd lengths, small pushes
        _stream("small-ragged", P=3, kx=61, ky=45, gx=96, gy=80, T=300, Tc=25, nw=97, dets=2),
        # an 8 x 8 scan in batches of 16 probes, 256 x 256 ROI, 0.3 meV energies, pushes of 32 frames
        _stream("scan-bf16", P=16, kx=256, ky=256, T=2048, Tc=32, nw=400),
        # the same in the FP32 arithmetic, for callers that want no split operands
        _stream("scan-fp32", P=2, kx=256, ky=256, T=2048, Tc=32, nw=400, prec="fp32"),
        # split FP16 with the complex spectra Psi kept for phase-resolved work
        _stream("scan-fp16-psi", P=4, kx=256, ky=256, T=2048, Tc=32, nw=400, prec="split_fp16", window="gauss",
                psi=True),
        # a chunk on its own FFT grid up to Nyquist, odd ROI, mean kept, Blackman-Harris window
        _stream("fft-grid", P=4, kx=191, ky=191, T=1000, Tc=50, nw=500, grid="fft", mean=False,
                window="blackmanharris"),
        # supercell partitions of uneven size pushed side by side, staging shorter than the segments
        dict(name="partitions", kind="group", shapes="5,128,3072;17,192,1024;8,256,2048;23,128,4096;4,384,512;11,192,1536",
             Tc=16, nw=300, k_stage=1024),
        # gradient of a spectral loss with respect to the exit waves, forward and backward
        dict(name="gradient", kind="grad", P=8, kx=128, ky=128, T=512, nw=200, emax=120.0, window="hann", radius=20.0,
             prec="fp32", segs=0, stride=0),
        # thick sample: long segments of full 1024 x 1024 frames cropped to the ROI, 1000 energies
        _stream("thick", P=4, kx=256, ky=256, gx=1024, gy=1024, T=8192, Tc=64, nw=1000, emax=150.0, ring=256),
        # Welch average of overlapping chunks, loss and gain sides, Bose factor, three detectors
        _stream("welch", P=4, kx=128, ky=128, T=512, Tc=32, nw=160, emin=-60.0, emax=60.0, segs=7, stride=256, skip=100,
                bose=300.0, dets=3),
        # frames left in pinned host memory by a CPU producer, read over the host link
        _stream("host-frames", P=4, kx=192, ky=192, gx=256, gy=256, T=1024, Tc=32, nw=300, host=True, ring=128),
        # probe batches one after another through a plan with pipelined segments
        _stream("pipelined", P=2, kx=256, ky=256, T=4096, Tc=64, nw=1000, emax=150.0, pipelined=True, batches=3,
                ring=512),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choices(["stream", "group", "grad"], [8, 2, 2])[0]
    if kind == "grad":
        c = dict(kind="grad", P=rng.randint(1, 12), kx=rng.randint(24, 160), ky=rng.randint(24, 160), T=_log(rng, 64, 1500),
                 nw=_log(rng, 30, 400), emax=rng.choice([60.0, 120.0, 200.0]), window=rng.choice(["hann", "rect", "tukey"]),
                 radius=float(rng.randint(4, 24)), prec=rng.choice(["fp32", "split_bf16"]), segs=rng.choice([0, 0, 3]),
                 stride=0)
        if c["segs"]:
            c["stride"] = c["T"] // 2
        return c
    if kind == "group":
        parts = ["%d,%d,%d" % (rng.randint(2, 20), rng.choice([64, 96, 128, 192, 250]), rng.choice([512, 1024, 1536, 2048, 700]))
                 for _ in range(rng.randint(2, 8))]
        return dict(kind="group", shapes=";".join(parts), Tc=rng.choice([8, 16, 32, 64]), nw=_log(rng, 100, 500),
                    k_stage=rng.choice([0, 256, 512, 1024]))
    while True:
        kx = _log(rng, 24, 384)
        c = _stream(P=_log(rng, 1, 32), kx=kx, ky=rng.choice([kx, max(16, kx - rng.randint(0, 40))]), T=_log(rng, 100, 8192),
                    Tc=rng.choice([8, 16, 20, 32, 50, 64, 100, 128]), nw=_log(rng, 40, 1200),
                    grid=rng.choices(["roi", "fft", "list"], [6, 1, 1])[0], emin=rng.choice([0.0, 0.0, -80.0, 20.0]),
                    emax=rng.choice([80.0, 120.0, 150.0, 250.0]),
                    window=rng.choice(["hann", "rect", "gauss", "tukey", "blackmanharris", "kaiser"]),
                    mean=rng.random() < 0.8, bose=rng.choice([0.0, 0.0, 300.0]),
                    prec=rng.choices(["split_bf16", "fp32", "split_fp16"], [6, 3, 2])[0], dets=rng.randint(1, 3),
                    psi=rng.random() < 0.2)
        c["wparam"] = {"tukey": 0.25, "kaiser": 3 * math.pi}.get(c["window"], 0.0)
        if c["grid"] == "fft":
            c["nw"] = min(c["nw"], c["T"])
            c["emin"] = 0.0
        if rng.random() < 0.3:      # cropped out of a larger grid
            c["gx"], c["gy"] = 2 * c["kx"], c["ky"] + 2 * rng.randint(0, 20)
        what = rng.choice(["", "", "", "welch", "host", "pipelined"])
        if what == "welch":
            c["T"] = min(c["T"], 1024)
            c["nw"] = min(c["nw"], c["T"])
            c.update(segs=rng.randint(2, 6), stride=c["T"] // rng.choice([1, 2]), skip=rng.choice([0, 37]), psi=False)
        if what == "host":
            c.update(host=True, ring=4 * c["Tc"])
        if what == "pipelined":
            c.update(prec="split_bf16", T=max(128, c["T"] // 32 * 32), pipelined=True, batches=rng.randint(2, 4))
            c["nw"] = min(c["nw"], c["T"])
        rows, frames = c["P"] * c["kx"] * c["ky"], _frames(c)
        cost = rows * frames * c["nw"] * c["batches"] * max(1, c["segs"] and 2) * (8 if c["prec"] == "fp32" else 1)
        held = c["P"] * c["gx"] * c["gy"] * (c["ring"] or frames) * 8
        if 4e6 < cost < 1.2e12 and held < 1.2e10 and rows * frames < (6e8 if c["host"] else 2.5e9) \
                and rows * c["nw"] < 3e8:
            return c


def _frames(c):
    return c.get("skip", 0) + (max(1, c.get("segs", 0)) - 1) * (c.get("stride", 0) or c["T"]) + c["T"]


def _energies(c):
    nw, lo, hi = c["nw"], c.get("emin", 0.0), c["emax"]
    j = np.arange(nw, dtype=np.float64)
    if c.get("grid") == "fft":
        return j * (H / (c["T"] * DT * 1e-3))
    if c.get("grid") == "list":
        return lo + (hi - lo) * (j / nw) ** 1.5
    return lo + j * ((hi - lo) / nw)


def _waves(P, kx, ky, gx, gy, n, seed):
    """n frames [n, P, gy, gx] complex64 on the GPU: unit-norm elastic part, 8 lines, noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    y = torch.arange(gy, device="cuda", dtype=torch.float32) - gy // 2
    x = torch.arange(gx, device="cuda", dtype=torch.float32) - gx // 2
    env = torch.exp(-(y[:, None] ** 2 + x[None, :] ** 2) / (2 * 8.0 ** 2))
    env = (env / env.norm()).expand(P, gy, gx).reshape(-1)
    rows, modes = env.numel(), 8

    def phase(*shape):
        return torch.rand(*shape, device="cuda", generator=g) * (2 * math.pi)

    psi0 = torch.polar(env, phase(rows))
    amp = torch.polar(1e-2 * env * (0.5 + 0.5 * torch.rand(modes, rows, device="cuda", generator=g)), phase(modes, rows))
    E = 5.0 + 95.0 * torch.rand(modes, device="cuda", generator=g, dtype=torch.float64)
    out = torch.empty(n, rows, dtype=torch.complex64, device="cuda")
    t = torch.arange(n, device="cuda", dtype=torch.float64)
    line = torch.polar(torch.ones(n, modes, dtype=torch.float64, device="cuda"),
                       2 * math.pi * torch.frac(t[:, None] * (E * (DT * 1e-3 / H)))).to(torch.complex64)
    noise = float(env.max()) * 1e-5
    step = max(1, (1 << 27) // rows)
    for a in range(0, n, step):
        b = min(n, a + step)
        f = out[a:b]
        torch.view_as_real(f).normal_(0.0, noise, generator=g)
        f += psi0
        f += line[a:b] @ amp
    return out.view(n, P, gy, gx)


def _detectors(c):
    d = [DetectorConfig(kind="circular", r_out=c.get("radius", 20.0)), DetectorConfig(kind="annular", r_in=12.0, r_out=28.0),
         DetectorConfig(kind="circular", cx=9.0, cy=-6.0, r_out=10.5)]
    return d[:c.get("dets", 1)]


def _config(c):
    gx, gy = c.get("gx", c["kx"]), c.get("gy", c["ky"])
    fft = c.get("grid") == "fft"
    return StreamConfig(n_probes=c["P"], kx=c["kx"], ky=c["ky"], T=c["T"], dt_fs=DT, pitch_row=gx,
                        pitch_frame=gx * gy * c["P"], pitch_probe=gx * gy, roi_x0=(gx - c["kx"]) // 2,
                        roi_y0=(gy - c["ky"]) // 2, E_meV=None if fft else list(_energies(c)), fft_bins=c["nw"] if fft else 0,
                        window=c["window"], window_param=c.get("wparam", 0.0), subtract_mean=c.get("mean", True),
                        bose_T_K=c.get("bose", 0.0), detectors=_detectors(c), welch_segments=c.get("segs", 0),
                        welch_stride=c.get("stride", 0), skip_init=c.get("skip", 0))


def _parts(case):
    return [_stream(P=p, kx=k, ky=k, T=t, nw=case["nw"], window=("hann", "gauss")[i % 2], Tc=case["Tc"])
            for i, (p, k, t) in enumerate(tuple(int(v) for v in s.split(",")) for s in case["shapes"].split(";"))]


def _ring(c, seed):
    n = _frames(c)
    if c.get("ring"):
        n = min(n, c["ring"])
    return _waves(c["P"], c["kx"], c["ky"], c.get("gx", c["kx"]), c.get("gy", c["ky"]), n, seed)


def _pushes(c, held):
    """(first held frame, frames) of each push: at most Tc frames, inside the held ring."""
    n, t = _frames(c), 0
    while t < n:
        k = min(c["Tc"], n - t, held - t % held)
        yield t % held, k
        t += k


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "grad":
        s.frames = _ring(case, seed).requires_grad_(True)
        s.plan = TacawPlan([_config(case)], precision=case["prec"])
        s.weights = _weights(case, seed)
        return s
    if case["kind"] == "group":
        parts = _parts(case)
        s.rings = [_waves(p["P"], p["kx"], p["ky"], p["kx"], p["ky"], 4 * p["Tc"], seed + 1000 * i)
                   for i, p in enumerate(parts)]
        s.plan = TacawPlan([_config(p) for p in parts], precision="split_bf16", k_stage=case["k_stage"])
        s.parts = parts
        # the k-th group push: every partition that still has frames
        s.calls = []
        for t in range(0, max(p["T"] for p in parts), case["Tc"]):
            ids = [i for i, p in enumerate(parts) if t < p["T"]]
            s.calls.append((ids, [_at(s.rings[i], t % (4 * case["Tc"])) for i in ids],
                            [min(case["Tc"], parts[i]["T"] - t) for i in ids]))
    else:
        waves = _ring(case, seed)
        if case["host"]:
            s.ring = torch.empty(waves.shape, dtype=waves.dtype, pin_memory=True)
            s.ring.copy_(waves)
        else:
            s.ring = waves
        del waves
        s.plan = TacawPlan([_config(case)], precision=case["prec"])
        if case["pipelined"]:
            s.plan.set_pipelined_segments(True)
        s.calls = [(_at(s.ring, t), k) for t, k in _pushes(case, s.ring.shape[0])]
    i = s.plan.info()
    n = case.get("batches", 1)
    s.I = [torch.empty(i["I_elems"], device="cuda") for _ in range(n)]
    s.S = [torch.empty(i["S_elems"], device="cuda") for _ in range(n)]
    s.psi = torch.empty(i["I_elems"], dtype=torch.complex64, device="cuda") if case.get("psi") else None
    return s


def _at(ring, t):
    return ring.data_ptr() + t * ring.stride(0) * 8


def _weights(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 7)
    return torch.randn(case["P"], 1, case["nw"], device="cuda", generator=g)


def run(s):
    c, cs = s.case, torch.cuda.current_stream()
    if c["kind"] == "grad":
        s.frames.grad = None
        S = spectrum(s.frames, s.plan)
        (S * s.weights).sum().backward()
        return {"S": S.detach(), "grad": s.frames.grad}
    for b in range(len(s.I)):
        s.plan.reset(cs)
        if c["kind"] == "group":
            for ids, at, n in s.calls:
                s.plan.push_group(ids, at, n, cs)
        else:
            for at, n in s.calls:
                s.plan.push(0, at, n, cs)
        if c.get("wait"):
            s.plan.finalize(s.I[b], s.S[b], s.psi, cs)
        else:
            s.plan.finalize_async(s.I[b], s.S[b], s.psi, cs)
    if c.get("pipelined"):
        s.plan.drain(cs)
    out = {"I": s.I, "S": s.S}
    if s.psi is not None:
        out["Psi"] = s.psi
    return out


def work(case):
    if case["kind"] == "group":
        ws = [work(p) for p in _parts(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    rows, n, nw = case["P"] * case["kx"] * case["ky"], _frames(case), case["nw"]
    if case["kind"] == "grad":
        # the aperture's frames read, the gradient written; two transforms of the aperture's rows
        ap = case["P"] * min(case["kx"] * case["ky"], math.pi * case["radius"] ** 2)
        return {"bytes": 8.0 * n * (ap + rows), "flops": 2 * ap * _transform(case["T"], nw) * max(1, case["segs"])}
    b = case["batches"]
    out = rows * nw * (12.0 if case["psi"] else 4.0)
    return {"bytes": b * (8.0 * rows * (n - case["skip"]) + out), "flops": b * rows * _transform(case["T"], nw) * max(1, case["segs"])}


def _transform(T, nw):
    """Flops of one fast transform of T frames to nw energies."""
    return 5.0 * (T + nw) * math.log2(T + nw)


# ---- FP64 restatement -------------------------------------------------------------------

def _window(c):
    T, t = c["T"], np.arange(c["T"], dtype=np.float64)
    w, a = c["window"], c.get("wparam", 0.0)
    if w == "rect" or T == 1:
        v = np.ones(T)
    elif w == "hann":
        v = 0.5 - 0.5 * np.cos(2 * np.pi * t / T)
    elif w == "gauss":
        v = np.exp(-0.5 * ((t - T / 2) / (a or T / 6)) ** 2)
    elif w == "tukey":
        e, v = a * T / 2, np.ones(T)
        v[t < e] = 0.5 * (1 - np.cos(np.pi * t[t < e] / e))
        v[t > T - e] = 0.5 * (1 - np.cos(np.pi * (T - t[t > T - e]) / e))
    elif w == "blackmanharris":
        x = 2 * np.pi * t / T
        v = 0.35875 - 0.48829 * np.cos(x) + 0.14128 * np.cos(2 * x) - 0.01168 * np.cos(3 * x)
    else:
        v = np.i0(a * np.sqrt(np.maximum(0.0, 1 - (2 * t / T - 1) ** 2))) / np.i0(a)
    return torch.from_numpy(v).cuda()


def _unit(cycles):
    return torch.polar(torch.ones_like(cycles), 2 * math.pi * torch.frac(cycles))


def _spectra(y, c):
    """Psi [rows, nw] of windowed series y [rows, T] in complex128."""
    T, nw = c["T"], c["nw"]
    if c.get("grid") == "fft":
        return torch.fft.fft(y)[:, :nw]
    t = torch.arange(T, dtype=torch.float64, device="cuda")
    cyc = torch.from_numpy(_energies(c) * (DT * 1e-3 / H)).cuda()
    if c.get("grid") == "list":
        return y @ _unit(-t[:, None] * cyc)
    # chirp-z: t j = (t^2 + j^2 - (j - t)^2) / 2
    d = (c["emax"] - c.get("emin", 0.0)) / nw * (DT * 1e-3 / H)
    j = torch.arange(nw, dtype=torch.float64, device="cuda")
    L = 1 << (T + nw - 1).bit_length()
    v = torch.zeros(L, dtype=torch.complex128, device="cuda")
    v[:nw] = _unit(j * j * (d / 2))
    if T > 1:
        k = torch.arange(1, T, dtype=torch.float64, device="cuda")
        v[L - T + 1:] = _unit(k * k * (d / 2)).flip(0)
    z = torch.fft.fft(y * _unit(-t * float(cyc[0])) * _unit(-t * t * (d / 2)), n=L)
    return torch.fft.ifft(z * torch.fft.fft(v))[:, :nw] * _unit(-j * j * (d / 2))


def _bose(c):
    E = _energies(c)
    if c.get("bose", 0.0) <= 0:
        return torch.ones(len(E), dtype=torch.float64, device="cuda")
    x = E / (KB * c["bose"])
    return torch.from_numpy(np.where(E == 0, 1.0, x / np.where(E == 0, 1.0, -np.expm1(-x)))).cuda()


def _masks(c):
    y = torch.arange(c["ky"], device="cuda", dtype=torch.float64) - c["ky"] // 2
    x = torch.arange(c["kx"], device="cuda", dtype=torch.float64) - c["kx"] // 2
    out = []
    for d in _detectors(c):
        r2 = (y[:, None] - d.cy) ** 2 + (x[None, :] - d.cx) ** 2
        m = r2 <= d.r_out ** 2
        if d.kind == "annular":
            m &= r2 > d.r_in ** 2
        out.append(m.reshape(-1).double())
    return torch.stack(out)


def _exact_stream(c, ring):
    """I [P, nw, npix] (float64), Psi or None, S [P, D, nw] of one stream."""
    P, kx, ky, T, nw = c["P"], c["kx"], c["ky"], c["T"], c["nw"]
    gx, gy = c.get("gx", kx), c.get("gy", ky)
    x0, y0, npix, n = (gx - kx) // 2, (gy - ky) // 2, kx * ky, _frames(c)
    segs, stride, skip = max(1, c.get("segs", 0)), c.get("stride", 0) or T, c.get("skip", 0)
    idx = torch.arange(n, device=ring.device) % ring.shape[0]
    w, B, D = _window(c), _bose(c), _masks(c)
    I = torch.zeros(P, nw, npix, dtype=torch.float64, device="cuda")
    Psi = torch.zeros(P, nw, npix, dtype=torch.complex128, device="cuda") if c.get("psi") else None
    step = max(1, min(npix, (1 << 27) // (T + nw)) // kx)
    for p in range(P):
        for r in range(0, ky, step):
            q = min(ky, r + step)
            f = ring[:, p, y0 + r:y0 + q, x0:x0 + kx].reshape(ring.shape[0], -1).cuda().to(torch.complex128)
            for i in range(segs):
                a = skip + i * stride
                y = f[idx[a:a + T].to(f.device)].T
                if c.get("mean", True):
                    y = y - y.mean(1, keepdim=True)
                z = _spectra((y * w).contiguous(), c)
                I[p, :, r * kx:q * kx] += (z.real ** 2 + z.imag ** 2).T * B[:, None] / segs
                if Psi is not None:
                    Psi[p, :, r * kx:q * kx] = z.T
    return I, Psi, torch.einsum("pek,dk->pde", I, D)


def _exact_grad(c, seed):
    """S and the gradient of sum(weights * S): g_t = 2 (w_t A_t - mean of w A), A = conj-transform of G."""
    f = _ring(c, seed)
    P, T, nw, npix = c["P"], c["T"], c["nw"], c["kx"] * c["ky"]
    segs, stride, n = max(1, c["segs"]), c["stride"] or T, _frames(c)
    D, w = _masks(c)[0], _window(c)
    pix = torch.nonzero(D).reshape(-1)
    t = torch.arange(T, dtype=torch.float64, device="cuda")
    W = _unit(-t[:, None] * torch.from_numpy(_energies(c) * (DT * 1e-3 / H)).cuda()) * w[:, None]     # [T, nw]
    c2 = _weights(c, seed).double().reshape(P, 1, nw)
    S = torch.zeros(P, 1, nw, dtype=torch.float64, device="cuda")
    grad = torch.zeros(n, P, npix, dtype=torch.complex128, device="cuda")
    for i in range(segs):
        y = f[i * stride:i * stride + T].reshape(T, P, npix)[:, :, pix].to(torch.complex128)
        y = y - y.mean(0)
        z = torch.einsum("tpk,te->pke", y, W)
        S += (z.real ** 2 + z.imag ** 2).sum(1)[:, None] / segs
        A = torch.einsum("pke,te->tpk", c2 * z, W.conj())
        grad[i * stride:i * stride + T, :, pix] += (2.0 / segs) * (A - A.mean(0))
    return {"S": S, "grad": torch.view_as_real(grad.reshape(f.shape)).reshape(*f.shape, 2)}


def exact(case, seed):
    if case["kind"] == "grad":
        out = _exact_grad(case, seed)
        out["grad"] = torch.view_as_complex(out["grad"])
        return out
    if case["kind"] == "group":
        got = [_exact_stream(p, _waves(p["P"], p["kx"], p["ky"], p["kx"], p["ky"], 4 * p["Tc"], seed + 1000 * i))
               for i, p in enumerate(_parts(case))]
    else:
        got = [_exact_stream(case, _ring(case, seed))]
    I = torch.cat([g[0].reshape(-1) for g in got])
    S = torch.cat([g[2].reshape(-1) for g in got])
    n = case.get("batches", 1)
    out = {"I": [I] * n, "S": [S] * n}
    if case.get("psi"):
        out["Psi"] = got[0][1].reshape(-1)
    return out


if __name__ == "__main__":
    r = random.Random(0)
    for case in listed() + [draw(r) for _ in range(6)]:
        print(case, work(case))
