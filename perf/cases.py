"""Timed cases of the FX correlator: what a program that uses this library has
it do, through its public entry points (`Correlator`, `autograd`, and the
batch calls of the C ABI).

A case is a dict of plain values. `kind` says which calls one pass makes:

  step    one block on the device: fused F-stage, then the X-stage
  layers  the three-call path (channelise, correct, correlate); every
          intermediate is an output
  beam    fused F-stage, then coherent beams
  stream  one block of a continuous stream (history, coarse shifts, lost-data
          flags), correlated
  train   correct + correlate forward and its adjoint, delays moving over the
          block (calibration by gradient descent)
  batch   many uneven correlation jobs in one launch
  host    one block from page-locked host memory to host visibilities

`listed()` holds the workloads of the configurations (LOFAR 16-bit and 8-bit
modes, the tiny block, the batching and the differentiation workload, the
beamformer), with the number of subbands that one GPU of several would carry,
and ragged ones; `draw` spreads over station counts, channel counts, spectra,
sample formats and precisions.
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1801_04834_gb300 as fx
from paper_1801_04834_gb300 import _abi, autograd

FS = 195312.5                       # complex sample rate of one subband (Hz)
FORMATS = {"ci16": _abi.FX_CI16, "ci8": _abi.FX_CI8, "ci4": _abi.FX_CI4}
SIGMA = {"ci16": 100.0, "ci8": 20.0, "ci4": 2.5}      # station noise, in counts
LIMIT = {"ci16": 32767, "ci8": 127, "ci4": 7}
PRECISIONS = {"f32": _abi.FX_F32, "f16": _abi.FX_F16, "bf16": _abi.FX_BF16, "f16_split": _abi.FX_F16_SPLIT,
              "tf32_split": _abi.FX_TF32_SPLIT}
RAW_BYTES = {"ci16": 4, "ci8": 2, "ci4": 1}           # per complex sample
DELAY_S = 5e-6                      # station delays are within +-5 us


def listed():
    return [
        # the tiny configuration: 8 stations, one subband; a user's first call and
        # every unit-sized job; launches and host time
        _c("tiny_f32", "step", stations=8, subbands=1, channels=64, spectra=768, precision="f32"),
        # LOFAR 16-bit mode at FP32 accuracy on the tensor cores, half of the 244 subbands
        _c("lofar16_tf32", "step", stations=64, subbands=122, channels=64, spectra=3072, precision="tf32_split"),
        # the same block through the default precision (FX_F32)
        _c("lofar16_f32", "step", stations=64, subbands=20, channels=64, spectra=3072, precision="f32"),
        # LOFAR 8-bit mode: 256 channels, FP16 operands, an eighth of the 488 subbands
        _c("lofar8_f16", "step", stations=64, subbands=61, channels=256, spectra=768, precision="f16", format="ci8"),
        # 8-bit mode with the accurate FP16 pair, a ragged array and integration
        _c("ragged8_split", "step", stations=50, subbands=24, channels=256, spectra=700, precision="f16_split",
           format="ci8"),
        # 78 fields (the largest array kept up with), odd integration length
        _c("fields78_tf32", "step", stations=78, subbands=16, channels=64, spectra=1001, precision="tf32_split"),
        # the beamformer requirement: 48 fields, 127 beams, Stokes I over 16 spectra
        _c("beams127", "beam", stations=48, subbands=40, channels=256, spectra=768, precision="f16", beams=127,
           output=1, tint=16),
        # a real-time stream: whole-sample delays, lost packets, FP32 accuracy
        _c("stream62", "stream", stations=62, subbands=12, channels=64, spectra=3072, precision="tf32_split",
           max_shift=64),
        # three separate calls, 4-bit samples, few channels, BF16 operands
        _c("layers_c16", "layers", stations=37, subbands=4, channels=16, spectra=2050, precision="bf16",
           format="ci4"),
        # the differentiation workload: 76 stations, 32 subbands, 768 spectra
        _c("train76", "train", stations=76, subbands=32, channels=64, spectra=768, precision="tf32_split"),
        # the batching workload: 48 uneven jobs
        _c("batch48", "batch", jobs=48, shape_seed=31, spectra_lo=256, spectra_hi=3072, precision="f16"),
        # host memory in and out, copies overlapped with the work
        _c("host8", "host", stations=64, subbands=8, channels=64, spectra=3072, precision="tf32_split", chunk=4),
    ]


def _c(name, kind, **kw):
    c = {"name": name, "kind": kind}
    if kind not in ("batch", "train"):
        c.update(taps=16, format="ci16")
    c.update(kw)
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["layers", "beam", "stream", "train", "batch", "host"])
    if kind == "batch":
        lo = _log(rng, 100, 800)
        return {"kind": kind, "jobs": rng.randint(3, 48), "shape_seed": rng.randrange(1 << 20), "spectra_lo": lo,
                "spectra_hi": rng.randint(lo, 3072), "precision": rng.choice(["f16", "bf16", "f16_split"])}
    c = {"kind": kind, "stations": _log(rng, 6, 96), "channels": rng.choice([16, 64, 64, 256]),
         "spectra": _log(rng, 60, 3072)}
    if kind == "train":
        c.update(precision=rng.choice(["f32", "tf32_split"]))
        most = 1 << 28
    else:
        c.update(taps=rng.choice([4, 8, 16, 16, 16]), format=rng.choice(["ci16", "ci16", "ci8", "ci4"]),
                 precision=rng.choice(["f32", "tf32_split", "f16", "bf16", "f16_split"]))
        most = {"step": 1 << 29, "layers": 1 << 26, "beam": 1 << 28, "stream": 1 << 28, "host": 1 << 27}[kind]
    if kind == "beam":
        c["stations"] = min(c["stations"], 64)
        c["precision"] = rng.choice(["f16", "bf16"])
        c["output"] = rng.choice([0, 1, 2])
        c["beams"] = _log(rng, 1, 222) if c["output"] else _log(rng, 1, 64)
        c["tint"] = rng.choice([1, 4, 16]) if c["output"] else 1
        c["spectra"] = max(c["tint"], c["spectra"] // c["tint"] * c["tint"])
        most //= max(1, c["beams"] // 32) if c["output"] == 0 else 1
    if kind == "stream":
        c["max_shift"] = rng.choice([0, 16, 100])
    per = c["stations"] * 2 * c["channels"] * c["spectra"]             # samples of one subband
    c["subbands"] = max(1, min(244, _log(rng, min(per, 1 << 17), most) // per))
    if kind == "host":
        c["chunk"] = rng.randint(1, min(4, c["subbands"]))
    return c


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------

def _taps(T, C):
    """Kaiser-windowed sinc prototype of T*C taps, unit sum."""
    L = T * C
    n = np.arange(L, dtype=np.float64)
    h = np.sinc((n - (L - 1) / 2.0) / C) * np.kaiser(L, 9.0)
    return (h / h.sum()).astype(np.float32)


def _centres(SB):
    return 150e6 + (np.arange(SB, dtype=np.float64) - SB // 2) * FS


def _calibration(case, seed):
    """Delays at the block's two ends [N], bandpass [N][C], gains [N][2][2] (host arrays)."""
    rng = np.random.default_rng([seed, 7])
    N, C = case["stations"], case["channels"]
    d0 = rng.uniform(-DELAY_S, DELAY_S, N)
    d1 = d0 + rng.uniform(-2e-8, 2e-8, N)             # fringe rate over one block
    bp = (1 + 0.05 * np.sin(2 * np.pi * (rng.uniform(1, 3, (N, 1)) * np.arange(C) / C + rng.uniform(0, 1, (N, 1)))))
    amp, ph = rng.uniform(0.8, 1.2, (N, 2)), rng.uniform(0, 2 * np.pi, (N, 2))
    g = np.stack([amp * np.cos(ph), amp * np.sin(ph)], -1)
    return d0, d1, bp.astype(np.float32), g.astype(np.float32)


def _sky(case, seed, n_samples, device="cuda"):
    """Station samples [SB][N][n_samples][2][re, im] (one packed byte for ci4):
    Gaussian noise plus one point source on a channel centre per subband."""
    N, SB, C, fmt = case["stations"], case["subbands"], case["channels"], case["format"]
    d0 = torch.from_numpy(_calibration(case, seed)[0]).cuda()
    last, dt = {"ci16": (2, torch.int16), "ci8": (2, torch.int8), "ci4": (1, torch.uint8)}[fmt]
    raw = torch.empty((SB, N, n_samples, 2, last), dtype=dt, device=device, pin_memory=device == "cpu")
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 13)
    t = torch.arange(n_samples, device="cuda")
    pol = torch.tensor([1.0, 0.75 * np.exp(1j * np.pi / 3)], dtype=torch.complex64, device="cuda")
    lim = LIMIT[fmt]
    for sb in range(SB):
        m = 1 + (seed + 5 * sb) % (C - 1) - C // 2
        z = torch.randn((N, n_samples, 2, 2), generator=g, device="cuda") * SIGMA[fmt]
        tone = torch.exp(2j * math.pi * ((m * t) % C).double() / C).to(torch.complex64)
        stat = torch.exp(-2j * math.pi * (_centres(SB)[sb] + m * FS / C) * d0).to(torch.complex64)
        z += torch.view_as_real((0.5 * SIGMA[fmt]) * (stat[:, None, None] * tone[None, :, None]) * pol)
        q = z.round_().clamp_(-lim, lim)
        if fmt == "ci4":
            qi = q.to(torch.int32) & 15
            raw[sb] = ((qi[..., 0] << 4) | qi[..., 1]).to(torch.uint8)[..., None]
        else:
            raw[sb].copy_(q.to(dt))
    return raw


def _correlator(case, **kw):
    return fx.Correlator(case["stations"], case["subbands"], case["channels"], case["spectra"],
                         taps=_taps(case.get("taps", 16), case["channels"]), centres=_centres(case["subbands"]),
                         n_taps=case.get("taps", 16), fmt=FORMATS[case.get("format", "ci16")],
                         precision=PRECISIONS[case["precision"]], **kw)


def _block_samples(case):
    return (case["spectra"] + case["taps"] - 1) * case["channels"]


def _chan(case, seed):
    """Channelised samples [SB][N][2][S][C][2]: noise of unit variance and a common
    signal seen with each station's delay at the block's middle."""
    N, SB, C, S = (case[k] for k in ("stations", "subbands", "channels", "spectra"))
    d0, d1 = _calibration(case, seed)[:2]
    f = torch.from_numpy(_centres(SB)[:, None] + (np.arange(C) - C // 2) * FS / C).cuda()      # [SB][C]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    chan = torch.randn((SB, N, 2, S, C, 2), generator=g, device="cuda")
    mid = torch.from_numpy((d0 + d1) / 2).cuda()
    for sb in range(SB):
        sig = torch.randn((2, S, C), dtype=torch.complex64, generator=g, device="cuda")
        ph = torch.exp(-2j * math.pi * mid[:, None] * f[sb]).to(torch.complex64)                # [N][C]
        chan[sb] += torch.view_as_real(sig[None] * ph[:, None, None, :])
    return chan


def _job_shapes(case):
    rng = random.Random(case["shape_seed"])
    return [(rng.randint(24, 96), rng.choice([16, 64, 256]), rng.randint(case["spectra_lo"], case["spectra_hi"]))
            for _ in range(case["jobs"])]


def _job_operands(case, seed):
    """Corrected operands of each job, planar [C][planes][I_pad][S_pad], and its shape."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 19)
    dt = torch.bfloat16 if case["precision"] == "bf16" else torch.float16
    out = []
    for N, C, S in _job_shapes(case):
        I, Ip, Sp = 2 * N, (2 * N + 15) // 16 * 16, (S + 63) // 64 * 64
        y = torch.randn((C, 2, I, S), generator=g, device="cuda") * 20
        y += torch.randn((C, 2, 1, S), generator=g, device="cuda") * 10       # a source all stations see
        split = case["precision"] == "f16_split"
        corr = torch.zeros((C, 4 if split else 2, Ip, Sp), dtype=dt, device="cuda")
        corr[:, :2, :I, :S] = y.to(dt)
        if split:
            corr[:, 2:, :I, :S] = (y - corr[:, :2, :I, :S].float()).to(dt)
        out.append((N, C, S, corr))
    return out


class _Batch:
    """A batch plan over jobs' operands and visibilities (the C ABI's fx_batch)."""

    def __init__(self, jobs, precision):
        self.lib = _abi.load()
        arr = (_abi.fx_job * len(jobs))()
        for a, (N, C, S, corr, vis) in zip(arr, jobs):
            a.n_stations, a.n_subbands, a.n_channels, a.n_spectra = N, 1, C, S
            a.d_corr, a.d_vis = corr.data_ptr(), vis.data_ptr()
        self.keep, self.plan = jobs, ctypes.c_void_p()
        _abi.check(self.lib.fx_batch_create(arr, len(jobs), precision, 0.0, ctypes.byref(self.plan)), "fx_batch_create")

    def __call__(self):
        s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        _abi.check(self.lib.fx_correlate_batched(self.plan, s), "fx_correlate_batched")
        return [vis for *_, vis in self.keep]

    def __del__(self):
        if self.plan:
            self.lib.fx_batch_destroy(self.plan)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        jobs = [(N, C, S, corr, torch.empty((1, C, N * (N + 1) // 2, 4, 2), device="cuda"))
                for N, C, S, corr in _job_operands(case, seed)]
        return {"kind": kind, "batch": _Batch(jobs, PRECISIONS[case["precision"]])}
    d0, d1, bp, g = _calibration(case, seed)
    if kind == "host":
        c = _correlator(case, host_chunk_subbands=case["chunk"])
        return {"kind": kind, "c": c, "raw": _sky(case, seed, _block_samples(case), "cpu"),
                "cal": tuple(torch.from_numpy(x).pin_memory() for x in (d0, d1, bp, g)),
                "vis": torch.empty(c.vis_shape(), pin_memory=True)}
    cal = tuple(torch.from_numpy(x).cuda() for x in (d0, d1, bp, g))
    if kind == "train":
        c = _correlator(case)
        rng = torch.Generator(device="cuda")
        rng.manual_seed(seed * 7919 + 23)
        grad = torch.randn(c.vis_shape(), generator=rng, device="cuda")
        return {"kind": kind, "c": c, "chan": _chan(case, seed), "bp": cal[2], "grad": grad,
                "leaves": [cal[3].requires_grad_(), cal[0].requires_grad_(), cal[1].requires_grad_()]}
    if kind == "stream":
        c = _correlator(case, streaming=True, max_coarse_shift=case["max_shift"])
        shift, flags = _stream_extras(case, seed)
        s = {"kind": kind, "c": c, "new": _sky(case, seed, case["spectra"] * case["channels"]), "cal": cal,
             "shift": torch.from_numpy(shift).cuda(), "flags": torch.from_numpy(flags).cuda(),
             "corr": torch.empty(c.corr_shape(), dtype=c.corr_dtype(), device="cuda"),
             "vis": torch.empty(c.vis_shape(), device="cuda")}
        run(s)                        # the stream is under way: the handle holds the block before
        return s
    c = _correlator(case, max_beams=case.get("beams", 0))
    s = {"kind": kind, "c": c, "raw": _sky(case, seed, _block_samples(case)), "cal": cal,
         "corr": torch.empty(c.corr_shape(), dtype=c.corr_dtype(), device="cuda")}
    if kind == "beam":
        beams, weights = _beam_extras(case, seed)
        s.update(delays=torch.from_numpy(beams).cuda(), weights=torch.from_numpy(weights).cuda(),
                 output=case["output"], tint=case["tint"],
                 out=torch.empty(c.beam_shape(case["beams"], case["output"], case["tint"]), device="cuda"))
    else:
        s["vis"] = torch.empty(c.vis_shape(), device="cuda")
    if kind == "layers":
        s["chan"] = torch.empty(c.chan_shape(), device="cuda")
    return s


def _stream_extras(case, seed):
    rng = np.random.default_rng([seed, 11])
    shift = rng.integers(0, case["max_shift"] + 1, case["stations"]).astype(np.int32)
    flags = (rng.uniform(size=(case["stations"], case["spectra"])) > 0.01).astype(np.float32)
    return shift, flags


def _beam_extras(case, seed):
    rng = np.random.default_rng([seed, 12])
    return (rng.uniform(-2e-6, 2e-6, (case["beams"], case["stations"])),
            rng.uniform(0.5, 1.5, case["stations"]).astype(np.float32))


def run(s):
    kind = s["kind"]
    if kind == "batch":
        return s["batch"]()
    c = s["c"]
    if kind == "host":
        d0, d1, bp, g = s["cal"]
        return c.process_host(s["raw"], d0, d1, bandpass=bp, gains=g, out=s["vis"])
    if kind == "train":
        gains, d0, d1 = s["leaves"]
        vis = autograd.correct_correlate(c, s["chan"], gains, d0, bandpass=s["bp"], delays_end=d1)
        return [vis.detach(), *torch.autograd.grad(vis, s["leaves"], s["grad"])]
    d0, d1, bp, g = s["cal"]
    if kind == "stream":
        _, vis, counts = c.stream_block(s["new"], d0, d1, coarse_shift=s["shift"], bandpass=bp, gains=g,
                                        flags=s["flags"], corr=s["corr"], vis=s["vis"])
        return [vis, counts]
    if kind == "layers":
        chan = c.channelize(s["raw"], out=s["chan"])
        corr = c.correct(chan, d0, d1, bandpass=bp, gains=g, out=s["corr"])
        return [chan, corr, c.correlate(corr, out=s["vis"])]
    corr = c.channelize_correct(s["raw"], d0, d1, bandpass=bp, gains=g, out=s["corr"])
    if kind == "beam":
        return c.beamform(corr, s["delays"], station_weights=s["weights"], output=s["output"], tint=s["tint"],
                          out=s["out"])
    return c.correlate(corr, out=s["vis"])


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    if case["kind"] == "batch":
        size = 8 if case["precision"] == "f16_split" else 4
        b = f = 0
        for N, C, S in _job_shapes(case):
            prods = C * N * (N + 1) // 2 * 4
            b += 2 * N * C * S * size + prods * 8
            f += prods * S * 8
        return {"bytes": b, "flops": f}
    N, SB, C, S = (case[k] for k in ("stations", "subbands", "channels", "spectra"))
    samples, prods = SB * N * 2 * S * C, SB * C * N * (N + 1) // 2 * 4
    xflops = 8 * prods * S
    if case["kind"] == "train":       # vis forward; K and M1, then the contraction, backward
        return {"bytes": 2 * samples * 8 + 2 * prods * 8, "flops": 3 * xflops + 3 * 14 * samples}
    T = case["taps"]
    fir_in = S * C if case["kind"] == "stream" else _block_samples(case)
    fflops = samples * (4 * T + 5 * math.log2(C) + 12)
    byt = SB * N * 2 * fir_in * RAW_BYTES[case["format"]]
    if case["kind"] == "beam":
        per = {0: 16, 1: 4, 2: 16}[case["output"]]
        return {"bytes": byt + SB * case["beams"] * C * (S // case["tint"]) * per,
                "flops": fflops + 8 * samples * case["beams"]}
    byt += prods * 8
    if case["kind"] == "layers":      # both intermediates are outputs and inputs of the next call
        size = {"f32": 8, "tf32_split": 8, "f16_split": 8}.get(case["precision"], 4)
        byt += samples * 2 * (8 + size)
    return {"bytes": byt, "flops": fflops + xflops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _samples64(case, raw):
    """Raw samples of one subband [N][L][2](re, im or byte) -> complex128 [N][2][L]."""
    if case["format"] == "ci4":
        b = raw[..., 0].to(torch.int32)
        re, im = b >> 4, b & 15
        re, im = re - 16 * (re > 7), im - 16 * (im > 7)
        z = torch.complex(re.double(), im.double())
    else:
        z = torch.complex(raw[..., 0].double(), raw[..., 1].double())
    return z.permute(0, 2, 1)


def _channels64(case, z):
    """[N][2][L] -> [N][2][S][C], ascending sky frequency."""
    C, S, T = case["channels"], case["spectra"], case["taps"]
    h = torch.from_numpy(_taps(T, C)).cuda().double().reshape(T, C)
    x = z.reshape(z.shape[0], 2, -1, C)
    u = sum(x[:, :, k:k + S] * h[k] for k in range(T))
    return torch.fft.fftshift(torch.fft.fft(u, dim=-1), dim=-1)


def _factor64(case, sb, d0, d1):
    """exp(2 pi i f_k tau_n(s)): [N][S][C]."""
    C, S = case["channels"], case["spectra"]
    f = torch.from_numpy(_centres(case["subbands"])[sb] + (np.arange(C) - C // 2) * FS / C).cuda()
    frac = torch.arange(S, device="cuda", dtype=torch.float64) / S
    tau = d0[:, None] + (d1 - d0)[:, None] * frac
    cycles = tau[:, :, None] * f
    return torch.exp(2j * math.pi * (cycles - torch.round(cycles).detach()))


def _vis64(y):
    """[N][2][S][C] -> [C][B][4][2], baselines i <= j at j(j+1)/2 + i."""
    N = y.shape[0]
    m = y.permute(3, 0, 1, 2).reshape(y.shape[3], 2 * N, y.shape[2])
    v = torch.matmul(m, m.conj().transpose(1, 2)).reshape(-1, N, 2, N, 2).permute(0, 1, 3, 2, 4)
    j, i = torch.tril_indices(N, N, device=y.device)
    return torch.view_as_real(v[:, i, j].reshape(-1, i.numel(), 4).contiguous())


def _planes64(case, y):
    """[N][2][S][C] -> the X-stage's operand layout of one subband (f32 or two planes)."""
    N, _, S, C = y.shape
    if case["precision"] == "f32":
        S16 = (S + 15) // 16 * 16
        out = torch.zeros((C, S16, N, 2), dtype=torch.complex128, device=y.device)
        out[:, :S] = y.permute(3, 2, 0, 1)
        return torch.view_as_real(out.reshape(C, S16 // 16, 16, N, 2).permute(0, 1, 3, 2, 4).contiguous())
    out = torch.zeros((C, 2, (2 * N + 15) // 16 * 16, (S + 63) // 64 * 64), dtype=torch.float64, device=y.device)
    rows = y.permute(3, 0, 1, 2).reshape(C, 2 * N, S)
    out[:, 0, :2 * N, :S], out[:, 1, :2 * N, :S] = rows.real, rows.imag
    return out


def _beams64(case, y, sb, delays, weights):
    C, S, tint = case["channels"], case["spectra"], case["tint"]
    f = torch.from_numpy(_centres(case["subbands"])[sb] + (np.arange(C) - C // 2) * FS / C).cuda()
    cycles = delays[:, :, None] * f
    w = weights[:, None] * torch.exp(2j * math.pi * (cycles - torch.round(cycles)))             # [b][N][C]
    b = torch.einsum("bnk,npsk->bksp", w, y)
    X, Y = b[..., 0], b[..., 1]
    if case["output"] == 0:
        return torch.view_as_real(b).reshape(*b.shape[:3], 4)
    ix, iy, xy = X.abs() ** 2, Y.abs() ** 2, X * Y.conj()
    st = [ix + iy] if case["output"] == 1 else [ix + iy, ix - iy, 2 * xy.real, 2 * xy.imag]
    st = [v.reshape(v.shape[0], C, S // tint, tint).sum(-1) for v in st]
    return st[0] if case["output"] == 1 else torch.stack(st, -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for N, C, S, corr in _job_operands(case, seed):
            v = corr[:, :, :2 * N, :S].double()
            y = torch.complex(v[:, 0], v[:, 1]) if v.shape[1] == 2 else torch.complex(v[:, 0] + v[:, 2], v[:, 1] + v[:, 3])
            out.append(_vis64(y.reshape(C, N, 2, S).permute(1, 2, 3, 0))[None])
        return out
    SB = case["subbands"]
    d0, d1, bp, g = (torch.from_numpy(x).cuda().double() for x in _calibration(case, seed))
    gc = torch.complex(g[..., 0], g[..., 1])
    if kind == "train":
        return _train64(case, seed, d0, d1, bp, g)
    if kind == "stream":
        raw = _sky(case, seed, case["spectra"] * case["channels"])
        shift, flags = (torch.from_numpy(x).cuda() for x in _stream_extras(case, seed))
    else:
        raw = _sky(case, seed, _block_samples(case))
    if kind == "beam":
        delays, weights = (torch.from_numpy(x).cuda() for x in _beam_extras(case, seed))
    chans, corrs, outs = [], [], []
    for sb in range(SB):
        z = _samples64(case, raw[sb])
        if kind == "stream":          # the block before was the same samples
            n, L = z.shape[2], _block_samples(case)
            at = torch.arange(L, device="cuda") + (2 * n - L) - shift[:, None]
            start = torch.where(at < 0, 0.0, 1.0)
            z = torch.cat([z, z], 2).gather(2, at.clamp(min=0)[:, None].expand(-1, 2, -1)) * start[:, None]
        x = _channels64(case, z)
        y = x * (_factor64(case, sb, d0, d1) * bp[:, None, :])[:, None] * gc[:, :, None, None]
        if kind == "stream":
            y = y * flags[:, None, :, None]
        if kind == "beam":
            outs.append(_beams64(case, y, sb, delays, weights.double()))
            continue
        if kind == "layers":
            chans.append(torch.view_as_real(x.contiguous()))
            if case["precision"] != "f16_split":
                corrs.append(_planes64(case, y))
        outs.append(_vis64(y))
    out = torch.stack(outs)
    if kind == "layers":
        return [torch.stack(chans), torch.stack(corrs) if corrs else None, out]
    if kind == "stream":
        j, i = torch.tril_indices(case["stations"], case["stations"], device="cuda")
        return [out, (flags.double() @ flags.double().T)[i, j]]
    return out


def _train64(case, seed, d0, d1, bp, g):
    chan = _chan(case, seed)
    rng = torch.Generator(device="cuda")
    rng.manual_seed(seed * 7919 + 23)
    N = case["stations"]
    grad = torch.randn((case["subbands"], case["channels"], N * (N + 1) // 2, 4, 2), generator=rng, device="cuda")
    leaves = [g.requires_grad_(), d0.requires_grad_(), d1.requires_grad_()]
    total, out = None, []
    for sb in range(case["subbands"]):
        y = torch.view_as_complex(chan[sb].double()) * (_factor64(case, sb, d0, d1) * bp[:, None, :])[:, None]
        v = _vis64(y * torch.view_as_complex(g)[:, :, None, None])
        got = torch.autograd.grad(v, leaves, grad[sb].double())
        total = got if total is None else [a + b for a, b in zip(total, got)]
        out.append(v.detach())
    return [torch.stack(out), *total]
