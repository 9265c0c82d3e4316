"""Fused F-stage at 256 channels: the phase factor of an output is an anchor at
channel k1 + 128 times up to eight steps of exp(2 pi i (fs / 16) tau). Against
the channelised block corrected in FP64, over long and fast-moving delays (so
that the step's angle covers the circle), runs that wrap the four row buffers,
and ragged ends.

Bound: both this call and fx_correct interpolate the phase angle in FP32, which
for a fast-moving delay is what decides (2^-24 of the phase travelled over the
block); fx_correct evaluates every factor by itself, so its error against FP64
measures that term for the same inputs. On top of it come here eight rotations
of two roundings of 2^-24 per component, a step rounded once (1.4e-6 in all)
and the two paths' sines, 4e-7 each, and FFT roundings: 2.3e-6 normwise.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def corrected64(c, chan, centres, d0, d1, bp, g):
    """[SB][C][2][I][S] from the channelised block."""
    x = torch.view_as_complex(chan.double())                                       # [SB][N][2][S][C]
    f = torch.from_numpy(centres[:, None] + (np.arange(256) - 128) * synth.SAMPLE_RATE_HZ / 256).cuda()
    tau = d0[:, None] + (d1 - d0)[:, None] * (torch.arange(c.S, device="cuda", dtype=torch.float64) / c.S)
    cyc = tau[None, :, :, None] * f[:, None, None, :]                               # [SB][N][S][C]
    y = x * (torch.exp(2j * np.pi * (cyc - torch.round(cyc))) * bp.double()[None, :, None, :])[:, :, None]
    y = y * torch.view_as_complex(g.double())[None, :, :, None, None]
    y = y.permute(0, 4, 1, 2, 3).reshape(c.SB, 256, c.I, c.S)
    return torch.stack([y.real, y.imag], 2)


@pytest.mark.parametrize("N,SB,S,tau", [(3, 2, 16, 5e-6), (2, 1, 83, 1e-4), (5, 1, 200, 2e-3), (1, 3, 64, 0.0)])
@pytest.mark.parametrize("fmt", [synth.CI16, synth.CI8])
def test_factors_against_fp64(N, SB, S, tau, fmt):
    import paper_1801_04834_gb300 as m
    rng = np.random.default_rng(S)
    blk = synth.make_block(7 + S, fmt, SB, N, 256, S, sigma=100.0 if fmt == synth.CI16 else 20.0)
    c = m.Correlator(N, SB, 256, S, taps=blk.taps, centres=blk.centres, n_taps=16, fmt=fmt, precision=m.FX_TF32_SPLIT)
    d0 = torch.from_numpy(rng.uniform(-tau, tau, N)).cuda()
    d1 = d0 + torch.from_numpy(rng.uniform(-tau, tau, N)).cuda() / 10
    bp = torch.from_numpy(rng.uniform(0.5, 1.5, (N, 256)).astype(np.float32)).cuda()
    g = torch.from_numpy(synth.random_gains(rng, N).astype(np.float32)).cuda()
    raw = torch.from_numpy(blk.raw).cuda()
    out = torch.full(c.corr_shape(), float("nan"), device="cuda")
    c.channelize_correct(raw, d0, d1, bandpass=bp, gains=g, out=out)
    chan = c.channelize(raw)
    two = c.correct(chan, d0, d1, bandpass=bp, gains=g)
    ref = corrected64(c, chan, blk.centres, d0, d1, bp, g)

    def rel(t):
        return ((t[:, :, :, :c.I, :S].double() - ref).norm() / ref.norm()).item()
    assert rel(out) < 1.5 * rel(two) + 2.3e-6, (rel(out), rel(two))
    assert torch.all(out[:, :, :, :, S:] == 0) and torch.all(out[:, :, :, c.I:] == 0)
    c.close()


@pytest.mark.parametrize("N,SB,S,tau", [(3, 2, 16, 5e-6), (2, 1, 83, 1e-4), (5, 1, 200, 2e-3), (1, 3, 1, 0.0)])
@pytest.mark.parametrize("fmt", [synth.CI16, synth.CI8])
def test_spectrum_blocked_factors_against_fp64(N, SB, S, tau, fmt):
    """The same factors and bound for FX_F32, whose stores swap spectra between lanes."""
    import paper_1801_04834_gb300 as m
    from paper_1801_04834_gb300.api import f32_unblock
    rng = np.random.default_rng(S)
    blk = synth.make_block(9 + S, fmt, SB, N, 256, S, sigma=100.0 if fmt == synth.CI16 else 20.0)
    c = m.Correlator(N, SB, 256, S, taps=blk.taps, centres=blk.centres, n_taps=16, fmt=fmt)
    d0 = torch.from_numpy(rng.uniform(-tau, tau, N)).cuda()
    d1 = d0 + torch.from_numpy(rng.uniform(-tau, tau, N)).cuda() / 10
    bp = torch.from_numpy(rng.uniform(0.5, 1.5, (N, 256)).astype(np.float32)).cuda()
    g = torch.from_numpy(synth.random_gains(rng, N).astype(np.float32)).cuda()
    raw = torch.from_numpy(blk.raw).cuda()
    out = torch.full(c.corr_shape(), float("nan"), device="cuda")
    c.channelize_correct(raw, d0, d1, bandpass=bp, gains=g, out=out)
    chan = c.channelize(raw)
    two = c.correct(chan, d0, d1, bandpass=bp, gains=g)
    ref = corrected64(c, chan, blk.centres, d0, d1, bp, g)

    def rel(t):
        y = f32_unblock(t, S).double().reshape(SB, 256, S, c.I, 2).permute(0, 1, 4, 3, 2)
        return ((y - ref).norm() / ref.norm()).item()
    assert rel(out) < 1.5 * rel(two) + 2.3e-6, (rel(out), rel(two))
    assert torch.all(f32_unblock(out, out.shape[2] * 16)[:, :, S:] == 0)
    c.close()
