"""Fused F-stage at 256 channels: the phase factor of an output is an anchor at
channel k1 + 128 times up to eight steps of exp(2 pi i (fs / 16) tau). Against
fx_channelize + fx_correct, which evaluate every factor by itself, over long
and fast-moving delays (so that the step's angle covers the circle), runs that
wrap the four row buffers, and ragged ends.

Bound per sample: eight rotations, each two roundings of 2^-24 per component,
and a step that is rounded once (8 x 2 x 2^-24 + 8 x 2^-24 = 1.4e-6), plus the
intrinsics' 4e-7 of the anchor here and of the factor there: 2.3e-6 normwise.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,SB,S,tau", [(3, 2, 16, 5e-6), (2, 1, 83, 1e-4), (5, 1, 200, 2e-3), (1, 3, 64, 0.0)])
@pytest.mark.parametrize("fmt", [synth.CI16, synth.CI8])
def test_factors_match_two_calls(N, SB, S, tau, fmt):
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
    ref = c.correct(c.channelize(raw), d0, d1, bandpass=bp, gains=g)
    e = ((out.double() - ref.double()).norm() / ref.double().norm()).item()
    assert e < 2.3e-6, e
    assert torch.all(out[:, :, :, :, S:] == 0) and torch.all(out[:, :, :, c.I:] == 0)
    c.close()
