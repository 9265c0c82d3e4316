"""The fused F-stage at 256 channels with FP32 operands against the whole chain in
FP64 (filter bank and correction): no further from it than the two separate
calls, which evaluate every phase factor by itself."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
C, T = 256, 16


@pytest.mark.parametrize("N,S", [(9, 100), (20, 300)])
@pytest.mark.parametrize("moving", [0.0, 2e-8])
def test_fused_no_further_from_fp64_than_two_calls(N, S, moving):
    import paper_1801_04834_gb300 as m
    rng = np.random.default_rng(N)
    blk = synth.make_block(5 + N, synth.CI16, 1, N, C, S, sigma=100.0)
    d0 = torch.from_numpy(rng.uniform(-5e-6, 5e-6, N)).cuda()
    d1 = d0 + moving * torch.from_numpy(rng.uniform(-1, 1, N)).cuda()
    bp = torch.from_numpy(rng.uniform(0.5, 1.5, (N, C)).astype(np.float32)).cuda()
    g = torch.from_numpy(synth.random_gains(rng, N).astype(np.float32)).cuda()
    raw = torch.from_numpy(blk.raw).cuda()
    c = m.Correlator(N, 1, C, S, taps=blk.taps, centres=blk.centres, n_taps=T)
    fused = c.channelize_correct(raw, d0, d1, bandpass=bp, gains=g)
    two = c.correct(c.channelize(raw), d0, d1, bandpass=bp, gains=g)

    x = torch.view_as_complex(raw[0].double()).permute(0, 2, 1).reshape(N, 2, S + T - 1, C)
    h = torch.from_numpy(np.asarray(blk.taps, np.float32)).cuda().double().reshape(T, C)
    u = sum(x[:, :, k:k + S] * h[k] for k in range(T))
    f = float(blk.centres[0]) + (torch.arange(C, device="cuda") - C // 2).double() * synth.SAMPLE_RATE_HZ / C
    tau = d0[:, None] + (d1 - d0)[:, None] * (torch.arange(S, device="cuda").double() / S)
    cyc = tau[:, :, None] * f
    factor = torch.exp(2j * np.pi * (cyc - torch.round(cyc))) * bp.double()[:, None, :]           # [N][S][C]
    y = torch.fft.fftshift(torch.fft.fft(u, dim=-1), dim=-1) * factor[:, None]
    y = y * torch.view_as_complex(g.double())[:, :, None, None]
    ref = torch.view_as_real(y.permute(3, 2, 0, 1).contiguous())[None]                            # [1][C][S][N][2][2]

    def rel(t):
        return ((m.f32_unblock(t, S).double() - ref).norm() / ref.norm()).item()
    assert rel(fused) <= rel(two), (rel(fused), rel(two))
    c.close()
