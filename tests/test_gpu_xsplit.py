"""X-stages on the tensor cores with FP32 operands (FX_TF32_SPLIT and, from 128
spectra on, FX_F32) on given operands against an FP64 product: small arrays
whose channels, or time segments, share a tile, ragged row blocks, integrations that end inside a
16-spectrum block, every accumulator chain length of FX_F32.

Bound: a real accumulator takes per 16 spectra at most 6 MMAs on a diagonal tile
(8 off the diagonal, where a chunk adds twice as many cross terms), each losing
up to 2^-24 of the running sum; chains of c such stages are summed in IEEE
FP32, and the split itself (BF16 cross terms, dropped lo lo') stays below 4 x
2^-24 with zero mean. So (8 c + 4) 2^-24 normwise.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -24


def correlator(N, SB, C, S, precision, **kw):
    import paper_1801_04834_gb300 as m
    return m.Correlator(N, SB, C, S, taps=synth.kaiser_sinc_taps(4, C), centres=synth.subband_centres(SB), n_taps=4,
                        precision=precision, **kw)


def operands(N, SB, C, S, seed):
    """[SB][C][S][N][2][2]: noise plus a signal all stations share."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    y = torch.randn((SB, C, S, N, 2, 2), generator=g, device="cuda") * 50
    return y + torch.randn((SB, C, S, 1, 1, 2), generator=g, device="cuda") * 30


def laid_out(c, y):
    import paper_1801_04834_gb300 as m
    if c.precision == 0:
        return m.f32_block(y)
    corr = torch.zeros(c.corr_shape(), device="cuda")
    corr[:, :, :, :c.I, :c.S] = y.reshape(c.SB, c.C, c.S, c.I, 2).permute(0, 1, 4, 3, 2)
    return corr


def product(y):
    SB, C, S, N = y.shape[:4]
    m = torch.view_as_complex(y.double()).reshape(SB, C, S, 2 * N).transpose(2, 3)
    v = torch.matmul(m, m.conj().transpose(2, 3)).reshape(SB, C, N, 2, N, 2).permute(0, 1, 2, 4, 3, 5)
    j, i = torch.tril_indices(N, N, device="cuda")
    return torch.view_as_real(v[:, :, i, j].reshape(SB, C, -1, 4).contiguous())


def rel(a, b):
    return ((a.double() - b).norm() / b.norm()).item()


# (stations, subbands, channels, spectra): 8 stations x 320 channels share tiles in
# pairs, 768 in fives with a remainder, 31 stations in pairs; 64 stations fill a
# tile, 65 to 130 need off-diagonal ones and ragged last blocks
SHAPES = [(1, 1, 16, 128), (8, 5, 64, 129), (8, 3, 256, 130), (31, 7, 64, 143), (32, 5, 64, 384), (33, 1, 64, 400),
          (64, 1, 16, 1537), (65, 1, 16, 385), (76, 2, 16, 200), (130, 1, 16, 1536),
          # few channels: time segments share a tile (8 of 96, 2 of 208, 4 of 240 with the
          # last one short, 2 of a block that ends inside the first of the second's stages)
          (8, 1, 64, 768), (24, 1, 16, 385), (13, 2, 16, 900), (3, 1, 16, 131)]


@pytest.mark.parametrize("N,SB,C,S", SHAPES)
@pytest.mark.parametrize("precision", [0, 4])
def test_given_operands(N, SB, C, S, precision):
    c = correlator(N, SB, C, S, precision)
    y = operands(N, SB, C, S, N + S)
    corr = laid_out(c, y)
    if precision == 0 and S % 16:                     # FX_F32: what lies past S is not read as a sample
        corr.reshape(SB, C, -1, N, 16, 2, 2)[:, :, -1, :, S % 16:] = float("nan")
    vis = torch.full(c.vis_shape(), float("nan"), device="cuda")
    c.correlate(corr, out=vis)
    stages = 4 if precision == 4 or S >= 1536 else 2 if S >= 384 else 1
    assert rel(vis, product(y)) < (8 * stages + 4) * ULP
    i, j = torch.tril_indices(N, N)
    auto = vis[:, :, torch.nonzero(i == j)[:, 0].cuda()]
    assert torch.all(auto[..., [0, 3], 1] == 0)       # X X* is real
    assert c.poll_status() == (0, 0)
    c.close()


def test_infinite_sample_stays_in_its_baselines():
    """FX_F32: as on the CUDA cores, an infinity or NaN only reaches baselines of its station."""
    N, SB, C, S = 20, 1, 16, 160
    y = operands(N, SB, C, S, 3)
    y[0, 2, 7, 4, 0, 0] = float("inf")
    y[0, 3, 9, 11, 1, 1] = float("nan")
    y[0, 4, 11, 1, 0, 1] = 3.4e38
    tc, cc = correlator(N, SB, C, S, 0), correlator(N, SB, C, S, 0, xf32_form="2x4")
    a, b = tc.correlate(laid_out(tc, y)), cc.correlate(laid_out(cc, y))
    assert torch.equal(torch.isfinite(a).all(-1), torch.isfinite(b).all(-1))
    assert torch.equal(torch.isinf(a[..., 0]), torch.isinf(b[..., 0]))
    tc.close()
    cc.close()


def test_forms_agree_and_accumulate():
    """The CUDA-core form (asked for by flag) agrees with the tensor-core one, and pieces
    added into the visibilities (fx_channelize_correlate) agree with the whole block."""
    N, SB, C, S = 20, 2, 64, 256
    rng = np.random.default_rng(5)
    blk = synth.make_block(9, synth.CI16, SB, N, C, S, sigma=100.0)
    import paper_1801_04834_gb300 as m
    kw = dict(taps=blk.taps, centres=blk.centres, n_taps=16)
    tau = torch.from_numpy(rng.uniform(-5e-6, 5e-6, N)).cuda()
    raw = torch.from_numpy(blk.raw).cuda()
    whole, cores = m.Correlator(N, SB, C, S, **kw), m.Correlator(N, SB, C, S, xf32_form="2x4", **kw)
    pieces = m.Correlator(N, SB, C, S, chunk_subbands=1, chunk_spectra=128, **kw)
    corr = whole.channelize_correct(raw, tau, tau)
    v = whole.correlate(corr)
    assert rel(v, cores.correlate(corr).double()) < 12 * ULP + S * ULP   # + the FMA chain's own bound
    assert rel(pieces.channelize_correlate(raw, tau, tau), v.double()) < 2 * 12 * ULP
    for c in (whole, cores, pieces):
        c.close()


@pytest.mark.parametrize("N,SB,C,S", [(3, 5, 64, 70), (8, 4, 256, 200), (17, 3, 256, 64), (31, 7, 64, 300)])
@pytest.mark.parametrize("precision", [1, 2, 3])
def test_channels_share_a_tile_16_bit(N, SB, C, S, precision):
    """FP16/BF16/split operands of small arrays, several channels per tile with a remainder
    (N = 8: six per tile; 17: five; 3 and 31: two): the same bits as a handle of one subband,
    whose channels are too few to share."""
    import paper_1801_04834_gb300 as m
    whole = correlator(N, SB, C, S, precision)
    taps = synth.kaiser_sinc_taps(4, 16)
    one = m.Correlator(N, 1, 16, S, taps=taps, centres=synth.subband_centres(1), n_taps=4, precision=precision)
    y = operands(N, SB, C, S, N).reshape(SB, C, S, 2 * N, 2).permute(0, 1, 4, 3, 2)
    dt = whole.corr_dtype()
    corr = torch.zeros(whole.corr_shape(), dtype=dt, device="cuda")
    corr[:, :, :2, :whole.I, :S] = y.to(dt)
    if precision == 3:
        corr[:, :, 2:, :whole.I, :S] = (y - y.to(dt).float()).to(dt)
    vis = torch.full(whole.vis_shape(), float("nan"), device="cuda")
    whole.correlate(corr, out=vis)
    for sb in range(SB):
        for c0 in range(0, C, 16):
            part = one.correlate(corr[sb:sb + 1, c0:c0 + 16].contiguous())
            assert torch.equal(vis[sb:sb + 1, c0:c0 + 16], part), (sb, c0)
    whole.close()
    one.close()
