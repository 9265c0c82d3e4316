"""The FP32 X-stage (FX_F32) on the tensor cores: bits that depend on nothing but
the operands."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def correlator(N, SB, C, S, **kw):
    import paper_1801_04834_gb300 as m
    return m.Correlator(N, SB, C, S, taps=synth.kaiser_sinc_taps(4, C), centres=synth.subband_centres(SB), n_taps=4, **kw)


# tiles with station slots that no station fills: time segments (7), groups of channels with
# an incomplete last one (9), a ragged tile (50), a ragged off-diagonal one (78), both (130)
@pytest.mark.parametrize("N,SB,C,S", [(7, 1, 16, 256), (9, 5, 64, 160), (50, 1, 16, 200), (78, 1, 16, 144),
                                      (130, 1, 16, 128)])
def test_same_bits_whatever_shared_memory_held(N, SB, C, S):
    """Raw samples of 0x7f7f, which another handle's F-stage leaves in shared memory, are
    words of the size at which the X-stage splits operands with more care."""
    import paper_1801_04834_gb300 as m
    c = correlator(N, SB, C, S)
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    corr = m.f32_block(torch.randn((SB, C, S, N, 2, 2), generator=g, device="cuda") * 50)
    seen = []
    for channels in (16, 64, 256):
        f = correlator(32, 8, channels, 64)
        tau = torch.zeros(32, dtype=torch.float64, device="cuda")
        for word in (0, 0x7f7f):
            f.channelize_correct(torch.full(f.raw_shape(), word, dtype=torch.int16, device="cuda"), tau, tau)
            seen.append(c.correlate(corr))
        f.close()
    assert all(torch.equal(seen[0], v) for v in seen[1:])
    assert c.poll_status() == (0, 0)
    c.close()


def product(y):
    SB, C, S, N = y.shape[:4]
    m = torch.view_as_complex(y.double()).reshape(SB, C, S, 2 * N).transpose(2, 3)
    v = torch.matmul(m, m.conj().transpose(2, 3)).reshape(SB, C, N, 2, N, 2).permute(0, 1, 2, 4, 3, 5)
    j, i = torch.tril_indices(N, N, device="cuda")
    return torch.view_as_real(v[:, :, i, j].reshape(SB, C, -1, 4).contiguous())


def operands(kind, N, C, S):
    g = torch.Generator(device="cuda")
    g.manual_seed(N * S)
    y = torch.randn((1, C, S, N, 2, 2), generator=g, device="cuda") * 50
    if kind == "common":                              # a signal all stations share
        y += torch.randn((1, C, S, 1, 1, 2), generator=g, device="cuda") * 30
    elif kind == "half":                              # every station loses half of its spectra
        y *= torch.randint(0, 2, (1, 1, S, N, 1, 1), generator=g, device="cuda")
    elif kind != "noise":                             # the first so many spectra of `kind` are there, spread out
        at = torch.randperm(S, generator=g, device="cuda")[int(kind):]
        y[:, :, at] = 0
    return y


@pytest.mark.parametrize("N", [8, 50, 76])            # time segments, one tile, off-diagonal tiles
@pytest.mark.parametrize("S", [128, 383, 384, 768, 1023, 1024, 1536])
@pytest.mark.parametrize("kind", ["noise", "common", "half"])
def test_no_less_accurate_than_the_fma_chain(N, S, kind):
    """Normwise over all baselines, over the cross baselines alone (whose sums are small
    where stations are uncorrelated), and the worst single baseline (over channels and pols)."""
    import paper_1801_04834_gb300 as m
    C = 16
    y = operands(kind, N, C, S)
    ref = product(y)
    i, j = torch.tril_indices(N, N, device="cuda")
    err = []
    for form in ("auto", "2x4"):
        c = correlator(N, 1, C, S, xf32_form=form)
        e = c.correlate(m.f32_block(y)).double() - ref
        per = (e.pow(2).sum((0, 1, 3, 4)) / ref.pow(2).sum((0, 1, 3, 4))).sqrt()
        cross = (e[:, :, i != j].norm() / ref[:, :, i != j].norm()).item()
        err.append(((e.norm() / ref.norm()).item(), cross, per.max().item()))
        c.close()
    assert all(a <= b for a, b in zip(*err)), err


@pytest.mark.parametrize("N", [8, 50, 76])
@pytest.mark.parametrize("S,live", [(128, 1), (128, 16), (1024, 1), (1024, 4), (1024, 16)])
def test_few_live_spectra(N, S, live):
    """Where a chain barely rounds, what is left is the product's own error. An operand keeps 23
    of its 24 bits (2^-24 of it RMS, at most 2^-23), lo lo' is 2^-24 RMS, and the accumulator
    loses up to 2^-24 of its value an MMA, 2 or 3 of them after the main term of a live
    spectrum (both K-steps and planes): 4 x 2^-24 normwise."""
    import paper_1801_04834_gb300 as m
    C = 16
    y = operands(str(live), N, C, S)
    c = correlator(N, 1, C, S)
    ref = product(y)
    assert ((c.correlate(m.f32_block(y)).double() - ref).norm() / ref.norm()).item() < 4 * 2.0 ** -24
    c.close()


@pytest.mark.parametrize("N,S", [(7, 256), (20, 160), (78, 144)])   # time segments, one tile, off-diagonal tiles
def test_infinities_as_on_the_cuda_cores(N, S):
    """Whole numbers have no low part, and an infinity times that would be a NaN: infinities keep
    their places and signs, NaNs theirs, and everything else its value (but for Im X X*)."""
    import paper_1801_04834_gb300 as m
    C = 16
    y = operands("noise", N, C, S).round()
    for k, (s, n, p, part, value) in enumerate([(7, 4, 0, 0, float("inf")), (S - 1, N - 1, 1, 1, float("-inf")),
                                                (S // 2, 2, 1, 0, float("nan")), (3, 0, 0, 1, 3.4e38)]):
        y[0, 3 * k + 1, s, n, p, part] = value
    vis = []
    for form in ("auto", "2x4"):
        c = correlator(N, 1, C, S, xf32_form=form)
        vis.append(c.correlate(m.f32_block(y)))
        assert c.poll_status() == (0, 0)
        c.close()
    i, j = torch.tril_indices(N, N, device="cuda")
    for v in vis:                                     # Im X X* is 0, or what its overflowing halves leave: no value to compare
        v[:, :, i == j, 0, 1] = v[:, :, i == j, 3, 1] = 0
    a, b = vis
    assert torch.equal(torch.isnan(a), torch.isnan(b))
    assert torch.equal(torch.isposinf(a), torch.isposinf(b)) and torch.equal(torch.isneginf(a), torch.isneginf(b))
    plain = [k for k in range(C) if k % 3 != 1 or k > 10]
    assert torch.equal(a[:, plain], b[:, plain])      # sums of whole numbers below 2^24: exact in both


@pytest.mark.parametrize("N,S", [(5, 300), (20, 1100), (64, 128)])
def test_cuda_core_form_at_any_length(N, S):
    """The FP32 FMA chain in 4 x 4 tiles (2 x 4 below 16 stations), also where the tensor cores
    are the default: per visibility the same chain as in 2 x 4 tiles, bit for bit."""
    import paper_1801_04834_gb300 as m
    C = 16
    y = operands("noise", N, C, S)
    corr, vis = m.f32_block(y), {}
    for form in ("4x4", "2x4", "auto"):
        c = correlator(N, 1, C, S, xf32_form=form)
        vis[form] = c.correlate(corr)
        c.close()
    assert torch.equal(vis["4x4"], vis["2x4"])
    assert not torch.equal(vis["4x4"], vis["auto"])   # the default is another form at this length
    ref = product(y)
    assert ((vis["4x4"].double() - ref).norm() / ref.norm()).item() < S * 2.0 ** -24


def test_cuda_core_form_full_shape_sampled():
    """The CUDA-core form at the LOFAR shape (64 stations, 10 subbands, 64 channels, 3072 spectra:
    256-thread blocks, 32-spectrum chunks) on sampled channels, held to the FP32 path's bound."""
    import paper_1801_04834_gb300 as m
    N, SB, C, S = 64, 10, 64, 3072
    c = correlator(N, SB, C, S, xf32_form="4x4")
    g = torch.Generator(device="cuda")
    g.manual_seed(180104834)
    corr = torch.randn(c.corr_shape(), generator=g, device="cuda") * 30
    vis = c.correlate(corr)
    y = m.f32_unblock(corr, S)
    for sb, k in ((0, 0), (4, 31), (9, 63)):
        ref = product(y[sb:sb + 1, k:k + 1].contiguous())[0, 0]
        assert ((vis[sb, k].double() - ref).norm() / ref.norm()).item() < 1e-5
    c.close()
