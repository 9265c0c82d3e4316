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
