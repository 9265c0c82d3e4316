"""fx_process_host over small arrays with FP32 operands, whose X-stage would rather
split time than channels where a launch has few of them: the bits of the
device-resident calls, whatever the chunk."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


# 1360 spectra: 8 MB of raw samples a subband, so the last chunk passes subband by subband
@pytest.mark.parametrize("N,SB,S", [(12, 5, 1360), (20, 5, 300), (7, 2, 300)])
@pytest.mark.parametrize("chunk", [1, 2, 5])
@pytest.mark.parametrize("precision", [0, 4])
def test_bits_of_the_device_calls(N, SB, S, chunk, precision):
    import paper_1801_04834_gb300 as m
    C = 64
    c = m.Correlator(N, SB, C, S, taps=synth.kaiser_sinc_taps(16, C), centres=synth.subband_centres(SB),
                     precision=precision, host_chunk_subbands=chunk)
    raw = synth.make_raw_torch(4, synth.CI16, SB, N, C, S)
    assert (raw[0].numel() * 2 >= 8 << 20) == (S == 1360)
    tau = torch.from_numpy(np.random.default_rng(1).uniform(-5e-6, 5e-6, N))
    ref = c.correlate(c.channelize_correct(raw, tau.cuda(), tau.cuda())).cpu()
    assert torch.equal(c.process_host(raw.cpu().pin_memory(), tau, tau), ref)
    c.close()
