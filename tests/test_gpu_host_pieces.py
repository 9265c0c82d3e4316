"""fx_process_host with subbands long enough (8 MB of raw samples) for the last
chunk to pass subband by subband: the same visibilities as the device-resident
calls, whatever the chunk (the last one whole, ragged, or the only one). FP16
at 34 stations: pieces and whole blocks run the same items, so the same bits."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [1, 2, 3, 5])
def test_last_chunk_in_pieces(chunk):
    import paper_1801_04834_gb300 as m
    SB, N, C, S = 5, 34, 64, 500
    c = m.Correlator(N, SB, C, S, taps=synth.kaiser_sinc_taps(16, C), centres=synth.subband_centres(SB),
                     precision=m.FX_F16, host_chunk_subbands=chunk)
    raw = synth.make_raw_torch(4, synth.CI16, SB, N, C, S)
    assert raw[0].numel() * 2 >= 8 << 20
    tau = torch.from_numpy(np.random.default_rng(1).uniform(-5e-6, 5e-6, N))
    ref = c.correlate(c.channelize_correct(raw, tau.cuda(), tau.cuda())).cpu()
    h_raw = raw.cpu().pin_memory()
    for _ in range(2):                                # the second call reuses every buffer and event
        assert torch.equal(c.process_host(h_raw, tau, tau), ref)
    c.close()
