"""The serving loop's aggregation, resampling and whitening kernels at the edges
of their tiles: strides whose new samples fill one and several blocks of
outputs or only a few of a warp's, whitening filters shorter than a warp and
not a multiple of it, a decimator longer than one block of taps, and emission
that starts inside a group of 4 samples.  References: the FP64 stream oracle's
cleaned series; from it, by direct sums, the decimated and whitened series of
any filter lengths, and the oracle's BBHnet.  Bound: relative L2 1e-5."""
import numpy as np
import pytest

import tests.test_gpu_serve as base
from oracle import fir as ofir, nets, stream as ostream
from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, rel_l2

pytestmark = pytest.mark.gpu


def direct_logits(cleaned, S, delta, f, h, Lb):
    n_det, n, _ = cleaned.shape
    c = np.zeros((n_det, n * S))
    for k in range(n):
        t = ostream.emit_times(k, S, delta)
        c[:, t[t >= 0]] = cleaned[:, k, t >= 0]
    hf, hw = (len(f) - 1) // 2, (len(h) - 1) // 2
    # known below c_end: decimated m with 2 m + hf < c_end, whitened n with n + hw < m_end
    params, head = synth.bbhnet_params(base.BBH_SEED)
    out = np.zeros(n)
    for k in range(n):
        c_end = (k + 1) * S - delta
        me = (c_end - hf - 1) // 2 + 1 if c_end > hf else 0
        x = np.zeros((1, n_det, Lb))
        for d in range(n_det):
            cp = np.concatenate([np.zeros(hf), c[d], np.zeros(hf)])
            dec = np.correlate(cp, f, "valid")[:2 * me:2][:me]
            ne = me - hw
            if ne > 0:
                w = np.correlate(np.concatenate([np.zeros(hw), dec]), h, "valid")[:ne]
                m = min(ne, Lb)
                x[0, d, Lb - m:] = w[ne - m:]
        out[k] = nets.bbhnet_forward(x, params, head, synth.bbhnet_layers())[0]
    return out


@pytest.mark.parametrize("mode", [G.GW_AGG_AVERAGE, G.GW_AGG_LATEST])
@pytest.mark.parametrize("strides,kh,kf,delta", [((2048, 1024), 257, 127, 512), ((8, 32), 31, 5, 0),
                                                 ((512, 16), 2049, 127, 7), ((256, 1024), 33, 1201, 1)])
def test_pipeline_edges(gpu_lib, monkeypatch, mode, strides, kh, kf, delta):
    monkeypatch.setattr(base, "KF", kf)
    nfft = 8192 if kh > 513 else 512
    _, psd = synth.psd_grid(base.FS2, nfft)
    f, h = ofir.lowpass_fir(kf, base.FC, base.FS), ofir.whitening_fir(psd, base.FS2, nfft, kh)
    ctx = Ctx()
    try:
        rig = base.Rig(ctx, G.GW_FP32, W=4096, max_stride=max(strides), mode=mode, delta=delta, Kh=kh, nfft=nfft)
        streams = [(1000 * kf + 10 * i, s, max(3, min(12, 4096 // s))) for i, s in enumerate(strides)]
        got = rig.run(streams, base.interleaved(streams, 3))
        monkeypatch.setattr(base, "KF", 127)  # the oracle's own resampling takes no other; its cleaned series has none
        for (seed, S, n), (cl, lg) in zip(streams, got):
            ref_cl, _ = rig.oracle(seed, S, n)
            strain = base.strain_emitted(seed, S, n, delta)
            assert rel_l2(cl - strain, ref_cl - strain) <= base.TOL32
            assert rel_l2(lg, direct_logits(ref_cl, S, delta, f, h, rig.Lb)) <= base.TOL32
    finally:
        ctx.close()
