"""FP32 FIR at the edges of its tiles: tap counts around the 16 taps of a block,
outputs that end inside a thread's run, few and many outputs (4, 8 or 16 per
thread), rows that are and are not 16-byte aligned, and a non-finite sample,
which may reach only the outputs whose taps cover it.  Reference: direct sums in
float64; the FP32 path's bound, rel-L2 1e-5."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, rel_l2

pytestmark = pytest.mark.gpu
BOUND = 1e-5


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = Ctx()
    yield c
    c.close()


def lowpass(ctx, taps):
    f = G.gw_fir_create_lowpass(ctx.h, 900.0, 4096.0, taps)
    ctx.objs.append((G.gw_fir_destroy, f))
    return f, G.gw_fir_taps(f)


@pytest.mark.parametrize("rows,taps,extra,offset", [(1, 3, 0, 0), (1, 15, 1, 1), (2, 17, 5, 0), (3, 31, 63, 2),
                                                   (1, 127, 4095, 0), (64, 33, 1000, 3), (5, 2049, 1, 0),
                                                   (300, 129, 2050, 0), (512, 65, 1027, 1), (1, 21001, 300, 0)])
def test_fir_and_adjoint(ctx, rows, taps, extra, offset):
    fir, h = lowpass(ctx, taps)
    n = taps + extra
    rng = np.random.default_rng(taps + rows)
    x = rng.standard_normal((rows, n)).astype(np.float32)
    dy = rng.standard_normal((rows, extra + 1)).astype(np.float32)
    buf = torch.zeros(offset + rows * n, device="cuda")
    buf[offset:] = torch.from_numpy(x.ravel()).cuda()
    y = torch.full((rows, extra + 1), float("nan"), device="cuda")
    dx = torch.full((rows, n), float("nan"), device="cuda")
    G.gw_whiten(fir, buf.data_ptr() + 4 * offset, rows, 1, n, y.data_ptr())
    dyd = torch.from_numpy(dy).cuda()
    G.gw_fir_backward(fir, dyd.data_ptr(), rows, 1, n, dx.data_ptr())
    torch.cuda.synchronize()
    some = sorted({0, rows // 2, rows - 1})
    ref = np.stack([np.correlate(x[r].astype(np.float64), h, "valid") for r in some])
    assert rel_l2(y.cpu().numpy()[some], ref) <= BOUND
    ref = np.stack([np.convolve(dy[r].astype(np.float64), h) for r in some])
    assert rel_l2(dx.cpu().numpy()[some], ref) <= BOUND


@pytest.mark.parametrize("taps", [17, 127])
def test_non_finite_sample_stays_in_its_outputs(ctx, taps):
    fir, _ = lowpass(ctx, taps)
    n, at = taps + 700, 400
    x = np.ones((1, n), np.float32)
    x[0, at] = np.inf
    xd = torch.from_numpy(x).cuda()
    y = torch.zeros(1, n - taps + 1, device="cuda")
    G.gw_whiten(fir, xd.data_ptr(), 1, 1, n, y.data_ptr())
    torch.cuda.synchronize()
    bad = ~np.isfinite(y.cpu().numpy()[0])
    covers = np.arange(n - taps + 1)
    covers = (covers <= at) & (at < covers + taps)
    assert not (bad & ~covers).any()


@pytest.mark.parametrize("batch,length", [(1, 2056), (3, 2300), (32, 4099)])
def test_band_loss(ctx, batch, length):
    _, psd = synth.psd_grid(4096.0, 8192)
    fir = G.gw_fir_create_band_loss(ctx.h, psd, 4096.0, 2049)
    ctx.objs.append((G.gw_fir_destroy, fir))
    g = G.gw_fir_taps(fir)
    rng = np.random.default_rng(length)
    s, p = (rng.standard_normal((batch, length)).astype(np.float32) for _ in range(2))
    sd, pd = torch.from_numpy(s).cuda(), torch.from_numpy(p).cuda()
    r = torch.zeros(batch, length - 2048, device="cuda")
    loss, dl = torch.zeros(1, device="cuda"), torch.full((1,), 3.0, device="cuda")
    dy = torch.zeros(batch, length, device="cuda")
    G.gw_band_loss(fir, sd.data_ptr(), pd.data_ptr(), batch, length, loss.data_ptr(), r.data_ptr())
    G.gw_band_loss_backward(fir, r.data_ptr(), batch, length, dl.data_ptr(), dy.data_ptr())
    torch.cuda.synchronize()
    ref = np.stack([np.correlate(a, g, "valid") for a in s.astype(np.float64) - p.astype(np.float64)])
    assert rel_l2(r.cpu().numpy(), ref) <= BOUND
    assert abs(loss.item() - np.mean(ref ** 2)) <= BOUND * np.mean(ref ** 2)
    dref = np.stack([np.convolve(a, g) for a in ref]) * (-2.0 / ref.size) * 3.0
    assert rel_l2(dy.cpu().numpy(), dref) <= BOUND
