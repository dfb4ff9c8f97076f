"""Tensor-core conv plans at the edges of their rules: batches with enough tiles
for several M sub-tiles per unit, items of one tile (padding rows zeroed once) and
of several, layers split over columns, and a FIR whose K-steps exceed the
parameter table.  References: the FP64 oracle (BBHnet logits within 0.05) and
direct sums in float64 (FIR rel-L2 2e-2), the BF16 path's bounds."""
import numpy as np
import pytest
import torch

from oracle import nets
from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = Ctx()
    yield c
    c.close()


@pytest.mark.parametrize("batch,length", [(700, 2048), (1, 2048), (19, 2048), (90, 512), (2, 6144)])
def test_bbhnet(ctx, batch, length):
    x = np.random.default_rng(length + batch).standard_normal((batch, 2, length)).astype(np.float32)
    xd = dev(x)
    m = ctx.bbhnet(6, G.GW_BF16)
    out = torch.full((batch,), float("nan"), device="cuda")
    G.gw_bbhnet_score(m, xd.data_ptr(), batch, length, out.data_ptr())
    G.gw_model_status(m)
    some = sorted({0, batch // 2, batch - 1})
    layers, head = synth.bbhnet_params(6)
    ref = nets.bbhnet_forward(x[some].astype(np.float64), layers, head, synth.bbhnet_layers())
    assert np.abs(out.cpu().numpy()[some] - ref).max() <= 0.05


@pytest.mark.parametrize("rows,taps,length", [(1, 9, 64), (2, 129, 1160), (3, 2049, 2056), (1, 2049, 12288),
                                              (5, 3073, 8192), (2, 4097, 4608), (700, 513, 1024), (64, 2049, 4160)])
def test_fir(ctx, rows, taps, length):
    f = G.gw_fir_create_lowpass(ctx.h, 900.0, 4096.0, taps, G.GW_BF16)
    ctx.objs.append((G.gw_fir_destroy, f))
    h = G.gw_fir_taps(f)
    x = np.random.default_rng(rows + taps).standard_normal((rows, length)).astype(np.float32)
    xd = dev(x)
    y = torch.full((rows, length - taps + 1), float("nan"), device="cuda")
    G.gw_whiten(f, xd.data_ptr(), rows, 1, length, y.data_ptr())
    torch.cuda.synchronize()
    # the FIR writes whole groups of 8 outputs
    n = (length - taps + 1) // 8 * 8
    some = sorted({0, rows // 2, rows - 1})
    ref = np.stack([np.correlate(x[r].astype(np.float64), h, "valid") for r in some])[:, :n]
    assert rel_l2(y.cpu().numpy()[some][:, :n], ref) <= 2e-2
