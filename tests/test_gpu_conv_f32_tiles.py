"""FP32 conv kernel over its tile choices: batches and lengths at which the
launch rule takes each tile (one window split over input channels up to full
launches), rows that end inside a tile, and inputs whose rows are and are not
16-byte aligned.  Reference: the FP64 oracle; the FP32 path's bound, rel-L2
1e-5."""
import numpy as np
import pytest

from oracle import nets
from paper_2108_12430_gb300 import synth

pytestmark = pytest.mark.gpu

BOUND = 1e-5


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    from tests.gpu_util import Ctx

    c = Ctx()
    yield c
    c.close()


# batch, length, floats before the first sample, samples between rows beyond the series
@pytest.mark.parametrize("batch,length,offset,slack", [(1, 8, 0, 0), (1, 40, 1, 3), (1, 4104, 0, 0), (3, 1016, 2, 1),
                                                      (5, 8, 3, 0), (9, 2072, 0, 4), (24, 4136, 1, 0),
                                                      (40, 8192, 0, 0)])
@pytest.mark.parametrize("standardise", [False, True])
def test_deepclean_tiles(ctx, batch, length, offset, slack, standardise):
    import torch
    from paper_2108_12430_gb300 import gwstream as G
    from tests.gpu_util import rel_l2

    rng = np.random.default_rng(batch * 1000 + length)
    step = 37
    n = length + (batch - 1) * step
    x = rng.standard_normal((21, n)).astype(np.float32)
    mean = rng.standard_normal(21).astype(np.float32) if standardise else None
    std = rng.uniform(0.5, 2.0, 21).astype(np.float32) if standardise else None
    ld = n + slack
    buf = torch.zeros(offset + 21 * ld, device="cuda")
    buf[offset:].view(21, ld)[:, :n] = torch.from_numpy(x).cuda()
    y = torch.full((batch, length), float("nan"), device="cuda")
    m = ctx.deepclean(2, G.GW_FP32, mean, std)
    G.gw_deepclean_forward(m, buf.data_ptr() + 4 * offset, ld, step, batch, length, y.data_ptr())
    torch.cuda.synchronize()
    some = sorted({0, batch // 2, batch - 1})
    w = np.stack([x[:, b * step:b * step + length] for b in some]).astype(np.float64)
    if standardise:
        w = (w - mean[:, None].astype(np.float64)) / std[:, None].astype(np.float64)
    ref = nets.deepclean_forward(w, synth.deepclean_params(2), synth.DEEPCLEAN_LAYERS)
    assert rel_l2(y.cpu().numpy()[some], ref) <= BOUND


@pytest.mark.parametrize("batch,length", [(1, 16), (1, 2048), (2, 1040), (7, 112), (33, 272), (200, 48), (48, 2048)])
def test_bbhnet_tiles(ctx, batch, length):
    import torch
    from paper_2108_12430_gb300 import gwstream as G
    from tests.gpu_util import dev

    x = np.random.default_rng(length + batch).standard_normal((batch, 2, length)).astype(np.float32)
    out = torch.full((batch,), float("nan"), device="cuda")
    xd = dev(x)
    G.gw_bbhnet_score(ctx.bbhnet(4), xd.data_ptr(), batch, length, out.data_ptr())
    torch.cuda.synchronize()
    some = sorted({0, batch // 2, batch - 1})
    layers, head = synth.bbhnet_params(4)
    ref = nets.bbhnet_forward(x[some].astype(np.float64), layers, head, synth.bbhnet_layers())
    assert np.abs(out.cpu().numpy()[some] - ref).max() <= BOUND * max(1.0, np.abs(ref).max())
