"""gw_band_loss with r in the memory of one of its inputs: at its start, inside it,
across either end.  The tiles that write r run beside the ones that still read the
inputs.  Loss and r have to be those of a call with r in memory of its own, bit
for bit."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = Ctx()
    yield c
    c.close()


@pytest.mark.parametrize("batch,length", [(1, 2049), (3, 4099), (32, 8192)])
@pytest.mark.parametrize("which", ["strain", "y_hat"])
@pytest.mark.parametrize("place", ["start", "inside", "before", "behind"])
def test_r_overlaps_an_input(ctx, batch, length, which, place):
    _, psd = synth.psd_grid(4096.0, 8192)
    fir = G.gw_fir_create_band_loss(ctx.h, psd, 4096.0, 2049)
    ctx.objs.append((G.gw_fir_destroy, fir))
    rng = np.random.default_rng(length)
    s, p = (torch.from_numpy(rng.standard_normal(batch * length).astype(np.float32)).cuda() for _ in range(2))
    n_r = batch * (length - 2048)
    loss = torch.zeros(2, device="cuda")
    ref = torch.zeros(n_r, device="cuda")
    G.gw_band_loss(fir, s.data_ptr(), p.data_ptr(), batch, length, loss.data_ptr(), ref.data_ptr())
    # the input in the middle of a larger buffer, r at an offset from its start
    buf = torch.zeros(n_r + batch * length + n_r, device="cuda")
    buf[n_r:n_r + batch * length] = s if which == "strain" else p
    at = n_r + {"start": 0, "inside": min(2048, batch * length - n_r), "before": -(n_r // 2),
                "behind": batch * length - (n_r + 1) // 2}[place]
    inp = buf.data_ptr() + 4 * n_r
    a, b = (inp, p.data_ptr()) if which == "strain" else (s.data_ptr(), inp)
    G.gw_band_loss(fir, a, b, batch, length, loss.data_ptr() + 4, buf.data_ptr() + 4 * at)
    torch.cuda.synchronize()
    assert torch.equal(buf[at:at + n_r], ref) and loss[0].item() == loss[1].item()
    assert np.isfinite(loss.cpu().numpy()).all() and loss[0].item() > 0
