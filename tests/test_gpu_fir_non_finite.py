"""A non-finite sample in the FP32 FIR: every output whose taps do not cover it is
written and near its reference, every output with a nonzero tap on it is not
finite.  The sample at the row's ends, inside a tile and at the edges of blocks of
taps; tap counts that end inside a block of 16, and more than one block."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G
from tests.gpu_util import Ctx, rel_l2
from tests.test_gpu_fir_tiles import BOUND, lowpass

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 64])
@pytest.mark.parametrize("taps", [17, 127, 2049, 4101])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_sample(gpu_lib, rows, taps, value):
    ctx = Ctx()
    try:
        fir, h = lowpass(ctx, taps)
        n, row = taps + 1500, rows // 2
        rng = np.random.default_rng(taps)
        for at in (0, 15, 16, 700, n // 2, taps - 1, n - 1):
            x = rng.standard_normal((rows, n)).astype(np.float32)
            ref = np.stack([np.correlate(r.astype(np.float64), h, "valid") for r in x])
            x[row, at] = value
            xd = torch.from_numpy(x).cuda()
            y = torch.full(ref.shape, float("nan"), device="cuda")
            G.gw_whiten(fir, xd.data_ptr(), rows, 1, n, y.data_ptr())
            torch.cuda.synchronize()
            got, m = y.cpu().numpy(), np.arange(n - taps + 1)
            tap = at - m  # the tap that each output has on the sample
            covers = (tap >= 0) & (tap < taps)
            clean = np.ones(ref.shape, bool)
            clean[row] = ~covers
            assert np.isfinite(got[clean]).all()
            assert rel_l2(np.where(clean, got, 0.0), np.where(clean, ref, 0.0)) <= BOUND
            hit = covers & (h[np.clip(tap, 0, taps - 1)].astype(np.float32) != 0.0)
            assert hit.any() or at in (0, n - 1)  # the window makes the end taps zero
            assert not np.isfinite(got[row][hit]).any()
    finally:
        ctx.close()
