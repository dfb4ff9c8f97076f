"""The training calls take float arrays at any float's address: input, prediction,
its gradient, parameters and their gradient one to three floats off a 16-byte
boundary give the bits of aligned ones (the vector and the scalar rows of every
kernel on the way)."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tc_data", [(G.GW_FP32, 0), (G.GW_BF16, 0), (G.GW_BF16, 1)])
@pytest.mark.parametrize("batch,length", [(1, 136), (3, 2056)])
def test_unaligned_arrays(gpu_lib, precision, tc_data, batch, length):
    rng = np.random.default_rng(length)
    params = synth.flatten_params(synth.deepclean_params(3))
    x = rng.standard_normal((batch, 21, length)).astype(np.float32)
    dy = rng.standard_normal((batch, length)).astype(np.float32)
    mean, std = rng.standard_normal(21).astype(np.float32), rng.uniform(0.5, 2.0, 21).astype(np.float32)
    ctx = Ctx()
    try:
        t = G.gw_trainer_create(ctx.h, 21, batch, length, 0, mean, std, precision=precision, tc_data=tc_data)
        ctx.objs.append((G.gw_trainer_destroy, t))

        def run(off):
            def at(a):
                b = torch.full((off + a.size,), float("nan"), device="cuda")
                b[off:] = torch.from_numpy(np.ascontiguousarray(a, np.float32).ravel()).cuda()
                return b

            pd, xd, dyd = at(params), at(x), at(dy)
            yd, dp = at(np.full(dy.shape, np.nan)), at(np.full(params.shape, np.nan))
            ptr = lambda b: b.data_ptr() + 4 * off  # noqa: E731
            G.gw_trainer_forward(t, ptr(pd), ptr(xd), batch, ptr(yd))
            G.gw_trainer_backward(t, ptr(dyd), ptr(dp))
            G.gw_trainer_status(t)
            return yd[off:].cpu().numpy(), dp[off:].cpu().numpy()

        y, g = run(0)
        assert np.isfinite(y).all() and np.isfinite(g).all()
        for off in (1, 2, 3):
            yo, go = run(off)
            assert np.array_equal(y, yo) and np.array_equal(g, go), off
    finally:
        ctx.close()
