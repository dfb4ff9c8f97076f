"""Tensor-core weight and bias gradients (BF16 operands, FP32 forward) at the
edges of their tiles: rows that end inside a segment of 8 positions or a chunk of
64, fewer chunks than CTAs, input channel counts around the 32 rows of a pass and
at the limit of the kernel, and one beyond it (the FP32 kernel).  Reference:
PyTorch float64 autograd; bound: rel-L2 1e-2 per parameter group (both operands
rounded to BF16, at most 2^-8 relative per product).  The output layer's bias
gradient is one sum of the random output gradients, which cancels; each term is
rounded by at most 2^-9 of its size, so it is held to 2^-8 of the sum of their
sizes."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev, rel_l2
from tests.test_gpu_wgrad_f32_tiles import raw_params, torch_forward

pytestmark = pytest.mark.gpu
BOUND = 1e-2


@pytest.mark.parametrize("batch,length,n_in", [(1, 16, 21), (2, 72, 1), (3, 520, 32), (1, 1096, 33), (5, 264, 36),
                                              (2, 136, 40), (40, 520, 21)])
def test_gradients(gpu_lib, batch, length, n_in):
    rng = np.random.default_rng(batch + length)
    params = raw_params(n_in, 3)
    x = rng.standard_normal((batch, n_in, length)).astype(np.float32)
    dy = rng.standard_normal((batch, length)).astype(np.float32)
    t = [{k: torch.from_numpy(np.asarray(v, np.float64)).requires_grad_(k not in ("mean", "var")) for k, v in p.items()}
         for p in params]
    torch_forward(torch.from_numpy(x.astype(np.float64)), t).backward(torch.from_numpy(dy.astype(np.float64)))
    ctx = Ctx()
    try:
        trainer = G.gw_trainer_create(ctx.h, n_in, batch, length, precision=G.GW_BF16)
        ctx.objs.append((G.gw_trainer_destroy, trainer))
        p, xd, dyd = dev(synth.flatten_params(params)), dev(x), dev(dy)
        yd, dp = torch.empty(batch, length, device="cuda"), torch.full_like(p, float("nan"))
        G.gw_trainer_forward(trainer, p.data_ptr(), xd.data_ptr(), batch, yd.data_ptr())
        G.gw_trainer_backward(trainer, dyd.data_ptr(), dp.data_ptr())
        G.gw_trainer_status(trainer)
        got, o = dp.cpu().numpy(), 0
        for layer, q in enumerate(t):
            for k in synth.PARAM_ORDER:
                if k not in q:
                    continue
                n = q[k].numel()
                if (layer, k) == (7, "b"):
                    assert abs(got[o] - q[k].grad.item()) <= 2.0 ** -8 * np.abs(dy).sum()
                elif k not in ("mean", "var"):
                    e = rel_l2(got[o:o + n], q[k].grad.numpy().ravel())
                    assert e <= BOUND, (layer, k, e)
                o += n
    finally:
        ctx.close()
