"""FP32 weight and bias gradients at the edges of their tiles: rows that end
inside a block of 8 positions, a run or a chunk, one to many items, and input
channel counts around the 8 of a warp.  Reference: PyTorch float64 autograd on
the CPU; the FP32 path's bound, rel-L2 1e-5 per parameter group (random output
gradients, so no group cancels)."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev, rel_l2

pytestmark = pytest.mark.gpu
BOUND = 1e-5


def raw_params(n_in, seed):
    """Raw parameters with n_in input channels."""
    params = synth.deepclean_params(seed)
    rng = np.random.default_rng(seed)
    params[0]["w"] = (rng.standard_normal((8, n_in, 7)) * np.sqrt(2.0 / (7 * n_in))).astype(np.float32)
    return params


def torch_forward(x, params):
    for p, (kind, _, _, _, stride, pad, _, out_pad, bn, act) in zip(params, synth.DEEPCLEAN_LAYERS):
        if kind == "conv":
            x = F.conv1d(x, p["w"], p["b"], stride=stride, padding=pad)
        else:
            x = F.conv_transpose1d(x, p["w"], p["b"], stride=stride, padding=pad, output_padding=out_pad)
        if bn:
            x = F.batch_norm(x, p["mean"], p["var"], p["gamma"], p["beta"], training=False, eps=1e-5)
        x = torch.tanh(x) if act == "tanh" else x
    return x[:, 0]


@pytest.mark.parametrize("batch,length,n_in,checkpoint",
                         [(1, 16, 21, 0), (2, 24, 1, 0), (3, 136, 8, 1), (1, 1032, 9, 0), (5, 264, 21, 0),
                          (2, 2056, 33, 0), (17, 1024, 21, 1), (40, 520, 24, 0)])
def test_gradients(gpu_lib, batch, length, n_in, checkpoint):
    rng = np.random.default_rng(batch + length)
    params = raw_params(n_in, 3)
    x = rng.standard_normal((batch, n_in, length)).astype(np.float32)
    dy = rng.standard_normal((batch, length)).astype(np.float32)
    t = [{k: torch.from_numpy(np.asarray(v, np.float64)).requires_grad_(k not in ("mean", "var")) for k, v in p.items()}
         for p in params]
    y = torch_forward(torch.from_numpy(x.astype(np.float64)), t)
    y.backward(torch.from_numpy(dy.astype(np.float64)))
    ctx = Ctx()
    try:
        trainer = G.gw_trainer_create(ctx.h, n_in, batch, length, checkpoint)
        ctx.objs.append((G.gw_trainer_destroy, trainer))
        p, xd, dyd = dev(synth.flatten_params(params)), dev(x), dev(dy)
        yd = torch.full((batch, length), float("nan"), device="cuda")
        dp = torch.full_like(p, float("nan"))
        G.gw_trainer_forward(trainer, p.data_ptr(), xd.data_ptr(), batch, yd.data_ptr())
        G.gw_trainer_backward(trainer, dyd.data_ptr(), dp.data_ptr())
        torch.cuda.synchronize()
        got, o = dp.cpu().numpy(), 0
        assert rel_l2(yd.cpu().numpy(), y.detach().numpy()) <= BOUND
        for layer, q in enumerate(t):
            for k in synth.PARAM_ORDER:
                if k not in q:
                    continue
                n = q[k].numel()
                if k in ("mean", "var"):
                    assert not got[o:o + n].any()
                else:
                    e = rel_l2(got[o:o + n], q[k].grad.numpy().ravel())
                    assert e <= BOUND, (layer, k, e)
                o += n
    finally:
        ctx.close()
