"""A trainer's memory, and its gradients where the weight gradients' partials of
all layers do not fit their buffer together and are added up in several groups:
short batches, input channel counts whose gradient buffers leave the partials
more or less room.  The byte counts are what a trainer took when its FP32 weight
gradients were one partial per 256 positions and layer (with the operand images
of tc_data); a budget that held one then holds one still."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev, rel_l2
from tests.test_gpu_wgrad_f32_tiles import raw_params, torch_forward

pytestmark = pytest.mark.gpu

# n_in, max_batch, length, precision, tc_data, checkpoint: bytes
TOOK = [((8, 1, 8192, G.GW_FP32, 0, 0), 3313920), ((8, 8, 4096, G.GW_FP32, 0, 0), 11868160),
        ((8, 8, 4096, G.GW_BF16, 0, 1), 9902080), ((21, 1, 16, G.GW_FP32, 0, 0), 536800),
        ((21, 1, 8192, G.GW_FP32, 0, 0), 4600608), ((21, 1, 8192, G.GW_BF16, 1, 0), 7056456),
        ((21, 8, 4096, G.GW_FP32, 0, 1), 15546912), ((21, 8, 4096, G.GW_BF16, 1, 0), 23868232),
        ((21, 32, 8192, G.GW_FP32, 0, 0), 132600352), ((21, 32, 8192, G.GW_BF16, 0, 0), 135221792),
        ((21, 32, 8192, G.GW_BF16, 1, 0), 173951816), ((21, 32, 8192, G.GW_BF16, 1, 1), 162417480),
        ((40, 8, 4096, G.GW_BF16, 1, 0), 34445640)]


@pytest.mark.parametrize("desc,took", TOOK)
def test_budget(gpu_lib, desc, took):
    n_in, batch, length, precision, tc_data, checkpoint = desc
    ctx = Ctx(budget=took)
    try:
        t = G.gw_trainer_create(ctx.h, n_in, batch, length, checkpoint, precision=precision, tc_data=tc_data)
        G.gw_trainer_destroy(t)
        assert G.gw_ctx_bytes_in_use(ctx.h) == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("precision,tc_data,bound", [(G.GW_FP32, 0, 1e-5), (G.GW_BF16, 0, 1e-2), (G.GW_BF16, 1, 4e-2)])
@pytest.mark.parametrize("batch,length,n_in,checkpoint", [(1, 8192, 8, 0), (1, 2304, 1, 1), (2, 4096, 21, 0),
                                                          (6, 2304, 9, 1), (1, 4096, 40, 0)])
def test_gradients_in_groups(gpu_lib, precision, tc_data, bound, batch, length, n_in, checkpoint):
    # bounds: the FP32 path's; BF16 operands as for the other gradient tests, per layer
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
        trainer = G.gw_trainer_create(ctx.h, n_in, batch, length, checkpoint, precision=precision, tc_data=tc_data)
        ctx.objs.append((G.gw_trainer_destroy, trainer))
        p, xd, dyd = dev(synth.flatten_params(params)), dev(x), dev(dy)
        yd, grads = torch.full((batch, length), float("nan"), device="cuda"), []
        for _ in range(2):  # the second step finds the buffer as the first left it
            dp = torch.full_like(p, float("nan"))
            G.gw_trainer_forward(trainer, p.data_ptr(), xd.data_ptr(), batch, yd.data_ptr())
            G.gw_trainer_backward(trainer, dyd.data_ptr(), dp.data_ptr())
            G.gw_trainer_status(trainer)
            grads.append(dp.cpu().numpy())
        assert np.array_equal(grads[0], grads[1])
        o = 0
        for layer, q in enumerate(t):
            a, b = [], []
            for k in synth.PARAM_ORDER:
                if k in q:
                    if k not in ("mean", "var"):
                        a.append(grads[0][o:o + q[k].numel()])
                        b.append(q[k].grad.numpy().ravel())
                    o += q[k].numel()
            assert rel_l2(np.concatenate(a), np.concatenate(b)) <= bound, layer
    finally:
        ctx.close()
