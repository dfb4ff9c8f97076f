"""Tensor-core conv epilogues at ragged sizes: lengths that end inside a row of
folded positions and inside a 128-row tile, few and many items, for each kind of
output (BF16 rows with and without a residual, e4m3, the training path's FP32
planes with the blocked copy).  References: the FP64 oracle, for e4m3 the same
network with every stored tensor rounded to e4m3 (noise inputs of a few hundred
samples leave little to average, so the format's own error against the exact
network exceeds the bound, 0.29 at 272 samples), and PyTorch float64 autograd;
bounds: BBHnet logits within 0.05 (BF16) and 0.25 (FP8) absolute, training
prediction rel-L2 2e-2 and gradients 4e-2 per layer."""
import numpy as np
import pytest
import torch

from oracle import layers as olayers, nets, quant
from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev, rel_l2
from tests.test_gpu_wgrad_f32_tiles import torch_forward

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx(gpu_lib):
    c = Ctx()
    yield c
    c.close()


def e4m3_forward(x, params, head, scales):
    """BBHnet with e4m3 storage (scales: n_layers + 1, the order of
    gw_model_calibrate) and FP64 accumulation; the stem on BF16 operands."""
    specs, s = synth.bbhnet_layers(), [float(v) for v in scales]

    def conv(h, i, rounded):
        _, _, _, _, stride, left, right, *_ = specs[i]
        p = params[i]
        w, b = olayers.fold_bn(p["w"], p["b"], p["gamma"], p["beta"], p["mean"], p["var"])
        if rounded:
            scale = np.float32(np.abs(w).max(axis=(1, 2), keepdims=True) / 448.0).astype(np.float64)
            w = quant.to_e4m3(np.float32(w / scale)) * scale
        else:
            w = quant.to_bf16(w)
        return olayers.conv1d(h, w, np.float32(b), stride, left, right)

    store = lambda v, scale: quant.to_e4m3(np.float32(v * scale)) / scale  # noqa: E731
    h = store(np.maximum(conv(quant.to_bf16(x), 0, False), 0.0), s[1])
    for blk in range(4):
        i, out = 1 + 3 * blk, s[4 + 3 * blk]
        a = store(np.maximum(conv(h, i, True), 0.0), s[i + 1])
        shortcut = store(conv(h, i + 2, True), out)
        h = store(np.maximum(conv(a, i + 1, True) + shortcut, 0.0), out)
    return olayers.linear(olayers.global_avg_pool(h), head["w"], head["b"])


@pytest.mark.parametrize("precision,bound", [(G.GW_BF16, 0.05), (G.GW_FP8, 0.25)])
@pytest.mark.parametrize("batch,length", [(1, 16), (3, 48), (5, 208), (33, 272), (2, 4112), (180, 1040)])
def test_bbhnet_ragged(ctx, precision, bound, batch, length):
    x = np.random.default_rng(length + batch).standard_normal((batch, 2, length)).astype(np.float32)
    xd = dev(x)
    m = ctx.bbhnet(4, precision)
    if precision == G.GW_FP8:
        scales = G.gw_model_calibrate(m, xd.data_ptr(), batch, length)
    out = torch.full((batch,), float("nan"), device="cuda")
    G.gw_bbhnet_score(m, xd.data_ptr(), batch, length, out.data_ptr())
    G.gw_model_status(m)
    some = sorted({0, batch // 2, batch - 1})
    layers, head = synth.bbhnet_params(4)
    if precision == G.GW_FP8:
        ref = e4m3_forward(x[some].astype(np.float64), layers, head, scales)
    else:
        ref = nets.bbhnet_forward(x[some].astype(np.float64), layers, head, synth.bbhnet_layers())
    assert np.abs(out.cpu().numpy()[some] - ref).max() <= bound


@pytest.mark.parametrize("batch,length,checkpoint", [(1, 16, 0), (3, 136, 0), (2, 1032, 1), (7, 2056, 0)])
def test_training_ragged(ctx, batch, length, checkpoint):
    rng = np.random.default_rng(batch + length)
    params = synth.deepclean_params(3)
    x = rng.standard_normal((batch, 21, length)).astype(np.float32)
    dy = rng.standard_normal((batch, length)).astype(np.float32)
    t = [{k: torch.from_numpy(np.asarray(v, np.float64)).requires_grad_(k not in ("mean", "var")) for k, v in p.items()}
         for p in params]
    y = torch_forward(torch.from_numpy(x.astype(np.float64)), t)
    y.backward(torch.from_numpy(dy.astype(np.float64)))
    trainer = G.gw_trainer_create(ctx.h, 21, batch, length, checkpoint, precision=G.GW_BF16, tc_data=1)
    ctx.objs.append((G.gw_trainer_destroy, trainer))
    p, xd, dyd = dev(synth.flatten_params(params)), dev(x), dev(dy)
    yd, dp = torch.full((batch, length), float("nan"), device="cuda"), torch.full_like(p, float("nan"))
    G.gw_trainer_forward(trainer, p.data_ptr(), xd.data_ptr(), batch, yd.data_ptr())
    G.gw_trainer_backward(trainer, dyd.data_ptr(), dp.data_ptr())
    G.gw_trainer_status(trainer)
    assert rel_l2(yd.cpu().numpy(), y.detach().numpy()) <= 2e-2
    got, o = dp.cpu().numpy(), 0
    for layer, q in enumerate(t):
        a, b = [], []
        for k in synth.PARAM_ORDER:
            if k in q:
                if k not in ("mean", "var"):
                    a.append(got[o:o + q[k].numel()])
                    b.append(q[k].grad.numpy().ravel())
                o += q[k].numel()
        assert rel_l2(np.concatenate(a), np.concatenate(b)) <= 4e-2, layer
