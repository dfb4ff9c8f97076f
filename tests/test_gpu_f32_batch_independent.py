"""FP32 results do not depend on how many items share a launch: a server's batch
is the bucket of a tick, which follows from arrival times.  Batches and lengths
on both sides of the FP32 conv's changes of tile, one window or segment alone
against the same one among others, bit for bit; and streams served alone and in
ticks of several buckets at the serving configuration's sizes."""
import numpy as np
import pytest
import torch

from paper_2108_12430_gb300 import gwstream as G, synth
from tests.gpu_util import Ctx, dev
from tests.test_gpu_serve import Rig

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = Ctx()
    yield c
    c.close()


@pytest.mark.parametrize("length", [40, 1016, 4096, 32768])
def test_deepclean_window(ctx, length):
    step, most = 64, 64
    x = dev(np.random.default_rng(length).standard_normal((21, length + (most - 1) * step)))
    m = ctx.deepclean(2)

    def run(first, n):
        y = torch.full((n, length), float("nan"), device="cuda")
        G.gw_deepclean_forward(m, x.data_ptr() + 4 * step * first, x.shape[1], step, n, length, y.data_ptr())
        torch.cuda.synchronize()
        return y.cpu().numpy()

    alone = {w: run(w, 1)[0] for w in (0, 1, 2, 7, most - 1)}
    for n in (2, 3, 8, 20, most):
        y = run(0, n)
        for w, ref in alone.items():
            if w < n:
                assert np.array_equal(y[w], ref), (n, w)


@pytest.mark.parametrize("length", [48, 512, 2048])
def test_bbhnet_segment(ctx, length):
    x = dev(np.random.default_rng(length).standard_normal((200, 2, length)))
    m = ctx.bbhnet(4)

    def run(first, n):
        out = torch.full((n,), float("nan"), device="cuda")
        G.gw_bbhnet_score(m, x[first].data_ptr(), n, length, out.data_ptr())
        torch.cuda.synchronize()
        return out.cpu().numpy()

    alone = {i: run(i, 1)[0] for i in (0, 1, 3, 15, 63, 199)}
    for n in (2, 4, 16, 48, 64, 200):
        out = run(0, n)
        for i, ref in alone.items():
            if i < n:
                assert out[i] == ref, (n, i)


@pytest.mark.parametrize("length", [136, 8192])
def test_training_prediction(ctx, length):
    most = 32
    x = dev(np.random.default_rng(length).standard_normal((most, 21, length)))
    p = dev(synth.flatten_params(synth.deepclean_params(3)))
    t = G.gw_trainer_create(ctx.h, 21, most, length)
    ctx.objs.append((G.gw_trainer_destroy, t))

    def run(first, n):
        y = torch.full((n, length), float("nan"), device="cuda")
        G.gw_trainer_forward(t, p.data_ptr(), x[first].data_ptr(), n, y.data_ptr())
        torch.cuda.synchronize()
        return y.cpu().numpy()

    alone = {i: run(i, 1)[0] for i in (0, 2, most - 1)}
    for n in (3, 8, most):
        y = run(0, n)
        for i, ref in alone.items():
            if i < n:
                assert np.array_equal(y[i], ref), (n, i)


@pytest.mark.parametrize("max_batch", [2, 4, 8, 64])
def test_serving_alone_and_in_the_mix(gpu_lib, max_batch):
    ctx = Ctx()
    try:
        kw = dict(W=32768, delta=0, Lb=2048, Kh=2049, nfft=8192, out_scale=1e-2)
        seeds = [(100 + 11 * i, S, 5) for i, S in enumerate((512, 512, 256, 128))]
        alone = Rig(ctx, G.GW_FP32, max_batch=1, **kw).run(seeds, [i for _ in range(5) for i in range(4)])
        streams = [seeds[i % 4] for i in range(max_batch)]
        rig = Rig(ctx, G.GW_FP32, max_streams=max_batch, max_batch=max_batch, max_wait_us=20000,
                  max_pending=5 * max_batch, **kw)
        got = rig.run(streams, [i for _ in range(5) for i in range(max_batch)])
        for i, (clean, logit) in enumerate(got):
            assert np.array_equal(clean, alone[i % 4][0]) and np.array_equal(logit, alone[i % 4][1])
    finally:
        ctx.close()
