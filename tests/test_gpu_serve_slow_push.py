"""Serving ticks whose ring update is slow beside the network.

The whole-network DeepClean kernel starts under the ring update and computes
the tiles that read only older samples; its last epilogue of a CTA's first
item then waits for the update (which reads pinned host memory) while the
slot's next item is already in the tensor cores.  64 streams of stride 1024
make the update long and give every CTA several items per slot.  Results have
to be the ones of the same streams served one at a time, bit for bit.
"""
import numpy as np
import pytest

from paper_2108_12430_gb300 import gwstream as G
from tests.gpu_util import Ctx
from tests.test_gpu_serve import Rig

pytestmark = pytest.mark.gpu
W, S, N, STREAMS = 32768, 1024, 4, 64


@pytest.mark.parametrize("max_batch", [48, 64])
def test_slow_ring_update_under_the_network(gpu_lib, max_batch):
    ctx = Ctx()
    try:
        kw = dict(W=W, max_stride=S, delta=0, Lb=2048, Kh=2049, nfft=8192, out_scale=1e-2)
        seeds = [(100 + 11 * i, S, N) for i in range(4)]
        alone = Rig(ctx, G.GW_BF16, max_batch=1, **kw).run(seeds, [i for _ in range(N) for i in range(4)])
        streams = [seeds[i % 4] for i in range(STREAMS)]
        rig = Rig(ctx, G.GW_BF16, max_streams=STREAMS, max_batch=max_batch, max_wait_us=20000, max_pending=N * STREAMS,
                  **kw)
        for _ in range(5):
            got = rig.run(streams, [i for _ in range(N) for i in range(STREAMS)])
            for i, (clean, logit) in enumerate(got):
                assert np.array_equal(clean, alone[i % 4][0]) and np.array_equal(logit, alone[i % 4][1])
    finally:
        ctx.close()
