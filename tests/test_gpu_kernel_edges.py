"""Sizes at which a kernel's tiles, remainders or dispatch rules could go wrong, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
import tt_synth
from test_gpu_pipeline import _compare_frame, _frames, _make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("net,enc,stride,hidden,K", [
    ((31, 33), (8,), (1,), 4, 1),            # one channel group, map narrower than a tile, odd rows (scalar stores)
    ((129, 67), (16, 40), (2, 2), 32, 2),    # odd columns at stride 2, five groups of 8, input channels in a partial chunk
    ((66, 9), (24,), (2,), 36, 3),           # three groups, a map lower than a tile
    ((96, 64), (64,), (1,), 16, 3),          # large enough for the blocks of four channel groups
    ((200, 150), (32,), (1,), 32, 1),
    ((64, 64), (16,), (1,), 16, 1),          # small map, 32 input channels: shared out over the warps of a block
])
def test_fp32_convolutions_at_the_edges_of_their_tiles(cuda_device, net, enc, stride, hidden, K):
    """Bound as for the other fp32 tests: fp32 sums of up to 9 * 72 products against the oracle's double sums, 1e-4."""
    wl = tt_synth.workload("cfg0-gain").with_(name="fp32-edges", src_w=net[0] + 7, src_h=net[1] + 5, net_w=net[0], net_h=net[1], enc_cout=enc,
                                              enc_stride=stride, hidden=hidden, n_tools=3, frame_kind="endoscopy")
    ctx, states, w = _make(wl, K)
    oras = [oracle.OraclePipeline(wl, w) for _ in range(K)]
    frames = _frames(wl, K, 2)
    for t in range(2):
        ctx.submit_frames([torch.from_numpy(frames[k][t]).to(cuda_device) for k in range(K)], states, frame_index=t)
        res = ctx.sync()
        for k in range(K):
            _compare_frame(ctx, states[k], res[k], oras[k].step(frames[k][t]), 1e-4, 1e-3, tag=f"edges k={k} t={t}")
    ctx.destroy()
