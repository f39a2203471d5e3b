"""Sizes at which a kernel's tiles, remainders or dispatch rules could go wrong, against the CPU oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import tt_synth
from paper_2402_04466_b200 import binding
from test_gpu_pipeline import _compare_frame, _frames, _make, _run_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("net,enc,stride,hidden,K", [
    ((31, 33), (8,), (1,), 4, 1),            # one channel group, map narrower than a tile, odd rows (scalar stores)
    ((129, 67), (16, 40), (2, 2), 32, 2),    # odd columns at stride 2, five groups of 8, input channels in a partial chunk
    ((66, 9), (24,), (2,), 36, 3),           # three groups, a map lower than a tile
    ((96, 64), (64,), (1,), 16, 3),          # large enough for the blocks of four channel groups
    ((200, 150), (32,), (1,), 32, 1),
    ((64, 64), (16,), (1,), 16, 1),          # small map, 32 input channels: shared out over the warps of a block
    ((40, 38), (24,), (1,), 12, 2),          # an odd number of channel groups, channels shared out by four
    ((130, 61), (8, 8), (1, 1), 20, 2),      # odd numbers of groups: shared out by two, and by nobody
    ((320, 240), (16, 32), (2, 2), 32, 3),   # eight output rows per block instead of four, the last rows of a tile empty
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


@pytest.mark.parametrize("shape", [
    dict(net_w=64, net_h=64, enc_cout=(16,), enc_stride=(1,), hidden=16),                # few warps: channels shared out
    dict(net_w=320, net_h=240, enc_cout=(16, 32), enc_stride=(2, 2), hidden=32),         # last layer shared out, cell not
    dict(net_w=158, net_h=120, enc_cout=(32, 64), enc_stride=(2, 2), hidden=64, precision="bf16"),   # bf16 model whose first layer runs here
])
def test_fp32_convolutions_give_a_stream_the_same_bits_whatever_shares_its_tick(cuda_device, shape):
    """How many warps add up a tile's channels decides the order of the sums: it must not follow from the number of streams in the tick
    or of multiprocessors left over.  Stream 0 alone against stream 0 among 2, 3, 5 and 8, and beside a reservation."""
    wl = tt_synth.workload("cfg0-gain").with_(name="neighbours", src_w=shape["net_w"] + 7, src_h=shape["net_h"] + 5, frame_kind="endoscopy", **shape)
    w = tt_synth.make_weights(wl)
    host = _frames(wl, 2, 2)
    frames = [[torch.from_numpy(f).to(cuda_device) for f in fs] for fs in host]
    runs = []
    for K, reserved in ((1, 0), (2, 0), (3, 0), (5, 0), (8, 0), (1, 60)):
        ctx = binding.Context(binding.make_config(wl, max_streams=K, reserved_sms=reserved), w)
        states = [ctx.state_create() for _ in range(K)]
        out = []
        for t in range(2):
            ctx.submit_frames([frames[min(k, 1)][t] for k in range(K)], states, frame_index=t)
            r = ctx.sync()[0]
            out += [ctx.fetch_probs(r), r["conf"]] + [ctx.debug_tensor(states[0], f"enc{l}") for l in range(len(wl.enc_cout))]
        runs.append(out + list(ctx.state_export(states[0])))
        ctx.destroy()
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("shape,K,pad", [
    (dict(src_w=214, src_h=120, net_w=160, net_h=120), 3, 5),                                    # rows not resized; odd pitch
    (dict(src_w=299, src_h=133, net_w=200, net_h=89), 3, 0),                                     # both axes down, a last tile of 4 columns and 5 rows
    (dict(src_w=203, src_h=157, net_w=132, net_h=100), 2, 64),                                   # both axes down, wide padding
    (dict(src_w=90, src_h=50, net_w=196, net_h=131, enc_stride=(1, 2, 2)), 3, 1),                # up-scaling, stride 1
    (dict(src_w=96, src_h=99, net_w=32, net_h=33, enc_cout=(64, 64), enc_stride=(1, 2)), 3, 0),  # every row on a frame row (a third), one tile wide
    (dict(src_w=960, src_h=720, enc_cout=(64, 128), enc_stride=(2, 2)), 8, 16),                  # 2400 tiles: five or six per block
])
def test_first_layer_kernel_equals_preprocessing_and_convolution_bit_for_bit(cuda_device, shape, K, pad):
    """One kernel resizes, normalises and convolves; with stage events on the two kernels it stands for run instead.  Same expressions, same
    order of products: the resized image, the first layer's map, every result and the state are the same bits, from frames with padded
    rows and from the same frames without padding."""
    wl = tt_synth.workload("cfg1-gain").with_(name="first", overlay=True, **{"hidden": 64, **shape})
    w = tt_synth.make_weights(wl)
    n = 2
    host = _frames(wl, K, n)
    runs, launches = [], []
    for separate, extra in ((False, pad), (True, pad), (False, 0)):
        cfg = binding.make_config(wl, max_streams=K)
        cfg.src_pitch = pitch = 3 * wl.src_w + extra
        ctx = binding.Context(cfg, w)
        states = [ctx.state_create() for _ in range(K)]
        ctx.set_profiling(separate)
        out = []
        for t in range(n):
            # stream k at k bytes behind an aligned address, the frame's last byte the buffer's last
            bufs = []
            for k in range(K):
                rows = np.full((wl.src_h, pitch), 201, np.uint8)
                rows[:, :3 * wl.src_w] = host[k][t].reshape(wl.src_h, -1)
                b = torch.empty(rows.size + k, dtype=torch.uint8, device=cuda_device)
                b[k:].copy_(torch.from_numpy(rows.reshape(-1)))
                bufs.append(b)
            ctx.submit_frames([bufs[k][k:] for k in range(K)], states, frame_index=t)
            res = ctx.sync()
            out += [a for i, r in enumerate(res) for a in (ctx.fetch_probs(r), ctx.fetch_masks(r), ctx.fetch_overlay(r), r["conf"], r["cx"],
                                                           ctx.debug_tensor(states[i], "pre"), ctx.debug_tensor(states[i], "enc0"))]
        if separate:
            assert ctx.get_stage_times()["preprocess"] > 0
        launches.append(ctx.get_counters()[0])
        runs.append(out + [a for s in states for a in ctx.state_export(s)])
        ctx.destroy()
    assert launches[0] == launches[2] == launches[1] - n          # one launch a tick fewer: the first layer did sample the frames itself
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("shape,K,pad", [
    (dict(src_w=640, src_h=480, net_w=320, net_h=240, enc_cout=(64, 64), enc_stride=(2, 2)), 8, 3),     # 600 tiles; 2 x 64 output channels
    (dict(src_w=420, src_h=310, net_w=200, net_h=140), 3, 7),
    (dict(src_w=402, src_h=258, net_w=100, net_h=65, enc_stride=(1, 2, 2)), 2, 1),
    (dict(src_w=400, src_h=260, net_w=100, net_h=65, enc_cout=(64, 64), enc_stride=(1, 2)), 2, 0),
])
def test_first_layer_whose_output_waits_in_the_operand_changes_no_bit(cuda_device, shape, K, pad):
    """Resize factors of 2 and more: the staged frame rows leave no room for the output beside three blocks."""
    test_first_layer_kernel_equals_preprocessing_and_convolution_bit_for_bit(cuda_device, shape, K, pad)


@pytest.mark.parametrize("net,enc,stride,hidden,K", [
    ((150, 110), (32, 128), (1, 2), 64, 2),            # 32 -> 128, 75 x 55 outputs: ragged in both directions
    ((66, 66), (64, 64), (1, 2), 64, 1),               # 64 -> 64, a last tile of one column and one row
    ((97, 131), (64, 64, 128, 128), (1, 2, 2, 2), 64, 3),   # odd inputs; 64 -> 128 resident, 128 -> 128 through the ring
    ((130, 70), (32, 64, 128, 256), (1, 2, 2, 2), 64, 2),   # 128 -> 256 through the ring
    ((128, 128), (64, 256), (2, 2), 64, 2),            # four groups of 64 resident outputs
    ((16, 12), (32, 64), (2, 2), 64, 1),               # a map smaller than one tile
])
def test_bf16_stride2_layers_at_the_edges_of_their_tiles(cuda_device, net, enc, stride, hidden, K):
    """The bounds of the other bf16 tests (_run_bf16): outputs 2e-2, intermediate maps 5e-2 of the oracle."""
    wl = tt_synth.workload("cfg1-gain").with_(name="s2", src_w=net[0] + 20, src_h=net[1] + 11, net_w=net[0], net_h=net[1], enc_cout=enc,
                                              enc_stride=stride, hidden=hidden)
    _run_bf16(cuda_device, wl, K, 2)


def test_stride2_layer_kernels_give_the_same_bits_at_small_and_large_batches(cuda_device):
    """One stream's 64 -> 128 channel layer runs as a few tiles per block on views fetched with their halo, eight streams' as many
    tiles per block with one box per tap: the same products in the same order, so a stream's maps, results and state must not
    change.  (The 32 -> 64 channel layer runs on views in both.)"""
    wl = tt_synth.workload("cfg1-gain").with_(name="s2-batch", src_w=800, src_h=500)
    K = 8
    host = [tt_synth.make_frames(wl.frame_kind, wl.stream_seed(s), 1, wl.src_w, wl.src_h)[0] for s in range(K)]
    frames = [torch.from_numpy(f).to(cuda_device) for f in host]

    def observe(ctx, st, r):
        return [ctx.debug_tensor(st, "enc1"), ctx.debug_tensor(st, "enc2"), ctx.fetch_probs(r), r["conf"], r["cx"], *ctx.state_export(st)]

    ctx, states, _ = _make(wl, K)
    ctx.submit_frames(frames, states)
    res = ctx.sync()
    batch = {k: observe(ctx, states[k], res[k]) for k in (0, 7)}
    ctx.destroy()
    for k in (0, 7):
        ctx, (st,), _ = _make(wl, 1)
        ctx.submit_frames([frames[k]], [st])
        (r,) = ctx.sync()
        for a, b in zip(batch[k], observe(ctx, st, r)):
            assert np.array_equal(a, b)
        ctx.destroy()


# groups of columns on 148, 128, 100 and 78 multiprocessors (0, 20, 48 and 70 reserved); single blocks, pairs of blocks beyond one round of units of 256
@pytest.mark.parametrize("hidden,net", [
    (64, (640, 840)),      # 70 tiles of one group of 256: cut into halves on 148, else whole
    (128, (640, 480)),     # 40 tiles x 512 columns: 192, 192 and 128, whole on 100, on pairs again 192, 192 and 128 on 78
    (128, (400, 300)),     # 21 ragged tiles x 512: halves, but 192, 192 and 128 on 78
    (256, (1280, 720)),    # 120 tiles x 1024, on pairs: several rounds of 256, the last cut into halves on 148 and 78, whole on 128 and 100
    (256, (368, 480)),     # 24 ragged tiles x 1024: five groups of 192 and one of 64 on 148 and, on pairs, on 78; whole on 128 and 100
])
def test_convlstm_column_groups_change_no_bit(cuda_device, hidden, net):
    """How many multiprocessors there are decides how the gates' columns are grouped into units, and whether these run on pairs of
    blocks: every form adds up the same products in the same order, so probabilities, confidences and state are the same bits."""
    wl = tt_synth.workload("cfg1-gain").with_(name="groups", src_w=net[0] + 30, src_h=net[1] + 20, net_w=net[0], net_h=net[1], hidden=hidden)
    host = _frames(wl, 1, 2)[0]
    w = tt_synth.make_weights(wl)
    runs = []
    for reserved in (0, 20, 48, 70):
        ctx = binding.Context(binding.make_config(wl, reserved_sms=reserved), w)
        st = ctx.state_create()
        out = []
        for t in range(2):
            ctx.submit_frames([torch.from_numpy(host[t]).to(cuda_device)], [st], frame_index=t)
            (r,) = ctx.sync()
            out += [ctx.fetch_probs(r), r["conf"]]
        runs.append(out + list(ctx.state_export(st)))
        ctx.destroy()
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("hidden,net,K", [
    (128, (400, 300), 5),     # 105 tiles: the last pair has no second tile; the second round cut into halves
    (64, (400, 300), 8),      # one group of columns
    (256, (368, 480), 3),     # 72 ragged tiles x 1024 columns: two rounds of whole groups
    (256, (368, 480), 2),     # 48: five groups of 192 and one of 64
    (512, (160, 120), 8),     # 24 tiles x 2048: ten groups of 192 and one of 128
])
def test_convlstm_on_pairs_of_blocks_changes_no_bit(cuda_device, hidden, net, K):
    """Beyond one round of units the ConvLSTM runs on pairs of blocks: every stream must get the bits it gets alone, on single blocks."""
    wl = tt_synth.workload("cfg1-gain").with_(name="pairs", src_w=net[0] + 30, src_h=net[1] + 20, net_w=net[0], net_h=net[1], hidden=hidden)
    frames = _frames(wl, K, 2)
    ctx, states, _ = _make(wl, K)
    for t in range(2):
        ctx.submit_frames([torch.from_numpy(frames[k][t]).to(cuda_device) for k in range(K)], states)
        res = ctx.sync()
    batch = [(*ctx.state_export(states[k]), ctx.fetch_probs(res[k])) for k in range(K)]
    ctx.destroy()
    ctx, (st,), _ = _make(wl, 1)
    for k in (0, K - 2, K - 1):
        ctx.state_reset(st)
        for t in range(2):
            ctx.submit_frames([torch.from_numpy(frames[k][t]).to(cuda_device)], [st])
            (r,) = ctx.sync()
        for a, b in zip(batch[k], (*ctx.state_export(st), ctx.fetch_probs(r))):
            assert np.array_equal(a, b)
    ctx.destroy()


@pytest.mark.parametrize("src,net,pad,K", [
    ((200, 150), (128, 64), 0, 1),       # one full tile column of 128
    ((200, 150), (129, 65), 3, 2),       # a tile column of one output: narrow tiles
    ((200, 150), (192, 90), 7, 3),       # half of the last wide tile: narrow tiles
    ((200, 150), (193, 90), 1, 1),       # more than half: wide tiles
    ((64, 40), (1, 1), 0, 8),
    ((1600, 900), (160, 90), 2, 2),      # ten source rows and columns per output: no tile of four rows fits
    ((2400, 1300), (40, 20), 0, 1),      # sixty: no tile fits, the kernel without staging
    ((90, 700), (300, 700), 5, 2),       # height not resized
])
def test_preprocess_at_the_edges_of_its_tiles(cuda_device, src, net, pad, K):
    """Bytes blended in fp32 by at most six roundings of values below 256, scaled to +-2: 2e-5 as in the stage tests."""
    (sw, sh), (nw, nh) = src, net
    frames = np.random.default_rng(5).integers(0, 256, (K, sh, sw, 3), dtype=np.uint8)
    buf = np.full((K, sh, 3 * sw + pad), 201, np.uint8)
    buf[:, :, :3 * sw] = frames.reshape(K, sh, 3 * sw)
    out = binding.preprocess(torch.from_numpy(buf.reshape(K, -1)).to(cuda_device), sw, sh, 3 * sw + pad, nw, nh).cpu().numpy()
    for k in range(K):
        assert np.max(np.abs(out[k] - oracle.preprocess(frames[k], nw, nh))) < 2e-5


@pytest.mark.parametrize("src,net,K", [
    ((504, 738), (224, 378), 8),         # 47.1 KB staged with wide tiles, beside 1 KB of tables
    ((534, 716), (297, 310), 8),         # ... with narrow tiles
    ((1920, 1080), (520, 292), 1),       # exactly 48 KB
    ((1280, 720), (320, 180), 1),        # tiles of four rows, the fewest that are staged ...
    ((1280, 720), (320, 180), 8),        # ... and the same frames without staging, beyond three rounds of them
    ((1280, 960), (640, 480), 4),        # two tiles of a block of different heights
])
def test_preprocess_whose_staging_takes_almost_48_kilobytes(cuda_device, src, net, K):
    """More than a kernel gets unasked, static variables included; and the largest resize factors that are staged.  Bound as above."""
    test_preprocess_at_the_edges_of_its_tiles(cuda_device, src, net, 3, K)


STAGED_SIZES = [                         # with the kernel that stages frame rows, whatever the batch (test_host_path.py asks the dispatch)
    ((40, 8), (20, 5), 0, 3),            # every thread's second column lies outside; fewer rows than runs of them
    ((300, 200), (127, 33), 1, 2),       # the second column of the last lane alone lies outside
    ((97, 61), (191, 95), 2, 8),         # narrow tiles, the last a column short; frame rows used by several output rows
    ((640, 360), (427, 241), 5, 5),      # rows that share a frame row with the one above, and rows that do not
    ((1280, 960), (1000, 562), 0, 8),    # several tiles a block, the copies of all but the first by one warp
    ((320, 240), (321, 240), 0, 8),      # the height not resized
]


@pytest.mark.parametrize("src,net,pad,K", STAGED_SIZES + [((300, 200), (64, 5), 0, 3)])     # the last: forty frame rows to an output row, none staged
def test_preprocess_of_a_frame_is_the_same_whatever_shares_its_launch(cuda_device, src, net, pad, K):
    """Tile heights, runs of rows and the blocks' shares depend on the batch; the bits of a frame do not.  Bound against the oracle as above."""
    test_preprocess_at_the_edges_of_its_tiles(cuda_device, src, net, pad, min(K, 2))
    (sw, sh), (nw, nh) = src, net
    frames = torch.from_numpy(np.random.default_rng(6).integers(0, 256, (K, sh * (3 * sw + pad)), dtype=np.uint8)).to(cuda_device)
    batch = binding.preprocess(frames, sw, sh, 3 * sw + pad, nw, nh)
    for k in range(K):
        assert torch.equal(binding.preprocess(frames[k:k + 1], sw, sh, 3 * sw + pad, nw, nh)[0], batch[k])


@pytest.mark.parametrize("from_tile", [0, 1, 2])
@pytest.mark.parametrize("src,net,pad,K", [
    ((97, 61), (191, 95), 2, 8),         # one tile a block
    ((1920, 1080), (1279, 717), 1, 4),   # two or three
    ((854, 720), (1216, 720), 3, 8),     # five or six narrow ones, the height not resized
])
def test_preprocess_whose_waits_run_out_still_makes_the_whole_image(cuda_device, src, net, pad, K, from_tile):
    """Behind a wait that gave up (here at once, the rows on their way) a block takes the rest of its tiles from memory: every float, the same bits."""
    (sw, sh), (nw, nh) = src, net
    frames = torch.from_numpy(np.random.default_rng(8).integers(0, 256, (K, sh * (3 * sw + pad)), dtype=np.uint8)).to(cuda_device)
    whole = binding.preprocess(frames, sw, sh, 3 * sw + pad, nw, nh)
    got = torch.full_like(whole, float("nan"))
    assert binding.load_library().tt_debug_preprocess_expired(frames.data_ptr(), K, frames.stride(0), sw, sh, 3 * sw + pad, got.data_ptr(), nw, nh,
                                                              255.0, 0.5, 0.25, from_tile, None) == 0
    torch.cuda.synchronize()
    assert torch.equal(got, whole)


_TWO_CONTEXTS = """
import ctypes as C, sys
import numpy as np
from paper_2402_04466_b200 import binding
cu, lib = C.CDLL("libcuda.so.1"), binding.load_library()
def do(name, *args):
    assert getattr(cu, name)(*args) == 0, name
def alloc(n):
    p = C.c_void_p()
    do("cuMemAlloc_v2", C.byref(p), C.c_size_t(n))
    return p
frame, out = np.random.default_rng(9).integers(0, 256, 1920 * 1080 * 3, dtype=np.uint8), []
def stage():
    src, dst, got = alloc(frame.size), alloc(3 * 520 * 292 * 4), np.zeros(3 * 520 * 292, np.float32)
    do("cuMemcpyHtoD_v2", src, frame.ctypes.data_as(C.c_void_p), C.c_size_t(frame.size))
    for _ in range(2):
        assert lib.tt_preprocess(src, 1, 0, 1920, 1080, 3 * 1920, dst, 520, 292, 255.0, 0.5, 0.25, None) == 0, lib.tt_last_error(None)
    do("cuCtxSynchronize")
    do("cuMemcpyDtoH_v2", got.ctypes.data_as(C.c_void_p), dst, C.c_size_t(got.nbytes))
    out.append(got)
do("cuInit", 0)
dev, first, second, popped = C.c_int(), C.c_void_p(), C.c_void_p(), C.c_void_p()
do("cuDeviceGet", C.byref(dev), 0)
do("cuDevicePrimaryCtxRetain", C.byref(first), dev)
do("cuCtxPushCurrent_v2", first)
stage()
do("cuCtxCreate_v2", C.byref(second), 0, dev)
stage()
do("cuCtxPopCurrent_v2", C.byref(popped))
stage()
assert out[0].any() and all(np.array_equal(out[0], x) for x in out[1:])
print("three alike")
"""


def test_calls_in_a_second_context_of_the_device(cuda_device):
    """More shared memory than a kernel gets unasked, in a context of its own that knows nothing of what the first one's kernels were given."""
    r = subprocess.run([sys.executable, "-c", _TWO_CONTEXTS], capture_output=True, text=True, timeout=240, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and "three alike" in r.stdout, r.stderr[-2000:]


@pytest.mark.parametrize("shape,K", [
    (dict(src_w=854, src_h=480, net_w=640, net_h=480, hidden=128), 5),                        # parts of 2 and 3 streams
    (dict(src_w=854, src_h=480, net_w=642, net_h=480, hidden=128), 6),                        # parts of 3; first layer on the fp32 kernel
    (dict(src_w=854, src_h=480, net_w=320, net_h=240, hidden=32, enc_cout=(16, 32), enc_stride=(2, 2), precision="fp32"), 6),
])
def test_a_tick_of_host_frames_in_parts_changes_nothing(cuda_device, shape, K):
    """Streams of large host frames are launched in parts as their frames arrive: results, maps, overlay, intermediate tensors and state
    are those of the same frames on the device, whose tick is not cut, and a tick counts once.  The middle stream's frame is on the device."""
    wl = tt_synth.workload("cfg1-gain").with_(name="parts", overlay=True, **shape)
    w = tt_synth.make_weights(wl)
    frames = _frames(wl, K, 3)
    runs, launches = [], []
    for host in (True, False):
        ctx = binding.Context(binding.make_config(wl, max_streams=K), w)
        states = [ctx.state_create() for _ in range(K)]
        out = []
        for t in range(3):
            fr = [torch.from_numpy(frames[k][t]) for k in range(K)]
            fr = [f.pin_memory() if host and k != K // 2 else f.to(cuda_device) for k, f in enumerate(fr)]
            before = ctx.get_counters()[0]
            ctx.submit_frames(fr, states, frame_index=t)
            res = ctx.sync()
            launches.append(ctx.get_counters()[0] - before)
            for k in range(K):
                out += [res[k][n] for n in ("conf", "cx", "cy", "count")] + [ctx.fetch_probs(res[k]), ctx.fetch_masks(res[k]), ctx.fetch_overlay(res[k])]
                out += [ctx.debug_tensor(states[k], n) for n in ["pre", "prob"] + [f"enc{l}" for l in range(len(wl.enc_cout))]]
        if wl.recurrent:
            for k in range(K):
                out += list(ctx.state_export(states[k]))
        assert ctx.get_counters()[1] == 3
        runs.append(out)
        ctx.destroy()
    assert launches[0] == launches[2] >= 2 * launches[3]        # the host ticks were cut
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("conf_mode", ["mean_sigmoid", "gap_linear"])
@pytest.mark.parametrize("K,ch,hm,wm,T", [
    (1, 4, 1, 1, 1),         # one pixel, four channels, one tool
    (2, 20, 9, 15, 8),       # 135 pixels: a second block of seven; channels in a partial chunk
    (3, 16, 8, 16, 5),       # one full block
    (8, 36, 16, 20, 7),      # ten full warps
    (2, 512, 13, 10, 3),     # widest state
])
def test_heads_of_a_planar_state_at_the_edges_of_their_blocks(cuda_device, K, ch, hm, wm, T, conf_mode):
    """fp32 sums of up to 512 products and fixed-point sums of 2^-30 against the oracle's double sums: 1e-4 as in the stage tests; sizes and
    centroids exactly those of the mask.  The second call finds the accumulators zeroed."""
    rng = np.random.default_rng(9)
    h = (rng.standard_normal((K, ch, hm, wm)) * 0.5).astype(np.float32)
    hw, cw = ((rng.standard_normal((T, ch)) * 2 / np.sqrt(ch)).astype(np.float32) for _ in range(2))
    hb, cb = ((rng.standard_normal(T) * 0.3).astype(np.float32) for _ in range(2))
    dev = [torch.from_numpy(a).to(cuda_device) for a in (hw, hb, cw, cb)]
    out = binding.postprocess(torch.from_numpy(h).to(cuda_device), False, *dev, conf_mode)
    again = binding.postprocess(torch.from_numpy(h).to(cuda_device), False, *dev, conf_mode)
    for k in range(K):
        z, p, m = oracle.head(h[k], hw, hb, 0.5)
        got = {n: out[n][k].cpu().numpy() for n in ("logits", "probs", "masks")}
        assert np.max(np.abs(got["logits"] - z)) < 1e-4 and np.max(np.abs(got["probs"] - p)) < 1e-4
        assert np.array_equal(got["masks"] != 0, got["logits"] > 0)
        r = out["results"][k]
        conf = oracle.conf_mean_sigmoid(p) if conf_mode == "mean_sigmoid" else oracle.conf_gap_linear(h[k], cw, cb)
        assert np.max(np.abs(r["conf"] - conf)) < 1e-4
        cx, cy, n = oracle.centroids(got["masks"])
        assert np.array_equal(r["count"], n) and np.array_equal(r["cx"], cx) and np.array_equal(r["cy"], cy)
        for f in ("conf", "cx", "cy", "count"):
            assert np.array_equal(r[f], again["results"][k][f])
