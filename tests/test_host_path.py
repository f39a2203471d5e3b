"""Host code of tt_submit_frames against a CUDA runtime that only writes down what it is asked for (no GPU needed)."""
import ctypes as C
import glob
import os
import random
import re
import subprocess

import numpy as np
import pytest

import tt_synth
from paper_2402_04466_b200 import binding
from paper_2402_04466_b200 import build as build_mod
from test_gpu_kernel_edges import STAGED_SIZES

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    """The library's own objects, linked with fake_cudart.c in the place of the CUDA runtime."""
    build_mod.build()
    objs = sorted(glob.glob(os.path.join(build_mod.OBJ_DIR, "*.o")))
    if not objs:                      # a checkout that came with the library alone
        build_mod.build(force=True)
        objs = sorted(glob.glob(os.path.join(build_mod.OBJ_DIR, "*.o")))
    d = tmp_path_factory.mktemp("fake")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build_mod._nvcc()))), "include")
    subprocess.run(["gcc", "-O1", "-fPIC", "-I", include, "-c", os.path.join(HERE, "fake_cudart.c"), "-o", str(d / "fake.o")], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", str(d / "libtt_fake.so"), *objs, str(d / "fake.o")], check=True)
    return str(d / "libtt_fake.so")


@pytest.fixture
def fake(fake_path, monkeypatch):
    monkeypatch.setattr(binding, "_LIB", None)
    monkeypatch.setattr(binding, "LIB_PATH", fake_path)
    lib = binding.load_library(build_if_missing=False)
    lib.fake_log.restype = C.c_char_p
    lib.fake_fail.argtypes = [C.c_char_p, C.c_int]
    lib.fake_pinned.argtypes = [C.c_void_p, C.c_size_t]
    lib.fake_reset()
    return lib


# copies of 124 us and 31 us of operations a stream, by the estimate: a tick of host frames runs in parts of one stream
WORKLOAD = dict(src_w=1920, src_h=1080, net_w=320, net_h=240, enc_cout=(16, 32), enc_stride=(2, 2), hidden=32, n_tools=3)


class Streams:
    """A context of K streams, each with a frame in pinned host memory of its own."""

    def __init__(self, lib, K, pad=0, workload=WORKLOAD, **options):
        wl = tt_synth.workload("cfg0-gain").with_(name="host-path", **workload)
        cfg = binding.make_config(wl, max_streams=K, **options)
        cfg.src_pitch = 3 * wl.src_w + pad
        self.lib, self.K, self.wl, self.bytes = lib, K, wl, wl.src_h * cfg.src_pitch
        self.ctx = binding.Context(cfg, tt_synth.make_weights(wl))
        self.states = [self.ctx.state_create() for _ in range(K)]
        self.frames = [np.full(self.bytes, 10 + k, np.uint8) for k in range(K)]
        for f in self.frames:
            lib.fake_pinned(f.ctypes.data, f.size)
        self.addr = [f.ctypes.data for f in self.frames]

    def submit(self, on_device=()):
        """Status and log of one tt_submit_frames."""
        fr = (binding.tt_frame * self.K)()
        for k in range(self.K):
            fr[k].data, fr[k].on_device = self.addr[k], int(k in on_device)
        status = self.ctx.submit_raw(self.K, fr, (C.c_void_p * self.K)(*[s.value for s in self.states]))
        log = self.lib.fake_log().decode().splitlines()
        self.lib.fake_reset()
        return status, log

    def sync(self):
        self.ctx.sync()
        self.lib.fake_reset()

    def mark(self):
        """Puts a value of its own into every stream's state: a stream that has taken a frame shows the other half of h, which holds another."""
        self.base = getattr(self, "base", 0.0) + 100.0
        for k, s in enumerate(self.states):
            x = np.full((self.wl.hidden, self.ctx.hm, self.ctx.wm), self.base + k, np.float32)
            self.ctx.state_import(s, x, x)
        self.lib.fake_reset()

    def advanced(self):
        return [k for k, s in enumerate(self.states) if self.ctx.state_export(s)[0].flat[0] != self.base + k]


def _first(log, *words):
    return next((i for i, line in enumerate(log) if line.startswith(words)), len(log))


def _copies(log):
    """[(from, bytes, to)] of the copies into device memory, pointer tables apart."""
    found = [re.match(r"copy in (\d+) from (0x\w+) to (0x\w+)", line) for line in log]
    return [(int(m[2], 16), int(m[1]), int(m[3], 16)) for m in found if m and int(m[1]) != 8 * binding.TT_MAX_STREAMS]


@pytest.mark.parametrize("warm", [0, 8])
@pytest.mark.parametrize("nth", [1, 2, 4])
def test_a_frame_that_cannot_be_copied_leaves_every_stream_as_it_was(fake, nth, warm):
    """A tick in parts launches nothing before all of its frames have been accepted, neither plainly nor from graphs."""
    s = Streams(fake, 4)
    for _ in range(warm):
        assert s.submit()[0] == binding.TT_OK
        s.sync()
    s.mark()
    fake.fake_fail(b"cudaMemcpyAsync", nth)
    status, log = s.submit()
    assert status == 4 and "failed cudaMemcpyAsync" in log       # TT_ERR_CUDA
    assert _first(log, "launch", "replay", "capture") == len(log) and log.count("drain") == 2
    assert "no stream has taken its frame" in s.ctx.last_error() and "cudaMemcpyAsync" in s.ctx.last_error()
    assert s.advanced() == []
    fake.fake_reset()
    status, log = s.submit()                                     # the caller tries again
    assert status == binding.TT_OK and [c[0] for c in _copies(log)] == s.addr
    last_copy = max(i for i, line in enumerate(log) if line.startswith("copy in") and " 64 " not in line)
    assert last_copy < _first(log, "launch", "replay", "capture")
    assert sum(line.startswith("wait") for line in log) == 4     # ... and was cut into four parts
    s.sync()
    assert s.advanced() == [0, 1, 2, 3]


@pytest.mark.parametrize("call,nth,taken", [
    ("cudaGraphLaunch", 1, 0), ("cudaGraphLaunch", 3, 2), ("cudaStreamWaitEvent", 2, 1), ("cudaEventRecord", 6, 4),   # the tick's last event
    ("cudaLaunchKernel", 5 + 3, 1),       # an encoder layer of the second part
    ("cudaLaunchKernel", 5 + 4, 1),       # its recurrent step
    ("cudaLaunchKernel", 5 + 5, 2),       # the heads behind it
])
def test_a_launch_that_fails_leaves_every_stream_before_or_behind_its_frame(fake, call, nth, taken):
    """Streams whose recurrent step had been enqueued have taken their frame, the others have not, the error names them, and nothing is left in
    flight: the next submit works on either."""
    s = Streams(fake, 4, plain_launches=call == "cudaLaunchKernel")
    for _ in range(8):
        assert s.submit()[0] == binding.TT_OK
        s.sync()
    s.mark()
    fake.fake_fail(call.encode(), nth)
    status, log = s.submit()
    assert status == 4 and f"failed {call}" in log and log[-2:] == ["drain", "drain"]
    error = s.ctx.last_error()
    assert (f"frames[0..{taken - 1}] have taken" if taken else "no stream has taken") in error
    assert s.advanced() == list(range(taken))
    with pytest.raises(binding.TTError):
        s.ctx.debug_tensor(s.states[0], "prob")                  # no completed submit's
    assert s.ctx.query() is False                                # nothing in flight
    s.mark()
    fake.fake_reset()
    assert s.submit()[0] == binding.TT_OK
    s.sync()
    assert s.advanced() == [0, 1, 2, 3]


@pytest.mark.parametrize("src,net,cout,stride", [
    ((854, 480), (640, 480), 32, 2), ((1920, 1080), (1280, 720), 64, 2),       # memory of its own for the output
    ((1920, 1080), (960, 540), 64, 2), ((1280, 960), (640, 480), 64, 2),       # twice the network's size
    ((1920, 1080), (856, 480), 32, 2), ((1920, 1080), (800, 448), 64, 2),
    ((1280, 720), (320, 180), 32, 1), ((1280, 720), (320, 180), 64, 1),
    ((1920, 1080), (768, 432), 64, 2),                                         # almost as much staging as the kernel takes
])
def test_the_first_layers_blocks_fit_and_its_grid_is_theirs(fake, src, net, cout, stride):
    """Three blocks to a multiprocessor unless the frame rows under their patches alone leave room for two, and as many blocks as fit at once."""
    w = dict(src_w=src[0], src_h=src[1], net_w=net[0], net_h=net[1], enc_cout=(cout, 64), enc_stride=(stride, 2), hidden=64, n_tools=3, precision="bf16")
    s = Streams(fake, 2, workload=w)
    log = s.submit(on_device=(0, 1))[1]
    (m,) = [m for m in (re.match(r"launch \S*conv_first_fused_kernelILi(\d+)ELi(\d)E(?:Lb([01])E)?\S* grid (\d+) 1 1 smem (\d+)", line) for line in log) if m]
    assert (int(m[1]), int(m[2])) == (cout, stride)
    own, grid, smem = int(m[3] or 1), int(m[4]), int(m[5])
    least = smem - own * 8 * 2048
    fits, could = (min(3, 228 * 1024 // (b + 2048)) for b in (smem, least))
    assert fits == could and (own or min(3, 228 * 1024 // (least + 8 * 2048 + 2048)) < could)
    assert could == 3 or least + 2048 > 228 * 1024 // 3
    ho, wo = ((n - 1) // stride + 1 for n in (net[1], net[0]))
    assert grid == min(2 * ((wo + 31) // 32) * ((ho + 7) // 8), fits * 148)
    s.sync()


def _parts(log):
    """Launch sequences of a tick that ran plainly: each begins with the resize (or the first layer that contains it)."""
    return sum(bool(re.match(r"launch \S*(preprocess|conv_first_fused)", line)) for line in log)


@pytest.mark.parametrize("on_device,parts", [
    ((), 8),                                  # 8 x (124 + 31) us one behind the other, or compute under the copies
    ((0, 1, 2, 3, 4, 5, 6), 2),               # one copy of 124 us, under 45 + 4 x 31 us of the first part
    ((0, 1, 2, 4, 5, 6, 7), 2),
    ((1, 2, 3, 4, 5, 6, 7), 1),               # nothing to compute before it has arrived
    ((0, 1, 2, 3, 4, 5, 6, 7), 1),
])
def test_a_tick_is_cut_by_the_frames_that_have_to_be_copied(fake, on_device, parts):
    """Frames that are on the device already do not arrive one behind the other."""
    s = Streams(fake, 8, plain_launches=True)
    status, log = s.submit(on_device)
    assert status == binding.TT_OK and _parts(log) == parts and len(_copies(log)) == 8 - len(on_device)
    s.sync()


@pytest.mark.parametrize("src,on_device,shift", [
    ((1917, 1081), (1,), 0),               # an aligned device frame whose overlay begins between 16-byte boundaries, in a part of its own
    ((1917, 1081), (1,), 1),
    ((1918, 1081), (), 0),
])
def test_no_kernel_runs_for_the_first_time_inside_a_capture(fake, src, on_device, shift):
    """Neither a tick nor a part of one is captured with a variant that has not run plainly before."""
    s = Streams(fake, 4, workload=dict(WORKLOAD, src_w=src[0], src_h=src[1]), overlay=True)
    for k in on_device:
        s.addr[k] += shift - s.addr[k] % 4
        fake.fake_pinned(s.addr[k], s.bytes)
    ran, captured = set(), set()
    for _ in range(9):
        status, log = s.submit(on_device)
        assert status == binding.TT_OK
        for line in log:
            if line.startswith("launch"):
                ran.add(line.split()[1])
            if line.startswith("capture"):
                assert line.split()[1] in ran
                captured.add(line.split()[1])
        s.sync()
    assert any("overlay_kernel" in k for k in captured)
    assert len([k for k in ran if "overlay_kernel" in k]) == 2      # word by word where frames and output allow it, byte by byte elsewhere


@pytest.mark.parametrize("K,pad,layout,on_device,expected", [
    (3, 0, "one", (), [(0, 3)]),                     # one buffer: one copy
    (3, 10, "one", (), [(0, 3)]),                    # rows padded to another pitch
    (4, 0, "one", (2,), [(0, 2), (3, 1)]),           # a frame in between that is on the device
    (3, 0, "gap", (), [(0, 1), (1, 1), (2, 1)]),     # 64 bytes between the frames
    (3, 0, "backwards", (), [(0, 1), (1, 1), (2, 1)]),
    (3, 0, "neighbours", (), [(0, 2), (2, 1)]),      # two page-locked ranges, one right behind the other
    (3, 0, "pageable", (), [(0, 1), (1, 1), (2, 1)]),
])
@pytest.mark.parametrize("cut", [False, True])
def test_frames_that_lie_one_behind_the_other_travel_as_one_copy(fake, K, pad, layout, on_device, expected, cut):
    """Every frame arrives in its place of the staging buffer, whatever travels together; no copy reaches over the edge of a part or out of a
    page-locked range, and none takes a frame that is on the device."""
    small = dict(WORKLOAD, src_w=340, src_h=250)
    s = Streams(fake, K, pad=pad, workload=WORKLOAD if cut else small, plain_launches=True)     # cut: parts of one stream
    fake.fake_unpin()
    step = s.bytes + (64 if layout == "gap" else 0)
    buf = np.repeat(np.arange(1, K + 1, dtype=np.uint8), step)
    base = buf.ctypes.data
    if layout == "neighbours":
        fake.fake_pinned(base, 2 * step)
        fake.fake_pinned(base + 2 * step, step)
    elif layout != "pageable":
        fake.fake_pinned(base, buf.size)
    order = range(K)[::-1] if layout == "backwards" else range(K)
    s.addr = [base + i * step for i in order]
    status, log = s.submit(on_device)
    assert status == binding.TT_OK
    assert _parts(log) == (K if cut else 1)
    copies = _copies(log)
    staging = copies[0][2] - next(n for n in range(K) if n not in on_device) * s.bytes
    got = [((to - staging) // s.bytes, size // s.bytes) for _, size, to in copies]
    assert all((to - staging) % s.bytes == 0 and size % s.bytes == 0 for _, size, to in copies)
    if cut:
        assert got == [(n, 1) for n in range(K) if n not in on_device]
    else:
        assert got == expected
    for n in range(K):
        if n not in on_device:
            staged = np.ctypeslib.as_array((C.c_uint8 * s.bytes).from_address(staging + n * s.bytes))
            assert np.array_equal(staged, buf[order[n] * step:order[n] * step + s.bytes])
    s.sync()


def test_preprocessing_is_refused_at_no_size(fake):
    """However the tile and its staging come out, the launch asks for the shared memory that it takes."""
    rng, at = random.Random(3), 0x7F0000000000        # addresses that nothing reads
    sizes = [(1920, 1080, 520, 292, 1), (504, 738, 224, 378, 8), (534, 716, 297, 310, 8)]
    for _ in range(1500):
        nw, nh = rng.randint(16, 1280), rng.randint(16, 960)
        sizes.append((max(2, int(nw * rng.uniform(0.3, 4.0))), max(2, int(nh * rng.uniform(0.3, 4.0))), nw, nh, rng.randint(1, 8)))
    for sw, sh, nw, nh, K in sizes:
        fake.fake_reset()
        assert fake.tt_preprocess(at, K, 3 * sw * sh, sw, sh, 3 * sw, at + 0x10000000, nw, nh, 255.0, 0.5, 0.25, None) == 0, (sw, sh, nw, nh, K)
        assert b"launch" in fake.fake_log()


@pytest.mark.parametrize("src,net,K,cols,smem", [                  # smem: two tiles of staged rows x bytes a row; 0: taps straight from memory
    ((1920, 1080), (1280, 720), 4, 128, 2 * 41 * 640),             # 26 output rows a tile
    ((1280, 960), (640, 480), 4, 128, 2 * 30 * 832),               # 14, where rounds of tiles alone would have 6 or 10
    ((320, 240), (1280, 960), 1, 128, 2 * 8 * 160),                # 22 instead of 18
    ((1920, 1080), (640, 360), 8, 128, 2 * 20 * 1216),             # 6, the fewest at any batch
    ((1920, 1080), (480, 270), 1, 128, 0),                         # 2 would fit
    ((1920, 1080), (608, 342), 1, 128, 2 * 15 * 1280),             # 4 in up to three rounds
    ((1920, 1080), (608, 342), 8, 128, 0),
    ((1280, 720), (320, 180), 4, 64, 2 * 18 * 832),
    ((1280, 720), (320, 180), 8, 64, 0),
    ((2400, 1300), (40, 20), 8, 64, 0),                            # none fits
])
def test_tiles_of_the_preprocessing_and_where_it_stages_none(fake, src, net, K, cols, smem):
    at = 0x7F0000000000
    assert fake.tt_preprocess(at, K, 3 * src[0] * src[1], *src, 3 * src[0], at + 0x10000000, *net, 255.0, 0.5, 0.25, None) == 0
    (line,) = [x for x in fake.fake_log().decode().splitlines() if x.startswith("launch")]
    assert line.endswith(f" smem {smem}") and (f"preprocess_staged_kernelILi{cols}E" if smem else "preprocess_direct_kernel") in line


@pytest.mark.parametrize("src,net,pad,K", STAGED_SIZES)
def test_sizes_that_are_there_for_the_staged_preprocessing_reach_it(fake, src, net, pad, K):
    at = 0x7F0000000000
    for batch in (1, K):
        fake.fake_reset()
        assert fake.tt_preprocess(at, batch, src[1] * (3 * src[0] + pad), *src, 3 * src[0] + pad, at + 0x10000000, *net, 255.0, 0.5, 0.25, None) == 0
        assert b"preprocess_staged_kernel" in fake.fake_log()


def test_kernel_attributes_are_set_in_every_context(fake):
    """Kernels of a context that came after another one (a device reset, a second context on the device) know nothing of what the first one's were given."""
    at = 0x7F0000000000
    wl = dict(WORKLOAD, src_w=854, src_h=480, net_w=640, net_h=480, enc_cout=(32, 64), hidden=128, precision="bf16")
    for _ in range(3):
        for _ in range(2):
            assert fake.tt_preprocess(at, 1, 3 * 1920 * 1080, 1920, 1080, 3 * 1920, at + 0x10000000, 520, 292, 255.0, 0.5, 0.25, None) == 0
            for hidden in (16, 128, 256, 512):
                args = (at, 1, 2, 9, 16, hidden, 3, at, at, None, None, 0, 0.5, at, at, at, at)
                assert fake.tt_postprocess_static(*args, None) == 0
        s = Streams(fake, 1, workload=wl, post_tc=False)
        assert s.submit(on_device=(0,))[0] == binding.TT_OK
        s.sync()
        s.ctx.destroy()
        fake.fake_new_context()


def test_the_static_scratch_is_looked_up_in_every_context(fake):
    """An address of a context that is gone is never handed to a kernel."""
    at, seen = 0x7F0000000000, []
    for _ in range(3):
        fake.fake_new_context()
        for again in range(2):
            fake.fake_reset()
            assert fake.tt_postprocess_static(at, 0, 1, 9, 16, 16, 3, at, at, None, None, 0, 0.5, at, at, at, at, None) == 0
            asked, cleared = (re.findall(rf"^{word} (0x\w+)", fake.fake_log().decode(), re.M) for word in ("symbol", "clear"))
            assert len(asked) == 1 - again
            seen.append(cleared[0])
    assert seen[0::2] == seen[1::2] and len(set(seen)) == 3


@pytest.mark.parametrize("net,enc,stride,hidden,K", [
    ((40, 30), (32, 64), (1, 1), 64, 1), ((40, 30), (32, 64), (1, 1), 64, 2), ((40, 30), (32, 64), (1, 1), 64, 3),
    ((160, 120), (16, 32), (2, 2), 64, 3), ((64, 64), (16,), (1,), 16, 1), ((320, 240), (16, 32), (2, 2), 32, 3), ((200, 150), (16,), (2,), 24, 2),
])
def test_a_multiprocessor_holds_no_more_blocks_of_an_fp32_convlstm_than_its_even_share(fake, net, enc, stride, hidden, K):
    """As a dependent it is placed where its predecessor leaves room, and blocks in a pile take as long as the pile is high."""
    s = Streams(fake, K, workload=dict(src_w=net[0], src_h=net[1], net_w=net[0], net_h=net[1], enc_cout=enc, enc_stride=stride, hidden=hidden, n_tools=3))
    log = s.submit(on_device=range(K))[1]
    lstm = [re.search(r"grid (\d+) (\d+) (\d+) smem (\d+)", line) for line in log if re.match(r"launch \S*conv3x3_simt_kernelILi1ELi2E", line)]
    assert len(lstm) == 1
    x, y, z, smem = (int(v) for v in lstm[0].groups())
    share = -(-x * y * z // 148)
    assert (share + 1) * (smem + 1024) > 228 * 1024 >= share * (smem + 1024)
    s.sync()


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",)])
def test_the_current_streams_handle_with_and_without_torchs_own_shortcut(monkeypatch, missing):
    """Names of torch that begin with an underscore may go; the public way to the handle stays."""
    import torch

    class Stream:
        cuda_stream = 77

    shortcut = {"_cuda_getDevice": lambda: 3, "_cuda_getCurrentRawStream": lambda device: 70 + device}
    monkeypatch.setattr(torch, "_C", type("C", (), {k: staticmethod(v) for k, v in shortcut.items() if k not in missing}))
    monkeypatch.setattr(torch.cuda, "current_stream", Stream)
    assert binding._stream_ptr(None) == (77 if missing else 73)
    assert binding._stream_ptr(Stream()) == 77 and binding._stream_ptr(5) == 5
