"""Host side of the launches, followed with a stand-in CUDA runtime of two devices (no GPU needed)."""
import ctypes
import glob
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2106_08034_gb300 import build as B
from paper_2106_08034_gb300 import synth
from paper_2106_08034_gb300 import wrls as W

HERE = os.path.dirname(os.path.abspath(__file__))
WIDTH, HEIGHT = 512, 300  # above the size where the two-wide blend becomes the default
PLANE = WIDTH * HEIGHT
BUF = np.zeros(32 * PLANE, np.float32)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """The library's objects linked with fake_cudart.cpp in place of the CUDA runtime."""
    B.build()
    sources = glob.glob(os.path.join(B.CSRC, "*.cu"))
    objs = [os.path.join(B.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in sorted(sources)]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    so = str(tmp_path_factory.mktemp("fake") / "libwrls_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    # -Bsymbolic: the library's calls reach the stand-in even where a CUDA runtime is loaded already
    cmd = ["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-o", so,
           os.path.join(HERE, "fake_cudart.cpp")] + objs
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    saved = W._lib, W.LIB_PATH
    W._lib, W.LIB_PATH = None, so
    try:
        W.lib().fake_launch_kernel.restype = ctypes.c_char_p
        yield W.lib()
    finally:
        W._lib, W.LIB_PATH = saved


@pytest.fixture()
def runtime(fake):
    fake.fake_set_device(0)
    fake.fake_fail_launches(0, 0)
    yield fake
    fake.fake_fail_launches(0, 0)
    fake.fake_set_device(0)


def at(plane):
    return BUF.ctypes.data + 4 * plane * PLANE


def frame(s):
    s.denoise(at(0), at(3), at(8), variance=at(5), features=at(16))


class Array:
    """A buffer with the attributes that the binding reads."""

    def __init__(self, a):
        self.shape, self.data_ptr = a.shape, lambda: a.ctypes.data


PAPER = [dict(), dict(state_precision=W.WRLS_STATE_BF16), dict(state_precision=W.WRLS_STATE_F16), dict(blend_mode=1)]
EXTENDED = [dict(n_gbuf=4, n_features=4), dict(n_gbuf=2, n_features=2), dict(weight_mode=2), dict(reproj_filter=1),
            dict(n_gbuf=4, n_features=4, blend_mode=1), dict(n_gbuf=4, n_features=4, feature_mode=1)]


@pytest.mark.parametrize("kw", PAPER + EXTENDED, ids=str)
def test_every_device_of_a_process_is_set_up(runtime, kw):
    """A kernel's opt-in to large shared memory belongs to a device: streams on a second one work too,
    through per-frame, sequence and batched calls and with every blend configuration."""
    for dev in (0, 1, 0):
        assert runtime.fake_set_device(dev) == 0
        p = W.wrls_params_default(**kw)
        s = W.Stream(WIDTH, HEIGHT, p)
        frame(s)
        W.wrls_denoise_sequence(s.handle, [(at(0), at(5), at(16), at(3), at(8 + 4 * (k & 1))) for k in range(4)])
        if kw in PAPER:
            b = W.wrls_batch_create(1)
            W.wrls_batch_tick(b, [(s.handle, at(0), None, None, at(3), at(8))])
            W.wrls_batch_destroy(b)
            W.wrls_batch_tick_static([(s.handle, at(0), None, None, at(3), at(8))])
            for cfg in range(W.BLEND_CONFIGS):
                if 4 <= cfg <= 7 and p.state_precision != W.WRLS_STATE_F32:
                    continue
                W.wrls_stream_set_blend_config(s.handle, cfg)
                frame(s)
        s.close()


def test_a_failed_launch_leaves_no_error_pending(runtime):
    """The status reports it; the caller's next check of the runtime's last error finds nothing."""
    s, e = W.Stream(WIDTH, HEIGHT, W.wrls_params_default()), W.Stream(WIDTH, HEIGHT, W.wrls_params_default(**EXTENDED[0]))
    frame(s)
    frame(e)
    samples = np.zeros((1, 5, HEIGHT, WIDTH), np.float32)
    planes = BUF.reshape(-1, HEIGHT, WIDTH)

    scene = W.vpt_scene_struct(synth.vpt_scene(WIDTH, HEIGHT, t=0, seed=1))
    io = [(at(0), at(5), at(16), at(3), at(8 + 4 * (k & 1))) for k in range(2)]
    calls = [lambda: frame(s), lambda: frame(e), lambda: W.wrls_denoise_sequence(s.handle, io),
             lambda: W.wrls_denoise_sequence(e.handle, io), lambda: s.write_state(at(0)), lambda: s.read_state(at(0)),
             lambda: W.wrls_reconstruct(Array(samples), Array(planes[:3])),
             lambda: W.wrls_velocity_from_world(Array(planes[:3]), np.eye(4), Array(planes[3:5])),
             lambda: W.wrls_render_vpt(scene, Array(samples), Array(planes[:3]))]
    for call in calls:
        for ok in range(2):  # the first or the second launch of the call fails
            runtime.fake_fail_launches(0, 0)
            call()
            n = runtime.fake_launches()
            call()
            if ok >= runtime.fake_launches() - n:
                continue
            runtime.fake_fail_launches(ok, 1)
            with pytest.raises(W.WrlsError) as err:
                call()
            assert err.value.status == W.WRLS_ERR_CUDA
            assert runtime.fake_last_error() == 0
    s.close()
    e.close()


def launched(runtime, call):
    """[(kernel, launched early)] of a call."""
    n = runtime.fake_launches()
    call()
    return [(runtime.fake_launch_kernel(k).decode(), runtime.fake_launch_early(k)) for k in range(n, runtime.fake_launches())]


def blends(runtime, call):
    """The blend configurations of a call: 2 (one CTA a tile), 8 or 9 (two-wide)."""
    out = set()
    for name, _ in launched(runtime, call):
        if "blend" in name:
            out.add(9 if "k_blend_tma2ILi8E" in name else 8 if "k_blend_tma2hILi16E" in name else
                    2 if "k_blendI" in name and "ELi16ELi2E" in name else name)
    return out


# two-wide configuration (9, 8) or 2 by default, through per-frame calls, sequences, a tick of one stream and
# a tick of four: by the waves of 64 x 16 tiles on 2 x 152 CTAs for the 16-bit formats
@pytest.mark.parametrize("width,height,f32,half", [
    (256, 256, (2, 2, 2, 2), (2, 2, 2, 2)),
    (361, 363, (2, 2, 2, 2), (2, 2, 2, 2)),      # 29 pixels short of 2^17
    (512, 256, (9, 9, 9, 9), (8, 2, 2, 8)),      # 128 tiles: 0.42 of a wave; four streams 1.68 waves
    (400, 400, (9, 9, 9, 9), (8, 2, 2, 8)),      # 175
    (643, 361, (9, 9, 9, 9), (8, 8, 8, 8)),      # 253: 0.83
    (608, 608, (9, 9, 9, 9), (2, 2, 2, 8)),      # 380: 1.25 waves, 5 waves of four streams
    (854, 480, (9, 9, 9, 9), (2, 2, 2, 8)),      # 420: 1.38 waves
    (800, 600, (9, 9, 9, 9), (8, 8, 8, 8)),      # 494: 1.63
    (1024, 512, (9, 9, 9, 9), (8, 8, 8, 8)),     # 2^19 pixels
    (16384, 8, (2, 2, 2, 2), (2, 2, 2, 2)),      # lower than a window
])
def test_default_blend_of_each_entry(runtime, width, height, f32, half):
    plane = width * height
    buf = np.zeros(40 * plane, np.float32)

    def at(p):
        return buf.ctypes.data + 4 * p * plane
    for prec, want in ((W.WRLS_STATE_F32, f32), (W.WRLS_STATE_BF16, half), (W.WRLS_STATE_F16, half)):
        ss = [W.Stream(width, height, W.wrls_params_default(state_precision=prec)) for _ in range(4)]
        s, b = ss[0], W.wrls_batch_create(4)
        io = [(at(0), None, None, at(3), at(5 + 3 * k)) for k in range(2)]
        tick = [(x.handle, at(0), None, None, at(3), at(5 + 3 * k)) for k, x in enumerate(ss)]
        calls = (lambda: s.denoise(at(0), at(3), at(5)), lambda: W.wrls_denoise_sequence(s.handle, io),
                 lambda: W.wrls_batch_tick(b, tick[:1]), lambda: W.wrls_batch_tick(b, tick))
        assert [blends(runtime, c) for c in calls] == [{w} for w in want]
        W.wrls_stream_set_blend_config(s.handle, 2)  # a configuration that was set holds for every entry
        assert [blends(runtime, c) for c in calls[:3]] == [{2}] * 3
        W.wrls_batch_destroy(b)
        for x in ss:
            x.close()


def test_autotune_times_what_frames_run(runtime):
    """The blend of a per-frame call is launched early; so are the launches that autotune compares."""
    s = W.Stream(WIDTH, HEIGHT, W.wrls_params_default())
    assert all(early for _, early in launched(runtime, lambda: frame(s)))
    log = launched(runtime, lambda: W.wrls_stream_autotune(s.handle, at(8), 3))
    assert len(log) == 1 + W.BLEND_CONFIGS * 4 and all(early for _, early in log)
    s.close()


def hints_offset():
    """Byte offset of KParams::hints (all members are 4 bytes wide)."""
    src = open(os.path.join(B.CSRC, "wrls_device.cuh")).read()
    body = re.sub(r"//[^\n]*", "", src[src.index("struct KParams {"):])
    body = body[body.index("{") + 1:body.index("};")]
    off = 0
    for name, array in re.findall(r"(?:float|int) (\w+)(\[kMaxTaps\])?;", body):
        if name == "hints":
            return off
        off += 4 * (25 if array else 1)
    raise AssertionError("KParams::hints not found")


# update tiles (32 x 8) against 152 SMs: early where every CTA finds an SM of its own or there are waves
@pytest.mark.parametrize("width,height,hold", [(128, 128, False), (152, 120, False), (160, 123, True), (200, 150, True),
                                               (361, 363, True), (512, 304, True), (512, 305, False), (1280, 720, False)])
@pytest.mark.parametrize("kw", [dict(), dict(state_precision=W.WRLS_STATE_BF16), dict(n_gbuf=4, n_features=4),
                                dict(reproj_filter=1), dict(blend_mode=1)], ids=str)
def test_frames_resident_at_once_hold_the_next_kernel(runtime, width, height, hold, kw):
    """The kernels of a per-frame call let the next one in early except on images whose CTAs share SMs
    and are all resident; sequences launch plainly, without either hint."""
    plane = width * height
    buf = np.zeros(32 * plane, np.float32)

    def at(p):
        return buf.ctypes.data + 4 * p * plane
    s = W.Stream(width, height, W.wrls_params_default(**kw))
    io = [(at(0), at(5), at(16), at(3), at(8 + 4 * k)) for k in range(2)]
    runtime.fake_watch(hints_offset())
    n = runtime.fake_launches()
    s.denoise(at(0), at(3), at(8), variance=at(5), features=at(16))
    assert [runtime.fake_watched(k) for k in range(n, n + 2)] == [256 + 512 * hold] * 2
    n = runtime.fake_launches()
    W.wrls_denoise_sequence(s.handle, io)
    assert all(runtime.fake_watched(k) < 256 for k in range(n, n + 4))
    runtime.fake_watch(-1)
    s.close()


@pytest.mark.parametrize("width,height,one", [(64, 64, True), (643, 320, True), (640, 364, False), (1920, 1080, False)])
def test_reconstruction_takes_one_pixel_a_thread_on_small_images(runtime, width, height, one):
    """Below 6 tiles an SM (912 of 32 x 8 on 152), with and without variance."""
    samples, out = np.zeros((2, 5, height, width), np.float32), np.zeros((4, height, width), np.float32)
    for var in (None, Array(out[3])):
        (name, early), = launched(runtime, lambda: W.wrls_reconstruct(Array(samples), Array(out[:3]), var))
        assert early and ("k_reconstructILb%dELi%dE" % (var is not None, 1 if one else 2)) in name


@pytest.mark.parametrize("width,height,small", [(128, 128, True), (320, 240, True), (320, 241, False), (361, 363, False)])
@pytest.mark.parametrize("kw,gbuf", [(dict(reproj_filter=1), False), (dict(weight_mode=2), False),
                                     (dict(weight_mode=2, feature_mode=1), False), (dict(n_gbuf=1, n_features=1), True),
                                     (dict(n_gbuf=4, n_features=4), True)], ids=str)
def test_extended_blend_of_small_images(runtime, width, height, small, kw, gbuf):
    """Without G-buffer entries, up to 2 tiles (32 x 8) an SM: one column a thread; else two columns."""
    plane = width * height
    buf = np.zeros(24 * plane, np.float32)

    def at(p):
        return buf.ctypes.data + 4 * p * plane
    s = W.Stream(width, height, W.wrls_params_default(**kw))
    log = launched(runtime, lambda: s.denoise(at(0), at(3), at(8), variance=at(5), features=at(16)))
    assert "k_update_ext" in log[0][0] and ("k_blend_extI" if small and not gbuf else "k_blend_ext2I") in log[1][0]
    s.close()
