"""The give-up paths of the bounded device-side waits: with a window's copy withheld the wait runs
out (about a second), the call's error word says so, and after a reset the stream works as a new
one, through every entry and state format whose kernels wait."""
import time

import pytest
import torch

from paper_2106_08034_gb300 import synth
from paper_2106_08034_gb300 import wrls as W

from helpers import cpu_frames

pytestmark = pytest.mark.gpu

WIDTH, HEIGHT = 80, 48  # 18 update tiles, all resident at once; wide enough for every window
BF16, F16 = dict(state_precision=W.WRLS_STATE_BF16), dict(state_precision=W.WRLS_STATE_F16)
G4, NEAREST = dict(n_gbuf=4, n_features=4), dict(reproj_filter=1)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2106_08034_gb300 import build as B
    B.build()
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"


@pytest.fixture(scope="module")
def frames():
    spec = synth.SceneSpec(WIDTH, HEIGHT, 6, seed=58, motion="orbit")
    return [(f["radiance"].cuda(), f["variance"].cuda(), f["features"][:4].contiguous().cuda(), f["motion"].cuda())
            for f in cpu_frames(spec)]


def call(entry, s, fr):
    outs = [torch.empty(3, HEIGHT, WIDTH, device="cuda") for _ in fr]
    if entry == "sequence":
        W.wrls_denoise_sequence(s.handle, [f + (o,) for f, o in zip(fr, outs)])
        return outs
    for (rad, var, feat, mot), o in zip(fr, outs):
        if entry == "frame":
            s.denoise(rad, mot, o, variance=var, features=feat)
        elif entry == "static tick":
            W.wrls_batch_tick_static([(s.handle, rad, None, None, mot, o)])
        else:
            b = W.wrls_batch_create(1)
            W.wrls_batch_tick(b, [(s.handle, rad, None, None, mot, o)])
            torch.cuda.synchronize()
            W.wrls_batch_destroy(b)
    return outs


@pytest.mark.parametrize("kw,entry,first", [
    (dict(), "sequence", 1), (dict(), "static tick", 1),
    (BF16, "frame", 1), (BF16, "sequence", 1), (BF16, "tick", 1), (BF16, "static tick", 1),
    (F16, "frame", 1), (F16, "static tick", 1),
    (G4, "frame", 1), (G4, "sequence", 1), (NEAREST, "frame", 1),
    (G4, "frame", 0),  # a first frame restarts without a copy in the update: the blend's wait alone
], ids=str)
def test_a_wait_that_runs_out_is_reported(frames, kw, entry, first):
    p = W.wrls_params_default(**kw)
    s, fresh = W.Stream(WIDTH, HEIGHT, p), W.Stream(WIDTH, HEIGHT, p)
    if first:
        call("frame", s, frames[:1])
    W.wrls_stream_check(s.handle)
    W.wrls_stream_set_debug(s.handle, W.WRLS_DEBUG_WITHHOLD_STAGE_COPY)
    t0 = time.time()
    call(entry, s, frames[1:3] if entry == "sequence" else frames[1:2])
    with pytest.raises(W.WrlsError) as e:
        W.wrls_stream_check(s.handle)
    assert e.value.status == W.WRLS_ERR_TIMEOUT
    # one limit and one more for copies in flight, in each kernel that waits
    assert 0.3 < time.time() - t0 < 15.0
    W.wrls_stream_set_debug(s.handle, 0)
    s.reset()
    got, want = call(entry, s, frames[3:]), call("frame", fresh, frames[3:])
    W.wrls_stream_check(s.handle)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    s.close()
    fresh.close()
