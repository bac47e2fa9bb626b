"""Per-frame calls, the input steps, the renderer and the state moves set up each kernel while the one
before finishes (programmatic dependent launch). Calls enqueued back to back give the bits of the
same calls with a synchronisation after each: no kernel reads its inputs or the state, or overwrites
either, ahead of its turn. Covered are frames whose inputs are rewritten in between on the same CUDA
stream, with a second stream object on it and with per-frame and sequence calls mixed; frames of one
stream with nothing in between; the chain from renderer to denoised frame; and state moves."""
import pytest
import torch

from paper_2106_08034_gb300 import synth
from paper_2106_08034_gb300 import wrls as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2106_08034_gb300 import build as B
    B.build()
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"


# below and above the size where the two-wide blend starts (2^17 pixels), one tile, many tiles
@pytest.mark.parametrize("wh", [(31, 7), (128, 128), (511, 256), (513, 257), (1283, 721)])
@pytest.mark.parametrize("kw", [dict(), dict(state_precision=W.WRLS_STATE_BF16), dict(n_gbuf=2, n_features=2)])
def test_back_to_back_frames(wh, kw):
    w, h = wh
    gen = torch.Generator(device="cuda").manual_seed(w)
    n = 10
    rads = [torch.rand(3, h, w, generator=gen, device="cuda") for _ in range(n)]
    mots = [2 * torch.rand(2, h, w, generator=gen, device="cuda") - 1 for _ in range(n)]
    feat = torch.rand(2, h, w, generator=gen, device="cuda") if "n_gbuf" in kw else None
    cs = torch.cuda.Stream()
    cs.wait_stream(torch.cuda.current_stream())

    def run(sync):
        outs = []
        with torch.cuda.stream(cs):
            a, b = (W.Stream(w, h, W.wrls_params_default(**kw), cuda_stream=cs) for _ in range(2))
            rad, mot = torch.empty_like(rads[0]), torch.empty_like(mots[0])
            for t in range(n):
                rad.copy_(rads[t])
                mot.copy_(mots[t])
                for s in (a, b) if t % 3 == 0 else (a,):
                    o = torch.empty(3, h, w, device="cuda")
                    if t == 5:  # two frames through the sequence entry in between
                        o2 = torch.empty(3, h, w, device="cuda")
                        W.wrls_denoise_sequence(s.handle, [(rad, None, feat, mot, o), (rads[t], None, feat, mots[t], o2)])
                        outs.append(o2)
                    else:
                        s.denoise(rad, mot, o, features=feat)
                    outs.append(o)
                    if sync:
                        cs.synchronize()
            cs.synchronize()
            for s in (a, b):
                W.wrls_stream_check(s.handle)
                s.close()
        return outs
    for x, y in zip(run(True), run(False)):
        assert torch.equal(x, y)


SIZES = [(31, 7), (128, 128), (513, 257), (1283, 721)]


def _repeat(run):
    """The outputs of run(sync=True) and of run(sync=False) are the same bits."""
    want, got = run(True), run(False)
    torch.cuda.synchronize()
    assert len(want) == len(got)
    for x, y in zip(want, got):
        assert torch.equal(x, y)


# nothing between the calls of one stream: the update of a frame is set up beside the blend of the frame
# before, which still reads the state copy that the update after the next one overwrites
@pytest.mark.parametrize("wh", SIZES)
@pytest.mark.parametrize("kw", [dict(), dict(state_precision=W.WRLS_STATE_BF16), dict(state_precision=W.WRLS_STATE_F16),
                                dict(blend_mode=1), dict(n_gbuf=2, n_features=2), dict(n_gbuf=2, n_features=2, blend_mode=1)],
                         ids=str)
def test_adjacent_frames_of_one_stream(wh, kw):
    w, h = wh
    gen = torch.Generator(device="cuda").manual_seed(w + 1)
    n = 12
    rads = [torch.rand(3, h, w, generator=gen, device="cuda") for _ in range(n)]
    mots = [6 * torch.rand(2, h, w, generator=gen, device="cuda") - 3 for _ in range(n)]
    feat = torch.rand(2, h, w, generator=gen, device="cuda") if "n_gbuf" in kw else None
    torch.cuda.synchronize()

    def run(sync):
        s = W.Stream(w, h, W.wrls_params_default(**kw))
        outs = [torch.empty(3, h, w, device="cuda") for _ in range(n)]
        state = torch.empty(s.state_planes, h, w, device="cuda")
        torch.cuda.synchronize()
        for t in range(n):
            s.denoise(rads[t], mots[t], outs[t], features=feat)
            if sync:
                torch.cuda.synchronize()
        s.read_state(state)
        W.wrls_stream_check(s.handle)
        s.close()
        return outs + [state]
    _repeat(run)


@pytest.mark.parametrize("wh", [(64, 40), (513, 257), (1284, 721)])
def test_renderer_inputs_and_frames_in_one_chain(wh):
    """Render, reconstruct, find the motion, denoise, the same buffers in every frame: each step's inputs
    are the outputs of the one ahead of it, and its outputs are what the frame before still read."""
    w, h = wh
    n = 6
    mats = [synth.orbit_camera(t, w, h) for t in range(n + 1)]

    def run(sync):
        s = W.Stream(w, h, W.wrls_params_default())
        smp, world = torch.empty(2, 5, h, w, device="cuda"), torch.empty(3, h, w, device="cuda")
        rad, var, mot = torch.empty(3, h, w, device="cuda"), torch.empty(h, w, device="cuda"), torch.empty(2, h, w, device="cuda")
        outs = [torch.empty(3, h, w, device="cuda") for _ in range(n)]
        kept = [torch.empty(6, h, w, device="cuda") for _ in range(n)]
        scenes = [W.vpt_scene_struct(synth.vpt_scene(w, h, t=t, seed=5)) for t in range(n)]
        torch.cuda.synchronize()
        for t in range(n):
            steps = [lambda: W.wrls_render_vpt(scenes[t], smp, world, frame=t), lambda: W.wrls_reconstruct(smp, rad, var),
                     lambda: W.wrls_velocity_from_world(world, mats[t], mot), lambda: s.denoise(rad, mot, outs[t])]
            for step in steps:
                step()
                if sync:
                    torch.cuda.synchronize()
            if t % 2:  # (half of the frames are followed by the next one's kernels at once)
                kept[t].copy_(torch.cat([rad, var[None], mot]))
        W.wrls_stream_check(s.handle)
        s.close()
        return [torch.nan_to_num(x, nan=-7.0) for x in outs + kept[1::2]]
    _repeat(run)


@pytest.mark.parametrize("wh", SIZES)
@pytest.mark.parametrize("precision", [W.WRLS_STATE_F32, W.WRLS_STATE_BF16, W.WRLS_STATE_F16])
def test_state_moves_between_frames(wh, precision):
    """write_state, a frame, read_state, into a buffer that the next write_state reads."""
    w, h = wh
    gen = torch.Generator(device="cuda").manual_seed(w + 2)
    n = 5
    rads = [torch.rand(3, h, w, generator=gen, device="cuda") for _ in range(n)]
    mots = [2 * torch.rand(2, h, w, generator=gen, device="cuda") - 1 for _ in range(n)]
    first = torch.zeros(25, h, w, device="cuda")
    first[[12, 16, 19, 21]] = 1.0
    first[22:] = torch.rand(3, h, w, generator=gen, device="cuda")
    torch.cuda.synchronize()

    def run(sync):
        a, b = (W.Stream(w, h, W.wrls_params_default(state_precision=precision)) for _ in range(2))
        state = first.clone()
        outs = [torch.empty(3, h, w, device="cuda") for _ in range(2 * n)]
        torch.cuda.synchronize()
        for t in range(n):
            for i, s in enumerate((a, b)):
                for step in (lambda: s.write_state(state), lambda: s.denoise(rads[t], mots[t], outs[2 * t + i]),
                             lambda: s.read_state(state)):
                    step()
                    if sync:
                        torch.cuda.synchronize()
        for s in (a, b):
            W.wrls_stream_check(s.handle)
            s.close()
        return outs + [state]
    _repeat(run)
