"""Per-frame calls set up each kernel while the one before finishes (programmatic dependent launch).
Frames enqueued back to back, their inputs rewritten in between on the same CUDA stream, give the
bits of the same frames with a synchronisation after every call: no kernel reads its inputs or the
state, or overwrites the state, ahead of its turn. Also with a second stream object on the same
CUDA stream and with per-frame and sequence calls mixed."""
import pytest
import torch

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
