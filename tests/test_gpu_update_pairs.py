"""The 16-bit update (two pixels a thread) against the oracle, one frame from a state read back.

The state before the frame is read from the stream (decoded exactly) and handed to the FP64
oracle, so one frame's arithmetic and encoding are compared alone. Rounding to p significant bits
moves a value by at most u = 2^-p of itself: 2^-8 (BF16) or 2^-11 (FP16; 2^-25 below its normal
range). P is
stored as its Cholesky factor L, so |dP_ij| <= (2u + u^2) sum_k |L_ik L_jk| <= 2.01 u sqrt(P_ii P_jj)
by Cauchy-Schwarz. On top of that the binary32 arithmetic may be off by some 20 roundings of the
largest operands: 4e-6 of their scale.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2106_08034_gb300 import wrls as W

from helpers import oracle_params_from

pytestmark = pytest.mark.gpu

IU = [(0, 0), (0, 1), (0, 2), (0, 3), (1, 1), (1, 2), (1, 3), (2, 2), (2, 3), (3, 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2106_08034_gb300 import build as B
    B.build()
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"


def _motion(kind, w, h, rng):
    m = np.zeros((2, h, w), np.float32)
    if kind == "pan":            # integral rows: two taps
        m[0] = 1.7
    elif kind == "drift":        # four taps, footprint inside the staged window
        m[0] = 0.6 + 0.5 * rng.random((h, w))
        m[1] = -0.4 + 0.5 * rng.random((h, w))
    elif kind == "scatter":      # footprint beyond the staged window: taps from global memory
        m[:] = 40 * (rng.random((2, h, w)) - 0.5)
    if kind != "static":
        m[:, rng.random((h, w)) < 0.03] = np.nan
    return m


# the 40 x 10 window exactly, one more or less, tiles cut in both pixels of a pair, no window
@pytest.mark.parametrize("wh", [(40, 10), (33, 9), (64, 8), (65, 13), (97, 20), (100, 3), (31, 40), (1, 1)])
@pytest.mark.parametrize("kind", ["static", "pan", "drift", "scatter"])
@pytest.mark.parametrize("precision", [W.WRLS_STATE_BF16, W.WRLS_STATE_F16])
def test_one_frame_against_the_oracle(wh, kind, precision):
    w, h = wh
    rng = np.random.default_rng(w * 100 + h + precision)
    feature_mode, init_mode = (1, 1) if kind == "pan" else (0, 0)
    p = W.wrls_params_default(state_precision=precision, feature_mode=feature_mode, init_mode=init_mode)
    s = W.Stream(w, h, p)
    out = torch.empty(3, h, w, device="cuda")
    st = torch.empty(25, h, w, device="cuda")
    for t in range(4):
        if t == 3:
            s.read_state(st)
            torch.cuda.synchronize()
            before = st.double().cpu().numpy().reshape(25, -1)
        rad = (0.5 + 0.2 * rng.standard_normal((3, h, w))).astype(np.float32)
        rad[:, rng.random((h, w)) < 0.05] = np.inf
        if w > 8:
            rad[1, :3, :5] = np.nan  # a neighbourhood without a sample
        mot = _motion(kind, w, h, rng)
        s.denoise(torch.from_numpy(rad).cuda(), torch.from_numpy(mot).cuda(), out)
    s.read_state(st)
    W.wrls_stream_check(s.handle)
    s.close()
    got = st.double().cpu().numpy().reshape(25, -1)
    ref = O.OracleStream(w, h, oracle_params_from(p))
    n = w * h
    ref.beta[:] = before[:12].T.reshape(n, 3, 4)
    ref.z[:] = before[22:].T
    for q, (a, b) in enumerate(IU):
        ref.P[:, a, b] = ref.P[:, b, a] = before[12 + q]
    ref.need_reset = False
    ref.frame(rad, mot)
    u, tiny = (2.0 ** -8, 0.0) if precision == W.WRLS_STATE_BF16 else (2.0 ** -11, 2.0 ** -25)
    scale = max(np.abs(ref.P).max(), np.abs(before[12:22]).max(), 1.0)
    assert np.all(np.abs(got[22:].T - ref.z) <= u * np.abs(ref.z) + tiny + 4e-6)
    beta = got[:12].T.reshape(n, 3, 4)
    assert np.all(np.abs(beta - ref.beta) <= u * np.abs(ref.beta) + tiny + 4e-6 * scale * (1 + np.abs(ref.beta).max()))
    d = np.sqrt(np.maximum(np.einsum("naa->na", ref.P), 0.0))
    for q, (a, b) in enumerate(IU):
        bound = 2.01 * u * d[:, a] * d[:, b] + 4 * tiny * scale + 4e-6 * scale
        assert np.all(np.abs(got[12 + q] - ref.P[:, a, b]) <= bound), (a, b)
