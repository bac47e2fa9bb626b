"""Parity of the CUDA input steps (pixel reconstruction filter, velocity from first-collision
world positions) with the FP64 oracle (oracle/wrls_oracle_upstream.c), through the C ABI,
and of the whole chain raw samples -> reconstruction -> velocity -> denoiser."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2106_08034_gb300 import synth
from paper_2106_08034_gb300 import wrls as W

from helpers import REL_TOL, oracle_params_from, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2106_08034_gb300 import build as B
    B.build()
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    W.lib()


def _rel_close(a, b, tol=REL_TOL, floor=1e-12):
    """Elementwise relative closeness with identical non-finite positions."""
    a = np.asarray(a, np.float64)
    b = np.asarray(b, np.float64)
    fa, fb = np.isfinite(a), np.isfinite(b)
    assert np.array_equal(fa, fb), "non-finite positions differ"
    err = np.abs(a[fa] - b[fa]) / np.maximum(np.abs(b[fa]), floor)
    return float(err.max()) if err.size else 0.0


@pytest.mark.parametrize("spp,sigma,radius,size", [(1, 0.5, 1.5, (97, 61)), (2, 0.5, 1.5, (250, 130)),
                                                   (4, 0.8, 0.9, (64, 40)), (8, 0.35, 1.5, (33, 17))])
def test_reconstruction_matches_oracle(spp, sigma, radius, size):
    W_, H_ = size
    sc = synth.Scene(synth.SceneSpec(W_, H_, 2, seed=81 + spp, motion="pan", firefly_frac=0.05))
    smp = synth.raw_samples(sc, 1, spp)
    smp[0, 1, 3, 4] = float("nan")          # missing colour
    smp[spp - 1, 3, 5, 6] = float("inf")    # missing offset
    smp[:, 0, 0, 0] = float("nan")          # a pixel without any valid sample
    p = W.wrls_recon_params_default(sigma=sigma, radius=radius)
    d = smp.cuda()
    rad = torch.empty(3, H_, W_, device="cuda")
    var = torch.empty(H_, W_, device="cuda")
    W.wrls_reconstruct(d, rad, var, p)
    torch.cuda.synchronize()
    ref, rvar = O.reconstruct(smp.numpy(), sigma=sigma, radius=radius)
    assert rel_err(rad.cpu().numpy(), ref) <= REL_TOL
    assert _rel_close(var.cpu().numpy(), rvar) <= REL_TOL
    W.wrls_reconstruct(d, rad, None, p)       # variance output is optional
    torch.cuda.synchronize()
    assert rel_err(rad.cpu().numpy(), ref) <= REL_TOL


def test_velocity_matches_oracle_full_hd():
    W_, H_ = 1920, 1080
    M_prev = synth.orbit_camera(9, W_, H_)
    world = synth.first_collision_world(W_, H_, synth.orbit_camera(10, W_, H_), seed=3)
    d = torch.from_numpy(world).cuda()
    for policy in (0, 1):
        mot = torch.empty(2, H_, W_, device="cuda")
        W.wrls_velocity_from_world(d, M_prev, mot, miss_policy=policy)
        torch.cuda.synchronize()
        ref = O.velocity(world, M_prev.astype(np.float32).astype(np.float64), policy)
        got = mot.cpu().numpy()
        fin = np.isfinite(ref)
        assert np.array_equal(fin, np.isfinite(got))
        assert np.abs(got[fin] - ref[fin]).max() <= 2e-3      # pixels
        assert np.abs(ref[fin]).max() > 1.0                   # the camera did move


def test_chain_samples_to_denoised_output():
    """Raw samples -> reconstruction -> velocity -> denoiser on the GPU, against the same
    chain of oracles fed with their own intermediate results (binary32 between the steps)."""
    W_, H_, T = 160, 96, 8
    spec = synth.SceneSpec(W_, H_, T, seed=85, motion="static", firefly_frac=0.02)
    sc = synth.Scene(spec)
    s = W.Stream(W_, H_)
    st = O.OracleStream(W_, H_, oracle_params_from(W.wrls_params_default()))
    rad = torch.empty(3, H_, W_, device="cuda")
    mot = torch.empty(2, H_, W_, device="cuda")
    out = torch.empty(3, H_, W_, device="cuda")
    for t in range(T):
        smp = synth.raw_samples(sc, t, 2)
        world = synth.first_collision_world(W_, H_, synth.orbit_camera(t, W_, H_), seed=t)
        M_prev = synth.orbit_camera(t - 1, W_, H_)
        W.wrls_reconstruct(smp.cuda(), rad)
        W.wrls_velocity_from_world(torch.from_numpy(world).cuda(), M_prev, mot)
        s.denoise(rad, mot, out)
        torch.cuda.synchronize()
        r_rad, _ = O.reconstruct(smp.numpy(), with_variance=False)
        r_mot = O.velocity(world, M_prev.astype(np.float32).astype(np.float64))
        ref, _, _ = st.frame(r_rad.astype(np.float32), r_mot.astype(np.float32))
        assert rel_err(out.cpu().numpy(), ref) <= REL_TOL, t
    s.close()


def test_input_steps_reject_bad_arguments():
    x = torch.zeros(1, 5, 8, 8, device="cuda")
    r = torch.empty(3, 8, 8, device="cuda")
    with pytest.raises(W.WrlsError):
        W.wrls_reconstruct(x, r, params=W.wrls_recon_params_default(radius=2.0))
    with pytest.raises(W.WrlsError):
        W.wrls_reconstruct(x, x[0, :3])              # output overlaps the samples
    with pytest.raises(W.WrlsError):
        W.wrls_velocity_from_world(r, np.full((4, 4), np.nan), torch.empty(2, 8, 8, device="cuda"))


# tiles of 32 x 8, two rows a thread: cut after either row, one row or column, several chunks of
# sample indices; `far` puts some offsets beyond half a pixel, so that the support is tested
@pytest.mark.parametrize("size", [(32, 8), (33, 9), (31, 7), (64, 1), (1, 17), (95, 23)])
@pytest.mark.parametrize("spp,radius,far", [(1, 1.5, False), (2, 1.5, True), (3, 1.2, False), (5, 0.6, True)])
def test_reconstruction_tile_edges(size, spp, radius, far):
    w, h = size
    gen = torch.Generator().manual_seed(w * 100 + h + spp)
    smp = torch.rand(spp, 5, h, w, generator=gen)
    smp[:, 3:] -= 0.5
    if far:
        smp[:, 3:][torch.rand(spp, 2, h, w, generator=gen) < 0.1] *= 2.5
    smp[:, 0][torch.rand(spp, h, w, generator=gen) < 0.1] = float("nan")
    smp[:, 4][torch.rand(spp, h, w, generator=gen) < 0.05] = float("-inf")
    d = smp.cuda()
    rad, var = torch.empty(3, h, w, device="cuda"), torch.empty(h, w, device="cuda")
    W.wrls_reconstruct(d, rad, var, W.wrls_recon_params_default(radius=radius))
    # the support test is binary32 on both sides
    ref, rvar = O.reconstruct(smp.numpy(), radius=float(np.float32(radius)))
    got = rad.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = np.isfinite(ref[0])
    # weights carry ex2's 2^-22 and the sums up to 9 spp roundings
    assert np.abs(got[:, fin] - ref[:, fin]).max(initial=0.0) <= (9 * spp + 8) * 2.0 ** -22
    gv = var.cpu().numpy()
    assert np.array_equal(np.isnan(gv), np.isnan(rvar))
    assert np.abs(gv - rvar)[np.isfinite(rvar)].max(initial=0.0) <= (spp + 8) * 2.0 ** -22


@pytest.mark.parametrize("size,shift", [((64, 5), 0), ((64, 5), 1), ((66, 5), 0), ((4, 3), 0), ((1, 1), 0)])
def test_velocity_widths_and_alignments(size, shift):
    """128-bit accesses where width and buffers allow them, else single values: the same bits."""
    w, h = size
    M = synth.orbit_camera(9, w, h)
    world = synth.first_collision_world(w, h, synth.orbit_camera(10, w, h), seed=3, miss_frac=0.2)
    buf, out = torch.empty(3 * h * w + 1, device="cuda"), torch.empty(2 * h * w + 1, device="cuda")
    d, mot = buf[shift:shift + 3 * h * w].view(3, h, w), out[shift:shift + 2 * h * w].view(2, h, w)
    d.copy_(torch.from_numpy(world))
    W.wrls_velocity_from_world(d, M, mot)
    got = mot.cpu().numpy()
    ref = O.velocity(world, M.astype(np.float32).astype(np.float64))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.nanmax(np.abs(got - ref), initial=0.0) <= 2e-3  # pixels, as at full HD


# sigma beyond 3e22 leaves a binary32 exponent factor of 0; infinity asks for a box filter
@pytest.mark.parametrize("sigma", [1e19, 1e23, float("inf")])
@pytest.mark.parametrize("size", [(61, 23), (33, 9)])
@pytest.mark.parametrize("radius,far", [(1.5, False), (1.2, True)])
def test_reconstruction_with_a_very_wide_filter(sigma, size, radius, far):
    """Samples outside the image or the support and missing samples still have weight 0."""
    w, h = size
    gen = torch.Generator().manual_seed(w + h)
    smp = torch.rand(2, 5, h, w, generator=gen)
    smp[:, 3:] -= 0.5
    if far:
        smp[:, 3:][torch.rand(2, 2, h, w, generator=gen) < 0.1] *= 2.5
    smp[:, 0][torch.rand(2, h, w, generator=gen) < 0.1] = float("nan")
    rad, var = torch.empty(3, h, w, device="cuda"), torch.empty(h, w, device="cuda")
    W.wrls_reconstruct(smp.cuda(), rad, var, W.wrls_recon_params_default(sigma=sigma, radius=radius))
    ref, rvar = O.reconstruct(smp.numpy(), sigma=float(np.float32(sigma)), radius=float(np.float32(radius)))
    got, gv = rad.cpu().numpy(), var.cpu().numpy()
    assert np.isfinite(ref).all() and np.isfinite(got).all()
    assert np.abs(got - ref).max() <= (9 * 2 + 8) * 2.0 ** -22  # as in the tile-edge test
    assert np.array_equal(np.isnan(gv), np.isnan(rvar))


# from 6 tiles an SM a thread takes two pixels: the same tile edges on images of that size, and the
# bits of the one-pixel form on a part of it
@pytest.mark.parametrize("size", [(1025, 225), (1056, 233), (991, 248)])
@pytest.mark.parametrize("spp,radius,far", [(1, 1.5, False), (2, 1.5, True), (5, 0.6, True)])
def test_reconstruction_two_pixels_a_thread(size, spp, radius, far):
    w, h = size
    gen = torch.Generator().manual_seed(w * 100 + h + spp)
    smp = torch.rand(spp, 5, h, w, generator=gen)
    smp[:, 3:] -= 0.5
    if far:
        smp[:, 3:][torch.rand(spp, 2, h, w, generator=gen) < 0.1] *= 2.5
    smp[:, 0][torch.rand(spp, h, w, generator=gen) < 0.1] = float("nan")
    p = W.wrls_recon_params_default(radius=radius)

    def run(s):
        d = s.contiguous().cuda()
        rad, var = torch.empty(3, *s.shape[2:], device="cuda"), torch.empty(*s.shape[2:], device="cuda")
        W.wrls_reconstruct(d, rad, var, p)
        only = torch.empty_like(rad)
        W.wrls_reconstruct(d, only, None, p)
        assert torch.equal(rad.nan_to_num(nan=-7.0), only.nan_to_num(nan=-7.0))
        return rad.cpu(), var.cpu()
    rad, var = run(smp)
    ref, rvar = O.reconstruct(smp.numpy(), radius=float(np.float32(radius)))
    got, fin = rad.numpy(), np.isfinite(ref[0])
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.abs(got[:, fin] - ref[:, fin]).max(initial=0.0) <= (9 * spp + 8) * 2.0 ** -22
    assert np.array_equal(np.isnan(var.numpy()), np.isnan(rvar))
    assert np.abs(var.numpy() - rvar)[np.isfinite(rvar)].max(initial=0.0) <= (spp + 8) * 2.0 ** -22
    y, x = h - 41, w - 67  # an inner part, and its pixels whose 3x3 neighbours lie in it
    prad, pvar = run(smp[:, :, y - 50:y, x - 90:x])
    assert torch.equal(prad[:, 1:-1, 1:-1].nan_to_num(nan=-7.0), rad[:, y - 49:y - 1, x - 89:x - 1].nan_to_num(nan=-7.0))
    assert torch.equal(pvar[1:-1, 1:-1].nan_to_num(nan=-7.0), var[y - 49:y - 1, x - 89:x - 1].nan_to_num(nan=-7.0))
