"""The workloads whose time is watched: the denoiser's calls over the range a renderer makes them.

A case is a dict of plain values; `listed()` gives the fixed ones and `draw(rng)` another one of
the same ranges. `prepare` makes a case's inputs on the GPU and the library objects a program
keeps, `run` is one pass through the public entry points of `paper_2106_08034_gb300.wrls`, and
`exact` restates the pass in 64-bit torch.

Denoising cases have `frames` frames in a pass. With `history` 0 a pass is a whole recorded clip:
the stream is reset, then its frames are denoised. With `history` > 0 it is a live stream: that
many frames were denoised before, and every pass takes the next ones of a ring of `ring` frames.
"""
import math

import numpy as np
import torch

from paper_2106_08034_gb300 import synth, wrls

PRECISION = {"f32": wrls.WRLS_STATE_F32, "bf16": wrls.WRLS_STATE_BF16, "f16": wrls.WRLS_STATE_F16}
# sizes of the batched streams: viewers of one server (the mixed workload of the benchmark, halved)
MIX = ((512, 512), (512, 512), (1280, 720), (1280, 720), (1920, 1080), (1920, 1080), (2560, 1440), (3840, 2160))
MAX_WORK = 3840 * 2160 * 8  # pixel-frames of the largest denoising pass


def denoise_case(name, kind, width, height, frames, state="f32", motion="orbit", history=0, ring=0, **options):
    case = {"name": name, "kind": kind, "width": width, "height": height, "frames": frames, "state": state,
            "motion": motion, "history": history, "ring": ring or frames + history, "fireflies": 0.05,
            "n_gbuf": 0, "weight_mode": 0, "blend_mode": 0, "feature_mode": 0, "reproj_filter": 0}
    case.update(options)
    return case


def listed():
    return [
        # a preview window, one call a frame: latency and launches are all there is
        denoise_case("preview 128x128", "frame", 128, 128, 1, motion="static", history=3, ring=8, fireflies=0.0),
        # a resizable viewport of odd size under a moving camera, one call a frame
        denoise_case("viewport 643x361", "frame", 643, 361, 4),
        # an interactive viewer at full HD, binary32 state, panning camera, one call a frame
        denoise_case("viewer 1080p f32", "frame", 1920, 1080, 1, motion="pan", history=3, ring=4),
        # a viewer at 1440p that halves its state with binary16, one call a frame
        denoise_case("viewer 1440p f16", "frame", 2560, 1440, 1, state="f16", history=3, ring=4),
        # offline denoising of a recorded full-HD clip, several frames in a call
        denoise_case("clip 1080p f32", "sequence", 1920, 1080, 8),
        # the largest: a 4K clip with the bfloat16 state
        denoise_case("clip 2160p bf16", "sequence", 3840, 2160, 8, state="bf16"),
        # a server's tick over viewers of mixed sizes, bfloat16 state (sessions cost memory)
        {"name": "tick of 8 viewers bf16", "kind": "tick", "streams": len(MIX), "state": "bf16", "history": 2,
         "ring": 3, "fireflies": 0.05},
        # a program whose frames live in pinned host memory
        denoise_case("host clip 1080p f32", "host", 1920, 1080, 6),
        # regression on noisy G-buffers (depth, normal) beside the temporal feature: 8 predictor entries
        denoise_case("G-buffer clip 1080p", "sequence", 1920, 1080, 4, n_gbuf=4, fireflies=0.0),
        # what a renderer does before each frame: filter its raw samples, find the pixels' motion
        {"name": "inputs 1080p 2 spp", "kind": "inputs", "width": 1920, "height": 1080, "spp": 2, "variance": True},
        # the renderer itself at full HD, with the noisy G-buffers
        {"name": "render 1080p 2 spp", "kind": "render", "width": 1920, "height": 1080, "spp": 2, "features": True},
        # moving a session to another process: state out of one stream, into another, and back out
        {"name": "session 1080p f16", "kind": "session", "width": 1920, "height": 1080, "state": "f16"},
    ]


def draw(rng):
    def size(lo, hi):  # pixels spread over their logarithm; aspect 1:1 to 21:9; odd sizes as often as even
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        aspect = rng.uniform(1.0, 2.34)
        return max(33, round(math.sqrt(n * aspect))), max(33, round(math.sqrt(n / aspect)))

    kind = rng.choice(["frame", "frame", "sequence", "sequence", "tick", "host", "inputs", "render", "session"])
    w, h = size(96 * 96, 3840 * 2160)
    if kind == "tick":
        return {"kind": kind, "streams": rng.randint(2, len(MIX)), "state": rng.choice(["f32", "bf16", "f16"]),
                "history": 2, "ring": 3, "fireflies": rng.choice([0.0, 0.05])}
    if kind == "inputs":
        w, h = size(96 * 96, 2560 * 1440)
        return {"kind": kind, "width": w, "height": h, "spp": rng.randint(1, 4), "variance": rng.random() < 0.5}
    if kind == "render":
        w, h = size(96 * 96, 1280 * 720)
        return {"kind": kind, "width": w, "height": h, "spp": rng.randint(1, 4), "features": rng.random() < 0.5}
    if kind == "session":
        w, h = size(96 * 96, 2560 * 1440)
        return {"kind": kind, "width": w, "height": h, "state": rng.choice(["f32", "bf16", "f16"])}
    options = {"fireflies": rng.choice([0.0, 0.05]), "motion": rng.choice(["static", "pan", "orbit", "orbit"])}
    if rng.random() < 0.3:  # the extended predictor and weights: binary32 state
        w, h = size(96 * 96, 1920 * 1080)
        options.update(rng.choice([{"n_gbuf": rng.randint(1, 4)}, {"weight_mode": 2}, {"reproj_filter": 1},
                                   {"n_gbuf": 2, "feature_mode": 1}]), fireflies=0.0)
        frames = rng.randint(2, 4)
    else:
        options.update(state=rng.choice(["f32", "f32", "bf16", "f16"]), blend_mode=rng.choice([0, 0, 0, 1]),
                       feature_mode=rng.choice([0, 0, 0, 1]), weight_mode=rng.choice([0, 0, 0, 1]))
        frames = rng.randint(2, 6)
    if kind == "host":  # bound by the host link, several times slower a pixel
        w, h = size(96 * 96, 1920 * 1080)
    frames = max(1, min(frames, MAX_WORK // (2 * w * h)))
    case = denoise_case("", kind, w, h, frames, **options)
    del case["name"]
    return case


# ---- inputs --------------------------------------------------------------------------------

def make_frames(width, height, count, seed, motion, fireflies):
    spec = synth.SceneSpec(width, height, count + 1, seed=seed, motion=motion, firefly_frac=fireflies)
    scene = synth.Scene(spec)
    return [scene.frame(t + 1, "cuda") for t in range(count)]


def needs(case):
    """(variance plane wanted, feature planes wanted)"""
    return case["weight_mode"] == 2, case["n_gbuf"]


def params_of(case):
    p = wrls.wrls_params_default(state_precision=PRECISION[case["state"]])
    for k in ("n_gbuf", "weight_mode", "blend_mode", "feature_mode", "reproj_filter"):
        if k in case:
            setattr(p, k, case[k])
    p.n_features = p.n_gbuf
    return p


def denoise_inputs(case, seed):
    """The ring of frames: (radiance, variance or None, G-buffer planes or None, motion) each."""
    var, g = needs(case)
    out = []
    for f in make_frames(case["width"], case["height"], case["ring"], seed, case["motion"], case["fireflies"]):
        out.append((f["radiance"], f["variance"] if var else None, f["features"][:g].contiguous() if g else None,
                    f["motion"]))
    return out


def mix_inputs(case, seed):
    return [[(f["radiance"], f["motion"]) for f in
             make_frames(w, h, case["ring"], seed * 100 + k, "orbit", case["fireflies"])]
            for k, (w, h) in enumerate(MIX[-case["streams"]:])]


def raw_inputs(case, seed):
    w, h = case["width"], case["height"]
    scene = synth.Scene(synth.SceneSpec(w, h, 2, seed=seed, motion="static", firefly_frac=0.05))
    samples = synth.raw_samples(scene, 1, case["spp"], "cuda")
    # collisions at a smooth depth behind each pixel, a tenth of the rays leave without one
    vp = synth.orbit_camera(1, w, h)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    inv = torch.from_numpy(np.linalg.inv(vp)).to("cuda", torch.float64)
    ys, xs = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64),
                            torch.arange(w, device="cuda", dtype=torch.float64), indexing="ij")
    ph = torch.rand(2, generator=gen, device="cuda", dtype=torch.float64) * 6.0
    depth = 0.94 + 0.04 * torch.sin(xs / w * 6.0 + ph[0]) * torch.cos(ys / h * 5.0 + ph[1])
    clip = torch.stack([(xs + 0.5) / w * 2 - 1, 1 - (ys + 0.5) / h * 2, depth, torch.ones_like(depth)])
    world = torch.einsum("ab,bhw->ahw", inv, clip)
    world = (world[:3] / world[3]).float()
    miss = torch.rand(h, w, generator=gen, device="cuda") < 0.1
    world = torch.where(miss[None], torch.full_like(world, float("nan")), world)
    return samples, world.contiguous(), synth.orbit_camera(0, w, h)


def session_state(case, seed):
    """A state such as a stream holds: models, positive definite P and features of smooth size."""
    w, h = case["width"], case["height"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    st = torch.empty(wrls.N_STATE, h, w, device="cuda")
    st[:12] = 0.4 * torch.randn(12, h, w, generator=gen, device="cuda")
    # P = L L^T, its condition in the hundreds at most as the recursion's is
    low = 0.2 * torch.randn(4, 4, h, w, generator=gen, device="cuda")
    low = low * torch.ones(4, 4, device="cuda").tril(-1)[:, :, None, None]
    low = low + torch.diag_embed(0.4 + 0.4 * torch.rand(h, w, 4, generator=gen, device="cuda")).permute(2, 3, 0, 1)
    p = (low[:, None].double() * low[None].double()).sum(2).float()
    k = 12
    for a in range(4):
        for b in range(a, 4):
            st[k] = p[a, b]
            k += 1
    st[22:] = torch.rand(3, h, w, generator=gen, device="cuda")
    return st


# ---- one pass ------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "inputs":
        samples, world, prev = raw_inputs(case, seed)
        _, _, h, w = samples.shape
        return {"kind": kind, "samples": samples, "world": world, "prev": prev,
                "radiance": torch.empty(3, h, w, device="cuda"), "motion": torch.empty(2, h, w, device="cuda"),
                "variance": torch.empty(h, w, device="cuda") if case["variance"] else None}
    if kind == "render":
        w, h, spp = case["width"], case["height"], case["spp"]
        return {"kind": kind, "scene": wrls.vpt_scene_struct(synth.vpt_scene(w, h, t=seed % 97, seed=seed)),
                "samples": torch.empty(spp, 5, h, w, device="cuda"), "world": torch.empty(3, h, w, device="cuda"),
                "features": torch.empty(7, h, w, device="cuda") if case["features"] else None}
    if kind == "session":
        st = session_state(case, seed)
        return {"kind": kind, "state": st, "back": torch.empty_like(st),
                "stream": wrls.Stream(case["width"], case["height"], params_of(case))}
    if kind == "tick":
        frames = mix_inputs(case, seed)
        streams = [wrls.Stream(w, h, params_of(case)) for w, h in MIX[-case["streams"]:]]
        outs = [torch.empty(3, s.height, s.width, device="cuda") for s in streams]
        s = {"kind": kind, "frames": frames, "streams": streams, "outs": outs, "at": 0,
             "batch": Batch(len(streams))}
        for _ in range(case["history"]):
            run(s)
        return s
    ring = denoise_inputs(case, seed)
    w, h, n = case["width"], case["height"], case["frames"]
    s = {"kind": kind, "n": n, "at": 0, "live": case["history"] > 0,
         "stream": wrls.Stream(w, h, params_of(case))}
    if kind == "host":
        s["ring"] = [tuple(None if t is None else t.cpu().pin_memory() for t in f) for f in ring]
        s["out"] = torch.empty(n, 3, h, w).pin_memory()
    else:
        s["ring"] = ring
        s["out"] = torch.empty(n, 3, h, w, device="cuda")
    s["outs"] = list(s["out"])
    if s["live"]:
        dst = torch.empty(3, h, w, device="cuda")
        for k in range(case["history"]):
            rad, var, feat, mot = ring[k]
            s["stream"].denoise(rad, mot, dst, variance=var, features=feat)
        s["at"] = case["history"]
    return s


class Batch:
    """Owns one batch executor."""

    def __init__(self, n):
        self.handle = wrls.wrls_batch_create(n)

    def __del__(self):
        wrls.wrls_batch_destroy(self.handle)


def run(state):
    kind = state["kind"]
    if kind == "inputs":
        wrls.wrls_reconstruct(state["samples"], state["radiance"], state["variance"])
        wrls.wrls_velocity_from_world(state["world"], state["prev"], state["motion"])
        out = {"radiance": state["radiance"], "motion": state["motion"]}
        if state["variance"] is not None:
            out["variance"] = state["variance"]
        return out
    if kind == "render":
        wrls.wrls_render_vpt(state["scene"], state["samples"], state["world"], state["features"], frame=1)
        out = {"samples": state["samples"], "world": state["world"]}
        if state["features"] is not None:
            out["features"] = state["features"]
        return out
    if kind == "session":
        state["stream"].write_state(state["state"])
        state["stream"].read_state(state["back"])
        return state["back"]
    if kind == "tick":
        k = state["at"] % len(state["frames"][0])
        state["at"] += 1
        wrls.wrls_batch_tick(state["batch"].handle, [(s.handle, f[k][0], None, None, f[k][1], o) for s, f, o in
                                                     zip(state["streams"], state["frames"], state["outs"])])
        return state["outs"]
    s, ring, n = state["stream"], state["ring"], state["n"]
    if not state["live"]:
        s.reset()
        state["at"] = 0
    if kind == "frame":
        for k in range(n):
            rad, var, feat, mot = ring[(state["at"] + k) % len(ring)]
            s.denoise(rad, mot, state["outs"][k], variance=var, features=feat)
    else:
        io = [ring[(state["at"] + k) % len(ring)] + (state["outs"][k],) for k in range(n)]
        (wrls.wrls_denoise_sequence if kind == "sequence" else wrls.wrls_denoise_sequence_host)(s.handle, io)
    state["at"] += n
    return state["out"]


# ---- what a pass cannot do without ------------------------------------------------------------

def planes_of(case):
    """(state values a pixel, bytes of one stored state a pixel)"""
    d = (4 if case.get("feature_mode", 0) == 0 else 1) + case.get("n_gbuf", 0)
    if case.get("n_gbuf", 0) or case.get("weight_mode", 0) == 2 or case.get("reproj_filter", 0):
        n = 3 * d + d * (d + 1) // 2 + 3
        return d, n, 4 * n
    return 4, 25, 100 if case["state"] == "f32" else 52


def denoise_work(pixels, case, frames, restarts):
    d, n, stored = planes_of(case)
    var, g = (case.get("weight_mode", 0) == 2), case.get("n_gbuf", 0)
    # state out, radiance and motion in, colour out; state in except on a restarted frame
    nbytes = pixels * (frames * (stored + 20 + 12 + 4 * var + 4 * g) + (frames - restarts) * stored)
    # four taps of n values; Eq. 8-14 (P p, the rank-1 updates of P and of three models); 25 neighbours
    flops = pixels * frames * (8 * n + 3 * d * d + 14 * d + 60 + 25 * (6 * d + 16))
    return {"bytes": nbytes, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "tick":
        return denoise_work(sum(w * h for w, h in MIX[-case["streams"]:]), case, 1, 0)
    px = case["width"] * case["height"]
    if kind == "inputs":
        spp = case["spp"]
        return {"bytes": px * (20 * spp + 12 + 4 * case["variance"] + 20), "flops": px * (9 * spp * 15 + 20 * spp + 45)}
    if kind == "render":
        # about 15 tentative collisions a sample, each a density of 12 Gaussians and a random number
        return {"bytes": px * (20 * case["spp"] + 12 + 28 * case["features"]), "flops": px * case["spp"] * 15 * 320}
    if kind == "session":
        stored = 100 if case["state"] == "f32" else 52
        return {"bytes": px * (200 + 2 * stored), "flops": px * 80}
    return denoise_work(px, case, case["frames"], 0 if case["history"] else 1)


# about four times the measured distance from 64 bits (1.3e-7, 2.8e-4 and 2.3e-3 of the result); "max" is
# a single channel of a firefly's neighbourhood, whose colour can cancel
DENOISE_TOL = {"f32": {"rel": 1e-6, "max": 1e-4}, "f16": {"rel": 1.2e-3, "max": 0.05},
               "bf16": {"rel": 1e-2, "max": 0.4}}
SESSION_TOL = {"f32": {"rel": 1e-7, "max": 1e-6}, "f16": {"rel": 2e-3, "max": 2e-2}, "bf16": {"rel": 1e-2, "max": 0.1}}


def tolerance(case):
    kind = case["kind"]
    if kind == "inputs":
        # measured against 64 bits: motion 1e-5 (a difference of two positions), colour and variance 1e-7
        return {"rel": 4e-5, "max": 4e-3}
    if kind == "render":
        # the decisions have to be the same, so that only the last bits of colours can move
        return {"rel": 1e-5, "max": 1e-3}
    if kind == "session":
        return SESSION_TOL[case["state"]]
    return DENOISE_TOL[case["state"]]


# ---- the same in 64 bits --------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "inputs":
        return exact_inputs(case, seed)
    if kind == "render":
        return None  # paths branch on random thresholds: another precision takes other paths
    if kind == "session":
        return session_state(case, seed).double()
    if kind == "tick":
        return [exact_denoise(dict(case, n_gbuf=0, weight_mode=0, blend_mode=0, feature_mode=0, reproj_filter=0),
                              [(f[0], None, None, f[1]) for f in fr], case["history"] + 1)[-1]
                for fr in mix_inputs(case, seed)]
    outs = exact_denoise(case, denoise_inputs(case, seed), case["history"] + case["frames"])
    return torch.stack(outs[case["history"]:])


def exact_denoise(case, ring, count):
    p = wrls.wrls_params_default()
    lam, hb, alpha, eps = (float(v) for v in (p.lambda_, p.h, p.alpha, p.eps))
    feat, g = case["feature_mode"] == 0, case["n_gbuf"]
    d = (4 if feat else 1) + g
    dev = "cuda"
    outs, beta, P, z = [], None, None, None
    for t in range(count):
        rad, var, gb, mot = ring[t % len(ring)]
        I = rad.double()
        H, W = I.shape[1:]
        ys, xs = torch.meshgrid(torch.arange(H, device=dev), torch.arange(W, device=dev), indexing="ij")
        # positions are 32-bit by definition: they decide which pixel is read
        qx, qy = xs.float() + mot[0], ys.float() + mot[1]
        ok = (qx >= 0) & (qx <= W - 1) & (qy >= 0) & (qy <= H - 1)
        if t == 0:
            ok = torch.zeros_like(ok)
        nb, nP = torch.zeros(3, d, H, W, dtype=torch.float64, device=dev), torch.zeros(d, d, H, W, dtype=torch.float64, device=dev)
        nP += torch.eye(d, device=dev, dtype=torch.float64)[:, :, None, None] * float(p.p0_delta)
        nz = I.clone()
        if t:
            cx, cy = torch.where(ok, qx, torch.zeros_like(qx)), torch.where(ok, qy, torch.zeros_like(qy))
            if case["reproj_filter"]:
                x0, y0 = torch.floor(cx + 0.5).long(), torch.floor(cy + 0.5).long()
                pick = [(x0, y0, torch.ones_like(cx, dtype=torch.float64))]
            else:
                x0, y0 = torch.floor(cx).long(), torch.floor(cy).long()
                fx, fy = cx.double() - x0, cy.double() - y0
                x1, y1 = (x0 + 1).clamp(max=W - 1), (y0 + 1).clamp(max=H - 1)
                pick = [(x0, y0, (1 - fx) * (1 - fy)), (x1, y0, fx * (1 - fy)), (x0, y1, (1 - fx) * fy), (x1, y1, fx * fy)]
            rb, rP, rz = torch.zeros_like(nb), torch.zeros_like(nP), torch.zeros_like(nz)
            for px, py, w in pick:
                rb += w * beta[:, :, py, px]
                rP += w * P[:, :, py, px]
                rz += w * z[:, py, px]
            pad = torch.nn.functional.pad(I[None], (1, 1, 1, 1), value=float("inf"))[0]
            lo = torch.stack([pad[:, a:a + H, b:b + W] for a in range(3) for b in range(3)]).amin(0)
            pad = torch.nn.functional.pad(I[None], (1, 1, 1, 1), value=-float("inf"))[0]
            hi = torch.stack([pad[:, a:a + H, b:b + W] for a in range(3) for b in range(3)]).amax(0)
            rz = alpha * torch.minimum(torch.maximum(rz, lo), hi) + (1 - alpha) * I
            nb, nP, nz = torch.where(ok, rb, nb), torch.where(ok, rP, nP), torch.where(ok, rz, nz)
            del rb, rP, rz
        beta, P, z = nb, nP, nz
        one = torch.ones(1, H, W, dtype=torch.float64, device=dev)
        pr = torch.cat([one] + ([z] if feat else []) + ([gb.double()] if g else []))
        m = torch.minimum(I.norm(dim=0), z.norm(dim=0)) + eps
        if case["weight_mode"] == 1:
            w = torch.ones_like(m)
        elif case["weight_mode"] == 2:
            w = torch.exp(-3 * var.double() / (m * m * hb * hb))
        else:
            w = torch.exp(-((I - z) ** 2).sum(0) / (m * m * hb * hb))
        k = (P * pr[None]).sum(1)
        gain = w / (lam + w * (pr * k).sum(0))
        beta = beta + (gain * (I - (beta * pr[None]).sum(1)))[:, None] * k[None]
        P = (P - gain * k[:, None] * k[None]) / lam
        # 5x5 blend
        num, den = torch.zeros_like(I), torch.zeros_like(m)
        nz_ = z.norm(dim=0)
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                a, b = slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx))
                c, e = slice(max(0, dy), H + min(0, dy)), slice(max(0, dx), W + min(0, dx))
                dist = ((z[:, a, b] - z[:, c, e]) ** 2).sum(0) / (torch.minimum(nz_[a, b], nz_[c, e]) + eps) ** 2
                wt = torch.exp(-(dx * dx + dy * dy) / (2.0 * float(p.sigma_s) ** 2) - dist / float(p.h_s) ** 2)
                who = pr[:, a, b] if case["blend_mode"] == 0 else pr[:, c, e]
                num[:, a, b] += wt * (beta[:, :, c, e] * who[None]).sum(1)
                den[a, b] += wt
        outs.append(num / den)
    return outs


def exact_inputs(case, seed):
    samples, world, prev = raw_inputs(case, seed)
    spp, _, H, W = samples.shape
    s = samples.double()
    rp = wrls.wrls_recon_params_default()
    num, den = torch.zeros(3, H, W, dtype=torch.float64, device="cuda"), torch.zeros(H, W, dtype=torch.float64, device="cuda")
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            a, b = slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx))
            c, e = slice(max(0, dy), H + min(0, dy)), slice(max(0, dx), W + min(0, dx))
            for k in range(spp):
                # the support is tested in 32 bits by definition
                fx, fy = dx + samples[k, 3, c, e], dy + samples[k, 4, c, e]
                ux, uy = dx + s[k, 3, c, e], dy + s[k, 4, c, e]
                w = torch.exp(-(ux * ux + uy * uy) / (2.0 * float(rp.sigma) ** 2))
                w = torch.where((fx.abs() <= rp.radius) & (fy.abs() <= rp.radius), w, torch.zeros_like(w))
                num[:, a, b] += w * s[k, :3, c, e]
                den[a, b] += w
    out = {"radiance": num / den}
    X = world.double()
    M = torch.from_numpy(np.asarray(prev, np.float32)).double().cuda()
    clip = torch.einsum("ab,bhw->ahw", M[:, :3], X) + M[:, 3][:, None, None]
    ys, xs = torch.meshgrid(torch.arange(H, device="cuda", dtype=torch.float64),
                            torch.arange(W, device="cuda", dtype=torch.float64), indexing="ij")
    vx = (clip[0] / clip[3] + 1) * W / 2 - 0.5 - xs
    vy = (1 - clip[1] / clip[3]) * H / 2 - 0.5 - ys
    mot = torch.stack([vx, vy])
    behind = ~(clip[3] > 0)
    mot = torch.where(behind[None], torch.full_like(mot, float("nan")), mot)
    out["motion"] = torch.where(torch.isfinite(X).all(0)[None], mot, torch.zeros_like(mot))
    if case["variance"]:
        if spp < 2:
            out["variance"] = torch.full((H, W), float("nan"), dtype=torch.float64, device="cuda")
        else:
            out["variance"] = s[:, :3].var(dim=0, unbiased=True).mean(0) / spp
    return out
