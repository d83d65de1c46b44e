"""The work that programs have this renderer do, as a list of timed cases.

Every case goes through the public entry points (`api.Renderer`,
`api.render_events_batch`, `api.EventFrames`, `api.event_quality` and the C
call `mcev_detect_batch_static`).  The kinds:

* frame     one frame of the event-camera loop (Alg. 1): the program holds the
            reference statistics of the previous frame as a checkpoint, renders
            the pair (t0, t1) and keeps events, sample counts, means and the
            updated reference;
* batch     the same for several independent cameras and scenes in one call;
* reference the first frame of the loop: every pixel at one sample count;
* samples   raw path samples of chosen pixels with their decision signatures;
* gradient  one step of inverse rendering: two mean images, the event loss and
            the gradients of texture and emission;
* quality   scoring one event video against another;
* detect    the allocation-free detector step on a caller's own path samples.
"""
import ctypes
import math
import random

import numpy as np
import torch

import scenegen as sg
from paper_2408_07996_gb300 import _lib as L
from paper_2408_07996_gb300.api import EventFrames, Renderer, event_loss, event_quality, render_events_batch


def listed():
    return [
        # the smallest frame: a 64x64 Cornell box, where launches and host latency are all there is
        dict(name="frame_indoor_64", kind="frame", scene="indoor", width=64, height=64, spp_min=16, spp_batch=16,
             spp_max=256, spp_ref=256, C=0.2, alpha=0.05, depth=4, variant=0, se_mode=0),
        # object motion at an ordinary size: 64 displaced spheres (327k triangles), one of them spinning
        dict(name="frame_objects_512", kind="frame", scene="spheres", width=512, height=512, n_spheres=64, level=4,
             n_spin=1, spp_min=256, spp_batch=32, spp_max=4096, spp_ref=4096, C=0.25, alpha=0.01, depth=4,
             variant=0, se_mode=0),
        # many moving objects (a per-frame instance hierarchy) on a 346x260 event-camera sensor, Welch standard error
        dict(name="frame_moving_346", kind="frame", scene="spheres", width=346, height=260, n_spheres=24, level=3,
             n_spin=12, spp_min=64, spp_batch=16, spp_max=1024, spp_ref=1024, C=0.2, alpha=0.05, depth=4,
             variant=0, se_mode=1),
        # the headline frame: camera flight over a 2.1M-triangle terrain with glossy patches, 1280x720
        dict(name="frame_terrain_720p", kind="frame", scene="terrain", width=1280, height=720, grid=1024, n_boxes=200,
             spp_min=512, spp_batch=64, spp_max=8192, spp_ref=2048, C=0.2, alpha=0.05, depth=6, variant=0, se_mode=0),
        # dataset generation: eight small sensors and scenes rendered together
        dict(name="batch_8", kind="batch", jobs=8, spp_min=16, spp_batch=16, spp_max=2048, C=0.2, alpha=0.05, depth=4),
        # start of a video on an odd-sized image: the reference frame at a fixed sample count
        dict(name="reference_641", kind="reference", scene="terrain", width=641, height=361, grid=512, n_boxes=60,
             spp=512, C=0.2, alpha=0.05, depth=5),
        # offline analysis of the sample distribution of a few thousand pixels, with decision signatures
        dict(name="samples_5001", kind="samples", scene="spheres", width=346, height=260, n_spheres=40, level=3,
             n_spin=1, n_pix=5001, k0=16, count=96, depth=4),
        # inverse rendering of texture and lights: forward at two times, loss, backward
        dict(name="gradient_256", kind="gradient", width=256, height=256, grid=158, tex=512, spp=64, depth=3),
        # scoring a 100-frame 720p event video
        dict(name="quality_720p", kind="quality", width=1280, height=720, frames=100, tau2=3, want_d2=False),
        # scoring a short odd-sized clip, with the per-event distances
        dict(name="quality_clip", kind="quality", width=203, height=199, frames=31, tau2=3, want_d2=True),
        # a host application's own 346x260 sensor: the rest of a frame's samples through the detector step
        dict(name="detect_346", kind="detect", width=346, height=260, spp_min=16, spp_batch=16, spp_max=256,
             C=0.2, alpha=0.05, variant=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["frame", "frame", "frame", "batch", "reference", "samples", "gradient", "quality", "quality",
                       "detect"])
    if kind in ("frame", "reference", "samples"):
        scene = rng.choice(["indoor", "spheres", "terrain"])
        case = dict(kind=kind, scene=scene, width=_log(rng, 33, 640), height=_log(rng, 31, 480), C=0.2,
                    alpha=rng.choice([0.01, 0.05]), depth=rng.randint(2, 6))
        if scene == "spheres":
            case.update(n_spheres=rng.randint(1, 48), level=rng.randint(2, 4))
            case["n_spin"] = rng.randint(0, case["n_spheres"])
        elif scene == "terrain":
            case.update(grid=_log(rng, 48, 512), n_boxes=rng.randint(0, 120))
        if kind == "frame":
            sub = rng.choice([16, 24, 32, 64])
            spp_max = _log(rng, 128, 4096)
            case.update(spp_min=rng.choice([16, 64, 100]), spp_batch=sub, spp_max=spp_max, spp_ref=min(spp_max, 1024),
                        variant=rng.choice([0, 0, 0, 1, 2, 3]), se_mode=rng.choice([0, 0, 1]))
        elif kind == "reference":
            case["spp"] = _log(rng, 32, 1024)
        else:
            case.update(n_pix=min(_log(rng, 100, 20000), case["width"] * case["height"]), k0=rng.randint(0, 300),
                        count=_log(rng, 16, 256))
        return case
    if kind == "batch":
        return dict(kind=kind, jobs=rng.randint(2, 8), spp_min=16, spp_batch=rng.choice([16, 32]),
                    spp_max=_log(rng, 256, 2048), C=0.2, alpha=rng.choice([0.01, 0.05]), depth=rng.randint(3, 5))
    if kind == "gradient":
        return dict(kind=kind, width=_log(rng, 64, 320), height=_log(rng, 64, 320), grid=_log(rng, 24, 200),
                    tex=rng.choice([64, 200, 512]), spp=_log(rng, 16, 128), depth=rng.randint(2, 4))
    if kind == "quality":
        return dict(kind=kind, width=_log(rng, 64, 1280), height=_log(rng, 48, 720), frames=_log(rng, 5, 100),
                    tau2=rng.choice([0, 1, 3, 9]), want_d2=rng.random() < 0.5)
    sub = rng.choice([16, 32, 64])
    return dict(kind=kind, width=_log(rng, 64, 640), height=_log(rng, 48, 480), spp_min=rng.choice([16, 64]),
                spp_batch=sub, spp_max=_log(rng, 160, 512), C=0.2, alpha=rng.choice([0.01, 0.05]),
                variant=rng.choice([0, 0, 1, 2]))


# ------------------------------------------------------------------ inputs
def _scene(case, seed):
    s = 1000 + seed
    if case["scene"] == "indoor":
        return sg.cornell_box(s), (0.0, 1.0), 2e-4
    if case["scene"] == "spheres":
        sc = sg.icosphere_field(s, n_spheres=case["n_spheres"], level=case["level"], n_frames=9, dt=4e-3,
                                n_spin=case["n_spin"], env_w=256, env_h=128)
        k = seed % 8
        return sc, (sc.key_times[k], sc.key_times[k + 1]), 1e-3
    sc = sg.terrain_with_boxes(s, grid=case["grid"], n_boxes=case["n_boxes"], n_frames=100)
    k = (7 * seed) % 99
    return sc, (sc.key_times[k], sc.key_times[k + 1]), 1e-2


def _renderer(case, scene, t_min, seed, spp_min=16):
    r = Renderer(case["width"], case["height"])
    r.upload(scene)
    r.set_params(t_min=t_min, max_depth=case["depth"], seed=20240815 + seed, spp_min=spp_min,
                 variant=case.get("variant", 0), se_mode=case.get("se_mode", 0))
    return r


def _videos(case, seed):
    """Events of a drifting grating seen by an ideal log sensor, and the same
    with events moved, dropped, flipped and added (what a cheaper renderer of
    the same scene gives)."""
    W, H, T = case["width"], case["height"], case["frames"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = np.random.default_rng(seed)
    kx, ky = rnd.uniform(0.02, 0.08, 2)
    vx, vy = rnd.uniform(0.3, 1.5, 2)
    x = torch.arange(W, device="cuda", dtype=torch.float64)
    y = torch.arange(H, device="cuda", dtype=torch.float64)[:, None]
    a = torch.empty((T, H, W), dtype=torch.int8, device="cuda")
    prev = None
    for t in range(T + 1):
        i = 0.5 + 0.25 * torch.sin(kx * (x - vx * t)) + 0.25 * torch.sin(ky * (y - vy * t) + 0.3 * torch.sin(0.05 * x))
        level = torch.floor(4.0 * i)
        if prev is not None:
            a[t - 1] = torch.sign(level - prev).to(torch.int8)
        prev = level
    at, ay, ax = torch.nonzero(a, as_tuple=True)
    pol = a[at, ay, ax]
    u = torch.rand(at.numel(), generator=g, device="cuda")
    pos = torch.stack([at, ay, ax])
    axis = torch.randint(0, 3, (at.numel(),), generator=g, device="cuda")
    step = 2 * torch.randint(0, 2, (at.numel(),), generator=g, device="cuda") - 1
    moved = (u >= 0.03) & (u < 0.08)
    pos = pos + torch.where(moved, step, 0) * (torch.arange(3, device="cuda")[:, None] == axis)
    lim = torch.tensor([T, H, W], device="cuda")[:, None]
    ok = (u >= 0.03) & ((pos >= 0) & (pos < lim)).all(0)
    pol = torch.where(torch.rand(at.numel(), generator=g, device="cuda") < 0.01, -pol, pol)
    flat = ((pos[0] * H + pos[1]) * W + pos[2])[ok]
    # events that meet in one voxel: their polarities add and are clipped, whatever the order
    tot = torch.zeros(T * H * W, dtype=torch.int32, device="cuda").index_add_(0, flat, pol[ok].to(torch.int32))
    b = tot.clamp_(-1, 1).to(torch.int8)
    n_extra = max(1, int(2e-4 * b.numel()))
    where = torch.randint(0, b.numel(), (n_extra,), generator=g, device="cuda")
    b[where] = 1
    b[where[: n_extra // 2]] = -1
    return a, b.view(T, H, W)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("frame", "reference", "samples"):
        scene, (t0, t1), t_min = _scene(case, seed)
        r = _renderer(case, scene, t_min, seed, case.get("spp_min", 16))
        st.update(r=r, t0=float(t0), t1=float(t1))
        if kind == "frame":
            r.render_reference(t0, case["spp_ref"])
            st["ref"] = r.get_state()
        elif kind == "samples":
            rng = np.random.default_rng(seed)
            pix = rng.choice(case["width"] * case["height"], case["n_pix"], replace=False).astype(np.int32)
            st["pixels"] = torch.from_numpy(pix).cuda()
        return st
    if kind == "batch":
        rng = np.random.default_rng(seed)
        runner = Renderer(8, 8)
        jobs = []
        for j in range(case["jobs"]):
            w, h = sg.BATCH_RESOLUTIONS[j % len(sg.BATCH_RESOLUTIONS)]
            level = 3 + (j // 4) % 2
            n = int(rng.integers(4, 60)) if level == 3 else int(rng.integers(2, 16))
            sc = sg.icosphere_field(5000 + 64 * seed + j, n_spheres=n, level=level, n_frames=9, dt=2e-3, env_w=128,
                                    env_h=64)
            shift = np.linspace(0.0, 0.08, 9)[:, None] * np.array([1.0, 0.0, 0.0])
            sc.cam_eye = sc.cam_eye + shift
            sc.cam_target = sc.cam_target + shift
            jobs.append((_renderer(dict(case, width=w, height=h), sc, 1e-3, seed + j), sc.key_times))
        # the program's frames so far, then a checkpoint before the frame in hand
        render_events_batch(runner, [(r, t[0], t[1]) for r, t in jobs], case["C"], case["alpha"], 64,
                            min(256, case["spp_max"]))
        st.update(runner=runner, jobs=[(r, float(t[1]), float(t[2])) for r, t in jobs],
                  refs=[r.get_state() for r, _ in jobs])
        return st
    if kind == "gradient":
        sc = sg.textured_room(3000 + seed, grid=case["grid"], tex_size=case["tex"])
        r = Renderer(case["width"], case["height"])
        r.upload(sc)
        r.set_params(t_min=6e-4, max_depth=case["depth"], seed=20240815 + seed)
        rng = np.random.default_rng(seed)
        target = (np.sign(rng.normal(size=(case["height"], case["width"]))) *
                  (rng.random((case["height"], case["width"])) < 0.2)).astype(np.int8)
        st.update(r=r, texture=torch.from_numpy(sc.texture).cuda().requires_grad_(True),
                  emission=torch.from_numpy(sc.mat_emit).cuda().requires_grad_(True),
                  target=torch.from_numpy(target).cuda())
        return st
    if kind == "quality":
        st["a"], st["b"] = _videos(case, seed)
        return st
    # detect: log-normal path radiances with some black paths, as a diffuse scene gives them; a twentieth of the
    # pixels has brightened or darkened since its reference
    n = case["width"] * case["height"]
    k = case["spp_max"] - case["spp_min"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    level = 0.5 * normal(n)
    sigma = 0.1 + 0.5 * torch.rand(n, generator=g, device="cuda")
    jump = torch.where(torch.rand(n, generator=g, device="cuda") < 0.05, 0.5 * normal(n), 0.02 * normal(n))
    st["L"] = torch.exp((level + jump)[:, None] + sigma[:, None] * normal(n, k))
    st["L"][torch.rand((n, k), generator=g, device="cuda") < 0.01] = 0.0
    state = torch.empty((6, n), dtype=torch.int32, device="cuda")
    first = torch.log(torch.exp((level + jump)[:, None] + sigma[:, None] * normal(n, case["spp_min"])) + 1e-3)
    state[0] = case["spp_min"]
    state[1] = first.mean(1).view(torch.int32)
    state[2] = (first.var(1) * (case["spp_min"] - 1)).view(torch.int32)
    state[3] = case["spp_max"]
    state[4] = (level + sigma / math.sqrt(case["spp_max"]) * normal(n)).view(torch.int32)
    state[5] = (sigma * sigma * (case["spp_max"] - 1)).view(torch.int32)
    st.update(state0=state, state=state.clone(), pixels=torch.randperm(n, generator=g, device="cuda").to(torch.int32),
              events=torch.zeros(n, dtype=torch.int8, device="cuda"),
              spp=torch.zeros(n, dtype=torch.int32, device="cuda"), mean=torch.zeros(n, device="cuda"),
              undecided=torch.zeros(n, dtype=torch.int32, device="cuda"))
    return st


# ------------------------------------------------------------------ one pass
def _state_out(r):
    n, mean, m2 = r.reference_arrays()
    return [n, mean, m2]


_QUALITY = ("n_a", "n_b", "matched_a", "matched_b", "none_a", "none_b", "sq_diff", "sum_dist_a", "sum_dist_b", "diag",
            "rmse", "psnr", "precision", "recall", "f1", "pscd")


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "frame":
        r = st["r"]
        r.set_state(st["ref"])
        o = r.render_events(st["t0"], st["t1"], case["C"], case["alpha"], case["spp_batch"], case["spp_max"])
        return [o["events"], o["spp"], o["mean"], _state_out(r)]
    if kind == "batch":
        for (r, _, _), ref in zip(st["jobs"], st["refs"]):
            r.set_state(ref)
        outs, _ = render_events_batch(st["runner"], st["jobs"], case["C"], case["alpha"], case["spp_batch"],
                                      case["spp_max"])
        return [[o["events"], o["spp"], o["mean"], _state_out(r)] for o, (r, _, _) in zip(outs, st["jobs"])]
    if kind == "reference":
        st["r"].render_reference(st["t0"], case["spp"])
        return _state_out(st["r"])
    if kind == "samples":
        radiance, sig = st["r"].trace_samples(st["t1"], st["pixels"], case["k0"], case["count"])
        return [radiance, sig]
    if kind == "gradient":
        tex, emi = st["texture"], st["emission"]
        tex.grad = emi.grad = None
        m0, m1 = EventFrames.apply(tex, emi, st["r"], 0.0, 1.0, case["spp"])
        loss = event_loss(m0, m1, st["target"], 0.2)
        loss.backward()
        return [m0.detach(), m1.detach(), loss.detach(), tex.grad, emi.grad]
    if kind == "quality":
        q = event_quality(st["a"], st["b"], tau2=case["tau2"], want_d2=case["want_d2"])
        out = {k: q[k] for k in _QUALITY}
        if case["want_d2"]:
            out.update(d2_a=q["d2_a"], d2_b=q["d2_b"])
        return out
    n = case["width"] * case["height"]
    s = st["state"]
    s.copy_(st["state0"])
    p = [ctypes.c_void_p(s[i].data_ptr()) for i in range(6)]
    args = L.DetectArgs(L=st["L"].data_ptr(), pixels=st["pixels"].data_ptr(), n_pix=n, n_total=n,
                        spp_r=case["spp_max"] - case["spp_min"], reserved0=0, k_base=case["spp_min"],
                        cur_n=p[0], cur_mean=p[1], cur_m2=p[2], ref_n=p[3], ref_mean=p[4], ref_m2=p[5],
                        events=st["events"].data_ptr(), spp_out=st["spp"].data_ptr(), mean_out=st["mean"].data_ptr(),
                        undecided=st["undecided"].data_ptr(), eps=1e-3, C=case["C"], alpha=case["alpha"],
                        spp_min=case["spp_min"], spp_batch=case["spp_batch"], spp_max=case["spp_max"],
                        variant=case["variant"], se_mode=0,
                        stream=ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    und = ctypes.c_int64(-1)
    L.check(L.load().mcev_detect_batch_static(ctypes.byref(args), ctypes.byref(und)), None, "mcev_detect_batch_static")
    return [st["events"], st["spp"], st["mean"], s[0], s[1].view(torch.float32), s[2].view(torch.float32), s[3],
            s[4].view(torch.float32), s[5].view(torch.float32), und.value]


# ------------------------------------------------------------------ what a pass cannot do without
def _triangles(case):
    if case["scene"] == "indoor":
        return 32
    if case["scene"] == "spheres":
        return case["n_spheres"] * 20 * 4 ** case["level"] + 2
    return 2 * (case["grid"] - 1) ** 2 + 12 * case["n_boxes"]


def _paths(n_paths, tris):
    """FLOP of n_paths path samples: at least one closest-hit and one shadow
    ray each, one two-box node (24 FLOP) per level of the hierarchy and one
    triangle test (25 FLOP) per ray."""
    return 2.0 * n_paths * (24.0 * math.log2(max(2, tris)) + 25.0)


def work(case):
    kind = case["kind"]
    if kind in ("frame", "reference", "samples"):
        n, tris = case["width"] * case["height"], _triangles(case)
        scene = 48 * tris
        if kind == "frame":
            # the reference in, the updated one, events, counts and means out; every pixel draws spp_min samples
            return dict(bytes=scene + 33 * n, flops=_paths(n * case["spp_min"], tris))
        if kind == "reference":
            return dict(bytes=scene + 12 * n, flops=_paths(n * case["spp"], tris))
        m = case["n_pix"] * case["count"]
        return dict(bytes=scene + 4 * case["n_pix"] + 8 * m, flops=_paths(m, tris))
    if kind == "batch":
        n = sum(w * h for w, h in (sg.BATCH_RESOLUTIONS[j % 4] for j in range(case["jobs"])))
        tris = 40000
        return dict(bytes=48 * tris * case["jobs"] + 33 * n, flops=_paths(n * case["spp_min"], tris))
    if kind == "gradient":
        n, tris = case["width"] * case["height"], 2 * (case["grid"] - 1) ** 2
        # two forward frames and their replays
        return dict(bytes=48 * tris + 17 * n + 24 * case["tex"] ** 2, flops=4 * _paths(n * case["spp"], tris))
    if kind == "quality":
        n = case["width"] * case["height"] * case["frames"]
        return dict(bytes=(10 if case["want_d2"] else 2) * n, flops=0)
    n, k = case["width"] * case["height"], case["spp_max"] - case["spp_min"]
    return dict(bytes=4 * n * k + (4 + 24 + 24 + 9) * n, flops=5.0 * n * k)


# ------------------------------------------------------------------ 64-bit values
def _sq_dist(mask):
    """Squared distance of every voxel to the nearest set voxel (2^30: none)."""
    inf = 1 << 30
    T, H, W = mask.shape
    x = torch.arange(W, device=mask.device).expand(mask.shape)
    left = torch.where(mask, x, -inf).cummax(2).values
    right = -torch.where(mask, x, inf).flip(2).neg().cummax(2).values.flip(2)
    d = torch.minimum(x - left, right - x).clamp_(max=1 << 14)
    best = torch.where(d >= 1 << 14, inf, d * d).to(torch.int32)
    for axis, ext in ((1, H), (0, T)):
        src, best = best, best.clone()
        for s in range(1, ext):
            if s * s >= int(best.max()):
                break
            hi, lo = best.narrow(axis, s, ext - s), best.narrow(axis, 0, ext - s)
            hi.copy_(torch.minimum(hi, src.narrow(axis, 0, ext - s) + s * s))
            lo.copy_(torch.minimum(lo, src.narrow(axis, s, ext - s) + s * s))
    return best.clamp_(max=inf)


def _quality_exact(case, seed):
    a, b = _videos(case, seed)
    T, H, W = a.shape
    diag = math.sqrt((W - 1) ** 2 + (H - 1) ** 2 + (T - 1) ** 2)
    out = dict(n_a=int((a != 0).sum()), n_b=int((b != 0).sum()),
               sq_diff=int(((a.to(torch.int32) - b.to(torch.int32)) ** 2).sum()), diag=diag)
    for key, q, v in (("a", a, b), ("b", b, a)):
        d2 = torch.full(a.shape, -1, dtype=torch.int32, device=a.device)
        for pol in (1, -1):
            d = _sq_dist(v == pol)
            d = torch.where(d >= 1 << 30, -2, d)
            d2 = torch.where(q == pol, d, d2)
        ev = d2[q != 0].to(torch.float64)
        out["matched_" + key] = int(((ev >= 0) & (ev <= case["tau2"])).sum())
        out["none_" + key] = int((ev < 0).sum())
        out["sum_dist_" + key] = float(torch.where(ev < 0, diag, ev.clamp(min=0).sqrt()).sum())
        out["d2_" + key] = d2
    mse = out["sq_diff"] / (4.0 * a.numel())
    out["rmse"] = math.sqrt(mse)
    out["psnr"] = -10.0 * math.log10(mse) if mse > 0 else math.inf
    out["precision"] = out["matched_a"] / out["n_a"] if out["n_a"] else 1.0
    out["recall"] = out["matched_b"] / out["n_b"] if out["n_b"] else 1.0
    pr = out["precision"] + out["recall"]
    out["f1"] = 2.0 * out["precision"] * out["recall"] / pr if pr > 0 else 0.0
    ma = out["sum_dist_a"] / out["n_a"] if out["n_a"] else 0.0
    mb = out["sum_dist_b"] / out["n_b"] if out["n_b"] else 0.0
    out["pscd"] = (ma + mb) / (2.0 * diag)
    keys = _QUALITY + (("d2_a", "d2_b") if case["want_d2"] else ())
    return {k: out[k] for k in keys}


def _t_quantile(p, nu):
    """p-quantile of Student's t with nu degrees of freedom (p < 1/2): the
    density integrated by Gauss-Legendre panels, inverted by bisection."""
    x, w = np.polynomial.legendre.leggauss(64)
    c = math.exp(math.lgamma(0.5 * (nu + 1)) - math.lgamma(0.5 * nu)) / math.sqrt(nu * math.pi)

    def below(t):          # P(T <= -t) = 1/2 - integral of the density over [0, t]
        s = 0.0
        for k in range(8):
            u = t * (k + 0.5 * (x + 1.0)) / 8.0
            s += float((w * (1.0 + u * u / nu) ** (-0.5 * (nu + 1))).sum()) * t / 16.0
        return 0.5 - c * s

    lo, hi = 0.0, 40.0
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if below(mid) > p else (lo, mid)
    return -0.5 * (lo + hi)


def _detect_exact(case, seed):
    st = prepare(case, seed)
    n_pix = case["width"] * case["height"]
    dt = torch.float64
    y = torch.log(st["L"].to(dt) + float(np.float32(1e-3)))
    pix = st["pixels"].long()
    s = st["state0"]
    f = [s[i][pix] if i in (0, 3) else s[i].view(torch.float32)[pix].to(dt) for i in range(6)]
    n, mean, m2 = f[0].to(dt), f[1], f[2]
    na, ma, va = f[3], f[4], f[5] / (f[3] - 1).to(dt)
    C = float(np.float32(case["C"]))
    alpha = float(np.float32(case["alpha"]))
    open_ = torch.ones(n_pix, dtype=torch.bool, device="cuda")
    k, col = case["spp_min"], 0
    while k < case["spp_max"]:
        sub = min(case["spp_batch"], case["spp_max"] - k)
        yb = y[:, col:col + sub]
        bm = yb.mean(1)
        b2 = ((yb - bm[:, None]) ** 2).sum(1)
        d = bm - mean
        tot = n + sub
        mean = torch.where(open_, mean + d * sub / tot, mean)
        m2 = torch.where(open_, m2 + b2 + d * d * n * sub / tot, m2)
        n = torch.where(open_, tot, n)
        k, col = k + sub, col + sub
        if k >= case["spp_max"]:
            break
        gap = (mean - ma).abs()
        if case["variant"] == 2:
            stop = gap < C
        else:
            t = (gap - C) / torch.sqrt((va + m2 / (n - 1)) / n)
            tc = _t_quantile(alpha if case["variant"] == 0 else 0.5 * alpha, k - 1)
            stop = t < tc if case["variant"] == 0 else (t < tc) | (t > -tc)
        open_ &= ~stop
    delta = mean - ma
    ev = torch.where(delta.abs() > C, torch.sign(delta), 0.0)
    hit = ev != 0

    def put(v, dtype):
        return torch.empty(n_pix, dtype=dtype, device="cuda").index_copy_(0, pix, v.to(dtype))

    return [put(ev, torch.int8), put(n, torch.int32), put(mean, dt), put(n, torch.int32), put(mean, dt), put(m2, dt),
            put(torch.where(hit, n, na.to(dt)), torch.int32), put(torch.where(hit, mean, ma), dt),
            put(torch.where(hit, m2, f[5]), dt), 0]


def exact(case, seed):
    if case["kind"] == "quality":
        return _quality_exact(case, seed)
    if case["kind"] == "detect":
        return _detect_exact(case, seed)
    # Monte Carlo path tracing: the 64-bit value needs a second renderer of the same random streams, minutes per frame
    return None
