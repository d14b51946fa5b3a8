"""Performance cases: the calls a program tracking surgical instruments makes.

Five kinds of call, each through the package's public entry points:

  eval   Tracker.eval_population on one population (losses and counts): what a
         program with its own optimiser or particle filter calls
  soft   soft_silhouette_loss, forward alone or with the backward pass through
         torch autograd: gradient refinement and gradient-based fitting
  search ask / eval_population / tell: CMA-ES with the population in the
         caller's hands (the stand-alone sampling and update)
  track  one camera frame: track_frame (mask on the device) or
         track_frame_host (mask in pinned host memory, with joint readings when
         there are two instruments)
  batch  Batch.track_frame: uneven instances tracked together
  serve  Server: camera streams with continuous batching

Images, meshes, population sizes and losses are the ones of this repository's
benchmark and tests: the 160x128 fit (about 1.5k triangles), the 640x512
tracking set (about 20k triangles, 64 candidates, 5 generations), the 700x493
paper-style set (look-at rotation, appearance and keypoint terms), and the
heterogeneous batch (320x256 to 1280x1024, 5k to 40k triangles, populations
to 256, one or two instruments).  Inputs are synthetic and seeded.
"""
import functools
import math

import numpy as np
import torch

from paper_2603_11404_gb300 import api
from paper_2603_11404_gb300 import workload as wl

LAMBDA_APP, KP_TAU, KP_LAMBDA = 0.5, 3.0, 5.0  # the weights of the paper-form benchmark
CUTOFF = 14.0  # reach of the soft silhouette in units of sigma


def _image(W, H, f):
    return {"W": W, "H": H, "f": float(f)}


C1, C2 = _image(160, 128, 200), _image(640, 512, 800)


def listed():
    return [
        # the smallest call: a population of the 160x128 fit
        dict(name="eval_160x128", kind="eval", mesh="c1", ni=1, lam=16, loss=wl.LOSS_XOR, rot=0, kp=False, **C1),
        # the ordinary fitness call: one generation of the 640x512 tracking set
        dict(name="eval_640x512", kind="eval", mesh="c2", ni=1, lam=64, loss=wl.LOSS_ONE_MINUS_IOU, rot=0, kp=False,
             **C2),
        # the paper's own objective on its odd image size (700 is no multiple of 32)
        dict(name="eval_700x493_paper", kind="eval", mesh="c2", ni=1, lam=64, loss=wl.LOSS_MSE_APP, rot=1, kp=True,
             **_image(700, 493, 700)),
        # the largest population: two instruments of 40k triangles each in a 1280x1024 image
        dict(name="eval_1280x1024_two", kind="eval", mesh="40000", ni=2, lam=256, loss=wl.LOSS_ONE_MINUS_IOU, rot=0,
             kp=False, **_image(1280, 1024, 1600)),
        # gradients of a whole population (gradient-based fitting)
        dict(name="soft_grad_640x512", kind="soft", mesh="c2", ni=1, lam=64, sigma=1.0, grad=True, **C2),
        # an optimiser's step on the best eight candidates: the small gradient call
        dict(name="soft_grad_top8", kind="soft", mesh="c2", ni=1, lam=8, sigma=1.0, grad=True, **C2),
        # the soft loss alone on the small fit, two instruments, odd image
        dict(name="soft_loss_101x77_two", kind="soft", mesh="800", ni=2, lam=32, sigma=1.0, grad=False,
             **_image(101, 77, 150)),
        # CMA-ES driven by the caller: two instruments, block-diagonal covariance
        dict(name="search_320x256_two", kind="search", mesh="5000", ni=2, lam=128, gens=3, **_image(320, 256, 400)),
        # a camera frame, mask on the device: the benchmark's step
        dict(name="track_640x512", kind="track", mesh="c2", ni=1, lam=64, gens=5, host=False, **C2),
        # a camera frame end to end from host memory, two instruments with joint readings
        dict(name="track_host_640x512_two", kind="track", mesh="c2", ni=2, lam=64, gens=5, host=True, **C2),
        # uneven instances tracked together
        dict(name="batch_24", kind="batch", n=24, gens=5, start=0),
        # eight camera streams, four frames each, submitted at once
        dict(name="serve_8_streams", kind="serve", streams=8, frames=4, lam=64, gens=5, mesh="c2", **C2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_image(rng, lo=101, hi=1280):
    W = _log(rng, lo, hi)
    H = max(64, int(W * rng.uniform(0.68, 0.82)))
    return _image(W, H, round(W * rng.uniform(1.0, 1.4), 1))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "soft", "soft", "search", "track", "track", "batch", "serve"])
    mesh = str(_log(rng, 1500, 40000))
    ni = rng.choice([1, 1, 2])
    if kind == "eval":
        img = _draw_image(rng)
        return dict(kind="eval", mesh=mesh, ni=ni, lam=_log(rng, 8, 256), loss=rng.choice([0, 1, 2]),
                    rot=rng.choice([0, 0, 1]), kp=rng.choice([False, False, True]), **img)
    if kind == "soft":
        img = _draw_image(rng, 101, 640)
        return dict(kind="soft", mesh=str(_log(rng, 800, 20000)), ni=ni, lam=_log(rng, 4, 64) // ni,
                    sigma=rng.choice([0.5, 1.0, 1.0]), grad=rng.choice([True, True, False]), **img)
    if kind == "search":
        return dict(kind="search", mesh=mesh, ni=ni, lam=_log(rng, 16, 256), gens=rng.randint(1, 4),
                    **_draw_image(rng, 101, 640))
    if kind == "track":
        return dict(kind="track", mesh=mesh, ni=ni, lam=_log(rng, 16, 128), gens=rng.randint(2, 10),
                    host=rng.choice([True, False]), **_draw_image(rng, 101, 960))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(3, 20), gens=rng.randint(2, 5), start=rng.randint(1, 23))
    return dict(kind="serve", streams=rng.randint(2, 8), frames=rng.randint(1, 4), lam=_log(rng, 16, 64),
                gens=rng.randint(2, 5), mesh=str(_log(rng, 1500, 20000)), **_draw_image(rng, 160, 640))


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _meshes(size):
    """The procedural instrument at one size (geometry: nothing in it depends on a seed)."""
    return wl.instrument_meshes(size)


def _scene(mesh, ni, W, H, f, rot=0):
    K = wl.Intrinsics(f, f, W / 2, H / 2, W, H)
    return wl.Scene(wl.instrument_frames(), _meshes(mesh), wl.Q_LB.copy(), wl.Q_UB.copy(), K, ni, rot)


def _case_scene(c):
    return _scene(c["mesh"], c["ni"], c["W"], c["H"], c["f"], c.get("rot", 0))


def _truth(rng, sc):
    return np.concatenate([wl.sample_state(rng, sc.K, rot_param=sc.rot_param) for _ in range(sc.n_instruments)])


def _observed(tr, state, rng):
    """The observed mask on the host: the silhouette at the true state, corrupted."""
    s = torch.from_numpy(state.astype(np.float32)).cuda()
    return wl.corrupt_mask(api.unpack_mask(tr.render(s), tr.width).cpu().numpy(), rng)


def _optimiser(tr, sc, lam, truth, rng, seed):
    start = truth + rng.normal(size=sc.d) * 0.5 * wl.default_scales(sc.d)
    return api.CMAES(tr, lam, start, wl.default_scales(sc.d), sigma0=1.0, seed=seed, block_diag=sc.d == 18)


def _readings(truth, rng, ni):
    """Joint readings with the encoder noise of the serving benchmark."""
    q = np.concatenate([truth[9 * b + 6: 9 * b + 9] for b in range(ni)])
    return (q + rng.normal(size=q.shape) * 0.02).astype(np.float32)


BATCH_IMAGES = [(320, 256), (640, 512), (960, 768), (1280, 1024)]
BATCH_LAMS = [32, 64, 128, 256]
BATCH_MESHES = ["5000", "10000", "20000", "40000"]


def _batch_instance(k):
    W, H = BATCH_IMAGES[k % 4]
    return dict(mesh=BATCH_MESHES[(k + k // 4) % 4], ni=2 if k % 3 == 0 else 1, W=W, H=H, f=1.25 * W,
                lam=BATCH_LAMS[(k // 4) % 4])


def _eval_inputs(c, seed):
    """(tracker, scene, params [lam, d] on the device, mask on the host, detections or None)"""
    sc = _case_scene(c)
    rng = np.random.default_rng(seed)
    truth = _truth(rng, sc)
    kw = dict(loss_kind=c["loss"], lambda_app=LAMBDA_APP) if c["kind"] == "eval" else {}
    tr = api.Tracker(sc, lambda_max=c["lam"], **kw)
    mask = _observed(tr, truth, rng)
    params = torch.from_numpy(wl.population_around(rng, truth, c["lam"])).cuda()
    obs = None
    if c.get("kp"):
        tr.set_keypoints((3, 4), (wl.JAW_TIP, wl.JAW_TIP), tau=KP_TAU, lambda_kpts=KP_LAMBDA)
        tips = tr.project_keypoints(torch.from_numpy(truth.astype(np.float32)).cuda()[None])[0].cpu().numpy()
        obs = torch.from_numpy(wl.noisy_detections(tips, rng)).cuda()
    return tr, sc, params, mask, obs


def prepare(case, seed):
    c, kind = case, case["kind"]
    rng = np.random.default_rng(seed)
    if kind in ("eval", "soft"):
        tr, sc, params, mask, obs = _eval_inputs(c, seed)
        if obs is not None:
            tr.set_keypoint_obs(obs)
        st = dict(c=c, tr=tr, params=params, mask=tr.pack_mask(torch.from_numpy(mask).cuda()), obs=obs)
        if kind == "soft":
            st["weights"] = torch.from_numpy(rng.uniform(0.5, 1.5, c["lam"]).astype(np.float32)).cuda()
        return st
    if kind in ("search", "track"):
        sc = _case_scene(c)
        truth = _truth(rng, sc)
        tr = api.Tracker(sc, loss_kind=wl.LOSS_ONE_MINUS_IOU, lambda_max=c["lam"])
        mask = _observed(tr, truth, rng)
        st = dict(c=c, tr=tr, es=_optimiser(tr, sc, c["lam"], truth, rng, seed))
        if c.get("host"):
            st["mask"] = torch.from_numpy(mask).pin_memory()
            st["joints"] = _readings(truth, rng, 2) if c["ni"] == 2 else None
        else:
            st["mask"] = tr.pack_mask(torch.from_numpy(mask).cuda())
        return st
    if kind == "batch":
        trs, opts, masks = [], [], []
        for k in range(c["start"], c["start"] + c["n"]):
            spec = _batch_instance(k)
            sc = _case_scene(spec)
            truth = _truth(rng, sc)
            tr = api.Tracker(sc, loss_kind=wl.LOSS_ONE_MINUS_IOU, lambda_max=spec["lam"])
            masks.append(tr.pack_mask(torch.from_numpy(_observed(tr, truth, rng)).cuda()))
            opts.append(_optimiser(tr, sc, spec["lam"], truth, rng, seed + k))
            trs.append(tr)
        b = api.Batch(trs, optimisers=opts, cluster=1, threads=256)  # the shape that the autotuner picks for it
        return dict(c=c, batch=b, masks=masks, keep=(trs, opts))
    # serve: every other stream has two instruments and joint readings
    srv = api.Server(max_active=c["streams"], max_streams=c["streams"], max_pending=64, max_pixels=c["W"] * c["H"],
                     max_lambda=c["lam"])
    frames, keep = [], []
    for k in range(c["streams"]):
        ni = 1 + k % 2
        sc = _scene(c["mesh"], ni, c["W"], c["H"], c["f"])
        truth = _truth(rng, sc)
        traj = wl.sinusoidal_trajectory(rng, truth, c["frames"])
        tr = api.Tracker(sc, loss_kind=wl.LOSS_ONE_MINUS_IOU, lambda_max=c["lam"])
        es = _optimiser(tr, sc, c["lam"], truth, rng, seed + k)
        sid = srv.add_stream(es, c["gens"], use_joint_reading=ni == 2)
        keep.append((tr, es))
        for f in range(c["frames"]):
            frames.append((f, sid, _observed(tr, traj[f], rng), _readings(traj[f], rng, 2) if ni == 2 else None))
    frames.sort(key=lambda x: x[:2])  # as they arrive: frame by frame over the streams
    return dict(c=c, server=srv, frames=frames, keep=keep)


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def run(state):
    c, kind = state["c"], state["c"]["kind"]
    if kind == "eval":
        loss, counts = state["tr"].eval_population(state["params"], state["mask"], counts=True)
        return {"loss": loss, "counts": counts}
    if kind == "soft":
        if not c["grad"]:
            return {"loss": api.soft_silhouette_loss(state["params"], state["tr"], state["mask"], c["sigma"])}
        x = state["params"].detach().requires_grad_(True)
        loss = api.soft_silhouette_loss(x, state["tr"], state["mask"], c["sigma"])
        (g,) = torch.autograd.grad(loss, x, state["weights"])
        return {"loss": loss.detach(), "grad": g}
    if kind == "search":
        es, tr = state["es"], state["tr"]
        for _ in range(c["gens"]):
            x = es.ask()
            loss = tr.eval_population(x, state["mask"])
            es.tell(loss)
        return {"population": x, "loss": loss}
    if kind == "track":
        if c["host"]:
            pose, loss = state["es"].track_frame_host(state["mask"], c["gens"], state["joints"])
            return {"pose": pose, "loss": loss}
        return {"pose": state["es"].track_frame(state["mask"], c["gens"])}
    if kind == "batch":
        return {"poses": state["batch"].track_frame(state["masks"], c["gens"])}
    srv = state["server"]
    results = []
    for f, sid, mask, joints in state["frames"]:
        while not srv.submit(sid, mask, joints, tag=f):  # staging full: make progress first
            srv.step()
            results += srv.poll()
    results += srv.run_until_idle()
    results.sort(key=lambda r: (r["stream"], r["tag"]))
    return {"poses": np.concatenate([r["pose"] for r in results]),
            "losses": np.array([r["best_loss"] for r in results], np.float32)}


# --------------------------------------------------------------------------
# What one pass cannot do without
# --------------------------------------------------------------------------
def _size(mesh):
    ms = _meshes(mesh)
    return sum(m.verts.shape[0] for m in ms), sum(m.tris.shape[0] for m in ms)


def _eval_work(mesh, ni, lam, W, H):
    """Vertex transforms and triangle set-ups of every candidate (16 operations
    per vertex, 40 per triangle) and 4 per covered pixel (the instrument covers
    about an eighth of the image); mesh, mask, population and losses once."""
    V, T = _size(mesh)
    flops = lam * ni * (16.0 * V + 40.0 * T + 4.0 * W * H / 8)
    return {"bytes": 12.0 * V + 12.0 * T + W * H / 8 + lam * (36.0 * ni + 20), "flops": flops}


def work(case):
    c, kind = case, case["kind"]
    if kind == "eval":
        return _eval_work(c["mesh"], c["ni"], c["lam"], c["W"], c["H"])
    if kind == "soft":
        # pixels within reach of the silhouette's outline see the triangles
        # within 14 sigma: about 40 operations per (pixel, triangle) pair, and as
        # many again for the gradient; the pairs are bounded by the triangles'
        # reach and by the image
        V, T = _size(c["mesh"])
        reach = min(math.pi * (CUTOFF * c["sigma"]) ** 2, c["W"] * c["H"])
        pairs = c["lam"] * c["ni"] * T * reach / 4
        w = _eval_work(c["mesh"], c["ni"], c["lam"], c["W"], c["H"])
        return {"bytes": w["bytes"], "flops": w["flops"] + 40.0 * pairs * (2 if c["grad"] else 1)}
    if kind in ("search", "track"):
        w = _eval_work(c["mesh"], c["ni"], c["lam"], c["W"], c["H"])
        d = 9 * c["ni"]
        update = 2.0 * c["lam"] * d * d + 20.0 * d ** 3
        raw = c["W"] * c["H"] if c.get("host") else 0
        return {"bytes": w["bytes"] + raw, "flops": c["gens"] * (w["flops"] + update)}
    if kind == "batch":
        specs = [_batch_instance(k) for k in range(c["start"], c["start"] + c["n"])]
        ws = [_eval_work(s["mesh"], s["ni"], s["lam"], s["W"], s["H"]) for s in specs]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": c["gens"] * sum(w["flops"] for w in ws)}
    ws = [_eval_work(c["mesh"], 1 + k % 2, c["lam"], c["W"], c["H"]) for k in range(c["streams"])]
    return {"bytes": sum(w["bytes"] + c["frames"] * c["W"] * c["H"] for w in ws),
            "flops": c["frames"] * c["gens"] * sum(w["flops"] for w in ws)}


# --------------------------------------------------------------------------
# The same outputs in 64 bits
# --------------------------------------------------------------------------
def _rot_axis(axis, ang):
    s, c = torch.sin(ang), torch.cos(ang)
    one, zero = torch.ones_like(s), torch.zeros_like(s)
    rows = {0: [one, zero, zero, zero, one, zero, zero, zero, one],
            1: [one, zero, zero, zero, c, -s, zero, s, c],
            2: [c, zero, s, zero, one, zero, -s, zero, c],
            3: [c, -s, zero, s, c, zero, zero, zero, one]}[axis]
    return torch.stack(rows, -1).reshape(ang.shape + (3, 3))


def _frames64(sc, x):
    """Rotations [n, F, 3, 3] and translations [n, F, 3] of every frame in the
    camera for the 9-vectors x [n, 9]."""
    lb, ub = torch.tensor(sc.q_lb, device=x.device), torch.tensor(sc.q_ub, device=x.device)
    q = lb + 0.5 * (ub - lb) * (1 - torch.cos(math.pi * (x[:, 6:9] - lb) / (ub - lb)))
    r = x[:, :3]
    if sc.rot_param == 1:
        R = _rot_axis(2, r[:, 2]) @ _rot_axis(1, r[:, 0]) @ _rot_axis(3, r[:, 1])
    else:
        t = r.norm(dim=1)
        k = r / t[:, None]
        z = torch.zeros_like(t)
        Kx = torch.stack([z, -k[:, 2], k[:, 1], k[:, 2], z, -k[:, 0], -k[:, 1], k[:, 0], z], -1).reshape(-1, 3, 3)
        s, c = torch.sin(t)[:, None, None], torch.cos(t)[:, None, None]
        R = c * torch.eye(3, device=x.device, dtype=x.dtype) + s * Kx + (1 - c) * k[:, :, None] * k[:, None, :]
    Rs, ts = [], []
    for f in sc.frames:
        J = _rot_axis(f.axis, f.coef * q[:, f.joint])
        o = torch.tensor([float(v) for v in f.offset], device=x.device, dtype=x.dtype).expand(x.shape[0], 3)
        P, pt = (R, x[:, 3:6]) if f.parent < 0 else (Rs[f.parent], ts[f.parent])
        Rs.append(P @ J)
        ts.append(pt + (P @ o[:, :, None])[:, :, 0])
    return torch.stack(Rs, 1), torch.stack(ts, 1)


def _project64(sc, x):
    """Offsets from the principal point [n, V, 2] and depths of the mesh's vertices."""
    verts, _, fr = sc.flat()
    v = torch.from_numpy(verts).to(x.device).double()
    fr = torch.from_numpy(fr).to(x.device).long()
    R, t = _frames64(sc, x)
    X = (R[:, fr] @ v[None, :, :, None])[..., 0] + t[:, fr]
    uv = torch.stack([sc.K.fx * X[..., 0] / X[..., 2], sc.K.fy * X[..., 1] / X[..., 2]], -1)
    return uv, X[..., 2]


def _pairs(j0, j1, i0, i1, step=4_000_000):
    """(triangle, column, row) of every pixel of the triangles' boxes, in pieces."""
    w, h = (j1 - j0 + 1).clamp(min=0), (i1 - i0 + 1).clamp(min=0)
    n = w * h
    ends = torch.cumsum(n, 0)
    total, a = int(ends[-1]) if n.numel() else 0, 0
    while a < total:
        k = torch.arange(a, min(total, a + step), device=n.device)
        t = torch.searchsorted(ends, k, right=True)
        o = k - (ends[t] - n[t])
        yield t, j0[t] + o % w[t], i0[t] + torch.div(o, w[t], rounding_mode="floor")
        a += step


def _exact_eval(case, seed):
    tr, sc, params, mask, obs = _eval_inputs(case, seed)
    K, W, H = sc.K, case["W"], case["H"]
    M = torch.from_numpy(mask).cuda().bool()
    _, tris, _ = sc.flat()
    tris = torch.from_numpy(tris).cuda().long()
    cx, cy = int(256 * K.cx), int(256 * K.cy)
    losses, counts = [], []
    for c in range(case["lam"]):
        S = torch.zeros(H * W, dtype=torch.bool, device="cuda")
        culled = 0
        for b in range(case["ni"]):
            uv, Z = _project64(sc, params[c:c + 1, 9 * b: 9 * b + 9].double())
            uv, Z = uv[0], Z[0]
            bad = (Z < K.z_near) | (uv.abs() > 16384).any(-1)
            P = torch.round(256 * uv).nan_to_num(0.0).clamp(-2 ** 40, 2 ** 40).long() + torch.tensor([cx, cy]).cuda()
            keep = ~bad[tris].any(1)
            culled += int((~keep).sum())
            p = P[tris[keep]]
            A = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
            p = torch.where((A < 0)[:, None, None], p[:, [0, 2, 1]], p)[A != 0]
            lo, hi = p.min(1).values, p.max(1).values
            box = [((lo[:, 0] + 255) >> 8).clamp(min=0), (hi[:, 0] >> 8).clamp(max=W - 1),
                   ((lo[:, 1] + 255) >> 8).clamp(min=0), (hi[:, 1] >> 8).clamp(max=H - 1)]
            for t, j, i in _pairs(*box):
                inside = torch.ones_like(t, dtype=torch.bool)
                for k in range(3):
                    a, d = p[t, k], p[t, (k + 1) % 3] - p[t, k]
                    e = d[:, 0] * (256 * i - a[:, 1]) - d[:, 1] * (256 * j - a[:, 0])
                    top_left = (d[:, 1] < 0) | ((d[:, 1] == 0) & (d[:, 0] > 0))
                    inside &= (e > 0) | ((e == 0) & top_left)
                S[(i * W + j)[inside]] = True
        Sm = S.reshape(H, W)
        s, I, m = int(Sm.sum()), int((Sm & M).sum()), int(M.sum())
        x, U = float(s + m - 2 * I), s + m - I
        loss = x if case["loss"] == 0 else (1.0 - I / U if U else 0.0) if case["loss"] == 1 else x + LAMBDA_APP * abs(s - m)
        if obs is not None:
            loss += KP_LAMBDA * _keypoints64(sc, params[c].double(), obs.double())
        losses.append(loss)
        counts.append([s, I, m, culled])
    return {"loss": torch.tensor(losses, dtype=torch.float64), "counts": torch.tensor(counts, dtype=torch.int32)}


def _keypoints64(sc, x, obs):
    total = 0.0
    pos = lambda a, b: max(0.0, math.hypot(a[0] - b[0], a[1] - b[1]) - KP_TAU)
    for b in range(sc.n_instruments):
        o = [float(v) for v in obs[b]]
        if o[4] == 0.0:
            continue
        R, t = _frames64(sc, x[None, 9 * b: 9 * b + 9])
        tip = torch.tensor(wl.JAW_TIP, device=x.device)
        p = []
        for f in (3, 4):
            X = (R[0, f] @ tip + t[0, f]).tolist()
            p.append((sc.K.fx * X[0] / X[2] + sc.K.cx, sc.K.fy * X[1] / X[2] + sc.K.cy))
        a, d = (o[0], o[1]), (o[2], o[3])
        mid = lambda u, v: ((u[0] + v[0]) / 2, (u[1] + v[1]) / 2)
        total += min(pos(a, p[0]) + pos(d, p[1]), pos(a, p[1]) + pos(d, p[0])) + pos(mid(a, d), mid(p[0], p[1]))
    return total


def _distance64(tri, px, py):
    """Signed distances of the pixel centres to their triangles (positively
    oriented [n, 3, 2]), and the nearest boundary points as (edge, position on
    it, unit vector from it to the centre, pointing outwards when inside)."""
    p = torch.stack([px, py], -1)
    inside = torch.ones_like(px, dtype=torch.bool)
    best = None
    for k in range(3):
        a, e = tri[:, k], tri[:, (k + 1) % 3] - tri[:, k]
        r = p - a
        L2 = (e * e).sum(-1)
        E = e[:, 0] * r[:, 1] - e[:, 1] * r[:, 0]
        s = (r * e).sum(-1) / L2
        t = s.clamp(0, 1)
        q = r - t[:, None] * e
        flat = (s > 0) & (s < 1)
        dist = torch.where(flat, E.abs() / L2.sqrt(), q.norm(dim=1))
        normal = torch.stack([-e[:, 1], e[:, 0]], -1) / L2.sqrt()[:, None] * torch.sign(E)[:, None]
        n = torch.where(flat[:, None], normal, q / q.norm(dim=1).clamp(min=1e-300)[:, None])
        inside &= E >= 0
        new = (dist, torch.full_like(px, k, dtype=torch.long), t, n)
        if best is None:
            best = new
        else:
            less = dist < best[0]
            best = tuple(torch.where(less[:, None] if u.dim() == 2 else less, u, v) for u, v in zip(new, best))
    sign = torch.where(inside, 1.0, -1.0).double()
    return best[0] * sign, best[1], best[2], best[3], sign


def _exact_soft(case, seed):
    _, sc, params, mask, _ = _eval_inputs(case, seed)
    rng = np.random.default_rng(seed)
    weights = torch.from_numpy(rng.uniform(0.5, 1.5, case["lam"]).astype(np.float32)).cuda().double()
    K, W, H, sigma = sc.K, case["W"], case["H"], case["sigma"]
    M = torch.from_numpy(mask).cuda().double().reshape(-1)
    _, tris, _ = sc.flat()
    tris = torch.from_numpy(tris).cuda().long()
    reach = CUTOFF * sigma
    losses, grads = [], []
    for c in range(case["lam"]):
        x = params[c].double().requires_grad_(True)
        uvs, work = [], []
        for b in range(case["ni"]):
            uv, Z = _project64(sc, x[None, 9 * b: 9 * b + 9])
            uv, Z = uv[0], Z[0].detach()
            uvs.append(uv)
            u = uv.detach()
            bad = (Z < K.z_near) | (u.abs() > 16384).any(-1)
            ids = tris[~bad[tris].any(1)]
            p = u[ids]
            A = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
            ids = torch.where((A < 0)[:, None], ids[:, [0, 2, 1]], ids)[A != 0]
            p = u[ids] + torch.tensor([K.cx, K.cy], device="cuda", dtype=torch.float64)
            lo, hi = p.min(1).values - reach, p.max(1).values + reach
            box = [torch.ceil(lo[:, 0]).long().clamp(min=0), torch.floor(hi[:, 0]).long().clamp(max=W - 1),
                   torch.ceil(lo[:, 1]).long().clamp(min=0), torch.floor(hi[:, 1]).long().clamp(max=H - 1)]
            work.append((ids, p, box))
        acc = torch.zeros(H * W, dtype=torch.float64, device="cuda")
        for ids, p, box in work:
            for t, j, i in _pairs(*box):
                d = _distance64(p[t], j.double(), i.double())[0]
                a = torch.where(d >= -reach, torch.nn.functional.softplus(d / sigma, threshold=1e9), 0.0)
                acc.index_add_(0, i * W + j, a)
        S = -torch.expm1(-acc)
        losses.append(float(((S - M) ** 2).sum()))
        if not case["grad"]:
            continue
        gS = 2 * (S - M) * torch.exp(-acc) / sigma * weights[c]
        gs = []
        for (ids, p, box), uv in zip(work, uvs):
            g = torch.zeros_like(uv)
            for t, j, i in _pairs(*box):
                d, k, s, n, sign = _distance64(p[t], j.double(), i.double())
                w = torch.where(d >= -reach, gS[i * W + j] * torch.sigmoid(d / sigma), 0.0) * sign
                for e, f in ((k, 1 - s), ((k + 1) % 3, s)):
                    v = ids[t].gather(1, e[:, None])[:, 0]
                    g.index_add_(0, v, -(w * f)[:, None] * n)
            gs.append(g)
        grads.append(torch.autograd.grad(uvs, x, gs)[0])
    out = {"loss": torch.tensor(losses, dtype=torch.float64)}
    if case["grad"]:
        out["grad"] = torch.stack(grads)
    return out


def exact(case, seed):
    if case["kind"] == "eval":
        return _exact_eval(case, seed)
    if case["kind"] == "soft":
        return _exact_soft(case, seed)
    # the searches draw their normals in FP32 and rank candidates by integer
    # pixel counts: a search in 64 bits draws other candidates and takes another
    # path, so these calls have no value of this kind
    return None
