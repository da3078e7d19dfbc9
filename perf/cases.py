"""What a user of this library has it do, as cases that can be timed and compared.

A case names one of these kinds of work and its sizes:

* ``search``   Plan.search: the shift-and-stack search of one field, or of
  several fields of one plan, from frames on the device to the sorted list
  in a buffer that the program keeps;
* ``noalloc``  search_noalloc: the same for callers that cannot allocate;
* ``refine``   Plan.refine: optimiser steps on the candidates of a search;
* ``grad``     refine_objective: the objective and its gradient by autograd;
* ``tracks``   Plan.link_tracks: a search's detections linked into tracks;
* ``median``   median_subtract: star removal over a group of frames;
* ``sumbin``   sum_frames and bin2x2 on one sequence.

Frames are made on the GPU from the seed: Gaussian noise, movers with a
Gaussian PSF, and, where the search normalises, what raw frames bring with
them: a sky level and noise of each frame's own, cosmic rays, masked stars.
"""
import math

import numpy as np
import torch

import paper_2303_07293_gb300 as st

FWHM = 3.0
CAPACITY = 1 << 20   # detections that a program keeps room for
MAX_TRACKS = 1 << 17


def _search(name, w, h, n, nv, hours, step_px, **kw):
    """step_px: how far adjacent velocities are apart over the whole baseline."""
    c = dict(name=name, kind="search", w=w, h=h, n=n, nv=nv, hours=hours, step_px=step_px,
             tau=5.0, mode="nearest", storage="f32", normalize=True, clip=10.0, movers=20,
             fields=1, graph=False)
    c.update(kw)
    return c


def listed():
    return [
        # a look at a short sequence with an integer grid (1 px per frame and
        # step): 16 frames of 128^2, used as given; launches and latency
        _search("tiny", 128, 128, 16, 21, 15.0, 15.0, normalize=False, clip=0.0, movers=3),
        # two hours on a 1024^2 camera, full blind grid, nearest shifts
        _search("mid", 1024, 1024, 64, 161, 2.0, 1.0),
        # the same frames at sub-pixel shifts
        _search("mid_bilinear", 1024, 1024, 64, 81, 2.0, 1.0, mode="bilinear"),
        # a night on a 2048^2 camera at 50 s cadence, 0.25 px/h steps: the
        # slow-mover part (+-12.5 px/h) of the blind grid
        _search("night", 2048, 2048, 256, 101, 255 * 50.0 / 3600, 0.885, movers=100),
        # several targets of a night in one plan: uneven lengths and sizes,
        # FP16 frames, the device part replayed as a graph
        _search("batch_f16", 1024, 1024, 120, 61, 3.0, 1.0, storage="f16", fields=6, graph=True),
        # a cropped, registered sequence: odd sizes, BF16 frames
        _search("ragged_bf16", 1021, 997, 45, 41, 1.5, 0.8, storage="bf16"),
        # continuous refinement of a search's best 4096 detections
        dict(name="refine_adam", kind="refine", w=2048, h=2048, n=300, cands=4096, steps=20,
             optimizer="adam", storage="f32"),
        # one value-and-gradient call of a user's own optimiser
        dict(name="grad", kind="grad", w=1024, h=1024, n=64, cands=512, storage="f32"),
        # the detections of a deep (4.5 sigma) search, linked
        dict(name="tracks", kind="tracks", w=1024, h=1024, n=64, nv=121, tau=4.5),
        # star removal for a group of 50 full frames
        dict(name="median_group", kind="median", w=2048, h=2048, n=50, masked=0.002),
        # star removal over a whole sequence
        dict(name="median_night", kind="median", w=1024, h=1024, n=200, masked=0.002),
        # sums of every 13 frames for slow movers, binning for fast ones
        dict(name="sum_bin", kind="sumbin", w=2048, h=2048, n=256, n_sum=13),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["noalloc", "refine", "grad", "tracks", "median", "median",
                                        "sumbin"])
    if kind == "search":
        while True:
            c = _search("", _log(rng, 64, 2048), _log(rng, 64, 2048), _log(rng, 8, 300),
                        rng.randrange(5, 162), round(rng.uniform(0.5, 8.0), 2),
                        round(rng.uniform(0.5, 1.0), 2),
                        mode=rng.choice(["nearest", "nearest", "nearest", "bilinear"]),
                        storage=rng.choice(["f32", "f32", "f16", "bf16"]),
                        normalize=rng.random() < 0.7, fields=rng.choice([1, 1, 1, 3]),
                        graph=rng.random() < 0.3)
            if rng.random() < 0.6:   # camera formats: rows of a whole number of 16 pixels
                c["w"] = max(64, c["w"] // 16 * 16)
            c["clip"] = 10.0 if c["normalize"] else 0.0
            px = sum(f["width"] * f["height"] * f["n_frames"] for f in _fields(c))
            cost = px * c["nv"] ** 2 * (4 if c["mode"] == "bilinear" else 1)
            if px <= 4 << 28 and 1e8 <= cost <= 6e11:
                break
    elif kind == "noalloc":
        c = dict(kind=kind, w=_log(rng, 32, 512), h=_log(rng, 32, 512), n=_log(rng, 8, 64),
                 nv=rng.randrange(5, 42), hours=2.0, step_px=round(rng.uniform(0.5, 4.0), 2),
                 tau=5.0, mode=rng.choice(["nearest", "bilinear"]), movers=2, normalize=False,
                 clip=0.0, fields=1, storage="f32")
    elif kind == "refine":
        c = dict(kind=kind, w=16 * rng.randrange(16, 97), h=rng.randrange(256, 1537),
                 n=_log(rng, 16, 200), cands=_log(rng, 32, 2048), steps=rng.randrange(2, 21),
                 optimizer=rng.choice(["adam", "gn"]), storage=rng.choice(["f32", "f16", "bf16"]))
    elif kind == "grad":
        c = dict(kind=kind, w=16 * rng.randrange(16, 97), h=rng.randrange(256, 1537),
                 n=_log(rng, 12, 100), cands=_log(rng, 8, 600), storage="f32")
    elif kind == "tracks":
        c = dict(kind=kind, w=16 * rng.randrange(16, 65), h=rng.randrange(256, 1025),
                 n=_log(rng, 16, 64), nv=rng.randrange(21, 122), tau=round(rng.uniform(4.5, 5.0), 2))
    elif kind == "median":
        n = _log(rng, 3, 300)
        side = min(2048, int(math.sqrt(2e8 / n)))
        c = dict(kind=kind, w=_log(rng, 64, side), h=_log(rng, 64, side), n=n,
                 masked=rng.choice([0.0, 0.002, 0.02]))
    else:
        n = _log(rng, 8, 256)
        side = min(2048, int(math.sqrt(1e9 / n)))
        c = dict(kind=kind, w=_log(rng, 64, side), h=_log(rng, 64, side), n=n,
                 n_sum=rng.randrange(2, min(n, 32)))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _fields(c):
    """The fields of a search case.  With several, lengths and sizes are
    uneven: from a third to the whole of the case's, in turn."""
    out = []
    for j in range(c["fields"]):
        share = 1.0 - 0.61 * ((j * 5) % c["fields"]) / c["fields"]
        half = 1 if c["fields"] == 1 or j % 3 != 2 else 2
        w, h = c["w"] // half, c["h"] // half
        n = max(8, int(c["n"] * share))
        t = np.arange(n) * (c["hours"] * share / max(n - 1, 1))
        dv = c["step_px"] / float(t[-1] - t[0])
        nv = c["nv"]
        out.append(dict(width=w, height=h, n_frames=n, t_ref=float(t[n // 2]),
                        vx0=-dv * (nv // 2), dvx=dv, nvx=nv, vy0=-dv * (nv // 2), dvy=dv, nvy=nv,
                        snr_threshold=c["tau"], min_coverage=0, times=t))
    return out


def _rng(seed, j):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 97 * j + 1)
    return g


def _frames(f, seed, j, movers, raw):
    """One field's frames [N][H][W]: unit noise and movers; raw: with sky,
    cosmic rays and masked stars."""
    n, h, w = f["n_frames"], f["height"], f["width"]
    g = _rng(seed, j)
    out = torch.empty((n, h, w), device="cuda", dtype=torch.float32)
    out.normal_(generator=g)
    u = torch.rand((max(movers, 1), 5), generator=g, device="cuda", dtype=torch.float64)
    if movers:
        dt = torch.from_numpy(f["times"] - f["t_ref"]).cuda()
        vx = f["vx0"] + u[:, 0] * (f["nvx"] - 1) * f["dvx"]
        vy = f["vy0"] + u[:, 1] * (f["nvy"] - 1) * f["dvy"]
        xs = (u[:, 2] * (w - 1))[:, None] + vx[:, None] * dt
        ys = (u[:, 3] * (h - 1))[:, None] + vy[:, None] * dt
        amp = 0.3 + 2.7 * u[:, 4]
        s2 = (FWHM / 2.354820045) ** 2
        d = torch.arange(-5, 6, device="cuda", dtype=torch.float64)
        px, py = torch.round(xs)[..., None, None] + d[None, :], torch.round(ys)[..., None, None] + d[:, None]
        val = amp[:, None, None, None] * torch.exp(
            -((px - xs[..., None, None]) ** 2 + (py - ys[..., None, None]) ** 2) / (2 * s2))
        px, py = torch.broadcast_tensors(px, py)
        i = torch.arange(n, device="cuda")[None, :, None, None].expand_as(px)
        ok = (px >= 0) & (px < w) & (py >= 0) & (py < h)
        flat = (i[ok] * h + py[ok].long()) * w + px[ok].long()
        # (sorted: movers that cross add up in one order)
        flat, at = torch.sort(flat, stable=True)
        uniq, inv = torch.unique_consecutive(flat, return_inverse=True)
        tot = torch.zeros(uniq.shape, device="cuda", dtype=torch.float64)
        tot.index_put_((inv,), torch.round(val[ok][at] * 2 ** 24) / 2 ** 24, accumulate=True)
        out.view(-1)[uniq] += tot.float()
    if raw:
        sky = torch.rand((n, 2), generator=g, device="cuda")
        level, sigma = 150.0 + 200.0 * sky[:, 0], 8.0 + 6.0 * sky[:, 1]
        hits = max(1, int(1e-5 * n * h * w))
        at = torch.randint(0, n * h * w, (hits,), generator=g, device="cuda")
        out.view(-1)[at] = 20.0 + 60.0 * (at % 4).float()
        for i in range(n):
            out[i].mul_(sigma[i]).add_(level[i])
        stars = max(1, (w * h) // 5000)
        sx = torch.randint(0, w, (stars,), generator=g, device="cuda")
        sy = torch.randint(0, h, (stars,), generator=g, device="cuda")
        mask = torch.zeros((h, w), device="cuda", dtype=torch.bool)
        for dy in range(-4, 5):
            for dx in range(-4, 5):
                if dx * dx + dy * dy <= 18:
                    mask[(sy + dy).clamp(0, h - 1), (sx + dx).clamp(0, w - 1)] = True
        out.masked_fill_(mask, float("nan"))
    return out


def _stars(c, seed):
    """A sequence with stationary stars, before star removal."""
    n, h, w = c["n"], c["h"], c["w"]
    g = _rng(seed, 0)
    out = torch.empty((n, h, w), device="cuda", dtype=torch.float32)
    out.normal_(generator=g)
    out += 200.0 + 3000.0 * torch.rand((h, w), generator=g, device="cuda") ** 200
    if c.get("masked", 0.0) > 0.0:
        k = max(1, int(c["masked"] * n * h * w))
        out.view(-1)[torch.randint(0, n * h * w, (k,), generator=g, device="cuda")] = float("nan")
    return out


def _refine_field(c):
    """The field whose detections are refined: an hour's steps of 0.25 px."""
    hours = c["n"] * 50.0 / 3600
    return _search("", c["w"], c["h"], c["n"], 41, hours, 0.25 * hours, tau=4.5,
                   storage=c["storage"], movers=100)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("median", "sumbin"):
        s = dict(case=case, frames=_stars(case, seed))
        if kind == "sumbin":
            s["times"] = np.arange(case["n"]) * (50.0 / 3600)
        return s
    c = case
    if kind == "tracks":
        c = _search("", case["w"], case["h"], case["n"], case["nv"], 2.0, 1.0, tau=case["tau"])
    elif kind in ("refine", "grad"):
        c = _refine_field(case)
    fields = _fields(c)
    frames = [_frames(f, seed, j, c["movers"], c["normalize"]) for j, f in enumerate(fields)]
    times = [f["times"] for f in fields]
    s = dict(case=case, fields=fields, frames=frames, times=times)
    if kind == "noalloc":
        return s
    s["plan"] = st.Plan(fields, storage=c["storage"], mode=c["mode"], normalize=c["normalize"],
                        cr_clip=c["clip"], use_graph=c["graph"])
    if kind == "search":
        s["out"] = torch.zeros((CAPACITY, 7), dtype=torch.int32, device="cuda")
        return s
    # the detections that tracks and refinement start from
    out, n, _ = s["plan"].search(frames, times)
    out = out[:n]
    if kind == "tracks":
        s["cands"] = out
        s["tracks"] = np.zeros(MAX_TRACKS, st.TRACK_DTYPE)
    else:
        snr = out[:, 5].view(torch.float32)
        top = torch.sort(snr, descending=True, stable=True).indices
        at = torch.arange(case["cands"], device="cuda") % top.shape[0]
        s["cands"] = out[top[at]].contiguous()
    if kind == "grad":
        f, k = fields[0], s["cands"][:, 2]
        xy = s["cands"][:, :2]
        g = _rng(seed, 7)
        jitter = torch.rand((xy.shape[0], 5), generator=g, device="cuda") - 0.5
        vx = f["vx0"] + (k % f["nvx"]).double() * f["dvx"]
        vy = f["vy0"] + torch.div(k, f["nvx"], rounding_mode="floor").double() * f["dvy"]
        theta = torch.stack([vx, vy, xy[:, 0].double(), xy[:, 1].double(),
                             1.0 + 0.0 * vx], 1).float()
        theta += jitter * torch.tensor([0.2, 0.2, 0.8, 0.8, 0.8], device="cuda")
        s["theta"], s["centre"] = theta.contiguous(), xy.contiguous()
    return s


def _cols(rec):
    return {k: rec[k] for k in rec.dtype.names}


def _detections(out, n, status):
    # columns x, y, k, field | stack, S/N (FP32) | n_cov; rows past n stay zero
    return dict(where=out[:, :4], value=out[:, 4:6].view(torch.float32), n_cov=out[:, 6], n=n,
                status=status)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "search":
        return _detections(*state["plan"].search(state["frames"], state["times"], CAPACITY,
                                                 out=state["out"]))
    if kind == "noalloc":
        f = state["fields"][0]
        out, n, status = st.search_noalloc(f, state["frames"][0], state["times"][0],
                                           mode=c["mode"], capacity=1 << 14)
        out[n:] = 0
        return _detections(out, n, status)
    if kind == "refine":
        rec, g = state["plan"].refine(state["cands"], steps=c["steps"], fwhm=FWHM, grad=True,
                                      optimizer=c["optimizer"])
        return dict(_cols(rec), grad=g)
    if kind == "grad":
        theta = state["theta"].clone().requires_grad_(True)
        J = st.refine_objective(theta, state["plan"], state["centre"], fwhm=FWHM)
        J.sum().backward()
        return dict(J=J.detach(), grad=theta.grad)
    if kind == "tracks":
        rec = state["plan"].link_tracks(state["cands"])
        state["tracks"][:len(rec)] = rec[:MAX_TRACKS]
        return dict(_cols(state["tracks"]), n=len(rec))
    if kind == "median":
        out, med = st.median_subtract(state["frames"], with_median=True)
        return dict(out=out, median=med)
    sums, t = st.sum_frames(state["frames"], state["times"], c["n_sum"])
    return dict(sums=sums, times=t, binned=st.bin2x2(state["frames"]))


def work(case):
    kind = case["kind"]
    if kind in ("search", "noalloc"):
        by = fl = 0
        for f in _fields(case):
            px = f["width"] * f["height"] * f["n_frames"]
            by += 4 * px
            fl += px * f["nvx"] * f["nvy"] * (8 if case["mode"] == "bilinear" else 1)
        return dict(bytes=by, flops=fl)
    if kind in ("refine", "grad"):
        evals = case["steps"] + 1 if kind == "refine" else 2
        n = case["cands"] * case["n"]
        size = 4 if case["storage"] == "f32" else 2
        return dict(bytes=min(n * 65 * 65, case["w"] * case["h"] * case["n"]) * size,
                    flops=14 * 4096 * n * evals)
    if kind == "tracks":
        # about the normal tail above the threshold, of which a third are maxima
        tail = 0.5 * math.erfc(case["tau"] / math.sqrt(2.0))
        n = case["w"] * case["h"] * case["nv"] ** 2 * tail / 3.0
        return dict(bytes=n * (28 + 48), flops=0)
    px = case["w"] * case["h"] * case["n"]
    if kind == "median":
        return dict(bytes=4 * (2 * px + case["w"] * case["h"]), flops=px)
    m = case["n"] // case["n_sum"]
    return dict(bytes=4 * (2 * px + px // 4 + m * case["w"] * case["h"]), flops=2 * px)


# --------------------------------------------------------- values in 64 bits

def _normalized(x, storage, clip):
    """Robust normalisation in 64 bits: 3-sigma clipped mean and deviation (at
    most 5 statistics), then rounded as the frames are stored."""
    x = x.double()
    out = torch.zeros_like(x)
    for i in range(x.shape[0]):
        r = x[i]
        v = r[torch.isfinite(r)]
        keep = torch.ones_like(v, dtype=torch.bool)
        mu, sd = v.mean(), v.std(unbiased=False)
        for _ in range(4):
            now = (v - mu).abs() <= 3.0 * sd
            if bool((now == keep).all()) or not bool(now.any()):
                break
            keep = now
            mu, sd = v[keep].mean(), v[keep].std(unbiased=False)
        z = ((r - mu) / sd).float()
        z = torch.where(torch.isfinite(r), z, torch.zeros_like(z))
        if clip > 0.0:
            z[z.abs() > clip] = 0.0
        out[i] = z.to({"f32": torch.float32, "f16": torch.float16,
                       "bf16": torch.bfloat16}[storage]).double()
    return out


def _exact_search(case, seed):
    f = _fields(case)[0]
    x = _frames(f, seed, 0, case["movers"], case["normalize"])
    x = _normalized(x, case["storage"], case["clip"]) if case["normalize"] else x.double()
    n, h, w = x.shape
    dt = f["times"] - f["t_ref"]
    tau = np.float32(f["snr_threshold"])
    thr = torch.tensor([float(np.float32(float(tau) * math.sqrt(k))) for k in range(n + 1)],
                       device="cuda", dtype=torch.float64)
    nmin = (n + 1) // 2
    got = []
    for k in range(f["nvx"] * f["nvy"]):
        sx = np.floor((f["vx0"] + (k % f["nvx"]) * f["dvx"]) * dt + 0.5).astype(int)
        sy = np.floor((f["vy0"] + (k // f["nvx"]) * f["dvy"]) * dt + 0.5).astype(int)
        S = torch.zeros((h, w), device="cuda", dtype=torch.float64)
        C = torch.zeros((h, w), device="cuda", dtype=torch.int64)
        for i in range(n):
            x0, x1 = max(0, -sx[i]), min(w, w - sx[i])
            y0, y1 = max(0, -sy[i]), min(h, h - sy[i])
            if x0 < x1 and y0 < y1:
                S[y0:y1, x0:x1] += x[i, y0 + sy[i]:y1 + sy[i], x0 + sx[i]:x1 + sx[i]]
                C[y0:y1, x0:x1] += 1
        ok = C >= nmin
        best = torch.where(ok, S, torch.full_like(S, -math.inf))
        pad = torch.nn.functional.pad(best, (1, 1, 1, 1), value=-math.inf)
        peak = ok & (S >= thr[C])
        for q, (dy, dx) in enumerate([(-1, -1), (-1, 0), (-1, 1), (0, -1), (0, 1), (1, -1),
                                      (1, 0), (1, 1)]):
            nb = pad[1 + dy:1 + dy + h, 1 + dx:1 + dx + w]
            peak &= (S > nb) if q < 4 else (S >= nb)
        at = peak.nonzero()
        if len(at):
            s, cv = S[at[:, 0], at[:, 1]], C[at[:, 0], at[:, 1]]
            got.append(torch.stack([s, s / torch.sqrt(cv.double())], 1))
    value = torch.zeros((CAPACITY if case["kind"] == "search" else 1 << 14, 2),
                        device="cuda", dtype=torch.float64)
    at = 0
    for g in got:
        value[at:at + len(g)] = g[:len(value) - at]
        at += len(g)
    # (positions, velocities and coverage are whole numbers)
    return dict(where=None, value=value, n_cov=None, n=None, status=None)


def _exact_grad(case, seed):
    s = prepare(case, seed)
    f, theta, centre = s["fields"][0], s["theta"].double(), s["centre"].double()
    img = _normalized(s["frames"][0], case["storage"], 10.0)
    s["plan"].close()
    n, h, w = img.shape
    dt = torch.from_numpy(f["times"] - f["t_ref"]).cuda()
    m = theta.shape[0]
    r = torch.arange(-32, 32, device="cuda", dtype=torch.float64)
    X = centre[:, 0, None, None] + r[None, None, :]
    Y = centre[:, 1, None, None] + r[None, :, None]
    X, Y = torch.broadcast_tensors(X, Y)
    sg = FWHM / (2.0 * 1.1774100225154747)
    dx, dy = X - theta[:, 2, None, None], Y - theta[:, 3, None, None]
    g = torch.exp(-(dx ** 2 + dy ** 2) / (2 * sg * sg))
    S = torch.zeros_like(g)
    gvx = torch.zeros(m, device="cuda", dtype=torch.float64)
    gvy = torch.zeros_like(gvx)
    for i in range(n):
        px, py = theta[:, 0] * dt[i], theta[:, 1] * dt[i]
        ux, uy = torch.floor(px), torch.floor(py)
        fx, fy = (px - ux)[:, None, None], (py - uy)[:, None, None]
        U, V = (X + ux[:, None, None]).long(), (Y + uy[:, None, None]).long()

        def tap(a, b):
            u, v = U + a, V + b
            ok = (u >= 0) & (v >= 0) & (u < w) & (v < h)
            return torch.where(ok, img[i][v.clamp(0, h - 1), u.clamp(0, w - 1)], 0.0)

        a0, a1, b0, b1 = tap(0, 0), tap(1, 0), tap(0, 1), tap(1, 1)
        S += (1 - fy) * ((1 - fx) * a0 + fx * a1) + fy * ((1 - fx) * b0 + fx * b1)
        gvx += dt[i] * (g * ((1 - fy) * (a1 - a0) + fy * (b1 - b0))).sum((1, 2))
        gvy += dt[i] * (g * ((1 - fx) * (b0 - a0) + fx * (b1 - a1))).sum((1, 2))
    F = theta[:, 4]
    gs, gg = (g * S).sum((1, 2)), (g * g).sum((1, 2))
    gx, gy = g * dx / sg ** 2, g * dy / sg ** 2
    J = F * gs - 0.5 * F * F * n * gg
    grad = torch.stack([F * gvx, F * gvy,
                        F * (gx * S).sum((1, 2)) - F * F * n * (g * gx).sum((1, 2)),
                        F * (gy * S).sum((1, 2)) - F * F * n * (g * gy).sum((1, 2)),
                        gs - F * n * gg], 1)
    return dict(J=J, grad=grad)


def _exact_median(case, seed):
    x = _stars(case, seed)
    n, h, w = x.shape
    med = torch.empty((h, w), device="cuda", dtype=torch.float64)
    for y in range(0, h, 64):
        v = x[:, y:y + 64]
        fin = torch.isfinite(v)
        cnt = fin.sum(0)
        v = torch.sort(torch.where(fin, v, torch.full_like(v, math.inf)), dim=0).values.double()
        lo = v.gather(0, ((cnt - 1).clamp(min=0) // 2)[None])[0]
        hi = v.gather(0, (cnt // 2).clamp(max=n - 1)[None])[0]
        med[y:y + 64] = torch.where(cnt > 0, 0.5 * (lo + hi), float("nan"))
    return dict(out=x.double() - med, median=med)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "noalloc"):
        small = work(case)["flops"] <= 1e11 and case["nv"] ** 2 * case["n"] <= 1e5
        if case["fields"] == 1 and case["mode"] == "nearest" and small:
            return _exact_search(case, seed)
        return None   # a search in plain torch takes minutes
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "median":
        return _exact_median(case, seed)
    if kind == "sumbin":
        x, q = _stars(case, seed), case["n_sum"]
        n, h, w = x.shape
        m = n // q
        t = np.arange(n) * (50.0 / 3600)
        sums = torch.stack([x[j * q:(j + 1) * q].double().sum(0) for j in range(m)])
        x = x[:, :h // 2 * 2, :w // 2 * 2]
        binned = torch.stack([f[0::2, 0::2].double() + f[0::2, 1::2] + f[1::2, 0::2] +
                              f[1::2, 1::2] for f in x])
        return dict(sums=sums, times=t[:m * q].reshape(m, q).mean(1), binned=binned)
    # refine: twenty steps of every candidate in 64 bits take minutes;
    # tracks: its numbers are those of the detections that it is given
    return None
