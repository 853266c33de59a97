"""Performance cases of the tracking filter: what a user's program has it do, through the
package's public entry points (Filter, Batch, Server, pf_step_frame_noalloc).

A case is a dict of plain values.  Kinds:
  track    a whole video of one tracker: reset, run over resident (or pinned host) frames,
           read every frame's estimate and weight statistics
  loop     closed loop: one host frame in, its estimate out, one frame a pass
  step     one frame of a caller that owns every buffer (pf_step_frame_noalloc): the new
           particles, likelihoods and the new state come back
  batch    many trackers of one precision over resident videos, every frame's estimates
  serve    camera streams of mixed precision on a server: one frame each, drained
Videos are the package's synthetic kind (a disk of level 228 on a background of 100, noise 5,
bouncing off the walls), rendered here on the GPU from the seed.
"""
import math
import random

import numpy as np
import torch

import paper_2308_00763_gb300 as pf

_BYTES = {"ref64": 8, "f32": 4, "f16": 2, "bf16": 2}
_DTYPE = {"ref64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_BG, _FG = 100.0, 228.0


def _track(name, precision, n, w, h, r, frames, sigma=(1.0, 1.0), drift=(0.0, 0.0), resampler="systematic",
           steps=0, host=False):
    c = dict(kind="track", precision=precision, n=n, w=w, h=h, r=r, frames=frames, sx=sigma[0], sy=sigma[1],
             dx=drift[0], dy=drift[1], resampler=resampler, steps=steps, host=host)
    return dict(c, name=name) if name else c


def _loop(name, precision, n, w, h, r):
    c = dict(kind="loop", precision=precision, n=n, w=w, h=h, r=r, frames=16, sx=1.0, sy=1.0, dx=0.0, dy=0.0)
    return dict(c, name=name) if name else c


def _step(name, precision, n, w, h, r, resampler="systematic"):
    c = dict(kind="step", precision=precision, n=n, w=w, h=h, r=r, sx=1.0, sy=1.0, dx=0.0, dy=0.0,
             resampler=resampler)
    return dict(c, name=name) if name else c


def _batch(name, precision, trackers, frames, n_lo, n_hi):
    c = dict(kind="batch", precision=precision, trackers=trackers, frames=frames, n_lo=n_lo, n_hi=n_hi)
    return dict(c, name=name) if name else c


def _serve(name, streams, n_lo, n_hi):
    c = dict(kind="serve", streams=streams, n_lo=n_lo, n_hi=n_hi)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a control loop on a small camera: the latency of one frame, host to estimate
        _loop("loop_f32_1k", "f32", 1000, 128, 128, 5),
        # the paper's motion model at its largest particle count, half precision
        _track("paper_f16_64k", "f16", 65536, 512, 512, 5, 50, sigma=(5.0, 2.0), drift=(1.0, 2.0)),
        # the benchmark's tracker in half precision and, as the usual default, in single
        _track("bench_f16_1m", "f16", 1 << 20, 512, 512, 5, 100),
        _track("bench_f32_1m", "f32", 1 << 20, 512, 512, 5, 50),
        # bfloat16 over host frames, a larger object, a ragged particle count
        _track("host_bf16_300k", "bf16", 300007, 1024, 768, 10, 32, host=True),
        # the FP64 mode that results are validated against
        _track("ref64_200k", "ref64", 200003, 512, 512, 5, 10),
        # the largest tracker of the size sweep
        _track("large_f16_16m", "f16", 1 << 24, 1024, 1024, 10, 20),
        # allocation-free step inside another engine, ragged count, single precision
        _step("step_f32_260k", "f32", 260001, 640, 480, 7),
        # two of the other resampling schemes
        _track("multinomial_f16_512k", "f16", 1 << 19, 512, 512, 5, 20, resampler="multinomial"),
        _track("metropolis_f32_128k", "f32", 131071, 512, 512, 5, 10, resampler="metropolis"),
        # many trackers of mixed size in one launch a frame (an offline batch of videos)
        _batch("batch_f16_256", "f16", 256, 6, 1000, 262144),
        # a multi-camera server, FP16 and FP32 streams
        _serve("serve_64", 64, 4096, 1 << 20),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["track"] * 6 + ["loop", "step", "batch", "serve"])
    precision = rng.choice(["f16", "f16", "f32", "f32", "bf16", "ref64"])
    w, h = rng.choice([(128, 128), (256, 256), (333, 217), (512, 512), (640, 480), (1024, 768), (1024, 1024)])
    r = rng.randint(3, 10 if w < 256 else 12)
    if kind == "loop":
        return _loop(None, precision, _log_int(rng, 1000, 65536), w, h, r)
    if kind == "step":
        return _step(None, precision, _log_int(rng, 4096, 1 << (18 if precision == "ref64" else 21)), w, h, r,
                     rng.choice(["systematic", "stratified"]))
    if kind == "batch":
        precision = rng.choice(["f16", "f32", "bf16"])
        return _batch(None, precision, rng.randint(16, 200), rng.randint(2, 5), 1000, _log_int(rng, 8192, 200000))
    if kind == "serve":
        return _serve(None, rng.randint(4, 60), 4096, _log_int(rng, 32768, 1 << 20))
    resampler = rng.choice(["systematic"] * 5 + ["stratified", "multinomial", "metropolis", "rejection", "gumbel"])
    paper = rng.random() < 0.25
    motion = dict(sigma=(5.0, 2.0), drift=(1.0, 2.0)) if paper else dict(sigma=(1.0, 1.0))
    # the sizes that each scheme and precision is run at, and no pass dearer than the largest
    # listed one
    top = {"systematic": 1 << 23, "stratified": 1 << 21, "multinomial": 1 << 20, "metropolis": 1 << 19,
           "rejection": 1 << 18, "gumbel": 8192}[resampler]
    if precision == "ref64":
        top = min(top, {"rejection": 1 << 15, "metropolis": 1 << 16, "gumbel": 2048}.get(resampler, 1 << 19))
    n = _log_int(rng, 1000, top)
    most = {"systematic": 64 << 20, "stratified": 32 << 20, "multinomial": 20 << 20, "metropolis": 6 << 20,
            "rejection": 2 << 20, "gumbel": 16384}[resampler]
    if precision == "ref64":
        most = min(most >> 4, 4 << 20) if resampler != "gumbel" else 4096
    frames = max(2, min(rng.randint(5, 60), most // n))
    return _track(None, precision, n, w, h, r, frames, resampler=resampler,
                  host=resampler == "systematic" and precision != "ref64" and rng.random() < 0.2, **motion)


# ---------------------------------------------------------------------------- inputs
def _video(w, h, r, frames, vel, rng, out=None):
    """(frames (T, H, W) uint8 on the GPU, start (x, y))."""
    margin = r + 16
    x0 = rng.uniform(margin, w - 1 - margin)
    y0 = rng.uniform(margin, h - 1 - margin)

    def fold(p, lo, hi):
        q = (p - lo) % (2.0 * (hi - lo))
        return lo + (2.0 * (hi - lo) - q if q > hi - lo else q)

    cx = torch.tensor([fold(x0 + t * vel[0], r, w - 1 - r) for t in range(frames)], device="cuda")
    cy = torch.tensor([fold(y0 + t * vel[1], r, h - 1 - r) for t in range(frames)], device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(rng.randrange(1 << 31))
    ys = torch.arange(h, dtype=torch.float32, device="cuda")
    xs = torch.arange(w, dtype=torch.float32, device="cuda")
    inside = (xs[None, None, :] - cx[:, None, None]) ** 2 + (ys[None, :, None] - cy[:, None, None]) ** 2 <= float(r * r)
    img = torch.where(inside, _FG, _BG) + 5.0 * torch.randn((frames, h, w), generator=g, device="cuda")
    return torch.floor(img + 0.5).clamp_(0, 255).to(torch.uint8), (x0, y0)


def _velocity(case, rng):
    """The object's motion: the filter's own drift if it has one, else 1 to 2.3 px a frame."""
    if case["dx"] or case["dy"]:
        return case["dx"], case["dy"]
    a, s = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(1.0, 2.3)
    return s * math.cos(a), s * math.sin(a)


def _kw(case, start, seed):
    return dict(init=start, sigma=(case["sx"], case["sy"]), drift=(case["dx"], case["dy"]), seed=seed,
                resampler=case.get("resampler", "systematic"), resampler_steps=case.get("steps", 0))


def _many(case, seed, count):
    """Specifications and videos of the trackers of a batch or the streams of a server."""
    rng = random.Random(seed)
    out = []
    for i in range(count):
        size = rng.choice([256, 512, 1024])
        c = dict(w=size, h=size, r=rng.randint(3, 12), n=_log_int(rng, case["n_lo"], case["n_hi"]),
                 frames=case.get("frames", 4), sx=2.0, sy=2.0, dx=0.0, dy=0.0,
                 precision=case.get("precision") or rng.choice(["f16", "f32"]))
        video, start = _video(size, size, c["r"], c["frames"], _velocity(c, rng), rng)
        out.append((c, video, start, 1000 + i + (seed << 16)))
    return out


def _disk_half_widths(r):
    return [math.isqrt(r * r - d * d) for d in range(-r, r + 1)]


def _likelihood64(frame, r, px, py):
    """The disk likelihood of pixels (px, py), in 64 bits (template pixels clamped to the frame)."""
    x0, x1 = int(px.min()) - r, int(px.max()) + r
    y0, y1 = int(py.min()) - r, int(py.max()) + r
    h, w = frame.shape
    ix = torch.arange(x0, x1 + 1, device="cuda").clamp_(0, w - 1)
    iy = torch.arange(y0, y1 + 1, device="cuda").clamp_(0, h - 1)
    roi = frame[iy][:, ix].to(torch.int64)
    pre = torch.zeros((roi.shape[0], roi.shape[1] + 1), dtype=torch.int64, device="cuda")
    pre[:, 1:] = roi.cumsum(1)
    cols, rows = x1 - x0 + 1 - 2 * r, y1 - y0 + 1 - 2 * r
    s = torch.zeros((rows, cols), dtype=torch.int64, device="cuda")
    area = 0
    for i, hw in enumerate(_disk_half_widths(r)):
        s += pre[i:i + rows, r + hw + 1:r + hw + 1 + cols] - pre[i:i + rows, r - hw:r - hw + cols]
        area += 2 * hw + 1
    like = (_FG - _BG) * (2.0 * s.double() - (_FG + _BG) * area) / (50.0 * area)
    return like[py - (y0 + r), px - (x0 + r)]


def _step_inputs(case, seed):
    """A frame and the particles of the frame before it, as a running tracker holds them."""
    rng = random.Random(seed)
    vel = _velocity(case, rng)
    video, start = _video(case["w"], case["h"], case["r"], 2, vel, rng)
    g = torch.Generator(device="cuda")
    g.manual_seed(rng.randrange(1 << 31))
    dt = _DTYPE[case["precision"]]
    half = case["precision"] in ("f16", "bf16")
    ax, ay = math.floor(start[0] + 0.5), math.floor(start[1] + 0.5)
    x = start[0] + 1.1 * torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
    y = start[1] + 1.1 * torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
    x, y = ((x - ax).to(dt), (y - ay).to(dt)) if half else (x.to(dt), y.to(dt))
    xa, ya = (x.double() + ax, y.double() + ay) if half else (x.double(), y.double())
    like = _likelihood64(video[0], case["r"], torch.floor(xa + 0.5).long(), torch.floor(ya + 0.5).long()).to(dt)
    m = float(like.max())
    s = float(torch.exp(like.double() - m).sum())
    if case["precision"] != "ref64":
        s = float(np.float32(s))
    scalars = dict(t=4, max_l=m, sum_e=s, anchor_x=ax, anchor_y=ay, next_anchor_x=ax, next_anchor_y=ay,
                   est_x=start[0], est_y=start[1])
    return video[1].contiguous(), x, y, like, scalars, start


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        many = _many(case, seed, case["trackers"])
        cfgs = [pf.make_config(c["w"], c["h"], c["n"], c["r"], c["precision"], **_kw(c, start, sd))
                for c, _, start, sd in many]
        b = pf.Batch(cfgs)
        b.set_videos([v for _, v, _, _ in many])
        return dict(kind=kind, batch=b, frames=case["frames"])
    if kind == "serve":
        many = _many(case, seed, case["streams"])
        server = pf.Server(4 << 30, max_streams=case["streams"], queue_depth=4)
        ids = [server.open(pf.make_config(c["w"], c["h"], c["n"], c["r"], c["precision"], **_kw(c, start, sd)))
               for c, _, start, sd in many]
        return dict(kind=kind, server=server, ids=ids, videos=[v for _, v, _, _ in many], t=0)
    if kind == "step":
        frame, x, y, like, scalars, start = _step_inputs(case, seed)
        cfg = pf.make_config(case["w"], case["h"], case["n"], case["r"], case["precision"], **_kw(case, start, seed))
        hdr = pf.PfStateHeader(magic=0x31534650, precision=cfg.precision, num_particles=case["n"], **scalars)
        out = [torch.empty_like(x) for _ in range(3)]
        return dict(kind=kind, cfg=cfg, hdr=hdr, frame=frame, ins=(x, y, like), outs=out)
    rng = random.Random(seed)
    video, start = _video(case["w"], case["h"], case["r"], case["frames"], _velocity(case, rng), rng)
    f = pf.Filter(case["w"], case["h"], case["n"], case["r"], case["precision"], **_kw(case, start, seed))
    if kind == "loop":
        return dict(kind=kind, filter=f, frames=video.cpu().numpy(), t=0)
    return dict(kind=kind, filter=f, frames=video.cpu().pin_memory() if case["host"] else video, count=case["frames"])


def _bounce(t, n):
    """Frame of a resident clip of n frames played forwards and backwards."""
    k = t % (2 * n - 2)
    return k if k < n else 2 * n - 2 - k


def run(state):
    kind = state["kind"]
    if kind == "track":
        f = state["filter"]
        f.reset()
        f.run(state["frames"])
        est, stats = f.estimates(0, state["count"], with_stats=True)
        return {"estimates": est, "stats": stats}
    if kind == "loop":
        f, t = state["filter"], state["t"]
        state["t"] = t + 1
        f.step(state["frames"][_bounce(t, len(state["frames"]))])
        return {"estimate": np.array(f.estimate(t))}
    if kind == "step":
        x, y, like = state["ins"]
        ox, oy, ol = state["outs"]
        frame = state["frame"]
        hdr = pf.pf_step_frame_noalloc(state["cfg"], state["hdr"], x.data_ptr(), y.data_ptr(), like.data_ptr(),
                                       frame.data_ptr(), frame.stride(0), ox.data_ptr(), oy.data_ptr(), ol.data_ptr())
        return {"x": ox, "y": oy, "likelihood": ol, "estimate": np.array([hdr.est_x, hdr.est_y]),
                "stats": np.array([hdr.max_l, hdr.sum_e])}
    if kind == "batch":
        b = state["batch"]
        b.reset()
        b.run(state["frames"])
        return {"estimates": np.stack([b.estimates(t) for t in range(state["frames"])])}
    s, t = state["server"], state["t"]
    state["t"] = t + 1
    for sid, v in zip(state["ids"], state["videos"]):
        s.submit(sid, v[_bounce(t, len(v))])
    s.drain()
    return {"estimates": np.array([s.result(sid, t) for sid in state["ids"]])}


# ---------------------------------------------------------------------------- work
def work(case):
    """Bytes: the previous frame's positions and likelihoods read, the new ones written, every
    frame after the first; host frames copied.  Operations: per particle and frame about 25
    (two normal draws, two coordinates, a likelihood, a weight, the sums, the CDF)."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        n = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])   # mean of the log-uniform law
        if kind == "batch":
            steps = case["trackers"] * n * case["frames"]
            return {"bytes": steps * _BYTES[case["precision"]] * (6 - 3 / case["frames"]), "flops": 25 * steps}
        return {"bytes": case["streams"] * n * 6 * 3, "flops": 25 * case["streams"] * n}
    b = _BYTES[case["precision"]]
    if kind in ("loop", "step"):
        return {"bytes": 6 * b * case["n"] + (case["w"] * case["h"] if kind == "loop" else 0), "flops": 25 * case["n"]}
    moved = 3 * b * case["n"] * (2 * case["frames"] - 1)
    if case["host"]:
        moved += case["w"] * case["h"] * case["frames"]
    per = 25.0
    if case["resampler"] == "metropolis":
        per += 3.0 * (case["steps"] or 64)    # a draw, a difference and a test per chain step
    return {"bytes": moved, "flops": per * case["n"] * case["frames"]}


# ---------------------------------------------------------------------------- exact
_M32 = 0xFFFFFFFF


def _mul_hi_lo(a, b):
    """High and low words of the 32 x 32-bit product a * b (b a tensor)."""
    p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
    s = p0 + ((p1 & 0xFFFF) << 16)
    return (p1 >> 16) + (s >> 32), s & _M32


def _philox(index, t, tag, seed):
    """Four words of Philox4x32-10 for counters (index, t, tag, 0), key = the 64-bit seed."""
    like = index if isinstance(tag, int) else index + 0 * tag
    c = [like, torch.full_like(like, t), tag + 0 * like, torch.zeros_like(like)]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        h0, l0 = _mul_hi_lo(0xD2511F53, c[0])
        h1, l1 = _mul_hi_lo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _uniform(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _normals(n, t, seed):
    w = _philox(torch.arange((n + 1) // 2, device="cuda"), t, 0, seed)
    out = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        rad, ang = torch.sqrt(-2.0 * torch.log(_uniform(a))), 2.0 * math.pi * _uniform(b)
        out.append((rad * torch.cos(ang), rad * torch.sin(ang)))
    return (torch.stack([out[0][0], out[1][0]], 1).reshape(-1)[:n],
            torch.stack([out[0][1], out[1][1]], 1).reshape(-1)[:n])


def _ancestors(case, like, m, s, t, seed):
    """The ancestor of every offspring of frame t (draws of frame t - 1)."""
    n = like.numel()
    scheme = case.get("resampler", "systematic")
    j = torch.arange(n, device="cuda")
    if scheme in ("systematic", "stratified", "multinomial"):
        c = (torch.exp(like - m).cumsum(0) * (1.0 / s)).clamp_(max=1.0)
        c[-1] = 1.0
        if scheme == "systematic":
            v = _uniform(_philox(torch.zeros(1, dtype=torch.int64, device="cuda"), t - 1, 1, seed)[0])
        else:
            v = _uniform(torch.stack(_philox(torch.arange((n + 3) // 4, device="cuda"), t - 1, 1, seed), 1).reshape(-1)[:n])
        u = v if scheme == "multinomial" else (j + v) * (1.0 / n)
        return torch.searchsorted(c, u).clamp_(max=n - 1)
    if scheme == "metropolis":
        k = j.clone()
        for b in range(case["steps"] or 64):
            w = _philox(torch.full_like(j, b // 2), t - 1, 5 + 256 * j, seed)
            kk = (w[2 * (b % 2)] * n) >> 32
            k = torch.where(torch.log(_uniform(w[2 * (b % 2) + 1])) <= like[kk] - like[k], kk, k)
        return k
    if scheme == "rejection":
        a, left = j.clone(), j.clone()
        for i in range(4096):
            w = _philox(torch.full_like(left, i // 2), t - 1, 6 + 256 * left, seed)
            kk = left if i == 0 else (w[2 * (i % 2)] * n) >> 32
            a[left] = kk
            left = left[~(torch.log(_uniform(w[2 * (i % 2) + 1])) <= like[kk] - m)]
            if not left.numel():
                break
        return a
    a = torch.empty_like(j)                      # Gumbel-max
    quads = torch.arange((n + 3) // 4, device="cuda")
    for j0 in range(0, n, 512):
        jj = j[j0:j0 + 512]
        w = _philox(quads[None, :].expand(jj.numel(), -1), t - 1, 4 + 256 * jj[:, None], seed)
        g = -torch.log(-torch.log(_uniform(torch.stack(w, 2).reshape(jj.numel(), -1)[:, :n])))
        a[j0:j0 + 512] = (like[None, :] + g).argmax(1)
    return a


def _frame64(case, frame, xa, ya, t, seed):
    """Propagate, score and weigh in 64 bits: (x, y, likelihood, max, sum, estimate)."""
    nx, ny = _normals(case["n"], t, seed)
    x, y = xa + case["dx"] + case["sx"] * nx, ya + case["dy"] + case["sy"] * ny
    like = _likelihood64(frame, case["r"], torch.floor(x + 0.5).long(), torch.floor(y + 0.5).long())
    m = float(like.max())
    w = torch.exp(like - m)
    s = float(w.sum())
    cx, cy = float(x[0]), float(y[0])
    est = (cx + float((w * (x - cx)).sum()) / s, cy + float((w * (y - cy)).sum()) / s)
    return x, y, like, m, s, est


def _track64(case, frames, start, seed, count):
    est, stats = [], []
    x = torch.full((case["n"],), start[0], dtype=torch.float64, device="cuda")
    y = torch.full((case["n"],), start[1], dtype=torch.float64, device="cuda")
    like = m = s = None
    for t in range(count):
        if t:
            a = _ancestors(case, like, m, s, t, seed)
            x, y = x[a], y[a]
        x, y, like, m, s, e = _frame64(case, frames[t], x, y, t, seed)
        est.append(e)
        stats.append((m, s))
    return np.array(est), np.array(stats)


def exact(case, seed):
    """The same filter in 64 bits with torch.  Past the first resampling a track in 16 or 32
    bits is another sample of the same filter: its estimates are compared, its weight sums
    have no such value."""
    kind = case["kind"]
    if kind == "batch":
        return {"estimates": np.stack([_track64(c, v, start, sd, c["frames"])[0]
                                       for c, v, start, sd in _many(case, seed, case["trackers"])], 1)}
    if kind == "serve":
        return {"estimates": np.concatenate([_track64(c, v, start, sd, 1)[0]
                                             for c, v, start, sd in _many(case, seed, case["streams"])])}
    if kind == "step":
        frame, x, y, like, st, _ = _step_inputs(case, seed)
        half = case["precision"] in ("f16", "bf16")
        ax, ay = (st["anchor_x"], st["anchor_y"]) if half else (0.0, 0.0)
        a = _ancestors(case, like.double(), st["max_l"], st["sum_e"], st["t"], seed)
        x, y, like, m, s, est = _frame64(case, frame, x.double()[a] + ax, y.double()[a] + ay, st["t"], seed)
        return {"x": x - ax, "y": y - ay, "likelihood": like if case["precision"] == "ref64" else None,
                "estimate": np.array(est), "stats": np.array([m, s]) if case["precision"] == "ref64" else None}
    rng = random.Random(seed)
    video, start = _video(case["w"], case["h"], case["r"], case["frames"], _velocity(case, rng), rng)
    if kind == "loop":
        return {"estimate": _track64(case, video, start, seed, 1)[0][0]}
    est, stats = _track64(case, video, start, seed, case["frames"])
    return {"estimates": est, "stats": stats if case["precision"] == "ref64" else None}
