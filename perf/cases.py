"""The work that users of this library have it do, as cases to be timed.

Every case goes through the public binding (paper_2207_12011_gb300.raypc) on
the seeded synthetic shell volumes of paper_2207_12011_gb300.synth: a volume
of six mantle-convection fields, a brush box drawn around one of the three
base brushes, an orbit camera and a transfer function, all from the seed. The
sizes are those of the library's own workloads (64^3 to 512^3 cells, 256^2 to
2048^2 pixels, FP32 and FP16 storage, 256-bin histograms, 64-view batches of
mixed image sizes, 100 000-line subsamples) and ragged ones between them.

listed() gives the cases, draw() more of the same ranges, prepare() a case's
state, run() one pass, work() the bytes and operations a pass cannot do
without, and exact() the floating outputs in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2207_12011_gb300 import raypc as rp
from paper_2207_12011_gb300 import synth

COLOR_VAR = 1            # T_anom: colours every volume here (each has at least two variables)


def listed():
    return [
        # the smallest interactive step: a brush edit on a 64^3 snapshot, its frame and its plots
        dict(name="frame_64_f32_256sq", kind="frame", n=64, store="f32", nvars=6, lods=0, brush="c1", w=256, h=256,
             bins=256),
        # the same step at the ordinary size: what every move of a brush handle costs
        dict(name="frame_256_f32_1024sq", kind="frame", n=256, store="f32", nvars=6, lods=2, brush="c2", w=1024,
             h=1024, bins=256),
        # and on a full-resolution snapshot in half storage at a display's size
        dict(name="frame_512_f16_1080p", kind="frame", n=512, store="f16", nvars=6, lods=2, brush="c3", w=1920,
             h=1080, bins=256),
        # playing a simulation: the next time step comes in, and the whole path runs on it
        dict(name="step_256_f32_1024sq", kind="step", n=256, store="f32", nvars=6, lods=2, brush="c2", w=1024,
             h=1024, bins=256),
        # the preparation of a large time step alone: storage, levels of detail, brick ranges
        dict(name="ingest_512_f16", kind="ingest", n=512, store="f16", nvars=6, lods=2, brush="c3"),
        # a parameter study: many views with a brush each, in one launch
        dict(name="batch_512_f16_32views", kind="batch", n=512, store="f16", nvars=6, lods=0, brush="c3", views=32,
             smallest=256, largest=2048),
        # many clients at once: coarse and full passes and plots of three time steps
        dict(name="serve_256_f16_24req", kind="serve", n=256, store="f16", nvars=6, lods=1, brush="c3", volumes=3,
             renders=16, hists=8, smallest=256, largest=1024, bins=256),
        # the plot of the whole data set, before anything is brushed
        dict(name="hist_512_f16_all", kind="hist", n=512, store="f16", nvars=6, lods=0, brush="", bins=256),
        # the plots inside a host application that owns all device memory; a ragged edge
        dict(name="hist_noalloc_250_f16", kind="noalloc", n=250, store="f16", nvars=6, lods=0, brush="c2", bins=256),
        # a resting camera: passes that refine a cut-open view of an odd-sized grid in an odd window
        dict(name="progressive_181_f32_1237x683", kind="progressive", n=181, store="f32", nvars=5, lods=0,
             brush="c2", w=1237, h=683, passes=4),
        # a moving camera: a coarse frame with depth, warped to the next viewpoint
        dict(name="preview_256_f16_960x540", kind="preview", n=256, store="f16", nvars=6, lods=1, brush="c1", w=960,
             h=540),
        # the plot's polylines and the selection of a million pathline seeds
        dict(name="lines_256_f32_100k", kind="lines", n=256, store="f32", nvars=6, lods=0, brush="c2", k=100000,
             npts=1 << 20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edge(rng, lo, hi):
    """A grid edge: half of them multiples of 16, as simulations have them, the rest anything."""
    n = _log_int(rng, lo, hi)
    return min(hi, max(lo, (n + 8) // 16 * 16)) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "step", "ingest", "batch", "serve", "hist", "noalloc",
                       "progressive", "preview", "lines"])
    c = dict(kind=kind, n=_edge(rng, 48, 512), store=rng.choice(["f32", "f16"]), nvars=rng.choice([3, 4, 5, 6, 6, 6]),
             lods=rng.choice([0, 1, 2]), brush=rng.choice(["c1", "c2", "c3"]))
    if kind in ("frame", "step", "progressive", "preview"):
        c["w"], c["h"] = _log_int(rng, 128, 2048), _log_int(rng, 128, 2048)
    if kind in ("frame", "step", "hist", "noalloc", "serve"):
        c["bins"] = rng.choice([64, 100, 256, 256, 512])
    if kind == "hist":
        c["brush"] = rng.choice(["", "c1", "c2", "c3"])
    if kind == "batch":
        c.update(n=_edge(rng, 96, 512), lods=0, views=_log_int(rng, 2, 24), smallest=rng.choice([160, 256, 333]),
                 largest=rng.choice([512, 1000, 2048]))
    if kind == "serve":
        c.update(n=_edge(rng, 96, 256), lods=1, volumes=rng.choice([1, 2, 3]), renders=rng.randrange(4, 20),
                 hists=rng.randrange(0, 8), smallest=rng.choice([160, 256, 333]), largest=rng.choice([512, 800, 1024]))
    if kind == "progressive":
        c.update(n=_edge(rng, 48, 320), passes=rng.randrange(2, 6), lods=0)
    if kind == "preview":
        c["lods"] = 1
    if kind == "lines":
        c.update(n=_edge(rng, 48, 384), k=_log_int(rng, 1000, 100000), npts=_log_int(rng, 1000, 1 << 22), lods=0)
    if kind == "ingest":
        c["lods"] = rng.choice([1, 2, 2])
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _volume(c, seed):
    return synth.make_shell_volume(c["n"], seed=synth.DEFAULT_SEED + 7 * seed, device="cuda")[: c["nvars"]].contiguous()


def _stored(c, src):
    """The values the volume holds (FP16 storage rounds to nearest even), as float32."""
    return src.half().float() if c["store"] == "f16" else src


def _brush(c, table, seed, base=None):
    spec = {k: v for k, v in synth.edited_spec(base or c["brush"], seed).items() if synth.VAR_INDEX[k] < c["nvars"]}
    return table.brush(spec)


def _camera(seed):
    r = np.random.default_rng(seed + 17)
    return synth.orbit_camera(r.uniform(0, 360), r.uniform(-60, 60), r.uniform(2.6, 3.4))


def _position_cut(c):
    """A position brush that cuts the shell open: the half x <= 0.3 and its outer 85 %."""
    lo = np.array([-np.inf, -np.inf, -np.inf, 0.615], np.float32)
    hi = np.array([0.3, np.inf, np.inf, np.inf], np.float32)
    return lo, hi, 0b1001


def _points(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    return torch.rand((c["npts"], 3), generator=g, device="cuda") * 2.0 - 1.0


def _inputs(c, seed):
    """Source volume, stored values, brush, transfer function and camera of a single-volume case."""
    src = _volume(c, seed)
    stored = _stored(c, src)
    table = synth.QuantileTable(stored)
    brush = _brush(c, table, seed) if c["brush"] else None
    tf = synth.make_tf(stored, synth.VAR_NAMES[COLOR_VAR])
    return src, stored, brush, tf, _camera(seed)


def _sizes(c, k):
    """k square image sizes, four steps from the smallest to the largest in turn."""
    ratio = c["largest"] / c["smallest"]
    four = [int(round(c["smallest"] * ratio ** (i / 3))) for i in range(4)]
    return [four[i % 4] for i in range(k)]


def _load(ctx, c, src, tf):
    v = ctx.load_volume(src, store=c["store"])
    v.build_bricks(n_lod=c["lods"])
    v.set_tf(tf.rgbs, tf.color_var, tf.v_lo, tf.v_hi)
    return v


def prepare(c, seed):
    kind = c["kind"]
    S = dict(case=c, kind=kind, seed=seed, order=tuple(range(c["nvars"])))
    ctx = S["ctx"] = rp.Context(torch.cuda.current_device())
    if kind == "serve":
        vols, tables = [], []
        for t in range(c["volumes"]):
            src = _volume(c, 100 * seed + t)
            stored = _stored(c, src)
            tables.append(synth.QuantileTable(stored))
            edges = synth.make_edges(stored, S["order"], c["bins"])
            vols.append((_load(ctx, c, src, synth.make_tf(stored, synth.VAR_NAMES[COLOR_VAR])), edges))
        r = np.random.default_rng(seed)
        sizes = _sizes(c, c["renders"])
        reqs = []
        for i in range(c["renders"] + c["hists"]):
            t = i % c["volumes"]
            b = _brush(c, tables[t], 1000 * seed + i)
            if i < c["renders"]:
                reqs.append(("render", vols[t][0], sizes[i], _camera(1000 * seed + i), b))
            else:
                reqs.append(("hist", vols[t][0], vols[t][1], None, b))
        S["reqs"] = reqs
        S["arrival"] = r.permutation(len(reqs)).tolist()
        S["server"] = rp.Server(ctx, num_streams=3, max_batch_pixels=8_000_000)
        return S
    src, stored, brush, tf, cam = _inputs(c, seed)
    S.update(brush=brush, tf=tf, cam=cam)
    if "bins" in c:
        S["edges"] = synth.make_edges(stored, S["order"], c["bins"])
    if kind == "noalloc":
        S["cells"] = stored.half() if c["store"] == "f16" else stored
        S["out"] = torch.empty((c["nvars"] - 1, c["bins"], c["bins"]), dtype=torch.int32, device="cuda")
        return S
    v = S["vol"] = _load(ctx, c, src, tf)
    if kind == "batch":
        table = synth.QuantileTable(stored)
        S["views"] = []
        for i, s in enumerate(_sizes(c, c["views"])):
            b = _brush(c, table, 1000 * seed + i)
            S["views"].append(dict(vol=v, cam=_camera(1000 * seed + i), w=s, h=s, lo=b.lo, hi=b.hi, mask=b.active_mask,
                                   out=torch.empty((s, s, 4), dtype=torch.float32, device="cuda")))
        S["batch"] = rp.Batch(ctx, c["views"])
    if kind in ("step", "ingest"):
        S["src"] = src
    if kind == "progressive":
        v.set_position_brush(*_position_cut(c))
        S["accum"] = torch.empty((c["h"], c["w"], 4), dtype=torch.float32, device="cuda")
    if kind == "preview":
        S["next"] = _next_camera(cam)
    if kind in ("preview", "lines"):
        v.set_brush(brush.lo, brush.hi, brush.active_mask)
    if kind == "lines":
        S["points"] = _points(c, seed)
    return S


def _next_camera(cam):
    """The camera a moment later: 2 degrees on around the y axis."""
    a = math.radians(2.0)
    x, y, z = cam.eye
    return synth.Camera((x * math.cos(a) + z * math.sin(a), y, z * math.cos(a) - x * math.sin(a)), cam.target, cam.up,
                        cam.tan_half_vfov)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(S):
    c, kind = S["case"], S["kind"]
    if kind == "serve":
        return _run_serve(S)
    if kind == "batch":
        return [img for img, _ in S["batch"].render(S["views"])]
    if kind == "noalloc":
        b = S["brush"]
        return rp.pc_histogram_noalloc(S["cells"], S["order"], S["edges"], lo=b.lo, hi=b.hi, active_mask=b.active_mask,
                                       use_brush=True, out=S["out"])
    v, b = S["vol"], S["brush"]
    if kind == "ingest":
        v.update(S["src"])
        v.build_bricks(n_lod=c["lods"])
        out = [v.bricks(lod) for lod in range(c["lods"] + 1)]
        return out + [v.sub_bricks(0, classify=False)[:2]] + [v.export(lod) for lod in range(1, c["lods"] + 1)]
    if kind == "hist":
        if b is not None:
            v.set_brush(b.lo, b.hi, b.active_mask)
        return v.pc_histogram(S["order"], S["edges"], use_brush=b is not None)
    if kind == "lines":
        lines = v.pc_subsample(S["seed"], c["k"], S["order"])
        return [*lines, v.filter_points(S["points"])]
    if kind == "preview":
        img, _, depth = v.render(S["cam"], c["w"], c["h"], lod=1, tf_skip=True, depth=True)
        warped, source = rp.warp_image(S["ctx"], S["cam"], S["next"], img, depth, with_src=True, fill_holes=True)
        return img, depth, warped, source
    if kind == "progressive":
        v.set_brush(b.lo, b.hi, b.active_mask)
        for p in range(c["passes"]):
            img, _ = v.render_progressive(S["cam"], c["w"], c["h"], S["seed"] & 0xFFFF, p, S["accum"])
        return img, S["accum"]
    if kind == "step":
        v.update(S["src"])
        v.build_bricks(n_lod=c["lods"])
    v.set_brush(b.lo, b.hi, b.active_mask)
    if kind == "step":
        tf = S["tf"]
        v.set_tf(tf.rgbs, tf.color_var, tf.v_lo, tf.v_hi)
    img, _ = v.render(S["cam"], c["w"], c["h"])
    return img, v.pc_histogram(S["order"], S["edges"], use_brush=True)


def _run_serve(S):
    srv, ids, out = S["server"], [None] * len(S["reqs"]), []
    for i in S["arrival"]:
        kind, vol, what, cam, b = S["reqs"][i]
        if kind == "render":
            ids[i] = srv.submit_render(vol, cam, what, what, lo=b.lo, hi=b.hi, mask=b.active_mask, coarse_lod=1)
        else:
            ids[i] = srv.submit_histogram(vol, S["order"], what, lo=b.lo, hi=b.hi, mask=b.active_mask)
    for rid in ids:
        r = srv.poll(rid, timeout_us=20_000_000)
        if not r["done"] or r["status"] != 0:
            raise RuntimeError(f"request {rid} ended with status {r['status']}, done {r['done']}")
        # the server owns the result's memory until it is released: a client keeps a copy
        out += [r["hist"].clone()] if "hist" in r else [r["coarse"].clone(), r["image"].clone()]
    torch.cuda.current_stream().synchronize()        # the copies are done before the memory is given back
    for rid in ids:
        srv.release(rid)
    return out


# ---------------------------------------------------------------------------
# The work a pass cannot do without
# ---------------------------------------------------------------------------
def _lattice(w, h, n, dist=3.0):
    """Lattice samples of a w x h frame (steps of 1/n) inside the shell's outer sphere."""
    th = math.tan(math.radians(22.5))
    sx = ((2 * np.arange(64) + 1) / 64 - 1) * th * w / h
    sy = ((2 * np.arange(64) + 1) / 64 - 1) * th
    q = sx[None, :] ** 2 + sy[:, None] ** 2
    disc = 1.0 - dist * dist * q / (1.0 + q)           # 1 - (distance of the ray to the centre)^2
    return float(2.0 * np.sqrt(np.maximum(disc, 0.0)).mean() * n * w * h)


SAMPLE_FLOPS = 32        # position 6, |p|^2 5, one trilinear interpolation 21


def work(c):
    kind, n, e = c["kind"], c["n"], 2 if c["store"] == "f16" else 4
    field = float(n) ** 3 * c["nvars"] * e
    counts = 4.0 * (c["nvars"] - 1) * c.get("bins", 0) ** 2
    image = 16.0 * c.get("w", 0) * c.get("h", 0)
    levels = sum(8.0 ** -k for k in range(1, c["lods"] + 1))
    nbrick = ((n + 7) // 8) ** 3 * c["nvars"] * 8.0
    if kind == "frame":
        return {"bytes": field + image + counts, "flops": SAMPLE_FLOPS * _lattice(c["w"], c["h"], n)}
    if kind == "step":
        return {"bytes": 4.0 * n ** 3 * c["nvars"] + field * (1 + levels) + nbrick + image + counts,
                "flops": SAMPLE_FLOPS * _lattice(c["w"], c["h"], n)}
    if kind == "ingest":
        nsub = ((n + 3) // 4) ** 3 * c["nvars"] * 8.0
        return {"bytes": 4.0 * n ** 3 * c["nvars"] + field * (1 + levels) + nbrick * (1 + levels) + nsub, "flops": 0.0}
    if kind == "batch":
        s = _sizes(c, c["views"])
        return {"bytes": field + 16.0 * sum(x * x for x in s), "flops": SAMPLE_FLOPS * sum(_lattice(x, x, n) for x in s)}
    if kind == "serve":
        s = _sizes(c, c["renders"])
        return {"bytes": c["volumes"] * field * (1 + levels) + 32.0 * sum(x * x for x in s) + c["hists"] * counts,
                "flops": SAMPLE_FLOPS * 1.5 * sum(_lattice(x, x, n) for x in s)}
    if kind in ("hist", "noalloc"):
        return {"bytes": field + counts, "flops": 0.0}
    if kind == "progressive":
        return {"bytes": field + 3.0 * image * c["passes"], "flops": SAMPLE_FLOPS * 0.65 * c["passes"] * _lattice(c["w"], c["h"], n)}
    if kind == "preview":
        return {"bytes": field / 8 + 2.5 * image, "flops": SAMPLE_FLOPS * _lattice(c["w"], c["h"], n / 2)}
    m = min(c["k"], int(3.5 * n ** 3 / 8))
    points = c["npts"] * 13.0 + min(field, c["npts"] * 0.45 * 8.0 * e)
    return {"bytes": m * (9.0 + 4 * c["nvars"] + c["nvars"] * e) + points, "flops": c["npts"] * 0.45 * 21.0}


# ---------------------------------------------------------------------------
# The floating outputs in 64 bits: the method's definitions in plain torch
# ---------------------------------------------------------------------------
def _lsr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _signed(u):
    return u - (1 << 64) if u >= 1 << 63 else u


def _jitter(seed, p, npix, dev):
    """Lattice offsets of progressive pass p: 1/2, or the top 24 bits of SplitMix64 per pixel."""
    if p == 0:
        return torch.full((npix,), 0.5, dtype=torch.float64, device=dev)
    z = torch.arange(1, npix + 1, dtype=torch.int64, device=dev) * _signed(0x9E3779B97F4A7C15) + _signed((seed << 32) | p)
    z = (z ^ _lsr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ _lsr(z, 27)) * _signed(0x94D049BB133111EB)
    return _lsr(z ^ _lsr(z, 31), 40).double() * 2.0 ** -24


def _interpolate(field, u):
    """Trilinear values of one variable at grid coordinates u ([m, 3], x y z), in 64 bits."""
    n = field.shape[0]
    u = u.clamp(0.0, n - 1.0)
    i = u.floor().clamp(max=n - 2)
    f, i = u - i, i.long()
    flat, base = field.reshape(-1), (i[:, 2] * n + i[:, 1]) * n + i[:, 0]
    at = lambda o: flat[base + o].double()  # noqa: E731
    lerp = lambda a, b, t: a + t * (b - a)  # noqa: E731
    rows = [lerp(at(o), at(o + 1), f[:, 0]) for o in (0, n, n * n, n * n + n)]
    return lerp(lerp(rows[0], rows[1], f[:, 1]), lerp(rows[2], rows[3], f[:, 1]), f[:, 2])


def _march(vol, brush, tf, cam, w, h, jitter=None, cut=None):
    """The emission-absorption frame of the stored values vol under a brush, early termination on."""
    dev, n = vol.device, vol.shape[-1]
    dt = float(np.float32(1.0 / n))
    a = torch.tensor(cam.as_array(), dtype=torch.float64, device=dev)
    eye, fwd = a[0:3], torch.nn.functional.normalize(a[3:6] - a[0:3], dim=0)
    right = torch.nn.functional.normalize(torch.linalg.cross(fwd, a[6:9]), dim=0)
    up = torch.linalg.cross(right, fwd)
    table = torch.tensor(tf.rgbs, dtype=torch.float64, device=dev)
    names = [v for v in range(vol.shape[0]) if (brush.active_mask >> v) & 1]
    out = torch.zeros((w * h, 4), dtype=torch.float64, device=dev)
    rin2, rout2 = float(np.float32(synth.R_IN) ** 2), float(np.float32(synth.R_OUT) ** 2)
    K = 2 * n + 2
    chunk = max(256, (1 << 23) // K)
    for p0 in range(0, w * h, chunk):
        pix = torch.arange(p0, min(w * h, p0 + chunk), device=dev)
        sx = ((2 * (pix % w) + 1).double() / w - 1.0) * float(a[9]) * w / h
        sy = (1.0 - (2 * (pix // w) + 1).double() / h) * float(a[9])
        d = torch.nn.functional.normalize(fwd + sx[:, None] * right + sy[:, None] * up, dim=1)
        b = d @ eye
        disc = rout2 - (eye - b[:, None] * d).square().sum(1)
        root = disc.clamp(min=0.0).sqrt()
        t0, t1 = (-b - root).clamp(min=0.0), -b + root
        j = 0.5 if jitter is None else jitter[pix][:, None]
        t = t0[:, None] + (torch.arange(K, device=dev) + j) * dt
        ray, k = torch.nonzero((t < t1[:, None]) & (disc > 0.0)[:, None], as_tuple=True)
        pos = eye + t[ray, k][:, None] * d[ray]
        r2 = pos.square().sum(1)
        ok = (r2 >= rin2) & (r2 <= rout2)
        if cut is not None:
            lo, hi, _ = cut
            ok &= (pos[:, 0] <= float(hi[0])) & (r2.sqrt() >= float(lo[3]))
        ray, k, pos = ray[ok], k[ok], pos[ok]
        u = pos * (0.5 * n) + (0.5 * n - 0.5)
        for v in names:
            s = _interpolate(vol[v], u)
            ok = (s >= float(brush.lo[v])) & (s <= float(brush.hi[v]))
            ray, k, u = ray[ok], k[ok], u[ok]
        s = ((_interpolate(vol[tf.color_var], u) - tf.v_lo) * (255.0 / (tf.v_hi - tf.v_lo))).clamp(0.0, 255.0)
        e = s.floor().clamp(max=254.0)
        f, e = (s - e)[:, None], e.long()
        rgbs = table[e] + f * (table[e + 1] - table[e])
        alpha = 1.0 - torch.exp(-rgbs[:, 3] * dt)
        through = torch.ones((len(pix), K + 1), dtype=torch.float64, device=dev)
        through[ray, k + 1] = 1.0 - alpha
        before = torch.cumprod(through, dim=1)[ray, k]
        wgt = torch.where(before > 2.0 ** -12, before * alpha, torch.zeros_like(alpha))
        part = torch.cat([wgt[:, None] * rgbs[:, :3], wgt[:, None]], dim=1)
        out[p0:p0 + len(pix)].index_add_(0, ray, part)
    return out.reshape(h, w, 4)


def _coarser(c, vol):
    """The next level: means of 2^3 cells, edges clamped, in the storage type."""
    n = vol.shape[-1]
    if n % 2:
        vol = torch.nn.functional.pad(vol[None], (0, 1, 0, 1, 0, 1), mode="replicate")[0]
    m = torch.nn.functional.avg_pool3d(vol[None].double(), 2)[0]
    return m.half().float() if c["store"] == "f16" else m.float()


def _ranges(vol, edge):
    """Min and max over the vertices e*b .. min(e*b + e, n-1) of every brick, as [b, b, b, v] twice."""
    n = vol.shape[-1]
    nb = (n + edge - 1) // edge
    pad = nb * edge + 1 - n
    got = []
    for sign in (-1.0, 1.0):
        # a replicated edge adds no new value
        x = torch.nn.functional.pad((vol * sign)[None], (0, pad) * 3, mode="replicate")[0]
        x = torch.nn.functional.max_pool3d(x[None], edge + 1, stride=edge)[0]
        got.append((x * sign)[:, :nb, :nb, :nb].permute(1, 2, 3, 0).contiguous().double())
    return tuple(got)


def exact(c, seed):
    kind = c["kind"]
    if kind in ("batch", "serve", "hist", "noalloc", "lines"):
        return None                          # counts and bytes, copies of stored values, or far too long in 64 bits
    src, stored, brush, tf, cam = _inputs(c, seed)
    if kind == "ingest":
        levels = [stored]
        for _ in range(c["lods"]):
            levels.append(_coarser(c, levels[-1]))
        return [_ranges(v, 8) for v in levels] + [_ranges(stored, 4)] + [v.double() for v in levels[1:]]
    if _lattice(c["w"], c["h"], c["n"]) * c.get("passes", 1) > 2e9:
        return None
    if kind == "preview":
        return _march(_coarser(c, stored), brush, tf, cam, c["w"], c["h"]), None, None, None
    if kind == "progressive":
        total = 0.0
        for p in range(c["passes"]):
            img = _march(stored, brush, tf, cam, c["w"], c["h"], _jitter(seed & 0xFFFF, p, c["w"] * c["h"], stored.device),
                         _position_cut(c))
            total = total + img
        return img, total / c["passes"]
    return _march(stored, brush, tf, cam, c["w"], c["h"]), None
