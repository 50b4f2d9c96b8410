"""Performance cases of the track-finding library: what its users run, over the real range of sizes.

Views are slabs of emulsion in 10 nm units (300 x 300 x 50 um, or the 1000 x 1000 x 50 um scan), grains are
fog plus straight tracks, with the seed window, tube radius and hit threshold of the shipped workloads
(synth.params).  Camera stacks are 1280 x 1024 x 40 frames or odd-sized crops of one.  Kinds of case:

* view   -- one view per call, host grains in, tracks out (View.load_host / find / fetch);
* batch  -- many views in one launch sequence, grains on the device (Batch.load / find / fetch);
* served -- views submitted one by one to the served loop and collected;
* frames -- raw camera frames on the device to grains (Frames.run / fetch);
* chain  -- raw frames to grains to tracks without leaving the device (Frames.to_batch / Batch.find);
* counts -- tube counts of caller-chosen grain pairs without allocation.
"""
import math

import numpy as np
import torch

from paper_1311_5334_gb300 import et, synth

UM = synth.UM
SLAB = (300 * UM, 300 * UM, 50 * UM)
SCAN = (1000 * UM, 1000 * UM, 50 * UM)
NOALLOC_MAX_GRAINS = 65536   # the documented limit of the allocation-free counts
VARIANT = dict(flags=et.FLAG_SINGLE_PASS | et.FLAG_ANGLE_CUT, cut=(9, 3, 4))


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # a nearly empty view at the edge of a plate: launches and latency are all there is
        dict(name="view_301", kind="view", fog=301, through=5, short=2),
        # one microscope view of the small workload, called for each view as it arrives
        dict(name="view_pr1", kind="view", fog=2000, through=20, short=0),
        # one crowded view with short heavily ionising tracks
        dict(name="view_dense", kind="view", fog=20000, through=200, short=100),
        # a large-field scan at the highest fog density
        dict(name="view_scan", kind="view", fog=1000000, through=4000, short=1000, scan=True),
        # a micro-batch as a microscope that buffers a few seconds makes it; another shape each time, so no graph
        dict(name="batch_17", kind="batch", views=17, graph=False, variant=False),
        # the throughput form: one captured launch sequence over 256 views of very different sizes
        dict(name="batch_256", kind="batch", views=256, graph=True, variant=False),
        # the other reading of the association with the background cut, on half a batch
        dict(name="batch_65_single_pass", kind="batch", views=65, graph=False, variant=True),
        # the served loop under a burst: 96 views submitted back to back, all results collected
        dict(name="served_96", kind="served", views=96),
        # one full camera stack, as an online filter sees it
        dict(name="frames_1", kind="frames", views=1, w=1280, h=1024, d=40, pad=0),
        # a block of full stacks kept in device memory
        dict(name="frames_24", kind="frames", views=24, w=1280, h=1024, d=40, pad=0),
        # an odd crop with padded rows, all the way from frames to tracks
        dict(name="chain_3_odd", kind="chain", views=3, w=1001, h=777, d=37, pad=23),
        # hypotheses of another program checked on a crowded view without any allocation
        dict(name="counts_29k", kind="counts", fog=20000, through=200, short=100, pairs=400001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "batch", "batch", "served", "frames", "chain", "counts"])
    if kind == "view":
        fog = _log(rng, 200, 60000)
        return dict(kind="view", fog=fog, through=max(1, fog // rng.randint(80, 120)), short=fog // rng.randint(200, 1000))
    if kind == "batch":
        return dict(kind="batch", views=_log(rng, 2, 240), graph=rng.random() < 0.5, variant=rng.random() < 0.25)
    if kind == "served":
        return dict(kind="served", views=_log(rng, 2, 200))
    if kind == "counts":
        fog = _log(rng, 500, 45000)
        return dict(kind="counts", fog=fog, through=fog // 100, short=fog // 200, pairs=_log(rng, 1000, 1500000))
    w, h, d = rng.randint(200, 1400), rng.randint(150, 1100), rng.randint(5, 48)
    if rng.random() < 0.4:
        w, h, d = 1280, 1024, 40
    return dict(kind=kind, views=_log(rng, 1, 24 if kind == "frames" else 8), w=w, h=h, d=d,
                pad=-w % 16 + 16 * rng.randint(0, 2))


# ---------------------------------------------------------------- inputs

def _grains(rng, extent, fog, through, short):
    """Grains of many views at once, by the recipe of synth.make_view: fog[v] uniform grains, through[v] isotropic
    crossing tracks (mean gap 3.3 um) and short[v] tracks of 10-50 um (mean gap 1.6 um) for view v, jittered,
    rounded, coincident ones dropped, in random order.  Returns (xyz int32 [n][3], offsets int64 [V + 1])."""
    fog, through, short = (np.asarray(a, dtype=np.int64) for a in (fog, through, short))
    nv = fog.size
    ext = np.asarray(extent, dtype=np.int64)
    e_um = ext / float(UM)
    pts = [rng.integers(0, ext, size=(int(fog.sum()), 3), dtype=np.int64)]
    view = [np.repeat(np.arange(nv), fog)]
    for count, gap, span in ((through, 3.3, None), (short, 1.6, (10.0, 50.0))):
        k = int(count.sum())
        if k == 0:
            continue
        cos = rng.uniform(-1.0, 1.0, k)
        phi = rng.uniform(0.0, 2.0 * math.pi, k)
        sin = np.sqrt(np.maximum(0.0, 1.0 - cos * cos))
        u = np.stack([sin * np.cos(phi), sin * np.sin(phi), cos], axis=1)
        p = rng.uniform(0.0, 1.0, (k, 3)) * e_um
        with np.errstate(divide="ignore", invalid="ignore"):
            a, b = (0.0 - p) / u, (e_um - p) / u
        t0, t1 = np.nanmax(np.minimum(a, b), axis=1), np.nanmin(np.maximum(a, b), axis=1)
        if span is not None:
            t1, t0 = np.minimum(t1, rng.uniform(*span, k)), np.zeros(k)
        steps = int(np.max(t1 - t0) / gap * 1.3) + 40
        t = t0[:, None] + np.cumsum(rng.exponential(gap, (k, steps)), axis=1)
        row, col = np.nonzero(t <= t1[:, None])
        q = p[row] + t[row, col][:, None] * u[row]
        q[:, :2] += rng.normal(0.0, 0.05, (q.shape[0], 2))
        q[:, 2] += rng.normal(0.0, 0.3, q.shape[0])
        pts.append(np.clip(np.rint(q * UM).astype(np.int64), 0, ext - 1))
        view.append(np.repeat(np.arange(nv), count)[row])
    pts, view = np.concatenate(pts), np.concatenate(view)
    key = ((view * ext[0] + pts[:, 0]) * ext[1] + pts[:, 1]) * ext[2] + pts[:, 2]
    keep = np.unique(key, return_index=True)[1]
    keep = keep[rng.permutation(keep.size)]
    keep = keep[np.argsort(view[keep], kind="stable")]
    offs = np.zeros(nv + 1, dtype=np.int64)
    offs[1:] = np.cumsum(np.bincount(view[keep], minlength=nv))
    return np.ascontiguousarray(pts[keep].astype(np.int32)), offs


def _batch_grains(rng, views):
    """Views of the batched workload: lognormal fog counts in [2k, 50k], tracks at 1 % of the fog."""
    fog = synth.lognormal_sizes(rng, views)
    return _grains(rng, SLAB, fog, np.rint(0.01 * fog).astype(np.int64), np.zeros_like(fog))


def _stacks(case, seed):
    """Raw frames on the device by the recipe of synth.render (dark Gaussian blobs, sensitivity pattern of one
    camera, noise): (uint8 [views][d][h][pitch], gain, thr)."""
    views, w, h, d = case["views"], case["w"], case["h"], case["d"]
    pitch = w + case["pad"]
    cam = np.random.default_rng([seed, 77])
    col = np.clip(cam.standard_normal(w), -2.5, 2.5)
    s = 1.0 + 0.08 * col[None, :] + 0.03 * np.clip(cam.standard_normal((h, w)), -3.0, 3.0)
    gain = np.clip(np.rint(128.0 / s), 0, 255).astype(np.uint8)
    thr = np.clip(np.rint(55.0 * s * gain / 128.0) + 10, 0, 255).astype(np.uint8)
    rng = np.random.default_rng([seed, 78])
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    ext = _stack_extent(w, h, d)
    area = w * h * d / float(1280 * 1024 * 40)
    sd = torch.from_numpy(s.astype(np.float32)).cuda()
    raw = torch.empty((views, d, h, pitch), dtype=torch.uint8, device="cuda")
    dz, dy, dx = (torch.from_numpy(a.ravel()).cuda() for a in
                  np.meshgrid(np.arange(-2, 3), np.arange(-3, 4), np.arange(-3, 4), indexing="ij"))
    for v in range(views):
        xyz, _ = _grains(rng, ext, [int(10000 * area)], [int(100 * area) + 1], [0])
        g = torch.from_numpy(xyz.astype(np.float32)).cuda()
        c = [g[:, k] * (synth.PITCH_DEN[k] / synth.PITCH_NUM[k]) for k in range(3)]
        amp = torch.from_numpy(rng.uniform(60.0, 110.0, xyz.shape[0]).astype(np.float32)).cuda()
        ix, iy, iz = (torch.round(c[k])[:, None].long() + o[None] for k, o in enumerate((dx, dy, dz)))
        wgt = amp[:, None] * torch.exp(-((ix - c[0][:, None]) ** 2 + (iy - c[1][:, None]) ** 2) / 2.0
                                       - (iz - c[2][:, None]) ** 2 / 1.28)
        ok = (ix >= 0) & (ix < w) & (iy >= 0) & (iy < h) & (iz >= 0) & (iz < d)
        # whole-number sums: the order of the additions leaves no trace
        sig = torch.zeros(d * h * w, dtype=torch.int32, device="cuda")
        sig.index_add_(0, ((iz * h + iy) * w + ix)[ok], torch.round(wgt[ok] * 1024.0).int())
        dark = torch.randn((d, h, w), generator=gen, device="cuda") * 3.0 + sig.view(d, h, w) / 1024.0 + 55.0
        raw[v, :, :, :w] = torch.clamp(torch.round(255.0 - sd[None] * dark), 0, 255).to(torch.uint8)
        if pitch > w:
            raw[v, :, :, w:] = torch.randint(0, 256, (d, h, pitch - w), generator=gen, device="cuda",
                                             dtype=torch.uint8)
    return raw, gain, thr


def _stack_extent(w, h, d):
    """A slab that holds every grain of a w x h x d stack."""
    return tuple(((n - 1) * num + den // 2) // den + 1
                 for n, num, den in zip((w, h, d), synth.PITCH_NUM, synth.PITCH_DEN))


def _grain_cap(case):
    """Grains a case can hold at most, whatever its seed draws (a track leaves well under 130 grains)."""
    if case["kind"] in ("batch", "served"):
        return min(case["views"] * 70000, case["views"] * 22000 + 500000)
    if case["kind"] in ("frames", "chain"):
        return case["views"] * (2000 + case["w"] * case["h"] * case["d"] // 2500)
    return case["fog"] + 130 * case["through"] + 60 * case["short"]


def _track_buffers(case):
    """Result buffers a program keeps: a track owns at least min_hits grains and a grain has one track."""
    n = _grain_cap(case)
    return np.zeros(n // synth.MIN_HITS + 1, dtype=et.TRACK_DTYPE), np.zeros(n, dtype=np.int32)


_context = []


def _ctx():
    """The program's context, made once."""
    if not _context:
        _context.append(et.Context(0))
    return _context[0]


class _State:
    """What a program keeps between calls; its handles are given back with it."""

    def __init__(self, kind, **kw):
        self.kind, self.owned = kind, []
        self.__dict__.update(kw)

    def own(self, handle):
        self.owned.append(handle)
        return handle

    def __del__(self):
        for h in self.owned:
            h.close()


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([seed, 1])
    s = _State(kind)
    if kind == "view":
        extent = SCAN if case.get("scan") else SLAB
        s.xyz, _ = _grains(rng, extent, [case["fog"]], [case["through"]], [case["short"]])
        s.view = s.own(_ctx().view(s.xyz, synth.params(extent)))
        s.out = _track_buffers(case)
    elif kind == "batch":
        xyz, s.offs = _batch_grains(rng, case["views"])
        s.xyz = torch.from_numpy(xyz).cuda()
        s.graph = case["graph"]
        s.batch = s.own(_ctx().batch(synth.params(SLAB, **(VARIANT if case["variant"] else {}))))
        s.out = _track_buffers(case) + (np.zeros(case["views"] + 1, dtype=np.int64),)
    elif kind == "served":
        xyz, offs = _batch_grains(rng, case["views"])
        s.views = [np.ascontiguousarray(xyz[offs[k]:offs[k + 1]]) for k in range(case["views"])]
        s.server = s.own(_ctx().server(synth.params(SLAB), 20 << 30))
        s.out = _track_buffers(case) + (np.zeros(case["views"] + 1, dtype=np.int64),)
    elif kind == "counts":
        xyz, _ = _grains(rng, SLAB, [case["fog"]], [case["through"]], [case["short"]])
        xyz = xyz[:NOALLOC_MAX_GRAINS]
        s.xyz = torch.from_numpy(xyz).cuda()
        s.pairs = torch.from_numpy(_near_pairs(rng, xyz, case["pairs"])).cuda()
        s.params = synth.params(SLAB)
        s.counts = torch.empty(s.pairs.shape[0], dtype=torch.int32, device="cuda")
    else:
        s.raw, gain, thr = _stacks(case, seed)
        fp = et.make_frame_params(case["w"], case["h"], case["d"], synth.PITCH_NUM, synth.PITCH_DEN,
                                  synth.GRAIN_THRESHOLD, row_pitch=case["w"] + case["pad"])
        s.frames = s.own(_ctx().frames(fp, gain, thr))
        offs, cap = np.zeros(case["views"] + 1, dtype=np.int64), _grain_cap(case)
        s.out = (np.zeros((cap, 3), dtype=np.int32), np.zeros(cap, dtype=np.int32), offs)
        if kind == "chain":
            s.out = _track_buffers(case) + (offs,)
            s.batch = s.own(_ctx().batch(synth.params(_stack_extent(case["w"], case["h"], case["d"]))))
    torch.cuda.synchronize()
    return s


def _near_pairs(rng, xyz, count):
    """Pairs of grains of neighbouring 15 um cubes, the hypotheses another program would ask about."""
    c = xyz // 1500
    order = np.lexsort((c[:, 2], c[:, 1], c[:, 0]))
    i = rng.integers(0, xyz.shape[0] - 1, count)
    j = np.minimum(i + rng.integers(1, 24, count), xyz.shape[0] - 1)
    return np.ascontiguousarray(np.stack([order[i], order[j]], axis=1).astype(np.int32))


# ---------------------------------------------------------------- one pass

TRACK_COLUMNS = ("seed_i", "seed_j", "nhits", "view", "member_offset", "count", "c", "u", "tmin", "tmax")


def _result(out):
    """The program's result buffers (zero behind the last track), a track's fields by name."""
    res = {k: out[0][k] for k in TRACK_COLUMNS}
    res["members"] = out[1]
    if len(out) > 2:
        res["offsets"] = out[2]
    return res


def run(state):
    s = state
    if s.kind == "view":
        s.view.load_host(s.xyz)
        s.view.find()
        s.view.fetch(out=s.out)
        return _result(s.out)
    if s.kind == "batch":
        s.batch.load(s.xyz, s.offs)
        s.batch.find(use_graph=s.graph)
        s.batch.fetch(out=s.out)
        return _result(s.out)
    if s.kind == "served":
        for tag, xyz in enumerate(s.views):
            if s.server.submit(xyz, tag) != et.OK:
                raise RuntimeError("the served loop refused a view")
        got = {}
        while len(got) < len(s.views):
            for r in s.server.poll(timeout_us=20000):
                got[int(r.tag)] = s.server.fetch(int(r.tag))
        tracks, members, offs = s.out
        n = m = 0
        for k in range(len(s.views)):
            t, g = got[k]
            tracks[n:n + t.shape[0]], members[m:m + g.shape[0]] = t, g
            n, m = n + t.shape[0], m + g.shape[0]
            offs[k + 1] = n
        return _result(s.out)
    if s.kind == "counts":
        et.tube_count_noalloc(s.xyz, s.params, s.pairs, s.counts, stream=torch.cuda.current_stream())
        return s.counts
    s.frames.run(s.raw)
    if s.kind == "frames":
        s.frames.fetch(out=s.out)
        return dict(zip(("xyz", "pulse", "offsets"), s.out))
    s.frames.to_batch(s.batch)
    s.batch.find()
    s.batch.fetch(out=s.out)
    return _result(s.out)


# ---------------------------------------------------------------- what a pass cannot do without

def _track_work(views, grains, extent):
    """Grains read once; per seed pair of the window 6 operations for the window test and 14 for each of the about
    three grains its tube holds; about one 64-byte track with 20 members per 100 grains."""
    vol = extent[0] * extent[1] * extent[2] / 1e6
    frac = min(1.0, 0.75 * 4.0 / 3.0 * math.pi * (20.0 ** 3 - 5.0 ** 3) / vol)
    seeds = views * 0.5 * grains * grains * frac
    return 12.0 * views * grains + 1.5 * views * grains, seeds * (6 + 3 * 14)


def work(case):
    kind = case["kind"]
    if kind == "view":
        extent = SCAN if case.get("scan") else SLAB
        b, f = _track_work(1, case["fog"] + 30 * case["through"] + 15 * case["short"], extent)
    elif kind in ("batch", "served"):
        # lognormal sizes: mean 16,150 grains, root mean square 19,800
        b, f = _track_work(case["views"], 19800, SLAB)
        b = case["views"] * 16150 * 13.5
    elif kind == "counts":
        n = case["fog"] + 30 * case["through"] + 15 * case["short"]
        b, f = 12.0 * n + 12.0 * case["pairs"], 14.0 * 3 * case["pairs"]
    else:
        vox = case["w"] * case["h"] * case["d"]
        grains = 12600.0 * vox / (1280 * 1024 * 40)
        b = case["views"] * (vox + 16.0 * grains) + 3.0 * case["w"] * case["h"]
        f = 1.0 * case["views"] * vox
        if kind == "chain":
            bt, ft = _track_work(case["views"], grains, _stack_extent(case["w"], case["h"], case["d"]))
            b, f = b + bt, f + ft
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in plain 64-bit arithmetic

def exact(case, seed):
    """The tracks of one small view by brute force (whole numbers) with a float64 fit; None for the rest, whose
    outputs are whole numbers or whose size is beyond brute force."""
    if case["kind"] != "view" or case["fog"] > 2600:
        return None
    rng = np.random.default_rng([seed, 1])
    xyz, _ = _grains(rng, SLAB, [case["fog"]], [case["through"]], [case["short"]])
    p = synth.params(SLAB)
    order = np.lexsort((xyz[:, 2], xyz[:, 1], xyz[:, 0]))
    g = xyz[order].astype(np.int64)                      # canonical order: index = rank
    n = g.shape[0]
    seeds = []
    for a in range(n):
        d = g[a + 1:] - g[a]
        d2 = (d * d).sum(1)
        b = np.nonzero((d2 >= p["seed_min"] ** 2) & (d2 < p["seed_max"] ** 2))[0] + a + 1
        seeds.append(np.stack([np.full(b.size, a), b], axis=1))
    seeds = np.concatenate(seeds)

    def inside(part):
        a, w = g[part[:, 0]][:, None], (g[part[:, 1]] - g[part[:, 0]])[:, None]
        c = np.cross(g[None] - a, w)
        return (c * c).sum(2) <= p["tube_r"] ** 2 * (w * w).sum(2)

    cands = []
    for k in range(0, seeds.shape[0], 512):
        part = seeds[k:k + 512]
        hit = inside(part)
        for i in np.nonzero(hit.sum(1) >= p["min_hits"])[0]:
            m = np.nonzero(hit[i])[0]
            cands.append((-m.size, int(part[i, 0]), int(part[i, 1]), m))
    cands.sort(key=lambda c: c[:3])
    used = np.zeros(n, dtype=bool)
    tracks = np.zeros(_grain_cap(case) // p["min_hits"] + 1, dtype=[
        (k, np.float64 if k in ("c", "u", "tmin", "tmax") else np.int64, (3,) if k in ("c", "u") else ())
        for k in TRACK_COLUMNS])
    members = np.zeros(_grain_cap(case), dtype=np.int64)
    nt = nm = 0
    for neg, lo, hi, m in cands:
        m = m[~used[m]]
        if m.size < p["min_hits"]:
            continue
        used[m] = True
        q = g[m].astype(np.float64)
        c = q.mean(0)
        u = np.linalg.eigh((q - c).T @ (q - c))[1][:, 2]
        u = u if u @ (g[hi] - g[lo]) > 0 else -u
        t = (q - c) @ u
        tracks[nt] = (order[lo], order[hi], m.size, 0, nm, -neg, c, u, t.min(), t.max())
        members[nm:nm + m.size] = np.sort(order[m])
        nt, nm = nt + 1, nm + m.size
    return _result((tracks, members))
