"""Performance cases of the Flow Fields matching loop: what a program does with it.

Every case goes through the public binding (``paper_1703_02563_gb300.ff``).  The frames are
seeded stand-ins for video: depth-ordered layers of value-noise texture with flat patches,
each with its own affine motion, so that frame 2 shows sub-pixel motion, occlusions and
regions where many feature vectors are equal.  Three-channel frames have the value spread of
8-bit CIELab (a full-range L, narrow a and b around 128).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1703_02563_gb300 import ff

OPS_PER_DIM = 11      # integer operations of one feature dimension of one matching error
SCHEDULES = {"basic": ff.FF_SCHED_BASIC, "plus": ff.FF_SCHED_PLUS, "fast": ff.FF_SCHED_PLUS_FAST,
             "fast_x2": ff.FF_SCHED_PLUS_FAST_X2}
BATCH_SIZES = ((320, 240), (640, 480), (1024, 436), (1242, 375))


def listed() -> list[dict]:
    return [
        # one tiny gray pair, device calls in order: latency of the shortest whole use
        dict(name="pair_gray_128x96", kind="pair", w=128, h=96, channels=1, scales=3, iters=4,
             radius=8, schedule="basic"),
        # an ordinary colour video pair (Sintel's frame shape), device calls in order
        dict(name="pair_lab_1024x436", kind="pair", w=1024, h=436, channels=3, scales=4, iters=6,
             radius=8, schedule="basic"),
        # a gray driving pair (KITTI's frame shape) from pinned host buffers in one call
        dict(name="host_gray_1242x375", kind="host", w=1242, h=375, channels=1, scales=4, iters=4,
             radius=12, schedule="basic", region_min=0),
        # a full-HD colour pair from pinned host buffers with the region filter: one large call
        dict(name="host_lab_1920x1080", kind="host", w=1920, h=1080, channels=3, scales=4, iters=6,
             radius=8, schedule="basic", region_min=150),
        # the fast schedule as the paper's real-time variant uses it: 2nd-finest grid, sparse
        # candidates, two backward flows, two-way check, region filter, one match per cell; odd size
        dict(name="fast_x2_2way_lab_1023x435", kind="two_way", w=1023, h=435, channels=3, scales=4,
             iters=4, radius=8, schedule="fast_x2", stride=2, region=150, cell=3, least=2),
        # the accurate schedule in one direction from a caller's own seeds, with costs; odd size
        dict(name="seeded_plus_gray_641x479", kind="seeded", w=641, h=479, channels=1, scales=4,
             iters=4, radius=8, schedule="plus"),
        # offline throughput: many colour pairs of mixed sizes, one captured graph per batch
        dict(name="batch_lab_mixed_x20", kind="batch", sizes="mixed", w=1242, h=480, pairs=20,
             slots=20, channels=3, scales=4, iters=6, radius=8, schedule="basic"),
        # a burst of host requests of many sizes through the serving loop until all are answered
        dict(name="serve_lab_x24", kind="serve", w=1920, h=1080, requests=24, slots=12, channels=3,
             scales=4, iters=6, radius=8, schedule="basic"),
        # feature extraction on its own, every level read out
        dict(name="features_lab_1242x375", kind="features", w=1242, h=375, channels=3, scales=4,
             tensor_cores=0),
        # the exact nearest-feature search on its own (seeds for another matcher)
        dict(name="knn_lab_1024x436", kind="knn", w=1024, h=436, channels=3, scales=4, leaf=8,
             stride=1),
        # the same search for a program that may not allocate, gray, every second candidate
        dict(name="knn_static_gray_640x480", kind="knn_static", w=640, h=480, channels=1, scales=4,
             leaf=8, stride=2),
        # the unrounded scale-space transform on the tensor cores, half precision, all levels
        dict(name="scalespace_fp16_lab_1242x375", kind="scalespace", w=1242, h=375, channels=3,
             scales=4, fp16=True),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case of the listed ones' ranges (odd sizes included), no dearer than they are."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["pair", "pair", "host", "two_way", "seeded", "batch", "serve",
                           "features", "knn", "knn_static", "scalespace"])
        w = _log_int(rng, 96, 1920)
        h = min(1080, max(64, int(w * rng.uniform(0.3, 0.8))))
        c = dict(kind=kind, w=w, h=h, channels=rng.choice([1, 3]), scales=rng.choice([3, 4]))
        if kind in ("pair", "host", "two_way", "seeded", "batch", "serve"):
            c.update(iters=rng.choice([4, 6]), radius=rng.choice([8, 12]), schedule="basic")
        if kind in ("pair", "seeded"):
            c["schedule"] = rng.choice(["basic", "plus", "fast"])
        if kind == "host":
            c["region_min"] = rng.choice([0, 150])
        if kind == "two_way":
            c.update(schedule=rng.choice(["basic", "fast_x2"]), stride=rng.choice([1, 2]),
                     region=rng.choice([50, 150]), cell=rng.choice([3, 4]), least=rng.choice([1, 2]))
        if kind == "batch":
            c.update(sizes="one", pairs=rng.randint(2, 20), slots=rng.choice([8, 16, 32]))
        if kind == "serve":
            c.update(requests=rng.randint(4, 20), slots=rng.choice([4, 8]))
        if kind == "features":
            c["tensor_cores"] = rng.choice([0, 1])
        if kind in ("knn", "knn_static"):
            c.update(leaf=rng.choice([4, 8]), stride=rng.choice([1, 2]))
        if kind == "scalespace":
            c["fp16"] = rng.choice([False, True])
        if work(c)["flops"] <= most and _points(c) <= 20e6:
            return c


# ----------------------------------------------------------------------------
# frames
# ----------------------------------------------------------------------------
def _noise(tables, period: float, x, y):
    """Value noise (smoothstep blend, octaves of half the period) at (x, y): [C, H, W]."""
    total, norm = 0.0, 0.0
    n = tables.shape[-1]
    for o in range(tables.shape[0]):
        gx, gy = x * (2.0 ** o / period), y * (2.0 ** o / period)
        x0, y0 = gx.floor(), gy.floor()
        fx, fy = gx - x0, gy - y0
        fx, fy = fx * fx * (3 - 2 * fx), fy * fy * (3 - 2 * fy)
        ix, iy = x0.long() % n, y0.long() % n
        jx, jy = (ix + 1) % n, (iy + 1) % n
        t = tables[o]
        v = ((t[:, iy, ix] * (1 - fx) + t[:, iy, jx] * fx) * (1 - fy)
             + (t[:, jy, ix] * (1 - fx) + t[:, jy, jx] * fx) * fy)
        total, norm = total + v * 0.6 ** o, norm + 0.6 ** o
    return total / norm


def _frames(seed: int, w: int, h: int, channels: int):
    """Two uint8 frames [C][H][W] on the GPU: 4 layers, displacements up to 0.15 of the width."""
    r = np.random.RandomState(seed % (1 << 32))
    y, x = torch.meshgrid(torch.arange(h, dtype=torch.float64, device="cuda"),
                          torch.arange(w, dtype=torch.float64, device="cuda"), indexing="ij")
    layers = []
    for k in range(4):
        tab = torch.from_numpy(r.rand(5, channels, 64, 64)).cuda()
        shape = torch.from_numpy(r.rand(3, 1, 64, 64)).cuda()
        flat = torch.from_numpy(r.rand(2, 1, 64, 64)).cuda()
        colour = torch.from_numpy(r.rand(channels)).cuda()
        a, s = math.radians(r.uniform(-10, 10)), r.uniform(0.9, 1.1)
        reach = 0.15 * w * (1.0 if k == 0 else r.uniform(0.4, 1.0))
        m = np.array([[s * math.cos(a) - 1, -s * math.sin(a)], [s * math.sin(a), s * math.cos(a) - 1]])
        t = r.uniform(-0.5, 0.5, 2) * reach
        # scaled so that the largest displacement at a frame corner is the layer's reach
        corners = np.array([[-w / 2, -h / 2], [w / 2, -h / 2], [-w / 2, h / 2], [w / 2, h / 2]])
        big = np.abs(corners @ m.T + t).max()
        m, t = m * min(1.0, reach / big), t * min(1.0, reach / big)
        layers.append((tab, shape, flat, colour, m + np.eye(2), t, r.uniform(24, 48)))
    out = []
    for second in (False, True):
        img = None
        for k, (tab, shape, flat, colour, m, t, period) in enumerate(layers):
            px, py = x - w / 2, y - h / 2
            if second:   # where this pixel of frame 2 comes from
                inv = np.linalg.inv(m)
                qx, qy = px - t[0], py - t[1]
                px, py = inv[0, 0] * qx + inv[0, 1] * qy, inv[1, 0] * qx + inv[1, 1] * qy
            px, py = px + 3000.0, py + 3000.0
            v = (0.5 + 2.0 * (_noise(tab, period, px, py) - 0.5)).clamp(0, 1)
            v = torch.where(_noise(flat, 40.0, px, py) > 0.68, colour[:, None, None], v)
            if img is None:
                img = v
            else:
                img = torch.where(_noise(shape, w / 3.0, px, py) > 0.62, v, img)
        if channels == 3:   # the spread of 8-bit CIELab
            img = torch.stack([img[0] * 255, 128 + (img[1] - 0.5) * 90, 128 + (img[2] - 0.5) * 90])
        else:
            img = img * 255
        out.append(img.round().clamp(0, 255).to(torch.uint8).contiguous())
    return out


def _pinned(t):
    return t.cpu().pin_memory()


def _config(case: dict, **more) -> ff.Config:
    return ff.Config(channels=case["channels"], scales=case["scales"], iters=case.get("iters", 4),
                     radius_q3=case.get("radius", 8), seed_leaf=case.get("leaf", 8),
                     seed_stride=case.get("stride", 1), max_width=case["w"], max_height=case["h"],
                     schedule=SCHEDULES[case.get("schedule", "basic")],
                     region_min=case.get("region_min", 0),
                     wht_tensor_cores=case.get("tensor_cores", 0), **more)


def _sizes(case: dict) -> list[tuple[int, int]]:
    """Frame sizes of a batch or of a burst of requests."""
    if case["kind"] == "batch":
        if case["sizes"] == "mixed":
            return [BATCH_SIZES[k % len(BATCH_SIZES)] for k in range(case["pairs"])]
        return [(case["w"], case["h"])] * case["pairs"]
    # requests: every one has its own size, spread over an eighth to all of the largest's width
    n = case["requests"]
    return [(max(64, int(case["w"] * (0.13 + 0.87 * ((7 * k) % n + 1) / n))),
             max(48, int(case["h"] * (0.2 + 0.8 * ((5 * k) % n + 1) / n)))) for k in range(n)]


class _Batch:
    """A batch object and its buffers, freed with the state."""

    def __init__(self, case: dict, seed: int):
        self.handle = ff.ff_batch_create(_config(case), 0, case["slots"],
                                         torch.cuda.current_stream())
        self.pairs = []
        for k, (w, h) in enumerate(_sizes(case)):
            i1, i2 = _frames(seed * 1000 + k, w, h, case["channels"])
            flow = lambda: torch.empty((h, w, 2), dtype=torch.int16, device="cuda")  # noqa: E731
            self.pairs.append(dict(img1=i1, img2=i2, w=w, h=h, pair_id=k, flow_fwd=flow(),
                                   flow_bwd=flow(),
                                   mask=torch.empty((h, w), dtype=torch.uint8, device="cuda")))
        self.descs = ff.pair_descs(self.pairs)

    def __del__(self):
        ff.ff_batch_destroy(self.handle)


class _Server:
    """A server, its requests' pinned frames and result buffers, freed with the state."""

    def __init__(self, case: dict, seed: int):
        cfg = _config(case)
        self.handle = ff.ff_server_create(cfg, 0, case["slots"] * ff.ff_slot_bytes(cfg),
                                          case["slots"])
        self.keep, self.requests, self.results = [], [], []
        for k, (w, h) in enumerate(_sizes(case)):
            i1, i2 = (_pinned(f) for f in _frames(seed * 1000 + k, w, h, case["channels"]))
            fwd = torch.empty((h, w, 2), dtype=torch.int16).pin_memory()
            mask = torch.empty((h, w), dtype=torch.uint8).pin_memory()
            self.keep.append((i1, i2))
            self.results.append((fwd, mask))
            self.requests.append(ff.host_pair(i1, i2, w, h, pair_id=k, flow_fwd=fwd, mask=mask))

    def __del__(self):
        ff.ff_server_destroy(self.handle)


# ----------------------------------------------------------------------------
# the contract: prepare, run, work, exact
# ----------------------------------------------------------------------------
def prepare(case: dict, seed: int):
    kind = case["kind"]
    st = {"kind": kind, "case": dict(case)}
    if kind == "batch":
        st["batch"] = _Batch(case, seed)
        return st
    if kind == "serve":
        st["server"] = _Server(case, seed)
        return st
    w, h, C = case["w"], case["h"], case["channels"]
    i1, i2 = _frames(seed, w, h, C)
    if kind == "scalespace":
        dims = [ff.level_dims(w, h, L) for L in range(case["scales"])]
        st.update(img=i1, out=[torch.empty((hl, wl, 9 * C), dtype=torch.float32, device="cuda")
                               for wl, hl in dims])
        return st
    if kind == "knn_static":
        # the level-0 features of both frames in the layout that the call takes: 16 or 32 bytes a pixel
        cfg = _config(case)
        ctx = ff.Context(cfg)
        P = 16 if C == 1 else 32
        st["feat"] = []
        for slot, img in enumerate((i1, i2)):
            ctx.features(slot, img)
            f = torch.zeros((h, w, P), dtype=torch.int8, device="cuda")
            f[..., :9 * C] = ctx.features_of(slot, 0)
            st["feat"].append(f)
        ctx.sync()
        ctx.close()
        wl, hl = ff.level_dims(w, h, case["scales"] - 1)
        st["idx"] = torch.empty((hl, wl, case["leaf"]), dtype=torch.int32, device="cuda")
        st["dist"] = torch.empty_like(st["idx"])
        return st
    ctx = ff.Context(_config(case))
    st.update(ctx=ctx, img1=i1, img2=i2)
    if kind == "host":
        st.update(img1=_pinned(i1), img2=_pinned(i2),
                  fwd=torch.empty((h, w, 2), dtype=torch.int16).pin_memory(),
                  bwd=torch.empty((h, w, 2), dtype=torch.int16).pin_memory(),
                  mask=torch.empty((h, w), dtype=torch.uint8).pin_memory())
    elif kind == "knn":
        ctx.features(0, i1)
        ctx.features(1, i2)
    elif kind == "seeded":
        # a coarse flow from elsewhere: smooth motion with some noise and some missing points
        r = np.random.RandomState(seed % (1 << 32))
        wl, hl = ff.level_dims(w, h, case["scales"] - 1)
        s = r.uniform(-0.05, 0.05, 2) * 8 * w + r.normal(0, 12, (hl, wl, 2))
        s = np.rint(s).astype(np.int16)
        s[r.rand(hl, wl) < 0.1] = ff.INVALID
        st["seeds"] = torch.from_numpy(s).cuda()
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        b = st["batch"]
        ff.ff_batch_run(b.handle, b.descs, len(b.pairs), use_graph=True)
        return [(p["flow_fwd"], p["flow_bwd"], p["mask"]) for p in b.pairs]
    if kind == "serve":
        v = st["server"]
        left = {ff.ff_server_submit(v.handle, q) for q in v.requests}
        while left:
            for ticket, status in ff.ff_server_poll(v.handle):
                if status != ff.FF_OK:
                    raise RuntimeError("a request failed")
                left.discard(ticket)
        return v.results
    case = st["case"]
    if kind == "scalespace":
        for L, out in enumerate(st["out"]):
            ff.ff_wht_coeffs_scalespace_tc(st["img"], case["w"], case["h"], case["w"],
                                           case["channels"], L, case["fp16"], out,
                                           torch.cuda.current_stream())
        return st["out"]
    if kind == "knn_static":
        ff.ff_seed_knn_static(st["feat"][0], st["feat"][1], case["w"], case["h"], case["channels"],
                              case["scales"], case["leaf"], case["stride"], st["idx"], st["dist"],
                              torch.cuda.current_stream())
        return st["idx"], st["dist"]
    ctx = st["ctx"]
    if kind == "knn":
        return ctx.seed_knn(ff.FF_FWD)
    if kind == "host":
        ff.ff_pair_host(ctx.ctx, st["img1"], st["img2"], case["w"], case["h"], 0, st["fwd"],
                        st["bwd"], st["mask"])
        return st["fwd"], st["bwd"], st["mask"]
    ctx.features(0, st["img1"])
    if kind == "features":
        return [ctx.features_of(0, L) for L in range(case["scales"])]
    ctx.features(1, st["img2"])
    if kind == "seeded":
        return ctx.match(ff.FF_FWD, 0, seeds_in=st["seeds"])
    fwd, cost = ctx.match(ff.FF_FWD, 0)
    bwd, _ = ctx.match(ff.FF_BWD, 0, with_cost=False)
    if kind == "two_way":
        bwd2, _ = ctx.match(ff.FF_BWD2, 0, with_cost=False)
        mask = ctx.filter_2way(fwd, bwd, bwd2)
        mask = ctx.region_filter(fwd, mask, case["region"])
        return fwd, cost, bwd, bwd2, mask, ctx.sparsify(fwd, bwd, bwd2, mask, case["cell"],
                                                        case["least"])
    return fwd, cost, bwd, ctx.filter(fwd, bwd)


def _points(case: dict) -> float:
    """Pixels of all frames of a case."""
    if case["kind"] in ("batch", "serve"):
        return float(sum(w * h for w, h in _sizes(case)))
    return float(case["w"] * case["h"])


def _seed_flops(case: dict, w: int, h: int) -> float:
    """The exact search's products: every coarsest-grid point against every candidate."""
    wl, hl = ff.level_dims(w, h, case["scales"] - 1)
    s = case.get("stride", 1)
    return 2.0 * 9 * case["channels"] * wl * hl * -(-w // s) * -(-h // s)


def _match_flops(case: dict, w: int, h: int) -> float:
    """Matching errors of one flow: two propagation candidates a point and sweep, one random one
    a point and search, one a carried point."""
    cfg = _config(case)
    n = 0
    for L in range(cfg.final_level(), case["scales"]):
        wl, hl = ff.level_dims(w, h, L)
        n += wl * hl * (2 * cfg.sweeps(L) + cfg.random_searches(L) + 0.25)
    return n * 9.0 * case["channels"] * OPS_PER_DIM


def _pair_work(case: dict, w: int, h: int, flows: int, seeded: bool = False) -> tuple[float, float]:
    C = case["channels"]
    wf, hf = ff.level_dims(w, h, _config(case).final_level())
    flops = flows * (_match_flops(case, w, h) + (0 if seeded else _seed_flops(case, w, h)))
    return 2.0 * C * w * h + flows * 4.0 * wf * hf, flops


def work(case: dict) -> dict:
    kind, w, h, C = case["kind"], case["w"], case["h"], case["channels"]
    levels = [ff.level_dims(w, h, L) for L in range(case["scales"])]
    points = sum(a * b for a, b in levels)
    wht = points * C * 2.0 * (8 * 8 * 3 + 8 * 3 * 3) / 8   # separable +-1 sums of the 8x8 windows
    if kind in ("batch", "serve"):
        each = [_pair_work(case, a, b, 2) for a, b in _sizes(case)]
        kept = sum(a * b for a, b in _sizes(case))
        return {"bytes": sum(e[0] for e in each) + kept, "flops": sum(e[1] for e in each)}
    if kind == "features":
        return {"bytes": float(C * w * h + 9 * C * points), "flops": wht}
    if kind == "scalespace":
        return {"bytes": float(case["scales"] * C * w * h + 36 * C * points),
                "flops": points * C * 2.0 * 64 * 9}
    if kind in ("knn", "knn_static"):
        s = case["stride"]
        cand = -(-w // s) * -(-h // s)
        nq = levels[-1][0] * levels[-1][1]
        return {"bytes": float(9 * C * (cand + nq) + 8 * case["leaf"] * nq),
                "flops": _seed_flops(case, w, h)}
    flows = {"pair": 2, "host": 2, "two_way": 3, "seeded": 1}[kind]
    nbytes, flops = _pair_work(case, w, h, flows, kind == "seeded")
    wf, hf = ff.level_dims(w, h, _config(case).final_level())
    nbytes += wf * hf * {"pair": 5, "host": 1, "two_way": 6, "seeded": 4}[kind]   # cost, masks
    return {"bytes": nbytes, "flops": flops + 2 * wht}


def exact(case: dict, seed: int):
    """The Walsh transform of the scale space in 64 bits, rounded nowhere for the tensor-core
    form, to the int8 codes for the features.  The searches and matches are whole numbers
    throughout, and the sweeps' order is serial: no 64-bit form of them is quicker."""
    kind = case["kind"]
    if kind not in ("features", "scalespace"):
        return None
    C, w, h = case["channels"], case["w"], case["h"]
    img = _frames(seed, w, h, C)[0].double()
    walsh = torch.ones(3, 8, dtype=torch.float64, device="cuda")
    walsh[1, 4:] = -1
    walsh[2, 2:6] = -1
    out = []
    for L in range(case["scales"]):
        n = 1 << L
        wl, hl = ff.level_dims(w, h, L)
        full = torch.nn.functional.pad(img[None], (0, wl * n - w, 0, hl * n - h),
                                       mode="replicate")[0]
        mean = full.reshape(C, hl, n, wl, n).mean(dim=(2, 4))
        if kind == "features":
            mean = (mean + 0.5).floor()
        pad = torch.nn.functional.pad(mean[None], (3, 4, 3, 4), mode="replicate")[0]
        win = pad.unfold(1, 8, 1).unfold(2, 8, 1)          # [C, hl, wl, 8 rows, 8 columns]
        co = torch.einsum("chwij,ui,vj->hwcuv", win, walsh, walsh).reshape(hl, wl, C, 9)
        if kind == "features":
            dc = ((co[..., :1] + 32) / 64).floor() - 128
            co = torch.cat([dc, ((co[..., 1:] + 8) / 16).floor()], dim=-1).clamp(-128, 127)
            co = co.to(torch.int8)
        out.append(co.reshape(hl, wl, 9 * C).contiguous())
    return out
