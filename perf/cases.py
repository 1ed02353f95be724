"""Cases that stand for the use of this library: what a program that segments
uint16 confocal volumes has it do, through the binding's public calls.

A "segment" case submits its frames as requests of one batch, waits, reads the
results back and releases them.  Channel 0 of a frame is the stem-cell channel
(nuclei on noise), channel 1 the vessel channel (tubes on noise); the front
end (`denoise`) runs on stem-cell channels, the MRF denoise (`mrf`) and the
distance map on vessel channels, the closing on every channel, as the paper
uses them.  A "register" case registers montage tiles; an "otsu" case takes
the Otsu level of one volume on a caller's stream.

Inputs are drawn on the GPU: noise N(200, 25), ellipsoidal nuclei of radius
4..9 with soft edges, vessels of radius 3..6 around curved centrelines, both
1200..1800 above the noise (one brightness per volume).
"""
import functools
import math

import numpy as np
import torch

import paper_1407_2089_gb300 as seg

DEVICE = "cuda:0"
WEIGHTS = (16, 16, 25)  # squared spacing 0.8 x 0.8 x 1.0 um in units of 0.2 um


def _segment(name, x, y, z, **more):
    case = {"kind": "segment", "x": x, "y": y, "z": z, "frames": 1, "channels": 1, "content": "nuclei",
            "host": False, "labels": "runs", "denoise": 0, "closing": 0, "mrf": 0, "distance": False,
            "min_volume": 30}
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # one small frame on the GPU, labels kept there: the smallest call, all latency
        _segment("single_frame", 128, 128, 32, labels="dense"),
        # one two-channel frame as it leaves the microscope: pinned host memory in, label runs and cells
        # in host memory out
        _segment("live_frame", 512, 512, 64, channels=2, host=True),
        # a stretch of a time-lapse resident on the GPU, every volume in one batch
        _segment("time_lapse", 512, 512, 64, frames=16, channels=2),
        # volumes of mixed sizes (64 to 1024 across, odd and even widths, 64 to 96 planes) in one batch
        {"name": "uneven_batch", "kind": "uneven", "volumes": 12, "dims_seed": 3, "lo": 64, "hi": 1024,
         "min_volume": 30},
        # one channel of the stitched montage, segmented whole: the largest call
        _segment("stitched_montage", 5530, 5530, 80, labels="dense"),
        # the stem-cell channel's denoise front end; the denoised images are read back too
        _segment("stem_denoise", 512, 512, 64, frames=4, denoise=8),
        # the vessel channel's MRF denoise, 20 steps
        _segment("vessel_mrf", 512, 512, 64, frames=4, content="vessels", mrf=20),
        # the vessel channel's distance map
        _segment("vessel_distance", 512, 512, 64, frames=4, content="vessels", distance=True),
        # 25-plane confocal frames, both channels, foreground closed with a small ball
        _segment("closed_frames", 512, 512, 25, frames=8, channels=2, closing=1),
        # one frame through every step the paper runs on its two channels, with each cell's distance to the
        # nearest vessel
        _segment("full_frame", 512, 512, 64, channels=2, labels="dense", denoise=8, closing=1, mrf=20,
                 distance=True),
        # montage registration, 3 x 3 tiles with a tenth of overlap
        {"name": "registration", "kind": "register", "nx": 3, "ny": 3, "x": 1024, "y": 1024, "z": 64,
         "overlap": 0.1, "rx": 4, "ry": 4, "rz": 1},
        # the allocation-free Otsu level of one resident volume (odd width)
        {"name": "otsu_level", "kind": "otsu", "x": 701, "y": 512, "z": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "live", "series", "uneven", "stitched", "denoise", "mrf", "distance", "closing",
                       "full", "register", "otsu"])
    mv = rng.choice([1, 10, 30, 30, 100])
    x, y, z = _log(rng, 64, 768), _log(rng, 64, 768), rng.randint(12, 80)
    if kind == "frame":
        return _segment(None, _log(rng, 24, 400), _log(rng, 24, 400), rng.randint(8, 48), labels="dense",
                        min_volume=mv)
    if kind == "live":
        return _segment(None, x, y, z, channels=rng.choice([1, 2]), host=True, min_volume=mv)
    if kind == "series":
        return _segment(None, x, y, z, frames=rng.randint(2, 12), channels=rng.choice([1, 2]), min_volume=mv)
    if kind == "uneven":
        return {"kind": "uneven", "volumes": rng.randint(3, 16), "dims_seed": rng.randint(0, 1 << 20),
                "lo": 48, "hi": 900, "min_volume": mv}
    if kind == "stitched":
        return _segment(None, _log(rng, 1200, 3500), _log(rng, 1200, 3500), rng.randint(24, 80), labels="dense",
                        min_volume=mv)
    if kind == "denoise":
        return _segment(None, x, y, z, frames=rng.randint(1, 5), denoise=rng.randint(3, 12), min_volume=mv)
    if kind == "mrf":
        return _segment(None, x, y, z, frames=rng.randint(1, 4), content="vessels", mrf=rng.randint(5, 30),
                        min_volume=mv)
    if kind == "distance":
        return _segment(None, x, y, z, frames=rng.randint(1, 5), content="vessels", distance=True, min_volume=mv)
    if kind == "closing":
        return _segment(None, x, y, z, frames=rng.randint(1, 8), channels=rng.choice([1, 2]),
                        closing=rng.randint(1, 4), min_volume=mv)
    if kind == "full":
        return _segment(None, x, y, z, channels=2, labels="dense", denoise=rng.randint(3, 10),
                        closing=rng.randint(0, 3), mrf=rng.randint(5, 25), distance=True, min_volume=mv)
    if kind == "register":
        return {"kind": "register", "nx": rng.randint(1, 3), "ny": rng.randint(2, 3), "x": _log(rng, 160, 900),
                "y": _log(rng, 160, 900), "z": rng.randint(16, 64), "overlap": rng.uniform(0.08, 0.2),
                "rx": rng.randint(1, 6), "ry": rng.randint(1, 6), "rz": rng.randint(0, 2)}
    return {"kind": "otsu", "x": x, "y": y, "z": z}


# ---- inputs ----------------------------------------------------------------

def _brightness(g):
    return 1200.0 + 600.0 * torch.rand(1, generator=g, device=DEVICE)


def _add_nuclei(vol, g, count):
    Z, Y, X = vol.shape
    half = 0.5 * _brightness(g)
    step = 22  # 2 * 9 + a gap: nuclei on a jittered grid never merge by chance alone
    n = [max(1, d // step) for d in (X, Y, Z)]
    total = n[0] * n[1] * n[2]
    count = min(count, total)
    cell = torch.randperm(total, generator=g, device=DEVICE)[:count]
    idx = torch.stack([cell % n[0], (cell // n[0]) % n[1], cell // (n[0] * n[1])], 1).float()
    size = torch.tensor([X, Y, Z], device=DEVICE, dtype=torch.float32)
    pitch = size / torch.tensor(n, device=DEVICE, dtype=torch.float32)
    c = (idx + 0.3 + 0.4 * torch.rand(count, 3, generator=g, device=DEVICE)) * pitch
    r = 4.0 + 5.0 * torch.rand(count, 3, generator=g, device=DEVICE)
    o = torch.arange(-12, 13, device=DEVICE)
    off = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    flat = vol.view(-1)
    for i in range(0, count, 1024):
        ci, ri = c[i:i + 1024], r[i:i + 1024]
        p = ci.round().long()[:, None, :] + off
        d = ((p.float() - ci[:, None, :]) / ri[:, None, :]).norm(dim=2)
        v = (half * torch.erfc((d - 1.0) * ri.mean(1, keepdim=True) / 2.12)).round().int()
        ok = (p >= 0).all(2) & (p < size.long()).all(2) & (v > 0)
        p, v = p[ok], v[ok]
        flat.index_add_(0, (p[:, 2] * Y + p[:, 1]) * X + p[:, 0], v)


def _add_vessels(vol, g, count):
    Z, Y, X = vol.shape
    half = 0.5 * _brightness(g)
    size = torch.tensor([X - 1, Y - 1, Z - 1], device=DEVICE, dtype=torch.float32)
    o = torch.arange(-9, 10, device=DEVICE)
    off = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    field = torch.zeros_like(vol).view(-1)
    for k in range(count):
        p = torch.rand(5, 3, generator=g, device=DEVICE) * size
        a = k % 2
        p[0, a], p[4, a] = 0.0, size[a]
        p = torch.cat([2 * p[:1] - p[1:2], p, 2 * p[4:] - p[3:4]])
        radius = 3.0 + 3.0 * torch.rand(1, generator=g, device=DEVICE)
        t = torch.linspace(0, 1, max(2, int(max(X, Y))), device=DEVICE)[:, None]
        for i in range(1, 5):
            q = 0.5 * (2 * p[i] + (p[i + 1] - p[i - 1]) * t
                       + (2 * p[i - 1] - 5 * p[i] + 4 * p[i + 1] - p[i + 2]) * t * t
                       + (3 * p[i] - p[i - 1] - 3 * p[i + 1] + p[i + 2]) * t * t * t)
            w = q.round().long()[:, None, :] + off
            d = (w.float() - q[:, None, :]).norm(dim=2)
            v = (half * torch.erfc((d - radius) / 1.41)).round().int()
            ok = (w >= 0).all(2) & (w <= size.long()).all(2) & (v > 0)
            w, v = w[ok], v[ok]
            field.scatter_reduce_(0, (w[:, 2] * Y + w[:, 1]) * X + w[:, 0], v, "amax")
    vol += field.view(Z, Y, X)


def _noisy(vol, seed, mean):
    """vol + N(mean, 25) rounded, as int16 (uint16 bits)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    out = torch.empty(vol.shape, dtype=torch.int16, device=DEVICE)
    for k in range(vol.shape[0]):
        noise = mean + 25.0 * torch.randn(vol.shape[1:], generator=g, device=DEVICE)
        out[k] = (vol[k] + noise.round().int()).clamp_(0, 32767).to(torch.int16)
    return out


def _volume(x, y, z, seed, content):
    """int16 (uint16 bits) [z][y][x] on the GPU."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    vol = torch.zeros(z, y, x, dtype=torch.int32, device=DEVICE)
    if content == "vessels":
        _add_vessels(vol, g, max(2, round(8 * x * y / (512 * 512))))
    else:
        _add_nuclei(vol, g, max(1, round(x * y * z / 40 ** 3)))
    return _noisy(vol, seed + 7, 200.0)


def _contents(case):
    return ["nuclei", "vessels"] if case["channels"] == 2 else [case["content"]]


def _uneven_dims(case):
    rng = np.random.default_rng(case["dims_seed"])
    dims = []
    for _ in range(case["volumes"]):
        a = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        dims.append((a, a, int(rng.integers(64, 97))))
    dims[0] = (case["lo"], case["lo"], 64)
    dims[-1] = (case["hi"], case["hi"], 96)
    return dims


@functools.lru_cache(maxsize=None)
def _context(window_us):
    """The handle that a program creates once and keeps."""
    stream = torch.cuda.Stream(DEVICE)
    return seg.seg_create(device=0, batch_window_us=window_us, order_stream=stream.cuda_stream), stream


def _layout(case, seed=0):
    """Tile positions of a montage in its own frame, as placed by the stage and as they are."""
    rng = np.random.default_rng(seed)
    r = [case["rx"], case["ry"], case["rz"]]
    step = [case["x"] - round(case["x"] * case["overlap"]), case["y"] - round(case["y"] * case["overlap"])]
    stage, true = [], []
    for j in range(case["ny"]):
        for i in range(case["nx"]):
            s = np.array([i * step[0] + r[0], j * step[1] + r[1], r[2]])
            stage.append(s)
            true.append(s + np.array([rng.integers(-(q // 2), q // 2 + 1) for q in r]))
    return np.array(stage), np.array(true)


def prepare(case, seed):
    kind = case["kind"]
    base = (seed * 1000003 + 17) % (1 << 40)
    if kind == "register":
        stage, true = _layout(case, base)
        d = np.array([case["x"], case["y"], case["z"]])
        ext = true.max(axis=0) + d
        whole = _volume(int(ext[0]), int(ext[1]), int(ext[2]), base, "nuclei")
        # each tile is taken on its own, with its own shot noise
        tiles = [_noisy(whole[t[2]:t[2] + d[2], t[1]:t[1] + d[1], t[0]:t[0] + d[0]], base + 1 + i, 0.0)
                 for i, t in enumerate(true)]
        return {"case": case, "tiles": tiles, "stage": stage}
    if kind == "otsu":
        return {"case": case, "volume": _volume(case["x"], case["y"], case["z"], base, "nuclei"),
                "result": torch.zeros(2, dtype=torch.int32, device=DEVICE)}
    if kind == "uneven":
        dims = _uneven_dims(case)
        frames = [_volume(*d, base + 101 * i, "nuclei")[None] for i, d in enumerate(dims)]
        case = dict(case, channels=1, content="nuclei", host=False, labels="dense", denoise=0, closing=0, mrf=0,
                    distance=False)
    else:
        frames = [torch.stack([_volume(case["x"], case["y"], case["z"], base + 101 * i + c, content)
                               for c, content in enumerate(_contents(case))]) for i in range(case["frames"])]
    where = {"device": "cpu", "pin_memory": True} if case["host"] else {"device": DEVICE}
    if case["host"]:
        frames = [f.cpu().pin_memory() for f in frames]
    vessel = [c == "vessels" for c in _contents(case)]
    state = {"case": case, "frames": frames, "vessel": vessel, "out": []}
    for f in frames:
        channels = []
        for v in vessel:
            # the cell table and the runs have room to spare; what a pass leaves unwritten stays zero
            b = {"cells": np.zeros((256 + 4 * (f[0].numel() // 40 ** 3), 64), dtype=np.uint8)}
            if case["labels"] == "dense":
                b["labels"] = torch.empty(f.shape[1:], dtype=torch.int32, **where)
            else:  # a dozen runs a row, twelve bytes each
                b["runs"] = torch.zeros(144 * max(f.shape[1] * f.shape[2], 64), dtype=torch.uint8, **where)
            if case["mrf"] and v or case["denoise"] and not v:
                b["denoised"] = torch.empty(f.shape[1:], dtype=torch.int16, **where)
            if case["distance"] and v:
                b["distance"] = torch.empty(f.shape[1:], dtype=torch.int32, **where)
            if case["distance"] and v and len(vessel) == 2:
                b["nearest"] = np.zeros(len(b["cells"]), dtype=np.uint32)
            channels.append(b)
        state["out"].append(channels)
    state["ctx"], state["stream"] = _context(0 if len(frames) == 1 else 2_000_000)
    torch.cuda.synchronize()
    return state


# ---- one pass --------------------------------------------------------------

def _table(b, cells):
    b["cells"][:len(cells)] = cells.view(np.uint8).reshape(-1, 64)
    return b["cells"]


def run(state):
    case = state["case"]
    if case["kind"] == "register":
        delta, edges = seg.seg_register_montage(state["tiles"], state["stage"], (case["rx"], case["ry"], case["rz"]))
        return {"delta": delta, "a": edges["a"], "b": edges["b"], "shift": edges["shift"], "score": edges["score"],
                "in_tree": edges["in_tree"]}
    if case["kind"] == "otsu":
        seg.seg_otsu_threshold_noalloc(state["volume"].data_ptr(), (case["x"], case["y"], case["z"]),
                                       state["result"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["result"]
    ctx, vessel = state["ctx"], state["vessel"]
    if case["labels"] == "dense" and not (case["denoise"] or case["mrf"] or case["distance"]) and \
            len(state["frames"]) == 1:
        # one frame at a time: the convenience call
        labels = [b["labels"] for b in state["out"][0]]
        got = seg.segment(ctx, state["frames"][0], min_volume=case["min_volume"], labels_out=labels,
                          closing_radius=case["closing"])
        return [{"labels": lab, "cells": _table(b, cells), "threshold": t}
                for b, (lab, cells, t) in zip(state["out"][0], got)]
    options = dict(
        min_volume=case["min_volume"], closing_radius=case["closing"], keep_host_input=case["host"],
        denoise_radius=[0 if v else case["denoise"] for v in vessel],
        mrf_iterations=[case["mrf"] if v else 0 for v in vessel],
        distance_weights=[WEIGHTS if v and case["distance"] else None for v in vessel])
    reqs = [seg.seg_submit_volume(ctx, f, **options) for f in state["frames"]]
    seg.seg_flush(ctx)
    cells, levels, steps, images = [], [], [], []
    for req, channels in zip(reqs, state["out"]):
        if seg.seg_wait(ctx, req) != seg.SEG_DONE:
            raise RuntimeError("request failed")
        for c, b in enumerate(channels):
            table, level = seg.seg_read_features(ctx, req, c)
            cells.append(_table(b, table))
            levels.append(level)
            if "labels" in b:
                images.append(seg.seg_read_labels(ctx, req, c, b["labels"]))
            else:
                seg.seg_read_label_runs(ctx, req, c, b["runs"])
                images.append(b["runs"])
            if "denoised" in b:
                steps.append(seg.seg_read_denoised(ctx, req, c, b["denoised"]))
                images.append(b["denoised"])
            if "distance" in b:
                images.append(seg.seg_read_distance(ctx, req, c, b["distance"]))
                if "nearest" in b:
                    nearest = seg.seg_read_cell_distance(ctx, req, 0, c)
                    b["nearest"][:len(nearest)] = nearest
                    images.append(b["nearest"])
        seg.seg_release(ctx, req)
    return {"cells": cells[0] if len(cells) == 1 else np.concatenate(cells), "levels": np.array(levels), "steps": np.array(steps, dtype=np.int64),
            "images": images}


# ---- what a pass cannot do without ------------------------------------------

def _overlap(d, n):
    return max(0, min(n, d + n) - max(0, d))


def work(case):
    kind = case["kind"]
    if kind == "register":
        # the products of the covariance at every shift of every overlapping pair
        stage, _ = _layout(case)
        dims, r = (case["x"], case["y"], case["z"]), (case["rx"], case["ry"], case["rz"])
        products, voxels = 0, 0
        for a in range(len(stage)):
            for b in range(a + 1, len(stage)):
                d = stage[b] - stage[a]
                if all(abs(int(d[k])) < dims[k] for k in range(3)):
                    per = [sum(_overlap(int(d[k]) + s, dims[k]) for s in range(-r[k], r[k] + 1)) for k in range(3)]
                    products += per[0] * per[1] * per[2]
                    voxels += 2 * _overlap(int(d[0]), dims[0]) * _overlap(int(d[1]), dims[1]) * \
                        _overlap(int(d[2]), dims[2])
        return {"bytes": 2.0 * voxels, "flops": 2.0 * products}
    smooth = 30.0  # three axes of five taps, per voxel
    if kind == "otsu":
        n = case["x"] * case["y"] * case["z"]
        return {"bytes": 2.0 * n, "flops": smooth * n}
    if kind == "uneven":
        n = sum(x * y * z for x, y, z in _uneven_dims(case))
        return {"bytes": 6.0 * n, "flops": smooth * n}
    n = case["x"] * case["y"] * case["z"] * case["frames"]
    total = {"bytes": 0.0, "flops": 0.0}
    for content in _contents(case):
        total["bytes"] += (6.0 if case["labels"] == "dense" else 2.0) * n
        total["flops"] += smooth * n
        if content == "nuclei" and case["denoise"]:
            # nine running sums (an addition, a subtraction and a scaling each), the difference and the median
            total["bytes"] += 2.0 * n
            total["flops"] += (9 * 3 + 1 + 54) * n
        if content == "vessels" and case["mrf"]:
            total["bytes"] += 2.0 * n
            total["flops"] += case["mrf"] * 15.0 * n
        if content == "vessels" and case["distance"]:
            total["bytes"] += 4.0 * n
            total["flops"] += 12.0 * n
    return total


# ---- the floating results in 64 bits ----------------------------------------

def exact(case, seed):
    """Only registration has floating results: every pair's best score."""
    if case["kind"] != "register":
        return None
    state = prepare(case, seed)
    stage, tiles = state["stage"], [t.to(torch.int64) for t in state["tiles"]]
    dims, r = (case["x"], case["y"], case["z"]), (case["rx"], case["ry"], case["rz"])
    scores = []
    for a in range(len(stage)):
        for b in range(a + 1, len(stage)):
            d0 = [int(v) for v in stage[b] - stage[a]]
            if not all(abs(d0[k]) < dims[k] for k in range(3)):
                continue
            best = -2.0
            for sz in range(-r[2], r[2] + 1):
                for sy in range(-r[1], r[1] + 1):
                    for sx in range(-r[0], r[0] + 1):
                        d = [d0[0] + sx, d0[1] + sy, d0[2] + sz]
                        if not all(_overlap(d[k], dims[k]) for k in range(3)):
                            continue
                        ia = tuple(slice(max(0, d[k]), min(dims[k], d[k] + dims[k])) for k in (2, 1, 0))
                        ib = tuple(slice(max(0, -d[k]), min(dims[k], dims[k] - d[k])) for k in (2, 1, 0))
                        p, q = tiles[a][ia], tiles[b][ib]
                        n = p.numel()
                        sa, sb, saa, sbb, sab = (int(v) for v in torch.stack(
                            [p.sum(), q.sum(), (p * p).sum(), (q * q).sum(), (p * q).sum()]).tolist())
                        va, vb = n * saa - sa * sa, n * sbb - sb * sb
                        if va and vb:
                            best = max(best, (n * sab - sa * sb) / math.sqrt(va * vb))
            scores.append(best)
    return {"delta": None, "a": None, "b": None, "shift": None,
            "score": torch.tensor(scores, dtype=torch.float64), "in_tree": None}
