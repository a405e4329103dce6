"""The work that is timed: passes through the public entry points over the range of real use.

A case names a ``kind`` of call and its sizes:

* ``stream``   ``Detector.detect`` on the frames of a small ring of buffers, one call per frame
  (a camera or video loop: each call gets the next buffer and waits for its keypoints);
* ``batch``    ``Detector.detect_batch`` on many frames, equal or of mixed sizes, with the default
  launch configuration or after ``Detector.autotune``;
* ``level``    ``of_detect_level_noalloc``, one level, asynchronous;
* ``learned``  ``of_detect_learned`` with the committed tile-proposal network;
* ``logits``   ``TileNet.logits`` on dense patches (labelling, threshold choice);
* ``train``    one training step of the network: loss and gradient, Adam, from the committed checkpoint;
* ``serve``    a burst of host frames through the serving loop: submit all, poll until all are back.

Frames are scenes of rectangles and checkerboards, blurred, with noise (and a 1/f background where
``pink``), rendered on the GPU from the seed; batches take each scene in up to eight variants (flips,
inversion).  Keypoint records are returned as bytes, so they are compared exactly.
"""

import json
import math

import numpy as np
import torch

import paper_2506_07164_gb300 as ofg
from paper_2506_07164_gb300 import learned

RECORD = 64  # bytes of one keypoint record
MIXED = ((720, 540), (1080, 720), (1440, 1080), (1920, 1080))  # frame sizes of a mixed batch
SERVED = ((640, 480), (1280, 720), (1920, 1080), (3840, 2160))  # frame sizes of the serving mix
TILE_MACS = 32 * 32 * 8 * 9 + 16 * 16 * 16 * 72 + 8 * 8 * 16 * 144 + 16


def listed():
    return [
        # The smallest call: one VGA frame, one level, no fallback (a tracker on a small camera).
        dict(name="stream_vga_1level", kind="stream", w=640, h=480, ring=2, levels=1, scale=1.2, t=20, t_lo=0,
             features=500, pink=False, aligned=True),
        # The ordinary call: a 1080p frame through the 8-level front end, one frame at a time.
        dict(name="stream_1080p", kind="stream", w=1920, h=1080, ring=2, levels=8, scale=1.2, t=20, t_lo=7,
             features=1000, pink=True, aligned=True),
        # A crop of a larger frame: odd size, rows at an odd pitch and offset, coarser pyramid.
        dict(name="stream_ragged", kind="stream", w=1283, h=717, ring=2, levels=4, scale=1.5, t=15, t_lo=5,
             features=1500, pink=True, aligned=False),
        # The largest single frame: 4K with many features.
        dict(name="stream_4k", kind="stream", w=3840, h=2160, ring=1, levels=8, scale=1.2, t=20, t_lo=7,
             features=2000, pink=True, aligned=True),
        # Two cameras' frames per call (a stereo pair), default configuration.
        dict(name="batch_stereo_720p", kind="batch", w=1280, h=720, frames=2, mixed=False, levels=8, scale=1.2, t=20,
             t_lo=7, features=1000, pink=True, aligned=True, tuned=False),
        # Frames of four sizes in one call, default configuration.
        dict(name="batch_mixed_64", kind="batch", w=1920, h=1080, frames=64, mixed=True, levels=8, scale=1.2, t=20,
             t_lo=7, features=1000, pink=True, aligned=True, tuned=False),
        # Offline throughput: 128 frames of 1080p, launch configuration tuned for the shape beforehand.
        dict(name="batch_1080p_128", kind="batch", w=1920, h=1080, frames=128, mixed=False, levels=8, scale=1.2, t=20,
             t_lo=7, features=1000, pink=True, aligned=True, tuned=True),
        # A caller that cannot allocate: one level of a 720p frame, queued on its stream.
        dict(name="level_720p", kind="level", w=1280, h=720, t=20, t_lo=7, features=1000, pink=True),
        # The learned front end on a batch of frames, committed network and threshold.
        dict(name="learned_1080p_16", kind="learned", w=1920, h=1080, frames=16, levels=8, scale=1.2, t=20, t_lo=7,
             features=1000),
        # Logits of many patches (choosing the threshold over a training set).
        dict(name="logits_16384", kind="logits", n=16384),
        # One training step at the trainer's batch size.
        dict(name="train_2048", kind="train", n=2048),
        # A burst of mixed frames at the server.
        dict(name="serve_24", kind="serve", frames=24, features=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream", "stream", "stream", "batch", "batch", "batch", "level", "learned", "logits", "train",
                       "serve"])
    opts = dict(levels=rng.choice([1, 2, 4, 6, 8, 8, 8]), scale=rng.choice([1.2, 1.2, 1.25, 1.5, 2.0]),
                t=rng.choice([10, 15, 20, 20, 30, 40]), t_lo=rng.choice([0, 5, 7, 7]), features=_log(rng, 100, 4000),
                pink=rng.random() < 0.7, aligned=rng.random() < 0.7)
    if kind == "stream":
        w = _log(rng, 320, 3840)
        return dict(kind=kind, w=w, h=int(w * rng.uniform(0.4, 0.8)), ring=rng.choice([1, 2, 3]), **opts)
    if kind == "batch":
        w = _log(rng, 320, 1920)
        return dict(kind=kind, w=w, h=int(w * rng.uniform(0.4, 0.8)), frames=_log(rng, 2, 96),
                    mixed=rng.random() < 0.5, tuned=False, **opts)
    if kind == "level":
        w = _log(rng, 320, 1900)
        return dict(kind=kind, w=w, h=int(w * rng.uniform(0.4, 0.56)), t=opts["t"], t_lo=opts["t_lo"],
                    features=opts["features"], pink=opts["pink"])
    if kind == "learned":
        w = _log(rng, 480, 1920)
        return dict(kind=kind, w=w, h=int(w * rng.uniform(0.45, 0.75)), frames=rng.randint(1, 12), levels=8, scale=1.2,
                    t=20, t_lo=7, features=_log(rng, 300, 2000))
    if kind == "logits":
        return dict(kind=kind, n=_log(rng, 64, 16384))
    if kind == "train":
        return dict(kind=kind, n=_log(rng, 64, 4096))
    return dict(kind=kind, frames=rng.randint(2, 32), features=_log(rng, 300, 2000))


# ------------------------------------------------------------------ inputs
def _scene(w, h, seed, pink):
    """One frame on the GPU: 200 rectangles (every other one rotated), 30 checkerboards, blur, noise."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    img = torch.full((h, w), 128.0, device="cuda")
    if pink:
        acc = torch.zeros((1, 1, h, w), device="cuda")
        for o in range(6):
            gw = 4 * 2**o + 2
            gh = max(2, round(gw * h / w) + 2)
            grid = torch.rand((1, 1, gh, gw), device="cuda", generator=gen) * 2 - 1
            acc += 0.5**o * torch.nn.functional.interpolate(grid, size=(h, w), mode="bilinear", align_corners=True)
        img += 40.0 * acc[0, 0] / acc.abs().max()
    yy = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] + 0.5
    xx = torch.arange(w, device="cuda", dtype=torch.float32)[None, :] + 0.5
    for i in range(200):
        cx, cy = rng.uniform(0, w), rng.uniform(0, h)
        sx, sy = rng.uniform(0.015, 0.2, size=2) * w
        ang = rng.uniform(0.0, np.pi) if i % 2 else 0.0
        val = rng.uniform(0.0, 255.0)
        ca, sa = math.cos(ang), math.sin(ang)
        ex, ey = 0.5 * (abs(sx * ca) + abs(sy * sa)), 0.5 * (abs(sx * sa) + abs(sy * ca))
        x0, x1 = max(0, int(cx - ex)), min(w, int(cx + ex) + 1)
        y0, y1 = max(0, int(cy - ey)), min(h, int(cy + ey) + 1)
        if x0 >= x1 or y0 >= y1:
            continue
        part = img[y0:y1, x0:x1]
        if ang == 0.0:
            part.fill_(val)
        else:
            dx, dy = xx[:, x0:x1] - cx, yy[y0:y1] - cy
            inside = ((dx * ca + dy * sa).abs() <= 0.5 * sx) & ((dy * ca - dx * sa).abs() <= 0.5 * sy)
            part.masked_fill_(inside, val)
    for _ in range(30):
        side = int(round(rng.uniform(0.04, 0.15) * w))
        sq = int(rng.integers(4, 13))
        a, b = rng.uniform(0.0, 255.0, size=2)
        px, py = int(rng.integers(0, max(1, w - side))), int(rng.integers(0, max(1, h - side)))
        x1, y1 = min(w, px + side), min(h, py + side)
        if x1 > px and y1 > py:
            odd = (((yy[: y1 - py] - 0.5) // sq) + ((xx[:, : x1 - px] - 0.5) // sq)) % 2
            img[py:y1, px:x1] = a + (b - a) * odd
    k = torch.exp(-0.5 * torch.arange(-3, 4, device="cuda", dtype=torch.float32) ** 2)
    k = k / k.sum()
    p = torch.nn.functional.pad(img[None, None], (3, 3, 3, 3), mode="replicate")
    p = sum(k[i] * p[:, :, :, i : i + w] for i in range(7))
    img = sum(k[i] * p[:, :, i : i + h] for i in range(7))[0, 0]
    img = img + 3.0 * torch.randn((h, w), device="cuda", generator=gen)
    return img.round().clamp(0, 255).to(torch.uint8)


def _placed(img, aligned):
    """The frame in a buffer of its own: rows at a multiple of 16 bytes, or a view one byte in at an odd pitch."""
    h, w = img.shape
    pitch = (w + 15) // 16 * 16 if aligned else (w + 2) | 1
    buf = torch.zeros((h, pitch), dtype=torch.uint8, device="cuda")
    view = buf[:, :w] if aligned else buf[:, 1 : w + 1]
    view.copy_(img)
    return view


def _sizes(case):
    if case.get("mixed"):
        s = case["w"] / 1920.0
        return [(max(96, int(MIXED[i % 4][0] * s)), max(96, int(MIXED[i % 4][1] * s))) for i in range(case["frames"])]
    return [(case["w"], case["h"])] * case.get("frames", case.get("ring", 1))


def _frames(case, seed):
    """A frame per size; each rendered scene serves up to eight frames of its size, in different variants."""
    out, made = [], {}
    for i, (w, h) in enumerate(_sizes(case)):
        scene, used = made.get((w, h), (None, 8))
        if used == 8:
            scene, used = _scene(w, h, 1000 * (seed % 1000003) + i, case.get("pink", True)), 0
        made[(w, h)] = (scene, used + 1)
        out.append(_placed(learned.frame_variants(scene, used), case.get("aligned", True)))
    return out


def _served(case, seed):
    """Host frames of the serving mix; every fifth frame repeats its predecessor's scene, shifted (a stereo pair)."""
    out = []
    for i in range(case["frames"]):
        if i % 5 == 4:
            out.append(np.ascontiguousarray(np.roll(out[-1], -9, axis=1)))
        else:
            w, h = SERVED[(i + seed) % 4]
            out.append(_scene(w, h, 1000 * (seed % 1000003) + i, True).cpu().numpy())
    return out


def _patches(n, seed):
    """n patches of 64 x 64 pixels cut from scenes, and labels (a third of them positive)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 1)
    scenes = torch.stack([_scene(1280, 720, 1000 * (seed % 1000003) + i, True) for i in range(4)])
    f = torch.randint(0, 4, (n,), device="cuda", generator=gen)
    y = torch.randint(0, 720 - 63, (n,), device="cuda", generator=gen)
    x = torch.randint(0, 1280 - 63, (n,), device="cuda", generator=gen)
    at = torch.arange(64, device="cuda")
    tiles = scenes[f[:, None, None], (y[:, None] + at)[:, :, None], (x[:, None] + at)[:, None, :]]
    tiles[::50, :16] = 0  # patches at an image's edge: zero halo
    labels = (torch.rand(n, device="cuda", generator=gen) < 0.33).float()
    return tiles.contiguous(), labels


def _meta():
    with open(learned.DEFAULT_META) as f:
        return json.load(f)


# ------------------------------------------------------------------ the calls
class _Server:
    """Owner of a server handle."""

    def __init__(self, features):
        self.h = ofg.of_server_create(max_w=3840, max_h=2160, levels=8, scale=1.2, fast_t=20, fast_t_lo=7,
                                      harris_k=0.04, n_features=features, slots=4, max_batch=16,
                                      memory_budget=12 << 30)

    def __del__(self):
        ofg.of_server_destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("stream", "batch", "learned"):
        st["frames"] = _frames(case, seed)
        n = 1 if kind == "stream" else len(st["frames"])
        st["det"] = ofg.Detector(max(f.shape[1] for f in st["frames"]), max(f.shape[0] for f in st["frames"]),
                                 max_levels=case["levels"], max_features=case["features"], max_batch=n,
                                 fast_t_lo=case["t_lo"])
        st["det"].out.zero_()
        st["args"] = dict(levels=case["levels"], scale=case["scale"], fast_t=case["t"], n_features=case["features"])
        if case.get("tuned"):
            st["det"].autotune(st["frames"], **st["args"])
        if kind == "learned":
            st["net"] = learned.TileNet(0).load(learned.DEFAULT_WEIGHTS)
            st["meta"] = _meta()
            st["descr"] = [(f, f.shape[1], f.shape[0], f.stride(0)) for f in st["frames"]]
    elif kind == "level":
        st["frame"] = _placed(_scene(case["w"], case["h"], seed, case["pink"]), True)
        st["out"] = torch.zeros(case["features"] * RECORD, dtype=torch.uint8, device="cuda")
        st["count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind in ("logits", "train"):
        st["tiles"], st["labels"] = _patches(case["n"], seed)
        st["net"] = learned.TileNet(0).load(learned.DEFAULT_WEIGHTS)
    else:
        st["frames"] = _served(case, seed)
        st["server"] = _Server(case["features"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "stream":
        return [st["det"].detect(f, **st["args"]).view(np.uint8) for f in st["frames"]]
    if kind == "batch":
        return st["det"].detect_batch(st["frames"], **st["args"])
    if kind == "level":
        ofg.of_detect_level_noalloc(st["frame"], case["w"], case["h"], st["frame"].stride(0), case["t"], case["t_lo"],
                                    0.04, case["features"], st["out"], st["count"],
                                    stream=torch.cuda.current_stream())
        return st["out"], st["count"]
    if kind == "learned":
        det, m = st["det"], st["meta"]
        ofg.of_detect_learned(det.h, st["descr"], case["levels"], case["scale"], case["t"], 0.04, case["features"],
                              st["net"].net, m["threshold"], m["min_confidence"], m["dilate"], det.out, det.counts,
                              want_stats=False)
        return det.out, det.counts
    if kind == "logits":
        return st["net"].logits(st["tiles"])
    if kind == "train":
        net = st["net"].net
        loss = ofg.of_tcnn_loss_grad(net, st["tiles"], st["labels"], case["n"], 4.0)
        ofg.of_tcnn_adam(net, 1e-4)
        return {"loss": np.float32(loss), "grad": ofg.of_tcnn_get_params(net, 2),
                "weights": ofg.of_tcnn_get_params(net, 0)}
    s = st["server"].h
    ids = [ofg.of_server_submit(s, f) for f in st["frames"]]
    got = {}
    while len(got) < len(ids):
        for r, kp in ofg.of_server_poll(s, 16, case["features"], wait_ms=50):
            got[r.id] = kp
    return np.concatenate([got[i] for i in ids]).view(np.uint8)


# ------------------------------------------------------------------ work and exact values
def _level_pixels(w, h, levels, scale):
    s, out = 1.0, []
    for _ in range(levels):
        out.append((int(w / s + 0.5), int(h / s + 0.5)))
        s *= scale
    return out


def work(case):
    """Bytes: frames or patches in, records, logits or gradients and weights out.  Operations: the score's three-input
    minima and maxima (81 per two pixels of every level's detect region), 8 per resized pixel, the network's
    multiply-adds (two operations each; a training step three times the forward pass's)."""
    kind = case["kind"]
    if kind in ("logits", "train"):
        n = case["n"]
        flops = 2.0 * TILE_MACS * n * (3 if kind == "train" else 1)
        return {"bytes": n * 4096.0 + (8.0 * ofg.of_tcnn_num_params() if kind == "train" else 4.0 * n), "flops": flops}
    if kind == "serve":
        sizes = [SERVED[i % 4] for i in range(case["frames"])]
    elif kind == "level":
        sizes = [(case["w"], case["h"])]
    else:
        sizes = _sizes(case)
    levels, scale = (1, 1.2) if kind == "level" else (case.get("levels", 8), case.get("scale", 1.2))
    total, ops = 0.0, 0.0
    for w, h in sizes:
        total += w * h + RECORD * case["features"]
        for l, (lw, lh) in enumerate(_level_pixels(w, h, levels, scale)):
            ops += 40.5 * max(0, lw - 38) * max(0, lh - 38) + (8.0 * lw * lh if l else 0.0)
            if kind == "learned":
                ops += 2.0 * TILE_MACS * math.ceil(max(0, lw - 38) / 32) * math.ceil(max(0, lh - 38) / 32)
    return {"bytes": total, "flops": ops}


def _params64(st):
    """The network's rounded weights (those its kernels use), split into their layers, in 64 bits."""
    p = torch.from_numpy(ofg.of_tcnn_get_params(st["net"].net, 1)).double().cuda()
    shapes = [(8, 1, 3, 3), (8,), (16, 8, 3, 3), (16,), (16, 16, 3, 3), (16,), (16,), (1,)]
    out, at = [], 0
    for s in shapes:
        n = math.prod(s)
        out.append(p[at : at + n].reshape(s).clone().requires_grad_(True))
        at += n
    return out


def _logits64(p, tiles):
    x = (tiles.double()[:, None] - 128.0) / 64.0
    for k in (0, 2, 4):
        # 3 x 3 windows at stride 2 as columns: a plain matrix product in 64 bits.
        c, s = x.shape[1], x.shape[2] // 2
        cols = torch.nn.functional.unfold(x, 3, padding=1, stride=2)
        x = torch.relu(p[k].reshape(p[k].shape[0], c * 9) @ cols + p[k + 1][:, None]).reshape(-1, p[k].shape[0], s, s)
    return x.mean(dim=(2, 3)) @ p[6] + p[7]


def exact(case, seed):
    if case["kind"] not in ("logits", "train"):
        return None
    st = prepare(case, seed)
    p = _params64(st)
    if case["kind"] == "logits":
        with torch.no_grad():
            return torch.cat([_logits64(p, t) for t in st["tiles"].split(2048)])
    n, loss = case["n"], 0.0
    for t, y in zip(st["tiles"].split(1024), st["labels"].split(1024)):
        z = _logits64(p, t)
        wt = torch.where(y > 0.5, 4.0, 1.0).double()
        part = (wt * (torch.nn.functional.softplus(z) - y.double() * z)).sum() / n
        part.backward()
        loss += float(part.detach())
    g = torch.cat([q.grad.reshape(-1) for q in p])
    # Adam from the checkpoint: master weights and moments as stored, bias-corrected, no decay.
    blob, k = ofg.of_tcnn_save(st["net"].net), ofg.of_tcnn_num_params()
    step = int(np.frombuffer(blob, np.int64, 1, 12)[0]) + 1
    w, m, v = (torch.from_numpy(np.frombuffer(blob, np.float32, k, 20 + 4 * k * i).astype(np.float64)).cuda()
               for i in range(3))
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    w = w - 1e-4 * (m / (1 - 0.9**step)) / ((v / (1 - 0.999**step)).sqrt() + 1e-8)
    return {"loss": np.float64(loss), "grad": g, "weights": w}
