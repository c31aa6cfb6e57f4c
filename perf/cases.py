"""What a user of the cascade-stage library has it do, as cases that can be timed.

A case is one pass of a serving loop on the GPU: the frames and the detector head of a batch are
in device memory, and the pass takes them through the public entry points of the package
(letterbox, decode + NMS, and what becomes of the detections: crops for one or two downstream
models, a chained second-level detector, or the device-side queue).  The detector itself is not
part of the library, so its output is drawn: background values around the recipe's logit mean and
a number of raised anchors in clusters of overlapping boxes, the way a detector reports objects.
Sizes are those of the repository's workloads and tests, and generic ones beside them."""
from __future__ import annotations

import math

import torch

import paper_2502_01277_b200 as octo

# Every field of a case.  `kind` says what happens to the detections: "crops" (one or two
# downstream models), "cascade" (a second detector runs on the crops, handed over on the device),
# "queue" (items wait on the device and leave in batches of `bz`).
_DEFAULTS = dict(
    kind="crops", batch=1, width=1920, height=1080, width2=0, height2=0,  # a second camera size, mixed in
    net=640, classes=80, planes=False, logits=True, multi_label=False, agnostic=False,
    raised=200, groups=25, jitter=0.15, spread=1.25,  # objects per frame and how their boxes scatter
    kept=29, max_det=300,                             # detections a frame is expected to yield, and the cap
    crop_w=224, crop_h=224, crop2_w=0, crop2_h=0,     # downstream models (a second one when crop2_w > 0)
    fit=False, norm=False,                            # aspect-preserving crops, mean / std
    net2=0, classes2=0, bz=0)

_MEAN, _STD = (0.485, 0.456, 0.406), (0.229, 0.224, 0.225)


def _case(**kw):
    return {**_DEFAULTS, **kw}


def listed():
    return [
        # one small frame: the smallest call, where launches and host work are all there is
        _case(name="tiny_b1", width=320, height=240, net=320, raised=40, groups=40, kept=38, crop_w=64, crop_h=64),
        # one camera at its frame rate
        _case(name="camera_b1"),
        # a few HD cameras; the detector exports probabilities, the classifier wants fitted, normalised crops
        _case(name="fitted_b4", batch=4, width=1280, height=720, logits=False, raised=150, groups=20, kept=22, fit=True,
              norm=True),
        # eight 1080p traffic cameras, vehicle crops
        _case(name="traffic_b8", batch=8, raised=150, groups=20, kept=23),
        # odd camera format, smaller detector with few classes, NMS across classes, plate-shaped crops
        _case(name="ragged_b13", batch=13, width=1277, height=717, net=416, classes=7, agnostic=True, raised=90, groups=15,
              kept=16, crop_w=96, crop_h=33),
        # an anchor-free detector with several labels per box
        _case(name="planes_b32", batch=32, planes=True, multi_label=True, kept=43),
        # mixed 720p / 1080p cameras feeding a vehicle classifier and a plate detector
        _case(name="two_branch_b64", batch=64, width=1280, height=720, width2=1920, height2=1080, raised=150, groups=20,
              kept=23, crop2_w=256, crop2_h=256),
        # a crowd seen by one camera, and by 32
        _case(name="crowd_b1", raised=5000, groups=250, jitter=0.25, spread=1.4, kept=770, max_det=1000, crop_w=128,
              crop_h=128),
        _case(name="crowd_b32", batch=32, raised=5000, groups=250, jitter=0.25, spread=1.4, kept=770, max_det=1000,
              crop_w=128, crop_h=128),
        # a throughput server: one batch for a whole GPU
        _case(name="server_b256", batch=256),
        # vehicles found in 16 frames, each crop through a second detector, its boxes cropped from the frame
        _case(name="cascade_b16", kind="cascade", batch=16, raised=150, groups=20, kept=23, crop_w=256, crop_h=256,
              net2=256, classes2=8),
        # two cameras feeding the queue of a model that takes batches of 64
        _case(name="queue_b2", kind="queue", batch=2, raised=150, groups=20, kept=23, bz=64),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = _case(batch=log_int(1, 256))
    if rng.random() < 0.5:
        c["width"], c["height"] = rng.choice([(320, 240), (640, 480), (1280, 720), (1920, 1080), (1080, 1920), (3840, 2160)])
    else:
        c["width"] = log_int(300, 2600)
        c["height"] = max(200, int(c["width"] * rng.uniform(0.5, 1.1)))
    c["net"] = rng.choice([320, 416, 512, 640, 640])
    c["classes"] = rng.choice([1, 7, 20, 80, 80])
    c["kind"] = rng.choice(["crops", "crops", "crops", "crops", "cascade", "queue"])
    head = rng.choice(["rows", "rows", "rows", "probabilities", "planes", "planes"])
    c["planes"], c["logits"] = head == "planes", head != "probabilities"
    variant = rng.choice(["", "", "multi", "agnostic"])
    c["multi_label"], c["agnostic"] = variant == "multi" and c["classes"] > 1, variant == "agnostic"
    if rng.random() < 0.2:  # a crowd
        c.update(raised=log_int(800, 5000), jitter=0.25, spread=1.4, max_det=1000)
        c["groups"] = max(1, c["raised"] // 20)
        c["kept"] = min(1000, 3 * c["groups"] + 80)
    else:
        c["raised"] = log_int(20, 300)
        c["groups"] = max(1, c["raised"] // rng.choice([1, 4, 8]))
        c["kept"] = c["groups"] + c["groups"] // 4 + 1
    if c["multi_label"]:
        c["kept"] = min(c["max_det"], 2 * c["kept"])
    anchors = _anchors(c["net"], c["planes"])
    if c["raised"] > anchors // 4:
        c["raised"] = anchors // 4
    c["crop_w"], c["crop_h"] = 8 * log_int(4, 32), log_int(24, 288)
    c["fit"], c["norm"] = rng.random() < 0.25, rng.random() < 0.25
    if c["kind"] == "crops" and rng.random() < 0.25:
        c["crop2_w"], c["crop2_h"] = 8 * log_int(4, 32), log_int(24, 288)
    elif c["kind"] == "cascade":
        c.update(net2=rng.choice([128, 192, 256]), classes2=8, fit=False, norm=False)
        c["crop_w"] = c["crop_h"] = c["net2"]
    elif c["kind"] == "queue":  # a few cameras, and a batch that takes about what they yield
        c["batch"] = log_int(1, 12)
        c["bz"] = 8 * max(2, min(100, c["batch"] * c["kept"] * rng.choice([1, 2, 3]) // 8))
    # no more work than the largest listed case
    most = max(_bytes(x) for x in listed() if not x["groups"] >= 250) * (0.4 if c["raised"] > 500 else 0.8)
    while c["batch"] > 1 and _bytes(c) > most:
        c["batch"] = c["batch"] * 3 // 4
    return c


# ---- inputs ----------------------------------------------------------------------------------

def _anchors(net, planes):
    return (1 if planes else 3) * sum((net // s) ** 2 for s in (8, 16, 32))


def _sizes(case):
    """(width, height) of every frame of the batch."""
    two = case["width2"] > 0
    return [(case["width2"], case["height2"]) if two and i % 2 else (case["width"], case["height"])
            for i in range(case["batch"])]


def _fitted(w, h, net):
    """Size of a frame inside the net x net detector input."""
    if w >= h:
        return net, max(1, (2 * h * net + w) // (2 * w))
    return max(1, (2 * w * net + h) // (2 * h)), net


def _items(case):
    """Slots of a downstream batch, per branch, that the caller provisions."""
    return case["batch"] * min(case["max_det"], case["kept"] + case["kept"] // 3 + 4)


def _frames(gen, sizes):
    """Camera-shaped frames: gradients, a sinusoid and noise per channel; rows padded to 16 bytes."""
    out = [None] * len(sizes)
    for w, h in sorted(set(sizes)):
        which = [i for i, s in enumerate(sizes) if s == (w, h)]
        pitch = (3 * w + 15) // 16 * 16
        buf = torch.zeros((len(which), h, pitch), dtype=torch.uint8, device="cuda")
        x = torch.arange(w, device="cuda").view(1, 1, w, 1) / w
        y = torch.arange(h, device="cuda").view(1, h, 1, 1) / h
        step = max(1, 40_000_000 // (3 * w * h))
        for lo in range(0, len(which), step):
            k = min(step, len(which) - lo)

            def uniform(a, b, *shape):
                return torch.empty(shape, device="cuda").uniform_(a, b, generator=gen)

            wave = torch.randint(1, 7, (2, k, 1, 1, 1), device="cuda", generator=gen)
            v = (uniform(60, 180, k, 1, 1, 3) + uniform(-60, 60, k, 1, 1, 3) * x + uniform(-60, 60, k, 1, 1, 3) * y
                 + 40 * torch.sin(2 * math.pi * (wave[0] * x + wave[1] * y) + uniform(0, 2 * math.pi, k, 1, 1, 3)))
            v += uniform(-8, 8, k, h, w, 3)
            buf[lo:lo + k, :, :3 * w] = v.round_().clamp_(0, 255).to(torch.uint8).view(k, h, 3 * w)
        for j, i in enumerate(which):
            out[i] = buf[j]
    return out


def _head(gen, case, n, net, classes, planes, logits, raised, groups, size, rows, multi_label, jitter, spread):
    """Detector head of n images: background anchors and `raised` anchors in `groups` clusters whose
    boxes (`size`: side range in head pixels) lie between head rows `rows`."""
    anchors = _anchors(net, planes)
    at = 4 if planes else 5  # first class value
    background = -7.0 if planes else -4.0

    def uniform(a, b, *shape):
        return torch.empty(shape, device="cuda").uniform_(a, b, generator=gen)

    head = torch.empty((n, at + classes, anchors) if planes else (n, anchors, at + classes), device="cuda")
    head.normal_(background, 1.0, generator=gen)
    value = head.transpose(1, 2) if planes else head  # [n, anchors, values]
    value[:, :, 0:2] = uniform(0, net, n, anchors, 2)
    value[:, :, 2:4] = uniform(8, 120, n, anchors, 2)
    # the clusters: centre, size and class of each, members scattered around it
    box = uniform(size[0], size[1], n, groups, 2)
    lo = torch.tensor([0.0, float(rows[0])], device="cuda") + box / 2
    hi = torch.tensor([float(net), float(rows[1])], device="cuda") - box / 2
    centre = torch.where(hi > lo, lo + (hi - lo) * uniform(0, 1, n, groups, 2), (lo + hi) / 2)
    label = torch.randint(0, classes, (n, groups), device="cuda", generator=gen)
    group = torch.arange(raised, device="cuda") % groups
    who = torch.rand((n, anchors), device="cuda", generator=gen).topk(raised, dim=1).indices
    image = torch.arange(n, device="cuda").view(n, 1).expand(n, raised)
    value[image, who, 0:2] = centre[:, group] + box[:, group] * uniform(-jitter, jitter, n, raised, 2)
    value[image, who, 2:4] = box[:, group] * uniform(1 / spread, spread, n, raised, 2)
    strong = torch.empty((3, n, raised), device="cuda").normal_(2.0, 0.5, generator=gen)
    if not planes:
        value[image, who, 4] = strong[0]
    value[image, who, at + label[:, group]] = strong[1]
    if multi_label:  # every other cluster carries a second label
        second = (label[:, group] + 1) % classes
        some = (group % 2 == 0).view(1, raised).expand(n, raised)
        value[image[some], who[some], at + second[some]] = strong[2][some]
    if not logits:
        value[:, :, (at if planes else 4):].sigmoid_()
    return head


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, net, sizes = case["batch"], case["net"], _sizes(case)
    u8 = lambda *shape: torch.zeros(shape, dtype=torch.uint8, device="cuda")  # noqa: E731
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    f16 = lambda *shape: torch.zeros(shape, dtype=torch.float16, device="cuda")  # noqa: E731
    s = dict(case=case, sizes=sizes, frames=_frames(gen, sizes))
    nh = min(_fitted(w, h, net)[1] for w, h in sizes)
    s["head"] = _head(gen, case, n, net, case["classes"], case["planes"], case["logits"], case["raised"], case["groups"],
                      (40 * net / 640, 200 * net / 640), ((net - nh) / 2, (net + nh) / 2), case["multi_label"],
                      case["jitter"], case["spread"])
    branches = [(case["crop_w"], case["crop_h"])] + ([(case["crop2_w"], case["crop2_h"])] if case["crop2_w"] else [])
    option = dict(keep_aspect=case["fit"], **(dict(mean=_MEAN, std=_STD) if case["norm"] else {}))
    s["stage"] = octo.Stage(net_size=net, max_batch=n, num_anchors=_anchors(net, case["planes"]), num_classes=case["classes"],
                            head_is_logits=case["logits"], max_det=case["max_det"], branches=branches,
                            class_agnostic=case["agnostic"], head_layout="planes" if case["planes"] else "rows",
                            multi_label=case["multi_label"], crop_options=[option] * len(branches))
    s["detector_input"] = f16(n, 3, net, net)
    s["dets"], s["counts"] = u8(n, case["max_det"], 32), i32(n)
    if case["kind"] == "queue":
        bz = case["bz"]
        s["queue"] = octo.Queue(max(64 * bz, 2 * n * case["max_det"]), case["crop_w"], case["crop_h"], max_bz=bz)
        if case["fit"] or case["norm"]:
            s["queue"].set_options(**option)
        s["crops"], s["records"], s["info"] = f16(bz, 3, case["crop_h"], case["crop_w"]), u8(bz, 48), i32(4)
        return s
    s["branches"] = [(f16(_items(case), 3, h, w), i32(n + 1), i32(2)) for w, h in branches]
    if case["kind"] == "cascade":
        m, net2, classes2 = _second(case), case["net2"], case["classes2"]
        s["head2"] = _head(gen, case, m, net2, classes2, False, True, 12, 3, (30, min(120, net2 / 2)), (0, net2), False, 0.15,
                           1.25)
        s["stage2"] = octo.Stage(net_size=net2, max_batch=m, num_anchors=_anchors(net2, False), num_classes=classes2,
                                 max_det=16, branches=((64, 32),))
        s["second"] = dict(dets=u8(m, 16, 32), counts=i32(m), crops=f16(8 * m, 3, 32, 64), offsets=i32(m + 1), n_items=i32(2))
    return s


def _second(case):
    """Images the second detector of a cascade runs on: the items a batch is expected to yield."""
    return max(1, min(octo.binding.OCTO_MAX_BATCH, case["batch"] * case["kept"]))


# ---- one pass --------------------------------------------------------------------------------

def run(s):
    stage = s["stage"]
    stage.preprocess(s["frames"], s["sizes"], out=s["detector_input"])
    # (the caller's detector runs here)
    stage.postprocess(s["head"], dets=s["dets"], counts=s["counts"])
    out = dict(detector_input=s["detector_input"], dets=s["dets"], counts=s["counts"])
    if "queue" in s:
        s["queue"].push(stage, 0)
        s["queue"].pop(s["case"]["bz"], out=s["crops"], items=s["records"], info=s["info"], max_wait=1)
        # a record starts with the address of its frame, which is another one in every process
        out.update(crops=s["crops"], records=s["records"][:, 8:], info=s["info"])
        return out
    for b, (crops, offsets, n_items) in enumerate(s["branches"]):
        stage.crop(b, crops.shape[0], out=crops, offsets=offsets, n_items=n_items)
        out["crops%d" % b], out["offsets%d" % b], out["n_items%d" % b] = crops, offsets, n_items
    if "stage2" in s:
        z, stage2 = s["second"], s["stage2"]
        stage2.adopt_items_device(stage, 0, s["head2"].shape[0])
        # (the caller's second detector runs here)
        stage2.postprocess(s["head2"], dets=z["dets"], counts=z["counts"])
        stage2.crop(0, z["crops"].shape[0], out=z["crops"], offsets=z["offsets"], n_items=z["n_items"])
        out["second"] = z
    return out


# ---- what a pass cannot do without -------------------------------------------------------------

def _head_bytes(images, anchors, classes, planes, logits, candidates):
    """Rows of logits are scanned by their objectness (one 32-byte sector each) and read whole where
    it passes; probabilities are read whole, as are the class planes of the planes layout."""
    if planes:
        return images * (4 * classes * anchors + candidates * 4 * 32)
    if not logits:
        return images * 4 * (5 + classes) * anchors
    return images * (32 * anchors + candidates * 4 * (5 + classes))


def _bytes(case):
    n, net, total = case["batch"], case["net"], 0.0
    pixels = 0.0  # of the frames' rectangles that become crops
    for w, h in _sizes(case):
        nw, nh = _fitted(w, h, net)
        tapped = h if nh >= h else nh if h % nh == 0 and (h // nh) % 2 else min(h, 2 * nh)
        total += 3 * w * tapped + 3 * net * net * 2
        side = min(120 * net / 640 * w / nw, w, h)
        pixels += min(case["kept"] * side * side, w * h)
    total += _head_bytes(n, _anchors(net, case["planes"]), case["classes"], case["planes"], case["logits"], case["raised"])
    per_item = [6 * case["crop_w"] * case["crop_h"], 6 * case["crop2_w"] * case["crop2_h"]]
    total += 3 * pixels + n * case["kept"] * (sum(per_item) + 32)
    if case["kind"] == "cascade":
        m = _second(case)
        total += _head_bytes(m, _anchors(case["net2"], False), case["classes2"], False, True, 12) + m * 4 * 6 * 64 * 32
    return total


def work(case):
    values = 3 * case["batch"] * (case["net"] ** 2 + case["kept"] * (case["crop_w"] * case["crop_h"] + case["crop2_w"] * case["crop2_h"]))
    return {"bytes": _bytes(case), "flops": 8.0 * values}  # two horizontal lerps, a vertical one and the scale per value


def tolerance(case):
    # Counts, indices, rectangles, scores and boxes are exact.  Pixels are binary16: a value that falls
    # close to a rounding boundary may come out one step (at most 2^-10 of itself) apart: 3e-5 to 8e-4 of
    # them do against bilinear sampling in 64 bits, a relative error of 4e-6 to 8e-6.
    return {"rel": 4e-5, "max": 1e-3}
