"""How the crop kernel cuts its work: bands of rows while there are fewer crops than tiles wanted, whole
crops above that, a finer cut of the last crops; heights around the groups of eight rows a band is made of,
widths below and above what one pass of the threads covers.  Every crop is compared with the oracle, within
the distance of one binary16 step (values below 1); slots past the last crop stay untouched."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_01277_b200 as octo
from gpu_harness import half_absdiff, run_stage_gpu
from test_gpu_parity import PIX_TOL, _check_dets

pytestmark = pytest.mark.gpu
SIDE = 256


def _check(count, crops, batch=1):
    rng = np.random.default_rng(count)
    anchors = count + 3
    head = np.zeros((batch, anchors, 6), dtype=np.float32)
    i = np.arange(count)
    for b in range(batch):  # boxes of different sizes that do not overlap: all are kept
        head[b, :count, 0], head[b, :count, 1] = 2 + 5.0 * (i % 48), 2 + 5.0 * (i // 48)
        head[b, :count, 2], head[b, :count, 3] = rng.uniform(1, 4.5, count), rng.uniform(1, 4.5, count)
        head[b, :count, 4], head[b, :count, 5] = 1.0, rng.uniform(0.3, 0.99, count)
    frames = [rng.integers(0, 256, (384, 3 * 512), dtype=np.uint8) for _ in range(batch)]
    sizes = [(512, 384)] * batch
    st = octo.Stage(net_size=SIDE, max_batch=batch, num_anchors=anchors, num_classes=1, head_is_logits=False,
                    max_det=1000, branches=crops)
    try:
        ref = oracle.run_stage(frames, sizes, head, SIDE, crops, logits=False, max_det=1000, do_letterbox=False,
                               threads=8)
        total = len(ref.items[0])
        assert total > 0
        res = run_stage_gpu(st, frames, sizes, head, max_items=[total + 2] * len(crops))
        _check_dets(res, ref)
        assert res.status == 0
        for k in range(len(crops)):
            assert res.n_items[k] == (total, total)
            it = res.items[k]
            assert np.array_equal(np.stack([it["rx0"], it["ry0"], it["rx1"], it["ry1"]], 1), ref.rects[k])
            assert half_absdiff(res.crops[k][:total], ref.crops[k][:total]) <= PIX_TOL
            assert np.all(res.crops[k][total:] == 0x7BFF)
    finally:
        st.close()


@pytest.mark.parametrize("count", [1, 2, 7, 60, 443, 444, 445, 900])
def test_row_bands(count):
    _check(count, ((8, 1), (16, 7), (24, 9), (224, 33)))


@pytest.mark.parametrize("count,batch", [(1, 1), (13, 1), (150, 2), (887, 2), (888, 2), (900, 3)])
def test_tall_and_wide_crops(count, batch):
    """At 900 x 3 crops every crop is one tile, except the last ones."""
    _check(count, ((16, 97), (264, 8), (40, 64)), batch)


@pytest.mark.parametrize("count", [55, 56, 58, 59, 83, 84])
def test_third_tiles(count):
    """Sixteen tiles a crop for 444 CTAs (148 SMs): third tiles for none of them, for a few (drawn from the counter), for
    an eighth and more (fixed), for nearly all; fourth tiles."""
    _check(count, ((8, 128), (40, 127)))


@pytest.mark.parametrize("first", [1, 5, 9, 13])
def test_rows_of_a_pass_four_at_a_time(first):
    """Passes of few rows: the source rows are requested four at a time, the last one to three by themselves."""
    _check(9, tuple((8, first + i) for i in range(4)))


def test_passes_of_64_rows():
    """Narrow rectangles reduced more than twofold, so many that most crops are one tile: passes of 32 output rows that
    stage two source rows for each, and of one row less."""
    w, h, net, count, batch = 512, 512, 256, 900, 2
    rng = np.random.default_rng(8)
    frames = [rng.integers(0, 256, (h, 3 * w), dtype=np.uint8) for _ in range(batch)]
    head = np.zeros((batch, count, 6), dtype=np.float32)
    i = np.arange(count)
    for b in range(batch):
        head[b, :, 0], head[b, :, 1] = 4 + 0.27 * i, 128 + (i % 7)
        head[b, :, 2], head[b, :, 3] = 2 + i % 5, 100 + i % 156
        head[b, :, 4], head[b, :, 5] = 1.0, 0.99 - 0.0005 * i
    crops = ((8, 64), (16, 40), (8, 33))
    st = octo.Stage(net_size=net, max_batch=batch, num_anchors=count, num_classes=1, head_is_logits=False, iou_thresh=1.0,
                    max_det=count, branches=crops)
    try:
        ref = oracle.run_stage(frames, [(w, h)] * batch, head, net, crops, logits=False, iou_thr=1.0, max_det=count,
                               do_letterbox=False, threads=8)
        res = run_stage_gpu(st, frames, [(w, h)] * batch, head, max_items=[count * batch] * len(crops))
        _check_dets(res, ref)
        assert res.status == 0 and res.n_items[0] == (count * batch, count * batch)
        for k in range(len(crops)):
            assert half_absdiff(res.crops[k], ref.crops[k]) <= PIX_TOL
    finally:
        st.close()


@pytest.mark.parametrize("batch,widths", [(1, (400, 408, 416, 424)), (9, (384, 392, 400, 408)), (65, (312, 320, 328, 336))])
def test_widest_crops_of_three_ctas(batch, widths):
    """Widths around the last of which an SM holds three CTAs, where the ring buffers are shorter: rectangles of which a
    pass stages from two rows to all it needs."""
    w, h, net = 2400, 160, 640
    scale, top = w / net, (net - 43) / 2
    rects = [(0, 2400), (100, 2170), (310, 1800), (500, 1790), (800, 1330), (900, 500), (30, 330), (1700, 90), (2300, 40)]
    rng = np.random.default_rng(batch)
    frames = [rng.integers(0, 256, (h, 3 * w), dtype=np.uint8) for _ in range(batch)]
    head = np.zeros((batch, len(rects), 6), dtype=np.float32)
    for i, (x, width) in enumerate(rects):
        head[:, i] = (x + width / 2) / scale, top + 20, width / scale, 36 if i % 2 else 8, 1.0, 0.9 - 0.02 * i
    crops = tuple((width, 24) for width in widths)
    st = octo.Stage(net_size=net, max_batch=batch, num_anchors=len(rects), num_classes=1, head_is_logits=False,
                    iou_thresh=1.0, branches=crops)
    try:
        ref = oracle.run_stage(frames, [(w, h)] * batch, head, net, crops, logits=False, iou_thr=1.0, do_letterbox=False,
                               threads=8)
        total = len(rects) * batch
        res = run_stage_gpu(st, frames, [(w, h)] * batch, head, max_items=[total] * len(crops))
        _check_dets(res, ref)
        assert res.status == 0
        for k in range(len(crops)):
            assert res.n_items[k] == (total, total)
            assert half_absdiff(res.crops[k], ref.crops[k]) <= PIX_TOL
    finally:
        st.close()


@pytest.mark.parametrize("width", [408, 416, 424])
def test_widest_queued_crops_of_three_ctas(width):
    w, h, net, rects = 2400, 160, 640, [(0, 2400), (310, 1800), (500, 1790), (30, 330)]
    frame = np.random.default_rng(width).integers(0, 256, (h, 3 * w), dtype=np.uint8)
    head = np.zeros((1, len(rects), 6), dtype=np.float32)
    for i, (x, side) in enumerate(rects):
        head[0, i] = (x + side / 2) * net / w, net / 2, side * net / w, 36 if i % 2 else 8, 1.0, 0.9 - 0.02 * i
    st = octo.Stage(net_size=net, max_batch=1, num_anchors=len(rects), num_classes=1, head_is_logits=False, iou_thresh=1.0,
                    branches=((8, 8),))
    q = octo.Queue(64, width, 24, max_bz=8)
    try:
        st.preprocess([torch.from_numpy(frame).cuda()], [(w, h)])
        dets, counts = st.postprocess(torch.from_numpy(head).cuda())
        q.push(st, 0)
        out, _, info = q.pop(8)
        d, c = octo.dets_to_numpy(dets, counts)
        assert c[0] == len(rects) and int(info[0]) == len(rects)
        got = out.view(torch.int16).cpu().numpy().view(np.uint16)
        for i in range(len(rects)):
            assert half_absdiff(got[i], oracle.crop(frame, w, h, d[0, i:i + 1], width, 24)) <= PIX_TOL
    finally:
        q.close()
        st.close()


@pytest.mark.parametrize("keep_aspect,oh", [(False, 3), (True, 2)])
def test_few_columns_of_a_16384_pixel_frame(keep_aspect, oh):
    """Four columns of a crop 8 pixels wide reach over 6144 pixels of such a frame, three of the seven that a rectangle of
    16384x4681 keeps in 8x2 over 7022: two of their rows need longer ring buffers.  Crops of a stage whose regions the
    host gives, and of a queue."""
    w, h, net = 16384, 4681, 64
    dev = torch.randint(0, 256, (h, 3 * w), dtype=torch.uint8, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
    frame = dev.cpu().numpy()
    rects = [(0, 16384), (0, 16000), (700, 16384), (4, 14600), (3000, 9000), (8000, 8100)]
    head = np.zeros((1, len(rects), 6), dtype=np.float32)
    for i, (lo, hi) in enumerate(rects):
        head[0, i] = (lo + hi) / 2 * net / w, net / 2, (hi - lo) * net / w, net, 1.0, 0.9 - 0.02 * i
    options = dict(keep_aspect=keep_aspect)
    whole = np.zeros(1, dtype=octo.ITEM_DTYPE)
    whole["rx1"], whole["ry1"] = w, h
    st = octo.Stage(net_size=net, max_batch=1, num_anchors=len(rects), num_classes=1, head_is_logits=False, iou_thresh=1.0,
                    branches=((8, oh), (16, oh)), crop_options=[options] * 2)
    q = octo.Queue(64, 8, oh, max_bz=8)
    try:
        q.set_options(**options)
        st.adopt_regions([dev], [(w, h)], whole)
        dets, counts = st.postprocess(torch.from_numpy(head).cuda())
        got = [st.crop(b, len(rects))[0] for b in range(2)]
        q.push(st, 0)
        got.append(q.pop(8)[0])
        d, c = octo.dets_to_numpy(dets, counts)
        assert c[0] == len(rects) and st.status() == 0
        for buf, ow in zip(got, (8, 16, 8)):
            crops = buf.view(torch.int16).cpu().numpy().view(np.uint16)
            for i in range(len(rects)):
                assert half_absdiff(crops[i], oracle.crop(frame, w, h, d[0, i:i + 1], ow, oh, **options)) <= PIX_TOL
    finally:
        q.close()
        st.close()
