"""NMS where its forms meet: candidate counts around a warp, the short path (512, with 4, 2 and 1 threads
per candidate), batches of classes, a class that the whole CTA takes (above 512, in blocks of 128), survivors
ordered by counting (96), by score buckets and by a network (above 1024, or 512 in half-sized CTAs), the half-sized
and the full on-chip capacity and what exceeds them; chains of overlapping boxes (as many rounds as
links), identical boxes, IoU values that lie exactly on the threshold, a small cap, clusters.  The oracle
makes the same binary32 decisions, so kept detections are bit-equal."""
import numpy as np
import pytest

import oracle
import paper_2502_01277_b200 as octo
from gpu_harness import run_stage_gpu
from paper_2502_01277_b200 import binding as B
from test_gpu_parity import _check_dets

pytestmark = pytest.mark.gpu
CLASSES, SIDE = 5, 256


def _boxes(rng, m, kind):
    """(cx, cy, w, h) of m boxes."""
    if kind == "chain":  # neighbours overlap above the threshold, the next but one does not
        i = np.arange(m)
        per = 60
        return np.stack([8 + 4.0 * (i % per), 6 + 12.0 * ((i // per) % 20), np.full(m, 10.0), np.full(m, 10.0)], 1)
    if kind == "apart":
        i = np.arange(m)
        return np.stack([2 + 5.0 * (i % 48), 2 + 5.0 * (i // 48), np.full(m, 4.0), np.full(m, 4.0)], 1)
    if kind == "powers":
        return np.concatenate([np.zeros((m, 2)), 2.0 ** rng.integers(-50, 67, (m, 1)) * 2.0 ** rng.integers(-2, 3, (m, 2))], 1)
    if kind == "huge":  # areas from 2^125 on: the sum of two may overflow
        return np.concatenate([np.zeros((m, 2)), 2.0 ** 63 * (1 + 0.25 * rng.integers(-2, 4, (m, 2)))], 1)
    if kind == "same":
        return np.tile(np.array([[100.0, 90.0, 30.0, 20.0]]), (m, 1))
    # a coarse grid of sizes and places: many IoU values are simple fractions, 1/2 among them
    return np.stack([rng.integers(4, 60, m) * 4.0, rng.integers(4, 40, m) * 4.0, rng.integers(1, 9, m) * 4.0,
                     rng.integers(1, 9, m) * 4.0], 1)


def _check(m, kind, share, cluster=0, agnostic=False, max_det=300, batch=1, iou=0.5, classes=CLASSES, sizes_of=None,
           crowded=None, half=False):
    """crowded: only so many images of the batch hold m candidates, the others 40.  sizes_of: candidates of each class.
    half: the first pass has to run half-sized CTAs."""
    rng = np.random.default_rng(m * 7 + len(kind))
    anchors = max(m, 4) + 3
    head = np.zeros((batch, anchors, 5 + classes), dtype=np.float32)
    for b in range(batch):
        k = m if crowded is None or b < crowded else min(m, 40)
        at = rng.permutation(anchors)[:k]
        head[b, at, :4] = _boxes(rng, m, kind)[:k]
        head[b, at, 4] = 1.0
        cls = np.where(rng.random(k) < share, 2, rng.integers(0, classes, k))
        if sizes_of is not None:
            cls = np.repeat(np.arange(classes), sizes_of)[:k]
        head[b, at, 5 + cls] = np.round(rng.uniform(0.3, 0.99, k) * 512) / 512  # ties in the score
        if kind == "chain":  # strongest first: every second link survives, one link settled per round
            head[b, at, 5:] = 0.0
            head[b, at, 7] = np.linspace(0.99, 0.3, k)
    frames, sizes = [np.zeros((192, 768), dtype=np.uint8)] * batch, [(256, 192)] * batch
    st = octo.Stage(net_size=SIDE, max_batch=batch, num_anchors=anchors, num_classes=classes, head_is_logits=False,
                    iou_thresh=iou, max_det=max_det, branches=((8, 8),), class_agnostic=agnostic)
    try:
        st.set_nms_cluster(cluster)
        ref = oracle.run_stage(frames, sizes, head, SIDE, ((8, 8),), logits=False, iou_thr=iou, max_det=max_det,
                               agnostic=agnostic, do_letterbox=False, do_crops=False)
        assert int(ref.n_cand[0]) == m
        for i in range(2):  # the counters are left clean
            res = run_stage_gpu(st, frames, sizes, head, max_items=[4])
            _check_dets(res, ref)
            if half and i == 0:
                assert st.last_nms_half_ctas()
        assert res.status & ~0x2 == (B.OCTO_STATUS_BIG_NMS if m > 8192 else 0)
        assert np.array_equal(res.offsets[0][:2], ref.offsets[0][:2])
    finally:
        st.close()


@pytest.mark.parametrize("m", [0, 1, 2, 31, 32, 33, 127, 130, 255, 256, 257, 400, 511, 512, 513])
@pytest.mark.parametrize("kind", ["grid", "chain", "same"])
@pytest.mark.parametrize("agnostic", [False, True])
def test_short_path(m, kind, agnostic):
    _check(m, kind, 0.5, agnostic=agnostic)


@pytest.mark.parametrize("m,share", [(513, 0.0), (520, 0.4), (640, 1.0), (640, 0.8), (1024, 0.5), (1024, 0.9),
                                     (1030, 1.0), (2100, 0.0), (2100, 0.2), (4097, 1.0), (8192, 0.3), (8200, 1.0),
                                     (8300, 0.0)])
@pytest.mark.parametrize("cluster", [1, 4])
def test_large_classes(m, share, cluster):
    _check(m, "grid", share, cluster=cluster, max_det=1000)


@pytest.mark.parametrize("m,share,kind,max_det", [(513, 0.0, "grid", 300), (513, 0.19, "grid", 1000), (2000, 0.21, "grid", 1000),
                                                  (2000, 0.25, "grid", 1000),
                                                  (1500, 0.0, "chain", 2), (1900, 0.0, "apart", 2000),
                                                  (900, 0.0, "same", 300), (8192, 0.1, "grid", 1000),
                                                  (8300, 0.0, "grid", 1000)])
def test_many_classes_on_one_cta(m, share, kind, max_det):
    """Classes of less than a quarter of the image: one warp per class (one of more: batches); full-sized CTAs and,
    with more images than SMs, half-sized ones."""
    for batch in (1, 160) if m <= 2000 else (1,):
        _check(m, kind, share, cluster=1, max_det=max_det, classes=40, batch=batch)
    if m <= 2000:
        _check(m, kind, share, max_det=max_det, classes=40, batch=160, half=True)


@pytest.mark.parametrize("sizes_of", [(256, 200, 200, 44), (257, 100, 100, 100, 43), (600, 60, 40, 20, 10),
                                      (250, 250, 250, 250), (1024, 512, 256, 129, 3), (3000, 1000, 60, 30, 6)])
@pytest.mark.parametrize("kind", ["grid", "apart"])
def test_half_sized_ctas(sizes_of, kind):
    """More images than SMs: batches of at most 512 candidates, ordered by counting and by words, classes above 256
    by the whole CTA, survivors below and above 512; the same images full-sized in the second pass when an image of
    more than 1024 candidates was reported."""
    _check(sum(sizes_of), kind, 0.0, classes=len(sizes_of), sizes_of=sizes_of, batch=160, crowded=4, half=True, max_det=1000)


@pytest.mark.parametrize("m", [400, 511, 600])
def test_half_sized_ctas_class_agnostic(m):
    _check(m, "grid", 0.0, batch=160, crowded=4, half=True, agnostic=True, max_det=1000)


@pytest.mark.parametrize("sizes_of,batch", [((6500, *[100] * 25), 1), ((6500, 500, 450, 400, 350, 300, 100, 400), 1),
                                            ((4000, 1100, 1000, 900, 800, 700, 512, 1), 1),
                                            ((3500, *[100] * 15), 160), ((3500, 250, 256, 200, 257, 190, 150, 200), 160)])
@pytest.mark.parametrize("cluster", [0, 1, 4])
def test_batches_of_an_image_beyond_the_chip(sizes_of, batch, cluster):
    """One class of more than a quarter beside smaller ones in images that do not fit on chip (8192, half-sized CTAs
    4096): batches with boxes from the head, ordered by counting (up to 128 a class) and by words."""
    if batch > 1 and cluster:
        return
    _check(sum(sizes_of), "grid", 0.0, classes=len(sizes_of), sizes_of=sizes_of, cluster=cluster, max_det=1000, batch=batch,
           crowded=2, half=batch > 1)


@pytest.mark.parametrize("m,classes,share", [(2600, 5, 0.0), (4200, 8, 0.0), (2600, 20, 0.16), (8192, 7, 0.0),
                                             (8192, 6, 0.0), (9000, 8, 0.0), (9000, 6, 0.1)])
@pytest.mark.parametrize("kind", ["grid", "powers"])
def test_a_warp_orders_a_class_by_a_network(m, classes, share, kind):
    """Classes of 512 to 1280 candidates on one CTA, on chip and off; the largest classes go to the whole CTA."""
    _check(m, kind, share, cluster=1, max_det=1000, classes=classes)


@pytest.mark.parametrize("m,max_det", [(120, 5), (256, 300), (600, 5), (600, 1), (1100, 70)])
@pytest.mark.parametrize("kind", ["grid", "chain"])
def test_cap_and_chains(m, max_det, kind):
    _check(m, kind, 1.0, max_det=max_det, batch=2)


@pytest.mark.parametrize("m", [96, 97, 700, 1500])
def test_many_survivors(m):
    """Boxes that do not overlap: every candidate survives (counting, score buckets, network)."""
    _check(m, "apart", 0.3, max_det=2000)


def test_thresholds_at_the_ends():
    for iou in (0.0, 1.0):
        _check(150, "grid", 0.7, iou=iou)
        _check(600, "grid", 0.7, iou=iou)


@pytest.mark.parametrize("iou", [0.0, 1e-45, 1e-38, 1e-30, 0.45])
@pytest.mark.parametrize("m", [150, 700, 1100])
def test_areas_and_thresholds_at_the_ends_of_binary32(m, iou):
    """Boxes around one point with sides from 2^-50 to 2^66: areas from underflow to overflow, quotients that
    round to zero, products with the threshold that underflow, sums of areas that overflow."""
    for kind in ("powers", "huge"):
        _check(m, kind, 0.3, iou=iou, max_det=1000)
        _check(m, kind, 0.0, iou=iou, max_det=1000, classes=40, cluster=1)
