"""The dense forms of the decode step at the sizes where they can go wrong: rows-layout probabilities
staged in tiles of 128 rows (partial tiles, rows whose length shares factors with the 32 banks, heads
that do not start every image on a 16-byte boundary), and planes heads in both warp splits with the
second look of multi-label heads at the anchors with a value above the threshold.  Oracle: the CPU
decode + NMS; every decision is made in the same individually rounded binary32 operations, so kept
detections are bit-equal."""
import numpy as np
import pytest

import oracle
import paper_2502_01277_b200 as octo
from gpu_harness import run_stage_gpu
from test_gpu_parity import _check_dets

pytestmark = pytest.mark.gpu


def _run(head, planes, num_anchors, num_classes, **kw):
    n, s = head.shape[0], 128
    frames = [np.zeros((96, 384), dtype=np.uint8) for _ in range(n)]
    sizes = [(128, 96)] * n
    st = octo.Stage(net_size=s, max_batch=n, num_anchors=num_anchors, num_classes=num_classes, max_det=300,
                    head_layout="planes" if planes else "rows", branches=((8, 8),), **kw)
    try:
        res = run_stage_gpu(st, frames, sizes, head, max_items=[4])
        ref = oracle.run_stage(frames, sizes, head, s, ((8, 8),), logits=kw.get("head_is_logits", True), max_det=300,
                               agnostic=kw.get("class_agnostic", False), layout="planes" if planes else "rows",
                               multi_label=kw.get("multi_label", False), do_letterbox=False, do_crops=False)
        _check_dets(res, ref)
        assert res.stats["candidates"] == int(ref.n_cand.sum())
        return res, ref
    finally:
        st.close()


def _boxes(rng, shape):
    return np.concatenate([rng.uniform(0, 128, shape + (2,)), rng.uniform(4, 60, shape + (2,))], -1).astype(np.float32)


@pytest.mark.parametrize("anchors", [1, 127, 128, 129, 401])
@pytest.mark.parametrize("classes", [1, 3, 11, 27, 80, 128])
@pytest.mark.parametrize("variant", ["single", "multi", "agnostic"])
def test_probability_rows(anchors, classes, variant):
    rng = np.random.default_rng(anchors * 131 + classes)
    head = np.zeros((2, anchors, 5 + classes), dtype=np.float32)
    head[..., :4] = _boxes(rng, (2, anchors))
    head[..., 4] = rng.uniform(0.2, 1.0, (2, anchors))
    few = rng.random((2, anchors, classes)) < 1.2 / classes  # about one label an anchor: the workspace holds two
    head[..., 5:] = np.where(few, np.round(rng.uniform(0, 1, few.shape) * 16) / 16, 0.01)  # ties among the classes
    if anchors > 4:
        head[0, 1, 4 + classes] = np.nan
        head[1, 2, 2] = 0.0
        head[1, anchors - 1, 3] = np.inf
    res, _ = _run(head, False, anchors, classes, head_is_logits=False, multi_label=variant == "multi",
                  class_agnostic=variant == "agnostic")
    assert res.status & ~0x2 == (0x1 if anchors > 4 else 0)


@pytest.mark.parametrize("classes", [1, 11, 58, 59, 123])
@pytest.mark.parametrize("variant", ["single", "multi", "agnostic"])
def test_probability_rows_of_any_sign(classes, variant):
    """Factors of both signs (two negative ones make a score), zeros of both signs and equal maxima at the ends of
    rows of 6 to 128 values, a value that is not finite at every position of a row."""
    anchors, rng = 300, np.random.default_rng(classes)
    head = np.zeros((2, anchors, 5 + classes), dtype=np.float32)
    head[..., :4] = _boxes(rng, (2, anchors))
    head[..., 4] = rng.choice([-1.0, -0.5, -0.0, 0.0, 0.25, 0.5, 1.0, 1.5], (2, anchors))
    head[..., 5:] = -0.01
    for k in (0, classes - 1, int(rng.integers(classes))):
        head[..., 5 + k] = rng.choice([-0.75, -0.5, 0.0, 0.5, 0.75, 1.0], (2, anchors))
    for e in range(5 + classes):
        head[1, 2 * e + 1, e] = (np.nan, np.inf, -np.inf)[e % 3]
    res, _ = _run(head, False, anchors, classes, head_is_logits=False, multi_label=variant == "multi",
                  class_agnostic=variant == "agnostic")
    assert res.status & 0x1


@pytest.mark.parametrize("anchors", [3, 4, 127, 128, 516, 1028])
@pytest.mark.parametrize("classes,logits", [(1, False), (39, True), (41, False), (128, True)])
@pytest.mark.parametrize("multi", [False, True])
def test_planes(anchors, classes, logits, multi):
    """Class counts around the planes eight groups of warps look at together, anchor counts around
    a CTA's share (128 or 32), in the vector and the scalar form (anchors not a multiple of four)."""
    _planes(2, anchors, classes, logits, multi)


@pytest.mark.parametrize("anchors,n", [(128 * 5, 512), (128 * 2 - 1, 512)])
def test_planes_wide_split(anchors, n):
    """Enough CTAs for four (eight) warps side by side along the anchors: vector and scalar form."""
    _planes(n, anchors, 9, True, True)


@pytest.mark.parametrize("classes", [2, 7, 8, 9, 10, 11, 40, 63, 64, 65])
@pytest.mark.parametrize("n,anchors", [(2, 516), (2, 517), (300, 64), (300, 66)])
@pytest.mark.parametrize("multi", [False, True])
def test_planes_around_a_batch_of_loads(classes, n, anchors, multi):
    """Class counts around the planes a thread has in flight (5 or 8, of one, two or eight groups of warps), in
    both splits of both forms, with values that are not finite in the first and the last plane."""
    _planes(n, anchors, classes, classes % 2 == 0, multi, bad=True)


def _planes(n, anchors, classes, logits, multi, bad=False):
    rng = np.random.default_rng(anchors * 17 + classes)
    head = np.full((n, 4 + classes, anchors), -6.0, dtype=np.float32)
    head[:, :4] = np.moveaxis(_boxes(rng, (n, anchors)), -1, 1)
    some = rng.random((n, 1, anchors)) < max(0.05, 3.0 / anchors)
    strong = some & (rng.random((n, classes, anchors)) < 1.2 / classes)  # about one label: the workspace holds two
    head[:, 4:] = np.where(strong, rng.normal(0.0, 1.5, strong.shape), -6.0)
    head[1, 4 + classes - 1, anchors - 1] = 3.0  # the last value of the head
    if not logits:
        head[:, 4:] = 1.0 / (1.0 + np.exp(-head[:, 4:]))
    if bad:
        head[0, 4 + classes - 1, 1] = np.nan
        head[1, 4, 2], head[1, 4 + classes - 1, 5] = np.inf, -np.inf
    res, _ = _run(head.astype(np.float32), True, anchors, classes, head_is_logits=logits, multi_label=multi and classes > 1)
    assert (res.status & 0x1 != 0) == bad
