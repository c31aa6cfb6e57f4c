"""How the crop kernel cuts its work: bands of rows while there are fewer crops than tiles wanted, whole
crops above that, a finer cut of the last crops; heights around the groups of eight rows a band is made of,
widths below and above what one pass of the threads covers.  Every crop is compared with the oracle, within
the distance of one binary16 step (values below 1); slots past the last crop stay untouched."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("first", [1, 5, 9, 13])
def test_rows_of_a_pass_four_at_a_time(first):
    """Passes of few rows: the source rows are requested four at a time, the last one to three by themselves."""
    _check(9, tuple((8, first + i) for i in range(4)))
