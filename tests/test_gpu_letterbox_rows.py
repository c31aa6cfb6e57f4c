"""Rows of a letterbox CTA: 1 to 8 by the width of the frames and the size of the grid; a row is staged behind a
barrier of its own and taken by one warp, or by several where a CTA has fewer rows than warps.
Every pixel of every frame against the oracle, within the distance of one binary16 step."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_01277_b200 as octo
from gpu_harness import half_absdiff
from test_gpu_parity import PIX_TOL

pytestmark = pytest.mark.gpu
S = 104

# (width, height, rows that fit, batches on both sides of the steps of the rule on 148 SMs, rows of a CTA there)
CASES = [(100, 37, 8, {1: 2, 14: 2, 15: 4, 56: 4, 57: 8}), (400, 90, 8, {15: 4, 91: 4, 92: 8}), (104, 104, 8, {1: 2, 15: 4, 57: 8}),
         (1300, 77, 7, {1: 2, 16: 2, 17: 3, 78: 3, 79: 7}), (1500, 100, 6, {1: 2, 16: 2, 17: 3, 65: 3, 66: 6}),
         (1800, 64, 5, {56: 2, 57: 5}), (2200, 90, 4, {14: 2, 15: 4}), (3000, 40, 3, {1: 2, 16: 2, 17: 3}),
         (4600, 20, 2, {1: 2, 30: 2}), (8192, 24, 1, {1: 1, 30: 1})]


def _rows(fit, n, long_table, sms=148):
    rows = min(fit, 8)
    while rows > 2 and 2 * n * -(-S // rows) < ((10 if long_table else 16) if rows > 4 else 5 if rows == 4 else 8) * sms:
        rows = rows // 2 if rows > 4 else 2
    return rows


def test_cases_reach_every_number_of_rows():
    reached = set()
    for w, h, fit, batches in CASES:
        slots = 1 if (w, h) == (S, S) else 2
        row = (3 * w + 15) // 16 * 16 + 16
        assert min(8, (56 * 1024 - 896) // (slots * row)) == fit
        for n, rows in batches.items():
            assert _rows(fit, n, 8 * S >= slots * row) == rows
            reached.add(rows)
    assert reached == set(range(1, 9))


@pytest.mark.parametrize("w,h,n", [(w, h, n) for w, h, _, batches in CASES for n in batches])
def test_rows_of_a_cta(w, h, n):
    rng = np.random.default_rng(w + n)
    pitch = (3 * w + 15) // 16 * 16
    imgs = [rng.integers(0, 256, (h, pitch), dtype=np.uint8) for _ in range(2)]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    st = octo.Stage(net_size=S, max_batch=n, num_anchors=64, num_classes=2, branches=((8, 8),))
    try:
        out = st.preprocess([dev[i % 2] for i in range(n)], [(w, h)] * n)
        got = out.view(torch.int16).cpu().numpy().view(np.uint16)
        want = [oracle.letterbox(i, w, h, S) for i in imgs]
        for i in range(n):
            assert half_absdiff(got[i], want[i % 2]) <= PIX_TOL
        assert st.status() == 0
    finally:
        st.close()
