"""Rows of a letterbox CTA: 8, 4 or 2 rows by the size of the grid, 7 to 1 for wide frames; a row is staged
behind a barrier of its own and taken by one warp, or by several where a CTA has fewer rows than warps.
Every pixel of every frame against the oracle, within the distance of one binary16 step."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_01277_b200 as octo
from gpu_harness import half_absdiff
from test_gpu_parity import PIX_TOL

pytestmark = pytest.mark.gpu


# (width, height): at S = 104 two source rows per output row of (3 w + 32) bytes leave room for fewer than 8 rows from
# 1150 pixels on; batches of 1, 23 and 30 frames give 13, 299 and 390 CTAs of 8 rows
@pytest.mark.parametrize("n", [1, 23, 30])
@pytest.mark.parametrize("w,h", [(104, 104), (100, 37), (1200, 77), (1500, 100), (2000, 61), (3000, 40), (4600, 20), (8192, 24)])
def test_rows_of_a_cta(n, w, h):
    rng = np.random.default_rng(w + n)
    pitch = (3 * w + 15) // 16 * 16
    imgs = [rng.integers(0, 256, (h, pitch), dtype=np.uint8) for _ in range(2)]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    st = octo.Stage(net_size=104, max_batch=n, num_anchors=64, num_classes=2, branches=((8, 8),))
    try:
        out = st.preprocess([dev[i % 2] for i in range(n)], [(w, h)] * n)
        got = out.view(torch.int16).cpu().numpy().view(np.uint16)
        want = [oracle.letterbox(i, w, h, 104) for i in imgs]
        for i in range(n):
            assert half_absdiff(got[i], want[i % 2]) <= PIX_TOL
        assert st.status() == 0
    finally:
        st.close()
