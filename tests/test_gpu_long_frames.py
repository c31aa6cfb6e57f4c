"""Frames whose rows span more than 4 GiB: one 4K camera of a row-interleaved buffer of many.  Everything a pass makes
of such a frame equals what it makes of a compact copy, bit for bit: letterbox, crops (boxes above, across and below the
4 GiB mark), the crops of a chained stage and of a queue."""
import numpy as np
import pytest
import torch

import paper_2502_01277_b200 as octo

pytestmark = pytest.mark.gpu

W, H, S = 3840, 2160, 640
PITCH = 192 * 3 * W  # 192 cameras side by side: row 1942 begins at 4 GiB
MARK = (1 << 32) / PITCH
CROPS = ((64, 64), (256, 256))
OPTIONS = [dict(keep_aspect=True, mean=(0.485, 0.456, 0.406), std=(0.229, 0.224, 0.225)), None]


def _head(boxes, anchors, classes=1):
    """One certain candidate per box (x1, y1, x2, y2, input pixels); scores fall from box to box."""
    head = np.zeros((1, anchors, 5 + classes), dtype=np.float32)
    for i, (x1, y1, x2, y2) in enumerate(boxes):
        head[0, i, :6] = (x1 + x2) / 2, (y1 + y2) / 2, x2 - x1, y2 - y1, 1.0, 0.95 - 0.02 * i
    return torch.from_numpy(head).cuda()


def _records(n, stage):
    return torch.zeros((n, stage.cfg.max_det, 32), dtype=torch.uint8, device="cuda")


def _pass(frame):
    scale, top = W / S, (S - S * H // W) // 2  # frame pixels per input pixel, canvas rows above
    rows = [(10, 50), (MARK - 300, MARK - 250), (MARK - 40, MARK + 30), (MARK + 1, MARK + 60), (2050, H), (5, H - 1)]
    boxes = [(60.0 * i + 5, top + lo / scale, 60.0 * i + 40, top + hi / scale) for i, (lo, hi) in enumerate(rows)]
    st = octo.Stage(net_size=S, max_batch=1, num_anchors=64, num_classes=1, head_is_logits=False, branches=CROPS, crop_options=OPTIONS)
    st2 = octo.Stage(net_size=256, max_batch=len(rows), num_anchors=64, num_classes=1, head_is_logits=False, branches=((40, 24),))
    q = octo.Queue(64, 48, 32, max_bz=16)
    out = {}
    try:
        out["input"] = st.preprocess([frame], [(W, H)])
        out["dets"], out["counts"] = st.postprocess(_head(boxes, 64), dets=_records(1, st))
        assert int(out["counts"][0]) == len(rows)
        for b, (ow, oh) in enumerate(CROPS):
            buf = torch.zeros((len(rows), 3, oh, ow), dtype=torch.float16, device="cuda")
            out["crops%d" % b], out["offsets%d" % b], out["items%d" % b] = st.crop(b, len(rows), out=buf)
        q.push(st, 0)
        buf = torch.zeros((16, 3, 32, 48), dtype=torch.float16, device="cuda")
        out["queue"], records, _ = q.pop(16, out=buf)
        out["records"] = records[:, 20:].clone()  # (without the address, size and pitch of the frame)
        head2 = _head([(10, 20, 200, 250), (150, 5, 255, 60)], 64).repeat(len(rows), 1, 1)
        st2.adopt_items_device(st, 1, len(rows))
        out["dets2"], out["counts2"] = st2.postprocess(head2, dets=_records(len(rows), st2))
        buf = torch.zeros((2 * len(rows), 3, 24, 40), dtype=torch.float16, device="cuda")
        st2.crop(0, 2 * len(rows), out=buf)
        out["crops of crops"] = buf
        st2.adopt_regions([frame], [(W, H)], st.item_table(1, len(rows)))
        out["dets2 again"], _ = st2.postprocess(head2, dets=_records(len(rows), st2))
        buf = torch.zeros((2 * len(rows), 3, 24, 40), dtype=torch.float16, device="cuda")
        st2.crop(0, 2 * len(rows), out=buf)
        out["crops of regions"] = buf
        torch.cuda.synchronize()
        assert st.status() == 0 and st2.status() == 0
    finally:
        st.close()
        st2.close()
        q.close()
    return out


def test_frame_of_more_than_4_gib():
    gen = torch.Generator(device="cuda").manual_seed(3)
    compact = torch.randint(0, 256, (H, 3 * W), dtype=torch.uint8, device="cuda", generator=gen)
    whole = torch.empty((H, PITCH), dtype=torch.uint8, device="cuda")
    frame = whole[:, 3 * W * 100:3 * W * 101]
    frame.copy_(compact)
    assert frame.stride(0) == PITCH and (H - 1) * PITCH > 1 << 32
    want, got = _pass(compact), _pass(frame)
    assert want["crops of crops"].any() and want["queue"].any()
    for name in want:
        assert torch.equal(got[name], want[name]), name
