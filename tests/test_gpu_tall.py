"""Batched frames taller than a single call takes: blobs around rows where the
fused kernel's queues and the pruning grid could run out of bits are those of a
short frame that holds the same rows, moved; bit for bit."""
import numpy as np
import pytest
import torch

from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog, synth

pytestmark = pytest.mark.gpu

HALF, W = 150, 40   # rows around each place; two strips


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


def _sorted(x, y, l, s, r):
    o = np.lexsort((l, x, y))
    return [np.asarray(v)[o] for v in (x, y, l, s, r)]


@pytest.mark.parametrize("h,places", [(70_000, [1 << 16, 30_000, 69_800]), ((1 << 21) + 400, [1 << 20, 1 << 21])])
def test_tall_batched_frame(h, places):
    crop = np.zeros((2 * HALF, W), np.float32)   # dark towards its ends: nothing there, nor in between
    crop[60:-60] = 0.2 + synth.small_blob_frame(7, 2 * HALF - 120, W, n_blobs=14)
    cfg = dog.small_frame_config(max_h=h, max_w=W, blob_cap=1024)
    det = dog.Detector(cfg)
    want = _sorted(*det.detect(torch.from_numpy(crop).cuda())[0].to_numpy())
    assert len(want[0]) >= 5
    tall = torch.zeros((h, W), dtype=torch.float32, device="cuda")
    for y in places:
        tall[y - HALF:y + HALF] = torch.from_numpy(crop).cuda()
    # small frames after it, so that it is not split into finer bands for the last wave
    frames = [tall] + [torch.zeros((8, 8), device="cuda") for _ in range(200)]
    out, counts, _ = det.detect_batched(frames)
    torch.cuda.synchronize()
    assert det.status() == 0 and int(counts[1:].max()) == 0
    x, y, l, s, r = _sorted(*dog.blobs_from_raw(out, int(counts[0])))
    assert len(x) == len(places) * len(want[0])
    for k, at in enumerate(sorted(places)):
        part = slice(k * len(want[0]), (k + 1) * len(want[0]))
        for got, w in zip((x, y - (at - HALF), l, s, r), want):
            assert np.array_equal(got[part], w)
