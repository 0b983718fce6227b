"""The 10-warp form of the fused kernel (ladders whose 12-warp form does not fit
the shared memory) at the edges of its 80-row blocks: responses, and so
candidates, bit for bit those of the 8-warp form."""
import numpy as np
import pytest
import torch

from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import autotune, dog, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("h,w", [(1, 33), (79, 64), (80, 65), (81, 31), (160, 97), (243, 40)])
def test_equals_eight_warp_form(h, w):
    img = torch.from_numpy(synth.small_blob_frame(3, h, w, n_blobs=6)).cuda()
    cfg = dog.small_frame_config(min_sigma=2.0, max_sigma=2.0 * 1.15 ** 13, ratio=1.15, n_levels=14, threshold=0.01,
                                 max_h=h, max_w=w)
    got = []
    for warps in (0, 8):
        det = dog.Detector(cfg)
        if warps:
            det.set_producer_warps(warps)
        D = det.debug_dog(img)
        cand = det.candidates(img)
        torch.cuda.synchronize()
        x, y, l, _, r = cand.to_numpy()
        order = np.lexsort((x, y, l))
        got.append((D, np.stack([x, y, l])[:, order], r[order]))
    assert torch.equal(got[0][0], got[1][0])
    assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][2], got[1][2])


def _form(det, img):
    """The fused kernel's instance (its number of warps first) that a call runs."""
    for _ in range(4):   # (a process's first trace may come back empty)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            det.candidates(img)
            torch.cuda.synchronize()
        names = [e.key for e in prof.key_averages() if "dog_fused_kernel" in e.key]
        if names:
            break
    assert len(names) == 1
    return names[0]


@pytest.mark.parametrize("cfg", [dog.small_frame_config(max_h=96, max_w=64), dog.plif_config(max_h=96, max_w=64),
                                 dog.small_frame_config(min_sigma=2.0, ratio=1.15, n_levels=14, max_h=96, max_w=64)])
def test_setting_the_reported_warps_changes_nothing(cfg):
    img = torch.from_numpy(synth.small_blob_frame(3, 96, 64, n_blobs=6)).cuda()
    det = dog.Detector(cfg)
    own, before = det.producer_warps, _form(det, img)
    det.set_producer_warps(own)
    assert det.producer_warps == own and _form(det, img) == before
    measure = autotune.frame_measure(det, img, reps=1)   # times 12 and 8, leaves the handle as it was
    measure(0, 1, 12), measure(0, 1, 8)
    assert det.producer_warps == own and _form(det, img) == before
    det.set_producer_warps(20 - own)   # the other one is a bound
    assert det.producer_warps == 20 - own
    after = _form(det, img)
    assert "<8," in after if own == 12 else after == before
