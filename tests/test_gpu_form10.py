"""The 10-warp form of the fused kernel (ladders whose 12-warp form does not fit
the shared memory) at the edges of its 80-row blocks: responses, and so
candidates, bit for bit those of the 8-warp form."""
import numpy as np
import pytest
import torch

from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog, synth

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
