"""The fused kernel at the edges of its blocks and forms: heights around
multiples of a block's rows, ladders that only the small forms hold, and frames
with non-finite pixels, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog, synth
from tests.test_gpu_detect import dev, full_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("warps", [8, 12])
@pytest.mark.parametrize("h", [63, 64, 65, 95, 96, 97, 129, 193])
def test_heights_around_a_block(h, warps):
    cfg = dog.plif_config(max_h=h, max_w=40)
    det = dog.Detector(cfg)
    det.set_producer_warps(warps)
    full_check(cfg, synth.plif_frame(synth.PLIF_SEED_BASE + h, h, 40), det=det)
    det.set_tiling(56)   # bands whose rows end inside a block, and a short last one
    full_check(cfg, synth.plif_frame(synth.PLIF_SEED_BASE + h, h, 40), det=det)


# radii that leave room for four warps, and for three (odd and even ladders)
@pytest.mark.parametrize("radii", [[54, 54, 54, 54, 55, 55, 55, 55, 55, 55],
                                   [48, 49, 50, 52, 53, 54, 56, 57, 58, 59, 61]])
def test_ladders_of_the_small_forms(radii):
    sig = [(r + 0.02 * i) / 4.0 for i, r in enumerate(radii)]
    cfg = dog.DetectorConfig(sigmas=sig, threshold=0.02, max_h=150, max_w=70, norm=1)
    det = dog.Detector(cfg)
    assert det.radii == radii
    full_check(cfg, synth.plif_frame(synth.PLIF_SEED_BASE + 3, 150, 70), det=det)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("at", [(70, 40), (3, 31), (139, 0)])
def test_non_finite_pixel_reaches_each_level_by_its_own_radius(bad, at):
    """A plane's response is non-finite within the radius of its wider level
    around the pixel (in both axes) and elsewhere bit for bit that of the frame
    without it, whichever levels are blurred together."""
    h, w = 140, 96
    cfg = dog.plif_config(max_h=h, max_w=w)
    det = dog.Detector(cfg)
    clean = synth.plif_frame(synth.PLIF_SEED_BASE + 5, h, w)
    img = clean.copy()
    img[at] = bad
    D0 = det.debug_dog(dev(clean)).cpu().numpy()
    D1 = det.debug_dog(dev(img)).cpu().numpy()
    dy = np.abs(np.arange(h) - at[0])[:, None]
    dx = np.abs(np.arange(w) - at[1])[None, :]
    for l in range(det.P):
        r = det.radii[l + 1]
        near = (dy <= r) & (dx <= r)
        assert not np.isfinite(D1[l][near]).any()
        np.testing.assert_array_equal(D1[l][~near], D0[l][~near])
    blobs, hist, _ = det.detect(dev(img))
    torch.cuda.synchronize()
    assert det.status() == 0 and int(hist.sum()) == blobs.n()


# ladders at the limit of the shared memory that three warps no longer hold; the
# first needs the most of all that were found
@pytest.mark.parametrize("radii", [[12, 12, 45, 46, 53, 53, 53, 55, 61, 61, 63],
                                   [12, 13, 42, 42, 54, 54, 57, 58, 61, 61, 63],
                                   [44, 45, 48, 49, 55, 55, 57, 59, 61, 61, 62],
                                   [48, 49, 50, 50, 53, 55, 58, 59, 59, 60, 61],
                                   [44, 45, 50, 50, 51, 56, 57, 58, 62, 62, 62]])
def test_ladders_of_the_smallest_form(radii):
    sig = [(r + 0.02 * i) / 4.0 for i, r in enumerate(radii)]
    cfg = dog.DetectorConfig(sigmas=sig, threshold=0.02, max_h=150, max_w=70, norm=1)
    det = dog.Detector(cfg)
    assert det.radii == radii
    img = synth.plif_frame(synth.PLIF_SEED_BASE + 3, 150, 70)
    full_check(cfg, img, det=det)
    # the batched and the differentiable calls hold them too
    single = det.detect(dev(img))
    out, counts, hists = det.detect_batched([dev(img)])
    assert int(counts[0]) == single[0].n() and torch.equal(hists[0], single[1])
    s = torch.tensor(sig, dtype=torch.float32, device="cuda")
    rec = dog.SoftMaxima(1 << 16, "cuda")
    H = det.soft_hist(dev(img), s, rec=rec)
    gi, gs = det.backward(dev(img), s, torch.ones_like(H), rec=rec)
    gi2, gs2 = det.backward(dev(img), s, torch.ones_like(H))
    assert 0 < int(rec.count) <= rec.cap and det.status() == 0
    assert torch.linalg.norm(gi - gi2) <= 1e-5 * torch.linalg.norm(gi2)
    assert torch.linalg.norm(gs - gs2) <= 1e-4 * torch.linalg.norm(gs2)


@pytest.mark.parametrize("sig", [[1.6 ** i for i in range(6)], [1.0, 5.0, 5.25, 12.0, 12.02], [0.5, 9.0, 15.0]])
def test_non_finite_pixel_beside_levels_of_very_different_radii(sig):
    """As above where one level of a pair has many taps fewer than the other, whole
    blocks of them, and for the differentiable form's maxima away from the pixel."""
    h, w, at = 190, 100, (97, 33)
    cfg = dog.DetectorConfig(sigmas=sig, threshold=0.02, max_h=h, max_w=w, norm=1)
    det = dog.Detector(cfg)
    clean = synth.plif_frame(synth.PLIF_SEED_BASE + 6, h, w)
    img = clean.copy()
    img[at] = np.inf
    D0, D1 = det.debug_dog(dev(clean)).cpu().numpy(), det.debug_dog(dev(img)).cpu().numpy()
    dy, dx = np.abs(np.arange(h) - at[0])[:, None], np.abs(np.arange(w) - at[1])[None, :]
    for l in range(det.P):
        near = (dy <= det.radii[l + 1]) & (dx <= det.radii[l + 1])
        assert not np.isfinite(D1[l][near]).any() and np.array_equal(D1[l][~near], D0[l][~near])
    s = torch.tensor(sig, dtype=torch.float32, device="cuda")
    sets = []
    for t in (clean, img):
        rec = dog.SoftMaxima(1 << 16, "cuda")
        det.soft_hist(dev(t), s, rec=rec)
        assert int(rec.count) <= rec.cap
        r = rec.buf[:int(rec.count)].cpu().numpy()
        far = np.maximum(np.abs(r[:, 0] - at[1]), np.abs(r[:, 1] - at[0])) > det.radii[-1] + 1
        sets.append({tuple(v) for v in r[far].tolist()})
    assert len(sets[0]) > 3 and sets[0] == sets[1]
