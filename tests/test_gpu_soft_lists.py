"""Soft backward from recorded maxima where its lists and tiles can go wrong:
frames narrower than the kernels (repeated mirror images), tile and cell edges,
frames too dense in maxima for the lists, and batches.  Against the FP64 oracle
with the tolerances of the other soft gradient tests (relative L2 1e-4), against
the recomputing backward (1e-5), or exactly where only the launch differs."""
import numpy as np
import pytest
import torch

import oracle
from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import _lib, dog, synth
from tests.test_gpu_soft import check_record_mask, setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


def _frame(h, w, seed=0):
    return synth.plif_frame(synth.GRAD_SEED_BASE + seed)[300:300 + h, 400:400 + w].copy()


def _flat_block(h, w):
    """Zeros but for noise along one edge: every voxel of the inside ties."""
    img = np.zeros((h, w), np.float32)
    img[:9] = _frame(9, w)
    return img


@pytest.mark.parametrize("shape", [(40, 7), (20, 150), (31, 33), (64, 65), (97, 40)])
def test_backward_from_record_small_frames(shape):
    img = _frame(*shape)
    cfg, det, p, sig0, sig = setup(img)
    t, s = torch.from_numpy(img).cuda(), torch.from_numpy(sig).cuda()
    rad = np.asarray(det.radii)
    rec = dog.SoftMaxima(1 << 16, "cuda")
    det.soft_hist(t, s, rec=rec)
    mask = check_record_mask(rec, img, sig, rad, p)
    Ho = oracle.soft_hist(img.astype(np.float64), sig.astype(np.float64), rad, p, sig0, mask)
    gH = (2.0 * (Ho - 0.5 * Ho.mean())).astype(np.float32)
    gi, gs = det.backward(t, s, torch.from_numpy(gH).cuda(), rec=rec)
    assert det.status() == 0
    oi, osg = oracle.soft_grad(img.astype(np.float64), sig.astype(np.float64), rad, p, sig0, gH.astype(np.float64),
                               mask)
    assert np.linalg.norm(gi.cpu().numpy() - oi) <= 1e-4 * np.linalg.norm(oi)
    assert np.linalg.norm(gs.cpu().numpy() - osg) <= 1e-4 * np.linalg.norm(osg)


def _grads(det, frames, s, gH, cap):
    """The batch call on its own forward's record; also the counts."""
    n, h, w = frames.shape
    buf = torch.empty((n, cap, 6), dtype=torch.int32, device="cuda")
    counts = torch.zeros(n, dtype=torch.int32, device="cuda")
    hist = torch.zeros(det.cfg.nbins, device="cuda")
    gi, gs = torch.empty_like(frames), torch.zeros(det.K, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    args = (det.h, frames.data_ptr(), n, h * w, h, w, w, s.data_ptr())
    assert det.lib.dog_soft_hist_batched(*args, hist.data_ptr(), buf.data_ptr(), cap, counts.data_ptr(), st) == 0
    assert det.lib.dog_backward_rec_batched(*args, buf.data_ptr(), counts.data_ptr(), cap, gH.data_ptr(),
                                            gi.data_ptr(), gs.data_ptr(), st) == 0
    return hist, gi, gs, counts


@pytest.mark.parametrize("kinds", ["n", "nn", "fn", "nfnf", "n" * 66])
@pytest.mark.parametrize("shape", [(150, 173)])
def test_batch_equals_single_frames(shape, kinds):
    """n: noise; f: flat (the dense form).  Listed frames are summed in the
    same order alone and in a batch; flat ones against the recomputing path."""
    imgs = [_frame(*shape, seed=i % 5) if k == "n" else _flat_block(*shape) for i, k in enumerate(kinds)]
    cfg, det, p, sig0, sig = setup(imgs[0])
    frames, s = torch.from_numpy(np.stack(imgs)).cuda(), torch.from_numpy(sig).cuda()
    gH = torch.linspace(-1.0, 2.0, cfg.nbins, device="cuda")
    hist, gi, gs, counts = _grads(det, frames, s, gH, 1 << 18)
    want_h, want_s = torch.zeros_like(hist), torch.zeros_like(gs)
    for b, k in enumerate(kinds):
        rec = dog.SoftMaxima(1 << 18, "cuda")
        det.soft_hist(frames[b], s, out=want_h, rec=rec)
        assert int(counts[b]) == int(rec.count) <= rec.cap
        if k == "n":
            one, _ = det.backward(frames[b], s, gH, grad_sigmas=want_s, rec=rec)
            assert torch.equal(gi[b], one)
        plain, _ = det.backward(frames[b], s, gH, grad_sigmas=want_s if k == "f" else None)
        assert torch.linalg.norm(gi[b] - plain) <= 1e-5 * torch.linalg.norm(plain)
    assert det.status() == 0
    torch.testing.assert_close(hist, want_h, rtol=1e-5, atol=1e-5)
    assert torch.linalg.norm(gs - want_s) <= 1e-4 * torch.linalg.norm(want_s)


def test_batch_replays_in_a_graph():
    """Captured before the lists have grown to the batch: several passes."""
    imgs = np.stack([_frame(120, 130, seed=i) for i in range(3)])
    cfg, det, p, sig0, sig = setup(imgs[0])
    frames, s = torch.from_numpy(imgs).cuda(), torch.from_numpy(sig).cuda()
    gH = torch.linspace(-1.0, 2.0, cfg.nbins, device="cuda")
    _grads(det, frames[:1], s, gH, 1 << 16)   # workspace of one frame
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _, gi, gs, _ = _grads(det, frames, s, gH, 1 << 16)
    g.replay()
    torch.cuda.synchronize()
    _, want_i, want_s, _ = _grads(det, frames, s, gH, 1 << 16)
    assert torch.equal(gi, want_i) and det.status() == 0
    torch.testing.assert_close(gs, want_s, rtol=1e-6, atol=0)


def test_tiles_reached_by_too_many_pairs():
    """A bump on every second pixel of every second row: 16 maxima in a cell of
    8 x 8, which the lists hold, and up to 790 pairs to a tile, which the tiles
    do not (those of the right edge do, with 150): some CTAs of a frame ask for
    the dense form while others are at work, beside frames that need none."""
    shape, n = (160, 200), 9
    bumps = np.zeros(shape, np.float32)
    bumps[::2, ::2] = 0.5
    imgs = [_frame(*shape, seed=i) + (i % 3 != 1) * bumps for i in range(n)]
    cfg, det, p, sig0, sig = setup(imgs[0])
    frames, s = torch.from_numpy(np.stack(imgs)).cuda(), torch.from_numpy(sig).cuda()
    gH = torch.linspace(-1.0, 2.0, cfg.nbins, device="cuda")
    _, gi, gs, counts = _grads(det, frames, s, gH, 1 << 14)
    assert int(counts.max()) <= 1 << 14 and det.status() == 0
    want_s = torch.zeros_like(gs)
    for b in range(n):
        plain, _ = det.backward(frames[b], s, gH, grad_sigmas=want_s)
        assert torch.linalg.norm(gi[b] - plain) <= 1e-5 * torch.linalg.norm(plain)
    assert torch.linalg.norm(gs - want_s) <= 1e-4 * torch.linalg.norm(want_s)


def test_a_graph_outlives_the_growth_of_the_lists():
    """A graph captured on the lists of its time replays after larger batches of
    the same frames have replaced them, twice, with other work between; the
    memory that the graph works on is not handed out again."""
    imgs = np.stack([_frame(120, 130, seed=i) for i in range(5)])
    cfg, det, p, sig0, sig = setup(imgs[0])
    frames, s = torch.from_numpy(imgs).cuda(), torch.from_numpy(sig).cuda()
    gH = torch.linspace(-1.0, 2.0, cfg.nbins, device="cuda")
    _grads(det, frames[:1], s, gH, 1 << 16)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _, gi, gs, _ = _grads(det, frames[:2], s, gH, 1 << 16)
    g.replay()
    torch.cuda.synchronize()
    want_i, want_s = gi.clone(), gs.clone()
    for n in (2, 5):
        gi.zero_()
        _, eager, _, _ = _grads(det, frames[:n], s, gH, 1 << 16)
        gs.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(gi, want_i) and torch.equal(eager[:2], want_i) and det.status() == 0
        torch.testing.assert_close(gs, want_s, rtol=1e-6, atol=0)


def test_a_wait_that_runs_out_is_reported():
    """The dense form's CTAs give up at once instead of waiting for one another:
    the status says so and the frame that wanted the form has no half-made
    gradient; the frame beside it and the next call are whole."""
    imgs = [_frame(150, 173), _flat_block(150, 173)]
    cfg, det, p, sig0, sig = setup(imgs[0])
    frames, s = torch.from_numpy(np.stack(imgs)).cuda(), torch.from_numpy(sig).cuda()
    gH = torch.linspace(-1.0, 2.0, cfg.nbins, device="cuda")
    _, want, _, _ = _grads(det, frames, s, gH, 1 << 18)
    assert det.status() == 0
    assert det.lib.dog_test_wait_limit(det.h, 0) == 0
    _, gi, _, _ = _grads(det, frames, s, gH, 1 << 18)
    assert det.status() == _lib.DOG_ERR_TIMEOUT
    assert torch.equal(gi[0], want[0]) and bool(gi[1].isnan().any())
    assert det.lib.dog_test_wait_limit(det.h, -1) == 0
    _, gi, _, _ = _grads(det, frames, s, gH, 1 << 18)
    assert det.status() == 0 and torch.equal(gi[0], want[0])
    assert torch.linalg.norm(gi[1] - want[1]) <= 1e-5 * torch.linalg.norm(want[1])
