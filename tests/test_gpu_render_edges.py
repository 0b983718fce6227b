"""Rendered counts where single precision cannot decide them, and tiles cut at
every side, against the CPU restatement bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("h,w,n,bg,gain,rn", [
    (31, 33, 9, 0.05, 2000.0, 4.0), (32, 15, 3, 0.05, 2000.0, 4.0), (1, 65, 5, 0.1, 3.7, 0.0),
    (34, 17, 400, 0.02, 900.0, 4.0),          # more spheres than one scan of the table
    (64, 64, 0, 0.0, 4096.0, 0.0),            # every value exactly on an edge (0.5 above a whole number)
    (64, 64, 0, 0.25, 1.0e-3, 0.0), (64, 64, 0, 1.0, 4000.5, 1.0e-6), (64, 64, 4, 0.5, 1.0e30, 2.0),
    (64, 64, 0, 0.5, 5.0, 3000.0),            # clipped at both ends
])
def test_counts_at_rounding_edges(h, w, n, bg, gain, rn):
    table = synth.sphere_table(synth.SPHERE_SEED_BASE + h * w, n=n, h=h, w=w, r_range=(1.0, 9.0))
    counts, inten = dog.render_spheres(torch.from_numpy(table).cuda(), h, w, ss=4, background=bg, gain=gain,
                                       read_noise=rn, seed=h + w, with_intensity=True)
    torch.cuda.synchronize()
    want_i, want_c = oracle.render_spheres(table, h, w, ss=4, background=bg, gain=gain, read_noise=rn, seed=h + w)
    assert np.array_equal(inten.cpu().numpy().view(np.uint32), want_i.view(np.uint32))
    assert np.array_equal(counts.cpu().numpy().view(np.uint16), want_c)


@pytest.mark.parametrize("spheres", [
    [(20.0, 30.0, -6.0, 0.7), (50.0, 10.0, -2.5, 0.4)],          # the radius enters squared
    [(3.0e7, 20.0, 3.0e7, 0.5), (40.0, -9.0e6, 9.0e6, 0.3)],     # an edge that single precision blurs over pixels
    [(20.0, 20.0, 5.0, float("inf"))],                           # inf * 0 outside the disc
    [(20.0, 20.0, float("nan"), 0.5), (float("nan"), 3.0, 4.0, 0.5), (30.0, 40.0, 0.0, 0.5)],
])
def test_spheres_out_of_the_ordinary(spheres):
    """The sum over all spheres as written, whatever tile or block a pixel is in."""
    table = np.array(spheres + [(33.0, 33.0, 7.0, 0.25)], np.float32)
    counts, inten = dog.render_spheres(torch.from_numpy(table).cuda(), 70, 80, ss=2, seed=5, with_intensity=True)
    torch.cuda.synchronize()
    want_i, want_c = oracle.render_spheres(table, 70, 80, ss=2, background=0.05, gain=2000.0, read_noise=4.0, seed=5)
    got_i = inten.cpu().numpy()
    assert np.array_equal(np.isnan(got_i), np.isnan(want_i))
    ok = ~np.isnan(want_i)
    assert np.array_equal(got_i[ok].view(np.uint32), want_i[ok].view(np.uint32))
    assert np.array_equal(counts.cpu().numpy().view(np.uint16)[ok], want_c[ok])


@pytest.mark.parametrize("gain", [1e-39, 3e-41, 2e-44, 1e-46])
def test_gains_below_single_precision(gain):
    """Bright intensities times a gain that single precision holds in a few bits
    or not at all, with sums of all sizes around a rounding edge."""
    table = np.zeros((0, 4), np.float32)
    bg = float(np.float32(min(40.0 / gain, 3.0e38)))   # 40 photons where a float can be that bright
    counts = dog.render_spheres(torch.from_numpy(table).cuda(), 300, 400, ss=1, background=bg, gain=gain,
                                read_noise=0.25, seed=3)
    torch.cuda.synchronize()
    _, want = oracle.render_spheres(table, 300, 400, ss=1, background=bg, gain=gain, read_noise=0.25, seed=3)
    assert np.array_equal(counts.cpu().numpy().view(np.uint16), want)


@pytest.mark.parametrize("h,w", [(639, 1000), (641, 1000), (1279, 1000), (1300, 1025)])
def test_frames_around_a_change_of_the_grid(h, w):
    """20, 21, 40 and 41 by 32 or 33 tiles: four, two, two and one CTA to a tile."""
    table = synth.sphere_table(synth.SPHERE_SEED_BASE + h, n=40, h=h, w=w, r_range=(3.0, 30.0))
    counts, inten = dog.render_spheres(torch.from_numpy(table).cuda(), h, w, ss=2, seed=h, with_intensity=True)
    torch.cuda.synchronize()
    want_i, want_c = oracle.render_spheres(table, h, w, ss=2, background=0.05, gain=2000.0, read_noise=4.0, seed=h)
    assert np.array_equal(inten.cpu().numpy().view(np.uint32), want_i.view(np.uint32))
    assert np.array_equal(counts.cpu().numpy().view(np.uint16), want_c)
