"""Stretch limits where the histogram's units, heads and tails of rows and the
derived last bin can go wrong: exact order statistics of the counts."""
import numpy as np
import pytest
import torch

from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("sat", [0.0, 0.3])
@pytest.mark.parametrize("top", [40, 4095, 60000])
@pytest.mark.parametrize("h,w,pad,skip", [(1, 1, 0, 0), (3, 7, 0, 0), (5, 8, 3, 1), (2, 511, 0, 0), (33, 512, 0, 3),
                                          (19, 513, 6, 5), (300, 1025, 0, 7), (2500, 40, 0, 0)])
def test_limits_are_order_statistics(h, w, pad, skip, top, sat):
    rng = np.random.default_rng(h * 10007 + w)
    v = rng.integers(0, top + 1, size=(h, w + pad)).astype(np.uint16)
    flat = torch.zeros(skip + v.size, dtype=torch.int16, device="cuda")   # rows of any alignment
    flat[skip:] = torch.from_numpy(v.view(np.int16).ravel()).cuda()
    img = flat[skip:].view(h, w + pad)[:, :w]
    s = np.sort(np.minimum(v[:, :w], 4095).ravel())
    k = min(int(np.floor(sat / 2 * s.size)), (s.size - 1) // 2)
    assert dog.stretch_limits(img, sat).tolist() == [s[k], s[s.size - 1 - k]]


@pytest.mark.parametrize("skip", [0, 1, 2, 3])
def test_scratch_of_any_alignment(skip):
    """The caller's scratch is 4096 int32 and nothing more: a part of a larger
    buffer that starts at any of its words."""
    from paper_2010_08486_gb300 import _lib
    v = np.random.default_rng(skip).integers(0, 5000, size=(61, 130)).astype(np.uint16)
    img = torch.from_numpy(v.view(np.int16)).cuda()
    work = torch.full((4096 + 8,), -1, dtype=torch.int32, device="cuda")
    lohi = torch.zeros(4, dtype=torch.int32, device="cuda")
    assert _lib.load().dog_stretch_limits(img.data_ptr(), 61, 130, 130, 0.1, work[skip:].data_ptr(),
                                          lohi[1:].data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    s = np.sort(np.minimum(v, 4095).ravel())
    k = int(np.floor(0.05 * s.size))
    assert lohi.tolist() == [0, s[k], s[s.size - 1 - k], 0]
    assert bool((work[:skip] == -1).all()) and bool((work[skip + 4096:] == -1).all())
