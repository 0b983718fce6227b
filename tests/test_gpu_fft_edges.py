"""The FFT backend's test kernel at its tile edges: a warp takes 30 columns by
four rows, a block eight warps.  Same rule and margin as the other FFT tests
(|D - D_oracle| <= 1e-5 * c_i * max|I|, candidates on every decidable voxel)."""
import pytest

from paper_2010_08486_gb300 import _lib
from paper_2010_08486_gb300 import build as libbuild
from paper_2010_08486_gb300 import dog, synth
from tests.test_gpu_fft import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("shape", [(32, 30), (33, 31), (4, 60), (5, 61), (31, 32), (1, 90), (64, 29), (65, 91), (3, 1)])
def test_tile_edges(shape):
    h, w = shape
    img = synth.small_blob_frame(11, h, w, n_blobs=3)
    _check(dog.small_frame_config(backend=_lib.BACKEND_FFT, max_h=h, max_w=w), img, name="edge_%dx%d" % shape)
