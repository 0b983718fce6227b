"""Pruning of given candidate lists against the oracle's greedy pruning: list
lengths around the shared-memory limit, sparse lists, lists so dense that the
conflict list overflows, and equal responses."""
import numpy as np
import pytest
import torch

import oracle
from paper_2010_08486_gb300 import _lib, build as libbuild, dog
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    libbuild.build()


@pytest.mark.parametrize("mode", [_lib.PRUNE_COALESCE, _lib.PRUNE_SUPPRESS])
@pytest.mark.parametrize("n,size", [(0, 9), (1, 9), (33, 40), (900, 24), (1500, 300), (3000, 150), (4095, 2000),
                                    (4096, 900), (4097, 900)])
def test_prune_of_a_list(n, size, mode):
    rng = np.random.default_rng(1000 * n + size)
    cfg = dog.plif_config(max_h=2048, max_w=2048, blob_cap=8192, prune=mode)
    det = dog.Detector(cfg)
    # distinct (x, y, level), in any order; responses in few values, so that ties are many
    cells = rng.choice(size * size * det.P, size=n, replace=False)
    level, pos = cells % det.P, cells // det.P
    x, y = pos % size, pos // size
    resp = (rng.integers(1, 40, n) / 64.0).astype(np.float32)
    sig = np.asarray(det.sigmas, np.float32)[level]
    raw = np.zeros((8192, 5), np.int32)
    raw[:n, 0], raw[:n, 1], raw[:n, 2] = x, y, level
    raw[:n, 3], raw[:n, 4] = sig.view(np.int32), resp.view(np.int32)
    cand = dog.BlobList(torch.from_numpy(raw).cuda(), torch.tensor(n, dtype=torch.int32, device="cuda"))
    out = det.prune(cand, 2048, 2048)
    torch.cuda.synchronize()
    want = oracle.prune(parity.blobs_to_oracle(x, y, level, sig, resp), parity.oracle_params(cfg))
    want.sigma = want.sigma.astype(np.float32).astype(np.float64)
    assert parity.same_blob_sets(parity.blobs_to_oracle(*out.to_numpy()), want)
    assert det.status() == 0


def test_candidates_far_apart():
    """A grid that spans the frame has cells of tens of thousands of rows here:
    candidates 2^16 rows apart, whose squared distance is 0 in 32 bits, do not
    conflict; close ones at the far end do."""
    h = 60_000_001
    cfg = dog.small_frame_config(max_h=64, max_w=64, blob_cap=64)
    det = dog.Detector(cfg)
    y = np.array([0, 65536, 131072, 30_000_000, 30_065_536, h - 1, h - 2], np.int32)
    x = np.array([3, 3, 3, 5, 5, 9, 9], np.int32)
    level = np.full(7, 2, np.int32)
    resp = (np.arange(1, 8) / 8.0).astype(np.float32)
    sig = np.asarray(det.sigmas, np.float32)[level]
    raw = np.zeros((64, 5), np.int32)
    raw[:7] = np.stack([x, y, level, sig.view(np.int32), resp.view(np.int32)], 1)
    cand = dog.BlobList(torch.from_numpy(raw).cuda(), torch.tensor(7, dtype=torch.int32, device="cuda"))
    out = det.prune(cand, h, 16)
    torch.cuda.synchronize()
    got = out.to_numpy()
    assert sorted(got[1].tolist()) == [0, 65536, 131072, 30_000_000, 30_065_536, h - 2] and det.status() == 0


@pytest.mark.parametrize("n", [5872, 5873, 9396, 9397, 23490, 23491, 46981])
def test_lists_at_the_sizes_of_the_shared_memory(n):
    """The largest lists of which the candidates and all arrays, the candidates,
    and two arrays fit the shared memory, and one more; and none of them."""
    rng = np.random.default_rng(n)
    size, cap = 1200, 65536
    cfg = dog.plif_config(max_h=2048, max_w=2048, blob_cap=cap)
    det = dog.Detector(cfg)
    cells = rng.choice(size * size * 8, size=n, replace=False)
    level, pos = cells % 8, cells // 8
    x, y = pos % size, pos // size
    resp = (rng.integers(1, 4000, n) / 4096.0).astype(np.float32)
    sig = np.asarray(det.sigmas, np.float32)[level]
    raw = np.zeros((cap, 5), np.int32)
    raw[:n, 0], raw[:n, 1], raw[:n, 2] = x, y, level
    raw[:n, 3], raw[:n, 4] = sig.view(np.int32), resp.view(np.int32)
    cand = dog.BlobList(torch.from_numpy(raw).cuda(), torch.tensor(n, dtype=torch.int32, device="cuda"))
    out = det.prune(cand, 2048, 2048)
    torch.cuda.synchronize()
    want = oracle.prune(parity.blobs_to_oracle(x, y, level, sig, resp), parity.oracle_params(cfg))
    want.sigma = want.sigma.astype(np.float32).astype(np.float64)
    assert parity.same_blob_sets(parity.blobs_to_oracle(*out.to_numpy()), want)
    assert det.status() == 0
