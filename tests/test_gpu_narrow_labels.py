"""The allocation-free labelling of grids of one to five voxels in x, whose words
are taken several at a time up to four voxels (and one at a time from five on): single
rows and planes, grids of a few words and of more words than a sweep of the launch
takes, bits past nx set, sparse and dense; labels and counts against scipy's
26-connected components numbered by their first voxel."""
import numpy as np
import pytest
import torch
from scipy import ndimage

from tests.test_gpu_ccl_stress import grid_words, run_noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300.build import build
    build()


def _reference(occ, t_np):
    lab, n = ndimage.label(occ, np.ones((3, 3, 3), int))
    size = np.bincount(lab.ravel(), minlength=n + 1)
    first = np.full(n + 1, occ.size, np.int64)
    np.minimum.at(first, lab.ravel(), np.arange(occ.size))
    kept = [k for k in np.argsort(first[1:], kind="stable") + 1 if size[k] >= t_np]
    new = np.zeros(n + 1, np.int32)
    new[kept] = np.arange(1, len(kept) + 1)
    return new[lab], n, len(kept)


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("ny,nz,density", [(1, 1, 1.0), (1, 40, 0.5), (33, 1, 0.4), (7, 9, 0.5), (97, 63, 0.12),
                                           (61, 130, 0.9), (1000, 640, 0.008)])
def test_narrow_grids(nx, ny, nz, density):
    from paper_1903_11785_gb300 import fvv
    rng = np.random.default_rng([nx, ny, nz])
    occ = rng.random((nz, ny, nx)) < (density if nx * ny * nz < 10 ** 6 else 0.0025)
    if ny == 1000:                       # more than 2048 blocks x 256 words; one component through them all
        occ[:, ny // 2, nx // 2] = True
    words = grid_words(occ, junk_past_nx=True)
    for t_np in (1, 3):
        ref, n, kept = _reference(occ, t_np)
        assert n <= 8192
        lab, counts = run_noalloc(fvv, words, (nx, ny, nz), t_np, 2 ** 31 - 1, fill=7)
        assert [int(c) for c in counts] == [n, kept, 0]
        assert np.array_equal(np.asarray(lab).reshape(occ.shape), ref)
