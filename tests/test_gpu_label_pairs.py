"""Words with the most pairs of touching runs (k_union lists a word's pairs
before it makes the unions): every second voxel of each row, the rows against
one another in or out of step, so that a run touches two runs of a row before
it, across word boundaries and up to the grid's ends, in whole and partial
words.  Labels, counts and boxes against the oracle's flood fill."""
import numpy as np
import pytest
import torch

from oracle import Oracle
from tests.test_gpu_ccl_stress import check_reconstruct_labeller, grid_rig, grid_words, make_lib_rig, oracle_labels

pytestmark = pytest.mark.gpu


def stripes(dims, phase, gap):
    """Voxels with (x + phase * (y + z)) even, but none in every gap-th plane."""
    nx, ny, nz = dims
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx]
    return ((x + phase * (y + z)) % 2 == 0) & ((z % gap != gap - 1) | (y % 5 == 0))


@pytest.mark.parametrize("dims", [(64, 12, 9), (33, 9, 7), (31, 5, 6), (97, 3, 4)])
@pytest.mark.parametrize("phase", [0, 1])
@pytest.mark.parametrize("gap", [2, 3])
def test_words_with_the_most_pairs(dims, phase, gap):
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA GPU"
    from paper_1903_11785_gb300 import fvv
    occ = stripes(dims, phase, gap)
    rig = grid_rig(dims, t_np=2)
    ref_lab, n_comp, rois = oracle_labels(rig, occ)
    assert Oracle(rig).ccl_uf(occ)[1] == n_comp > 0
    r = make_lib_rig(fvv, rig, rois)
    try:
        for _ in range(5):
            check_reconstruct_labeller(fvv, r, grid_words(occ, junk_past_nx=True), ref_lab, n_comp, rois,
                                       int(occ.sum()))
    finally:
        r.close()
