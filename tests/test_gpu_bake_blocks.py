"""The bake's kernels for blocks of 8^3 and more, and the slot numbering over several tiles of
blocks, against the FP64 oracle bake: grids that do not fill the last tile of 4,096 blocks,
items that split a block along each axis (64^3), every remainder of the blob chunks, broad
blobs that all reach every block, alpha codes, and blobs too faint to keep a block. The bands
are those of test_gpu_bake.py: the kernel's factors per axis keep each within its budget."""
import numpy as np
import pytest

import oracle
from paper_2103_14645_gb300 import renderer, synth
from tests.test_gpu_bake import BMIN, DEV, EXTENT, TAU, _check_bake, _compare_blocks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,B,n_blob,std", [(264, 8, 40, (0.03, 0.08)), (136, 8, 1, (0.2, 0.3)), (80, 16, 5, (0.05, 0.1)),
                                            (96, 32, 64, (0.2, 0.5)), (64, 32, 62, (0.1, 0.4)), (192, 64, 6, (0.05, 0.2))])
def test_separable_bake_matches_oracle(N, B, n_blob, std):
    f = synth.analytic_field(N + B, n_blob=n_blob, std=std, peak=(2.0, 60.0))
    _, atl, _, _, ndiff = _check_bake(N, B, 400.0, f)
    assert ndiff <= 1e-4 * atl.size + 2


def test_alpha_codes_of_separable_blocks():
    f = synth.analytic_field(5, n_blob=9, std=(0.05, 0.1), peak=(20.0, 80.0))
    field = renderer.bake_field(f["blobs"], f["colors"], f["jitter"], TAU)
    ind, atl = renderer.bake(96, 32, BMIN, EXTENT, 100.0, field, DEV, flags=renderer.FLAG_ALPHA_ATLAS)
    ind, atl = ind.cpu().numpy(), atl.cpu().numpy()
    blocks = np.flatnonzero((ind >= 0).ravel())
    _, content, raw = oracle.bake_blocks(96, 32, BMIN, EXTENT, 100.0, f["blobs"], f["colors"], f["jitter"], blocks,
                                         alpha_codes=True)
    _compare_blocks(atl[ind.ravel()[blocks]], content, raw)


def test_blobs_below_the_threshold_keep_nothing():
    f = synth.analytic_field(6, n_blob=8, std=(0.1, 0.2), peak=(1.0, 1.0))
    f["blobs"][:, 4] = 0.1 * TAU * 64 / EXTENT / 8            # all together a tenth of sigma_tau
    field = renderer.bake_field(f["blobs"], f["colors"], f["jitter"], TAU)
    ind, atl = renderer.bake(64, 16, BMIN, EXTENT, 10.0, field, DEV)
    assert bool((ind == -1).all()) and atl.shape[0] == 0


def test_atlas_of_a_counted_bake():
    """max_blocks None counts first and then only writes the atlas: the same scene as one call
    with room, for blocks on both sides of 8^3."""
    for N, B in ((64, 4), (64, 8), (96, 32)):
        f = synth.analytic_field(N, n_blob=12, std=(0.05, 0.1), peak=(20.0, 80.0))
        field = renderer.bake_field(f["blobs"], f["colors"], f["jitter"], TAU)
        ind, atl = renderer.bake(N, B, BMIN, EXTENT, 100.0, field, DEV)
        ind1, atl1 = renderer.bake(N, B, BMIN, EXTENT, 100.0, field, DEV, max_blocks=atl.shape[0] + 3)
        assert atl.shape[0] > 0 and bool((ind == ind1).all()) and bool((atl == atl1).all())


@pytest.mark.parametrize("B", [8, 16, 32, 64])
def test_a_blob_narrower_than_any_voxel_adds_nothing(B):
    """A finite blob whose exponent leaves binary32 a voxel away (s = 5e-20: k = 2.9e38) contributes
    exactly 0 between the voxel centres: the codes of the field without it."""
    f = synth.analytic_field(B, n_blob=3, std=(0.3, 0.6), peak=(20.0, 80.0))
    out = []
    for blobs in (f["blobs"], np.concatenate([f["blobs"], [[-1.7031, -1.7011, -1.7057, 5e-20, 10.0]]]).astype(np.float32)):
        field = renderer.bake_field(blobs, f["colors"], f["jitter"], TAU)
        out.append(renderer.bake(B, B, (-2.0,) * 3, 4.0, 100.0, field, DEV))
    (ind, atl), (ind_n, atl_n) = out
    assert bool((ind == ind_n).all()) and bool((atl == atl_n).all())
    assert float((atl[..., 0] > 0).float().mean()) > 0.1
