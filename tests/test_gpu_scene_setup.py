"""What snerg_create builds from an indirection grid and an atlas, read back and compared with
numpy on every block edge: the per-octant block and voxel distance maps and the apron-padded
atlas. Densities are sparse and random (single voxels, empty blocks, an unreferenced slot), the
grids have edges on both sides of the block-map kernel's 32- and 64-block limits and block
counts that do not fill the last thread block. The workspace layout is described in
test_gpu_distance_maps.py; the padded atlas follows the distance planes."""
import numpy as np
import pytest
import torch

from paper_2103_14645_gb300 import renderer

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _align(v):
    return (v + 255) & ~255


def _cone_distance(occ, octant, cap):
    """min(cap, Chebyshev distance to the nearest set cell of the cone), occ [..., n, n, n] (z, y, x)."""
    D = np.where(occ, 0, cap).astype(np.int32)
    n = occ.shape[-1]
    for bit, axis in ((0, -1), (1, -2), (2, -3)):
        src = np.moveaxis(D, axis, -1)
        if (octant >> bit) & 1:
            src = src[..., ::-1]
        out = src.copy()
        for d in range(1, min(n, cap)):
            out[..., :n - d] = np.minimum(out[..., :n - d], np.maximum(d, src[..., d:]))
        if (octant >> bit) & 1:
            out = out[..., ::-1]
        D = np.moveaxis(out, -1, axis)
    return D


@pytest.mark.parametrize("G,B,p_block,shift", [(9, 2, 0.3, 0), (5, 4, 0.4, 0), (7, 8, 0.2, 0), (5, 16, 0.3, 0),
                                               (3, 32, 0.6, 0), (1, 32, 1.0, 0), (3, 64, 0.3, 1), (33, 4, 0.01, 0),
                                               (64, 2, 0.003, 1), (65, 2, 0.002, 0)])
def test_workspace_matches_numpy(G, B, p_block, shift):
    rng = np.random.default_rng(100 * G + B)
    N, P, cells = G * B, B + 2, G ** 3
    occupied = np.sort(rng.choice(cells, max(1, int(round(p_block * cells))), replace=False))
    nb = len(occupied) + 1                                     # one slot is not referenced
    slots = rng.permutation(nb)[:len(occupied)]
    ind = np.full(cells, -1, np.int32)
    ind[occupied] = slots
    ind = ind.reshape(G, G, G)
    atlas = rng.integers(0, 256, (nb, B, B, B, 8), dtype=np.uint8)
    density = rng.uniform(size=(nb, B, B, B)) < rng.choice([0.0, 2.0 / B ** 3, 0.02, 0.3, 0.98], nb)[:, None, None, None]
    atlas[..., 0] *= density
    # an atlas that is 8-byte aligned and no more
    buf = torch.zeros(atlas.size + 8 * shift, dtype=torch.uint8, device=DEV)
    t_atlas = buf[8 * shift:].view(atlas.shape)
    t_atlas.copy_(torch.from_numpy(atlas))
    r = renderer.Renderer(N, B, (-1.0, -1.0, -1.0), 2.0, 5.0, (1.0, 1.0, 1.0), torch.from_numpy(ind).to(DEV), t_atlas)
    ws = r.workspace.cpu().numpy()
    o_ind = 256
    o_blk = _align(_align(_align(o_ind + 8 * cells * 4) + cells) + 2 * cells)
    o_vskip = _align(o_blk + nb * 4)
    o_pad = _align(o_vskip + 8 * nb * P ** 3)
    got_ind = ws[o_ind:o_ind + 8 * cells * 4].view(np.int32).reshape(8, G, G, G)
    got_skip = ws[o_vskip:o_vskip + 8 * nb * P ** 3].reshape(8, nb, P, P, P)
    got_pad = ws[o_pad:o_pad + nb * P ** 3 * 8].reshape(nb, P, P, P, 8)
    for o in range(8):
        want = np.where(ind >= 0, ind, -np.maximum(_cone_distance(ind >= 0, o, 32), 1))
        np.testing.assert_array_equal(got_ind[o], want, err_msg=f"block map, octant {o}")
    dense = np.zeros((G, B, G, B, G, B, 8), np.uint8)
    z, y, x = np.nonzero(ind >= 0)
    for k in range(len(z)):
        dense[z[k], :, y[k], :, x[k]] = atlas[ind[z[k], y[k], x[k]]]
    padded = np.pad(dense.reshape(N, N, N, 8), ((1, 1), (1, 1), (1, 1), (0, 0)), mode="edge")
    set_ = atlas[..., 0] != 0
    want_skip = np.stack([_cone_distance(set_, o, 255) for o in range(8)])
    for k in range(len(z)):
        b, s = (z[k], y[k], x[k]), ind[z[k], y[k], x[k]]
        lo = [i * B for i in b]
        want = padded[lo[0]:lo[0] + P, lo[1]:lo[1] + P, lo[2]:lo[2] + P]
        np.testing.assert_array_equal(got_pad[s], want, err_msg=f"padded atlas, block {b}")
        # apron cells outside the grid repeat the voxel that they clamp to, the others hold 255
        plane = np.pad(want_skip[:, s], ((0, 0), (1, 1), (1, 1), (1, 1)), mode="edge")
        for a in range(3):
            for face, at_border in ((0, b[a] == 0), (P - 1, b[a] == G - 1)):
                if not at_border:
                    np.moveaxis(plane, a + 1, 0)[face] = 255
        np.testing.assert_array_equal(got_skip[:, s], plane, err_msg=f"distance planes, block {b}")
    unused = [s for s in range(nb) if s not in set(slots.tolist())]
    assert (got_pad[unused] == 0).all()
    r.close()
