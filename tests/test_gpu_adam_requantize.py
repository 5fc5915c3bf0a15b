"""snerg_adam_requantize_atlas: the optimiser step and the new codes in one pass over the
values, against the two calls it stands for and the padded atlas that it has to leave behind
(interior, aprons of neighbouring blocks, clamped grid border), for gradients that touch a few
voxels of a few blocks, all of them, or none, over steps whose moments outlive the gradient."""
import numpy as np
import pytest
import torch

import oracle
from paper_2103_14645_gb300 import renderer

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _align(v):
    return (v + 255) & ~255


def _padded(r, ind, atlas):
    """(stored blocks' padded copies in the workspace, what they have to be)"""
    G, B, nb = ind.shape[0], r.B, r.nb
    P, N = B + 2, G * B
    o = _align(_align(_align(256 + 32 * G ** 3) + G ** 3) + 2 * G ** 3)
    o = _align(_align(o + nb * 4) + 8 * nb * P ** 3)
    ws = r.workspace.cpu().numpy()
    got = ws[o:o + nb * P ** 3 * 8].reshape(nb, P, P, P, 8)
    dense = np.zeros((G, B, G, B, G, B, 8), np.uint8)
    for z, y, x in np.argwhere(ind >= 0):
        dense[z, :, y, :, x] = atlas[ind[z, y, x]]
    pad = np.pad(dense.reshape(N, N, N, 8), ((1, 1),) * 3 + ((0, 0),), mode="edge")
    want = np.zeros_like(got)
    for z, y, x in np.argwhere(ind >= 0):
        want[ind[z, y, x]] = pad[z * B:z * B + P, y * B:y * B + P, x * B:x * B + P]
    return got, want


@pytest.mark.parametrize("G,B,touched", [(4, 2, 0.2), (3, 8, 0.01), (2, 32, 0.001), (2, 64, 0.0005), (1, 4, 1.0), (3, 4, 0.0)])
def test_one_pass_matches_the_two_calls(G, B, touched):
    rng = np.random.default_rng(10 * G + B)
    cells = G ** 3
    occupied = rng.choice(cells, max(1, (2 * cells) // 3), replace=False)
    nb = len(occupied) + 1                                # one slot is not referenced
    ind = np.full(cells, -1, np.int32)
    ind[occupied] = rng.permutation(nb)[:len(occupied)]
    ind = ind.reshape(G, G, G)
    atlas = rng.integers(0, 256, (nb, B, B, B, 8), dtype=np.uint8)
    t_ind, t_atlas = torch.from_numpy(ind).to(DEV), torch.from_numpy(atlas).to(DEV)
    r = [renderer.Renderer(G * B, B, (-1.0,) * 3, 2.0, 5.0, (1.0,) * 3, t_ind, t_atlas) for _ in range(2)]
    val = [(t_atlas.float() / 255.0).contiguous() for _ in range(2)]
    m, v = ([torch.zeros_like(val[0]) for _ in range(2)] for _ in range(2))
    out = [torch.zeros_like(t_atlas) for _ in range(2)]
    for step in range(1, 4):
        g = np.zeros(atlas.shape, np.float32)
        if step < 3:                                      # the third step: moments without a gradient
            on = rng.uniform(size=atlas.shape[:4]) < touched
            g[on, 1:] = rng.normal(size=(int(on.sum()), 7))
        grad = torch.from_numpy(g).to(DEV)
        r[0].adam_requantize_atlas(val[0], m[0], v[0], grad, step, lr=0.02, atlas_out=out[0])
        renderer.adam_step(val[1], m[1], v[1], grad, step, lr=0.02)
        r[1].requantize_atlas(val[1], out[1])
        # the two kernels may fuse a product and a sum differently: each sum of two terms below 2
        # is then off by an ulp of 1, also where the terms cancel
        for a in (val, m, v):
            np.testing.assert_allclose(a[0].cpu().numpy(), a[1].cpu().numpy(), rtol=1e-6, atol=step * 1.2e-7)
        codes = atlas.copy()
        codes[..., 1:] = oracle.requantize(val[0].cpu().numpy()[..., 1:])
        used = sorted(ind[ind >= 0].tolist())
        np.testing.assert_array_equal(out[0].cpu().numpy()[used], codes[used])
        got, want = _padded(r[0], ind, codes)
        np.testing.assert_array_equal(got[used], want[used])
    if touched:
        # codes did change, also where a voxel has copies: beside a stored neighbour, at the grid's border
        at = np.argwhere(ind >= 0)                         # z, y, x of the stored blocks
        new = (out[0].cpu().numpy()[ind[ind >= 0]] != atlas[ind[ind >= 0]])[..., 1:].any(-1)
        block, *local = np.nonzero(new)
        shared = border = False
        for axis in range(3):
            for face, step in ((0, -1), (B - 1, 1)):
                beside = at[block[local[axis] == face]]
                beside[:, axis] += step
                inside = (beside[:, axis] >= 0) & (beside[:, axis] < G)
                border |= bool((~inside).any())
                shared |= bool((ind[tuple(beside[inside].T)] >= 0).any())
        assert new.any() and border and (shared or G == 1)


def test_arguments():
    t_ind = torch.zeros((1, 1, 1), dtype=torch.int32, device=DEV)
    atlas = torch.zeros((1, 2, 2, 2, 8), dtype=torch.uint8, device=DEV)
    r = renderer.Renderer(2, 2, (-1.0,) * 3, 2.0, 5.0, (1.0,) * 3, t_ind, atlas)
    t = [torch.zeros(atlas.shape, device=DEV) for _ in range(4)]
    for kw in ({"step": 0}, {"step": 1, "lr": -1.0}, {"step": 1, "betas": (1.0, 0.9)}, {"step": 1, "eps": 0.0}):
        with pytest.raises(renderer.SnergError):
            r.adam_requantize_atlas(*t, **kw)
    with pytest.raises(ValueError):
        r.adam_requantize_atlas(t[0][:, :1], *t[1:], step=1)
