"""snerg_render_rays_noalloc over block edges and grid sizes: its two-sided block map (one word or
two of blocks per row, the largest grid, a single block), stencils inside a block and across its
faces, and probes beyond a run's end, against the ordinary ray-list call on the same rays."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2103_14645_gb300 import renderer, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("G,B,p_block,n", [(1, 8, 1.0, 500), (7, 2, 0.5, 3000), (33, 4, 0.02, 3000), (64, 2, 0.01, 3000),
                                           (5, 16, 0.4, 90001), (2, 64, 0.7, 129)])
def test_matches_render_rays(G, B, p_block, n):
    rng = np.random.default_rng(31 * G + B)
    cells = G ** 3
    occupied = rng.choice(cells, max(1, int(p_block * cells)), replace=False)
    ind = np.full(cells, -1, np.int32)
    ind[occupied] = rng.permutation(len(occupied))
    atlas = rng.integers(0, 256, (len(occupied), B, B, B, 8), dtype=np.uint8)
    atlas[..., 0] *= rng.uniform(size=atlas.shape[:4]) < 0.15
    cams = synth.orbit_cameras(rng, [(200, 150)] * 3, 1.6, 50.0)
    sc = synth.custom_scene(G * B, B, ind.reshape(G, G, G), atlas, 40.0, synth.init_mlp(rng), cams)
    pix_np = synth.random_pixels(rng, cams, n)
    t_ind, t_atl, pix, mlp = (torch.from_numpy(a).to(DEV) for a in (sc.ind, sc.atlas, pix_np, sc.mlp))
    want = renderer.Renderer.from_scene(sc, DEV).render_rays(cams, pix, mlp)
    out = torch.full((n, 3), float("nan"), device=DEV)
    status = torch.full((1,), -1, dtype=torch.int32, device=DEV)
    desc = renderer.SceneDesc(sc.N, sc.B, (ctypes.c_float * 3)(*sc.bmin), sc.extent, sc.sigma_max,
                              (ctypes.c_float * 3)(*sc.bg), 0, 0)
    code = renderer.load_library().snerg_render_rays_noalloc(
        ctypes.byref(desc), t_ind.data_ptr(), t_atl.data_ptr(), sc.nb, cams.ctypes.data, 3, pix.data_ptr(), n,
        mlp.data_ptr(), out.data_ptr(), status.data_ptr(), torch.cuda.current_stream(DEV).cuda_stream)
    torch.cuda.synchronize()
    assert code == 0 and int(status.item()) == 0
    # the same samples composited with the same weights: FP32 rounding of the MLP's sums only
    assert float((out - want).abs().max()) <= 2e-6
