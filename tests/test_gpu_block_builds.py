"""The march is built with the block edge and the density / alpha choice as constants for edges of
8 to 64; debug outputs run the build that reads both from the scene. Every build has to give the
same pixels, bit for bit, and the same gradients up to the order of FP32 sums, on blocks whose
rays enter, leave and cross stencils at every face."""
import numpy as np
import pytest
import torch

from paper_2103_14645_gb300 import renderer, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("flags", [0, 4])
@pytest.mark.parametrize("G,B", [(12, 2), (9, 4), (7, 8), (5, 16), (3, 32), (2, 64)])
def test_every_build_renders_the_same(G, B, flags):
    rng = np.random.default_rng(10 * G + B + flags)
    cells = G ** 3
    occupied = rng.choice(cells, max(1, (3 * cells) // 5), replace=False)
    ind = np.full(cells, -1, np.int32)
    ind[occupied] = rng.permutation(len(occupied))
    atlas = rng.integers(0, 256, (len(occupied), B, B, B, 8), dtype=np.uint8)
    atlas[..., 0] *= rng.uniform(size=atlas.shape[:4]) < 0.08
    cams = synth.orbit_cameras(rng, [(401, 299), (150, 170)], 1.5, 50.0)
    sc = synth.custom_scene(G * B, B, ind.reshape(G, G, G), atlas, 0.3 * G * B, synth.init_mlp(rng), cams, flags=flags)
    r = renderer.Renderer.from_scene(sc, DEV)
    r.set_mlp(sc.mlp)
    w = torch.from_numpy(sc.mlp).to(DEV)
    for mlp in (None, w):
        want = r.render(cams, mlp, counts=True)["rgb"]             # the build with members
        assert torch.equal(r.render(cams, mlp), want)
        assert torch.equal(r.render(cams, mlp, persistent=True), want)
        assert torch.equal(r.render(cams, mlp, persistent=True, tile=(8, 8), ctas_per_sm=4), want)
        assert torch.equal(r.render(cams[:1], mlp, schedule=True), want[:401 * 299])
        pix = torch.from_numpy(synth.random_pixels(rng, cams, 100001)).to(DEV)
        at = torch.where(pix[:, 0] == 0, pix[:, 2] * 401 + pix[:, 1], 401 * 299 + pix[:, 2] * 150 + pix[:, 1]).long()
        for n in (100001, 777):
            p = pix[:n].contiguous()
            assert torch.equal(r.render_rays(cams, p, mlp), want[at[:n]])
    rgb, state = r.render_rays_recorded(cams, pix, w)
    assert torch.equal(rgb, want[at])
    up = torch.from_numpy(rng.normal(size=(100001, 3)).astype(np.float32)).to(DEV)
    ga, gm = torch.zeros(sc.atlas.shape, device=DEV), torch.zeros(883, device=DEV)
    dbg = r.render_rays(cams, pix, w, aux=True, counts=True)
    r.backward(cams, pix, w, up, ga, gm, fwd_aux=dbg["aux"], fwd_counts=dbg["counts"])
    ra, rm = torch.empty_like(ga), torch.empty_like(gm)
    r.backward_recorded(cams, pix, w, up, state, ra, rm)
    own_a, own_m = torch.zeros_like(ga), torch.zeros_like(gm)
    r.backward(cams, pix, w, up, own_a, own_m)
    r.check_status()
    for x, y in ((ra, ga), (rm, gm), (own_a, ga), (own_m, gm)):
        assert float((x - y).abs().max()) <= 2e-5 * float(y.abs().max())
