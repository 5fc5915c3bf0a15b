"""The render that records its composited samples and the adjoint that scatters them, against the
plain pair of calls: the same colours and per-ray state bit for bit, the same gradients up to the
order of FP32 sums, for rays with fewer, exactly and more samples than a record holds, every
scene flag of the ray-list path, and ray counts on both sides of the launch rules."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2103_14645_gb300 import renderer, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _scene(flags, sigma_vox, seed):
    ind, atl = synth.gauss_grid(64, 8, 0.4, 0.6, seed)
    cams = synth.orbit_cameras(np.random.default_rng(seed), [(300, 200)] * 2, 1.7, 45.0)
    return synth.custom_scene(64, 8, ind, atl, sigma_vox * 32.0, synth.init_mlp(np.random.default_rng(seed + 1)), cams,
                              flags=flags)


@pytest.mark.parametrize("flags,sigma_vox,n", [(0, 0.6, 1), (0, 0.05, 700), (1, 0.6, 9728), (4, 0.6, 9729), (8, 0.05, 20000),
                                               (5, 0.3, 77825), (0, 0.3, 150000), (0, 5.0, 155649)])
def test_recorded_pair_matches_the_plain_pair(flags, sigma_vox, n):
    sc = _scene(flags, sigma_vox, 3)
    r = renderer.Renderer.from_scene(sc, DEV)
    w = torch.from_numpy(sc.mlp).to(DEV)
    rng = np.random.default_rng(n)
    pix = torch.from_numpy(synth.random_pixels(rng, sc.cameras, n)).to(DEV)
    g = torch.from_numpy(rng.normal(size=(n, 3)).astype(np.float32)).to(DEV)
    a = r.render_rays(sc.cameras, pix, w, aux=True, counts=True)
    rgb, state = r.render_rays_recorded(sc.cameras, pix, w)
    assert torch.equal(a["rgb"], rgb)
    if sigma_vox == 0.05 and n > 100:
        assert int(a["counts"][:, 1].max()) > 32           # some rays march on past their record
    ga, gm = torch.zeros(sc.atlas.shape, device=DEV), torch.zeros(883, device=DEV)
    r.backward(sc.cameras, pix, w, g, ga, gm, fwd_aux=a["aux"], fwd_counts=a["counts"])
    ra, rm = torch.full_like(ga, 7.0), torch.full_like(gm, 7.0)       # overwritten
    r.backward_recorded(sc.cameras, pix, w, g, state, ra, rm)
    r.check_status()
    for x, y in ((ra, ga), (rm, gm)):
        assert float((x - y).abs().max()) <= 2e-5 * float(y.abs().max()) + 1e-7
    assert bool((ra[..., 0] == 0).all())
    only = torch.full_like(gm, 3.0)
    r.backward_recorded(sc.cameras, pix, w, g, state, None, only)
    assert float((only - gm).abs().max()) <= 2e-5 * float(gm.abs().max()) + 1e-7


def test_autograd_and_large_fine_tuning_take_the_record():
    sc = _scene(0, 0.3, 4)
    r = renderer.Renderer.from_scene(sc, DEV)
    pix = torch.from_numpy(synth.random_pixels(np.random.default_rng(1), sc.cameras, 5000)).to(DEV)
    w = torch.from_numpy(sc.mlp).to(DEV).requires_grad_()
    vals = (torch.from_numpy(sc.atlas).to(DEV).float() / 255.0).requires_grad_()
    target = torch.rand((5000, 3), device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
    loss = ((renderer.render_rays_autograd(r, sc.cameras, pix, w, vals) - target) ** 2).sum()
    loss.backward()
    ga, gm, ls = torch.zeros_like(vals), torch.zeros(883, device=DEV), torch.zeros(1, device=DEV)
    r.train_rays(sc.cameras, pix, w.detach(), target, ga, gm, loss=ls)
    loss = float(loss.detach())
    assert abs(loss - float(ls)) <= 1e-5 * float(ls)
    assert float((vals.grad - ga).abs().max()) <= 2e-5 * float(ga.abs().max())
    assert float((w.grad - gm).abs().max()) <= 2e-5 * float(gm.abs().max())
    ft = [renderer.FineTuner(r, sc.mlp, atlas=sc.atlas, atlas_lr=1e-3) for _ in range(2)]
    ft[1].fused_rays = 0                                   # the separate calls
    for f in ft:
        f.step(sc.cameras, pix, target)
    assert float((ft[0].ma - ft[1].ma).abs().max()) <= 2e-5 * float(ft[0].ma.abs().max())
    assert float((ft[0].m - ft[1].m).abs().max()) <= 2e-5 * float(ft[0].m.abs().max())


def test_no_rays_and_arguments():
    lib = renderer.load_library()
    assert lib.snerg_state_bytes(0) == 0 and lib.snerg_state_bytes(3) == 3 * (48 + 33 * 8)
    sc = _scene(0, 0.6, 5)
    r = renderer.Renderer.from_scene(sc, DEV)
    w = torch.from_numpy(sc.mlp).to(DEV)
    pix = torch.zeros((4, 3), dtype=torch.int32, device=DEV)
    rgb, state = r.render_rays_recorded(sc.cameras, pix, w)
    gm = torch.ones(883, device=DEV)
    with pytest.raises(ValueError):                        # the state of another number of rays
        r.backward_recorded(sc.cameras, pix[:2].contiguous(), w, rgb[:2].contiguous(), state, None, gm)
    none, P = ctypes.c_void_p(None), sc.cameras.ctypes.data
    assert lib.snerg_render_rays_recorded(r.handle, P, 2, pix.data_ptr(), 4, w.data_ptr(), rgb.data_ptr(), none, none) == 1
    assert lib.snerg_render_backward_recorded(r.handle, P, 2, pix.data_ptr(), 4, w.data_ptr(), rgb.data_ptr(), none, none,
                                              gm.data_ptr(), none) == 1
    # a refused call leaves the gradients alone: no rays' pixels, weights or upstream gradient, no
    # cameras, an unaligned atlas gradient
    ga = torch.ones(sc.atlas.size + 1, device=DEV)
    args = [r.handle, P, 2, pix.data_ptr(), 4, w.data_ptr(), rgb.data_ptr(), state.data_ptr(), ga.data_ptr(), gm.data_ptr(), none]
    for i, v in ((3, none), (5, none), (6, none), (1, none), (2, 0), (8, ga.data_ptr() + 4)):
        assert lib.snerg_render_backward_recorded(*args[:i], v, *args[i + 1:]) == 1
        assert bool((ga == 1).all()) and bool((gm == 1).all()), i
    with pytest.raises(ValueError):                        # too short for the sums
        r.backward_recorded(sc.cameras, pix, w, rgb, state, None, gm[:882])
    rgb, state = r.render_rays_recorded(sc.cameras, pix[:0], w)
    ga = torch.ones(sc.atlas.shape, device=DEV)
    r.backward_recorded(sc.cameras, pix[:0], w, rgb, state, ga, gm)
    assert rgb.shape == (0, 3) and not bool(ga.any()) and not bool(gm.any())


def test_rays_beyond_the_record_limit_keep_the_small_state(monkeypatch):
    sc = _scene(0, 0.3, 4)
    r = renderer.Renderer.from_scene(sc, DEV)
    n = 60000
    pix = torch.from_numpy(synth.random_pixels(np.random.default_rng(1), sc.cameras, n)).to(DEV)
    w = torch.from_numpy(sc.mlp).to(DEV).requires_grad_()
    vals = (torch.from_numpy(sc.atlas).to(DEV).float() / 255.0).requires_grad_()
    target = torch.rand((n, 3), device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
    grads, kept, moments = [], [], []
    for limit in (n, n - 1):
        monkeypatch.setattr(renderer, "RECORD_MAX_RAYS", limit)
        before = torch.cuda.memory_allocated()
        rgb = renderer.render_rays_autograd(r, sc.cameras, pix, w, vals)
        kept.append(torch.cuda.memory_allocated() - before)
        grads.append(torch.autograd.grad(rgb, (w, vals), rgb.detach() - target))
        del rgb
        ft = renderer.FineTuner(r, sc.mlp, atlas=sc.atlas, atlas_lr=0.0)
        ft.fused_rays = 0
        ft.step(sc.cameras, pix, target)
        moments.append((ft.m.clone(), ft.ma.clone()))
    assert kept[0] >= (12 + 312) * n and kept[1] <= (12 + 48) * n + 4096
    for a, b in (grads, moments):
        for x, y in zip(a, b):
            assert float((x - y).abs().max()) <= 2e-5 * float(y.abs().max())


def test_no_state_is_kept_without_a_backward():
    sc = _scene(0, 0.3, 4)
    r = renderer.Renderer.from_scene(sc, DEV)
    n = 200000
    pix = torch.from_numpy(synth.random_pixels(np.random.default_rng(1), sc.cameras, n)).to(DEV)
    w = torch.from_numpy(sc.mlp).to(DEV).requires_grad_()
    vals = (torch.from_numpy(sc.atlas).to(DEV).float() / 255.0).requires_grad_()
    want = renderer.render_rays_autograd(r, sc.cameras, pix, w, vals)
    assert want.requires_grad
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    with torch.no_grad():
        rgb = renderer.render_rays_autograd(r, sc.cameras, pix, w, vals)
    assert torch.equal(rgb, want) and not rgb.requires_grad
    assert torch.cuda.max_memory_allocated() - before <= 12 * n + (2 << 20)       # the colours
    with torch.inference_mode():
        assert torch.equal(renderer.render_rays_autograd(r, sc.cameras, pix, w, vals), want)
