"""Launches that leave the chip part empty run fewer rays per warp (1, 2, 4, 8 or 16 lanes). Which
rays share a warp changes no ray: images, row ranges, scheduled frames and ray lists of every
size class, on both sides of each class's limit, are compared bit for bit with launches of 32 rays
per warp, and the adjoint's sums (which rows a thread block adds up depends on the lanes) with the
same rays in many small calls. The sizes follow from the launch rules and the device's SMs."""
import numpy as np
import pytest
import torch

from paper_2103_14645_gb300 import renderer, synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
LANES = (1, 2, 4, 8, 16)
N = 64                                                     # the scene's grid


def _most(lanes, rule):
    """The most rays that take no more than `lanes` per warp."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count

    def side(d, lo, hi):
        return min(max(N // d, lo), hi)
    warps = {"image": [side(8, 36, 56), side(10, 40, 80), side(10, 36, 96), side(12, 40, 96), side(14, 28, 96)],
             "list": [28, 28, 28, side(16, 20, 28), side(16, 16, 28)], "debug list": [16] * 5,
             "adjoint": [9, 9, side(32, 10, 12), side(32, 11, 14), side(20, 10, 14)]}[rule]
    return sms * warps[LANES.index(lanes)] * lanes


def _lanes(n, rule):
    return next((l for l in LANES if n <= _most(l, rule)), 32)


@pytest.fixture(scope="module")
def scene():
    sc = synth.make_scene("gauss64")
    r = renderer.Renderer.from_scene(sc, DEV)
    r.set_mlp(sc.mlp)
    return sc, r, torch.from_numpy(sc.mlp).to(DEV)


def _camera(W, H):
    return np.asarray([synth.look_at_camera((1.5, -1.1, 0.9), (0.0, 0.0, 0.0), W, H, 45.0, 0)])


def _image(lanes, over):
    """A ragged image of `lanes` rays per warp, near the class's limit, or the next class (over)."""
    n = _most(lanes, "image")
    W = int((4 * n / 3) ** 0.5) | 1
    H = n // W
    if over:
        H += 1 + (n - W * H == 0)
    assert _lanes(W * H, "image") == (32 if over and lanes == 16 else 2 * lanes if over else lanes)
    return W, H


@pytest.mark.parametrize("size", [(1, 1), (7, 3), (61, 37)] + [(l, over) for l in LANES for over in (False, True)])
def test_images_of_every_size_class(scene, size):
    W, H = _image(*size) if isinstance(size[1], bool) else size
    _, r, w = scene
    cam = _camera(W, H)
    want = r.render(cam, w, counts=True)["rgb"]            # debug outputs: 32 rays per warp
    assert torch.equal(r.render(cam, w), want)
    stored = r.render(cam, None, counts=True)["rgb"]
    assert torch.equal(r.render(cam, None), stored)
    for _ in range(3):
        assert torch.equal(r.render(cam, None, schedule=True), stored)
    rows = (H // 3, H - H // 4)
    out = torch.full((W * H, 3), -1.0, device=DEV)
    r.render(cam, w, out=out, rows=rows)
    inside = torch.zeros(H, dtype=torch.bool, device=DEV)
    inside[rows[0]:rows[1]] = True
    inside = inside[:, None].expand(H, W).reshape(-1)
    assert torch.equal(out[inside], want[inside]) and bool((out[~inside] == -1.0).all())
    r.check_status()


@pytest.mark.parametrize("rule", ["list", "debug list"])
@pytest.mark.parametrize("lanes,more", [(0, 1), (0, 33)] + [(l, more) for l in LANES for more in (0, 1)] +
                         [(per, more) for per in (40, 70, 80, 140, 160) for more in (0, 1)])
def test_ray_lists_of_every_size_class(scene, lanes, more, rule):
    # 40, 70, 80, 140, 160: 4, 7, 8, 14, 16 CTAs per SM of 128 rays, where the builds change
    n = more + (0 if lanes == 0 else _most(1, "debug list") * 32 * lanes // 40 if lanes >= 40 else _most(lanes, rule))
    assert lanes in (0, 40, 70, 80, 140, 160) or _lanes(n, rule) == (lanes if not more else 2 * lanes)
    _, r, w = scene
    cam = _camera(1021, 523)
    image = r.render(cam, w, counts=True)["rgb"]
    pix = synth.random_pixels(np.random.default_rng(n), cam, n)
    t = torch.from_numpy(pix).to(DEV)
    want = image[t[:, 2].long() * 1021 + t[:, 1].long()]
    assert torch.equal(r.render_rays(cam, t, w), want)
    out = r.render_rays(cam, t, w, aux=True, counts=True)
    assert torch.equal(out["rgb"], want)
    r.check_status()


@pytest.mark.parametrize("lanes,more", [(0, 5)] + [(l, more) for l in LANES for more in (0, 1)])
def test_adjoint_sums_of_every_size_class(scene, lanes, more):
    n = more + (_most(lanes, "adjoint") if lanes else 0)
    assert lanes == 0 or _lanes(n, "adjoint") == (lanes if not more else 2 * lanes)
    sc, r, w = scene
    cam = _camera(640, 479)
    rng = np.random.default_rng(n)
    pix = torch.from_numpy(synth.random_pixels(rng, cam, n)).to(DEV)
    target = torch.from_numpy(rng.uniform(size=(n, 3)).astype(np.float32)).to(DEV)

    def step(lots):
        g_atlas = torch.zeros(sc.atlas.shape, device=DEV)
        g_mlp, loss = torch.zeros(883, device=DEV), torch.zeros(1, device=DEV)
        rgb = torch.empty((n, 3), device=DEV)
        b_atlas, b_mlp = torch.zeros_like(g_atlas), torch.zeros_like(g_mlp)
        for i in range(0, n, lots):
            sl = slice(i, min(i + lots, n))
            out = rgb[sl]
            r.train_rays(cam, pix[sl].contiguous(), w, target[sl].contiguous(), g_atlas, g_mlp, loss=loss, out=out)
            r.backward(cam, pix[sl].contiguous(), w, 2.0 * (out - target[sl]), b_atlas, b_mlp)
        return rgb, loss, g_atlas, g_mlp, b_atlas, b_mlp

    whole, small = step(n), step(2000)
    assert torch.equal(whole[0], small[0])
    # FP32 sums of up to n terms in another order
    for a, b in zip(whole[1:], small[1:]):
        scale = float(b.abs().max())
        assert float((a - b).abs().max()) <= 2e-5 * scale + 1e-7
    assert float((whole[2] - whole[4]).abs().max()) <= 2e-5 * float(whole[2].abs().max())
    r.check_status()


def test_images_on_several_streams(scene):
    """A handle whose images come in on several streams gives them more rays per warp again (here 8
    and 16 instead of 4, beside the 4 of the first calls): the same colours."""
    _, r, _ = scene
    W, H = _image(4, False)
    cam = _camera(W, H)
    want = r.render(cam, None, counts=True)["rgb"]
    streams = [torch.cuda.Stream() for _ in range(8)]
    torch.cuda.synchronize()
    for _ in range(2):
        outs = []
        for s in streams:
            with torch.cuda.stream(s):
                outs.append(r.render(cam, None))
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in outs)
