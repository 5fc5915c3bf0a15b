"""What the renderer is timed on: the calls a program makes of it, over the sizes it is used at.

A scene is thin closed shells in a mostly empty grid, hollow inside, stored in B^3
macroblocks with seeded smooth colours and features: the structure of a baked object after
culling, made on the GPU from the seed. Cameras look at it from around the unit cube at a
39 degree field of view. A case has one geometry, and the seed turns and mirrors it, so that
every seed stores as many blocks: the colours, the slot order, the network, the cameras and
the rays are the seed's own.

`exact` follows the documented arithmetic contract: the sample lattice, the nearest voxel
and the early exit are decided in binary32 with one rounding per operation, and everything
that is summed or evaluated along the ray is 64 bit.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2103_14645_gb300 import renderer, synth

DEV = "cuda"
BMIN = (-1.0, -1.0, -1.0)
EXTENT = 2.0
SIGMA_VOX = 5.0          # optical depth of a voxel at code 255: an opaque surface is 2 to 4 samples deep
TAU_ALPHA = 0.005        # a block whose largest opacity is below this is not stored
BG = (1.0, 1.0, 1.0)
RADIUS = 2.2             # cameras' distance from the centre of the cube
FOV = 39.0
LR = 3e-4
ATLAS_LR = 2e-3
BETAS = (0.9, 0.999)
EPS = 1e-8


def listed():
    return [
        # a thumbnail or a low-resolution preview: the smallest call, where latency counts
        {"name": "view_200", "kind": "view", "N": 512, "B": 32, "W": 200, "H": 200, "flags": 0, "weights": "stored",
         "dest": "device"},
        # the frame that the paper times: 800 x 800 pixels of a 1024^3 grid
        {"name": "view_800", "kind": "view", "N": 1024, "B": 32, "W": 800, "H": 800, "flags": 0, "weights": "stored",
         "dest": "device"},
        # a full-HD frame of a large grid handed to the host (display, encoder), alpha atlas,
        # an odd image size, network weights in a tensor
        {"name": "view_hd_host", "kind": "view", "N": 2048, "B": 32, "W": 1919, "H": 1079, "flags": 4,
         "weights": "tensor", "dest": "host"},
        # an interactive viewer: consecutive frames of a moving camera with the tile schedule
        {"name": "orbit_800", "kind": "orbit", "N": 1024, "B": 32, "W": 800, "H": 800, "flags": 0, "frames": 12},
        # an offline job (test set, light field): many cameras of mixed sizes in one launch
        {"name": "batch_64", "kind": "batch", "N": 1024, "B": 32, "cams": 64, "flags": 0},
        # scattered pixels of several views (picking, metrics on a subset), forward only
        {"name": "rays_262k", "kind": "rays", "N": 1024, "B": 32, "n": 262147, "flags": 1, "weights": "tensor"},
        # the same for a host application that owns all memory: smaller blocks, no handle
        {"name": "rays_noalloc_65k", "kind": "noalloc", "N": 768, "B": 16, "n": 65537, "flags": 0},
        # the render inside somebody's own training loop: forward and backward through autograd
        {"name": "autograd_65k", "kind": "autograd", "N": 512, "B": 32, "n": 65536, "flags": 0},
        # fine-tuning the network after a bake
        {"name": "finetune_mlp_16k", "kind": "finetune", "N": 1024, "B": 32, "n": 16384, "flags": 0, "atlas": False},
        # fine-tuning the network and the baked colours and features
        {"name": "finetune_atlas_65k", "kind": "finetune", "N": 512, "B": 32, "n": 65536, "flags": 0, "atlas": True},
        # opening a scene: device tensors to the first frame on the screen
        {"name": "open_1024", "kind": "open", "N": 1024, "B": 32, "W": 800, "H": 800, "flags": 0},
        # baking a field into a new scene
        {"name": "bake_1024", "kind": "bake", "N": 1024, "B": 32, "blobs": 64, "flags": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, n_max, g_max):
    """Block edge and grid size: powers of two and others, up to n_max voxels a side."""
    B = rng.choice([8, 16, 32, 32, 32, 64])
    G = _log_int(rng, max(4, 256 // B), min(n_max // B, g_max))
    return {"N": B * G, "B": B}


def draw(rng):
    kind = rng.choice(["view", "view", "orbit", "batch", "rays", "rays", "noalloc", "autograd", "finetune", "finetune",
                       "open", "bake"])
    if kind == "view":
        W = _log_int(rng, 160, 1920)
        return {"kind": kind, **_grid(rng, 2048, 64), "W": W, "H": max(90, int(W * rng.uniform(0.55, 1.0))),
                "flags": rng.choice([0, 0, 1, 2, 4, 5, 8]), "weights": rng.choice(["stored", "tensor"]),
                "dest": rng.choice(["device", "device", "host"])}
    if kind == "orbit":
        W = _log_int(rng, 320, 1280)
        return {"kind": kind, **_grid(rng, 1024, 64), "W": W, "H": int(W * rng.uniform(0.55, 1.0)),
                "flags": rng.choice([0, 0, 4]), "frames": rng.randint(6, 12)}
    if kind == "batch":
        return {"kind": kind, **_grid(rng, 1024, 64), "cams": _log_int(rng, 3, 64), "flags": rng.choice([0, 0, 1, 4, 8])}
    if kind in ("rays", "noalloc"):
        c = {"kind": kind, **_grid(rng, 1024, 64), "n": _log_int(rng, 1000, 262144),
             "flags": rng.choice([0, 1] if kind == "noalloc" else [0, 0, 1, 4, 8])}
        return c if kind == "noalloc" else dict(c, weights=rng.choice(["stored", "tensor"]))
    if kind == "autograd":
        return {"kind": kind, **_grid(rng, 512, 32), "n": _log_int(rng, 1000, 131072),
                "flags": rng.choice([0, 0, 1, 4, 8])}
    if kind == "finetune":
        atlas = rng.random() < 0.5
        return {"kind": kind, **_grid(rng, 512 if atlas else 1024, 32 if atlas else 64),
                "n": _log_int(rng, 1000, 65536 if atlas else 1000000), "flags": rng.choice([0, 0, 1, 4]), "atlas": atlas}
    if kind == "open":
        W = _log_int(rng, 160, 1280)
        return {"kind": kind, **_grid(rng, 1024, 64), "W": W, "H": int(W * rng.uniform(0.55, 1.0)),
                "flags": rng.choice([0, 0, 4])}
    return {"kind": kind, **_grid(rng, 1024, 64), "blobs": rng.randint(4, 64), "flags": rng.choice([0, 4])}


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _turn(seed):
    """The seed's order of the axes and which of them it mirrors."""
    rng = np.random.default_rng([seed, 3])
    return [int(i) for i in rng.permutation(3)], [bool(b) for b in rng.integers(0, 2, 3)]


def _scene(case, seed):
    """(ind int32 [G,G,G], atlas uint8 [nb,B,B,B,8], mlp float32 [883]) on the GPU."""
    N, B = case["N"], case["B"]
    G = N // B
    shape = np.random.default_rng([N, B])
    shells = [(shape.uniform(0.38, 0.62, 3) * N, shape.uniform(0.15, 0.25, 3) * N) for _ in range(3)]
    rng = np.random.default_rng([seed, N, B])
    axes, flips = _turn(seed)
    freq, phase = rng.uniform(-12.0, 12.0, (7, 3)), rng.uniform(0.0, 2.0 * math.pi, 7)
    mlp = torch.from_numpy(synth.init_mlp(rng)).to(DEV)

    def distance(p, c, r):          # about the distance (in voxels) from the ellipsoid's surface
        c, r = torch.tensor(c, dtype=torch.float32, device=DEV), torch.tensor(r, dtype=torch.float32, device=DEV)
        a = (p - c) / r
        k0, k1 = a.norm(dim=-1), (a / r).norm(dim=-1).clamp_min(1e-12)
        return k0 * (k0 - 1.0) / k1

    ax = torch.arange(G, device=DEV)
    bz, by, bx = torch.meshgrid(ax, ax, ax, indexing="ij")
    blocks = torch.stack([bx, by, bz], -1).reshape(-1, 3)
    centre = (blocks.float() + 0.5) * B
    near = torch.zeros(blocks.shape[0], dtype=torch.bool, device=DEV)
    for c, r in shells:
        near |= distance(centre, c, r).abs() <= (0.87 * B + 4.0) * float(r.max() / r.min())
    cand = blocks[near]
    la = torch.arange(B, device=DEV)
    lz, ly, lx = torch.meshgrid(la, la, la, indexing="ij")
    local = torch.stack([lx, ly, lz], -1).reshape(-1, 3).float() + 0.5
    q_min = math.ceil(-math.log(1.0 - TAU_ALPHA) / SIGMA_VOX * 255.0)
    chunk = max(1, (1 << 24) // B ** 3)
    wt = torch.tensor(freq, dtype=torch.float32, device=DEV)
    pt = torch.tensor(phase, dtype=torch.float32, device=DEV)
    kept, parts = [], []
    for i in range(0, cand.shape[0], chunk):
        b = cand[i:i + chunk]
        p = b[:, None, :].float() * B + local
        dens = torch.zeros(p.shape[:2], device=DEV)
        for c, r in shells:
            dens = torch.maximum(dens, torch.exp(-distance(p, c, r) ** 2))
        q = torch.floor(dens * 255.0 + 0.5)
        keep = q.amax(1) >= q_min
        if not bool(keep.any()):
            continue
        # the geometry's blocks and voxels, turned
        b, q = b[keep][:, axes], q[keep].view(-1, B, B, B).permute(0, *(1 + 2 - axes[2 - i] for i in range(3)))
        for i in range(3):
            if flips[i]:
                b[:, i] = G - 1 - b[:, i]
                q = q.flip(3 - i)
        q, p = q.reshape(-1, B ** 3), b[:, None, :].float() * B + local
        a = torch.empty((q.shape[0], B ** 3, 8), dtype=torch.uint8, device=DEV)
        a[..., 0] = q.to(torch.uint8)
        for c in range(7):
            x = (p[..., 0] * wt[c, 0] + p[..., 1] * wt[c, 1] + p[..., 2] * wt[c, 2]) / N + pt[c]
            a[..., 1 + c] = torch.floor((0.5 + 0.5 * torch.sin(x)) * 255.0 + 0.5).to(torch.uint8)
        kept.append(b)
        parts.append(a)
    kept = torch.cat(kept)
    order = torch.from_numpy(rng.permutation(kept.shape[0])).to(DEV)     # slots in no spatial order
    kept, atlas = kept[order], torch.cat(parts)[order].reshape(-1, B, B, B, 8).contiguous()
    ind = torch.full((G, G, G), -1, dtype=torch.int32, device=DEV)
    ind[kept[:, 2], kept[:, 1], kept[:, 0]] = torch.arange(kept.shape[0], dtype=torch.int32, device=DEV)
    return ind, atlas, mlp


def _sigma_max(case):
    return SIGMA_VOX * case["N"] / EXTENT


def _cameras(case, seed):
    rng = np.random.default_rng([seed, 7])
    if case["kind"] == "batch":
        sizes = [(200, 200), (400, 400), (800, 800), (1280, 720), (1920, 1080), (533, 401)]
        return synth.orbit_cameras(rng, [sizes[(5 * i + 2) % len(sizes)] for i in range(case["cams"])], RADIUS, FOV)
    if case["kind"] == "orbit":
        # a small closed loop, so that one pass follows on the last
        W, H, n = case["W"], case["H"], case["frames"]
        az0, el0 = rng.uniform(0.0, 2.0 * math.pi), math.radians(rng.uniform(-30.0, 50.0))
        cams = np.zeros(n, synth.CAMERA_DTYPE)
        for i in range(n):
            az = az0 + math.radians(8.0) * math.sin(2.0 * math.pi * i / n)
            el = el0 + math.radians(5.0) * math.cos(2.0 * math.pi * i / n)
            pos = RADIUS * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
            cams[i] = synth.look_at_camera(pos, (0.0, 0.0, 0.0), W, H, FOV, 0)
        return cams
    sizes = [(case["W"], case["H"])] if "W" in case else [(800, 800)] * 8
    return synth.orbit_cameras(rng, sizes, RADIUS, FOV)


def _rays(case, cams, seed):
    rng = np.random.default_rng([seed, 11])
    return torch.from_numpy(synth.random_pixels(rng, cams, case["n"])).to(DEV)


def _values(seed, n):
    """Seeded observed colours / upstream gradients, [n, 3]."""
    g = torch.Generator(device=DEV).manual_seed(seed * 2 + 1)
    return torch.rand((n, 3), generator=g, device=DEV)


def _field(case, seed):
    f = synth.analytic_field(seed, n_blob=case["blobs"])
    f["blobs"] = synth.analytic_field(case["blobs"], n_blob=case["blobs"])["blobs"]
    axes, flips = _turn(seed)
    f["blobs"][:, :3] = f["blobs"][:, axes] * np.where(flips, -1.0, 1.0)
    return f


def _renderer(case, ind, atlas):
    return renderer.Renderer(case["N"], case["B"], BMIN, EXTENT, _sigma_max(case), BG, ind, atlas, flags=case["flags"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "bake":
        f = _field(case, seed)
        return {"case": case, "field": renderer.bake_field(f["blobs"], f["colors"], f["jitter"], TAU_ALPHA)}
    ind, atlas, mlp = _scene(case, seed)
    cams = _cameras(case, seed)
    s = {"case": case, "cams": cams, "mlp": mlp}
    if kind == "open":
        return dict(s, ind=ind, atlas=atlas, weights=mlp.cpu().numpy())
    if kind == "noalloc":
        n = case["n"]
        desc = renderer.SceneDesc(case["N"], case["B"], (ctypes.c_float * 3)(*BMIN), EXTENT, _sigma_max(case),
                                  (ctypes.c_float * 3)(*BG), 0, case["flags"])
        return dict(s, ind=ind, atlas=atlas, desc=desc, lib=renderer.load_library(), pix=_rays(case, cams, seed),
                    out=torch.zeros((n, 3), device=DEV), status=torch.zeros(1, dtype=torch.int32, device=DEV))
    r = _renderer(case, ind, atlas)
    s["r"] = r
    if kind in ("view", "orbit", "batch"):
        r.set_mlp(mlp.cpu().numpy())
        n = sum(int(c["W"]) * int(c["H"]) for c in cams)
        if case.get("dest") == "host":
            s["out"] = torch.zeros((n, 3)).pin_memory()
        elif kind == "orbit":
            s["out"] = torch.zeros((case["frames"], case["W"] * case["H"], 3), device=DEV)
        else:
            s["out"] = torch.zeros((n, 3), device=DEV)
        return s
    s["pix"] = _rays(case, cams, seed)
    if kind == "rays":
        r.set_mlp(mlp.cpu().numpy())
    elif kind == "autograd":
        s["grad"] = _values(seed, case["n"]) - 0.5
        s["mlp"] = mlp.requires_grad_()
        s["values"] = (atlas.float() / 255.0).requires_grad_()
    else:
        s["target"] = _values(seed, case["n"])
        host = atlas.cpu().numpy() if case["atlas"] else None
        s["ft"] = renderer.FineTuner(r, mlp.cpu().numpy(), lr=LR, betas=BETAS, eps=EPS, atlas=host,
                                     atlas_lr=ATLAS_LR if case["atlas"] else None)
    return s


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(s):
    case, cams = s["case"], s.get("cams")
    kind = case["kind"]
    if kind == "view":
        mlp = s["mlp"] if case["weights"] == "tensor" else None
        if case["dest"] == "host":
            return s["r"].render_to_host(cams, s["out"], mlp)
        return s["r"].render(cams, mlp, out=s["out"])
    if kind == "orbit":
        for i in range(case["frames"]):
            s["r"].render(cams[i:i + 1], None, out=s["out"][i], schedule=True)
        return s["out"]
    if kind == "batch":
        return s["r"].render(cams, None, out=s["out"], persistent=True)
    if kind == "rays":
        return s["r"].render_rays(cams, s["pix"], s["mlp"] if case["weights"] == "tensor" else None)
    if kind == "noalloc":
        code = s["lib"].snerg_render_rays_noalloc(
            ctypes.byref(s["desc"]), s["ind"].data_ptr(), s["atlas"].data_ptr(), s["atlas"].shape[0], cams.ctypes.data,
            cams.shape[0], s["pix"].data_ptr(), case["n"], s["mlp"].data_ptr(), s["out"].data_ptr(),
            s["status"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if code:
            raise RuntimeError("snerg_render_rays_noalloc: status %d" % code)
        return {"rgb": s["out"], "status": s["status"]}
    if kind == "autograd":
        rgb = renderer.render_rays_autograd(s["r"], cams, s["pix"], s["mlp"], s["values"])
        g_mlp, g_values = torch.autograd.grad(rgb, (s["mlp"], s["values"]), s["grad"])
        return {"rgb": rgb.detach(), "g_mlp": g_mlp, "g_values": g_values}
    if kind == "finetune":
        ft = s["ft"]
        out = {"loss": ft.step(cams, s["pix"], s["target"]), "mlp": ft.mlp, "m": ft.m, "v": ft.v}
        if case["atlas"]:
            out.update(shadow=ft.shadow, ma=ft.ma, va=ft.va, codes=ft.codes)
        return out
    if kind == "open":
        s["r"] = _renderer(case, s["ind"], s["atlas"])      # the program keeps its renderer
        s["r"].set_mlp(s["weights"])
        return s["r"].render(cams, None)
    ind, atlas = renderer.bake(case["N"], case["B"], BMIN, EXTENT, 200.0, s["field"], DEV, flags=case["flags"])
    return {"ind": ind, "atlas": atlas}


# ---------------------------------------------------------------------------------------
# what a pass cannot do without, and how far results may be off
# ---------------------------------------------------------------------------------------
# A ray of these scenes composites about 2.5 samples (hits and misses together), each of
# which needs about 4 voxels of 8 bytes that the sample before it did not; neighbouring
# pixels of one view share about half of them, scattered rays none.
_SAMPLES = 2.5
_RAY_FLOPS = 2 * 850 * 0.5 + _SAMPLES * 2 * 8 * 8


def _stored_blocks(case):
    """About the stored blocks of a scene: three ellipsoids of mean radius 0.2 N, shells two blocks deep."""
    return 3 * 4.0 * math.pi * (0.2 * case["N"] / case["B"]) ** 2 * 1.6


def work(case):
    kind = case["kind"]
    voxels = _SAMPLES * 4 * 8
    if kind == "bake":
        kept = 0.143 * case["N"] ** 3 * case["blobs"] / 64
        return {"bytes": 8 * kept + 4 * (case["N"] / case["B"]) ** 3, "flops": kept * (16 * 4 * 2 + 7 * 4)}
    if kind in ("rays", "noalloc"):
        return {"bytes": case["n"] * (24 + voxels), "flops": case["n"] * _RAY_FLOPS}
    if kind in ("autograd", "finetune"):
        n, vals = case["n"], _stored_blocks(case) * case["B"] ** 3 * 8
        atlas = {"autograd": 4 * vals}.get(kind, 29 * vals if case.get("atlas") else 0)
        return {"bytes": n * (36 + voxels + (2 * voxels * 4 if atlas else 0)) + atlas, "flops": 3 * n * _RAY_FLOPS}
    if kind == "batch":
        n = sum(int(c["W"]) * int(c["H"]) for c in _cameras(case, 0))
    else:
        n = case["W"] * case["H"] * case.get("frames", 1)
    b = n * (12 + voxels / 2)
    if kind == "open":      # the codes read, and a device layout with its empty-space map written
        b += _stored_blocks(case) * case["B"] ** 3 * (8 + 8 + 8)
    return {"bytes": b, "flops": n * _RAY_FLOPS}


def tolerance(case):
    """About four times what the renderer was seen to be off 64 bits, or between two runs."""
    kind = case["kind"]
    if kind == "bake":              # codes whose exact value lies at a rounding boundary: 1e-5 to 3e-5 of them
        return {"rel": 0.0, "differ": 1e-4}
    if kind == "finetune":
        # the loss and the moments are sums over the rays in any order: 5e-7; a first Adam step
        # divides g by |g|, so a single value whose gradient nearly cancels may move either way
        return {"rel": 2e-6, "max": 0.02, "differ": 1e-5}
    if kind == "autograd":          # gradients: sums over the rays in any order, 4e-7
        return {"rel": 2e-6, "max": 1e-4}
    return {"rel": 4e-7, "max": 2e-5}      # colours: 1e-7


# ---------------------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------------------
def _network(w, x):
    w1, b1, w2, b2, w3, b3 = torch.split(w, [544, 16, 256, 16, 48, 3])
    h = torch.relu(x @ w1.view(16, 34).T + b1)
    h = torch.relu(h @ w2.view(16, 16).T + b2)
    return torch.sigmoid(h @ w3.view(3, 16).T + b3)


def _inputs(cv, d):
    enc = [f(2.0 ** l * d) for l in range(4) for f in (torch.sin, torch.cos)]
    return torch.cat([cv, d, *enc], 1)


def _march(case, ind, atlas, mlp, cams, pix, record=None):
    """Composites [n, 7] (decoded), transmittance, samples composited, per-sample colours and
    directions of rays pix [n, 3], 64 bit; `record` receives every composited sample."""
    N, B = case["N"], case["B"]
    lg, f32, f64 = B.bit_length() - 1, torch.float32, torch.float64
    n, flags = pix.shape[0], case["flags"]
    cell = atlas.reshape(-1, 8)
    ci = pix[:, 0].long()

    def per_ray(name):
        return torch.from_numpy(np.ascontiguousarray(cams[name])).to(DEV)[ci]

    c2w = per_ray("c2w")
    dc = [(pix[:, 1].float() + 0.5 - per_ray("cx")) / per_ray("fx"), -((pix[:, 2].float() + 0.5 - per_ray("cy")) / per_ray("fy"))]
    d = [c2w[:, 4 * i] * dc[0] + c2w[:, 4 * i + 1] * dc[1] - c2w[:, 4 * i + 2] for i in range(3)]
    norm = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
    d = [x / norm for x in d]
    scale = torch.tensor(np.float32(N) / np.float32(EXTENT), device=DEV)
    o = [(c2w[:, 4 * i + 3] - BMIN[i]) * scale for i in range(3)]
    t0, t1 = torch.full((n,), -math.inf, device=DEV), torch.full((n,), math.inf, device=DEV)
    hit = torch.ones(n, dtype=torch.bool, device=DEV)
    for i in range(3):
        ta, tb, zero = -o[i] / d[i], (float(N) - o[i]) / d[i], d[i] == 0
        t0 = torch.where(zero, t0, torch.maximum(t0, torch.minimum(ta, tb)))
        t1 = torch.where(zero, t1, torch.minimum(t1, torch.maximum(ta, tb)))
        hit &= ~(zero & ((o[i] < 0) | (o[i] > N)))
    t0 = t0.clamp_min(0.0)
    hit &= t0 < t1
    kappa = np.float32(float(np.float32(_sigma_max(case))) * (EXTENT / N) / 255.0)
    tau_max, t_min = np.float32(math.log(1000.0)), np.float32(1e-3)
    acc = torch.zeros((n, 7), dtype=f64, device=DEV)
    per = torch.zeros((n, 3), dtype=f64, device=DEV)
    T, T32, tau = (torch.full((n,), v, dtype=t, device=DEV) for v, t in ((1.0, f64), (1.0, f32), (0.0, f32)))
    count = torch.zeros(n, dtype=torch.int32, device=DEV)
    done = torch.zeros(n, dtype=torch.bool, device=DEV)
    live = torch.nonzero(hit).flatten()
    k = 0
    while live.numel():
        lo, ld, l0, l1 = [x[live] for x in o], [x[live] for x in d], t0[live], t1[live]
        for k in range(k, k + 32):
            t = l0 + (k + 0.5)
            u = [lo[i] + t * ld[i] for i in range(3)]
            j = [torch.floor(x).clamp_(0, N - 1).to(torch.int32) for x in u]
            slot = ind[j[2] >> lg, j[1] >> lg, j[0] >> lg].long()
            loc = ((((j[2] & (B - 1)) << lg) + (j[1] & (B - 1))) << lg) + (j[0] & (B - 1))
            on = cell[slot.clamp_min(0) * B ** 3 + loc, 0] > 0
            at = torch.nonzero(on & (slot >= 0) & (t < l1) & ~done[live]).flatten()
            if not at.numel():
                continue
            ray = live[at]
            x = [u[i][at] - 0.5 for i in range(3)]
            low = [torch.floor(v) for v in x]
            f = [x[i] - low[i] for i in range(3)]
            g = [1.0 - v for v in f]
            where, q = [], []
            for c in range(8):
                p = [(low[i].long() + ((c >> i) & 1)).clamp(0, N - 1) for i in range(3)]
                sl = ind[p[2] >> lg, p[1] >> lg, p[0] >> lg].long()
                w = torch.where(sl >= 0, sl * B ** 3 + ((((p[2] & (B - 1)) << lg) + (p[1] & (B - 1))) << lg) + (p[0] & (B - 1)), -1)
                where.append(w)
                q.append(cell[w.clamp_min(0)] * (w >= 0)[:, None])
            q = torch.stack(q, 1)
            e = [q[:, c, 0].float() * g[0] + q[:, c + 1, 0].float() * f[0] for c in (0, 2, 4, 6)]
            s32 = (e[0] * g[1] + e[1] * f[1]) * g[2] + (e[2] * g[1] + e[3] * f[1]) * f[2]
            fd = [v.to(f64) for v in f]
            tw = torch.stack([math.prod(fd[i] if (c >> i) & 1 else 1.0 - fd[i] for i in range(3)) for c in range(8)], 1)
            s = (tw[:, :, None] * q.to(f64)).sum(1)
            if flags & 4:
                a32 = s32 * torch.tensor(np.float32(1.0 / 255.0), device=DEV)
                T32[ray] = T32[ray] * (1.0 - a32)
                stop = T32[ray] < torch.tensor(t_min, device=DEV)
                left = 1.0 - s[:, 0] / 255.0
            else:
                tau[ray] = tau[ray] + s32 * torch.tensor(kappa, device=DEV)
                stop = tau[ray] > torch.tensor(tau_max, device=DEV)
                left = torch.exp(-s[:, 0] * float(kappa))
            wk = T[ray] * (1.0 - left)
            T[ray] = T[ray] * left
            acc[ray] += wk[:, None] * (s[:, 1:] / 255.0)
            count[ray] += 1
            done[ray] |= stop
            if flags & 2:
                cv = s[:, 1:] / 255.0
                dr = torch.stack([v[ray] for v in d], 1).to(f64)
                per[ray] += wk[:, None] * (cv[:, :3] + _network(mlp.to(f64), _inputs(cv, dr)))
            if record is not None:
                record.append((ray, torch.stack(where, 1), tw * wk[:, None]))
        k += 1
        live = live[(l0 + (k + 0.5) < l1) & ~done[live]]
    return acc, T, count, per, torch.stack(d, 1).to(f64)


def _shade(case, acc, T, count, per, d, w):
    cv, left = acc, T
    if case["flags"] & 1:
        a = 1.0 - T
        sc = torch.where(a > 0, torch.clamp(1.5 * a, max=1.0) / a.clamp_min(1e-300), torch.ones_like(a))
        cv, left = acc * sc[:, None], 1.0 - a * sc
    if case["flags"] & 2:
        return per + left[:, None] * torch.tensor(BG, dtype=torch.float64, device=DEV)
    rgb = cv[:, :3]
    if not case["flags"] & 8:
        rgb = rgb + torch.where((count > 0)[:, None], _network(w, _inputs(cv, d)), torch.zeros_like(rgb))
    return rgb + left[:, None] * torch.tensor(BG, dtype=torch.float64, device=DEV)


def _gradients(case, ind, atlas, mlp, cams, pix, upstream):
    """rgb, dL/dweights and dL/dvalues for dL/drgb = upstream(rgb)."""
    record = []
    acc, T, count, per, d = _march(case, ind, atlas, mlp, cams, pix, record)
    acc, w = acc.requires_grad_(), mlp.detach().to(torch.float64).requires_grad_()
    rgb = _shade(case, acc, T, count, per, d, w)
    g = upstream(rgb.detach())
    g_acc, g_w = torch.autograd.grad(rgb, (acc, w), g, allow_unused=True)
    g_values = torch.zeros((atlas.numel() // 8, 8), dtype=torch.float64, device=DEV)
    for ray, where, tw in record:
        ok = where >= 0
        v = tw[:, :, None] * g_acc[ray][:, None, :]
        g_values[:, 1:].index_add_(0, where[ok], v[ok])
    return rgb.detach(), torch.zeros_like(w) if g_w is None else g_w, g_values.reshape(atlas.shape)


def _adam(p, g, lr):
    m, v = (1.0 - BETAS[0]) * g, (1.0 - BETAS[1]) * g * g
    return p - lr * (m / (1.0 - BETAS[0])) / (torch.sqrt(v / (1.0 - BETAS[1])) + EPS), m, v


def _exact_bake(case, seed):
    N, B = case["N"], case["B"]
    G, f64 = N // B, torch.float64
    f = {k: torch.from_numpy(v.astype(np.float64)).to(DEV) for k, v in _field(case, seed).items()}
    v = EXTENT / N
    pos = [BMIN[i] + (torch.arange(N, dtype=f64, device=DEV) + 0.5) * v for i in range(3)]
    half = 0.5 / f["blobs"][:, 3] ** 2

    def axis(i, off):               # [blobs, N]: the blob's factor along one axis
        return torch.exp(-half[:, None] * (pos[i] + off - f["blobs"][:, i:i + 1]) ** 2)

    e = [axis(i, 0.0) for i in range(3)]
    top = torch.zeros((G, G, G), dtype=f64, device=DEV)
    for z in range(N):
        s = torch.einsum("by,bx->yx", e[1] * (f["blobs"][:, 4] * e[2][:, z])[:, None], e[0])
        top[z // B] = torch.maximum(top[z // B], s.view(G, B, G, B).amax((1, 3)))
    keep = 1.0 - torch.exp(-top * v) >= float(np.float32(TAU_ALPHA))
    ind = torch.full((G, G, G), -1, dtype=torch.int32, device=DEV)
    ind[keep] = torch.arange(int(keep.sum()), dtype=torch.int32, device=DEV)
    j = f["jitter"] * v
    je = [torch.stack([axis(i, j[s, i]) for s in range(16)], 1) for i in range(3)]      # [blobs, 16, N]
    phase = (f["colors"][:, None, :3] * j[None]).sum(-1)                                  # [7, 16]
    atlas = torch.empty((int(keep.sum()), B, B, B, 8), dtype=torch.uint8, device=DEV)
    for z in range(N):
        bz = z // B
        if not bool(keep[bz].any()):
            continue
        a = (je[2][:, :, z] * f["blobs"][:, 4:5])[:, :, None] * je[1]
        s = (a.reshape(-1, N).T @ je[0].reshape(-1, N)) / 16.0                            # [y, x]
        ch = [1.0 - torch.exp(-s * v) if case["flags"] & 4 else s / float(np.float32(200.0))]
        for c in range(7):
            w = f["colors"][c]
            arg = w[0] * pos[0][None, :] + w[1] * pos[1][:, None] + w[2] * pos[2][z] + w[3]
            ch.append(0.5 + 0.5 * (torch.sin(arg) * torch.cos(phase[c]).mean() + torch.cos(arg) * torch.sin(phase[c]).mean()))
        q = torch.floor(torch.stack(ch, -1) * 255.0 + 0.5).clamp_(0, 255).to(torch.uint8)
        q = q.view(G, B, G, B, 8).permute(0, 2, 1, 3, 4)                                  # [by, bx, y, x, 8]
        atlas[ind[bz][keep[bz]].long(), z % B] = q[keep[bz]]
    return {"ind": ind, "atlas": atlas}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None                 # tens of millions of rays
    if kind == "bake":
        return _exact_bake(case, seed)
    ind, atlas, mlp = _scene(case, seed)
    cams = _cameras(case, seed)
    if kind in ("rays", "noalloc", "autograd", "finetune"):
        pix = _rays(case, cams, seed)
    else:
        pix = torch.from_numpy(synth.all_pixels(cams)).to(DEV)
    if kind == "autograd":
        up = (_values(seed, case["n"]) - 0.5).to(torch.float64)
        rgb, g_mlp, g_values = _gradients(case, ind, atlas, mlp, cams, pix, lambda c: up)
        return {"rgb": rgb, "g_mlp": g_mlp, "g_values": g_values}
    if kind == "finetune":
        target = _values(seed, case["n"]).to(torch.float64)
        rgb, g_mlp, g_values = _gradients(case, ind, atlas, mlp, cams, pix, lambda c: 2.0 * (c - target))
        p, m, v = _adam(mlp.to(torch.float64), g_mlp, LR)
        out = {"loss": ((rgb - target) ** 2).sum().reshape(1), "mlp": p, "m": m, "v": v}
        if case["atlas"]:
            shadow, ma, va = _adam((atlas.float() / 255.0).to(torch.float64), g_values, ATLAS_LR)
            codes = torch.floor(shadow * 255.0 + 0.5).clamp_(0, 255).to(torch.uint8)
            codes[..., 0] = atlas[..., 0]
            out.update(shadow=shadow, ma=ma, va=va, codes=codes)
        return out
    parts = [_shade(case, *_march(case, ind, atlas, mlp, cams, p), mlp.to(torch.float64)) for p in pix.split(1 << 21)]
    rgb = torch.cat(parts)
    if kind == "noalloc":
        return {"rgb": rgb, "status": None}
    return rgb.view(case["frames"], -1, 3) if kind == "orbit" else rgb
