"""The performance cases: what users of the renderer have it do, from the
smallest interactive frame to a 1M-voxel view, each through the public calls.

Scenes are a procedural quadruped (24 joints, capsules, a band of leaf voxels
around their surface) with the sizes of the repository's presets: 3k, 20k,
200k and 1M voxels.  The geometry of a size is fixed; features, densities,
pose, camera and network weights follow the seed.
"""
import functools
import math
import os

import numpy as np
import torch
import torch.nn.functional as nnf

import paper_2202_05628_gb300 as art
from paper_2202_05628_gb300 import proposal as art_proposal

UNET = (32, 64, 128, 256)  # the shading U-Net's widths
OPACITY = (32, 64)         # the opacity branch's
STORE = {"f32": "f32", "bf16": "bf16", "bf16_skip": "bf16", "fp8_skip": "bf16"}  # voxel features of a frame's form
NET = {"f32": "f32", "bf16": "bf16", "bf16_skip": "bf16", "fp8_skip": "fp8"}     # its network's arithmetic


def listed():
    return [
        # the smallest real frame: a 20k-voxel preview at 128 x 128 with the three-layer network, FP32 (launches count)
        dict(name="frame_20k_tiny_f32", kind="frame", form="f32", net="tiny", voxels=20000, C=16, W=128, H=128),
        # the plain FP32 form of a full animal: 1M voxels at 1024 x 1024, U-Net in FP32
        dict(name="frame_1m_f32", kind="frame", form="f32", net="unet", voxels=1000000, C=32, W=1024, H=1024),
        # the product form: BF16 features and network, learned depth interval with its coarse check
        dict(name="frame_1m_bf16_skip", kind="frame", form="bf16_skip", net="unet", voxels=1000000, C=32, W=1024, H=1024),
        # a mid-sized animal in a window of odd proportions (ragged tiles at every level), the FP8 variant
        dict(name="frame_200k_fp8_ragged", kind="frame", form="fp8_skip", net="unet", voxels=200000, C=32, W=712, H=504),
        # the network alone on a full-HD feature map, as a host that renders its own maps calls it
        dict(name="shade_bf16_1080p", kind="shade", form="bf16", net="unet", C=32, W=1920, H=1080),
        # the same in FP32 on a small ragged window
        dict(name="shade_f32_ragged", kind="shade", form="f32", net="unet", C=32, W=424, H=248),
        # the paper's two-branch network (appearance, then opacity from [A, I_f])
        dict(name="shade_two_branch_bf16", kind="shade", form="bf16", net="two_branch", C=32, W=1024, H=1024),
        # feature and opacity maps of a tiny scene at odd sizes, FP32 (a unit test's or a thumbnail's call)
        dict(name="maps_3k_f32_odd", kind="maps", store="f32", voxels=3000, C=8, W=219, H=141),
        # a VR stereo pair in one pass: 1M voxels, two 1920 x 1080 eyes 6.4 cm apart, BF16
        dict(name="stereo_1m_bf16", kind="stereo", store="bf16", voxels=1000000, C=32, W=1920, H=1080),
        # a training step of the feature table: 65,536 rays over 8 views at 512 x 512, forward and backward
        dict(name="step_200k_8views", kind="step", voxels=200000, C=16, W=512, H=512, views=8, rays=8192),
        # view-dependent features (spherical harmonics of degree 2)
        dict(name="sh2_1m_f32", kind="sh", store="f32", degree=2, voxels=1000000, C=32, W=1024, H=1024),
        # the stable (tile, depth) pair sort as a building block, an odd count
        dict(name="sort_900k", kind="sort", pairs=900001, bits=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _window(rng, lo, hi, step):
    """A size with about hi * hi pixels at most, sides in multiples of step."""
    w, h = _log(rng, lo, hi), _log(rng, lo, hi)
    return max(step, w // step * step), max(step, h // step * step)


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "shade", "shade", "maps", "stereo", "step", "sh", "sort"])
    voxels = _log(rng, 3000, 1000000)
    if kind == "frame":
        if rng.random() < 0.2:
            W, H = _window(rng, 61, 260, 1)
            return dict(kind=kind, form="f32", net="tiny", voxels=_log(rng, 3000, 60000), C=rng.choice([8, 16, 32]), W=W, H=H)
        W, H = _window(rng, 64, 1024, 8)
        return dict(kind=kind, form=rng.choice(["f32", "bf16", "bf16_skip", "fp8_skip"]), net="unet", voxels=voxels, C=32, W=W, H=H)
    if kind == "shade":
        W, H = _window(rng, 64, 1024, 8)
        if rng.random() < 0.3:
            return dict(kind=kind, form=rng.choice(["f32", "bf16"]), net="two_branch", C=32, W=W, H=H)
        return dict(kind=kind, form=rng.choice(["f32", "bf16"]), net="unet", C=32, W=W, H=H)
    if kind == "maps":
        W, H = _window(rng, 63, 1024, 1)
        return dict(kind=kind, store=rng.choice(["f32", "f16", "bf16"]), voxels=voxels, C=rng.choice([8, 16, 32]), W=W, H=H)
    if kind == "stereo":
        W, H = _window(rng, 200, 1080, 1)
        return dict(kind=kind, store=rng.choice(["f32", "bf16"]), voxels=voxels, C=32, W=W, H=H)
    if kind == "step":
        side = _log(rng, 64, 512)
        return dict(kind=kind, voxels=_log(rng, 3000, 200000), C=rng.choice([8, 16]), W=side, H=max(63, side - rng.randrange(9)),
                    views=rng.randint(1, 8), rays=max(256, side * side // 32))
    if kind == "sh":
        W, H = _window(rng, 63, 1024, 1)
        return dict(kind=kind, store="f32", degree=rng.randint(0, 2), voxels=voxels, C=rng.choice([8, 16, 32]), W=W, H=H)
    return dict(kind="sort", pairs=_log(rng, 1000, 900001), bits=rng.choice([16, 24, 32]))


# ------------------------------------------------------------------ the scene

# 24 joints: (parent, x, y, z) in template metres; body along +x, up +y.
JOINTS = [(-1, -.100, .200, 0), (0, -.040, .205, 0), (1, .020, .210, 0), (2, .080, .210, 0), (3, .110, .240, 0), (4, .130, .270, 0), (5, .160, .290, 0),
          (3, .080, .180, .045), (7, .085, .110, .045), (8, .080, .040, .045), (9, .095, .012, .045),
          (3, .080, .180, -.045), (11, .085, .110, -.045), (12, .080, .040, -.045), (13, .095, .012, -.045),
          (0, -.100, .180, .045), (15, -.085, .110, .045), (16, -.105, .045, .045), (17, -.090, .012, .045),
          (0, -.100, .180, -.045), (19, -.085, .110, -.045), (20, -.105, .045, -.045), (21, -.090, .012, -.045), (0, -.140, .220, 0)]
TIPS = {24: (.215, .280, 0), 25: (-.230, .265, 0), 26: (.117, .012, .045), 27: (.117, .012, -.045), 28: (-.068, .012, .045), 29: (-.068, .012, -.045)}
TIP_OF = {6: 24, 23: 25, 10: 26, 14: 27, 18: 28, 22: 29}  # leaf joint -> its tip
CAPSULES = [(0, 1, .056), (1, 2, .060), (2, 3, .057), (3, 5, .036), (5, 6, .031), (6, 24, .042),
            (7, 8, .024), (8, 9, .019), (9, 10, .016), (11, 12, .024), (12, 13, .019), (13, 14, .016),
            (15, 16, .026), (16, 17, .020), (17, 18, .016), (19, 20, .026), (20, 21, .020), (21, 22, .016),
            (0, 23, .028), (23, 25, .016), (10, 26, .014), (14, 27, .014), (18, 28, .014), (22, 29, .014)]
PARENT = np.array([j[0] for j in JOINTS], np.int32)


def _distance(p, a, b):
    """Distance of points p [n, 3] to the segment a b."""
    ab = b - a
    t = ((p - a) @ ab / (ab @ ab)).clamp(0.0, 1.0)
    return (p - a - t[:, None] * ab).norm(dim=1)


def _band(points, caps, depth, band):
    """Voxels whose centre lies in the band around the capsules, and their signed distance."""
    h, f = 1.0 / (1 << depth), 8
    nc = (1 << depth) // f

    def sdf(p):
        d = torch.full((len(p),), 1e9, dtype=torch.float64, device="cuda")
        for a, b, r in caps:
            d = torch.minimum(d, _distance(p, points[a], points[b]) - r)
        return d

    g = torch.arange(nc, device="cuda", dtype=torch.float64)
    cells = torch.cartesian_prod(g, g, g)
    d = sdf((cells + 0.5) * (f * h) - 0.5)
    half = 0.5 * math.sqrt(3.0) * f * h
    cells = cells[(d + half >= band[0]) & (d - half <= band[1])]
    s = torch.arange(f, device="cuda", dtype=torch.float64)
    ijk = (cells[:, None] * f + torch.cartesian_prod(s, s, s)[None]).reshape(-1, 3)
    d = sdf((ijk + 0.5) * h - 0.5)
    keep = (d >= band[0]) & (d <= band[1])
    return ijk[keep], d[keep]


@functools.lru_cache(maxsize=6)
def _geometry(voxels):
    """Joints, voxels, skinning and signed distances of the quadruped scaled to about `voxels` leaf voxels in a 1 m cube."""
    depth, band, fur = ((7, (-.02, .02), False) if voxels < 8000 else (8, (-.015, .015), False) if voxels < 60000 else
                        (9, (-.01, .02), True) if voxels < 450000 else (10, (-.01, .02), True))
    raw = np.array([j[1:] for j in JOINTS] + [TIPS[k] for k in sorted(TIPS)])
    raw = raw - 0.5 * (raw.min(0) + raw.max(0))
    scale, best = 0.5, None
    for _ in range(9):
        pts = torch.tensor(raw * scale, device="cuda")
        ijk, sd = _band(pts, [(a, b, 0.3 * r * scale) for a, b, r in CAPSULES], depth, band)
        if best is None or abs(len(ijk) - voxels) < abs(len(best[1]) - voxels):
            best = (pts, ijk, sd)
        if abs(len(ijk) - voxels) <= 0.01 * voxels:
            break
        scale *= math.sqrt(voxels / max(len(ijk), 1))
    pts, ijk, sd = best
    order = torch.argsort((ijk[:, 0] * 4096 + ijk[:, 1]) * 4096 + ijk[:, 2])
    ijk, sd = ijk[order], sd[order]
    centre = (ijk + 0.5) / (1 << depth) - 0.5
    dist = []
    for j in range(24):  # a joint's bone ends at the mean of its children, or at its tip
        kids = [k for k in range(24) if PARENT[k] == j]
        dist.append(_distance(centre, pts[j], pts[kids].mean(0) if kids else pts[TIP_OF[j]]))
    dk, idx = torch.stack(dist, 1).topk(4, dim=1, largest=False)
    w = torch.exp(-0.5 * (dk ** 2 - dk[:, :1] ** 2) / 0.05 ** 2)
    w = (w / w.sum(1, keepdim=True)).float()
    return dict(depth=depth, rest=pts[:24].float().cpu().numpy(), ijk=ijk.to(torch.int32).cpu().numpy().astype(np.uint16),
                jidx=idx.to(torch.uint8).cpu().numpy(), w=(w / w.sum(1, keepdim=True)).cpu().numpy(),
                fade=torch.exp(-sd.clamp(min=0.0) * (math.log(100.0) / 0.02)).float() if fur else None,
                centroid=centre.mean(0).cpu().numpy())


def _pose(rng, walk):
    """A frame of a walk cycle, or random joint rotations of up to 30 degrees."""
    aa = np.zeros((24, 3))
    if not walk:
        ax = rng.standard_normal((24, 3))
        aa = ax / np.linalg.norm(ax, axis=1, keepdims=True) * np.deg2rad(rng.uniform(0.0, 30.0, (24, 1)))
    else:
        ph = 2.0 * math.pi * rng.integers(60) / 60.0
        for top, off in ((7, 0.0), (11, math.pi), (15, math.pi), (19, 0.0)):
            bend = math.radians(10.0) * (1.0 - math.cos(ph + off)) * (-1.0 if top < 15 else 1.0)
            aa[top, 2], aa[top + 1, 2], aa[top + 2, 2] = math.radians(25.0) * math.sin(ph + off), bend, -0.5 * bend
        for j in (1, 2, 3):
            aa[j, 1] = math.radians(5.0) * math.sin(ph + 0.4 * j)
        aa[4, 2], aa[23, 1] = math.radians(6.0) * math.sin(2.0 * ph), math.radians(15.0) * math.sin(ph)
    return aa.astype(np.float32), np.zeros(3, np.float32), np.zeros(3, np.float32)


def _camera(target, W, H, azimuth, shift=0.0):
    """A camera 2 m from the target at 15 degrees elevation, 40 degrees vertical field of view: (fx, fy, cx, cy, [R | t])."""
    az, el = math.radians(azimuth), math.radians(15.0)
    eye = target + 2.0 * np.array([math.cos(el) * math.sin(az), math.sin(el), math.cos(el) * math.cos(az)])
    z = (target - eye) / np.linalg.norm(target - eye)
    x = np.cross(z, (0.0, 1.0, 0.0))
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(z, x), z])
    t = -R @ eye
    t[0] -= shift
    f = float(np.float32(0.5 * H / math.tan(math.radians(20.0))))
    return f, f, 0.5 * W, 0.5 * H, np.concatenate([R, t[:, None]], 1).astype(np.float32)


def _unet_layers(g, cin, ch, cout):
    """(weights [cout][k][k][cin], bias) of a U-Net's layers in execution order, He-normal."""
    shapes, prev = [], cin
    for c in ch:
        shapes, prev = shapes + [(c, prev, 3), (c, c, 3)], c
    for l in range(len(ch) - 2, -1, -1):
        shapes += [(ch[l], ch[l + 1] + ch[l], 3), (ch[l], ch[l], 3)]
    return _layers(g, shapes + [(cout, ch[0], 1)])


def _layers(g, shapes):
    return [((math.sqrt(2.0 / (k * k * ci)) * g.standard_normal((co, k, k, ci))).astype(np.float32),
             (0.05 * g.standard_normal(co)).astype(np.float32)) for co, ci, k in shapes]


def _net_layers(case, seed):
    g, C = np.random.default_rng([seed, 7]), case["C"]
    if case["net"] == "tiny":
        return [_layers(g, [(32, C, 3), (32, 32, 3), (4, 32, 3)])]
    if case["net"] == "two_branch":
        return [_unet_layers(g, C, UNET, 3), _unet_layers(g, 4, OPACITY, 1)]
    return [_unet_layers(g, C, UNET, 4)]


def _inputs(case, seed):
    """What the case's user has: arrays made from the seed alone."""
    rng = np.random.default_rng([seed, 1])
    dev = torch.Generator(device="cuda").manual_seed(seed)
    kind, x = case["kind"], {}
    if kind == "sort":
        n = case["pairs"]
        tile = torch.randint(0, 350, (n,), device="cuda", generator=dev)  # a few hundred busy tiles, 17 bits of depth
        depth = torch.randint(0, 1 << 17, (n,), device="cuda", generator=dev)
        x["keys"] = ((tile * 67 << 17) | depth).to(torch.int32)
        x["vals"] = torch.randperm(n, device="cuda", generator=dev).to(torch.int32)
        return x
    W, H, C = case["W"], case["H"], case["C"]
    if kind in ("frame", "shade"):
        x["layers"] = _net_layers(case, seed)
    if kind == "shade":  # an animal-sized covered region: F of the size the composite gives, zero outside
        yy, xx = torch.meshgrid(torch.linspace(-1, 1, H, device="cuda"), torch.linspace(-1, 1, W, device="cuda"), indexing="ij")
        a, b = rng.uniform(0.3, 0.6, 2)
        A = (1.2 * (1.0 - (xx / a) ** 2 - (yy / b) ** 2)).clamp(0.0, 1.0)
        A = A * (0.7 + 0.3 * torch.rand((H, W), device="cuda", generator=dev))
        x["A"] = A.contiguous()
        x["F"] = (0.4 * A[..., None] * torch.randn((H, W, C), device="cuda", generator=dev)).contiguous()
        return x
    geo = _geometry(case["voxels"])
    n = len(geo["ijk"])
    dens = nnf.softplus(torch.randn(n, device="cuda", generator=dev)) * 20.0
    x["density"] = dens * geo["fade"] if geo["fade"] is not None else dens
    x["features"] = 0.5 * torch.randn((n, C), device="cuda", generator=dev)
    if kind == "sh":
        x["sh"] = 0.5 * torch.randn((n, (case["degree"] + 1) ** 2, C), device="cuda", generator=dev)
    x["geo"], x["pose"] = geo, _pose(rng, walk=kind in ("frame", "stereo"))
    az = 45.0 * rng.integers(8)
    if kind == "stereo":
        x["cams"] = [_camera(geo["centroid"], W, H, az, s) for s in (-0.032, 0.032)]
    else:
        x["cams"] = [_camera(geo["centroid"], W, H, az + 45.0 * v) for v in range(case.get("views", 1))]
    if kind == "step":
        x["target"] = [0.2 * torch.randn((H, W, C), device="cuda", generator=dev) for _ in x["cams"]]
        x["mask"] = [(torch.rand((H, W, 1), device="cuda", generator=dev) < case["rays"] / (W * H)).float() for _ in x["cams"]]
    return x


# ------------------------------------------------------------- the user's calls


def _flat(layers):
    return np.concatenate([art.flat_params(part) for part in layers])


def prepare(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    s = dict(case=case, r=art.Renderer())
    if kind == "sort":
        s["keys"], s["vals"] = x["keys"], x["vals"]
        s["k"], s["v"] = torch.empty_like(x["keys"]), torch.empty_like(x["vals"])
        return s
    r, W, H, C = s["r"], case["W"], case["H"], case["C"]
    if "geo" in x:
        g = x["geo"]
        r.load_octree(g["depth"], np.full(3, -0.5, np.float32), 1.0, g["ijk"], g["jidx"], g["w"], x["features"].cpu().numpy(),
                      x["density"].cpu().numpy(), STORE[case["form"]] if kind == "frame" else case.get("store", "f32"))
        r.load_skeleton(PARENT, g["rest"])
        for v, c in enumerate(x["cams"]):
            r.set_camera(v, W, H, *c, 0.5, 3.5)
        s["pose"] = x["pose"]
    else:
        r.set_camera(0, W, H, *_camera(np.zeros(3), W, H, 0.0), 0.5, 3.5)
    if kind in ("frame", "shade"):
        net, dt = case["net"], NET[case["form"]]
        if net == "tiny":
            r.load_shader(art.ART_NET_TINY, C, [32], 4, _flat(x["layers"]), dt)
        elif net == "unet":
            r.load_shader(art.ART_NET_UNET, C, list(UNET), 4, _flat(x["layers"]), dt)
        else:
            r.load_shader(art.ART_NET_TWO_BRANCH, C, list(UNET), 4, _flat(x["layers"]), dt, list(OPACITY))
        if case["form"].endswith("skip"):
            path = os.path.join(os.path.dirname(art.__file__), "weights", "proposal_quadruped_1m_1024.bin")
            r.load_proposal(art_proposal.load(path)[0])
            r.set_config(skip=art.SKIP_LEARNED, max_missed=1e-3, margin=1)
        s["rgba"] = torch.empty((H, W, 4), device="cuda")
    if kind == "shade":
        s["F"], s["A"] = x["F"].bfloat16() if NET[case["form"]] == "bf16" else x["F"], x["A"]
    if kind in ("maps", "stereo", "sh"):
        r.set_pose(*x["pose"])
        dt = torch.bfloat16 if case["store"] == "bf16" else torch.float32
        s["F"] = [torch.empty((H, W, C), dtype=dt, device="cuda") for _ in x["cams"]]
        s["A"] = [torch.empty((H, W), device="cuda") for _ in x["cams"]]
    if kind == "sh":
        r.load_sh_features(case["degree"], x["sh"])
    if kind == "step":
        s["leaves"] = [x["features"].requires_grad_(), x["density"].requires_grad_(), torch.from_numpy(x["geo"]["w"]).cuda().requires_grad_()]
        s["target"], s["mask"] = x["target"], x["mask"]
    return s


def run(s):
    case, r = s["case"], s["r"]
    kind = case["kind"]
    if kind == "frame":
        r.render_frame(0, *s["pose"], s["rgba"])
        return s["rgba"]
    if kind == "shade":
        dt = NET[case["form"]]
        if case["net"] == "two_branch":
            r.shade_with_opacity(0, s["F"], s["A"], s["rgba"], dt)
        else:
            r.shade(0, s["F"], s["rgba"], dt)
        return s["rgba"]
    if kind in ("maps", "sh", "stereo"):
        dt = "bf16" if case["store"] == "bf16" else "f32"
        r.set_pose(*s["pose"])
        if kind == "stereo":
            r.render_views([0, 1], s["F"], s["A"], dt)
        else:
            r.render_feature_maps(0, s["F"][0], s["A"][0], dt)
        return [*s["F"], *s["A"]]
    if kind == "step":
        F, A, loss = [], [], 0.0
        for v in range(case["views"]):
            f, a = art.render_features(r, v, *s["leaves"], s["pose"])
            loss = loss + ((f - s["target"][v]) * s["mask"][v]).square().sum()
            F.append(f.detach())
            A.append(a.detach())
        return [*F, *A, *torch.autograd.grad(loss, s["leaves"])]
    s["k"].copy_(s["keys"])
    s["v"].copy_(s["vals"])
    r.sort_pairs(s["k"], s["v"], case["bits"])
    return [s["k"], s["v"]]


# ------------------------------------------------------------------------ work


def _unet_macs(W, H, cin, ch, cout):
    """Multiply-adds of a U-Net, the upsampled inputs counted at four taps a pixel (nearest x2 repeats a pixel, so nine taps fold into four)."""
    t, prev = 0, cin
    for l, c in enumerate(ch):
        t, prev = t + (W >> l) * (H >> l) * c * 9 * (prev + c), c
    for l in range(len(ch) - 2, -1, -1):
        t += (W >> l) * (H >> l) * ch[l] * (9 * ch[l] + 4 * ch[l + 1] + 9 * ch[l])
    return t + W * H * ch[0] * cout


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return dict(bytes=16 * case["pairs"], flops=0)
    W, H, C, px = case["W"], case["H"], case["C"], case["W"] * case["H"]
    if kind == "shade" or kind == "frame":
        macs = px * 9 * (32 * C + 32 * 32 + 4 * 32) if case["net"] == "tiny" else _unet_macs(W, H, C, UNET, 4)
        if case["net"] == "two_branch":
            macs += _unet_macs(W, H, 4, OPACITY, 1)
    if kind == "shade":
        return dict(bytes=px * (C * (4 if case["form"] == "f32" else 2) + 16), flops=2 * macs)
    n = case["voxels"]
    voxel = n * (8 + 4 + 16 + 4)  # position, joints, weights, density
    skin = 2 * n * (4 * 12 + 60)  # the blend and its inverse
    if kind == "frame":
        return dict(bytes=voxel + n * C * (4 if case["form"] == "f32" else 2) + 16 * px, flops=2 * macs + skin)
    if kind == "sh":
        return dict(bytes=voxel + n * C * 4 * (case["degree"] + 1) ** 2 + px * (C + 1) * 4, flops=skin)
    if kind == "step":
        return dict(bytes=case["views"] * px * (C * 8 + 8) + 2 * n * (C + 5) * 4 + n * 12, flops=3 * skin)
    es, views = (2 if case["store"] != "f32" else 4), (2 if kind == "stereo" else 1)
    return dict(bytes=voxel + n * C * es + views * px * (C * (2 if case["store"] == "bf16" else 4) + 4), flops=skin)


# ------------------------------------------------ the same in 64 bits, in torch


def _rodrigues(r):
    th = np.linalg.norm(r)
    if th == 0.0:
        return np.eye(3)
    k = r / th
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    return np.eye(3) + math.sin(th) * K + (1.0 - math.cos(th)) * K @ K


def _joint_maps(pose, rest):
    """Per joint the map [24, 3, 4] from its rest to its posed frame."""
    aa, R, T = (np.asarray(v, np.float64) for v in pose)
    rest, M = rest.astype(np.float64), []
    for j in range(24):
        p = PARENT[j]
        Rp, Tp = (_rodrigues(R), T) if p < 0 else M[p]
        off = rest[j] - (rest[p] if p >= 0 else 0.0)
        M.append((Rp @ _rodrigues(aa[j]), Rp @ off + Tp))
    return torch.tensor(np.stack([np.concatenate([m, (t - m @ rest[j])[:, None]], 1) for j, (m, t) in enumerate(M)]), device="cuda")


def _warp(geo, w, pose):
    """Blended maps: (linear part [n, 3, 3], warped centre [n, 3])."""
    A = torch.zeros((len(w), 3, 4), dtype=torch.float64, device="cuda")
    G, jidx = _joint_maps(pose, geo["rest"]), torch.from_numpy(geo["jidx"]).cuda().long()
    for k in range(4):
        A = A + w[:, k, None, None] * G[jidx[:, k]]
    c = (torch.from_numpy(geo["ijk"].astype(np.int32)).cuda().double() + 0.5) / (1 << geo["depth"]) - 0.5
    return A[:, :, :3], (A[:, :, :3] @ c[:, :, None])[:, :, 0] + A[:, :, 3]


def _rays(cam, pix, W):
    fx, fy, cx, cy, M = cam
    M = torch.tensor(M, device="cuda").double()
    dc = torch.stack([(pix % W + 0.5 - cx) / fx, (pix // W + 0.5 - cy) / fy, torch.ones_like(pix, dtype=torch.float64)], 1)
    d = dc @ M[:, :3]
    return -M[:, :3].T @ M[:, 3], d / d.norm(dim=1, keepdim=True)


def _span(lin, cw, o, d, h):
    """Entry and exit distances of rays o + t d through the warped voxels, clipped to [0.5, 3.5]."""
    inv = torch.linalg.inv(lin) * (2.0 / h)
    u, du = (inv @ (o - cw)[:, :, None])[:, :, 0], (inv @ d[:, :, None])[:, :, 0]
    du = torch.where(du == 0.0, torch.full_like(du, 1e-300), du)
    a, b = (-1.0 - u) / du, (1.0 - u) / du
    return torch.minimum(a, b).amax(1).clamp(min=0.5), torch.maximum(a, b).amin(1).clamp(max=3.5)


@torch.no_grad()
def _hits(lin, cw, cam, W, H, h):
    """(voxel, pixel) of every hit, front to back within each pixel."""
    fx, fy, cx, cy, M = cam
    M = torch.tensor(M, device="cuda").double()
    sign = torch.cartesian_prod(*[torch.tensor([-1.0, 1.0], dtype=torch.float64, device="cuda")] * 3) * (0.5 * h)
    X = (cw[:, None] + (lin[:, None] @ sign[None, :, :, None])[..., 0]) @ M[:, :3].T + M[:, 3]
    u, v = X[..., 0] / X[..., 2] * fx + cx, X[..., 1] / X[..., 2] * fy + cy
    x0, x1 = (u.amin(1) - 0.51).ceil().clamp(0, W).long(), (u.amax(1) - 0.49).floor().clamp(-1, W - 1).long()
    y0, y1 = (v.amin(1) - 0.51).ceil().clamp(0, H).long(), (v.amax(1) - 0.49).floor().clamp(-1, H - 1).long()
    ok = (torch.linalg.det(lin) >= 1e-3) & (X[..., 2].amin(1) > 1e-6)
    nx, ny = (x1 - x0 + 1).clamp(min=0) * ok, (y1 - y0 + 1).clamp(min=0)
    cnt = nx * ny
    vid = torch.repeat_interleave(torch.arange(len(cnt), device="cuda"), cnt)
    k = torch.arange(len(vid), device="cuda") - (cnt.cumsum(0) - cnt)[vid]
    pix = (y0[vid] + k // nx[vid]) * W + x0[vid] + k % nx[vid]
    o, d = _rays(cam, pix, W)
    t0, t1 = _span(lin[vid], cw[vid], o, d, h)
    hit = t1 > t0
    vid, pix, t0, t1 = vid[hit], pix[hit], t0[hit], t1[hit]
    for key in (lambda: t1, lambda: t0, lambda: pix):  # by pixel, then entry, then exit, then voxel
        order = torch.argsort(key(), stable=True)
        vid, pix, t0, t1 = vid[order], pix[order], t0[order], t1[order]
    return vid, pix


def _composite(lin, cw, sigma, feat, cam, W, H, h):
    """F [H, W, C] and A [H, W]; feat(voxel, ray direction) gives the hits' features."""
    vid, pix = _hits(lin, cw, cam, W, H, h)
    o, d = _rays(cam, pix, W)
    t0, t1 = _span(lin[vid], cw[vid], o, d, h)
    tau = sigma[vid] * (t1 - t0)
    before = tau.cumsum(0) - tau
    first = torch.zeros(W * H, dtype=torch.long, device="cuda")
    count = torch.bincount(pix, minlength=W * H)
    first[1:] = count.cumsum(0)[:-1]
    before = before - before[first[pix]] if len(pix) else before
    keep = (torch.exp(-before) >= 1e-4).double()  # the stop comes after the hit that crosses it
    w = torch.exp(-before) * -torch.expm1(-tau) * keep
    f = feat(vid, d)
    F = torch.zeros((W * H, f.shape[1]), dtype=torch.float64, device="cuda").index_add(0, pix, w[:, None] * f)
    s = torch.zeros(W * H, dtype=torch.float64, device="cuda").index_add(0, pix, tau * keep)
    return F.reshape(H, W, -1), -torch.expm1(-s).reshape(H, W)


def _conv(x, layer, act):
    w, b = (torch.from_numpy(v).cuda().double() for v in layer)
    y = nnf.conv2d(x, w.permute(0, 3, 1, 2), b, padding=w.shape[1] // 2)
    return y.relu() if act else y.sigmoid()


def _unet(x, layers, levels):
    it, skip = iter(layers), []
    for l in range(levels):
        x = _conv(_conv(x, next(it), True), next(it), True)
        if l + 1 < levels:
            skip.append(x)
            x = nnf.max_pool2d(x, 2)
    for s in reversed(skip):
        x = torch.cat([nnf.interpolate(x, scale_factor=2, mode="nearest"), s], 1)
        x = _conv(_conv(x, next(it), True), next(it), True)
    return _conv(x, next(it), False)


def _shade(case, layers, F, A):
    x = F.permute(2, 0, 1)[None]
    if case["net"] == "tiny":
        y = _conv(_conv(_conv(x, layers[0][0], True), layers[0][1], True), layers[0][2], False)
    else:
        y = _unet(x, layers[0], 4)
        if case["net"] == "two_branch":
            y = torch.cat([y, _unet(torch.cat([A[None, None], y], 1), layers[1], 2)], 1)
    return y[0].permute(1, 2, 0).contiguous()


def _harmonics(degree, d):
    """Real orthonormal spherical harmonics without the Condon-Shortley phase, [hits, (degree + 1)^2], degree <= 2."""
    x, y, z = d.unbind(1)
    c0, c1, c2 = math.sqrt(0.25 / math.pi), math.sqrt(0.75 / math.pi), math.sqrt(3.75 / math.pi)
    Y = [torch.full_like(x, c0), c1 * y, c1 * z, c1 * x, c2 * x * y, c2 * y * z, math.sqrt(0.3125 / math.pi) * (3.0 * z * z - 1.0),
         c2 * x * z, 0.5 * c2 * (x * x - y * y)]
    return torch.stack(Y[:(degree + 1) ** 2], 1)


def exact(case, seed):
    if case["kind"] == "sort":
        return None
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "shade":
        F = x["F"].bfloat16() if NET[case["form"]] == "bf16" else x["F"]
        return _shade(case, x["layers"], F.double(), x["A"].double())
    W, H, geo = case["W"], case["H"], x["geo"]
    h = 1.0 / (1 << geo["depth"])
    leaves = [x["features"].double(), x["density"].double(), torch.from_numpy(geo["w"]).cuda().double()]
    for v in leaves:
        v.requires_grad_(kind == "step")
    f, sigma, w = leaves
    lin, cw = _warp(geo, w, x["pose"])
    if kind == "sh":
        U, _, Vh = torch.linalg.svd(lin.cpu())  # R^T of the polar decomposition lin = R S maps a ray into the canonical frame
        rot = (U @ Vh).cuda()

        def feat(vid, d):
            Y = _harmonics(case["degree"], (d[:, None] @ rot[vid])[:, 0])
            out = torch.zeros((len(vid), case["C"]), dtype=torch.float64, device="cuda")
            for k in range(Y.shape[1]):
                out += Y[:, k, None] * x["sh"][vid, k].double()
            return out
    else:
        def feat(vid, d):
            return f[vid]
    maps = [_composite(lin, cw, sigma, feat, c, W, H, h) for c in x["cams"]]
    if kind == "frame":
        return _shade(case, x["layers"], *maps[0])
    F, A = [m[0] for m in maps], [m[1] for m in maps]
    if kind == "step":
        loss = sum(((a - t) * m).square().sum() for a, t, m in zip(F, x["target"], x["mask"]))
        return [v.detach() for v in F + A] + list(torch.autograd.grad(loss, leaves))
    return F + A
