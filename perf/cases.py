"""Timed cases of the rasterizer and the matching stages, through their public entry points.

The workloads are the package's own: an aerial scene of 1 km x 1 km (Gaussians over a rolling ground and in building
clusters) seen from about 300 m at up to 3840x2160, the small scene in front of an identity camera, 32-channel feature
maps, and the dense stage's matching, PnP and localisation. Everything is drawn from the seed, on the GPU.

``exact`` is the same mathematics in 64 bits in plain torch. The choices that define the result (depth order, tile
rectangles, which pixels a Gaussian reaches) are made as the scene's binary32 numbers make them.
"""
import math

import numpy as np
import torch

from paper_2507_15683_gb300 import gsr

AERIAL_VISIBLE = 0.16  # share of the aerial scene that one view sees


# ---- the cases ------------------------------------------------------------------------------------
def listed():
    return [
        # one small preview: launches and latency are all there is
        {"name": "render_tiny", "kind": "render", "scene": "tiny", "n": 1000, "sh": 0, "feat": False, "w": 128, "h": 128},
        # the forward render of a full frame
        {"name": "render_1080p", "kind": "render", "scene": "aerial", "n": 1_000_000, "sh": 3, "feat": False,
         "w": 1920, "h": 1080},
        # candidate views of a coarse search, with the feature map, in one graph launch
        {"name": "features_16x270p", "kind": "render_batch", "scene": "aerial", "n": 2_000_000, "sh": 3, "feat": True,
         "w": 480, "h": 270, "views": 16},
        # one step of a pose optimiser on a small ragged crop, with a pixel mask
        {"name": "grad_ragged", "kind": "grad", "scene": "aerial", "n": 60_000, "sh": 1, "w": 333, "h": 251,
         "weight": True},
        # the headline: loss and pose gradient of a full frame
        {"name": "grad_1080p", "kind": "grad", "scene": "aerial", "n": 1_000_000, "sh": 3, "w": 1920, "h": 1080,
         "weight": False},
        # the pyramid's last level on a large scene, the photo in pinned host memory
        {"name": "grad_host_4k", "kind": "grad_host", "scene": "aerial", "n": 3_000_000, "sh": 3, "w": 3840, "h": 2160,
         "weight": False},
        # eight pose candidates refined together: one batched step
        {"name": "grad_8x540p", "kind": "grad_batch", "scene": "aerial", "n": 500_000, "sh": 3, "w": 960, "h": 540,
         "views": 8},
        # a whole pose refinement with the default options
        {"name": "refine_540p", "kind": "refine", "scene": "aerial", "n": 500_000, "sh": 3, "w": 960, "h": 540},
        # which Gaussians does this view see
        {"name": "visibility_1080p", "kind": "visibility", "scene": "aerial", "n": 1_000_000, "sh": 3, "w": 1920,
         "h": 1080},
        # dense matching of a photo's feature map against a rendered one
        {"name": "match_1080p", "kind": "match", "w": 1920, "h": 1080},
        # the pose from dense matches
        {"name": "pnp_500k", "kind": "pnp", "w": 1920, "h": 1080, "matches": 490_000, "hyps": 128},
        # a whole localisation: three rounds of render, match and PnP
        {"name": "localize_540p", "kind": "localize", "scene": "aerial", "n": 1_000_000, "sh": 3, "feat": True,
         "w": 960, "h": 536, "hyps": 128, "rounds": 3},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["render", "render_batch", "grad", "grad", "grad_host", "grad_batch", "refine", "visibility",
                       "match", "pnp", "localize"])
    w = log(96, 1920)
    c = {"kind": kind, "w": w, "h": max(64, int(w * rng.uniform(0.5, 0.8)))}
    if kind == "match":
        c.update(w=8 * log(16, 240), h=8 * log(12, 135))
    elif kind == "pnp":
        c.update(w=log(160, 1920), h=log(120, 1080), hyps=log(16, 512))
        c["matches"] = log(500, max(1000, min(490_000, c["w"] * c["h"] // 2)))
    else:
        c.update(scene="aerial", n=log(2_000, 1_000_000), sh=rng.randint(0, 3))
        if kind == "render":
            c["feat"] = rng.random() < 0.5
        elif kind in ("grad", "grad_host"):
            c["weight"] = rng.random() < 0.5
        elif kind == "render_batch":
            w = log(96, 640)
            c.update(w=w, h=max(64, int(w * rng.uniform(0.5, 0.8))), views=rng.randint(2, 16), feat=rng.random() < 0.5)
        elif kind == "grad_batch":
            w = log(96, 960)
            c.update(w=w, h=max(64, int(w * rng.uniform(0.5, 0.8))), views=rng.randint(2, 8))
        elif kind == "refine":
            w = log(96, 960)
            c.update(n=log(2_000, 500_000), w=w, h=max(64, int(w * rng.uniform(0.5, 0.6))))
        elif kind == "localize":
            w = 8 * log(24, 160)
            c.update(n=log(200_000, 1_000_000), feat=True, w=w, h=8 * max(12, int(w * rng.uniform(0.5, 0.6)) // 8),
                     hyps=log(32, 256), rounds=rng.randint(2, 3))
    return c


def work(case):
    """Bytes of the inputs read once and the outputs written once, and the operations of the mathematics: per pixel about
    20 blended Gaussians, 12 operations each for colour, depth and transmittance, 64 more with features, and 3 times
    the forward's for a gradient; per similarity of a match 64 + 8."""
    kind, px = case["kind"], case["w"] * case["h"]
    if kind == "match":
        cells = px // 64
        return {"bytes": 2 * 32 * 4 * px + 16 * px, "flops": 72.0 * cells * cells + 72.0 * 4096 * cells * 0.7}
    if kind == "pnp":
        return {"bytes": 32 * case["matches"] + 8 * px, "flops": 30.0 * case["matches"] * 2.3 * case["hyps"]}
    n, views = case["n"], case.get("views", 1)
    vis = n if case["scene"] == "tiny" else AERIAL_VISIBLE * n
    scene = 16 * n + vis * (32 + 12 * (case["sh"] + 1) ** 2 + (64 if case.get("feat") else 0))
    blends = 20.0 * px * views
    if kind in ("render", "render_batch"):
        return {"bytes": scene + views * px * (28 + (128 if case["feat"] else 0)),
                "flops": blends * (12 + (64 if case["feat"] else 0))}
    if kind == "visibility":
        return {"bytes": scene + 37 * n, "flops": blends * 36}
    if kind == "localize":
        cells = px // 64
        r = case["rounds"]
        return {"bytes": scene + 2 * 128 * px * r, "flops": r * (blends * 76 + 72.0 * cells * cells)}
    steps = 50 if kind == "refine" else 1
    return {"bytes": scene + steps * views * px * (16 + (4 if case.get("weight") else 0)),
            "flops": steps * blends * 36}


# ---- inputs ---------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _scene_arrays(case, seed):
    """The scene's arrays, on the GPU."""
    g, n = _gen(seed), case["n"]
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    nrm = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    K = (case["sh"] + 1) ** 2
    sh = nrm(n, K, 3) * 0.05
    sh[:, 0] = rnd(n, 3)
    q = nrm(n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    if case["scene"] == "tiny":
        means = torch.cat([rnd(n, 2) * 4 - 2, rnd(n, 1) * 4 + 4], 1)
        scales, opac = torch.exp(nrm(n, 3) * 0.5 - 3.0), torch.sigmoid(nrm(n))
    else:
        nb = n // 20  # in 500 building clusters; the rest on the ground
        ground = torch.cat([rnd(n - nb, 2) * 1000.0, nrm(n - nb, 1) * 20.0], 1)
        at = (rnd(500, 2) * 1000.0)[(rnd(nb) * 500).long().clamp(max=499)]
        means = torch.cat([ground, torch.cat([at + nrm(nb, 2) * 5.0, rnd(nb, 1) * 60.0], 1)], 0)
        scales, opac = torch.exp(nrm(n, 3) * 0.7 + math.log(0.5)), torch.sigmoid(nrm(n) * 1.5 + 1.0)
    d = {"means": means, "scales": scales, "quats": q, "opacities": opac, "sh": sh, "sh_degree": case["sh"],
         "feats_bf16": None}
    if case.get("feat"):
        f = nrm(n, 32)
        d["feats_bf16"] = (f / f.norm(dim=1, keepdim=True)).to(torch.bfloat16).view(torch.int16)
    return {k: v.contiguous() if isinstance(v, torch.Tensor) else v for k, v in d.items()}


def _look(centre, yaw, pitch):
    """World-to-camera matrix (x right, y down, z forward); yaw 0 = +y, pitch from the nadir."""
    hd = np.array([math.sin(yaw), math.cos(yaw), 0.0])
    fwd = math.cos(pitch) * np.array([0.0, 0.0, -1.0]) + math.sin(pitch) * hd
    right = np.array([math.cos(yaw), -math.sin(yaw), 0.0])
    R = np.stack([right, np.cross(fwd, right), fwd])
    T = np.eye(4)
    T[:3, :3] = R
    T[:3, 3] = -R @ np.asarray(centre, np.float64)
    return T


def _near(T, r, deg, metres):
    """T turned by deg about a random axis through the camera and moved by metres in a random direction."""
    a, d = r.standard_normal(3), r.standard_normal(3)
    a, d = a / np.linalg.norm(a), d / np.linalg.norm(d)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    th = math.radians(deg)
    R = (np.eye(3) + math.sin(th) * K + (1 - math.cos(th)) * K @ K) @ T[:3, :3]
    out = np.eye(4)
    out[:3, :3] = R
    out[:3, 3] = -R @ (-T[:3, :3].T @ T[:3, 3] + metres * d)
    return out


def _camera(case):
    f = 128.0 if case.get("scene") == "tiny" else case["w"] * 1400.0 / 1920.0
    return {"width": case["w"], "height": case["h"], "fx": f, "fy": f, "cx": case["w"] / 2, "cy": case["h"] / 2}


def _poses(case, seed):
    """Per view: the pose that the photo was taken from and the one that is rendered."""
    r = np.random.default_rng(int(seed) + 1)
    if case.get("scene") == "tiny":
        return [(np.eye(4), _near(np.eye(4), r, 1.0, 0.05))]
    out = []
    for _ in range(case.get("views", 1)):
        c = (r.uniform(400, 600), r.uniform(180, 300), r.uniform(280, 320))
        T = _look(c, r.uniform(-0.3, 0.3), math.radians(r.uniform(25, 35)))
        out.append((T, _near(T, r, 2.0, 5.0)))
    return out


def _photo(rgb, depth, seed, view):
    """A photo and its depth from a noiseless render: sensor noise."""
    g = _gen(seed * 101 + view)
    n = torch.randn(4, *depth.shape, generator=g, device="cuda")
    return (rgb.float() + 0.02 * n[:3]).contiguous(), (depth.float() + 0.5 * n[3]).contiguous()


def _weight(case, seed):
    g = _gen(seed + 5)
    return torch.rand(case["h"], case["w"], generator=g, device="cuda") * (
        torch.rand(case["h"], case["w"], generator=g, device="cuda") > 0.2)


def _feature_maps(case, seed):
    """Two 32-channel maps of one scene: smooth fields, the second shifted by a few pixels, both a little noisy."""
    g, h, w = _gen(seed), case["h"], case["w"]
    base = torch.randn(1, 32, h // 5 + 16, w // 5 + 16, generator=g, device="cuda")
    base = torch.nn.functional.interpolate(base, size=(h + 32, w + 32), mode="bilinear", align_corners=False)[0]
    dx, dy = (int(v) for v in np.random.default_rng(int(seed)).integers(2, 20, 2))
    out = []
    for y, x in ((0, 0), (dy, dx)):
        f = base[:, y:y + h, x:x + w] + 0.1 * torch.randn(32, h, w, generator=g, device="cuda")
        out.append((0.2 * f).contiguous())
    return out


def _words(shape, seed):
    return torch.from_numpy(np.random.default_rng(int(seed) + 9).integers(0, 2 ** 32, shape, dtype=np.uint64)
                            .astype(np.uint32).view(np.int32)).cuda()


def _pnp_inputs(case, seed):
    """A rendered depth map, and matches of its pixels with the query's: 70 % true to half a pixel, 30 % wrong."""
    r = np.random.default_rng(int(seed) + 3)
    g, h, w, K = _gen(seed), case["h"], case["w"], case["matches"]
    T = _look((500.0, 200.0, 300.0), 0.0, math.radians(30.0))
    Tq = _near(T, r, 2.0, 5.0)
    cam = _camera(case)
    z = torch.nn.functional.interpolate(300.0 + 60.0 * torch.rand(1, 1, h // 24 + 2, w // 24 + 2, generator=g,
                                                                   device="cuda"), size=(h, w), mode="bilinear")[0, 0]
    alpha = 0.4 + 0.6 * torch.rand(h, w, generator=g, device="cuda")
    depth = (z * alpha).contiguous()
    rp = torch.randperm(h * w, generator=g, device="cuda")[:K].sort().values
    X = _lift(depth, alpha, rp, cam, T)
    p = X @ torch.from_numpy(Tq[:3, :3].T.copy()).cuda() + torch.from_numpy(Tq[:3, 3].copy()).cuda()
    x = torch.floor(p[:, 0] / p[:, 2] * cam["fx"] + cam["cx"]).long()
    y = torch.floor(p[:, 1] / p[:, 2] * cam["fy"] + cam["cy"]).long()
    wrong = (torch.rand(K, generator=g, device="cuda") < 0.3) | (x < 0) | (x >= w) | (y < 0) | (y >= h)
    any_ = torch.randint(0, h * w, (K,), generator=g, device="cuda")
    q = torch.where(wrong, any_, y * w + x)
    m = torch.stack([torch.arange(K, device="cuda"), q, rp], 1).to(torch.int32).contiguous()
    return cam, T, depth, alpha.contiguous(), m, _words((case["hyps"], 3), seed)


def _lift(depth, alpha, rp, cam, T):
    z = depth.reshape(-1)[rp].double() / alpha.reshape(-1)[rp].double()
    w = depth.shape[1]
    d = torch.stack([z * ((rp % w).double() + 0.5 - cam["cx"]) / cam["fx"],
                     z * (torch.div(rp, w, rounding_mode="floor").double() + 0.5 - cam["cy"]) / cam["fy"], z], 1)
    return (d - torch.from_numpy(T[:3, 3].copy()).cuda()) @ torch.from_numpy(T[:3, :3].copy()).cuda()


class State(dict):
    """What a program keeps between calls; its handles are given back with it."""


def prepare(case, seed):
    kind, s = case["kind"], State(case=case)
    if kind == "match":
        s["matcher"] = gsr.Matcher(case["h"], case["w"])
        s["maps"] = _feature_maps(case, seed)
        return s
    if kind == "pnp":
        s["args"] = _pnp_inputs(case, seed)
        s["solver"] = gsr.PnP(case["matches"], case["hyps"])
        return s
    arrays = _scene_arrays(case, seed)
    s["scene"] = S = gsr.Scene(arrays)
    s["cam"] = cam = _camera(case)
    poses = _poses(case, seed)
    s["T"] = [q for _, q in poses]
    s["cams"] = [cam] * len(poses)
    if kind == "render_batch":
        v, h, w = len(poses), case["h"], case["w"]
        new = lambda *sh, **k: torch.empty((v,) + sh, device="cuda", **k)  # noqa: E731
        s["out"] = {"rgb": new(3, h, w), "depth": new(h, w), "alpha": new(h, w), "final_T": new(h, w),
                    "last_idx": new(h, w, dtype=torch.int32)}
        if case["feat"]:
            s["out"]["feats"] = new(32, h, w)
        s["outs"] = [{k: t[i] for k, t in s["out"].items()} for i in range(v)]
        S.render_batch(s["cams"], s["T"], s["outs"])  # a graph launch does not grow the workspace: the first call does
    elif kind in ("grad", "grad_host", "grad_batch", "refine"):
        photos = []
        for i, (T, _) in enumerate(poses):
            o = S.render(cam, T)
            photos.append(_photo(o["rgb"], o["depth"], seed, i))
        s["rgb"], s["depth"] = [p[0] for p in photos], [p[1] for p in photos]
        s["weight"] = _weight(case, seed) if case.get("weight") else None
        if kind == "grad_host":
            for k in ("rgb", "depth"):
                s[k] = [t.cpu().pin_memory() for t in s[k]]
            s["weight"] = None if s["weight"] is None else s["weight"].cpu().pin_memory()
        s["loss"] = gsr.pose_loss_function()
    elif kind == "localize":
        s["query"] = S.render(cam, poses[0][0])["feats"]
        s["matcher"] = gsr.Matcher(case["h"], case["w"])
        s["solver"] = gsr.PnP(case["h"] * case["w"], case["hyps"])
        s["words"] = _words((case["rounds"], case["hyps"], 3), seed)
    return s


def _fixed(t, rows, fill=0):
    """A list of any length as an array of `rows` rows."""
    return torch.nn.functional.pad(t, (0, 0) * (t.dim() - 1) + (0, rows - t.shape[0]), value=fill)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "render":
        return s["scene"].render(s["cam"], s["T"][0])
    if kind == "render_batch":
        s["scene"].render_batch(s["cams"], s["T"], s["outs"], graph=True)
        return s["out"]
    if kind == "grad":  # a torch optimiser's step: the pose's tangent is a float32 parameter
        xi = torch.zeros(6, requires_grad=True)
        loss = s["loss"].apply(xi, s["scene"], s["cam"], s["T"][0], s["rgb"][0], s["depth"][0], s["weight"])
        loss.backward()
        return {"loss": loss.detach(), "grad": xi.grad}
    if kind == "grad_host":  # the images are binary32, and so is the step that the gradient is for
        loss, grad = s["scene"].render_pose_grad_host(s["cam"], s["T"][0], s["rgb"][0], s["depth"][0], s["weight"])
        return {"loss": torch.tensor(loss, dtype=torch.float32), "grad": torch.from_numpy(grad).float()}
    if kind == "grad_batch":
        loss, grad = s["scene"].render_pose_grad_batch(s["cams"], s["T"], s["rgb"], s["depth"])
        return {"loss": torch.from_numpy(loss).float(), "grad": torch.from_numpy(grad).float()}
    if kind == "refine":
        p = gsr.pose(s["T"][0])
        hist = gsr.gs_refine_pose(s["scene"].handle, gsr.camera(s["cam"]), p, s["rgb"][0].data_ptr(),
                                  s["depth"][0].data_ptr(), None, gsr.gs_refine_defaults(),
                                  torch.cuda.current_stream().cuda_stream)
        return {"T": gsr.pose_matrix(p).astype(np.float32), "loss": hist.astype(np.float32)}
    if kind == "visibility":
        r = s["scene"].visibility(s["cam"], s["T"][0])
        r["ids"], r["uv_visible"] = _fixed(r["ids"], case["n"], -1), _fixed(r["uv_visible"], case["n"])
        return r
    if kind == "match":
        r, cells = s["matcher"].match(*s["maps"]), case["h"] * case["w"] // 64
        for k in ("coarse", "coarse_prob", "fine", "fine_prob"):
            r[k] = _fixed(r[k], cells * (64 if "fine" in k else 1), 0 if "prob" in k else -1)
        return r
    if kind == "pnp":
        r = s["solver"].solve(*s["args"])
        found = r["hyp_counts"] >= 0  # a sample without a solution has no pose
        r["hyp_poses"] = torch.where(found[..., None], r["hyp_poses"], 0.0)
        r["valid_index"] = _fixed(r["valid_index"], case["matches"], -1)
        r["points"] = _fixed(r["points"], case["matches"])
        return r
    return gsr.dense_localize(s["scene"], s["matcher"], s["solver"], s["cam"], s["T"][0], s["query"], s["words"],
                              n_rounds=case["rounds"])


# ---- the same in 64 bits --------------------------------------------------------------------------
def _basis(d, deg):
    """Real spherical harmonics of unit vectors, degree by degree."""
    x, y, z = d.unbind(-1)
    Y = [torch.full_like(x, math.sqrt(1 / (4 * math.pi)))]
    if deg >= 1:
        c = math.sqrt(3 / (4 * math.pi))
        Y += [-c * y, c * z, -c * x]
    if deg >= 2:
        a, b, e = math.sqrt(15 / (4 * math.pi)), math.sqrt(5 / (16 * math.pi)), math.sqrt(15 / (16 * math.pi))
        Y += [a * x * y, -a * y * z, b * (3 * z * z - 1), -a * x * z, e * (x * x - y * y)]
    if deg >= 3:
        a, b = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi))
        c, e, f = math.sqrt(21 / (32 * math.pi)), math.sqrt(7 / (16 * math.pi)), math.sqrt(105 / (16 * math.pi))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
              -c * x * (5 * z * z - 1), f * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _skew(v):
    z = torch.zeros_like(v[0])
    return torch.stack([torch.stack([z, -v[2], v[1]]), torch.stack([v[2], z, -v[0]]), torch.stack([-v[1], v[0], z])])


def _splats(a, cam, R, t, deg):
    """Centre, conic, depth and colour of Gaussians (64 bits, differentiable)."""
    q = a["quats"]
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(-1)
    M = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(-1, 3, 3)
    M = M * a["scales"][:, None, :]
    p = a["means"] @ R.T + t
    px, py, pz = p.unbind(-1)
    fx, fy = cam["fx"], cam["fy"]
    lx, ly = 1.3 * 0.5 * cam["width"] / fx, 1.3 * 0.5 * cam["height"] / fy
    zero = torch.zeros_like(pz)
    J = torch.stack([fx / pz, zero, -fx * (px / pz).clamp(-lx, lx) / pz,
                     zero, fy / pz, -fy * (py / pz).clamp(-ly, ly) / pz], -1).view(-1, 2, 3)
    B = J @ (R @ M)
    C = B @ B.transpose(1, 2)
    ca, cb, cc = C[:, 0, 0] + 0.3, C[:, 0, 1], C[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    d = a["means"] + R.T @ t
    d = d / d.norm(dim=1, keepdim=True)
    rgb = ((_basis(d, deg)[..., None] * a["sh"]).sum(1) + 0.5).clamp(min=0)
    return torch.stack([fx * px / pz + cam["cx"], fy * py / pz + cam["cy"], cc / det, -cb / det, ca / det, pz,
                        rgb[:, 0], rgb[:, 1], rgb[:, 2]], -1)


def _tiles(a, cam, T):
    """Tile lists in depth order, from the binary32 projection: (Gaussian of each entry, start of each tile, grid)."""
    R, t = (torch.from_numpy(T[:3, k].astype(np.float32)).cuda() for k in (slice(0, 3), 3))
    m, s, q = a["means"], a["scales"], a["quats"]
    row = lambda k: ((R[k, 0] * m[:, 0] + R[k, 1] * m[:, 1]) + R[k, 2] * m[:, 2]) + t[k]  # noqa: E731
    px, py, pz = row(0), row(1), row(2)
    nr = (((q[:, 0] * q[:, 0] + q[:, 1] * q[:, 1]) + q[:, 2] * q[:, 2]) + q[:, 3] * q[:, 3]).sqrt()
    w, x, y, z = (q[:, k] / nr for k in range(4))
    xx, yy, zz, xy, xz, yz, wx, wy, wz = x * x, y * y, z * z, x * y, x * z, y * z, w * x, w * y, w * z
    r = [[1 - 2 * (yy + zz), 2 * (xy - wz), 2 * (xz + wy)], [2 * (xy + wz), 1 - 2 * (xx + zz), 2 * (yz - wx)],
         [2 * (xz - wy), 2 * (yz + wx), 1 - 2 * (xx + yy)]]
    M = [[r[i][j] * s[:, j] for j in range(3)] for i in range(3)]
    dot = lambda u, v: (u[0] * v[0] + u[1] * v[1]) + u[2] * v[2]  # noqa: E731
    S = [[dot(M[min(i, j)], M[max(i, j)]) for j in range(3)] for i in range(3)]
    f = lambda v: torch.tensor(v, dtype=torch.float32, device="cuda")  # noqa: E731
    fx, fy, cx, cy = f(cam["fx"]), f(cam["fy"]), f(cam["cx"]), f(cam["cy"])
    lx, ly = f(1.3) * (f(0.5 * cam["width"]) / fx), f(1.3) * (f(0.5 * cam["height"]) / fy)
    ix, iy = px / pz, py / pz
    u, v = fx * ix + cx, fy * iy + cy
    xh, yh, pz2 = torch.minimum(lx, torch.maximum(-lx, ix)) * pz, torch.minimum(ly, torch.maximum(-ly, iy)) * pz, pz * pz
    j00, j02, j11, j12 = fx / pz, -((fx * xh) / pz2), fy / pz, -((fy * yh) / pz2)
    A = [[j00 * R[0, k] + j02 * R[2, k] for k in range(3)], [j11 * R[1, k] + j12 * R[2, k] for k in range(3)]]
    U = [[dot(A[i], [S[0][k], S[1][k], S[2][k]]) for k in range(3)] for i in range(2)]
    ca, cb, cc = dot(U[0], A[0]) + 0.3, dot(U[0], A[1]), dot(U[1], A[1]) + 0.3
    det = ca * cc - cb * cb
    mid = 0.5 * (ca + cc)
    rad = torch.ceil(3.0 * (mid + (mid * mid - det).clamp(min=0.1).sqrt()).sqrt())
    tx, ty = (cam["width"] + 15) // 16, (cam["height"] + 15) // 16
    x0, x1 = torch.floor((u - rad) * 0.0625).clamp(min=0), torch.floor((u + rad) * 0.0625).clamp(max=tx - 1)
    y0, y1 = torch.floor((v - rad) * 0.0625).clamp(min=0), torch.floor((v + rad) * 0.0625).clamp(max=ty - 1)
    gid = ((pz >= 0.2) & (det > 0) & (rad > 0) & (x0 <= x1) & (y0 <= y1)).nonzero()[:, 0]
    x0, x1, y0, y1 = (b[gid].long() for b in (x0, x1, y0, y1))
    wide = x1 - x0 + 1
    cnt = wide * (y1 - y0 + 1)
    rec = torch.repeat_interleave(torch.arange(len(gid), device="cuda"), cnt)
    local = torch.arange(len(rec), device="cuda") - (cnt.cumsum(0) - cnt)[rec]
    tile = (y0[rec] + local // wide[rec]) * tx + x0[rec] + local % wide[rec]
    depth = torch.argsort(pz[gid], stable=True)  # positive: the order of the bits; ties by index
    rank = torch.empty_like(depth)
    rank[depth] = torch.arange(len(depth), device="cuda")
    order = torch.argsort(tile * max(1, len(gid)) + rank[rec])
    start = torch.zeros(tx * ty + 1, dtype=torch.long, device="cuda")
    start[1:] = torch.bincount(tile, minlength=tx * ty).cumsum(0)
    return gid, rec[order], start, tx, ty


def _walk(sp, opac, lists, cam, step):
    """Front to back over all tiles at once: step(tiles, records, pixels, alpha, w, e, dx, dy) per list position, where
    e = alpha where it still follows the exponent (below the cap). Returns T and the tiles' pixels."""
    _, rec, start, tx, ty = lists
    n = (start[1:] - start[:-1])
    act = torch.argsort(n, descending=True)
    lane = torch.arange(256, device="cuda")
    X = (torch.arange(tx * ty, device="cuda") % tx)[:, None] * 16 + lane % 16
    Y = torch.div(torch.arange(tx * ty, device="cuda"), tx, rounding_mode="floor")[:, None] * 16 + lane // 16
    out = (X >= cam["width"]) | (Y >= cam["height"])
    Tr = torch.ones(tx * ty, 256, dtype=torch.float64, device="cuda")
    done = out.clone()
    nmax = int(n.max()) if len(n) else 0
    for k in range(nmax):
        if k % 16 == 0:
            act = act[(n[act] > k) & ~done[act].all(1)]
            if not len(act):
                break
            sizes = n[act].cpu().numpy()
        m = int(np.searchsorted(-sizes, -k, side="left"))  # tiles with more than k entries come first
        tl = act[:m]
        if m == 0:
            continue
        r = rec[start[tl] + k]
        s = sp[r]
        dx = s[:, 0:1] - (X[tl] + 0.5)
        dy = s[:, 1:2] - (Y[tl] + 0.5)
        pw = -0.5 * (s[:, 2:3] * dx * dx + s[:, 4:5] * dy * dy) - s[:, 3:4] * dx * dy
        oe = opac[r][:, None] * torch.exp(pw)
        al = oe.clamp(max=0.99)
        T0, d0 = Tr[tl], done[tl]
        take = ~d0 & (pw <= 0) & (al >= 1.0 / 255.0)
        T1 = T0 * (1 - al)
        stop = take & (T1 < 1e-4)
        acc = take & ~stop
        al = torch.where(acc, al, 0.0)
        step(tl, r, s, al, al * T0, torch.where(oe < 0.99, al, 0.0), dx, dy, T0)
        Tr[tl] = torch.where(acc, T1, T0)
        done[tl] = d0 | stop
    return Tr


def _image(t, cam, tx, ty):
    """(tiles, 256, c) to (c, h, w)."""
    c = t.shape[2]
    return (t.view(ty, tx, 16, 16, c).permute(4, 0, 2, 1, 3).reshape(c, ty * 16, tx * 16)
            [:, :cam["height"], :cam["width"]].contiguous())


def _tiled(img, tx, ty):
    """(c, h, w) to (tiles, 256, c), zeros beyond the image."""
    c, h, w = img.shape
    p = torch.zeros(c, ty * 16, tx * 16, dtype=torch.float64, device="cuda")
    p[:, :h, :w] = img
    return p.view(c, ty, 16, tx, 16).permute(1, 3, 2, 4, 0).reshape(ty * tx, 256, c)


def _render64(a, cam, T, deg, keep=False):
    lists = _tiles(a, cam, T)
    gid, _, start, tx, ty = lists
    b = {k: v[gid].double() for k, v in a.items() if k in ("means", "scales", "quats", "opacities", "sh")}
    R, t = (torch.from_numpy(np.ascontiguousarray(T[:3, k])).cuda() for k in (slice(0, 3), 3))
    sp = _splats(b, cam, R, t, deg)
    f = None if a["feats_bf16"] is None else a["feats_bf16"].view(torch.bfloat16)[gid].double()
    acc = torch.zeros(tx * ty, 256, 4, dtype=torch.float64, device="cuda")
    F = None if f is None else torch.zeros(tx * ty, 256, 32, dtype=torch.float64, device="cuda")

    def step(tl, r, s, al, w, e, dx, dy, T0):
        acc[tl] += w[..., None] * torch.cat([s[:, 6:9], s[:, 5:6]], 1)[:, None, :]
        if F is not None:
            F[tl] += w[..., None] * f[r][:, None, :]

    Tr = _walk(sp, b["opacities"], lists, cam, step)
    img = _image(acc, cam, tx, ty)
    Ti = _image(Tr[..., None], cam, tx, ty)[0]
    o = {"rgb": img[:3], "depth": img[3], "alpha": 1 - Ti, "final_T": Ti, "last_idx": None}
    if F is not None:
        o["feats"] = _image(F, cam, tx, ty)
    return (o, lists, b, sp, acc) if keep else o


def _pull(lists, b, sp, cam, G, acc):
    """dL/d(centre, conic, depth, colour) of every listed Gaussian, for pixel gradients G of (r, g, b, depth)."""
    total = (acc * G).sum(2)
    seen = torch.zeros_like(total)
    out = torch.zeros(len(sp), 9, dtype=torch.float64, device="cuda")

    def step(tl, r, s, al, w, e, dx, dy, T0):
        g = G[tl]
        c = (g * torch.cat([s[:, 6:9], s[:, 5:6]], 1)[:, None, :]).sum(2)
        now = seen[tl] + w * c
        seen[tl] = now
        e = e * (T0 * c - (total[tl] - now) / (1 - al))
        A, B, C = s[:, 2:3], s[:, 3:4], s[:, 4:5]
        rows = [-(e * (A * dx + B * dy)), -(e * (B * dx + C * dy)), -0.5 * e * dx * dx, -e * dx * dy, -0.5 * e * dy * dy,
                w * g[..., 3], w * g[..., 0], w * g[..., 1], w * g[..., 2]]
        out.index_add_(0, r, torch.stack([x.sum(1) for x in rows], 1))

    _walk(sp, b["opacities"], lists, cam, step)
    return out


def _grad64(a, cam, T, deg, rgb, depth, weight):
    o, lists, b, sp, acc = _render64(dict(a, feats_bf16=None), cam, T, deg, keep=True)
    px = cam["width"] * cam["height"]
    w = torch.ones_like(o["depth"]) if weight is None else weight.double()
    dr, dd = o["rgb"] - rgb.double(), o["depth"] - depth.double()
    dw = float(np.float32(0.1))
    loss = ((dr.abs().sum(0) / 3 + dw * dd.abs()) * w).sum() / px
    G = torch.cat([dr.sign() * w / (3 * px), (dw * dd.sign() * w / px)[None]])
    ct = _pull(lists, b, sp, cam, _tiled(G, lists[3], lists[4]), acc)
    xi = torch.zeros(6, dtype=torch.float64, device="cuda", requires_grad=True)
    E = torch.eye(3, dtype=torch.float64, device="cuda") + _skew(xi[3:])
    R, t = (torch.from_numpy(np.ascontiguousarray(T[:3, k])).cuda() for k in (slice(0, 3), 3))
    Rx, tx = E @ R, E @ t + xi[:3]
    if len(b["means"]):
        # the camera centre moves with rho alone: -R^T (E^T t + rho) at the first order
        (_splats_at(b, cam, Rx, tx, R, t, xi, deg) * ct).sum().backward()
    return loss, torch.zeros(6) if xi.grad is None else xi.grad


def _splats_at(b, cam, Rx, tx, R, t, xi, deg):
    """_splats at the moved pose, the view direction taken from the moved camera centre."""
    s = _splats(b, cam, Rx, tx, deg)
    d = b["means"] + R.T @ t + R.T @ xi[:3]
    d = d / d.norm(dim=1, keepdim=True)
    rgb = ((_basis(d, deg)[..., None] * b["sh"]).sum(1) + 0.5).clamp(min=0)
    return torch.cat([s[:, :6], rgb], 1)


def _visibility64(a, cam, T, deg):
    n = len(a["means"])
    R, t = (torch.from_numpy(np.ascontiguousarray(T[:3, k])).cuda() for k in (slice(0, 3), 3))
    p = a["means"].double() @ R.T + t
    uv = torch.stack([cam["fx"] * p[:, 0] / p[:, 2] + cam["cx"], cam["fy"] * p[:, 1] / p[:, 2] + cam["cy"]], 1)
    o, lists, b, sp, acc = _render64(a, cam, T, deg, keep=True)
    G = torch.zeros_like(acc)
    G[..., :3] = 1.0
    ct = _pull(lists, b, sp, cam, G, acc)
    m = b["means"].clone().requires_grad_(True)
    (_splats(dict(b, means=m), cam, R, t, deg) * ct).sum().backward()
    grad = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    grad[lists[0]] = m.grad
    return {"mask": None, "uv": uv, "grad": grad, "ids": None, "uv_visible": None, "n_visible": None}


def _match64(fq, fr, tau=0.1):
    def codes(f):
        c, h, w = f.shape
        m = f.double().view(c, h // 8, 8, w // 8, 8).mean((2, 4)).reshape(c, -1).T
        return m / m.norm(dim=1, keepdim=True)

    q, r = codes(fq), codes(fr)
    n, step = len(q), 2048
    lr = torch.cat([torch.logsumexp(q[i:i + step] @ r.T / tau, 1) for i in range(0, n, step)])
    lc = torch.cat([torch.logsumexp(r[i:i + step] @ q.T / tau, 1) for i in range(0, n, step)])
    rb = torch.cat([(2 * (q[i:i + step] @ r.T) / tau - lc).argmax(1) for i in range(0, n, step)])
    cb = torch.cat([(2 * (r[i:i + step] @ q.T) / tau - lr).argmax(1) for i in range(0, n, step)])
    i = (cb[rb] == torch.arange(n, device="cuda")).nonzero()[:, 0]
    prob = torch.exp(2 * (q[i] * r[rb[i]]).sum(1) / tau - lr[i] - lc[rb[i]])
    # the fine level's millions of choices hold near ties: its list has no one value in 64 bits
    return {"codes_q": None, "codes_r": None, "lse_row": lr, "lse_col": lc, "row_best": None, "col_best": None,
            "coarse": None, "coarse_prob": _fixed(prob, n), "fine": None, "fine_prob": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "match":
        return _match64(*_feature_maps(case, seed))
    if kind == "pnp":
        cam, T, depth, alpha, m, _ = _pnp_inputs(case, seed)
        rp = m[:, 2].long()
        # the pose is the end of a search over random samples: only what leads to it has a value of its own
        X = _lift(depth, alpha, rp[alpha.reshape(-1)[rp] >= 0.5], cam, T)
        return {"points": _fixed(X, case["matches"])}
    if kind in ("refine", "localize"):
        return None  # fifty renders and gradients; three whole rounds: far over 20 seconds
    a, cam, poses, deg = _scene_arrays(case, seed), _camera(case), _poses(case, seed), case["sh"]
    if kind == "render":
        return _render64(a, cam, poses[0][1], deg)
    if kind == "visibility":
        return _visibility64(a, cam, poses[0][1], deg)
    if kind == "render_batch":
        o = [_render64(a, cam, T, deg) for _, T in poses]
        return {k: None if o[0][k] is None else torch.stack([x[k] for x in o]) for k in o[0]}
    res = []
    for i, (T, Tq) in enumerate(poses):
        o = _render64(dict(a, feats_bf16=None), cam, T, deg)
        rgb, depth = _photo(o["rgb"], o["depth"], seed, i)
        res.append(_grad64(a, cam, Tq, deg, rgb, depth, _weight(case, seed) if case.get("weight") else None))
    if kind == "grad_batch":
        return {"loss": torch.stack([x for x, _ in res]), "grad": torch.stack([g for _, g in res])}
    return {"loss": res[0][0], "grad": res[0][1]}
