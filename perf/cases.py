"""Performance cases of the tracking library: what a user's program has it do.

A case is one call (or the short fixed sequence of calls a tracking thread
makes) through the C ABI on device-resident inputs, from the smallest call (one
camera, one frame, where latency counts) to the largest batch (32 full-HD
frames with 100 000 map points each).  Sizes are those of the repository's
workloads: 752x480 pinhole frames, 512x512 fisheye frames, 1920x1080 stress
frames, and the 640x480 to 1280x720 camera streams of the served loop with 500
to 4000 keypoints and 1000 to 20 000 map points.

Kinds of case:
  stereo    ft_stereo_match_pinhole of one frame
  fisheye   ft_stereo_match_fisheye of one frame (with triangulation)
  search    ft_search_local_points of one pinhole frame
  pose      ft_optimize_pose of one frame's matches
  extract   ft_extract_orb of a call's images
  track     ft_track_batch: stereo matching and search of every frame in one
            launch; options: the last frame's points instead of the local map,
            pose optimization after the search, pyramids built from level 0
  trackfish ft_track_batch of fisheye frames

Images are either "scene" (overlapping flat shapes with power-law sizes, a
mild texture, blur and sensor noise: edges and corners about as frequent as in
indoor and outdoor footage) or "texture" (band-limited noise: foliage, gravel,
carpet; about a third of its pixels are corners).

Inputs are drawn on the GPU from the seed.  exact() evaluates the floating
point outputs in 64 bits with torch alone.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch
import torch.nn.functional as TF

from paper_2509_10757_gb300 import _lib as L
from paper_2509_10757_gb300 import scenes
from paper_2509_10757_gb300.batch import Context, OrbOutputs, pinhole_struct, pose_struct, rig_struct, stream_handle

NL = 8                                   # pyramid levels
SC32 = scenes.level_scales32()           # the FP32 level scales the interface defines
DEV = "cuda"


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # one frame of a small camera: only the stereo step (depth for new keypoints)
        dict(name="stereo_640x480", kind="stereo", w=640, h=480, left=500, content="scene"),
        # one fisheye frame at full size: brute-force matching of the overlap, triangulation
        dict(name="fisheye_512x512", kind="fisheye", left=1500),
        # relocalization against a large map in a 720p frame: keypoints beyond the on-chip stage
        dict(name="search_1280x720", kind="search", w=1280, h=720, left=4000, points=20000),
        # motion-only refinement of one frame's pose
        dict(name="pose_752x480", kind="pose", w=752, h=480, left=1200, points=3000),
        # one camera live: a frame at a time through the fused call
        dict(name="track_1", kind="track", frames=1, w=752, h=480, left=1200, points=3000, last=False, pose=False,
             images=False, content="scene"),
        # a few cameras, motion-model tracking: the last frame's points, then the pose
        dict(name="track_last_pose_16", kind="track", frames=16, w=752, h=480, left=1250, points=1800, last=True,
             pose=True, images=False, content="texture"),
        # many cameras of one server: the batched workload
        dict(name="track_64", kind="track", frames=64, w=752, h=480, left=1250, points=3500, last=False, pose=False,
             images=False, content="texture"),
        # the same server when only level-0 images are on the device: pyramids, tracking, pose
        dict(name="track_images_pose_64", kind="track", frames=64, w=752, h=480, left=1250, points=3500, last=False,
             pose=True, images=True, content="scene"),
        # many fisheye rigs of one server
        dict(name="track_fisheye_32", kind="trackfish", frames=32, left=1500, points=6000),
        # full-HD cameras with dense keypoints against large maps
        dict(name="track_1080p_32", kind="track", frames=32, w=1920, h=1080, left=8000, points=100000, last=False,
             pose=False, images=False, content="texture"),
        # one stereo pair through the keypoint extractor
        dict(name="extract_2", kind="extract", images=2, w=752, h=480, slots=1200, content="texture"),
        # the server's 64 stereo pairs through the keypoint extractor
        dict(name="extract_128", kind="extract", images=128, w=752, h=480, slots=1200, content="scene"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng):
    """An image size of the served shapes, or an odd one in their range."""
    if rng.random() < 0.5:
        return rng.choice([(640, 480), (752, 480), (1280, 720)])
    return rng.randint(400, 1281), rng.randint(300, 721)


def draw(rng):
    kind = rng.choice(["stereo", "fisheye", "search", "pose", "track", "track", "trackfish", "extract"])
    content = rng.choice(["scene", "texture"])
    if kind == "fisheye":
        return dict(kind=kind, left=_log_int(rng, 300, 4000))
    if kind == "trackfish":
        return dict(kind=kind, frames=_log_int(rng, 1, 32), left=_log_int(rng, 500, 2000),
                    points=_log_int(rng, 1000, 8000))
    w, h = _size(rng)
    if kind == "stereo":
        return dict(kind=kind, w=w, h=h, left=_log_int(rng, 300, 4000), content=content)
    if kind == "search":
        return dict(kind=kind, w=w, h=h, left=_log_int(rng, 500, 4000), points=_log_int(rng, 1000, 20000))
    if kind == "pose":
        return dict(kind=kind, w=w, h=h, left=_log_int(rng, 500, 4000), points=_log_int(rng, 1000, 8000))
    if kind == "extract":
        return dict(kind=kind, images=_log_int(rng, 1, 48), w=w, h=h, slots=_log_int(rng, 500, 2000), content=content)
    return dict(kind=kind, frames=_log_int(rng, 1, 64), w=w, h=h, left=_log_int(rng, 500, 2500),
                points=_log_int(rng, 1000, 12000), last=rng.random() < 0.3, pose=rng.random() < 0.4,
                images=rng.random() < 0.3, content=content)


# --------------------------------------------------------------------------
# random inputs, on the GPU
# --------------------------------------------------------------------------
class Rand:
    """Seeded draws on the device (and a few scalars on the host)."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 7919 + 13)
        self.np = np.random.default_rng(int(seed))

    def uni(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def ints(self, lo, hi, *shape):
        return torch.randint(lo, hi, shape, generator=self.g, device=DEV)

    def octaves(self, n):
        p = torch.as_tensor(scenes.octave_probs(), device=DEV)
        return torch.multinomial(p, n, replacement=True, generator=self.g)

    def desc(self, n):
        return self.ints(0, 256, n, 32).to(torch.uint8)

    def flipped(self, desc, p):
        """Descriptors with each bit flipped with probability p."""
        bits = torch.rand((desc.shape[0], 32, 8), generator=self.g, device=DEV) < p
        w = (1 << torch.arange(8, device=DEV)).to(torch.uint8)
        return desc ^ (bits.to(torch.uint8) * w).sum(-1).to(torch.uint8)

    def perm(self, n):
        return torch.randperm(n, generator=self.g, device=DEV)


def _blur(img, sigma):
    r = int(math.ceil(3 * sigma))
    x = torch.arange(-r, r + 1, device=DEV, dtype=torch.float32)
    k = torch.exp(-0.5 * (x / sigma) ** 2)
    k = k / k.sum()
    img = TF.pad(img[:, None], (r, r, r, r), mode="reflect")
    img = TF.conv2d(TF.conv2d(img, k.view(1, 1, 1, -1)), k.view(1, 1, -1, 1))
    return img[:, 0]


def _bytes(img):
    return img.round().clamp(0, 255).to(torch.uint8)


def _images(R, n, w, h, content):
    """n images (uint8) of one kind of content."""
    noise = _blur(torch.randn((n, h, w), generator=R.g, device=DEV), 1.5)
    noise = (noise - noise.mean()) / noise.std()
    if content == "texture":
        return _bytes(128 + 45 * noise)
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    img = (R.uni(60, 190, n, 1, 1) + R.uni(-60, 60, n, 1, 1) * xx / w).float()
    shapes = 400
    size = (8 * (1 - R.uni(0, 1, shapes, n, 1, 1) * (1 - (8 / (w / 4)) ** 2)) ** -0.5).float()
    aspect, ang = R.uni(0.3, 1, shapes, n, 1, 1).float(), R.uni(0, math.pi, shapes, n, 1, 1)
    cx, cy = R.uni(0, w, shapes, n, 1, 1).float(), R.uni(0, h, shapes, n, 1, 1).float()
    val, box = R.uni(15, 240, shapes, n, 1, 1).float(), R.uni(0, 1, shapes, n, 1, 1) < 0.6
    c, s = torch.cos(ang).float(), torch.sin(ang).float()
    for i in range(shapes):
        dx, dy = xx - cx[i], yy - cy[i]
        u, v = (c[i] * dx + s[i] * dy) / size[i], (c[i] * dy - s[i] * dx) / (size[i] * aspect[i])
        inside = torch.where(box[i], torch.maximum(u.abs(), v.abs()) < 1, u * u + v * v < 1)
        img = torch.where(inside, val[i], img)
    img = _blur(img + 12 * noise, 0.7)
    return _bytes(img + 2 * torch.randn(img.shape, generator=R.g, device=DEV))


def _stereo_scenes(R, n, cam, content):
    """n scenes: left and right images, plane labels per left pixel, plane depths."""
    w, h = cam.width, cam.height
    left = _images(R, n, w, h, content)
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    out = []
    for i in range(n):
        sx, sy, depth = R.uni(0, w, 6), R.uni(0, h, 6), R.uni(1, 10, 6)
        label = ((xx[..., None] - sx) ** 2 + (yy[..., None] - sy) ** 2).argmin(-1)
        disp = cam.fx * cam.b / depth
        best = torch.full((h, w), math.inf, device=DEV, dtype=torch.float64)
        src = torch.full((h, w), -1.0, device=DEV, dtype=torch.float64)
        for k in range(6):
            xl = xx + disp[k]
            xi = xl.round().long()
            seen = (xi < w) & (label.gather(1, xi.clamp(max=w - 1)) == k) & (depth[k] < best)
            best = torch.where(seen, depth[k], best)
            src = torch.where(seen, xl, src)
        x0 = src.clamp(0, w - 1).floor().long()
        f = (src - x0).clamp(0, 1)
        lf = left[i].double()
        right = lf.gather(1, x0) * (1 - f) + lf.gather(1, (x0 + 1).clamp(max=w - 1)) * f
        right = torch.where(src >= 0, right, R.uni(0, 255, h, w)) + 2 * R.normal(h, w)
        out.append((left[i], _bytes(right), label, depth))
    return out


def _pyramid_layout(w, h):
    """Per level (width, height, pitch, offset), then the bytes of all levels."""
    levels, total = [], 0
    for sc in SC32:
        lw, lh = int(math.floor(np.float32(w) / sc + 0.5)), int(math.floor(np.float32(h) / sc + 0.5))
        pitch = (lw + 15) // 16 * 16
        levels.append((lw, lh, pitch, total))
        total += (pitch * lh + 255) // 256 * 256
    return levels, total


class Pyramid:
    """An image's levels in one buffer (rows padded to 16 bytes) and their
    struct; not filled: only level 0 is there."""

    def __init__(self, img, buf=None, filled=True):
        layout, total = _pyramid_layout(img.shape[1], img.shape[0])
        self.buf = torch.zeros(total, dtype=torch.uint8, device=DEV) if buf is None else buf
        self.levels = []
        p = self.struct = L.ft_pyramid()
        p.nlevels = NL
        for l, (lw, lh, pitch, off) in enumerate(layout):
            rows = self.buf[off:off + pitch * lh].view(lh, pitch)
            if l == 0:
                rows[:, :lw] = img
            elif filled:
                f = TF.interpolate(img[None, None].float(), size=(lh, lw), mode="bilinear", align_corners=False)
                rows[:, :lw] = _bytes(f[0, 0])
            self.levels.append(rows[:, :lw])
            p.data[l], p.width[l], p.height[l], p.pitch[l] = rows.data_ptr(), lw, lh, pitch


def _keypoints(R, n, w, h):
    """Random level pixels: x, y (FP32, level 0), octave."""
    o = R.octaves(n)
    sc = torch.as_tensor(SC32, device=DEV)[o]
    lw, lh = (w / sc + 0.5).floor(), (h / sc + 0.5).floor()
    u, v = (R.uni(0, 1, n) * lw).floor().float(), (R.uni(0, 1, n) * lh).floor().float()
    return u * sc, v * sc, o


class Keypoints:
    def __init__(self, x, y, o, desc):
        self.x, self.y = x.float().contiguous(), y.float().contiguous()
        self.oct, self.desc = o.to(torch.int8).contiguous(), desc.contiguous()
        self.n = len(self.x)

    def struct(self):
        return L.ft_keypoints(self.n, self.x.data_ptr(), self.y.data_ptr(), self.oct.data_ptr(), self.desc.data_ptr())


def _poses(R):
    """The true pose and the tracker's estimate of it (2 cm and 0.5 degrees off)."""
    rot = scenes.random_rotation(R.np, 10.0)
    centre = R.np.normal(0.0, 1.0, 3)
    return rot, centre, scenes.make_pose(*scenes.perturb_pose(R.np, rot, centre))


def _local_map(R, n, unproject, w, h, rot, centre, kps, depth, flip_p):
    """Map points: 60 % behind keypoints, the rest random; some behind the
    camera, outside the image or facing away.  Returns pos, nrm, desc, skip,
    octave and the keypoint of each point (-1: none)."""
    na = min(int(0.6 * n), kps.n)
    pick = R.perm(kps.n)[:na]
    u = torch.cat([kps.x[pick].double(), R.uni(0, w, n - na)])
    v = torch.cat([kps.y[pick].double(), R.uni(0, h, n - na)])
    z = torch.cat([depth[pick], R.uni(1, 10, n - na)])
    octave = torch.cat([kps.oct[pick].long(), R.octaves(n - na)])
    desc = torch.cat([R.flipped(kps.desc[pick], flip_p), R.desc(n - na)])
    rt, ct = torch.as_tensor(rot, device=DEV), torch.as_tensor(centre, device=DEV)
    P = unproject(u, v, z) @ rt + ct
    bad = R.uni(0, 1, n)[:, None]
    P = torch.where(bad < 0.03, 2 * ct - P, P)
    P = torch.where((bad >= 0.03) & (bad < 0.06), P + 3 * rt[0] * z[:, None], P)
    view = P - ct
    dist = view.norm(dim=1, keepdim=True)
    view = view / dist
    a = torch.linalg.cross(view, R.normal(n, 3))
    a = a / (a.norm(dim=1, keepdim=True) + 1e-12)
    th = math.radians(25.0) * R.uni(0, 1, n)[:, None]
    nrm = view * torch.cos(th) + torch.linalg.cross(a, view) * torch.sin(th)
    nrm = torch.where(R.uni(0, 1, n)[:, None] < 0.04, -nrm, nrm)
    dmax = dist[:, 0] * 1.2 ** octave.double() * R.uni(0.9, 1.1, n)
    pos = torch.cat([P, (dmax / 1.2 ** (NL - 1))[:, None]], 1).float().contiguous()
    nrm = torch.cat([nrm, dmax[:, None]], 1).float().contiguous()
    skip = (R.uni(0, 1, n) < 0.05).to(torch.uint8)
    owner = torch.cat([pick, torch.full((n - na,), -1, device=DEV)])
    return dict(pos=pos, nrm=nrm, desc=desc.contiguous(), skip=skip, oct=octave, owner=owner, n=n)


def _pinhole_frame(R, cam, scene, n_left, n_map, dense):
    """One frame as a tracker has it before the call: keypoints of both images,
    taken flags, poses, local map."""
    w, h = cam.width, cam.height
    distract, flip = (0.4, 0.08) if dense else (0.2, 0.05)
    x, y, o = _keypoints(R, n_left, w, h)
    desc = R.desc(n_left)
    if scene is None:
        z = R.uni(1, 10, n_left)
    else:
        z = scene[3][scene[2][y.round().long().clamp(0, h - 1), x.round().long().clamp(0, w - 1)]]
    left = Keypoints(x, y, o, desc)
    sc = torch.as_tensor(SC32, device=DEV)[o]
    xr = x.double() - cam.fx * cam.b / z
    keep = xr >= 0
    xt = ((xr / sc).round().float() * sc)[keep]
    nd = int(round(distract * n_left))
    dx, dy, do = _keypoints(R, nd, w, h)
    perm = R.perm(len(xt) + nd)
    right = Keypoints(torch.cat([xt, dx])[perm], torch.cat([y[keep], dy])[perm], torch.cat([o[keep], do])[perm],
                      torch.cat([R.flipped(desc[keep], flip), R.desc(nd)])[perm])
    rot, centre, pose = _poses(R)

    def unproject(u, v, zz):
        return torch.stack([(u - cam.cx) / cam.fx * zz, (v - cam.cy) / cam.fy * zz, zz], 1)

    m = _local_map(R, n_map, unproject, w, h, rot, centre, left, z, flip)
    taken = (R.uni(0, 1, n_left) < 0.1).to(torch.uint8)
    return dict(left=left, right=right, pose=pose, map=m, taken=taken, depth=z)


def _last_points(R, m, pose):
    """The last frame's points: the map's with their octaves as last observed,
    and the last pose (2 cm to the side)."""
    n = m["n"]
    o = (m["oct"] + R.ints(-1, 2, n)).clamp(0, NL - 1)
    o = torch.where(R.uni(0, 1, n) < 0.02, torch.full_like(o, -1), o).to(torch.int8)
    rot = pose.R.reshape(3, 3).astype(np.float64)
    last = scenes.make_pose(rot, pose.O.astype(np.float64) + 0.02 * rot[0])
    v = L.ft_last_frame_view(n, m["pos"].data_ptr(), m["desc"].data_ptr(), o.data_ptr(), m["skip"].data_ptr(),
                             pose_struct(last))
    return dict(oct=o, view=v)


def _kb8_theta(cam, u, v):
    """Normalized pixel, its radius, the ray's angle to the axis, and where the
    lens model has such an angle (at most 2 rad, where the model still rises)."""
    mx, my = (u - cam.cx) / cam.fx, (v - cam.cy) / cam.fy
    thd = torch.hypot(mx, my)
    k = [float(x) for x in cam.k]
    th = thd.clone()
    for _ in range(20):
        t = th * th
        f = th * (1 + t * (k[0] + t * (k[1] + t * (k[2] + t * k[3])))) - thd
        slope = 1 + t * (3 * k[0] + t * (5 * k[1] + t * (7 * k[2] + t * 9 * k[3])))
        th = th - f / slope
    return mx, my, thd, th, (f.abs() <= 2e-6) & (slope > 0) & (th >= 0) & (th <= 2)


def _kb8_unproject(cam, u, v, dist):
    mx, my, thd, th, _ = _kb8_theta(cam, u, v)
    s = torch.where(thd > 0, torch.sin(th) / thd.clamp(min=1e-300), torch.ones_like(thd))
    return torch.stack([mx * s, my * s, torch.cos(th)], 1) * dist[:, None]


def _kb8_project(cam, P):
    rho = torch.hypot(P[:, 0], P[:, 1])
    th = torch.atan2(rho, P[:, 2])
    t = th * th
    k = [float(x) for x in cam.k]
    s = th * (1 + t * (k[0] + t * (k[1] + t * (k[2] + t * k[3])))) / rho.clamp(min=1e-300)
    s = torch.where(rho > 0, s, torch.zeros_like(s))
    return cam.fx * P[:, 0] * s + cam.cx, cam.fy * P[:, 1] * s + cam.cy


def _fisheye_frame(R, rig, n_left, n_map):
    """One fisheye frame: 60 % of the left keypoints in the overlap with a true
    right keypoint, right distractors up to the left count."""
    w, h = rig.left.width, rig.left.height
    nov = int(round(0.6 * n_left))
    x = torch.cat([R.uni(rig.lap_l0, rig.lap_l1, nov), R.uni(0, rig.lap_l0 - 1, n_left - nov)])
    y, o, desc, dist = R.uni(0, h - 1, n_left), R.octaves(n_left), R.desc(n_left), R.uni(1, 10, n_left)
    order = R.perm(n_left)
    x = x[order].float()
    left = Keypoints(x, y, o, desc)
    Rrl = torch.as_tensor(rig.R_rl, device=DEV).double().view(3, 3)
    trl = torch.as_tensor(rig.t_rl, device=DEV).double()
    Pr = _kb8_unproject(rig.left, left.x.double(), left.y.double(), dist) @ Rrl.T + trl
    ur, vr = _kb8_project(rig.right, Pr)
    ok = ((order < nov) & (Pr[:, 2] > 0.1) & (ur >= rig.lap_r0) & (ur <= rig.lap_r1) & (vr >= 0) & (vr < h))
    true = ok.nonzero()[:, 0]
    nd = n_left - len(true)
    perm = R.perm(n_left)
    right = Keypoints(torch.cat([ur[true], R.uni(0, w - 1, nd)])[perm], torch.cat([vr[true], R.uni(0, h - 1, nd)])[perm],
                      torch.cat([o[true], R.octaves(nd)])[perm],
                      torch.cat([R.flipped(desc[true], 0.05), R.desc(nd)])[perm])
    rot, centre, pose = _poses(R)
    m = _local_map(R, n_map, lambda a, b, d: _kb8_unproject(rig.left, a, b, d), w, h, rot, centre, left, dist, 0.05)
    c_rl = -rig.R_rl.reshape(3, 3).T.astype(np.float64) @ rig.t_rl
    O_right = (pose.O + pose.R.reshape(3, 3).T @ c_rl).astype(np.float32)
    return dict(left=left, right=right, pose=pose, map=m, O_right=O_right,
                taken=(R.uni(0, 1, n_left) < 0.1).to(torch.uint8),
                taken_r=(R.uni(0, 1, n_left) < 0.1).to(torch.uint8))


# --------------------------------------------------------------------------
# outputs: one tensor per kind of output, every frame's part at a multiple of
# 16 entries
# --------------------------------------------------------------------------
class Outputs:
    def __init__(self):
        self.size, self.type, self.tail, self.at, self.t = {}, {}, {}, {}, {}

    def want(self, frame, name, n, dtype, *tail):
        off = self.size.get(name, 0)
        self.at[frame, name] = (off, n)
        self.size[name] = off + (n + 15) // 16 * 16
        self.type[name], self.tail[name] = dtype, tail

    def make(self):
        for k, n in self.size.items():
            self.t[k] = torch.zeros((max(n, 16),) + self.tail[k], dtype=self.type[k], device=DEV)

    def ptr(self, frame, name):
        t = self.t[name]
        return t.data_ptr() + self.at[frame, name][0] * t[0].numel() * t.element_size()

    def of(self, frame, name):
        off, n = self.at[frame, name]
        return self.t[name][off:off + n]


I32, F32, I8 = torch.int32, torch.float32, torch.int8
STEREO = (("best_r", I32), ("dist", I32), ("sad_shift", I32), ("sad_best", I32), ("u_right", F32), ("depth", F32))


def _want_search(o, f, side, n_map, n_kp):
    o.want(f, "level_" + side, n_map, I8)
    o.want(f, "proj_" + side, n_map, F32, 4)
    for k in ("mp_kp_", "mp_d1_", "mp_d2_"):
        o.want(f, k + side, n_map, I32)
    o.want(f, "kp_mp_" + side, n_kp, I32)


def _search_cam(o, f, side):
    return L.ft_search_cam_out(*(o.ptr(f, k + side) for k in ("level_", "proj_", "mp_kp_", "mp_d1_", "mp_d2_", "kp_mp_")))


def _map_view(m):
    return L.ft_map_view(m["n"], m["pos"].data_ptr(), m["nrm"].data_ptr(), m["desc"].data_ptr(), m["skip"].data_ptr())


# --------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------
class State:
    pass


def _inputs(case, seed):
    """The case's inputs alone (shared by prepare and exact)."""
    R = Rand(seed)
    s = State()
    s.case, s.R = case, R
    kind = case["kind"]
    if kind in ("fisheye", "trackfish"):
        s.rig = scenes.fisheye_rig(int(seed) * 31 + 7)
        s.frames = [_fisheye_frame(R, s.rig, case["left"], case.get("points", 1000))
                    for _ in range(case.get("frames", 1))]
        return s
    if kind == "extract":
        n = case["images"]
        pool = []
        for at in range(0, n, 8):
            pool += list(_images(R, min(8, n - at), case["w"], case["h"], case["content"]))
        s.pyr = [Pyramid(i) for i in pool]
        return s
    s.cam = scenes.pinhole_camera(case["w"], case["h"])
    n = case.get("frames", 1)
    s.pyr, sc = [], []
    if kind in ("stereo", "track"):
        sc = _stereo_scenes(R, min(n, 8 if case["w"] < 1500 else 2), s.cam, case["content"])
        built = case.get("images", False)
        s.levels = torch.zeros((n, 2, _pyramid_layout(case["w"], case["h"])[1]), dtype=torch.uint8, device=DEV)
        for f in range(n):
            s.pyr.append(tuple(Pyramid(sc[f % len(sc)][i], s.levels[f, i], not built) for i in range(2)))
    s.frames = []
    for f in range(n):
        # the batch is ragged: counts vary by a fifth around the case's
        q = 1.0 if n == 1 else 0.8 + 0.4 * ((f * 29) % 64) / 63.0
        s.frames.append(_pinhole_frame(R, s.cam, sc[f % len(sc)] if sc else None, int(case["left"] * q),
                                       int(case.get("points", 500) * q), case["w"] >= 1500))
    if kind == "track" and case["last"]:
        for fr in s.frames:
            fr["last"] = _last_points(R, fr["map"], fr["pose"])
    if kind in ("search", "pose"):
        # the stereo step's right coordinates, as an earlier call left them
        fr = s.frames[0]
        ur = fr["left"].x.double() - s.cam.bf / fr["depth"] + 0.3 * R.normal(fr["left"].n)
        s.u_right = torch.where(R.uni(0, 1, fr["left"].n) < 0.7, ur, torch.full_like(ur, -1)).float()
    if kind == "pose":
        # the search's matches: the points' own keypoints, one in ten a wrong one
        fr, m = s.frames[0], s.frames[0]["map"]
        wrong = R.ints(0, fr["left"].n, m["n"])
        kp = torch.where((R.uni(0, 1, m["n"]) < 0.1) & (m["owner"] >= 0), wrong, m["owner"])
        s.mp_kp = torch.where(m["skip"] != 0, torch.full_like(kp, -1), kp).to(I32)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind, o = case["kind"], Outputs()
    s.out = o
    n = case.get("frames", 1)
    if kind == "extract":
        area = sum(p.struct.width[l] * p.struct.height[l] for p in s.pyr for l in range(NL))
        s.ctx = Context(arena_bytes=(64 << 20) + 3 * area, max_frames=max(64, case["images"]))
        s.orb = OrbOutputs(case["images"], scenes.orb_level_caps(case["slots"]), scenes.orb_pattern())
        s.arr = (L.ft_pyramid * case["images"])(*(p.struct for p in s.pyr))
        lay = s.orb.lay
        for name, _, tail in OrbOutputs.KEYS + (("n_level", None, ()),):
            # one view of every image's array of this name: images lie a fixed distance apart
            off, dt, shape = lay.items[lay.index[0, name]][1:]
            step = lay.size // case["images"]
            t = s.orb.dev.view(getattr(torch, dt.name))
            size = dt.itemsize
            strides = (step // size,) + tuple(int(np.prod(shape[i + 1:])) for i in range(len(shape)))
            o.t[name] = t.as_strided((case["images"],) + tuple(shape), strides, off // size)
        return s
    for f, fr in enumerate(s.frames):
        nl, nr, nm = fr["left"].n, fr["right"].n, fr["map"]["n"]
        if kind in ("stereo", "track"):
            for k, dt in STEREO:
                o.want(f, k, nl, dt)
        if kind in ("fisheye", "trackfish"):
            for k in ("r_idx", "d1", "d2"):
                o.want(f, k, nl, I32)
            o.want(f, "depth", nl, F32)
            o.want(f, "xyz", nl, F32, 4)
        if kind in ("search", "track", "trackfish"):
            _want_search(o, f, "l", nm, nl)
        if kind == "trackfish":
            _want_search(o, f, "r", nm, nr)
        if kind == "pose" or case.get("pose"):
            o.want(f, "Rt", 12, F32)
            o.want(f, "inlier", nm, I8)
            o.want(f, "n_inliers", 1, I32)
    o.make()
    many = kind in ("track", "trackfish")
    per = 1 << 20
    if many:
        fr = max(s.frames, key=lambda q: q["map"]["n"])
        per += 256 * (fr["left"].n + fr["right"].n) + 80 * fr["map"]["n"]
    s.ctx = Context(arena_bytes=(64 << 20) + per * n, max_frames=max(64, n), use_graphs=many)
    if not many:
        fr = s.frames[0]
        s.pose = pose_struct(fr["pose"])
        s.left, s.right = fr["left"].struct(), fr["right"].struct()
        if kind == "fisheye":
            s.rig_c = rig_struct(s.rig)
            s.fish_out = L.ft_fisheye_out(*(o.ptr(0, k) for k in ("r_idx", "d1", "d2", "depth", "xyz")))
        else:
            s.cam_c = pinhole_struct(s.cam)
            v = s.view = L.ft_frame_view(camera=L.FT_CAMERA_PINHOLE, pinhole=s.cam_c, left=s.left, right=s.right)
            v.taken_left = fr["taken"].data_ptr()
            s.map_c = _map_view(fr["map"])
        if kind == "stereo":
            s.stereo = L.ft_stereo_frame(s.left, s.right, s.pyr[0][0].struct, s.pyr[0][1].struct)
            s.stereo_out = L.ft_stereo_out(*(o.ptr(0, k) for k, _ in STEREO))
        if kind in ("search", "pose"):
            s.view.u_right = s.u_right.data_ptr()
        if kind == "search":
            s.search_out = L.ft_search_out(left=_search_cam(o, 0, "l"))
        if kind == "pose":
            s.pose_out = L.ft_pose_out(o.ptr(0, "Rt"), o.ptr(0, "inlier"), o.ptr(0, "n_inliers"))
        return s
    s.jobs = (L.ft_frame_job * n)()
    s.pose_outs = []
    for f, fr in enumerate(s.frames):
        j = s.jobs[f]
        j.left, j.right = fr["left"].struct(), fr["right"].struct()
        j.taken_left = fr["taken"].data_ptr()
        j.pose = pose_struct(fr["pose"])
        j.map = _map_view(fr["map"])
        j.search.left = _search_cam(o, f, "l")
        if kind == "trackfish":
            j.camera, j.fisheye = L.FT_CAMERA_FISHEYE, rig_struct(s.rig)
            j.taken_right = fr["taken_r"].data_ptr()
            j.O_right[:] = [float(v) for v in fr["O_right"]]
            j.fisheye_out = L.ft_fisheye_out(*(o.ptr(f, k) for k in ("r_idx", "d1", "d2", "depth", "xyz")))
            j.search.right = _search_cam(o, f, "r")
            continue
        j.camera, j.pinhole = L.FT_CAMERA_PINHOLE, pinhole_struct(s.cam)
        j.pyr_left, j.pyr_right = s.pyr[f][0].struct, s.pyr[f][1].struct
        j.build_pyramids = int(case["images"])
        j.stereo = L.ft_stereo_out(*(o.ptr(f, k) for k, _ in STEREO))
        if case["last"]:
            j.last = C.pointer(fr["last"]["view"])
        if case["pose"]:
            s.pose_outs.append(L.ft_pose_out(o.ptr(f, "Rt"), o.ptr(f, "inlier"), o.ptr(f, "n_inliers")))
            j.pose_out = C.pointer(s.pose_outs[-1])
    s.batch = L.ft_batch(n=n, frames=C.cast(s.jobs, C.POINTER(L.ft_frame_job)))
    if case.get("images"):
        o.t["levels"] = s.levels
    return s


def run(s):
    kind, lib, ctx, st = s.case["kind"], s.ctx.lib, s.ctx.ptr, stream_handle()
    if kind in ("track", "trackfish"):
        r = lib.ft_track_batch(ctx, st, None, C.byref(s.batch))
    elif kind == "stereo":
        r = lib.ft_stereo_match_pinhole(ctx, st, None, C.byref(s.cam_c), C.byref(s.stereo), C.byref(s.stereo_out))
    elif kind == "fisheye":
        r = lib.ft_stereo_match_fisheye(ctx, st, None, C.byref(s.rig_c), C.byref(s.left), C.byref(s.right),
                                        C.byref(s.fish_out))
    elif kind == "search":
        r = lib.ft_search_local_points(ctx, st, None, C.byref(s.view), C.byref(s.pose), C.byref(s.map_c),
                                       C.byref(s.search_out))
    elif kind == "pose":
        r = lib.ft_optimize_pose(ctx, st, None, C.byref(s.view), C.byref(s.pose), C.byref(s.map_c),
                                 C.c_void_p(s.mp_kp.data_ptr()), C.byref(s.pose_out))
    else:
        r = lib.ft_extract_orb(ctx, st, None, len(s.arr), s.arr, C.byref(s.orb.params), s.orb.outs)
    L.check(r, kind)
    return s.out.t


# --------------------------------------------------------------------------
# work
# --------------------------------------------------------------------------
def _level_pixels(w, h):
    return [int(math.floor(w / float(s) + 0.5)) * int(math.floor(h / float(s) + 0.5)) for s in SC32]


def work(case):
    kind = case["kind"]
    if kind == "extract":
        px = sum(_level_pixels(case["w"], case["h"]))
        # every level pixel read once, a record and descriptor written per slot; per pixel the 16
        # circle comparisons, per slot the moments (two multiply-adds of 709 pixels), the 512
        # smoothed samples (9 operations each, separable) and their rotation
        return dict(bytes=float(case["images"] * (px + 57 * case["slots"])),
                    flops=float(case["images"] * (16 * px + case["slots"] * (4 * 709 + 512 * (9 + 6)))))
    n, nl, nm = case.get("frames", 1), case["left"], case.get("points", 0)
    b = f = 0.0
    if kind in ("stereo", "track"):
        # 41-byte keypoint records, 28 bytes written per left keypoint, 352 bytes of patches per match;
        # per match 11 shifts of 121 differences
        nr = nl * 1.1
        b += 41 * (nl + nr) + 28 * nl + 352 * 0.85 * nl
        f += 0.85 * nl * 11 * 121 * 3 + 20 * nl * 8 * 3
        if case.get("images"):
            px = _level_pixels(case["w"], case["h"])
            b += 2 * sum(px)                # level 0 read, the other levels written, both images
            f += 2 * sum(px[1:]) * 9
    if kind in ("fisheye", "trackfish"):
        b += 41 * 2 * nl + 32 * nl
        f += (0.6 * nl) * (0.7 * nl) * 8 * 3
    if kind in ("search", "track", "trackfish"):
        sides = 2 if kind == "trackfish" else 1
        b += 65 * nm + sides * (29 * nm + 5 * nl) + (41 * nl if kind == "search" else 0)
        f += sides * nm * (60 + 4 * 8 * 3)
    if kind == "pose" or case.get("pose"):
        obs = min(0.6 * nm, nl)
        b += 5 * nm + 28 * obs
        f += 40 * obs * 160
    return dict(bytes=n * b, flops=n * f)


# --------------------------------------------------------------------------
# exact: the floating point outputs in 64 bits
# --------------------------------------------------------------------------
SC64 = torch.as_tensor(SC32.astype(np.float64))


def _hamming(a, b):
    """[n, m] Hamming distances of descriptor rows."""
    w = torch.arange(8, device=DEV, dtype=torch.uint8)

    def signs(d):
        return (((d[:, :, None] >> w) & 1).reshape(len(d), 256).float() * 2 - 1)

    return ((256 - signs(a) @ signs(b).T) / 2).round().long()


def _exact_stereo(cam, fr, pyr):
    le, ri, sc = fr["left"], fr["right"], SC64.to(DEV)
    x, y, o = le.x.double(), le.y.double(), le.oct.long()
    xr, yr, orr = ri.x.double(), ri.y.double(), ri.oct.long()
    b, bf = float(np.float32(cam.b)), float(np.float32(cam.bf))
    r, row, maxd = 2 * sc[orr], y.floor(), bf / b
    ok = ((yr - r).floor() <= row[:, None]) & (row[:, None] <= (yr + r).ceil())
    ok &= (o[:, None] - orr).abs() <= 1
    ok &= (xr <= x[:, None]) & (xr >= x[:, None] - maxd)
    d = _hamming(le.desc, ri.desc)
    key = torch.where(ok, d * (1 << 20) + torch.arange(ri.n, device=DEV), torch.full_like(d, 1 << 40)).min(1).values
    matched, j = (key >> 20) < 75, key & 0xfffff
    ur = torch.full((le.n,), -1.0, dtype=torch.float64, device=DEV)
    depth, sadb = ur.clone(), torch.full((le.n,), -1, device=DEV)
    for l in range(NL):
        a, c = pyr[0].levels[l].long(), pyr[1].levels[l].long()
        h, w = a.shape
        i = ((o == l) & matched).nonzero()[:, 0]
        u, v, u0 = ((q / sc[l] + 0.5).floor().long() for q in (x[i], y[i], xr[j[i]]))
        ins = (v >= 5) & (v <= h - 6) & (u >= 5) & (u <= w - 6) & (u0 >= 10) & (u0 <= w - 11)
        i, u, v, u0 = i[ins], u[ins], v[ins], u0[ins]
        if not len(i):
            continue
        k = torch.arange(-5, 6, device=DEV)
        rows = v[:, None, None] + k[None, :, None]
        p = a[rows, u[:, None, None] + k] - a[v, u][:, None, None]
        sad = []
        for s in range(-5, 6):
            q = c[rows, u0[:, None, None] + s + k] - c[v, u0 + s][:, None, None]
            sad.append((p - q).abs().sum((1, 2)))
        sad = torch.stack(sad, 1)
        best = (sad * 16 + torch.arange(11, device=DEV)).argmin(1)
        inner = (best > 0) & (best < 10)
        i, u0, sad, best = i[inner], u0[inner], sad[inner], best[inner][:, None]
        s1, s2, s3 = (sad.gather(1, best + q)[:, 0].double() for q in (-1, 0, 1))
        sub = sc[l] * (u0 + best[:, 0] - 5 + (s1 - s3) / (2 * (s1 + s3 - 2 * s2)))
        disp = x[i] - sub
        good = (disp >= 0) & (disp < maxd)
        zero = disp <= 0
        sub, disp = torch.where(zero, x[i] - 0.01, sub), torch.where(zero, torch.full_like(disp, 0.01), disp)
        i = i[good]
        ur[i], depth[i], sadb[i] = sub[good], bf / disp[good], s2[good].long()
    acc = sadb[sadb >= 0].sort().values
    if len(acc):
        drop = (sadb >= 0) & (sadb.double() >= float(np.float32(1.5) * np.float32(1.4)) * acc[len(acc) // 2].double())
        ur[drop], depth[drop] = -1.0, -1.0
    return ur, depth


def _pose64(pose):
    t = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=DEV)  # noqa: E731
    return t(pose.R).view(3, 3), t(pose.t), t(pose.O)


def _exact_proj(m, Rw, t, O, cam, last):
    """(u, v, u_right, viewing cosine) of the points in view, zeros elsewhere."""
    P, N = m["pos"].double(), m["nrm"].double()
    c = P[:, :3] @ Rw.T + t
    z = c[:, 2]
    if isinstance(cam, scenes.PinholeCamera):
        u, v = cam.fx * c[:, 0] / z + cam.cx, cam.fy * c[:, 1] / z + cam.cy
        ur = u - cam.bf / z
    else:
        u, v = _kb8_project(cam, c)
        ur = torch.full_like(u, -1.0)
    ok = (z > 0) & (u >= cam.min_x) & (u <= cam.max_x) & (v >= cam.min_y) & (v <= cam.max_y) & (m["skip"] == 0)
    vc = torch.zeros_like(u)
    if last is not None:
        ok &= (last["oct"] >= 0) & (last["oct"] < NL)
    else:
        d = P[:, :3] - O
        dist = d.norm(dim=1)
        vc = (d * N[:, :3]).sum(1) / dist
        ok &= (dist >= 0.8 * P[:, 3]) & (dist <= 1.2 * N[:, 3]) & (vc >= 0.5)
    return torch.where(ok[:, None], torch.stack([u, v, ur, vc], 1), torch.zeros(1, device=DEV, dtype=torch.float64))


def _exact_fisheye(rig, fr):
    le, ri = fr["left"], fr["right"]
    la = (le.x >= rig.lap_l0) & (le.x <= rig.lap_l1)
    ra = (ri.x >= rig.lap_r0) & (ri.x <= rig.lap_r1)
    d = _hamming(le.desc, ri.desc)
    key = d * (1 << 20) + torch.arange(ri.n, device=DEV)
    key = torch.where(la[:, None] & ra, key, torch.full_like(key, 256 << 20)).topk(2, largest=False, sorted=True).values
    d1, d2 = key[:, 0] >> 20, key[:, 1] >> 20
    ok = la & (d1 < 256) & (d1.double() < 0.7 * d2.double())
    j = (key[:, 0] & 0xfffff).clamp(max=ri.n - 1)
    one = torch.ones(le.n, device=DEV, dtype=torch.float64)
    l = _kb8_unproject(rig.left, le.x.double(), le.y.double(), one)
    r = _kb8_unproject(rig.right, ri.x[j].double(), ri.y[j].double(), one)
    Rm = torch.as_tensor(rig.R_rl, device=DEV).double().view(3, 3)
    Cn = (-(Rm.T @ torch.as_tensor(rig.t_rl, device=DEV).double())).expand_as(l)
    dd = r @ Rm
    nn_ = torch.linalg.cross(l, dd)
    n2 = (nn_ * nn_).sum(1)
    s = (torch.linalg.cross(Cn, dd) * nn_).sum(1) / n2
    t = (torch.linalg.cross(Cn, l) * nn_).sum(1) / n2
    X = 0.5 * (s[:, None] * l + Cn + t[:, None] * dd)
    ok &= _kb8_theta(rig.left, le.x.double(), le.y.double())[4]
    ok &= _kb8_theta(rig.right, ri.x[j].double(), ri.y[j].double())[4]
    ok &= (n2 > 1e-10 * (l * l).sum(1) * (dd * dd).sum(1)) & (s > 0) & (t > 0) & (X[:, 2] > 1e-4)
    depth = torch.where(ok, X[:, 2], -one)
    xyz = torch.where(ok[:, None], torch.cat([X, one[:, None]], 1), torch.zeros(1, device=DEV, dtype=torch.float64))
    return depth, xyz


def _exact_pose(s):
    """Motion-only Gauss-Newton with Huber weights, four rounds of ten steps."""
    fr, cam = s.frames[0], s.cam
    m = (s.mp_kp >= 0).nonzero()[:, 0]
    k = s.mp_kp[m].long()
    P, sc = fr["map"]["pos"][m, :3].double(), SC64.to(DEV)[fr["left"].oct[k].long()]
    obs = torch.stack([fr["left"].x[k], fr["left"].y[k], s.u_right[k]], 1).double()
    st = obs[:, 2] >= 0
    w, th = 1 / sc ** 2, torch.where(st, 7.815, 5.991).double()
    Rw, t, _ = _pose64(fr["pose"])
    inl = torch.ones(len(m), dtype=torch.bool, device=DEV)

    def residuals():
        c = P @ Rw.T + t
        iz = 1 / c[:, 2]
        u, v = cam.fx * c[:, 0] * iz + cam.cx, cam.fy * c[:, 1] * iz + cam.cy
        e = obs - torch.stack([u, v, u - cam.bf * iz], 1)
        e[:, 2] = torch.where(st, e[:, 2], torch.zeros_like(iz))
        return c, iz, e, w * (e * e).sum(1)

    for _ in range(4):
        if inl.sum() < 3:
            break
        for _ in range(10):
            c, iz, e, chi = residuals()
            use = inl & (c[:, 2] > 0)
            hw = torch.where(chi <= th, torch.ones_like(chi), (th / chi).sqrt()) * w * use
            D = torch.zeros(len(m), 3, 3, dtype=torch.float64, device=DEV)
            D[:, 0, 0] = D[:, 2, 0] = cam.fx * iz
            D[:, 1, 1] = cam.fy * iz
            D[:, 0, 2] = -cam.fx * c[:, 0] * iz ** 2
            D[:, 1, 2] = -cam.fy * c[:, 1] * iz ** 2
            D[:, 2, 2] = D[:, 0, 2] + cam.bf * iz ** 2
            D[:, 2] *= st[:, None]
            J = torch.cat([torch.linalg.cross(c[:, None].expand_as(D), D), D], 2)
            H = (J.transpose(1, 2) @ (J * hw[:, None, None])).sum(0)
            g = (J * (hw[:, None] * e)[:, :, None]).sum((0, 1))
            d = torch.linalg.solve(H, g)
            wx = torch.zeros(4, 4, dtype=torch.float64, device=DEV)
            wx[0, 1], wx[0, 2], wx[1, 2] = -d[2], d[1], -d[0]
            wx[1, 0], wx[2, 0], wx[2, 1] = d[2], -d[1], d[0]
            wx[:3, 3] = d[3:]
            T = torch.linalg.matrix_exp(wx)
            Rw, t = T[:3, :3] @ Rw, T[:3, :3] @ t + T[:3, 3]
        c, _, _, chi = residuals()
        inl = (c[:, 2] > 0) & ~(chi > th)
    return torch.cat([Rw.reshape(9), t])


CIRCLE = ((0, -3), (1, -3), (2, -2), (3, -1), (3, 0), (3, 1), (2, 2), (1, 3),
          (0, 3), (-1, 3), (-2, 2), (-3, 1), (-3, 0), (-3, -1), (-2, -2), (-1, -3))


def _exact_corners(img, cap):
    """The level's first `cap` corners by (score, y, x): x, y, cos, sin."""
    h, w = img.shape
    if h <= 38 or w <= 38 or cap == 0:
        e = torch.zeros(0, device=DEV, dtype=torch.float64)
        return e, e, e, e
    a = img.short()
    c = a[3:h - 3, 3:w - 3]
    d = torch.stack([a[3 + dy:h - 3 + dy, 3 + dx:w - 3 + dx] - c for dx, dy in CIRCLE])
    best = torch.full_like(c, -256)
    for i in range(16):
        arc = d[[(i + q) % 16 for q in range(9)]]
        best = torch.maximum(best, torch.maximum(arc.min(0).values, -arc.max(0).values))
    score = TF.pad((best.int() - 1), (3, 3, 3, 3), value=-1)
    keep = torch.zeros_like(score, dtype=torch.bool)
    keep[19:h - 19, 19:w - 19] = True
    score = torch.where(keep & (score >= 20), score, torch.full_like(score, -1))
    # a larger key wins: the score, then the earlier raster position
    pos = torch.arange(h * w, device=DEV).view(h, w)
    key = torch.where(score >= 0, score.long() * (1 << 25) + ((1 << 25) - 1 - pos), torch.full_like(pos, -1))
    near = TF.max_pool2d(TF.pad(key.double(), (1, 1, 1, 1), value=-1.0)[None], 3, stride=1)[0].long()
    key = key[(key >= 0) & (key == near)].sort(descending=True).values[:cap]
    p = (1 << 25) - 1 - (key & ((1 << 25) - 1))
    y, x = p // w, p % w
    r = torch.arange(-15, 16, device=DEV)
    disk = (r[:, None] ** 2 + r[None] ** 2 <= 225).double()
    patch = img[y[:, None, None] + r[None, :, None], x[:, None, None] + r].double() * disk
    m10, m01 = (patch * r).sum((1, 2)), (patch * r[:, None]).sum((1, 2))
    nm = torch.hypot(m10, m01)
    one = torch.ones_like(nm)
    return x.double(), y.double(), torch.where(nm > 0, m10 / nm, one), torch.where(nm > 0, m01 / nm, 0 * one)


def _like(case, seed, names):
    """Zeros in 64 bits, laid out as prepare() lays the outputs out."""
    s = prepare(case, seed)
    return s, {k: (torch.zeros_like(s.out.t[k], dtype=torch.float64) if k in names else None) for k in s.out.t}


def exact(case, seed):
    kind = case["kind"]
    if kind == "extract":
        s, out = _like(case, seed, ("x", "y", "cs"))
        caps, slot = scenes.orb_level_caps(case["slots"]), 0
        out["x"].fill_(-1e9), out["y"].fill_(-1e9)
        out["cs"][:, :, 0] = 1.0
        for l, cap in enumerate(caps):
            for i, p in enumerate(s.pyr):
                x, y, c, sn = _exact_corners(p.levels[l], cap)
                at = slice(slot, slot + len(x))
                out["x"][i, at], out["y"][i, at] = x * float(SC32[l]), y * float(SC32[l])
                out["cs"][i, at, 0], out["cs"][i, at, 1] = c, sn
            slot += cap
        return out
    s, out = _like(case, seed, ("u_right", "depth", "proj_l", "proj_r", "xyz") + (("Rt",) if kind == "pose" else ()))

    def put(f, name, v):
        off, n = s.out.at[f, name]
        out[name][off:off + n] = v

    for f, fr in enumerate(s.frames):
        if kind in ("stereo", "track"):
            if case.get("images"):      # the built levels: bilinear from level 0, as prepare() fills them
                s.pyr[f] = tuple(Pyramid(p.levels[0].contiguous()) for p in s.pyr[f])
            ur, depth = _exact_stereo(s.cam, fr, s.pyr[f])
            put(f, "u_right", ur)
            put(f, "depth", depth)
        if kind in ("fisheye", "trackfish"):
            depth, xyz = _exact_fisheye(s.rig, fr)
            put(f, "depth", depth)
            put(f, "xyz", xyz)
        if kind in ("search", "track", "trackfish"):
            Rw, t, O = _pose64(fr["pose"])
            cam = s.rig.left if kind == "trackfish" else s.cam
            put(f, "proj_l", _exact_proj(fr["map"], Rw, t, O, cam, fr.get("last")))
        if kind == "trackfish":
            Rm = torch.as_tensor(s.rig.R_rl, device=DEV).double().view(3, 3)
            tr = torch.as_tensor(s.rig.t_rl, device=DEV).double()
            O_r = torch.as_tensor(fr["O_right"], device=DEV).double()
            put(f, "proj_r", _exact_proj(fr["map"], Rm @ Rw, Rm @ t + tr, O_r, s.rig.right, None))
        if kind == "pose":
            put(f, "Rt", _exact_pose(s))
    return out
