"""The work this library is used for, as timed cases.

Every case goes through the public entry points of `paper_1311_6811_gb300` on a
scene rendered on the GPU from a seed: calibrated cameras on a ring around the
grid, a per-pixel Gaussian colour background, and a body of ten capsules (two
bodies in the largest scene) that stands or walks in it.

Voxel lists are written in an order the library leaves unspecified, so they are
returned as what the later stages make of them (surface counts, silhouettes),
not as they stand.
"""

import math
import random

import numpy as np
import torch

from paper_1311_6811_gb300 import autograd, psfs

_DTYPES = ("f32", "f16", "bf16")
_NOISE_VAR = 4.0   # sensor noise, variance per channel


def listed():
    return [
        # the oracle-sized rig, one frame per call with the default
        # configuration: a live preview, where latency and launches count
        dict(name="frame_64", kind="frame", nx=64, ny=64, nz=64, cams=4, width=320, height=240, dtype="f32",
             bodies=1, frames=1, tuned=False),
        # the benchmark's rig, one frame per call: an interactive capture that
        # cannot wait for later frames
        dict(name="frame_128", kind="frame", nx=128, ny=128, nz=128, cams=8, width=640, height=480, dtype="f32",
             bodies=1, frames=1, tuned=True),
        # the large rig: two bodies, 16 HD cameras, 16-bit maps
        dict(name="frame_256_f16", kind="frame", nx=256, ny=256, nz=256, cams=16, width=1280, height=720,
             dtype="f16", bodies=2, frames=1, tuned=False),
        # the benchmark itself: a recorded 100-frame walk
        dict(name="sequence_128", kind="sequence", nx=128, ny=128, nz=128, cams=8, width=640, height=480,
             dtype="f32", bodies=1, frames=100, tuned=True),
        # the same rig with 16-bit maps, whole frame groups
        dict(name="sequence_128_f16", kind="sequence", nx=128, ny=128, nz=128, cams=8, width=640, height=480,
             dtype="f16", bodies=1, frames=64, tuned=True),
        # a short clip on a rig whose grid, image and frame count divide nothing
        dict(name="sequence_odd_bf16", kind="sequence", nx=101, ny=86, nz=74, cams=5, width=496, height=377,
             dtype="bf16", bodies=1, frames=13, tuned=True),
        # frames of unrelated rigs in one launch: a processing service
        dict(name="batch_16", kind="batch", rigs=16, rig_seed=64, dtype="f32"),
        # the adjoint of one frame with the forward recomputed: gradient checks
        # and background fitting frame by frame
        dict(name="adjoint_128", kind="adjoint", nx=128, ny=128, nz=128, cams=8, width=640, height=480, dtype="f32",
             bodies=1, frames=1, tuned=True),
        # a training step of the background model over 16 frames: background
        # update, forward, loss, gradients of mean and variance
        dict(name="train_128", kind="train", nx=128, ny=128, nz=128, cams=8, width=640, height=480, dtype="f32",
             bodies=1, frames=16, tuned=True),
        # what follows the reconstruction of a walk: smoothing, surface voxels,
        # silhouettes in every camera
        dict(name="track_128", kind="track", nx=128, ny=128, nz=128, cams=8, width=640, height=480, frames=100,
             bodies=1),
        # the same stages on rows that are not whole 16-byte units
        dict(name="track_odd", kind="track", nx=93, ny=110, nz=77, cams=5, width=470, height=351, frames=9, bodies=1),
        # the tracker's particle weights of one frame
        dict(name="weights_200", kind="weights", particles=200, kt=8, kw=4, cams=8, width=640, height=480, bodies=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case: any kind, any grid from 40 to 190 voxels a side, 2 to 12
    cameras, images from 160 to 960 pixels wide."""
    kind = rng.choice(["frame", "frame", "sequence", "sequence", "adjoint", "train", "track", "weights", "batch"])
    if kind == "batch":
        return dict(kind="batch", rigs=rng.randint(3, 16), rig_seed=rng.randrange(10000), dtype=rng.choice(_DTYPES))
    case = dict(kind=kind, cams=rng.randint(2, 12), width=_log_int(rng, 160, 960), height=_log_int(rng, 120, 720),
                bodies=rng.randint(1, 2))
    if kind == "weights":
        case.update(particles=_log_int(rng, 16, 400), kt=rng.randint(4, 12), kw=rng.randint(2, 6))
        return case
    case.update(nx=_log_int(rng, 40, 190), ny=_log_int(rng, 40, 190), nz=_log_int(rng, 40, 190))
    if kind in ("sequence", "train"):
        # sequences need whole 16-byte frames and a voxel count of fours
        case["width"] = (case["width"] + 15) // 16 * 16
        case["nz"] = (case["nz"] + 3) // 4 * 4
    if kind == "track":
        case.update(frames=_log_int(rng, 1, 48))
        return case
    case.update(dtype=rng.choice(_DTYPES), tuned=kind != "adjoint" and rng.random() < 0.5,
                frames=_log_int(rng, 2, 48) if kind == "sequence" else rng.randint(2, 18) if kind == "train" else 1)
    return case


# --------------------------------------------------------------------------- #
# scenes
# --------------------------------------------------------------------------- #
def _rot(axis, a):
    c, s = math.cos(a), math.sin(a)
    if axis == 0:
        return np.array([[1, 0, 0], [0, c, -s], [0, s, c]])
    if axis == 1:
        return np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]])
    return np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])


def _ring(g, n, width, height, focal, target_z):
    """`n` pinhole cameras on a 3 m ring, heights 1.2 to 2.2 m, looking at the
    grid's centre with up to 2 degrees of jitter."""
    cams = []
    for k in range(n):
        az = 2.0 * math.pi * k / n
        centre = np.array([3.0 * math.cos(az), 3.0 * math.sin(az), g.uniform(1.2, 2.2)])
        fwd = np.array([0.0, 0.0, target_z]) - centre
        fwd /= np.linalg.norm(fwd)
        right = np.cross(fwd, [0.0, 0.0, 1.0])
        right /= np.linalg.norm(right)
        R = np.stack([right, np.cross(fwd, right), fwd])
        for axis in range(3):
            R = _rot(axis, math.radians(g.uniform(-2.0, 2.0))) @ R
        K = np.array([[focal, 0, width / 2], [0, focal, height / 2], [0, 0, 1.0]])
        cams.append(dict(width=width, height=height, K=K, R=R, t=-R @ centre, centre=centre))
    return cams


def _body(phase, xy, heading, spread, swing):
    """Ten capsules (a, b, radius): torso, head, and two parts per limb."""
    lean = _rot(2, heading)
    hip = np.array([xy[0], xy[1], 0.88])

    def part(base, flex, abd, length, radius):
        d = lean @ (_rot(0, abd) @ (_rot(1, -flex) @ np.array([0.0, 0.0, -1.0])))
        return base, base + length * d, radius

    chest = hip + np.array([0.0, 0.0, 0.55])
    caps = [(hip, chest, 0.14), (chest + [0, 0, 0.15], chest + [0, 0, 0.25], 0.10)]
    for side in (1.0, -1.0):
        s = swing * math.sin(phase + (0.0 if side > 0 else math.pi))
        leg = part(hip + lean @ np.array([0.0, 0.09 * side, -0.02]), s, side * 0.08, 0.42, 0.075)
        arm = part(chest + lean @ np.array([0.0, 0.19 * side, -0.04]), -s, side * spread, 0.30, 0.045)
        caps += [leg, part(leg[1], s - 0.5 * swing, side * 0.08, 0.42, 0.055)]
        caps += [arm, part(arm[1], 0.4 - s, side * spread, 0.28, 0.04)]
    return caps


def _walk(g, frames, bodies):
    """Capsules of every frame: each body walks a circle of 0.35 m."""
    tracks = [dict(c=(0.0, 0.0) if bodies == 1 else (-0.35 + 0.7 * b, 0.25 * (-1) ** b), a=g.uniform(0, 6.28),
                   p=g.uniform(0, 6.28), w=g.uniform(5.0, 7.0), v=g.uniform(1.7, 2.8), s=g.uniform(0.1, 0.9),
                   q=g.uniform(0.3, 0.5)) for b in range(bodies)]
    out = []
    for f in range(frames):
        caps = []
        for t in tracks:
            ang = t["a"] + t["v"] * f / 30.0
            xy = (t["c"][0] + 0.35 * math.cos(ang), t["c"][1] + 0.35 * math.sin(ang))
            caps += _body(t["p"] + t["w"] * f / 30.0, xy, ang + math.pi / 2, t["s"], t["q"])
        out.append(caps)
    return out


def _caps_tensor(caps):
    return (torch.tensor(np.array([c[0] for c in caps]), dtype=torch.float32, device="cuda"),
            torch.tensor(np.array([c[1] for c in caps]), dtype=torch.float32, device="cuda"),
            torch.tensor([c[2] for c in caps], dtype=torch.float32, device="cuda"))


def _rays(cam):
    """Unit world directions of the pixel centres, [H * W][3]."""
    y, x = torch.meshgrid(torch.arange(cam["height"], device="cuda") + 0.5,
                          torch.arange(cam["width"], device="cuda") + 0.5, indexing="ij")
    f = cam["K"][0, 0]
    d = torch.stack([(x - cam["width"] / 2) / f, (y - cam["height"] / 2) / f, torch.ones_like(x)], -1).reshape(-1, 3)
    d = d @ torch.tensor(cam["R"], dtype=torch.float32, device="cuda")
    return d / d.norm(dim=1, keepdim=True)


def _labels(rays, centre, caps):
    """Index of the nearest capsule each ray meets, -1 for none."""
    A, B, r = caps
    O = torch.tensor(centre, dtype=torch.float32, device="cuda")
    e, w0 = B - A, O - A
    b = e @ rays.T                                   # [caps][pixels]
    d = w0 @ rays.T
    c, ee = (e * e).sum(1)[:, None], (e * w0).sum(1)[:, None]
    t = ((ee - b * d) / (c - b * b).clamp_min(1e-9)).clamp_(0.0, 1.0)
    s = (t * b - d).clamp_min_(0.0)                  # depth of closest approach
    dist2 = (w0 * w0).sum(1)[:, None] - 2.0 * t * ee + t * t * c + s * s - 2.0 * s * (t * b - d)
    depth, label = torch.where(dist2 <= (r * r)[:, None], s, torch.inf).min(0)
    return torch.where(depth.isfinite(), label, -1)


class _Scene:
    """One rig, its background and the images of a walk."""

    def __init__(self, case, seed, images=True):
        g = np.random.default_rng(seed)
        tg = torch.Generator(device="cuda").manual_seed(seed)
        K, W, H, F = case["cams"], case["width"], case["height"], case.get("frames", 1)
        nx, ny, nz = case.get("nx", 128), case.get("ny", 128), case.get("nz", 128)
        side = 3.0 if case["bodies"] > 1 else 2.2
        vs = side / max(nx, ny, nz)
        self.grid = dict(nx=nx, ny=ny, nz=nz, origin=(-nx * vs / 2, -ny * vs / 2, 0.0), voxel_size=vs)
        self.cams = _ring(g, K, W, H, 0.9375 * W, side / 2)
        self.walk = _walk(g, F, case["bodies"])
        self.colours = torch.tensor(g.uniform(0, 255, (10 * case["bodies"], 3)), dtype=torch.float32, device="cuda")
        if not images:
            return
        self.mean = torch.empty((K, H, W, 3), device="cuda").uniform_(40, 200, generator=tg)
        sigma = torch.empty((K, H, W, 3), device="cuda").uniform_(3, 8, generator=tg)
        self.var = sigma * sigma + _NOISE_VAR
        self.images = torch.empty((F, K, H, W, 3), dtype=torch.uint8, device="cuda")
        std, sd = self.var.sqrt().view(K, -1, 3), math.sqrt(_NOISE_VAR)
        rays = [_rays(c) for c in self.cams]
        for f in range(F):
            caps = _caps_tensor(self.walk[f])
            z = torch.randn((K, H * W, 3), device="cuda", generator=tg)
            for k in range(K):
                lab = _labels(rays[k], self.cams[k]["centre"], caps)
                img = torch.where((lab >= 0)[:, None], self.colours[lab.clamp_min(0)] + sd * z[k],
                                  self.mean[k].view(-1, 3) + std[k] * z[k])
                self.images[f, k] = img.round_().clamp_(0, 255).to(torch.uint8).view(H, W, 3)

    def masks(self, frame):
        """Rendered silhouettes, uint8 [K][H][W]."""
        caps = _caps_tensor(self.walk[frame])
        return torch.stack([(_labels(_rays(c), c["centre"], caps) >= 0).to(torch.uint8).view(c["height"], c["width"])
                            for c in self.cams])

    def posterior(self, frame, tg):
        """A posterior grid as the reconstruction leaves it: near 1 inside the
        body, near 0 outside, a noisy surface in between."""
        A, B, r = _caps_tensor(self.walk[frame])
        o, vs = self.grid["origin"], self.grid["voxel_size"]
        x, y, z = (o[a] + (torch.arange(self.grid[n], device="cuda") + 0.5) * vs for a, n in enumerate(("nx", "ny", "nz")))
        best = None
        for a, b, rad in zip(A, B, r):
            e = b - a
            px, py, pz = (x - a[0])[None, None, :], (y - a[1])[None, :, None], (z - a[2])[:, None, None]
            t = ((px * e[0] + py * e[1] + pz * e[2]) / (e * e).sum()).clamp_(0, 1)
            d = ((px - t * e[0]) ** 2 + (py - t * e[1]) ** 2 + (pz - t * e[2]) ** 2).sqrt_() - rad
            best = d if best is None else torch.minimum(best, d)
        noise = torch.empty_like(best).normal_(generator=tg)
        return torch.sigmoid(-best * (4.0 / vs) + noise)


_TUNED = set()   # rigs this process has tuned; later handles of the kind start with the choice


def _reconstructor(case, sc):
    n = case["nx"] * case["ny"] * case["nz"]
    rec = psfs.Reconstructor(sc.grid, sc.cams, map_dtype=case.get("dtype", "f32"), capacity=max(1, n // 8))
    if hasattr(sc, "mean"):
        rec.set_background(sc.mean, sc.var)
    if case.get("tuned"):
        key = tuple(case[k] for k in ("nx", "ny", "nz", "cams", "width", "height", "dtype"))
        if key not in _TUNED:
            psfs.psfs_autotune(rec.handle, sc.images[0])
            _TUNED.add(key)
    return rec


def _rigs(case):
    """The rigs of a batch: cubes of 96 to 192, 4 to 12 cameras, two image sizes."""
    r = random.Random(case["rig_seed"])
    out = []
    for _ in range(case["rigs"]):
        n = r.choice([96, 128, 160, 192])
        w, h = r.choice([(640, 480), (960, 540)])
        out.append(dict(nx=n, ny=n, nz=n, cams=r.randint(4, 12), width=w, height=h, bodies=1, frames=1,
                        dtype=case["dtype"]))
    return out


def _particles(sc, count, g):
    """The body's ten cylinders in world coordinates under displaced poses,
    float32 [count][10][7]."""
    base = np.array([[*a, *b, r] for a, b, r in sc.walk[0][:10]])
    out = np.repeat(base[None], count, 0)
    shift = g.normal(0.0, 0.04, (count, 1, 3))
    out[:, :, 0:3] += shift + g.normal(0.0, 0.02, (count, 10, 3))
    out[:, :, 3:6] += shift + g.normal(0.0, 0.02, (count, 10, 3))
    return out.astype(np.float32)


# --------------------------------------------------------------------------- #
# the cases
# --------------------------------------------------------------------------- #
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.kind, s.case = case["kind"], case
    if s.kind == "batch":
        s.recs, s.keep, frames = [], [], []
        for n, rig in enumerate(_rigs(case)):
            sc = _Scene(rig, seed * 1000 + n)
            rec = _reconstructor(rig, sc)
            occ, lst, cnt = rec.alloc_outputs()
            s.recs.append(rec)
            s.keep.append((sc.images, occ, lst, cnt))
            frames.append((rec.handle, sc.images[0], occ, lst, rec.capacity, cnt))
        s.batch = _Batch(frames)
        return s
    if s.kind == "weights":
        sc = _Scene(case, seed, images=False)
        s.rec = psfs.Reconstructor(sc.grid, sc.cams)
        s.masks = sc.masks(0)
        s.cyl = torch.from_numpy(_particles(sc, case["particles"], np.random.default_rng(seed + 1))).cuda()
        s.weights = torch.empty(case["particles"], device="cuda")
        s.terms = torch.empty((case["particles"], case["cams"], 2), device="cuda")
        return s
    F, shape = case["frames"], (case["nz"], case["ny"], case["nx"])
    sc = _Scene(case, seed, images=s.kind != "track")
    s.rec = _reconstructor(case, sc)
    tg = torch.Generator(device="cuda").manual_seed(seed + 1)
    if s.kind == "track":
        s.occ = torch.stack([sc.posterior(f, tg) for f in range(F)])
        s.smoothed = torch.empty_like(s.occ)
        s.lists = torch.empty((F, s.rec.capacity), dtype=torch.int32, device="cuda")
        s.surface = torch.empty((F, s.rec.capacity), dtype=torch.int32, device="cuda")
        s.counts = torch.zeros(F, dtype=torch.int32, device="cuda")
        s.surface_counts = torch.zeros(F, dtype=torch.int32, device="cuda")
        s.masks = torch.empty((F, case["cams"], case["height"], case["width"]), dtype=torch.uint8, device="cuda")
        return s
    s.images = sc.images
    if s.kind == "frame":
        s.out = s.rec.alloc_outputs()
    elif s.kind == "sequence":
        s.occ = torch.empty((F, *shape), device="cuda")
        s.lists = torch.empty((F, s.rec.capacity), dtype=torch.int32, device="cuda")
        s.counts = torch.zeros(F, dtype=torch.int32, device="cuda")
    elif s.kind == "adjoint":
        s.d_occ = torch.randn(shape, device="cuda", generator=tg)
        s.grads = (torch.empty(sc.mean.shape[:3], device="cuda"), torch.empty_like(sc.mean), torch.empty_like(sc.var))
    else:
        s.mean, s.var = sc.mean.requires_grad_(), sc.var.requires_grad_()
        s.target = torch.stack([sc.posterior(f, tg) for f in range(F)])
    return s


class _Batch:
    """A batch in its graph of per-frame launches, freed with its state."""

    def __init__(self, frames):
        self.handle = psfs.psfs_batch_create(frames)
        psfs.psfs_batch_set_config(self.handle, *psfs.BATCH_CONFIGS[-1][:3], launch=1)

    def __del__(self):
        psfs.psfs_batch_destroy(self.handle)


def run(s):
    if s.kind == "frame":
        occ, _, cnt = s.rec.reconstruct(s.images[0], s.out)
        return {"occupancy": occ, "count": cnt}
    if s.kind == "sequence":
        psfs.psfs_reconstruct_sequence(s.rec.handle, s.images.shape[0], s.images, s.occ, s.lists, s.rec.capacity,
                                       s.counts)
        return {"occupancy": s.occ, "counts": s.counts}
    if s.kind == "batch":
        psfs.psfs_batch_run(s.batch.handle)
        return {"occupancy": [k[1] for k in s.keep], "counts": [k[3] for k in s.keep]}
    if s.kind == "adjoint":
        psfs.psfs_backward(s.rec.handle, s.images[0], s.d_occ, *s.grads)
        return dict(zip(("d_slm", "d_mean", "d_var"), s.grads))
    if s.kind == "train":
        occ = autograd.psfs_occupancy_sequence(s.rec, s.images, s.mean, s.var)
        loss = 0.5 * (occ - s.target).square().sum()
        d_mean, d_var = torch.autograd.grad(loss, (s.mean, s.var))
        return {"occupancy": occ.detach(), "d_mean": d_mean, "d_var": d_var}
    if s.kind == "track":
        F, cap = s.occ.shape[0], s.rec.capacity
        psfs.psfs_smooth(s.rec.handle, F, s.occ, s.smoothed, s.lists, cap, s.counts)
        psfs.psfs_surface(s.rec.handle, F, s.lists, cap, s.counts, s.surface, cap, s.surface_counts)
        psfs.psfs_reproject(s.rec.handle, F, s.surface, cap, s.surface_counts, s.masks)
        return {"smoothed": s.smoothed, "counts": s.counts, "surface_counts": s.surface_counts, "masks": s.masks}
    psfs.psfs_particle_weights(s.rec.handle, s.cyl, s.masks, s.weights, s.terms, s.case["kt"], s.case["kw"])
    return {"weights": s.weights, "terms": s.terms}


def work(case):
    if case["kind"] == "batch":
        parts = [work(dict(r, kind="frame")) for r in _rigs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    K, pix = case["cams"], case["cams"] * case["width"] * case["height"]
    if case["kind"] == "weights":
        samples = case["particles"] * K * 10 * (case["kt"] * case["kw"] + 2 * case["kt"])
        return {"bytes": pix + case["particles"] * (280 + 4 + 8 * K), "flops": 40 * samples}
    vox, F = case["nx"] * case["ny"] * case["nz"], case["frames"]
    if case["kind"] == "track":
        return {"bytes": F * (8 * vox + pix), "flops": F * 9 * vox}
    # images once a frame, the background (mean and variance) once, the grid once a frame;
    # per pixel and frame the two exponentials' worth of Eq. 1-2, per voxel and camera a projection and an add
    by, fl = F * (3 * pix + 4 * vox) + 24 * pix, F * (20 * pix + 12 * K * vox)
    if case["kind"] == "adjoint":
        by, fl = by + 28 * pix, 2 * fl
    if case["kind"] == "train":
        by, fl = by + 4 * F * vox + 24 * pix, 2 * fl
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------- #
# the same in 64 bits, written from the model's equations
# --------------------------------------------------------------------------- #
_PD, _PFA = 0.9, 0.1
_Q = 0.5 * (_PD + _PFA)


def _pixels(sc, k):
    """Pixel of every voxel centre in camera k, and whether it is seen."""
    cam, o, vs = sc.cams[k], sc.grid["origin"], sc.grid["voxel_size"]
    P = cam["K"] @ np.concatenate([cam["R"], cam["t"][:, None]], 1)
    x, y, z = (o[a] + (torch.arange(sc.grid[n], device="cuda", dtype=torch.float64) + 0.5) * vs
               for a, n in enumerate(("nx", "ny", "nz")))
    u, v, w = (P[r, 0] * x[None, None, :] + P[r, 1] * y[None, :, None] + (P[r, 2] * z + P[r, 3])[:, None, None]
               for r in range(3))
    px, py = torch.floor(u / w), torch.floor(v / w)
    W, H = cam["width"], cam["height"]
    seen = (w > 0) & (px >= 0) & (px < W) & (py >= 0) & (py < H)
    return torch.where(seen, py * W + px, 0.0).long().reshape(-1), seen.reshape(-1)


def _slm(sc, f, k):
    """Silhouette likelihood of camera k's pixels (Eq. 1-2), [H * W]."""
    mu, var = sc.mean[k].double(), sc.var[k].double()
    d = sc.images[f, k].double() - mu
    r = -3.0 * math.log(256.0) + (0.5 * (2 * math.pi * var).log() + 0.5 * d * d / var).sum(-1)
    return torch.sigmoid(r).reshape(-1)


def _ab(s):
    a = _PD * s + (1 - _PD) * (1 - s)
    return a, _Q * s + (1 - _Q) * (1 - s)


def _occupancy(sc, f, pixels):
    L = 0.0
    for k, (pix, seen) in enumerate(pixels):
        a, b = _ab(_slm(sc, f, k))
        L = L + torch.where(seen, (a / b).log()[pix], 0.0)
    return torch.sigmoid(L)   # prior 1/2


def _gradients(sc, f, pixels, occ, d_occ):
    """dLoss/dSLM, dLoss/dmean, dLoss/dvar of one frame."""
    dL = d_occ.double().reshape(-1) * occ * (1 - occ)
    out = []
    for k, (pix, seen) in enumerate(pixels):
        s = _slm(sc, f, k)
        a, b = _ab(s)
        acc = torch.zeros_like(s).index_add_(0, pix, torch.where(seen, dL, 0.0))
        ds = acc * ((2 * _PD - 1) / a - (2 * _Q - 1) / b)
        dr = (ds * s * (1 - s))[:, None]
        var = sc.var[k].double().view(-1, 3)
        d = sc.images[f, k].double().view(-1, 3) - sc.mean[k].double().view(-1, 3)
        out.append((ds, -dr * d / var, dr * (0.5 / var - 0.5 * d * d / var ** 2)))
    K, H, W = sc.mean.shape[:3]
    return (torch.stack([o[0] for o in out]).view(K, H, W), torch.stack([o[1] for o in out]).view(K, H, W, 3),
            torch.stack([o[2] for o in out]).view(K, H, W, 3))


def _weights(sc, case, cyl, masks):
    kt, kw, W, H = case["kt"], case["kw"], case["width"], case["height"]
    A, B, rad = cyl[..., 0:3].double(), cyl[..., 3:6].double(), cyl[..., 6:7].double()
    t = (torch.arange(kt, device="cuda", dtype=torch.float64) + 0.5) / kt
    w = (2 * torch.arange(kw, device="cuda", dtype=torch.float64) + 1) / kw - 1
    terms = []
    for k, cam in enumerate(sc.cams):
        P = torch.tensor(cam["K"] @ np.concatenate([cam["R"], cam["t"][:, None]], 1), device="cuda")
        u = B - A
        n = torch.linalg.cross(u, 0.5 * (A + B) - torch.tensor(cam["centre"], device="cuda"))
        n = n / n.norm(dim=-1, keepdim=True)
        m = masks[k].bool()
        pad = torch.nn.functional.pad(m[None, None].double(), (1, 1, 1, 1), value=1.0)[0, 0].bool()
        inner = pad[:-2, 1:-1] & pad[2:, 1:-1] & pad[1:-1, :-2] & pad[1:-1, 2:]

        def misses(image, ws):
            X = (A + 0)[:, :, None, None] + t[:, None, None] * u[:, :, None, None] + \
                ws[None, :, None] * (rad * n)[:, :, None, None]
            h = X @ P[:, :3].T + P[:, 3]
            x, y = torch.floor(h[..., 0] / h[..., 2]), torch.floor(h[..., 1] / h[..., 2])
            ok = (h[..., 2] > 0) & (x >= 0) & (x < W) & (y >= 0) & (y < H)
            hit = image.reshape(-1)[torch.where(ok, y * W + x, 0.0).long()] & ok
            return 1.0 - hit.double().mean(dim=(1, 2, 3))

        terms.append(torch.stack([misses(m & ~inner, torch.tensor([-1.0, 1.0], device="cuda", dtype=torch.float64)),
                                  misses(m, w)], 1))
    terms = torch.stack(terms, 1)
    return {"weights": torch.exp(-terms.sum(dim=(1, 2))), "terms": terms}


def exact(case, seed):
    if case["kind"] == "batch":
        occ = []
        for n, rig in enumerate(_rigs(case)):
            sc = _Scene(rig, seed * 1000 + n)
            px = [_pixels(sc, k) for k in range(rig["cams"])]
            occ.append(_occupancy(sc, 0, px).view(rig["nz"], rig["ny"], rig["nx"]))
        return {"occupancy": occ, "counts": [None] * len(occ)}
    if case["kind"] == "weights":
        sc = _Scene(case, seed, images=False)
        cyl = torch.from_numpy(_particles(sc, case["particles"], np.random.default_rng(seed + 1))).cuda()
        return _weights(sc, case, cyl, sc.masks(0))
    shape = (case["nz"], case["ny"], case["nx"])
    tg = torch.Generator(device="cuda").manual_seed(seed + 1)
    F = case["frames"]
    sc = _Scene(case, seed, images=case["kind"] != "track")
    if case["kind"] == "track":
        out = []
        ones = torch.ones((1, 1, *shape), device="cuda", dtype=torch.float64)
        box = torch.ones((1, 1, 3, 3, 3), device="cuda", dtype=torch.float64)
        n = torch.nn.functional.conv3d(ones, box, padding=1)
        for f in range(F):
            p = sc.posterior(f, tg).double()[None, None]
            for dim in (2, 3, 4):   # separable box sums
                edges = [0] * 6
                edges[8 - 2 * dim] = edges[9 - 2 * dim] = 1   # pad() counts from the last dimension
                q = torch.nn.functional.pad(p, edges)
                p = sum(q.narrow(dim, o, shape[dim - 2]) for o in range(3))
            out.append((p / n)[0, 0])
        return {"smoothed": torch.stack(out), "counts": None, "surface_counts": None, "masks": None}
    pixels = [_pixels(sc, k) for k in range(case["cams"])]
    if case["kind"] == "frame":
        return {"occupancy": _occupancy(sc, 0, pixels).view(shape), "count": None}
    if case["kind"] == "sequence":
        return {"occupancy": torch.stack([_occupancy(sc, f, pixels).view(shape) for f in range(F)]), "counts": None}
    if case["kind"] == "adjoint":
        d_occ = torch.randn(shape, device="cuda", generator=tg)
        grads = _gradients(sc, 0, pixels, _occupancy(sc, 0, pixels), d_occ)
        return dict(zip(("d_slm", "d_mean", "d_var"), grads))
    occs, dm, dv = [], 0.0, 0.0
    for f in range(F):
        occ = _occupancy(sc, f, pixels)
        target = sc.posterior(f, tg).double().reshape(-1)
        _, m, v = _gradients(sc, f, pixels, occ, occ - target)
        occs.append(occ.view(shape))
        dm, dv = dm + m, dv + v
    return {"occupancy": torch.stack(occs), "d_mean": dm, "d_var": dv}
