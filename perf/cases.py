"""Performance cases: what a user of the package has it do, over the sizes it is used at.

Six kinds of case, each through public entry points:

  build     vbm.build: volume -> Gaussians (transfer function, wavelet pyramid, selection, map);
            run once per volume and transfer function, from a 32^3 test cube to a 512^3 simulation
  pyramid   vbm.tf_apply + vbm.dwt3d: the RGBA wavelet pyramid alone, for programs that select
            coefficients themselves
  targets   vbm.render_dvr: the ray-marched supervision images of a volume
  view      vbm.Plan.forward: one frame of an interactive viewer (no gradient)
  step      FineTuner.step_graph: one fine-tuning iteration of a whole batch, the package's main loop
  loop      a program's own training loop: autograd render, vbm.loss, backward, vbm.adam

Inputs are made on the GPU from the seed alone: synthetic fields (blobs with band-limited noise, or
noisy shells), splats placed where such a field has detail, with the scales, opacities and colours of
a set some iterations into its fine-tuning, and targets marched through the same field.

The fine-tuning cases run at the learning rates of the end of an annealed schedule (a thousandth of
the initial ones), so that a pass repeated thousands of times stays the same work.
"""

import math

import numpy as np
import torch

from paper_2601_09417_gb300 import vbm
from paper_2601_09417_gb300.autograd import render
from paper_2601_09417_gb300.finetune import FineTuner, default_lrs

DEVICE = "cuda"

# The eight-knot transfer function of the package's workloads: zero opacity near 0.
KNOTS_X = np.arange(8) / 7.0
KNOTS_RGBA = np.array([[0.00, 0.00, 0.00, 0.00], [0.10, 0.10, 0.60, 0.00], [0.10, 0.50, 0.90, 0.02],
                       [0.20, 0.80, 0.60, 0.06], [0.60, 0.90, 0.20, 0.12], [0.95, 0.75, 0.10, 0.25],
                       [0.95, 0.35, 0.10, 0.45], [1.00, 1.00, 1.00, 0.70]])

CAMERA = np.dtype([("R", "f4", 9), ("t", "f4", 3), ("fx", "f4"), ("fy", "f4"), ("cx", "f4"), ("cy", "f4"),
                   ("znear", "f4"), ("width", "i4"), ("height", "i4"), ("pad", "i4")])

# Launch configurations of the fine-tuner: its defaults, the one its usage example gives, and the ones
# its autotuner settles on for large batches and for batches of many sets.
CONFIGS = {
    "default": {},
    "example": dict(tile=(8, 8), ppt=1, group_lanes=4, bwd_ppt=2, bwd_group_lanes=4, persistent=True),
    "large": dict(tile=(8, 8), ppt=2, group_lanes=4, persistent=True, segment_len=512, recompute=True),
    "uneven": dict(tile=(8, 8), ppt=2, group_lanes=4, bwd_group_lanes=8, persistent=True, segment_len=512),
    "tall": dict(tile=(8, 16), ppt=4, group_lanes=4, bwd_group_lanes=8, persistent=True, segment_len=-1),
}


def listed():
    return [
        # the smallest volume: a test cube, where launches and host round trips count
        dict(name="build 32", kind="build", nx=32, ny=32, nz=32, levels=2, budget=10000),
        # a cropped scan, no two edges alike
        dict(name="build ragged", kind="build", nx=224, ny=160, nz=96, levels=4, budget=240000),
        # a simulation time step, the largest volume of the package's workloads
        dict(name="build 512", kind="build", nx=512, ny=512, nz=512, levels=5, budget=3000000),
        # a scan's RGBA pyramid
        dict(name="pyramid 256", kind="pyramid", nx=256, ny=256, nz=256, levels=4),
        # supervision images of a small volume, and of the largest
        dict(name="targets 128", kind="targets", nx=128, ny=128, nz=128, views=8, width=512, height=512, step=0.5),
        dict(name="targets 512", kind="targets", nx=512, ny=512, nz=512, views=8, width=1024, height=1024, step=0.5),
        # a viewer's frame of the largest set at full HD
        dict(name="view 1080p", kind="view", count=2883451, edge=512, width=1920, height=1080),
        # fine-tuning: a first try on one small view with the defaults, the usage example's batch, the
        # largest batch, and many small sets of uneven sizes at once
        dict(name="step small", kind="step", count=3370, edge=32, sets=1, views=1, width=128, height=128,
             config="default"),
        dict(name="step medium", kind="step", count=99654, edge=128, sets=1, views=8, width=512, height=512,
             config="example"),
        dict(name="step large", kind="step", count=2883451, edge=512, sets=1, views=8, width=1024, height=1024,
             config="large"),
        dict(name="step uneven", kind="step", count=872010, edge=128, sets=32, views=4, width=256, height=256,
             config="uneven"),
        # a training loop of one's own, on images of odd size
        dict(name="loop odd", kind="loop", count=12007, edge=72, views=3, width=509, height=347),
    ]


def _between(rng, lo, hi):
    """A whole number from lo to hi, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, multiple):
    e = [max(multiple, multiple * round(_between(rng, 32, 512) / multiple)) for _ in range(3)]
    return [min(512, x) for x in e]


def draw(rng):
    kind = rng.choice(["build", "pyramid", "targets", "view", "step", "step", "loop"])
    if kind in ("build", "pyramid"):
        levels = rng.randint(1, 5)
        nx, ny, nz = _edges(rng, 1 << levels)
        case = dict(kind=kind, nx=nx, ny=ny, nz=nz, levels=levels)
        if kind == "build":
            case["budget"] = max(100, int(nx * ny * nz * rng.uniform(0.02, 0.1)) if nx * ny * nz < 2 ** 25 else
                                 int(nx * ny * nz * 0.022))
        return case
    if kind == "targets":
        nx, ny, nz = _edges(rng, 1)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, views=rng.randint(1, 8), width=_between(rng, 64, 1024),
                    height=_between(rng, 64, 1024), step=rng.choice([0.5, 0.5, 1.0]))
    if kind == "view":
        count = _between(rng, 3000, 2800000)
        return dict(kind=kind, count=count, edge=_edge_for(count), width=_between(rng, 320, 1920),
                    height=_between(rng, 240, 1080))
    if kind == "loop":
        count = _between(rng, 500, 12000)
        return dict(kind=kind, count=count, edge=_edge_for(count), views=rng.randint(1, 3),
                    width=_between(rng, 32, 509), height=_between(rng, 32, 347))
    sets = rng.choice([1, 1, 1, rng.randint(2, 24)])
    views = rng.randint(1, 8) if sets == 1 else rng.randint(1, 4)
    count = _between(rng, 2000, 2000000 if sets == 1 else 600000)
    side = 1024 if sets == 1 else 256
    return dict(kind=kind, count=count, edge=_edge_for(count) if sets == 1 else 64, sets=sets, views=views,
                width=_between(rng, 64, side), height=_between(rng, 64, side),
                config=rng.choice(sorted(CONFIGS)))


def _edge_for(count):
    """Edge of the volume that keeps about `count` coefficients (4.5% of its voxels), a multiple of 8."""
    return int(min(512, max(32, 8 * round((count / 0.045) ** (1 / 3) / 8))))


# ------------------------------------------------------------------ inputs

def _noise(dims, gen, power, k_max):
    """Zero-mean, unit-std field with amplitude |k|^-power up to k_max cycles along an axis."""
    nx, ny, nz = dims
    spec = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device=DEVICE))
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device=DEVICE)[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=DEVICE)[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device=DEVICE)[None, None, :]
    k = (kx * kx + ky * ky + kz * kz).sqrt()
    spec *= torch.where((k >= 1) & (k <= k_max), k.clamp(min=1) ** -power, torch.zeros_like(k))
    f = torch.fft.irfftn(spec, s=(nz, ny, nx))
    return (f - f.mean()) / f.std()


def _field(dims, gen, shells):
    """A scalar field in [0, 1]: five noisy shells round a core, or blobs with band-limited noise."""
    nx, ny, nz = dims
    if shells:
        z, y, x = (((torch.arange(n, device=DEVICE) + 0.5) / n - 0.5) for n in (nz, ny, nx))
        r = (x[None, None, :] ** 2 + y[None, :, None] ** 2 + z[:, None, None] ** 2).sqrt()
        n = _noise(dims, gen, 11 / 6, max(dims) / 4)
        f = torch.exp(-r * r / (2 * 0.05 ** 2))
        for rel, amp in zip((0.2, 0.35, 0.5, 0.65, 0.8), (0.4, 0.5, 0.6, 0.7, 0.8)):
            R = rel / 2
            f += amp * torch.exp(-(r - R * (1 + 0.1 * n)) ** 2 / (2 * 0.015 ** 2))
        return f.clamp_(0, 1).contiguous()
    blobs = max(4, min(64, round(4 * (nx * ny * nz) / 32 ** 3)))
    amp = 0.2 + 0.8 * torch.rand(blobs, generator=gen, device=DEVICE)
    axis = []
    for n in (nz, ny, nx):
        c = n * (0.2 + 0.6 * torch.rand((blobs, 1), generator=gen, device=DEVICE))
        s = (1.5 + 3.5 * torch.rand((blobs, 1), generator=gen, device=DEVICE)) * max(1.0, n / 96)
        axis.append(torch.exp(-((torch.arange(n, device=DEVICE) + 0.5)[None] - c) ** 2 / (2 * s * s)))
    planes = (amp[:, None, None] * axis[0][:, :, None] * axis[1][:, None, :]).reshape(blobs, nz * ny)
    f = (planes.t() @ axis[2]).reshape(nz, ny, nx)
    f += 0.05 * _noise(dims, gen, 2.0, 16)
    return f.clamp_(0, 1).contiguous()


def _transfer(f, dtype):
    """The transfer function on a tensor of scalars: shape + (4,), from the knots as float32 holds them."""
    x = torch.tensor(KNOTS_X.astype(np.float32), device=DEVICE).to(dtype)
    rgba = torch.tensor(KNOTS_RGBA.astype(np.float32), device=DEVICE).to(dtype)
    f = f.to(dtype).clamp(0, 1)
    i = (torch.bucketize(f, x, right=True) - 1).clamp(0, len(x) - 2)
    t = ((f - x[i]) / (x[i + 1] - x[i]))[..., None]
    return (1 - t) * rgba[i] + t * rgba[i + 1]


def _orbit(dims, views, width, height):
    """Cameras on an orbit at 1.8 times the longest edge, as packed records."""
    recs = np.zeros(views, dtype=CAMERA)
    centre, reach = np.asarray(dims) / 2.0, 1.8 * max(dims)
    focal = (height / 2.0) / math.tan(math.radians(30))
    for v in range(views):
        az, el = 2 * math.pi * v / views + math.pi / 7, math.radians(20 if v % 2 == 0 else -20)
        back = np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
        f = -back
        r = np.cross(f, [0.0, 0.0, 1.0])
        r /= np.linalg.norm(r)
        R = np.stack([r, np.cross(f, r), f])
        recs[v]["R"] = R.reshape(9)
        recs[v]["t"] = -R @ (centre + reach * back)
        for key, val in (("fx", focal), ("fy", focal), ("cx", width / 2.0), ("cy", height / 2.0), ("znear", 0.2),
                         ("width", width), ("height", height)):
            recs[v][key] = val
    return recs


def _march(field, cams, step, dtype):
    """Emission-absorption images (views, 4, H, W) in plain torch: midpoint samples, trilinear, black background.
    Every camera has the same image size; all views' rays march together."""
    nz, ny, nx = field.shape
    W, H = int(cams[0]["width"]), int(cams[0]["height"])
    flat, box = field.reshape(-1).to(dtype), torch.tensor([nx, ny, nz], dtype=dtype, device=DEVICE)
    rays = []
    for cam in cams:
        R = torch.tensor(cam["R"].astype(np.float64).reshape(3, 3), dtype=dtype, device=DEVICE)
        t = torch.tensor(cam["t"].astype(np.float64), dtype=dtype, device=DEVICE)
        px = (torch.arange(W, device=DEVICE, dtype=dtype) + 0.5 - float(cam["cx"])) / float(cam["fx"])
        py = (torch.arange(H, device=DEVICE, dtype=dtype) + 0.5 - float(cam["cy"])) / float(cam["fy"])
        d = px[None, :, None] * R[0] + py[:, None, None] * R[1] + R[2]
        rays.append(((-(R * t[:, None]).sum(0)).expand(H * W, 3), d.reshape(-1, 3)))
    o, d = (torch.cat([r[k] for r in rays]) for k in (0, 1))
    d = d / d.norm(dim=1, keepdim=True)
    ta, tb = (0 - o) / d, (box - o) / d
    t0 = torch.minimum(ta, tb).amax(1).clamp(min=0)
    t1 = torch.maximum(ta, tb).amin(1)
    hit = (t1 > t0).nonzero()[:, 0]
    o, d, t0, t1 = o[hit].t().contiguous(), d[hit].t().contiguous(), t0[hit], t1[hit]
    C, T = torch.zeros((len(hit), 3), dtype=dtype, device=DEVICE), torch.ones(len(hit), dtype=dtype, device=DEVICE)
    dx, dy, dz = int(nx > 1), nx * int(ny > 1), nx * ny * int(nz > 1)
    for m in range(int(((t1 - t0) / step).ceil().max().item()) if len(hit) else 0):
        begin = t0 + m * step
        seg = (t1 - begin).clamp(0, step)
        tm = begin + 0.5 * seg
        corner, frac = [], []
        for k, n in enumerate((nx, ny, nz)):
            q = (o[k] + tm * d[k] - 0.5).clamp(0, n - 1)
            i = q.floor().clamp(max=max(n - 2, 0))
            corner.append(i.long())
            frac.append(q - i)
        at = (corner[2] * ny + corner[1]) * nx + corner[0]
        fx, fy, fz = frac
        val = 0
        for bz, wz in ((0, 1 - fz), (dz, fz)):
            for by, wy in ((0, 1 - fy), (dy, fy)):
                val = val + wz * wy * torch.lerp(flat[at + bz + by], flat[at + bz + by + dx], fx)
        rgba = _transfer(val, dtype)
        a = 1 - (1 - rgba[:, 3]) ** seg
        C += (T * a)[:, None] * rgba[:, :3]
        T = T * (1 - a)
    img = torch.zeros((len(cams) * H * W, 4), dtype=dtype, device=DEVICE)
    img[hit, :3] = C
    img[hit, 3] = 1 - T
    return img.reshape(len(cams), H, W, 4).permute(0, 3, 1, 2).contiguous()


def _splats(field, count, gen):
    """Gaussians P[14][count] where the field has detail, some iterations into their fine-tuning."""
    alpha = _transfer(field, torch.float32)[..., 3][None, None]
    nz, ny, nx = field.shape
    levels = max(1, min(3, int(math.log2(min(nx, ny, nz) / 8))))
    share = ([1.0], [0.67, 0.33], [0.64, 0.32, 0.04])[levels - 1]
    rows, left = [], count
    for j in range(1, levels + 1):
        s = 1 << j
        hi = torch.nn.functional.max_pool3d(alpha, s)
        detail = (hi + torch.nn.functional.max_pool3d(-alpha, s)).reshape(-1)
        cz, cy, cx = hi.shape[2:]
        for code in range(1, 8):
            last = j == levels and code == 7
            n = min(left if last else int(count * share[j - 1] / 7), detail.numel())
            left -= n
            noise = -torch.log(-torch.log(torch.rand(detail.numel(), generator=gen, device=DEVICE).clamp(1e-6, 1 - 1e-6)))
            at = torch.topk(torch.log(detail + 1e-4) + 0.3 * noise, n).indices.sort().values
            o = torch.tensor([code & 1, (code >> 1) & 1, code >> 2], device=DEVICE, dtype=torch.float32)[:, None]
            k = torch.stack([at % cx, (at // cx) % cy, at // (cx * cy)]).float()
            P = torch.empty((14, n), device=DEVICE)
            P[0:3] = s * k + 0.5 + o * (s / 2) + 0.1 * s * torch.randn((3, n), generator=gen, device=DEVICE)
            P[3:6] = torch.log(s * (0.34 + 0.09 * o)) - 0.1 + 0.15 * torch.randn((3, n), generator=gen, device=DEVICE)
            P[6:10] = 0.05 * torch.randn((4, n), generator=gen, device=DEVICE)
            P[6] += 1
            P[10] = -4.6 + 1.2 * torch.randn(n, generator=gen, device=DEVICE)
            P[11:14] = torch.exp(-2 + torch.randn((3, n), generator=gen, device=DEVICE)).clamp(max=1.5)
            rows.append(P)
    if left:    # more than the field has cells: any place inside it
        P = rows[0][:, torch.randint(rows[0].shape[1], (left,), generator=gen, device=DEVICE)].clone()
        P[0:3] += torch.randn((3, left), generator=gen, device=DEVICE)
        rows.append(P)
    return torch.cat(rows, dim=1).contiguous()


class State:
    """What a program keeps between calls."""

    def __init__(self, **kw):
        self.__dict__.update(kw)


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _scene(case, seed):
    """(params, camera records, targets, scene offsets, view -> scene) of a step or loop case."""
    gen = _generator(seed)
    sets = case.get("sets", 1)
    if sets == 1:
        dims = (case["edge"],) * 3
        field = _field(dims, gen, shells=case["edge"] >= 384)
        cams = _orbit(dims, case["views"], case["width"], case["height"])
        targets = _march(field, cams, case["edge"] / 48.0, torch.float32)[:, :3].contiguous()
        return _splats(field, case["count"], gen), cams, targets, None, None
    # sets of uneven sizes, each with its own field and cameras
    edges = torch.tensor([32, 48, 64, 96, 128])
    pick = torch.randint(5, (sets,), generator=torch.Generator().manual_seed(sets))     # a case's sizes are its own
    edges = edges[pick].clamp(max=case["edge"]).tolist()
    weight = [e ** 3 for e in edges]
    counts = [max(1, int(case["count"] * w / sum(weight))) for w in weight]
    P, cams, targets, offset, view_scene = [], [], [], [0], []
    for i, (e, n) in enumerate(zip(edges, counts)):
        field = _field((e, e, e), gen, shells=False)
        c = _orbit((e, e, e), case["views"], case["width"], case["height"])
        P.append(_splats(field, n, gen))
        cams.append(c)
        targets.append(_march(field, c, e / 20.0, torch.float32)[:, :3])
        offset.append(offset[-1] + P[-1].shape[1])
        view_scene += [i] * case["views"]
    return (torch.cat(P, 1).contiguous(), np.concatenate(cams), torch.cat(targets).contiguous(),
            np.asarray(offset, dtype=np.int64), np.asarray(view_scene, dtype=np.int32))


def _lrs(case):
    return [1e-3 * lr for lr in default_lrs(case["edge"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("build", "pyramid", "targets"):
        dims = (case["nx"], case["ny"], case["nz"])
        field = _field(dims, _generator(seed), shells=min(dims) >= 384)
        tf = vbm.make_tf(KNOTS_X, KNOTS_RGBA)
        if kind == "build":
            return State(kind=kind, field=field, dims=dims, tf=tf, bank=vbm.bank_build(case["levels"]),
                         select=vbm.make_select(case["budget"]), capacity=2 * case["budget"] + 1024)
        if kind == "pyramid":
            return State(kind=kind, field=field, dims=dims, tf=tf, levels=case["levels"],
                         out=torch.empty((4,) + tuple(field.shape), device=DEVICE),
                         tmp=torch.empty(2 * field.numel(), device=DEVICE))
        cams = _orbit(dims, case["views"], case["width"], case["height"])
        return State(kind=kind, field=field, dims=dims, tf=tf, cams=vbm.cameras_to_device(cams), views=case["views"],
                     width=case["width"], height=case["height"], step=case["step"],
                     out=torch.empty((case["views"], 4, case["height"], case["width"]), device=DEVICE))
    W, H = case["width"], case["height"]
    if kind == "view":
        gen = _generator(seed)
        dims = (case["edge"],) * 3
        params = _splats(_field(dims, gen, shells=case["edge"] >= 384), case["count"], gen)
        n = params.shape[1]
        plan = vbm.Plan([0, n], 1, W, H, tile_w=8, tile_h=8, pair_capacity=vbm.default_pair_capacity(n),
                        flags=vbm.PLAN_PERSISTENT, pixels_per_thread=2, group_lanes=4)
        return State(kind=kind, params=params, plan=plan, cams=vbm.cameras_to_device(_orbit(dims, 1, W, H)),
                     img=torch.zeros((1, 3, H, W), device=DEVICE), alpha=torch.zeros((1, H, W), device=DEVICE))
    params, cams, targets, offset, view_scene = _scene(case, seed)
    if kind == "step":
        return State(kind=kind, tuner=FineTuner(params, cams, targets, scene_offset=offset, view_scene=view_scene,
                                                lrs=_lrs(case), **CONFIGS[case["config"]]))
    n, V = params.shape[1], case["views"]
    params.requires_grad_(True)
    return State(kind=kind, params=params, cams=vbm.cameras_to_device(cams), targets=targets, n=n, lrs=_lrs(case),
                 plan=vbm.Plan([0, n], V, W, H, pair_capacity=vbm.default_pair_capacity(n * V)),
                 m=torch.zeros((14, n), device=DEVICE), v=torch.zeros((14, n), device=DEVICE),
                 step=torch.zeros(1, dtype=torch.int32, device=DEVICE), ws=vbm.loss_workspace(V, H, W),
                 loss=torch.zeros(1, dtype=torch.float64, device=DEVICE), dimg=torch.empty_like(targets))


def run(s):
    if s.kind == "build":
        params, n = vbm.build(s.field, s.dims, s.tf, s.bank, s.select, s.capacity)
        return {"params": params, "n": n}
    if s.kind == "pyramid":
        vbm.tf_apply(s.field, s.tf, s.out)
        vbm.dwt3d(s.out, 4, s.dims, s.levels, 0, s.tmp)
        return s.out
    if s.kind == "targets":
        vbm.render_dvr(s.field, s.dims, s.tf, s.cams, s.views, s.width, s.height, s.step, s.out)
        return s.out
    if s.kind == "view":
        s.plan.forward(s.params, s.cams, s.img, alpha=s.alpha)
        return {"img": s.img, "alpha": s.alpha}
    if s.kind == "step":
        s.tuner.step_graph()
        t = s.tuner
        return {"params": t.params, "m": t.m, "v": t.v, "img": t.img, "loss": t.loss}
    V, _, H, W = s.targets.shape
    img = render(s.params, s.plan, s.cams)
    vbm.loss(img, s.targets, V, H, W, 0.2, 1.0 / img.numel(), s.loss, s.dimg, s.ws)
    grad, = torch.autograd.grad(img, s.params, s.dimg)
    with torch.no_grad():
        vbm.adam(s.params, grad, s.m, s.v, s.n, s.step, s.lrs)
    return {"params": s.params, "m": s.m, "v": s.v, "img": img, "loss": s.loss, "grad": grad}


def work(case):
    """Bytes: each input read once, each output written once.  Flops: the arithmetic of the method; where
    it depends on the data, of a typical set (the kept share of a budget, half of the images' rays inside
    the box, thirty splats evaluated per pixel)."""
    kind = case["kind"]
    if kind in ("build", "pyramid"):
        n = case["nx"] * case["ny"] * case["nz"]
        flops = n * (12 + 4 * 3 * 8 * 2 * (1 - 8.0 ** -case["levels"]) * 8 / 7)
        if kind == "pyramid":
            return {"bytes": 20 * n, "flops": flops}
        return {"bytes": 4 * n + 56 * 0.6 * case["budget"], "flops": flops + 40 * n}
    pixels = case["width"] * case["height"] * case.get("views", 1) * case.get("sets", 1)
    if kind == "targets":
        samples = 0.5 * pixels * 0.8 * (case["nx"] + case["ny"] + case["nz"]) / 3 / case["step"]
        return {"bytes": 4 * case["nx"] * case["ny"] * case["nz"] + 16 * pixels, "flops": 70 * samples}
    n = case["count"]
    if kind == "view":
        return {"bytes": 56 * n + 16 * pixels, "flops": 250 * n + 30 * 21 * pixels}
    items = n * case["views"]
    return {"bytes": 6 * 56 * n + 24 * pixels, "flops": 650 * items + (30 * 82 + 3 * 392) * pixels}


# ------------------------------------------------- the same in 64 bits, plain torch

def _cdf97():
    """The 9-tap low-pass and 7-tap dual of the Cohen-Daubechies-Feauveau 9/7 pair, from their construction:
    cos^8(w/2) P(sin^2(w/2)) with P = 1 + 4x + 10x^2 + 20x^3, the real root to the short filter."""
    roots = np.roots([20.0, 10.0, 4.0, 1.0])
    xr = float(roots[np.argmin(abs(roots.imag))].real)
    for _ in range(4):
        xr -= np.polyval([20, 10, 4, 1.0], xr) / np.polyval([60, 20, 4.0], xr)
    q = np.polydiv([20.0, 10.0, 4.0, 1.0], [20.0, -20.0 * xr])[0]
    sin2, cos4 = np.array([-0.25, 0.5, -0.25]), np.convolve([0.25, 0.5, 0.25], [0.25, 0.5, 0.25])
    short = np.convolve(cos4, np.array([0, 1.0, 0]) - sin2 / xr)
    pair = q[0] * np.convolve(sin2, sin2)
    pair[1:4] += q[1] * sin2
    pair[2] += q[2]
    long = np.convolve(cos4, pair)
    return long * (math.sqrt(2) / long.sum()), short * (math.sqrt(2) / short.sum())


def _exact_pyramid(field, levels):
    out = _transfer(field, torch.float64).permute(3, 0, 1, 2).contiguous()
    low, dual = _cdf97()
    high = [(-1.0) ** abs(n) * dual[n + 3] for n in range(-3, 4)]
    nz, ny, nx = field.shape
    for j in range(levels):
        region = out[:, :nz >> j, :ny >> j, :nx >> j]
        for axis in (3, 2, 1):
            n = region.shape[axis]
            at = torch.arange(0, n, 2, device=DEVICE)
            a = sum(w * region.index_select(axis, (at + k - 4) % n) for k, w in enumerate(low))
            d = sum(w * region.index_select(axis, (at + 1 + k - 3) % n) for k, w in enumerate(high))
            region = torch.cat([a, d], axis)
        out[:, :nz >> j, :ny >> j, :nx >> j] = region
    return out


def _project(P, cam, tile):
    """The splats of one view in 64 bits, as the renderer defines them, in depth order."""
    R = torch.tensor(cam["R"].astype(np.float64).reshape(3, 3), device=DEVICE)
    t = torch.tensor(cam["t"].astype(np.float64), device=DEVICE)
    f, (cx, cy), (W, H) = float(cam["fx"]), (float(cam["cx"]), float(cam["cy"])), (int(cam["width"]), int(cam["height"]))
    order = (R[2] @ P[0:3].detach() + t[2]).argsort(stable=True)
    P = P[:, order]
    p = R @ P[0:3] + t[:, None]
    q = P[6:10] / P[6:10].norm(dim=0, keepdim=True)
    w, x, y, z = q
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                       1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                       1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)
    M = rot * torch.exp(P[3:6]).t()[:, None, :]
    xz, yz = p[0] / p[2], p[1] / p[2]
    xc = xz.clamp((-0.15 * W - cx) / f, (1.15 * W - cx) / f)
    yc = yz.clamp((-0.15 * H - cy) / f, (1.15 * H - cy) / f)
    zero = torch.zeros_like(xz)
    J = torch.stack([f / p[2], zero, -f * xc / p[2], zero, f / p[2], -f * yc / p[2]], -1).reshape(-1, 2, 3)
    V = J @ R @ M
    S = V @ V.transpose(1, 2)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * c - b * b
    opac = torch.sigmoid(P[10])
    u, v = f * xz + cx, f * yz + cy
    with torch.no_grad():
        mid = 0.5 * (a + c)
        k = torch.sqrt(2 * torch.log(255 * opac).clamp(min=0)).clamp(max=3)
        r = torch.ceil(k * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        seen = (p[2] > float(cam["znear"])) & (det > 0) & (opac >= 1 / 255)
        lo = [torch.floor((torch.floor(m) - r) / tile) for m in (u, v)]
        hi = [torch.floor((torch.floor(m) + r) / tile) for m in (u, v)]
    return dict(u=u, v=v, A=c / det, B=-b / det, C=a / det, o=opac, rgb=P[11:14], seen=seen, lo=lo, hi=hi)


def _render_rows(s, rows, W, tile):
    """Rows of the image (3, len(rows), W) by compositing every splat at every pixel."""
    y, x = torch.meshgrid(rows.double(), torch.arange(W, device=DEVICE).double(), indexing="ij")
    x, y = x.reshape(-1, 1), y.reshape(-1, 1)
    tx, ty = torch.floor(x / tile), torch.floor(y / tile)
    # splats that no pixel of these rows lists
    near = s["seen"] & (s["lo"][1] <= ty.max()) & (s["hi"][1] >= ty.min())
    at = near.nonzero()[:, 0]
    u, v, A, B, C, o = (s[k][at] for k in ("u", "v", "A", "B", "C", "o"))
    dx, dy = u - (x + 0.5), v - (y + 0.5)
    power = -0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy
    alpha = (o * torch.exp(power)).clamp(max=0.99)
    with torch.no_grad():
        on = (power <= 0) & (alpha >= 1 / 255) & (s["lo"][0][at] <= tx) & (s["hi"][0][at] >= tx) \
            & (s["lo"][1][at] <= ty) & (s["hi"][1][at] >= ty)
    alpha = torch.where(on, alpha, torch.zeros_like(alpha))
    keep = torch.cumprod(1 - alpha, 1)
    live = keep.detach() >= 1e-4        # false from the splat on that would take it below
    before = torch.cat([torch.ones_like(keep[:, :1]), keep[:, :-1]], 1)
    weight = torch.where(live, alpha * before, torch.zeros_like(alpha))
    return (s["rgb"][:, at] @ weight.t()).reshape(3, len(rows), W)


def _exact_step(case, seed):
    """One training step from the prepared state: image, loss, gradient and Adam's update."""
    params, cams, targets, _, _ = _scene(case, seed)
    tile, V, H, W = 16, case["views"], case["height"], case["width"]
    P = params.double().requires_grad_(True)
    rows = max(1, int(4e8 / (W * P.shape[1])))
    img = torch.empty((V, 3, H, W), dtype=torch.float64, device=DEVICE)

    def blocks():
        for v in range(V):
            for r in range(0, H, rows):
                yield v, torch.arange(r, min(H, r + rows), device=DEVICE)

    with torch.no_grad():
        for v, r in blocks():
            img[v][:, r] = _render_rows(_project(P, cams[v], tile), r, W, tile)
    x, y = img.clone().requires_grad_(True), targets.double()
    g = torch.exp(-(torch.arange(11, device=DEVICE).double() - 5) ** 2 / 4.5)
    g = g / g.sum()

    def window(m):
        m = torch.nn.functional.pad(m.reshape(-1, H, W), (5, 5, 5, 5))
        m = sum(g[k] * m[:, :, k:k + W] for k in range(11))
        return sum(g[k] * m[:, k:k + H] for k in range(11)).reshape(V, 3, H, W)

    mx, my = window(x), window(y)
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = (2 * mx * my + c1) * (2 * (window(x * y) - mx * my) + c2) / (
        (mx * mx + my * my + c1) * (window(x * x) - mx * mx + window(y * y) - my * my + c2))
    loss = 0.8 * (x - y).abs().mean() + 0.2 * (1 - ssim).mean()
    dimg, = torch.autograd.grad(loss, x)
    grad = torch.zeros_like(P)
    for v, r in blocks():
        part, = torch.autograd.grad(_render_rows(_project(P, cams[v], tile), r, W, tile), P, dimg[v][:, r])
        grad += part
    lr = torch.tensor(np.repeat(_lrs(case), [3, 3, 4, 1, 3]), device=DEVICE)[:, None]
    m, v2 = 0.1 * grad, 0.001 * grad * grad
    new = P.detach() - lr * (m / 0.1) / ((v2 / 0.001).sqrt() + 1e-15)
    out = {"params": new, "m": m, "v": v2, "img": img, "loss": loss.detach().reshape(1)}
    if case["kind"] == "loop":
        out["grad"] = grad
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "pyramid":
        dims = (case["nx"], case["ny"], case["nz"])
        return _exact_pyramid(_field(dims, _generator(seed), shells=min(dims) >= 384), case["levels"])
    if kind == "targets":
        dims = (case["nx"], case["ny"], case["nz"])
        field = _field(dims, _generator(seed), shells=min(dims) >= 384)
        return _march(field, _orbit(dims, case["views"], case["width"], case["height"]), case["step"], torch.float64)
    pairs = case.get("count", 0) * case.get("views", 1) * case.get("width", 0) * case.get("height", 0)
    if kind == "loop" or (kind == "step" and case["sets"] == 1 and case["config"] == "default" and pairs < 1.2e10):
        return _exact_step(case, seed)
    # build: which coefficients are kept is decided on rounded float32 magnitudes; view and the larger
    # steps: compositing every splat at every pixel takes too long
    return None
