"""The work that programs have this simulator do, as cases to be timed.

Each case is one call (or one training step) through the public Python binding
of the C ABI: rendering transients of a scene, the detector's steps on a cube,
a gradient step through the differentiable splat, the paper's depth-map forward
model, and a burst of requests to the server. The sizes are those of the
benchmark's workloads, of the paper's dataset (128 x 128 scans, 1024 bins of
32 ps) and of the serving trace; ``draw`` spreads over the same ranges.

``exact`` is the definition in 64 bits with plain torch: the sum over every
(scan point, surface point) pair, the taps of the jitter, and the depth-map
model's convolution summed over its nonzeros.
"""
import math
import random

import numpy as np
import torch

from paper_2506_03747_gb300 import nlos
from paper_2506_03747_gb300.autograd import NlosSplat

C = 299792458.0
DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------
def _simulate(name, **kw):
    c = dict(name=name, kind="simulate", scan_nx=64, scan_ny=64, wall_half=1.0, scan_mode="confocal",
             cos_mode="object", num_bins=512, bin_ps=8.0, fwhm_ps=60.0, padding="zero", standoff=1.0,
             scene="union", points=262144, refresh=True, occluders=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call a program makes: one confocal preview of a flat glyph
        # without jitter, where launches and latency are what it costs
        _simulate("preview_plane32", scan_nx=32, scan_ny=32, wall_half=0.5, num_bins=256, bin_ps=16.0,
                  fwhm_ps=0.0, standoff=0.0, scene="glyph", points=1024, refresh=False),
        # a dataset renderer's ordinary scene: new surface samples, then the
        # confocal transient with stand-off and jitter
        _simulate("render_union64"),
        # the largest single scene of the benchmark: a non-confocal 128 x 128 scan
        # of a million-point heightfield
        _simulate("render_heightfield128", scan_nx=128, scan_ny=128, scan_mode="nonconfocal",
                  num_bins=1024, bin_ps=4.0, fwhm_ps=30.0, standoff=1.5, scene="heightfield",
                  points=1048576),
        # a user's own scanner: a rectangular scan and an odd number of bins and
        # points, wall cosines, edge bins continued under the jitter
        _simulate("render_ragged", scan_nx=75, scan_ny=52, scan_mode="nonconfocal",
                  cos_mode="object_wall", num_bins=701, bin_ps=6.5, fwhm_ps=45.0, padding="replicate",
                  scene="heightfield", points=40001),
        # the paper's dataset entry by the direct sum: a 128 x 128 depth map under
        # Eq. 1 as printed (no cosines), 1024 bins of 32 ps, 70 ps jitter
        _simulate("dataset_depthmap128", scan_nx=128, scan_ny=128, cos_mode="none", num_bins=1024,
                  bin_ps=32.0, fwhm_ps=70.0, standoff=0.0, scene="depthmap", points=16384),
        # a scene that shadows itself: the union's own solids as occluders
        _simulate("render_occluded64", occluders=True, refresh=False),
        # the detector on a rendered cube: per-transient energy and Poisson counts
        dict(name="detect_cube128", kind="detect", scan_nx=128, scan_ny=128, num_bins=1024,
             noise_mode="peak", photons=100.0),
        # the detector's timing jitter on a cube that came from elsewhere
        dict(name="jitter_cube128", kind="jitter", traces=16384, num_bins=1024, fwhm_bins=7.5,
             padding="zero"),
        # one step of shape and albedo recovery on a glyph scene: the splat
        # forward and the gradients, at 60 ps jitter (3.2 bins standard deviation)
        dict(name="train_glyph64", kind="train", scan_nx=64, scan_ny=64, scan_mode="confocal",
             cos_mode="object", num_bins=512, bin_ps=8.0, fwhm_ps=60.0, points=65536),
        # the same for a fast detector (30 ps: 1.6 bins), non-confocal
        dict(name="train_sharp32", kind="train", scan_nx=32, scan_ny=32, scan_mode="nonconfocal",
             cos_mode="object", num_bins=512, bin_ps=8.0, fwhm_ps=30.0, points=16384),
        # the paper's own forward model on its dataset shape
        dict(name="lct_dataset128", kind="lct", n=128, m=1024, bin_ps=32.0, wall_half=1.0,
             albedo=True),
        # eight requests of mixed sizes at once, as a serving process gets them
        dict(name="serve_burst8", kind="serve", requests=8, trace=5, side_lo=16, side_hi=128,
             bins_lo=256, bins_hi=1024, points_lo=10000, points_hi=200000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate"] * 5 + ["detect", "jitter", "train", "train", "lct", "serve"])
    if kind == "simulate":
        scene = rng.choice(["glyph", "union", "heightfield", "depthmap"])
        nx = _log(rng, 12, 160)
        ny = nx if rng.random() < 0.5 else _log(rng, 12, 160)
        pts = _log(rng, 500, 1200000)
        while nx * ny * pts > 1.7e10:
            pts = max(500, pts // 2)
        bin_ps = rng.uniform(4.0, 32.0)
        standoff = rng.choice([0.0, 1.0, 1.5])
        return dict(kind=kind, scan_nx=nx, scan_ny=ny, wall_half=rng.choice([0.5, 1.0]),
                    scan_mode=rng.choice(["confocal", "nonconfocal"]),
                    cos_mode=rng.choice(["none", "object", "object_wall"]),
                    num_bins=_log(rng, 200, 2048), bin_ps=bin_ps,
                    fwhm_ps=rng.choice([0.0, rng.uniform(30.0, 70.0)]),
                    padding=rng.choice(["zero", "zero", "replicate"]), standoff=standoff, scene=scene,
                    points=pts, refresh=rng.random() < 0.6,
                    occluders=scene == "union" and rng.random() < 0.5)
    if kind == "detect":
        return dict(kind=kind, scan_nx=_log(rng, 16, 160), scan_ny=_log(rng, 16, 160),
                    num_bins=_log(rng, 200, 1500), noise_mode=rng.choice(["peak", "peak", "paper_nr"]),
                    photons=math.exp(rng.uniform(math.log(5.0), math.log(500.0))))
    if kind == "jitter":
        return dict(kind=kind, traces=_log(rng, 256, 20000), num_bins=_log(rng, 200, 2048),
                    fwhm_bins=rng.uniform(1.0, 18.0), padding=rng.choice(["zero", "replicate"]))
    if kind == "train":
        nx = _log(rng, 12, 64)
        bin_ps = rng.uniform(4.0, 16.0)
        return dict(kind=kind, scan_nx=nx, scan_ny=_log(rng, 12, 64),
                    scan_mode=rng.choice(["confocal", "nonconfocal"]),
                    cos_mode=rng.choice(["none", "object", "object_wall"]),
                    num_bins=_log(rng, 200, 1024), bin_ps=bin_ps, fwhm_ps=rng.uniform(30.0, 70.0),
                    points=_log(rng, 1000, 65536))
    if kind == "lct":
        return dict(kind=kind, n=2 ** rng.randint(4, 7), m=2 ** rng.randint(6, 10),
                    bin_ps=rng.uniform(16.0, 48.0), wall_half=rng.choice([0.5, 1.0]),
                    albedo=rng.random() < 0.7)
    return dict(kind=kind, requests=rng.randint(1, 12), trace=rng.randint(0, 10 ** 6), side_lo=16,
                side_hi=_log(rng, 32, 128), bins_lo=256, bins_hi=_log(rng, 300, 1024), points_lo=5000,
                points_hi=_log(rng, 10000, 200000))


# ---------------------------------------------------------------------------
# Inputs, on the GPU and from the seed alone.
# ---------------------------------------------------------------------------
class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def u(self, *shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def n(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def beta22(self, n):  # the middle of three uniforms
        return self.u(3, n).sort(dim=0).values[1]


def _records(pos, nrm, albedo, area):
    return torch.cat([pos, nrm, albedo[:, None], area[:, None]], dim=1).float().contiguous()


def _grid(n, half):
    c = -half + (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * (2.0 * half / n)
    return torch.meshgrid(c, c, indexing="xy")


def _glyph(r, points, half):
    """A fronto-parallel plane with a blocky albedo mask (8 x 8 blocks of 0 or 1)."""
    n = math.isqrt(points - 1) + 1
    x, y = _grid(n, half)
    z = r.u(1, lo=0.45, hi=0.55).expand(n * n)
    mask = (r.u(8, 8) < 0.5).double()
    k = (torch.arange(n, device=DEV) * 8) // n
    alb = mask[k][:, k].reshape(-1)
    nrm = torch.zeros(n * n, 3, device=DEV, dtype=torch.float64)
    nrm[:, 2] = -1.0
    area = torch.full((n * n,), (2.0 * half / n) ** 2, device=DEV, dtype=torch.float64)
    pos = torch.stack([x.reshape(-1), y.reshape(-1), z], dim=1)
    return _records(pos, nrm, alb, area)[:points].contiguous()


def _heightfield(r, points, half):
    """Samples of a smooth random surface 0.4 to 1.5 m from the wall."""
    n = math.isqrt(points - 1) + 1
    x, y = _grid(n, half)
    z = torch.zeros_like(x)
    c, sg, amp = r.u(32, 2, lo=-half, hi=half), r.u(32, lo=0.1, hi=0.5), r.u(32, lo=-1.0, hi=1.0)
    zx, zy = torch.zeros_like(x), torch.zeros_like(x)
    for k in range(32):
        dx, dy = x - c[k, 0], y - c[k, 1]
        e = amp[k] * torch.exp(-(dx * dx + dy * dy) / (2.0 * sg[k] ** 2))
        z += e
        zx -= e * dx / sg[k] ** 2
        zy -= e * dy / sg[k] ** 2
    lo, scale = z.min(), 1.1 / (z.max() - z.min())
    z, zx, zy = 0.4 + scale * (z - lo), scale * zx, scale * zy
    s = torch.sqrt(1.0 + zx * zx + zy * zy)
    nrm = torch.stack([zx / s, zy / s, -1.0 / s], dim=-1).reshape(-1, 3)
    pos = torch.stack([x, y, z], dim=-1).reshape(-1, 3)
    area = ((2.0 * half / n) ** 2 * s).reshape(-1)
    return _records(pos, nrm, r.beta22(n * n), area)[:points].contiguous()


def _depthmap(r, points, half):
    """A depth map's pixels (a bump on a tilted plane), facing the wall."""
    n = math.isqrt(points - 1) + 1
    x, y = _grid(n, half)
    c = r.u(2, lo=-0.4, hi=0.4)
    z = 0.8 + 0.3 * torch.exp(-((x - c[0]) ** 2 + (y - c[1]) ** 2) / 0.1) + 0.1 * x
    pos = torch.stack([x, y, z], dim=-1).reshape(-1, 3)
    nrm = torch.zeros(n * n, 3, device=DEV, dtype=torch.float64)
    nrm[:, 2] = -1.0
    area = torch.full((n * n,), (2.0 * half / n) ** 2, device=DEV, dtype=torch.float64)
    return _records(pos, nrm, 0.2 + 0.8 * r.beta22(n * n), area)[:points].contiguous()


def _solids(r, half):
    """Three spheres and two boxes 0.3 to 1.2 m from the wall (kind, a, b)."""
    out = []
    for _ in range(3):
        rad = float(r.u(1, lo=0.1, hi=0.3))
        u = r.u(3).tolist()
        out.append((0, [(2 * u[0] - 1) * (half - rad), (2 * u[1] - 1) * (half - rad),
                        0.3 + rad + u[2] * (0.9 - 2 * rad)], [rad, 0.0, 0.0]))
    for _ in range(2):
        s, u = r.u(3, lo=0.1, hi=0.5).tolist(), r.u(3).tolist()
        a = [-half + u[0] * (2 * half - s[0]), -half + u[1] * (2 * half - s[1]),
             0.3 + u[2] * (0.9 - s[2])]
        out.append((1, a, [a[i] + s[i] for i in range(3)]))
    return out


def _union(r, points, half):
    """Area-uniform samples of the solids' outer surface, and the solids."""
    solids = _solids(r, half)
    areas = []
    for kind, a, b in solids:
        s = [b[i] - a[i] for i in range(3)]
        areas.append(4 * math.pi * b[0] ** 2 if kind == 0 else
                     2 * (s[0] * s[1] + s[1] * s[2] + s[0] * s[2]))
    got_p, got_n, n_got, tried = [], [], 0, 0
    while n_got < points:
        m = 2 * points
        edges = torch.tensor(np.cumsum(areas) / sum(areas), device=DEV)
        which = torch.bucketize(r.u(m), edges).clamp_(max=len(solids) - 1)
        v = r.n(m, 3)
        v = v / v.norm(dim=1, keepdim=True)
        t, f = r.u(m, 3), r.u(m)
        pos, nrm = torch.zeros_like(v), torch.zeros_like(v)
        for i, (kind, a, b) in enumerate(solids):
            lo = torch.tensor(a, device=DEV, dtype=torch.float64)
            if kind == 0:
                p_i, n_i = lo + b[0] * v, v
            else:
                hi = torch.tensor(b, device=DEV, dtype=torch.float64)
                s = hi - lo
                fa = torch.stack([s[1] * s[2], s[0] * s[2], s[0] * s[1]]).repeat_interleave(2)
                face = torch.bucketize(f, torch.cumsum(fa, 0) / fa.sum()).clamp_(max=5)
                axis, side = face // 2, face % 2
                one = torch.nn.functional.one_hot(axis, 3).double()
                p_i = (lo + t * s) * (1 - one) + one * torch.where(side[:, None] == 1, hi, lo)
                n_i = one * (2.0 * side[:, None] - 1.0)
            sel = (which == i)[:, None]
            pos, nrm = torch.where(sel, p_i, pos), torch.where(sel, n_i, nrm)
        keep = torch.ones(m, device=DEV, dtype=torch.bool)
        for i, (kind, a, b) in enumerate(solids):
            lo = torch.tensor(a, device=DEV, dtype=torch.float64)
            if kind == 0:
                inside = (pos - lo).norm(dim=1) < b[0]
            else:
                hi = torch.tensor(b, device=DEV, dtype=torch.float64)
                inside = ((pos > lo) & (pos < hi)).all(dim=1)
            keep &= ~(inside & (which != i))
        got_p.append(pos[keep])
        got_n.append(nrm[keep])
        n_got += int(keep.sum())
        tried += m
    area = sum(areas) * (n_got / tried) / points
    rec = _records(torch.cat(got_p)[:points], torch.cat(got_n)[:points], r.u(points, lo=0.2, hi=1.0),
                   torch.full((points,), area, device=DEV, dtype=torch.float64))
    occ = np.zeros((len(solids), 8), np.float32)
    for i, (kind, a, b) in enumerate(solids):
        occ[i, 0], occ[i, 1:4], occ[i, 4:7] = kind, a, b
    return rec, occ


def _scene(kind, r, points, half):
    if kind == "union":
        return _union(r, points, half)
    f = {"glyph": _glyph, "heightfield": _heightfield, "depthmap": _depthmap}[kind]
    return f(r, points, half), None


_NEAREST_Z = {"glyph": 0.45, "union": 0.3, "heightfield": 0.4, "depthmap": 0.7}


def _params(c):
    standoff, near = c.get("standoff", 0.0), 2.0 * _NEAREST_Z[c["scene"]]
    # with stand-off, or a window too short to reach the scene from the wall, the window
    # starts at the nearest part of the scene seen from the wall centre
    short = c["num_bins"] * c["bin_ps"] * 1e-12 * C < near + 0.3
    return dict(scan_nx=c["scan_nx"], scan_ny=c["scan_ny"], wall_half_x=c["wall_half"],
                wall_half_y=c["wall_half"], scan_mode=c["scan_mode"], laser_xy=(0.0, 0.0),
                cos_mode=c["cos_mode"], num_bins=c["num_bins"], bin_width_s=c["bin_ps"] * 1e-12,
                jitter_fwhm_s=c["fwhm_ps"] * 1e-12, jitter_padding=c.get("padding", "zero"),
                bin_mode=c.get("bin_mode", "nearest"), standoff_m=standoff,
                standoff_mode="euclidean" if standoff else "constant",
                window_start_m=2.0 * standoff + near if standoff or short else 0.0,
                noise_mode="none")


def _train_params(c):
    return _params(dict(c, wall_half=0.5, scene="glyph", bin_mode="splat"))


def _train_inputs(c, seed):
    """The base points, the albedo and normal offset of this step, and the
    gradient of the step's loss with respect to the transient."""
    r = _Rand(seed)
    pts = _glyph(r, c["points"], 0.5)
    pts[:, 6] = 0.1 + 0.9 * pts[:, 6]
    n = pts.shape[0]
    albedo = (pts[:, 6].double() * r.u(n, lo=0.8, hi=1.2)).float()
    depth = (2e-3 * r.n(n)).float()
    g = r.n(c["scan_nx"] * c["scan_ny"], c["num_bins"]).float()
    return pts, albedo, depth, g


def _cube(r, traces, bins):
    """A rendered cube: a peak per transient over a dim tail, few of the peaks bright
    (about one bin in a hundred above 30 of 100 peak photons)."""
    b = torch.arange(bins, device=DEV, dtype=torch.float32)
    at = r.u(traces, 1, lo=0.1 * bins, hi=0.8 * bins).float()
    h = torch.exp(r.u(traces, 1, lo=math.log(0.01), hi=0.0)).float()
    t = (b - at) / (0.02 * bins)
    tau = h * torch.exp(-0.5 * t * t) + 0.02 * h * (t > 0) * torch.exp(-t.clamp(min=0) / 4)
    return 1e-3 * tau * (0.9 + 0.2 * torch.rand(tau.shape, generator=r.g, device=DEV))


def _requests(c):
    """Sizes and modes of a burst's requests: the same for every seed."""
    rng = random.Random(c["trace"])
    out = []
    for _ in range(c["requests"]):
        side = _log(rng, c["side_lo"], c["side_hi"])
        out.append(dict(scan_nx=side, scan_ny=side, wall_half=1.0,
                        scan_mode=rng.choice(["confocal", "nonconfocal"]), cos_mode="object",
                        num_bins=_log(rng, c["bins_lo"], c["bins_hi"]), bin_ps=rng.uniform(4.0, 16.0),
                        fwhm_ps=rng.uniform(30.0, 70.0), standoff=1.0,
                        scene=rng.choice(["union", "heightfield"]),
                        points=_log(rng, c["points_lo"], c["points_hi"])))
    return out


def _depth_map(c, seed):
    r = _Rand(seed)
    n, m = c["n"], c["m"]
    x, y = _grid(n, 1.0)
    p = r.u(2, lo=-0.5, hi=0.5)
    z = 0.2 + 0.15 * torch.exp(-((x - p[0]) ** 2 + (y - p[1]) ** 2) / 0.1) + 0.05 * x
    depth = torch.round(z * m).to(torch.int32).clamp_(0, m - 1)
    depth[r.u(n, n) < 0.05] = -1  # pixels without a surface
    albedo = (0.2 + 0.8 * r.beta22(n * n)).reshape(n, n).float() if c["albedo"] else None
    return depth.contiguous(), albedo


class _DeviceView:
    """Server-owned device memory as a tensor (CUDA array interface)."""

    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False),
                                         "version": 3}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "simulate":
        pts, occ = _scene(case["scene"], _Rand(seed), case["points"], case["wall_half"])
        scene = nlos.scene_create(_params(case), pts)
        if case["occluders"]:
            nlos.scene_set_occluders(scene, occ)
        tau = torch.empty(scene.num_scan, scene.num_bins, device=DEV)
        return dict(case=case, scene=scene, points=pts, tau=tau)
    if kind == "detect":
        traces = case["scan_nx"] * case["scan_ny"]
        r = _Rand(seed)
        tau = _cube(r, traces, case["num_bins"])
        if case["noise_mode"] == "paper_nr":
            # that mode's scale is the cube's variance: intensities whose variance times
            # intensity gives the photon level
            var = tau.double().var(unbiased=False)
            k = (case["photons"] * 10 ** 0.2 / (var * tau.max().double())) ** (1.0 / 3.0)
            tau = (tau * k).float()
        prm = nlos.params(scan_nx=case["scan_nx"], scan_ny=case["scan_ny"], num_bins=case["num_bins"],
                          noise_mode=case["noise_mode"], peak_photons=case["photons"],
                          dark_per_bin=1e-3, nr_db=2.0, seed=seed)
        scene = nlos.scene_create(prm, torch.empty(0, 8, device=DEV))
        return dict(case=case, scene=scene, tau=tau.contiguous(),
                    counts=torch.empty(tau.shape, device=DEV, dtype=torch.int32),
                    energy=torch.empty(traces, device=DEV, dtype=torch.float64))
    if kind == "jitter":
        tau = _cube(_Rand(seed), case["traces"], case["num_bins"]).contiguous()
        return dict(case=case, tau=tau, out=torch.empty_like(tau))
    if kind == "train":
        pts, albedo, depth, g = _train_inputs(case, seed)
        scene = nlos.scene_create(_train_params(case), pts)
        return dict(case=case, scene=scene, albedo=albedo.requires_grad_(True),
                    depth=depth.requires_grad_(True), g=g)
    if kind == "lct":
        depth, albedo = _depth_map(case, seed)
        plan = nlos.Lct(case["n"], case["m"], case["wall_half"], case["bin_ps"] * 1e-12)
        return dict(case=case, plan=plan, depth=depth, albedo=albedo,
                    tau=torch.empty(case["n"], case["n"], case["m"], device=DEV))
    r = _Rand(seed)
    reqs = [(nlos.params(_params(q)), _scene(q["scene"], r, q["points"], 1.0)[0].cpu().numpy(), q)
            for q in _requests(case)]
    return dict(case=case, server=nlos.server_create(16 << 30), requests=reqs)


def run(state):
    kind = state["case"]["kind"]
    if kind == "simulate":
        if state["case"]["refresh"]:
            nlos.scene_set_points(state["scene"], state["points"])
        nlos.simulate(state["scene"], state["tau"])
        return state["tau"]
    if kind == "detect":
        nlos.detect(state["scene"], state["tau"], state["counts"], state["energy"])
        return state["counts"], state["energy"]
    if kind == "jitter":
        tau = state["tau"]
        nlos.jitter(tau, state["out"], tau.shape[0], tau.shape[1], state["case"]["fwhm_bins"], 1.0,
                    padding=state["case"]["padding"])
        return state["out"]
    if kind == "train":
        a, d = state["albedo"], state["depth"]
        tau = NlosSplat.apply(a, d, state["scene"])
        ga, gd = torch.autograd.grad(tau, (a, d), grad_outputs=state["g"])
        return tau.detach(), ga, gd
    if kind == "lct":
        state["plan"].forward(state["depth"], state["albedo"], state["tau"])
        return state["tau"]
    srv = state["server"]
    tickets = [srv.submit(prm, pts) for prm, pts, _ in state["requests"]]
    ptrs = []
    for t in tickets:
        st, tau = nlos.EBUSY, None
        while st == nlos.EBUSY:
            st, tau, _, _ = srv.poll(t, 1000)
        ptrs.append(tau)
    out = [torch.as_tensor(_DeviceView(p, (q["scan_nx"] * q["scan_ny"], q["num_bins"])),
                           device=DEV).clone() for p, (_, _, q) in zip(ptrs, state["requests"])]
    torch.cuda.current_stream().synchronize()  # the server owns the results until they are released
    for t in tickets:
        srv.release(t)
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
def _landing(c, prm):
    """The share of (scan point, surface point) pairs that carry weight into the window."""
    pts, _ = _scene(c["scene"], _Rand(1), min(c["points"], 16384), c["wall_half"])
    sx, sy, off = _spots(prm)
    k = torch.arange(0, sx.numel(), max(1, sx.numel() // 64) | 1, device=DEV)
    u, w = _pairs(prm, pts.double(), sx[k], sy[k], off[k])
    return float(((u >= 0) & (u < c["num_bins"]) & (w != 0)).double().mean())


def work(case):
    kind = case["kind"]
    if kind == "simulate":
        n = case["scan_nx"] * case["scan_ny"]
        # about 24 operations for each pair that lands in the window
        return {"bytes": 32.0 * case["points"] + 4.0 * n * case["num_bins"],
                "flops": 24.0 * n * case["points"] * _landing(case, _params(case))}
    if kind == "detect":
        n = case["scan_nx"] * case["scan_ny"] * case["num_bins"]
        return {"bytes": 8.0 * n + 8.0 * case["scan_nx"] * case["scan_ny"], "flops": 30.0 * n}
    if kind == "jitter":
        n = case["traces"] * case["num_bins"]
        taps = 2 * math.ceil(2 * case["fwhm_bins"] / (2 * math.sqrt(2 * math.log(2)))) + 1
        return {"bytes": 8.0 * n, "flops": 2.0 * taps * n}
    if kind == "train":
        n = case["scan_nx"] * case["scan_ny"]
        # the pair's geometry twice and six terms of the splat each way
        return {"bytes": 32.0 * case["points"] + 8.0 * n * case["num_bins"] + 16.0 * case["points"],
                "flops": 100.0 * n * case["points"]}
    if kind == "lct":
        n, m = case["n"], case["m"]
        # the convolution over its nonzeros: one addition a (pixel, scan point) pair
        return {"bytes": 8.0 * n * n + 4.0 * n * n * m, "flops": 1.0 * n ** 4}
    t = {"bytes": 0.0, "flops": 0.0}
    for q in _requests(case):
        w = work(dict(q, kind="simulate"))
        t = {k: t[k] + w[k] for k in t}
    return t


# ---------------------------------------------------------------------------
# The definition in 64 bits.
# ---------------------------------------------------------------------------
def _spots(p):
    nx, ny, wx, wy, h = p["scan_nx"], p["scan_ny"], p["wall_half_x"], p["wall_half_y"], p["standoff_m"]
    x = -wx + (torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5) * (2 * wx / nx)
    y = -wy + (torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5) * (2 * wy / ny)
    sx, sy = x.repeat(ny), y.repeat_interleave(nx)
    if p["standoff_mode"] == "constant":
        legs = torch.full_like(sx, 2 * h)
    else:
        d = torch.sqrt(sx * sx + sy * sy + h * h)
        legs = d + (d if p["scan_mode"] == "confocal" else h)  # the laser spot is the wall centre
    return sx, sy, (legs - p["window_start_m"]) / (C * p["bin_width_s"])


def _leg(pts, sx, sy):
    """Length, object cosine and wall cosine of the leg from each spot to each point."""
    dx, dy = pts[None, :, 0] - sx[:, None], pts[None, :, 1] - sy[:, None]
    z = pts[None, :, 2]
    r = torch.sqrt(dx * dx + dy * dy + z * z)
    cos = -(dx * pts[None, :, 3] + dy * pts[None, :, 4] + z * pts[None, :, 5]) / r
    return r, cos, z / r


def _factor(cos_mode, r, cos, wall):
    f = 1.0 / (r * r)
    if cos_mode != "none":
        f = f * cos.clamp(min=0)
    return f * wall if cos_mode == "object_wall" else f


def _pairs(p, pts, sx, sy, off):
    """Bin coordinate and weight of every pair of some spots with all points."""
    r, cos, wall = _leg(pts, sx, sy)
    f = _factor(p["cos_mode"], r, cos, wall)
    q = (pts[:, 6] * pts[:, 7])[None]
    if p["scan_mode"] == "confocal":
        rl, fl = r, f
    else:
        zero = torch.zeros(1, device=DEV, dtype=torch.float64)
        rl, cl, wl = _leg(pts, zero, zero)
        fl = _factor(p["cos_mode"], rl, cl, wl)
    return (r + rl) / (C * p["bin_width_s"]) + off[:, None], q * f * fl


def _hidden(occ, pts, sx, sy):
    """Whether the segment from a spot to a point runs inside a solid for more than
    0.004 of its length."""
    hid = torch.zeros(sx.numel(), pts.shape[0], device=DEV, dtype=torch.bool)
    dx, dy = pts[None, :, 0] - sx[:, None], pts[None, :, 1] - sy[:, None]
    dz = pts[None, :, 2].expand_as(dx)
    for k, a0, a1, a2, b0, b1, b2, _ in occ.astype(np.float64).tolist():
        if k == 0:
            fx, fy = (sx - a0)[:, None], (sy - a1)[:, None]
            A = dx * dx + dy * dy + dz * dz
            Bq = fx * dx + fy * dy - a2 * dz
            disc = Bq * Bq - A * (fx * fx + fy * fy + a2 * a2 - b0 * b0)
            sq = torch.sqrt(disc.clamp(min=0))
            chord = ((-Bq + sq) / A).clamp(max=1) - ((-Bq - sq) / A).clamp(min=0)
            chord = torch.where(disc > 0, chord, torch.zeros_like(chord))
        else:
            t0, t1 = torch.zeros_like(dx), torch.ones_like(dx)
            for o, d, lo, hi in ((sx[:, None], dx, a0, b0), (sy[:, None], dy, a1, b1), (0.0, dz, a2, b2)):
                ta, tb = (lo - o) / d, (hi - o) / d
                t0, t1 = torch.maximum(t0, torch.minimum(ta, tb)), torch.minimum(t1, torch.maximum(ta, tb))
            chord = t1 - t0
        hid |= chord > 4e-3
    return hid


def _blur(tau, sigma, padding):
    radius = math.ceil(2 * sigma) if sigma > 0 else 0
    if radius == 0:
        return tau
    j = torch.arange(-radius, radius + 1, device=DEV, dtype=torch.float64)
    taps = torch.exp(-j * j / (2 * sigma * sigma))
    taps = (taps / taps.sum()).tolist()
    B = tau.shape[1]
    out = torch.zeros_like(tau)
    for k, t in zip(range(-radius, radius + 1), taps):
        b = torch.arange(B, device=DEV) - k
        v = tau[:, b.clamp(0, B - 1)]
        out += t * (v if padding == "replicate" else v * ((b >= 0) & (b < B)))
    return out


def _sigma(p):
    return p["jitter_fwhm_s"] / (2 * math.sqrt(2 * math.log(2))) / p["bin_width_s"]


def _exact_transient(p, pts, occ=None):
    pts = pts.double()
    sx, sy, off = _spots(p)
    n, B = sx.numel(), p["num_bins"]
    tau = torch.zeros(n * B, device=DEV, dtype=torch.float64)
    lit = None
    if occ is not None and p["scan_mode"] != "confocal":
        zero = torch.zeros(1, device=DEV, dtype=torch.float64)
        lit = ~_hidden(occ, pts, zero, zero)
    step = max(1, (1 << 25) // max(1, pts.shape[0]))
    for s in range(0, n, step):
        e = min(n, s + step)
        u, w = _pairs(p, pts, sx[s:e], sy[s:e], off[s:e])
        ok = (u >= 0) & (u < B) & (w != 0)
        if occ is not None:
            ok &= ~_hidden(occ, pts, sx[s:e], sy[s:e])
            if lit is not None:
                ok &= lit
        row = torch.arange(s, e, device=DEV)[:, None].expand_as(u)[ok]
        tau.index_add_(0, row * B + u[ok].floor().long(), w[ok])
    return _blur(tau.view(n, B), _sigma(p), p["jitter_padding"])


def _exact_train(c, seed):
    base, albedo, depth, g = _train_inputs(c, seed)
    p = _train_params(c)
    pts = base.double()
    pts[:, :3] += depth.double()[:, None] * pts[:, 3:6]
    pts[:, 6] = albedo.double()
    sx, sy, off = _spots(p)
    n, B, P, sg = sx.numel(), p["num_bins"], pts.shape[0], _sigma(p)
    nz, q, area = pts[None, :, 5], (pts[:, 6] * pts[:, 7])[None], pts[None, :, 7]
    zero = torch.zeros(1, device=DEV, dtype=torch.float64)
    tau = torch.zeros(n * B, device=DEV, dtype=torch.float64)
    gf = g.double().reshape(-1)
    ga, gd = (torch.zeros(P, device=DEV, dtype=torch.float64) for _ in range(2))

    def leg(lx, ly):  # factor, its derivative along the normal, length, cosine
        r, cos, wall = _leg(pts, lx, ly)
        f = _factor(c["cos_mode"], r, cos, wall)
        fc = torch.ones_like(cos) if c["cos_mode"] == "none" else cos.clamp(min=0)
        dfc = torch.zeros_like(cos) if c["cos_mode"] == "none" else -(1 - cos * cos) / r * (cos > 0)
        fw, dfw = ((wall, (nz + wall * cos) / r) if c["cos_mode"] == "object_wall" else
                   (torch.ones_like(cos), torch.zeros_like(cos)))
        return f, (dfc * fw + fc * dfw) / r ** 2 + fc * fw * 2 * cos / r ** 3, r, cos

    step = max(1, (1 << 24) // P)
    reach = 6.0 * sg
    for s in range(0, n, step):
        e = min(n, s + step)
        fd, dfd, rd, cd = leg(sx[s:e], sy[s:e])
        fl, dfl, rl, cl = (fd, dfd, rd, cd) if c["scan_mode"] == "confocal" else leg(zero, zero)
        u = (rd + rl) / (C * p["bin_width_s"]) + off[s:e, None]
        w, dw, du = q * fd * fl, q * (dfd * fl + fd * dfl), -(cd + cl) / (C * p["bin_width_s"])
        j = u.floor()
        row = torch.arange(s, e, device=DEV, dtype=torch.float64)[:, None] * B
        g0, g1 = torch.zeros_like(u), torch.zeros_like(u)
        for k in range(-math.ceil(reach) - 1, math.ceil(reach) + 2):
            b = j + k
            x = b + 0.5 - u
            phi = torch.exp(-x * x / (2 * sg * sg)) / (sg * math.sqrt(2 * math.pi))
            phi = phi * ((x.abs() < reach) & (b >= 0) & (b < B))
            at = (row + b.clamp(0, B - 1)).long().reshape(-1)
            tau.index_add_(0, at, (w * phi).reshape(-1))
            v = gf[at].view_as(u) * phi
            g0 += v
            g1 += v * x
        ga += (area * fd * fl * g0).sum(0)
        gd += (dw * g0 + w * du * g1 / (sg * sg)).sum(0)
    return tau.view(n, B), ga, gd


def _exact_lct(c, seed):
    """The depth-map model's convolution, summed over the map's voxels and the
    point-spread function's one node a column."""
    depth, albedo = _depth_map(c, seed)
    n, m = c["n"], c["m"]
    d = depth.reshape(-1).long()
    ok = (d >= 0) & (d < m)
    j = (d + 1).double()
    val = (albedo.reshape(-1).double() if c["albedo"] else torch.full_like(j, 0.5)) / (j * m * m)
    row = ((d + 1) ** 2 + m - 1) // m - 1
    px = torch.arange(n * n, device=DEV) // n
    py = torch.arange(n * n, device=DEV) % n
    slope = c["wall_half"] / (m * C * (c["bin_ps"] * 1e-12))
    node = -1.0 + 2.0 * torch.arange(2 * n, device=DEV, dtype=torch.float64) / (2 * n - 1)
    dz = 2.0 / (2 * m - 1)
    target = 16.0 * slope * slope * (node[:, None] ** 2 + node[None, :] ** 2)
    k = torch.round((target + 1.0) / dz)
    has = (k >= 0) & (k < 2 * m) & ((target - (-1.0 + k * dz)).abs() <= 0.5 * dz + 1e-12)
    k = torch.where(has, k - m, torch.full_like(k, 10.0 * m)).long()
    vol = torch.zeros(n * n * m, device=DEV, dtype=torch.float64)
    px, py, row, val = px[ok], py[ok], row[ok], val[ok]
    out = torch.arange(n * n, device=DEV)
    for s in range(0, n * n, max(1, (1 << 24) // (n * n))):
        o = out[s:s + max(1, (1 << 24) // (n * n))]
        t = row[None] + k[(o // n)[:, None] - px[None] + n, (o % n)[:, None] - py[None] + n]
        sel = (t >= 0) & (t < m)
        vol.index_add_(0, (o[:, None] * m + t)[sel], val[None].expand_as(t)[sel])
    jt = torch.arange(1, m + 1, device=DEV)
    return vol.view(n, n, m)[:, :, (jt * jt + m - 1) // m - 1] * (m / jt.double() ** 4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "simulate":
        pts, occ = _scene(case["scene"], _Rand(seed), case["points"], case["wall_half"])
        return _exact_transient(_params(case), pts, occ if case["occluders"] else None)
    if kind == "detect":  # the counts are whole numbers
        tau = prepare(case, seed)["tau"]
        return None, tau.double().sum(dim=1)
    if kind == "jitter":
        tau = _cube(_Rand(seed), case["traces"], case["num_bins"])
        sigma = case["fwhm_bins"] / (2 * math.sqrt(2 * math.log(2)))
        return _blur(tau.double(), sigma, case["padding"])
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "lct":
        return _exact_lct(case, seed)
    r = _Rand(seed)
    return [_exact_transient(_params(q), _scene(q["scene"], r, q["points"], 1.0)[0])
            for q in _requests(case)]
