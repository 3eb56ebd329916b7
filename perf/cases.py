"""The work that a user of this package has it do, as cases that can be timed and compared.

Every case goes through the public entry points of `paper_2301_08068_gb300.rmp`: one state per
control step (synchronous and asynchronous), LiDAR scans, batches of states, combined policies,
closed-loop rollouts, the ESDF policy, the request server and the refresh of a map.  Scenes,
states and scans are made here from the seed alone (torch on the GPU, numpy for the small
draws), with the sizes of this repository's own workloads; `exact` evaluates the same
definitions in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2301_08068_gb300 import rmp as R

TRUNC = 0.3          # TSDF truncation, m
CLEAR = 0.3          # clearance of a free point, m
STATIC = dict(eta_rep=88.0, nu_rep=1.4, eta_damp=140.0, nu_damp=1.2, r=2.4, c=0.2, eps=1e-3,
              min_range=0.0)
LIDAR = dict(eta_rep=1.2, nu_rep=1.5, eta_damp=3.0, nu_damp=1.0, r=1.3, c=1.0, eps=1e-3,
             min_range=0.2)
ALPHA, BETA = 10.0, 15.0   # attractor gains of the static-map tuning

# The maps: the two dense grids, the 40 m and 100 m hashed TSDF maps, the 10 m planning cube
# (200 small obstacles), and two survey sites 1.5 km apart in one frame (few blocks in a huge
# extent).  kind, extent (m), voxel size (m), primitives, size range (m), max range (m)
MAPS = {
    "dense64": ("dense", (6.4, 6.4, 6.4), 0.1, 20, (0.1, 0.75), 5.0),
    "dense128": ("dense", (6.4, 6.4, 6.4), 0.05, 40, (0.1, 0.75), 10.0),
    "hashed40": ("hashed", (40.0, 40.0, 10.0), 0.1, 200, (0.2, 2.0), 10.0),
    "hashed100": ("hashed", (100.0, 100.0, 20.0), 0.2, 2500, (0.2, 2.0), 10.0),
    "cube10": ("hashed", (10.0, 10.0, 10.0), 0.1, 200, (0.2, 0.6), 10.0),
    "sites": ("sites", (24.0, 24.0, 8.0), 0.1, 60, (0.2, 2.0), 10.0),
}
SITE_STEP = (15200, 14400, 512)   # voxels from the first site to the second


def listed():
    return [
        # one control step on a small onboard grid: latency only
        dict(name="eval_dense64_1k", kind="eval", map="dense64", rays=1024, sync=True,
             records=False, fp64=False, cubic=False),
        # the benchmark's control step: 65536 rays through the hashed 40 m map
        dict(name="eval_hashed40_64k", kind="eval", map="hashed40", rays=65536, sync=True,
             records=False, fp64=False, cubic=False),
        # the largest single request, on the 100 m map, device-resident state and result
        dict(name="eval_hashed100_262k", kind="eval", map="hashed100", rays=262144, sync=False,
             records=False, fp64=False, cubic=False),
        # a ragged ray count with hit records and per-ray policies (visualisation, logging),
        # FP64 reduction and the spline weight
        dict(name="eval_hashed40_records_20k", kind="eval", map="hashed40", rays=20011,
             sync=False, records=True, fp64=True, cubic=True),
        # one 64 x 1024 LiDAR scan per control step
        dict(name="scan_64x1024", kind="scan", beams=64, columns=1024, points=65536, sync=True,
             records=False, fp64=False),
        # a full OS-0 scan with the per-point policies, device-resident
        dict(name="scan_128x2048_records", kind="scan", beams=128, columns=2048, points=262144,
             sync=False, records=True, fp64=False),
        # many candidate states of a planner, uneven ray counts
        dict(name="batch_256_uneven", kind="batch", map="hashed40", states=256, ray_lo=4096,
             ray_hi=65536, host=False, fp64=False),
        # one control step of a fleet: raycast policy and goal attractor
        dict(name="combined_128x256", kind="combined", states=128, rays=256, mean=True),
        # the closed loop of the planning experiment (whole call, host in and out)
        dict(name="rollout_128x1024", kind="rollout", states=128, rays=1024, steps=48, esdf=False),
        # the single-query comparison policy for a large set of states
        dict(name="esdf_16k_states", kind="esdf", states=16384, prims=200, goals=True),
        # a burst of requests of many sizes over three resident maps, through the server
        dict(name="served_burst_96", kind="served", requests=96, ray_lo=1024, ray_hi=262144),
        # a new map from the mapper (blocks on the device), then the control step on it
        dict(name="map_refresh_hashed40", kind="refresh", map="hashed40", rays=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "scan", "batch", "batch", "combined", "rollout",
                       "esdf", "served", "refresh"])
    any_map = ["dense64", "dense128", "hashed40", "hashed100", "cube10", "sites"]
    if kind == "eval":
        return dict(kind=kind, map=rng.choice(any_map), rays=_log_int(rng, 64, 262144),
                    sync=rng.random() < 0.5, records=rng.random() < 0.25,
                    fp64=rng.random() < 0.25, cubic=rng.random() < 0.25)
    if kind == "scan":
        beams, columns = rng.choice([16, 32, 64, 128]), rng.choice([512, 1024, 2048])
        return dict(kind=kind, beams=beams, columns=columns,
                    points=rng.randrange(beams * columns // 2, beams * columns + 1),
                    sync=rng.random() < 0.5, records=rng.random() < 0.5, fp64=rng.random() < 0.25)
    if kind == "batch":
        n = _log_int(rng, 2, 256)
        lo = _log_int(rng, 64, 8192)
        return dict(kind=kind, map=rng.choice(any_map), states=n, ray_lo=lo,
                    ray_hi=lo * rng.choice([1, 2, 5, 8]), host=rng.random() < 0.5,
                    fp64=rng.random() < 0.25)
    if kind == "combined":
        return dict(kind=kind, states=_log_int(rng, 8, 512), rays=_log_int(rng, 16, 2048),
                    mean=rng.random() < 0.7)
    if kind == "rollout":
        return dict(kind=kind, states=_log_int(rng, 8, 128), rays=_log_int(rng, 16, 1024),
                    steps=rng.randrange(8, 49), esdf=rng.random() < 0.3)
    if kind == "esdf":
        return dict(kind=kind, states=_log_int(rng, 16, 65536), prims=_log_int(rng, 5, 1000),
                    goals=rng.random() < 0.7)
    if kind == "served":
        lo = _log_int(rng, 64, 4096)
        return dict(kind=kind, requests=rng.randrange(8, 97), ray_lo=lo,
                    ray_hi=lo * rng.choice([4, 16, 64]))
    return dict(kind=kind, map=rng.choice(any_map[:5]), rays=_log_int(rng, 256, 65536))


# ------------------------------------------------------------------------------ inputs
def _cuda(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).cuda()


class Scene:
    """Boxes and spheres in [0, extent): kinds (True = sphere), centres, half-extents."""

    def __init__(self, extent, n, size, rng, boxes_only=False):
        self.extent = np.asarray(extent, np.float64)
        self.center = rng.uniform(0.0, 1.0, (n, 3)) * self.extent
        self.size = rng.uniform(size[0], size[1], (n, 3))
        self.sphere = np.zeros(n, bool) if boxes_only else rng.uniform(size=n) < 0.5
        self.size[self.sphere] = self.size[self.sphere, :1]      # radius in every component
        self.c, self.h = _cuda(self.center), _cuda(self.size)
        self.s = _cuda(self.sphere)

    def sdf(self, p, i=None):
        """Signed distances of points p (..., m, 3) to primitives i (broadcast), FP64."""
        c, h, s = (self.c, self.h, self.s) if i is None else (self.c[i], self.h[i], self.s[i])
        q = p - c
        ball = q.square().sum(-1).sqrt() - h[..., 0]
        a = q.abs() - h
        box = a.clamp_min(0.0).square().sum(-1).sqrt() + a.amax(-1).clamp_max(0.0)
        return torch.where(s, ball, box)

    def volume(self, dims, vs, fill):
        """min(fill, union's SDF) at the voxel centres, (nz, ny, nx) FP32 on the GPU."""
        nx, ny, nz = dims
        vol = torch.full((nz * ny * nx,), fill, dtype=torch.float32, device="cuda")
        reach = int(math.ceil((2.0 * self.size.max() + 2.0 * max(fill, 0.0)) / vs)) + 2
        k = torch.arange(reach, device="cuda")
        lo = ((self.c - self.h - fill) / vs).floor().long() if fill > 0 else \
            ((self.c - self.h) / vs).floor().long()
        per = max(1, (1 << 24) // reach ** 3)
        for i0 in range(0, len(self.center), per):
            i = torch.arange(i0, min(i0 + per, len(self.center)), device="cuda")
            z, y, x = (lo[i, a].view(-1, 1) + k for a in (2, 1, 0))
            z, y, x = z[:, :, None, None], y[:, None, :, None], x[:, None, None, :]
            ok = (z >= 0) & (z < nz) & (y >= 0) & (y < ny) & (x >= 0) & (x < nx)
            shape = ok.shape
            p = torch.stack([x.expand(shape), y.expand(shape), z.expand(shape)], -1)
            p = (p.double() + 0.5) * vs
            d = self.sdf(p, i.view(-1, 1, 1, 1)).float()
            at = (x + nx * (y + ny * z)).expand(shape)[ok]
            vol.scatter_reduce_(0, at, d[ok], "amin")
        return vol.view(nz, ny, nx)

    def free_points(self, n, rng, lo=0.0, hi=1.0):
        out = np.zeros((0, 3))
        while len(out) < n:
            p = rng.uniform(lo, hi, (max(64, 3 * n), 3)) * self.extent
            t = _cuda(p)
            d = torch.cat([self.sdf(q[:, None, :]).amin(1) for q in t.split(4096)])
            out = np.concatenate([out, p[(d > CLEAR).cpu().numpy()]])
        return out[:n]


def _blocks(vol):
    """(keys, tsdf) of the 8^3 blocks that reach into the truncation band, on the GPU."""
    nz, ny, nx = vol.shape
    b = vol.view(nz // 8, 8, ny // 8, 8, nx // 8, 8).permute(0, 2, 4, 1, 3, 5)
    some = (b < TRUNC).flatten(3).any(-1)
    at = some.nonzero()
    tsdf = b[some].reshape(-1, 512).clamp(-TRUNC, TRUNC).contiguous()
    return at.flip(1).int().contiguous(), tsdf


class World:
    """A scene, its map description on the GPU and its occupancy (for free voxels and exact)."""

    def __init__(self, name, rng):
        self.name = name
        self.kind, extent, self.vs, n, size, self.max_range = MAPS[name]
        self.scenes = [Scene(extent, n, size, rng, self.kind == "dense")
                       for _ in range(2 if self.kind == "sites" else 1)]
        dims = [-(-int(round(e / self.vs)) // 8) * 8 for e in extent]
        self.offsets = [(0, 0, 0), SITE_STEP][:len(self.scenes)]
        if self.kind == "dense":
            vol = self.scenes[0].volume(dims, self.vs, 0.0)
            self.occ = [vol < 0.0]
            self.dense = self.occ[0].to(torch.uint8).contiguous()
        else:
            keys, tsdf, self.occ = [], [], []
            for sc, off in zip(self.scenes, self.offsets):
                vol = sc.volume(dims, self.vs, TRUNC)
                self.occ.append(vol <= 0.0)
                kk, tt = _blocks(vol)
                keys.append(kk + torch.tensor(off, dtype=torch.int32, device="cuda") // 8)
                tsdf.append(tt)
            self.keys, self.tsdf = torch.cat(keys).contiguous(), torch.cat(tsdf).contiguous()

    def desc(self):
        if self.kind == "dense":
            return R.dense_desc(self.dense, self.vs, (0.0, 0.0, 0.0))
        return R.hashed_desc(self.keys, self.tsdf, self.vs)

    def states(self, n, rng):
        """n rows of [x, xdot] at free points and their sites."""
        site = rng.integers(0, len(self.scenes), n)
        x = np.zeros((n, 3))
        for s, sc in enumerate(self.scenes):
            m = int((site == s).sum())
            if m:
                x[site == s] = sc.free_points(m, rng) + np.asarray(self.offsets[s]) * self.vs
        return np.concatenate([x, rng.normal(size=(n, 3))], 1), site


_context = []


def _ctx():
    if not _context:
        _context.append(R.Context(0))
    return _context[0]


class Held:
    """What a user's program keeps: inputs, uploaded maps, workspaces, output buffers."""

    def __init__(self, case):
        self.case, self.maps, self.esdfs, self.servers = case, [], [], []

    def upload(self, world):
        m = R.rmp_map_upload(_ctx().handle, world.desc())
        self.maps.append(m)
        return m

    def __del__(self):
        try:
            for s in self.servers:
                s.close()
            for m in self.maps:
                R.rmp_map_release(_ctx().handle, m)
            for e in self.esdfs:
                R.rmp_esdf_release(_ctx().handle, e)
        except Exception:
            pass


def _params(base, max_range, fp64=False, cubic=False):
    return R.make_params(dict(base, reduce_mode=int(fp64), w_mode=int(cubic)), max_range)


def _result_buffer(n):
    """n device results and their fields as views: f, sum A, sum A f, eig, counts."""
    buf = torch.zeros(n * R.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    v = buf.view(torch.float64).view(n, 18)
    c = buf.view(torch.int32).view(n, 36)
    return buf, dict(f=v[:, 0:3], sumA=v[:, 3:9], sumAf=v[:, 9:12], eig=v[:, 12:15],
                     counts=c[:, 30:35])


def _lidar_points(case, rng):
    """Scan of the 40 m scene from a free point: analytic first hits plus N(0, 0.02 m), NaN
    without a return within 30 m; beam-major, the first `points` of the scan."""
    _, extent, _, n, size, _ = MAPS["hashed40"]
    sc = Scene(extent, n, size, rng)
    o = _cuda(sc.free_points(1, rng)[0])
    fov = 90.0 if case["beams"] >= 128 else 45.0
    el = np.deg2rad(np.linspace(-fov / 2, fov / 2, case["beams"]))
    az = 2 * np.pi * np.arange(case["columns"]) / case["columns"]
    e, a = np.meshgrid(el, az, indexing="ij")
    u = np.stack([np.cos(e) * np.cos(a), np.cos(e) * np.sin(a), np.sin(e)], -1).reshape(-1, 3)
    u = _cuda(u[:case["points"]])
    t = torch.full((len(u),), math.inf, dtype=torch.float64, device="cuda")
    for i in range(n):
        c, h = sc.c[i], sc.h[i]
        if sc.sphere[i]:
            b = ((o - c) * u).sum(1)
            disc = b * b - ((o - c).square().sum() - h[0] ** 2)
            ti = -b - disc.clamp_min(0.0).sqrt()
            hit = (disc >= 0) & (ti >= 0)
        else:
            t1, t2 = (c - h - o) / u, (c + h - o) / u
            ti = torch.minimum(t1, t2).nan_to_num(-math.inf, math.inf, -math.inf).amax(1)
            tf = torch.maximum(t1, t2).nan_to_num(math.inf, math.inf, -math.inf).amin(1)
            hit = (ti <= tf) & (ti >= 0)
        t = torch.where(hit & (ti < t), ti, t)
    noise = _cuda(rng.normal(0.0, 0.02, len(u)))
    t = torch.where(t <= 30.0, t + noise, torch.full_like(t, math.nan))
    return (u * t[:, None]).float().contiguous(), rng.normal(size=3)


def _uneven(rng, n, lo, hi):
    return np.rint(np.exp(rng.uniform(math.log(lo), math.log(hi + 0.49), n))).astype(np.int64)


def _inputs(case, seed):
    """Everything made from the seed: used by prepare and by exact alike."""
    rng = np.random.default_rng(int(seed))
    kind = case["kind"]
    if kind == "scan":
        pts, v = _lidar_points(case, rng)
        return dict(points=pts, state=np.concatenate([np.zeros(3), v]))
    if kind in ("eval", "refresh", "batch"):
        w = World(case["map"], rng)
        n = case.get("states", 1)
        st, site = w.states(n, rng)
        rays = _uneven(rng, n, case["ray_lo"], case["ray_hi"]) if kind == "batch" else \
            np.array([case["rays"]])
        return dict(worlds=[w], world_of=np.zeros(n, int), states=st, sites=site, rays=rays)
    if kind == "served":
        ws = [World(m, rng) for m in ("dense128", "hashed40", "hashed100")]
        n = case["requests"]
        of = rng.integers(0, 3, n)
        st, site = np.zeros((n, 6)), np.zeros(n, int)
        for i, w in enumerate(ws):
            m = int((of == i).sum())
            if m:
                st[of == i], site[of == i] = w.states(m, rng)
        return dict(worlds=ws, world_of=of, states=st, sites=site,
                    rays=_uneven(rng, n, case["ray_lo"], case["ray_hi"]))
    if kind == "esdf":
        # at the density of the 10 m planning cube
        edge = 10.0 * (case["prims"] / 200.0) ** (1.0 / 3.0)
        sc = Scene((edge,) * 3, case["prims"], (0.2, 0.6), rng)
        n = case["states"]
        x = rng.uniform(0.0, edge, (n, 3))
        return dict(scene=sc, states=np.concatenate([x, rng.normal(size=(n, 3))], 1),
                    goals=rng.uniform(0.0, edge, (n, 3)))
    w = World("cube10", rng)                      # combined, rollout
    n, sc = case["states"], w.scenes[0]
    if kind == "combined":
        x, v = sc.free_points(n, rng), rng.normal(size=(n, 3))
    else:
        x, v = sc.free_points(n, rng, (0.05,) * 3, (0.15, 0.95, 0.95)), np.zeros((n, 3))
    goals = sc.free_points(n, rng, (0.85, 0.05, 0.05), (0.95,) * 3)
    return dict(worlds=[w], world_of=np.zeros(n, int), states=np.concatenate([x, v], 1),
                sites=np.zeros(n, int), rays=np.full(n, case["rays"]), goals=goals)


def _primitives(sc):
    class P:
        pass
    out = []
    for i in range(len(sc.center)):
        p = P()
        p.kind, p.center, p.size = ("sphere" if sc.sphere[i] else "box"), sc.center[i], sc.size[i]
        out.append(p)
    return out


def prepare(case, seed):
    s = Held(case)
    i = _inputs(case, seed)
    kind, ctx = case["kind"], _ctx().handle
    s.ctx = ctx
    if kind == "scan":
        s.points, s.x, s.v = i["points"], i["state"][:3].copy(), i["state"][3:].copy()
        s.params = _params(LIDAR, 30.0, case["fp64"])
        s.state = _cuda(i["state"])
        s.per_ray = torch.zeros((case["points"], 9), device="cuda") if case["records"] else None
    elif kind == "eval":
        w = i["worlds"][0]
        s.map = s.upload(w)
        s.x, s.v = i["states"][0, :3].copy(), i["states"][0, 3:].copy()
        s.state = _cuda(i["states"][0])
        s.params = _params(STATIC, w.max_range, case["fp64"], case["cubic"])
        n = case["rays"]
        s.hits = s.per_ray = None
        if case["records"]:
            s.hits = torch.zeros(n * 24, dtype=torch.uint8, device="cuda")
            s.per_ray = torch.zeros((n, 9), device="cuda")
            w6 = s.hits.view(torch.int32).view(n, 6)
            s.rec = dict(voxel=w6[:, 0:4], d=s.hits.view(torch.float32).view(n, 6)[:, 4],
                         outcome=w6[:, 5], per_ray=s.per_ray)
    elif kind == "batch":
        w = i["worlds"][0]
        s.map = s.upload(w)
        s.params = _params(STATIC, w.max_range, case["fp64"])
        s.n, s.max_rays = case["states"], int(i["rays"].max())
        s.host_states, s.host_rays = i["states"], i["rays"].astype(np.uint32)
        s.states, s.rays = _cuda(i["states"]), _cuda(i["rays"].astype(np.int32))
    elif kind == "served":
        s.map = [s.upload(w) for w in i["worlds"]]
        s.params = [_params(STATIC, w.max_range) for w in i["worlds"]]
        s.server = R.Server(_ctx(), max_rays=int(max(i["rays"].max(), 1)))
        s.servers.append(s.server)
        s.requests = [(s.map[k], i["states"][b, :3].copy(), i["states"][b, 3:].copy(),
                       int(i["rays"][b]), s.params[k]) for b, k in enumerate(i["world_of"])]
    elif kind == "esdf":
        s.esdf = R.rmp_esdf_upload(ctx, _primitives(i["scene"]))
        s.esdfs.append(s.esdf)
        s.params = _params(STATIC, 10.0)
        s.n, s.states = case["states"], _cuda(i["states"])
        s.goals = _cuda(i["goals"]) if case["goals"] else None
        s.query = torch.zeros((s.n, 4), dtype=torch.float64, device="cuda")
    elif kind == "refresh":
        s.desc_of = i["worlds"][0]
        s.x, s.v = i["states"][0, :3].copy(), i["states"][0, 3:].copy()
        s.params = _params(STATIC, s.desc_of.max_range)
    else:
        w = i["worlds"][0]
        s.map, s.n = s.upload(w), case["states"]
        s.params = _params(STATIC, w.max_range)
        if kind == "combined":
            s.states, s.goals = _cuda(i["states"]), _cuda(i["goals"])
            s.rays = _cuda(i["rays"].astype(np.int32))
        else:
            s.robots = np.concatenate([i["states"], i["goals"]], 1)
            s.rollout = R.rollout_params(ALPHA, BETA, 0.01, 0.2, case["steps"], 10, case["rays"],
                                         metric_mean=True)
            if case["esdf"]:
                s.esdf = R.rmp_esdf_upload(ctx, _primitives(w.scenes[0]))
                s.esdfs.append(s.esdf)
    if kind in ("eval", "scan") and not case["sync"]:
        s.ws = torch.zeros(R.rmp_workspace_bytes(), dtype=torch.uint8, device="cuda")
        R.rmp_workspace_init(s.ws)
        s.out, s.fields = _result_buffer(1)
    if kind in ("batch", "combined"):
        most = s.max_rays if kind == "batch" else case["rays"]
        s.ws = torch.empty(R.rmp_batch_workspace_bytes(s.n, most), dtype=torch.uint8,
                           device="cuda")
    if kind in ("batch", "combined", "esdf"):
        s.out, s.fields = _result_buffer(s.n)
    return s


def run(s):
    case, kind, ctx = s.case, s.case["kind"], s.ctx
    if kind == "eval":
        if case["sync"]:
            out = R.rmp_raycast_eval(ctx, s.map, s.x, s.v, case["rays"], s.params, hits=s.hits,
                                     per_ray=s.per_ray)
        else:
            R.rmp_raycast_eval_async(ctx, s.map, s.state, case["rays"], s.params, s.ws, s.out,
                                     hits=s.hits, per_ray=s.per_ray)
            out = s.fields
        return [out, s.rec] if case["records"] else out
    if kind == "scan":
        if case["sync"]:
            out = R.rmp_scan_eval(ctx, s.points, s.x, s.v, s.params, per_ray=s.per_ray)
        else:
            R.rmp_scan_eval_async(ctx, s.points, s.state, s.params, s.ws, s.out,
                                  per_ray=s.per_ray)
            out = s.fields
        return [out, s.per_ray] if case["records"] else out
    if kind == "batch":
        if case["host"]:
            got = R.rmp_raycast_eval_batch(ctx, s.map, s.host_states, s.host_rays, s.params)
            return _stacked(got)
        R.rmp_raycast_eval_batch_async(ctx, s.map, s.states, s.rays, s.n, s.max_rays, s.params,
                                       s.ws, s.out)
        return s.fields
    if kind == "combined":
        R.rmp_combined_eval_batch_async(ctx, s.map, s.states, s.rays, s.n, case["rays"], s.params,
                                        s.goals, ALPHA, BETA, s.ws, s.out,
                                        metric_mean=case["mean"])
        return s.fields
    if kind == "esdf":
        R.rmp_esdf_eval_async(ctx, s.esdf, s.states, s.goals, s.n, s.params, ALPHA, BETA, s.out,
                              query=s.query)
        return [s.fields, s.query]
    if kind == "served":
        tickets = [s.server.submit(*q) for q in s.requests]
        return _stacked([s.server.wait(t)[0] for t in tickets])
    if kind == "refresh":
        m = R.rmp_map_upload(ctx, s.desc_of.desc())
        out = R.rmp_raycast_eval(ctx, m, s.x, s.v, case["rays"], s.params)
        R.rmp_map_release(ctx, m)
        return out
    if case["esdf"]:
        got = R.rmp_rollout_esdf(ctx, s.map, s.esdf, s.robots, s.params, s.rollout)
    else:
        got = R.rmp_rollout(ctx, s.map, s.robots, s.params, s.rollout)
    return dict(x=np.stack([g["x"] for g in got]), xdot=np.stack([g["xdot"] for g in got]),
                path=np.array([g["path_length"] for g in got]),
                smoothness=np.array([g["smoothness"] for g in got]),
                status=np.array([[g["status"], g["steps"], g["smooth_n"]] for g in got]))


def _stacked(got):
    return dict(f=np.stack([g["f"] for g in got]), sumA=np.stack([g["sumA"] for g in got]),
                sumAf=np.stack([g["sumAf"] for g in got]), eig=np.stack([g["eig"] for g in got]),
                counts=np.array([[g["n_rays"], g["n_hits"], g["n_active"], g["rank"], g["status"]]
                                 for g in got]))


# ------------------------------------------------------------------------------ work
def _reach_bytes(name):
    """One bit per voxel of the map within the range of a state."""
    kind, extent, vs, _, _, rng = MAPS[name]
    return np.prod([min(e, 2 * rng) for e in extent]) / vs ** 3 / 8


def work(case):
    kind = case["kind"]
    per_ray, res = 150.0, R.RESULT_BYTES + 48      # direction, policy, nine sums
    if kind == "eval":
        return dict(bytes=_reach_bytes(case["map"]) + res + (60 if case["records"] else 0) * case["rays"],
                    flops=per_ray * case["rays"])
    if kind == "scan":
        return dict(bytes=(12 + (36 if case["records"] else 0)) * case["points"] + res,
                    flops=100.0 * case["points"])
    if kind == "batch":
        lo, hi = case["ray_lo"], case["ray_hi"]
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        _, extent, vs, _, _, _ = MAPS[case["map"]]
        whole = np.prod(extent) / vs ** 3 / 8
        return dict(bytes=whole + res * case["states"], flops=per_ray * mean * case["states"])
    if kind == "combined":
        return dict(bytes=125e3 + (res + 28) * case["states"],
                    flops=per_ray * case["rays"] * case["states"])
    if kind == "rollout":
        if case["esdf"]:
            return dict(bytes=200 * 56.0, flops=case["steps"] * 200 * 20.0 * case["states"])
        return dict(bytes=125e3 + 168.0 * case["states"],
                    flops=per_ray * case["rays"] * case["states"] * case["steps"])
    if kind == "esdf":
        return dict(bytes=56.0 * case["prims"] + (res + 56) * case["states"],
                    flops=20.0 * case["prims"] * case["states"])
    if kind == "served":
        lo, hi = case["ray_lo"], case["ray_hi"]
        return dict(bytes=sum(_reach_bytes(m) for m in ("dense128", "hashed40", "hashed100")),
                    flops=per_ray * (hi - lo) / math.log(hi / lo) * case["requests"])
    _, extent, vs, _, _, _ = MAPS[case["map"]]
    voxels = np.prod(extent) / vs ** 3       # refresh: a byte a voxel, or TSDF in a third of the blocks
    return dict(bytes=voxels * (1.0 if "dense" in case["map"] else 4.0 / 3.0) + res,
                flops=per_ray * case["rays"])


# ------------------------------------------------------------------------------ exact
def _fma(a, b, c):
    return (a.double() * b.double() + c.double() if torch.is_tensor(c)
            else a.double() * b.double() + float(c)).float()


def _directions(i):
    """Directions of Halton indices i (int64): the FP32 recipe that defines them."""
    u = torch.zeros_like(i, dtype=torch.float64)
    for k in range(24):
        u += ((i >> k) & 1).double() * 2.0 ** -(k + 1)
    num, q = torch.zeros_like(i), i.clone()
    for _ in range(20):
        num = num * 3 + q % 3
        q = q // 3
    u, v = u.float(), (num.double() / 3.0 ** 20).float()
    z, st = 1.0 - 2.0 * u, 2.0 * (u * (1.0 - u)).sqrt()
    w = v * 8.0
    o = w.int()
    t = w - o.float()
    a = torch.where(o % 2 == 1, 1.0 - t, t) * torch.tensor(math.pi / 4, dtype=torch.float32, device=i.device)
    a2 = a * a
    f = [torch.tensor(1.0 / math.factorial(n), dtype=torch.float32, device=i.device)
         for n in range(13)]
    ps = (-f[11]).expand_as(a)
    for c in (f[9], -f[7], f[5], -f[3]):
        ps = _fma(ps, a2, c)
    sa = _fma(a2 * a, ps, a)
    pc = f[12].expand_as(a)
    for c in (-f[10], f[8], -f[6], f[4], -f[2]):
        pc = _fma(pc, a2, c)
    ca = _fma(a2, pc, torch.ones_like(a))
    swap = ((o + 1) & 2) != 0
    c, s = torch.where(swap, sa, ca), torch.where(swap, ca, sa)
    c = torch.where((o >= 2) & (o <= 5), -c, c)
    s = torch.where(o >= 4, -s, s)
    return torch.stack([st * c, st * s, z], 1)


def _march(occ, is_dense, P, D, R_fx, vs):
    """Entry distance of the first occupied voxel per ray (inf: none); P (n, 3) 2^-16 voxels in
    the volume's frame, D (n, 3) 2^-24; exact crossings in 64-bit integers."""
    n = len(P)
    nz, ny, nx = occ.shape
    lim = torch.tensor([nx, ny, nz], device=P.device)
    out = torch.full((n,), math.inf, dtype=torch.float64, device=P.device)
    A, s, k = D.abs(), torch.where(D > 0, 1, -1), P >> 16
    N = torch.where(D > 0, (k << 16) + 65536 - P, torch.where(D < 0, P - (k << 16), 1))
    idx = torch.arange(n, device=P.device)
    d = torch.zeros(n, dtype=torch.float64, device=P.device)
    alive = torch.ones(n, dtype=torch.bool, device=P.device)
    for it in range(1 << 20):
        inside = ((k >= 0) & (k < lim)).all(1)
        kc = torch.where(inside[:, None], k, 0)
        hit = inside & occ[kc[:, 2], kc[:, 1], kc[:, 0]] & alive
        out[idx[hit]] = d[hit]
        alive &= ~hit
        if is_dense:
            alive &= inside
        else:      # beyond the volume and moving away: nothing occupied is left ahead
            alive &= ~(((k < 0) & (s < 0)) | ((k >= lim) & (s > 0))).any(1)
        y = N[:, 1] * A[:, 0] < N[:, 0] * A[:, 1]
        nw, aw = torch.where(y, N[:, 1], N[:, 0]), torch.where(y, A[:, 1], A[:, 0])
        zz = N[:, 2] * aw < nw * A[:, 2]
        ax = torch.where(zz, 2, torch.where(y, 1, 0))
        nn, aa = torch.where(zz, N[:, 2], nw), torch.where(zz, A[:, 2], aw)
        alive &= (nn << 24) <= R_fx * aa
        d = nn.double() / aa.clamp_min(1).double() * 256.0 * vs
        step = torch.nn.functional.one_hot(ax, 3)
        k, N = k + s * step, N + 65536 * step
        if it % 8 == 7:
            if not alive.any():
                break
            k, N, A, s, d, idx = k[alive], N[alive], A[alive], s[alive], d[alive], idx[alive]
            alive = alive[alive]
    return out


def _policy(base, cubic, u, d, v, valid):
    """Per-ray (n_active contribution, f, A (6), A f (3)), FP64."""
    r = -u
    d = torch.where(valid, d, 1.0)
    vu = (v * u).sum(1)
    z = torch.where(vu > 0, vu * vu, 0.0) * base["eta_damp"] / (d / base["nu_damp"] + base["eps"])
    fr = base["eta_rep"] * torch.exp(-d / base["nu_rep"]) + z
    x = d / base["r"]
    w = torch.where(x < 1.0, (1 - x) ** 2 * (1 + 2 * x) if cubic else (1 - x) ** 2, 0.0)
    c = base["c"]
    sc = z / (z + c * torch.log1p(torch.exp(-2 * c * z)))
    al = torch.where(valid, w * sc * sc, 0.0)
    A = al[:, None] * torch.stack([r[:, 0] * r[:, 0], r[:, 0] * r[:, 1], r[:, 0] * r[:, 2],
                                   r[:, 1] * r[:, 1], r[:, 1] * r[:, 2], r[:, 2] * r[:, 2]], 1)
    f = torch.where(valid, fr, 0.0)[:, None] * r
    return f, A, (al * fr * (r * r).sum(1))[:, None] * r


def _resolve(S, b, always=False):
    """f, eig of Eq. (1); f is None where a sum is too near to singular to say."""
    S, b = S.cpu().numpy(), b.cpu().numpy()
    M = S[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)
    lam, Q = np.linalg.eigh(M)
    top = lam[:, 2:3]
    keep = (lam > 1e-12 * top) & (top > 1e-300)
    inv = np.where(keep, 1.0 / np.where(keep, lam, 1.0), 0.0)
    f = np.einsum("nij,nj->ni", Q, inv * np.einsum("nji,nj->ni", Q, b))
    poor = (top[:, 0] > 0) & (lam[:, 0] < 1e-5 * top[:, 0])
    return (None if poor.any() and not always else f), lam


def _raycast_sums(w, base, cubic, states, sites, rays, want_rays=False):
    """sum A, sum A f per state in 64 bits (and, for one state, d and the per-ray values)."""
    S = torch.zeros((len(states), 6), dtype=torch.float64, device="cuda")
    b = torch.zeros((len(states), 3), dtype=torch.float64, device="cuda")
    R_fx = int(np.rint(w.max_range / w.vs * 65536.0))
    extra = None
    order = np.argsort(sites, kind="stable")
    at = 0
    while at < len(order):
        group, total = [], 0
        while at < len(order) and (not group or (total + rays[order[at]] <= 1 << 21 and
                                                 sites[order[at]] == sites[group[0]])):
            group.append(order[at])
            total += int(rays[order[at]])
            at += 1
        n = torch.as_tensor(np.asarray(rays)[group], device="cuda")
        g = torch.repeat_interleave(torch.arange(len(group), device="cuda"), n)
        first = torch.cumsum(n, 0) - n
        i = torch.arange(total, device="cuda") - first[g] + 1
        u32 = _directions(i)
        D = (u32 * 16777216.0).round().long()
        P = np.rint(states[group][:, :3] / w.vs * 65536.0).astype(np.int64)
        P -= np.asarray(w.offsets[sites[group[0]]], np.int64) << 16
        P = _cuda(P)
        d = _march(w.occ[sites[group[0]]], w.kind == "dense", P[g], D, R_fx, w.vs)
        v = _cuda(states[group][:, 3:])[g]
        f, A, Af = _policy(base, cubic, u32.double(), d, v, d.isfinite())
        gi = torch.as_tensor(np.asarray(group), device="cuda")
        S.index_add_(0, gi[g], A)
        b.index_add_(0, gi[g], Af)
        if want_rays:
            extra = (d, torch.cat([f, A], 1))
    return (S, b, extra) if want_rays else (S, b)


def _attractor(S, b, x, v, goals, rays, mean):
    if mean:
        S, b = S / rays[:, None], b / rays[:, None]
    e = goals - x
    z = e.square().sum(1).sqrt()
    c = STATIC["c"]
    h = z + c * torch.log1p(torch.exp(-2 * c * z))
    S = S + torch.tensor([1.0, 0, 0, 1.0, 0, 1.0], dtype=torch.float64, device=S.device)
    return S, b + ALPHA * e / h[:, None] - BETA * v


def _esdf_query(sc, x):
    """Distance (>= 0) and gradient of the nearest primitive, (n,) and (n, 3)."""
    ds, gs = [], []
    for p in x.split(max(1, (1 << 23) // len(sc.center))):
        sd = sc.sdf(p[:, None, :])
        best, j = sd.min(1)
        q, h = p - sc.c[j], sc.h[j]
        ball = q / q.square().sum(1, keepdim=True).sqrt()
        a = q.abs() - h
        o = a.clamp_min(0.0) * torch.where(q < 0, -1.0, 1.0)
        l = o.square().sum(1, keepdim=True).sqrt()
        face = torch.nn.functional.one_hot(a.argmax(1), 3) * torch.where(q < 0, -1.0, 1.0)
        box = torch.where(l > 0, o / l.clamp_min(1e-300), face)
        ds.append(best.clamp_min(0.0))
        gs.append(torch.where(sc.s[j][:, None], ball, box))
    return torch.cat(ds), torch.cat(gs)


def _esdf_sums(sc, x, v):
    d, g = _esdf_query(sc, x)
    _, S, b = _policy(STATIC, False, -g, d, v, torch.ones_like(d, dtype=torch.bool))
    return S, b, d, g


def _fields(S, b, always=False):
    f, eig = _resolve(S, b, always)
    return dict(f=f, sumA=S, sumAf=b, eig=eig)


def _rollout_exact(case, i):
    w = i["worlds"][0]
    st, goals, n = i["states"].copy(), i["goals"], case["states"]
    status, steps = np.zeros(n, int), np.zeros(n, int)
    path, sm, smn = np.zeros(n), np.zeros(n), np.zeros(n, int)
    seg0, prev, have = st[:, :3].copy(), np.zeros((n, 3)), np.zeros(n, bool)
    occ = w.occ[0].cpu().numpy()
    dims = np.array(occ.shape[::-1])
    for _ in range(case["steps"]):
        on = np.nonzero(status == 0)[0]
        if not len(on):
            break
        x, v = _cuda(st[on, :3]), _cuda(st[on, 3:])
        if case["esdf"]:
            S, b, _, _ = _esdf_sums(w.scenes[0], x, v)
            S, b = _attractor(S, b, x, v, _cuda(goals[on]), None, False)
        else:
            S, b = _raycast_sums(w, STATIC, False, st[on], i["sites"][on], i["rays"][on])
            S, b = _attractor(S, b, x, v, _cuda(goals[on]), _cuda(i["rays"][on].astype(float)), True)
        f, _ = _resolve(S, b, True)
        vn = st[on, 3:] + f * 0.01
        xn = st[on, :3] + vn * 0.01
        path[on] += np.linalg.norm(xn - st[on, :3], axis=1)
        st[on, :3], st[on, 3:] = xn, vn
        steps[on] += 1
        for r in on:
            if steps[r] % 10 == 0:
                seg = st[r, :3] - seg0[r]
                seg0[r] = st[r, :3]
                if have[r]:
                    a, c = np.linalg.norm(prev[r]), np.linalg.norm(seg)
                    if a > 0 and c > 0:
                        sm[r] += 1.0 - math.acos(min(1.0, max(-1.0, prev[r] @ seg / (a * c)))) / math.pi
                        smn[r] += 1
                prev[r], have[r] = seg, True
            k = np.floor(np.rint(st[r, :3] / w.vs * 65536.0) / 65536.0).astype(int)
            inside = (k >= 0).all() and (k < dims).all()
            if inside and occ[k[2], k[1], k[0]]:
                status[r] = R.RMP_ROLLOUT_COLLIDED
            elif np.linalg.norm(st[r, :3] - goals[r]) < 0.2:
                status[r] = R.RMP_ROLLOUT_REACHED
            elif steps[r] >= case["steps"]:
                status[r] = R.RMP_ROLLOUT_TIMEOUT
    return dict(x=st[:, :3], xdot=st[:, 3:], path=path,
                smoothness=np.where(smn > 0, sm / np.maximum(smn, 1), 1.0), status=None)


def exact(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    one = lambda d: {k: None if v is None else v[0] for k, v in d.items()}  # noqa: E731
    if kind == "rollout":
        return _rollout_exact(case, i)
    if kind == "scan":
        p = i["points"].double()
        d = p.square().sum(1).sqrt()
        ok = d.isfinite() & (d > 0) & (d >= LIDAR["min_range"]) & (d <= 30.0)
        u = torch.where(ok[:, None], p / d[:, None], 0.0)
        v = _cuda(i["state"][3:])[None, :]
        f, A, Af = _policy(LIDAR, False, u, d, v, ok)
        out = _fields(A.sum(0, keepdim=True), Af.sum(0, keepdim=True))
        out = one(out) if case["sync"] else out
        return [out, torch.cat([f, A], 1)] if case["records"] else out
    if kind == "esdf":
        x, v = _cuda(i["states"][:, :3]), _cuda(i["states"][:, 3:])
        S, b, d, g = _esdf_sums(i["scene"], x, v)
        if case["goals"]:
            S, b = _attractor(S, b, x, v, _cuda(i["goals"]), None, False)
        return [_fields(S, b, case["goals"]), torch.cat([d[:, None], g], 1)]
    if kind == "eval" and case["records"]:
        S, b, (d, per) = _raycast_sums(i["worlds"][0], STATIC, case["cubic"], i["states"],
                                       i["sites"], i["rays"], True)
        out = _fields(S, b)
        return [one(out) if case["sync"] else out,
                dict(voxel=None, d=None, outcome=None, per_ray=per)]
    n = len(i["states"])
    S = torch.zeros((n, 6), dtype=torch.float64, device="cuda")
    b = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    for k, w in enumerate(i["worlds"]):
        at = np.nonzero(i["world_of"] == k)[0]
        if len(at):
            S[at], b[at] = _raycast_sums(w, STATIC, case.get("cubic", False), i["states"][at],
                                         i["sites"][at], i["rays"][at])
    if kind == "combined":
        S, b = _attractor(S, b, _cuda(i["states"][:, :3]), _cuda(i["states"][:, 3:]),
                          _cuda(i["goals"]), _cuda(i["rays"].astype(float)), case["mean"])
        return _fields(S, b, True)
    out = _fields(S, b)
    return one(out) if kind == "refresh" or (kind == "eval" and case["sync"]) else out
