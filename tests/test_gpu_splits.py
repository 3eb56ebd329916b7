"""The cuts of the work over CTAs, warps and lanes where they change: ESDF states on both sides
of 8, 16 and 32 states a CTA, ties and distances that FP32 cannot tell apart, coordinates past
FP32; batches with more states than one run of the set-up kernel takes and with total loads on
both sides of the march's segment cuts; scans whose last warp is ragged, with the per-point rows;
batches with a CTA per state, rollouts with a CTA per robot."""
from fractions import Fraction as F

import numpy as np
import pytest

import oracle as O
from paper_2301_08068_gb300 import rmp as R
from paper_2301_08068_gb300 import workloads as W

from gpu_helpers import (assert_hits_exact, assert_per_ray_close, assert_result_close,
                         scan_abs_term, torch_cuda)
from test_gpu_batch import run_batch
from test_gpu_esdf import check_states, run_esdf, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch_cuda()
    c = R.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 8, 9, 1216, 1217, 2432, 2433])
def test_esdf_states_per_cta(ctx, n):
    _, prims = scene(40)
    rng = np.random.default_rng(n)
    states = np.concatenate([rng.uniform(-1.0, 11.0, (n, 3)), rng.normal(0.0, 1.0, (n, 3))], 1)
    goals = rng.uniform(0.0, 10.0, (n, 3))
    eid = R.rmp_esdf_upload(ctx.handle, prims)
    try:
        check_states(ctx, eid, O.prims_array(prims), states, goals, W.PARAMS_STATIC_MAP)
    finally:
        R.rmp_esdf_release(ctx.handle, eid)


@pytest.mark.parametrize("gap", [0.0, 1e-13, 1e-9, 1e-7])
@pytest.mark.parametrize("n", [2, 33, 97])
def test_esdf_ties(ctx, gap, n):
    """n spheres and boxes at the same distance of a state but for the gap, which FP32 cannot
    tell: the first minimum of a sequential scan wins, here in every lane and every turn."""
    rng = np.random.default_rng(n)
    sign = np.sign(rng.normal(size=(n, 3)))
    # both 0.5 sqrt(3) away: the sphere 2 sqrt(3) less its radius, the box from its corner
    prims = [W.Primitive("sphere", 5.0 + 2.0 * sign[i], np.array([1.5 * np.sqrt(3.0)])) if i % 3
             else W.Primitive("box", 5.0 + 2.0 * sign[i], np.full(3, 1.5)) for i in range(n)]
    for i, p in enumerate(prims):
        p.center[0] += gap * ((7 * i) % n) * sign[i, 0]
    pr = O.prims_array(prims)
    states = np.zeros((20, 6))
    states[:, :3] = 5.0
    states[1:, :3] += rng.normal(0.0, 1e-13, (19, 3))
    states[:, 3:] = rng.normal(0.0, 1.0, (20, 3))
    eid = R.rmp_esdf_upload(ctx.handle, prims)
    try:
        check_states(ctx, eid, pr, states, None, W.PARAMS_STATIC_MAP)
    finally:
        R.rmp_esdf_release(ctx.handle, eid)


def test_esdf_beyond_fp32(ctx):
    """Primitives and states so far away that FP32 holds neither the squares nor the coordinates:
    the query equals the oracle's bit for bit."""
    far = [W.Primitive("sphere", np.array([1e20, -3e19, 2.0]), np.array([4e18])),
           W.Primitive("box", np.array([-1e60, 0.0, 1e59]), np.array([1e40, 2.0, 1e30])),
           W.Primitive("sphere", np.array([1.0, 2.0, 3.0]), np.array([0.5]))]
    pr = O.prims_array(far)
    x = np.array([[0.0, 0.0, 0.0], [1e17, -1e18, 2.0], [3e19, 1e19, -1e19], [-1e59, 1e58, 0.0],
                  [-9.9e59, 1.0, 1e59], [1.2, 2.1, 3.3], [1e20, 0.0, 0.0]])
    states = np.concatenate([x, np.full((len(x), 3), -0.25)], 1)
    eid = R.rmp_esdf_upload(ctx.handle, far)
    try:
        _, q = run_esdf(ctx, eid, states, None, R.make_params(W.PARAMS_STATIC_MAP, 10.0))
        po = O.make_params(W.PARAMS_STATIC_MAP, 10.0)
        for i, s in enumerate(states):
            assert np.array_equal(q[i], O.esdf_eval(pr, s[:3], s[3:], po)[1]), i
    finally:
        R.rmp_esdf_release(ctx.handle, eid)


@pytest.mark.parametrize("n_states,total", [(1216, 9000), (1217, 19000), (2500, 40000),
                                            (2500, 90000), (1217, 200000)])
def test_batch_many_states(ctx, n_states, total):
    """Set-up runs of 8 and of more states a CTA, states without rays and invalid ones among
    them, 1, 2 and 4 segments marched: a state's result is bitwise the one it has alone."""
    wl = W.hashed_workload(n_states=8, state_seed_index=21)
    mid, om = ctx.upload(wl.map), O.OracleMap(wl.map)
    rng = np.random.default_rng(total)
    counts = rng.multinomial(total, rng.dirichlet(np.full(n_states, 0.3))).astype(np.uint32)
    states = np.stack([np.concatenate([wl.states[b % 8].x, wl.states[b % 8].xdot])
                       for b in range(n_states)])
    bad = rng.choice(n_states, 9, replace=False)
    counts[bad] = 100
    states[bad, rng.integers(0, 6, 9)] = np.nan
    pg, po = R.make_params(wl.params, wl.max_range), O.make_params(wl.params, wl.max_range)
    try:
        res, h, _, _ = run_batch(ctx, mid, states, counts, pg)
        for b in range(n_states):
            if b in bad:                # a position is checked; a velocity only ends in the sums
                at_x = np.isnan(states[b, :3]).any()
                assert res[b]["status"] == (R.RMP_ERR_INVALID_ARG if at_x else 0)
            elif counts[b] == 0:
                assert res[b]["status"] == 0 and res[b]["n_rays"] == 0
                assert np.all(res[b]["f"] == 0.0)
        good = np.setdiff1d(np.flatnonzero(counts), bad)
        for b in [*good[:3], *good[-3:], *rng.choice(good, 14), int(np.argmax(counts))]:
            ro, ho, por = O.raycast_eval(om, states[b, :3], states[b, 3:], int(counts[b]), po)
            assert_hits_exact(h[b, :counts[b]], ho)
            assert_result_close(res[b], ro, por)
            alone = run_batch(ctx, mid, states[b:b + 1], counts[b:b + 1], pg, want=False)[0][0]
            for key in ("f", "sumA", "sumAf", "eig"):
                assert np.array_equal(alone[key], res[b][key]), (b, key)
    finally:
        R.rmp_map_release(ctx.handle, mid)


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 4097, 77825])
def test_scan_rows_ragged(ctx, n):
    """The per-point rows, which a warp writes together: against the oracle, and nothing is
    written past the last point."""
    sw = W.lidar_workload()
    pts = sw.points[np.random.default_rng(n).integers(0, len(sw.points), n)]
    torch = torch_cuda()
    per = torch.full(((n + 7) * 9,), -7.5, dtype=torch.float32, device="cuda")
    rg = R.rmp_scan_eval(ctx.handle, torch.from_numpy(pts).cuda(), sw.x, sw.xdot,
                         R.make_params(sw.params, sw.max_range), per_ray=per[:9 * n])
    got = per.cpu().numpy().reshape(-1, 9).astype(np.float64)
    assert np.all(got[n:] == -7.5)
    ro, por = O.scan_eval(pts, sw.x, sw.xdot, O.make_params(sw.params, sw.max_range))
    at = scan_abs_term(pts, sw.x, sw.xdot, sw.params)
    assert_per_ray_close(got[:n], por, at)
    assert_result_close(rg, ro, por, at)


@pytest.mark.parametrize("n_states,red,lgs,cells", [(1, 0, -1, -1), (8, 1, -1, -1), (152, 0, -1, -1),
                                                    (153, 0, 2, -1), (153, 1, 1, 0), (304, 0, 0, 0),
                                                    (305, 0, -1, -1)])
@pytest.mark.parametrize("dense", [True, False])
def test_batch_cta_per_state(ctx, dense, n_states, red, lgs, cells):
    """A CTA per state (max_rays 1024) and the packed chunks of the persistent grid (1025) give the
    same records, rows and sums, for invalid states and states without rays too; likewise combined
    with the attractor."""
    torch = torch_cuda()
    wl = W.dense_box_workload(n_states=6, jitter=True) if dense \
        else W.hashed_workload(n_states=6, state_seed_index=52)
    mid = ctx.upload(wl.map)
    rng = np.random.default_rng(n_states)
    states = np.stack([np.concatenate([wl.states[b % 6].x, wl.states[b % 6].xdot])
                       for b in range(n_states)])
    counts = rng.choice([0, 1, 2, 31, 32, 33, 64, 100, 255, 256, 257, 511, 777, 1023, 1024], n_states)
    counts[0] = 1024
    if n_states > 8:
        states[3, 1], states[4, 0], states[5, 4] = np.nan, 1e9, np.nan
        counts[6] = 1500                                  # more rays than max_rays
    counts = counts.astype(np.uint32)
    p = R.make_params(dict(wl.params, reduce_mode=red), wl.max_range)
    R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, lgs)
    R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, cells)
    try:
        a, ha, pa, _ = run_batch(ctx, mid, states, counts, p, max_rays=1024)
        o, ho, po, _ = run_batch(ctx, mid, states, counts, p, max_rays=1025)
        assert np.array_equal(ha, ho[:, :1024])
        assert np.array_equal(pa, po[:, :1024], equal_nan=True)
        for b in range(n_states):
            for key, want in o[b].items():
                assert np.array_equal(a[b][key], want, equal_nan=True), (b, key)
        st, nr = torch.tensor(states, device="cuda"), torch.tensor(counts.astype(np.int32)).cuda()
        gl = torch.tensor(states[:, :3] + rng.normal(size=(n_states, 3)), device="cuda")
        for mean in (False, True):
            got = []
            for mr in (1024, 1025):
                ws = torch.empty(R.rmp_batch_workspace_bytes(n_states, mr), dtype=torch.uint8,
                                 device="cuda")
                out = torch.empty((n_states, R.RESULT_BYTES), dtype=torch.uint8, device="cuda")
                R.rmp_combined_eval_batch_async(ctx.handle, mid, st, nr, n_states, mr, p, gl, 10.0,
                                                15.0, ws, out, metric_mean=mean)
                got.append(out.cpu().numpy())
            for b in range(n_states):
                a, o = (R.result_from_bytes(g[b].tobytes()) for g in got)
                for key, want in o.items():
                    assert np.array_equal(a[key], want, equal_nan=True), (b, key)
    finally:
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, -1)
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, -1)
        R.rmp_map_release(ctx.handle, mid)


def fma(a, b, c):
    """a b + c rounded once, elementwise."""
    return np.array([float(F(x) * F(y) + F(z)) for x, y, z in zip(a, b, c)])


@pytest.mark.parametrize("rays,mean,red,lgs,steps", [
    (1, False, 0, -1, 40), (31, True, 0, -1, 40), (64, True, 1, -1, 12), (257, True, 0, 1, 12),
    (300, False, 1, 0, 12), (1000, True, 0, -1, 12), (1024, False, 0, -1, 300),
    (1025, True, 0, -1, 8), (4096, True, 0, -1, 4), (4097, True, 0, -1, 3)])
@pytest.mark.parametrize("dense", [True, False])
def test_rollout_cta_per_robot(ctx, dense, rays, mean, red, lgs, steps):
    """Every number of robots and so of warps a CTA, and rollouts evaluated together per step,
    give a robot the same bits; the path is that of combined evaluations and Euler steps.  Among
    the robots: one at its goal, a fast one that hits or leaves, one too far away, NaN."""
    wl = W.dense_box_workload(n_states=6, jitter=True) if dense \
        else W.hashed_workload(n_states=6, state_seed_index=52)
    mid = ctx.upload(wl.map)
    torch = torch_cuda()
    rng = np.random.default_rng(rays)
    robots = np.array([np.concatenate([s.x, s.xdot, s.x + rng.uniform(-3, 3, 3)]) for s in wl.states])
    robots = np.concatenate([robots, robots[:5]])
    robots[6, 6:] = robots[6, :3] + 1e-4
    robots[7, 3:6] = [60.0, -80.0, 10.0]
    robots[8, :3] = 1e9
    robots[9, 3:6] = np.nan
    robots[10, :3] = np.nan
    many = np.tile(robots, (28, 1))                       # 308 robots
    p = R.make_params(dict(wl.params, reduce_mode=red), wl.max_range)
    rp = R.rollout_params(10.0, 15.0, 0.01, 0.05, steps, 3, rays, metric_mean=mean)
    R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, lgs)
    try:
        ref = R.rmp_rollout(ctx.handle, mid, robots, p, rp)
        for n in (1, 152, 153, 305):
            got = R.rmp_rollout(ctx.handle, mid, many[:n], p, rp)
            for b in range(n):
                for key, want in ref[b % 11].items():
                    assert np.array_equal(got[b][key], want, equal_nan=True), (n, b, key)
        x, v, goal = robots[:8, :3].copy(), robots[:8, 3:6].copy(), robots[:8, 6:]
        nr = torch.full((8,), rays, dtype=torch.int32, device="cuda")
        ws = torch.empty(R.rmp_batch_workspace_bytes(8, rays), dtype=torch.uint8, device="cuda")
        out = torch.empty((8, R.RESULT_BYTES), dtype=torch.uint8, device="cuda")
        gl = torch.tensor(goal, device="cuda")
        for step in range(max(r["steps"] for r in ref[:8])):
            st = torch.tensor(np.concatenate([x, v], 1), device="cuda")
            R.rmp_combined_eval_batch_async(ctx.handle, mid, st, nr, 8, rays, p, gl, 10.0, 15.0, ws,
                                            out, metric_mean=mean)
            o = out.cpu().numpy()
            for b in range(8):
                if step < ref[b]["steps"]:
                    v[b] = fma(R.result_from_bytes(o[b].tobytes())["f"], [0.01] * 3, v[b])
                    x[b] = fma(v[b], [0.01] * 3, x[b])
        for b in range(8):
            assert np.array_equal(ref[b]["x"], x[b]) and np.array_equal(ref[b]["xdot"], v[b]), b
        assert ref[6]["status"] == R.RMP_ROLLOUT_REACHED and ref[8]["status"] == R.RMP_ROLLOUT_FAILED
        assert ref[10]["status"] == R.RMP_ROLLOUT_FAILED
    finally:
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, -1)
        R.rmp_map_release(ctx.handle, mid)


@pytest.mark.parametrize("n", [1, 9, 1217, 2433])
def test_esdf_rollout_states_per_cta(ctx, n):
    """8, 16 and 32 robots a CTA: each robot's path is the one it has among few, robots that stop
    early and an invalid one beside it."""
    wl = W.hashed_workload(n_states=6, state_seed_index=52)
    _, prims = scene(40)
    rng = np.random.default_rng(5)
    robots = np.concatenate([rng.uniform(0.5, 9.5, (12, 3)), rng.normal(0.0, 1.0, (12, 3)),
                             rng.uniform(0.5, 9.5, (12, 3))], 1)
    robots[1, 6:] = robots[1, :3] + 1e-4                  # at its goal
    robots[2, 0] = np.nan
    mid, eid = ctx.upload(wl.map), R.rmp_esdf_upload(ctx.handle, prims)
    p = R.make_params(wl.params, wl.max_range)
    rp = R.rollout_params(10.0, 15.0, 0.01, 0.05, 45, 4, 1)
    try:
        one = [R.rmp_rollout_esdf(ctx.handle, mid, eid, robots[b:b + 1], p, rp)[0] for b in range(12)]
        got = R.rmp_rollout_esdf(ctx.handle, mid, eid, np.tile(robots, (n // 12 + 1, 1))[:n], p, rp)
        for b in range(n):
            for key, want in one[b % 12].items():
                assert np.array_equal(got[b][key], want, equal_nan=True), (b, key)
        assert one[1]["steps"] == 1 and one[2]["status"] == R.RMP_ROLLOUT_FAILED
    finally:
        R.rmp_map_release(ctx.handle, mid)
        R.rmp_esdf_release(ctx.handle, eid)


def test_map_memory_reused(ctx):
    """Maps uploaded and released in turn by several threads, each on a stream of its own: the
    memory one gives back serves another, and every evaluation is the one of a fresh context."""
    import threading
    torch = torch_cuda()
    wls = [W.dense_box_workload(n_states=1, jitter=True), W.hashed_workload(n_states=1, state_seed_index=52)]
    want = []
    for wl in wls:
        c = R.Context(0)
        s = wl.states[0]
        want.append(R.rmp_raycast_eval(c.handle, c.upload(wl.map), s.x, s.xdot, 2000,
                                       R.make_params(wl.params, wl.max_range)))
        c.close()
    bad = []

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for j in range(6):
                wl, w = wls[(i + j) % 2], want[(i + j) % 2]
                mid = ctx.upload(wl.map)
                s = wl.states[0]
                got = R.rmp_raycast_eval(ctx.handle, mid, s.x, s.xdot, 2000,
                                         R.make_params(wl.params, wl.max_range))
                R.rmp_map_release(ctx.handle, mid)
                if any(not np.array_equal(got[k], w[k]) for k in w):
                    bad.append((i, j))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


@pytest.mark.parametrize("contexts", [1, 2])
def test_rollouts_from_several_threads(ctx, contexts):
    """Rollouts of 2000 rays, whose CTAs want 66 KB of shared memory, while three other threads keep
    asking for rollouts of 16 rays, on one context and on two: every call succeeds and gives
    what it gives alone."""
    import ctypes as C
    import threading
    wl = W.hashed_workload(n_states=32, state_seed_index=52)
    p = R.make_params(wl.params, wl.max_range)
    robots = np.stack([np.concatenate([s.x, s.xdot, s.x + 3.0]) for s in wl.states])
    other = R.Context(0) if contexts == 2 else ctx
    rp = [R.rollout_params(10.0, 15.0, 0.01, 0.05, 1, 1, rays) for rays in (2000, 16)]
    jobs = [(ctx, ctx.upload(wl.map), 32, rp[0]), (other, other.upload(wl.map), 1, rp[1])]
    fn = R.lib().rmp_rollout

    def call(i):
        c, mid, n, r = jobs[i]
        out = (R.rmp_rollout_result_t * n)()
        st = fn(c.handle, mid, robots.ctypes.data, n, C.byref(p), C.byref(r), None, out)
        return st, bytes(out)

    want = [call(0), call(1)]
    assert want[0][0] == 0 and want[1][0] == 0
    bad, done = [], threading.Event()

    def work(i):
        if i == 0:
            bad.extend(g[0] for g in (call(0) for _ in range(1500)) if g != want[0])
            done.set()
        else:
            while not done.is_set():
                g = call(1)
                if g != want[1]:
                    bad.append(g[0])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c, mid, _, _ in jobs:
        R.rmp_map_release(c.handle, mid)
    if contexts == 2:
        other.close()
    assert not bad, (len(bad), bad[:3])


@pytest.mark.parametrize("cells", [-1, 0])
@pytest.mark.parametrize("block,least", [(64, 12), (128, 6), (256, 2)])
def test_launch_info_of_the_kernel_that_runs(ctx, block, least, cells):
    """Resident CTAs per SM are those of the variant launched at this CTA size: 64- and 128-thread
    CTAs run one that is bounded to 768 threads an SM (85 registers), 256-thread ones one bounded
    to 512."""
    wl = W.hashed_workload(n_states=1, state_seed_index=52)
    mid = ctx.upload(wl.map)
    p = R.make_params(wl.params, wl.max_range)
    R.rmp_tune_set(ctx.handle, R.RMP_TUNE_BLOCK, block)
    R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, cells)
    try:
        info = R.rmp_eval_launch_info(ctx.handle, mid, 262144, p)
        assert info["block"] == block and info["ctas_per_sm"] >= least, info
    finally:
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_BLOCK, 0)
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, -1)
        R.rmp_map_release(ctx.handle, mid)


@pytest.mark.parametrize("n_states,max_rays", [(40, 1100), (3000, 40), (300, 500)])
def test_batches_back_to_back_on_one_workspace(ctx, n_states, max_rays):
    """Batches of other states and counts follow one another on one workspace without a wait, each
    resident beside its predecessor: every result is the one the batch has on its own.  The
    packed grid with few and with many states, and a CTA per state; single evaluations between
    them."""
    torch = torch_cuda()
    wl = W.hashed_workload(n_states=64, state_seed_index=23)
    mid = ctx.upload(wl.map)
    pg = R.make_params(wl.params, wl.max_range)
    rng = np.random.default_rng(n_states)
    sets = []
    for i in range(3):
        pick = rng.integers(0, 64, n_states)
        st = np.stack([np.concatenate([wl.states[b].x, wl.states[b].xdot]) for b in pick])
        counts = rng.integers(0, max_rays + 1, n_states).astype(np.int32)
        sets.append((torch.tensor(st, device="cuda"), torch.tensor(counts, device="cuda")))
    ws = torch.empty(R.rmp_batch_workspace_bytes(n_states, max_rays), dtype=torch.uint8, device="cuda")
    one = torch.empty(R.rmp_workspace_bytes(), dtype=torch.uint8, device="cuda")
    R.rmp_workspace_init(one)

    def batch(i, out):
        R.rmp_raycast_eval_batch_async(ctx.handle, mid, *sets[i], n_states, max_rays, pg, ws, out)

    def buffer():
        return torch.zeros((n_states, R.RESULT_BYTES), dtype=torch.uint8, device="cuda")

    want, single = [buffer() for _ in sets], torch.zeros(R.RESULT_BYTES, dtype=torch.uint8, device="cuda")
    for i, out in enumerate(want):
        batch(i, out)
        torch.cuda.synchronize()
    R.rmp_raycast_eval_async(ctx.handle, mid, sets[0][0][0], 700, pg, one, single)
    got, alone = [buffer() for _ in range(24)], torch.zeros_like(single)
    torch.cuda.synchronize()
    for j, out in enumerate(got):
        batch(j % 3, out)
        if j % 5 == 4:
            R.rmp_raycast_eval_async(ctx.handle, mid, sets[0][0][0], 700, pg, one, alone)
    torch.cuda.synchronize()
    assert torch.equal(single, alone)
    for j, out in enumerate(got):
        assert torch.equal(out, want[j % 3]), j
    R.rmp_map_release(ctx.handle, mid)
