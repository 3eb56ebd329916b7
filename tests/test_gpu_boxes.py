"""The box field of the march where it can go wrong: grids that are not multiples of 8, single
blocks, random occupancy from nearly empty to half full (boxes of every extent), states on
voxel boundaries and centres (ties), outside and far from a hashed map's blocks, the pole ray
of Halton offset 0, and segments.  Hit records equal the oracle's voxel-by-voxel march byte for
byte, with the boxes and (knob off) voxel by voxel."""
import numpy as np
import pytest

import oracle as O
from paper_2301_08068_gb300 import rmp as R
from paper_2301_08068_gb300 import workloads as W

from gpu_helpers import assert_hits_exact, gpu_raycast, torch_cuda

pytestmark = pytest.mark.gpu
VS = 0.1


@pytest.fixture(scope="module")
def ctx():
    torch_cuda()
    c = R.Context(0)
    yield c
    c.close()


def check(ctx, m, xs, n, max_range):
    mid, om = ctx.upload(m), O.OracleMap(m)
    knobs = ((-1, -1), (-1, 0), (-1, 2), (0, 0), (0, -1))      # voxel boxes, log2 segments
    try:
        for i, x in enumerate(xs):
            d = dict(W.PARAMS_STATIC_MAP, halton_offset=i & 1)
            v = np.array([0.4, -0.9, 0.2])
            _, ho, _ = O.raycast_eval(om, x, v, n, O.make_params(d, max_range))
            for cells, lgs in knobs:
                R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, cells)
                R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, lgs)
                _, hg, _ = gpu_raycast(ctx, mid, x, v, n, R.make_params(d, max_range))
                assert_hits_exact(hg, ho)
    finally:
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, -1)
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_LG_SEGMENTS, -1)
        R.rmp_map_release(ctx.handle, mid)


@pytest.mark.parametrize("dims", [(1, 1, 1), (8, 8, 8), (9, 7, 17), (24, 1, 65), (71, 64, 50)])
@pytest.mark.parametrize("density", [0.001, 0.03, 0.5])
def test_dense_grids(ctx, dims, density):
    rng = np.random.default_rng([*dims, int(1000 * density)])
    occ = (rng.uniform(size=dims[::-1]) < density).astype(np.uint8)
    ext = np.array(dims) * VS
    free = np.argwhere(occ == 0)[:, ::-1]
    xs = [ext * rng.uniform(size=3), ext * 0.5, ext + 0.05, np.array([-0.01, 0.02, 0.03])]
    if len(free):
        k = free[rng.integers(len(free))]
        xs += [(k + 0.5) * VS, k * VS + 1e-9]
    check(ctx, W.DenseMap(occ, VS, np.zeros(3)), xs, 777, 4.0)


@pytest.mark.parametrize("far", [False, True])      # a far block: the hash layout
@pytest.mark.parametrize("density", [0.0005, 0.02, 0.4])
def test_hashed_blocks(ctx, far, density):
    rng = np.random.default_rng([int(far), int(10000 * density)])
    keys = np.unique(rng.integers(-4, 5, (60, 3)), axis=0).astype(np.int32)
    if far:
        keys = np.concatenate([keys, [[9000, -7000, 800]]]).astype(np.int32)
    tsdf = np.where(rng.uniform(size=(len(keys), 512)) < density, -0.1, 0.2).astype(np.float32)
    tsdf[-1, 100] = -0.1                            # the far block is occupied
    xs = [rng.uniform(-3.0, 3.0, 3), np.zeros(3), np.array([0.05, -0.05, 0.15]),
          np.array([-30.0, 2.0, 1.0]), np.array([1.0, 6.0, -28.0]), np.array([4.1, 4.1, 4.1])]
    check(ctx, W.HashedMap(keys, tsdf, VS), xs, 777, 45.0)


def test_empty_hashed_map(ctx):
    keys = np.array([[0, 0, 0], [3, -2, 1]], np.int32)
    tsdf = np.full((2, 512), 0.2, np.float32)
    check(ctx, W.HashedMap(keys, tsdf, VS), [np.zeros(3), np.array([5.0, -5.0, 5.0])], 100, 20.0)


@pytest.mark.parametrize("axis,size", [(0, 66000), (1, 65600), (2, 70001)])
def test_dense_long_axis(ctx, axis, size):
    """More than 65535 voxels ahead on one axis, where the far face's crossing no longer fits 32
    bits (2^16 a voxel): states near both ends and 65535 to 65540 voxels before either face, among
    obstacles a few voxels away."""
    dims = [9, 10, 9]
    dims[axis] = size
    rng = np.random.default_rng(size)
    occ = (rng.uniform(size=dims[::-1]) < 0.01).astype(np.uint8)
    xs = []
    for k in (2, 65536, 65537, 65539, 65541, size - 1 - 65535, size - 1 - 65536, size - 1 - 65539,
              size - 3):
        c = np.array([4, 4, 4])
        c[axis] = min(max(k, 0), size - 1)
        occ[tuple(c[::-1])] = 0
        xs.append((c + 0.5) * VS)
    check(ctx, W.DenseMap(occ, VS, np.zeros(3)), xs, 333, 4.0)


@pytest.mark.parametrize("kind", ["dense", "grid", "hash"])
def test_uploaded_without_box_field(ctx, kind):
    """RMP_TUNE_CELL_SKIP 0 at the upload leaves the box field out, 4 KB per occupied block;
    evaluations give the oracle's records whatever the knob says then."""
    rng = np.random.default_rng(11)
    if kind == "dense":
        occ = (rng.uniform(size=(40, 33, 70)) < 0.02).astype(np.uint8)
        m, xs, r = W.DenseMap(occ, VS, np.zeros(3)), [np.array([3.0, 1.6, 2.0]), np.zeros(3) + 0.01], 4.0
        occupied = 9 * 5 * 5
    else:
        keys = np.unique(rng.integers(-4, 5, (60, 3)), axis=0).astype(np.int32)
        if kind == "hash":
            keys = np.concatenate([keys, [[9000, -7000, 800]]]).astype(np.int32)
        tsdf = np.where(rng.uniform(size=(len(keys), 512)) < 0.05, -0.1, 0.2).astype(np.float32)
        tsdf[:, 7] = -0.1
        m, xs, r = W.HashedMap(keys, tsdf, VS), [np.array([0.05, -0.05, 0.15]), np.array([4.1, 4.1, 4.1])], 20.0
        occupied = len(keys)
    size = []
    for knob in (-1, 0):
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, knob)
        mid = ctx.upload(m)
        size.append(R.rmp_map_info(ctx.handle, mid)["device_bytes"])
        R.rmp_map_release(ctx.handle, mid)
    assert size[0] - size[1] == 4096 * occupied, size
    upload = ctx.upload
    try:                                            # as check does, on a map without a field
        ctx.upload = lambda mm: (R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, 0), upload(mm))[1]
        check(ctx, m, xs, 500, r)
    finally:
        del ctx.upload
        R.rmp_tune_set(ctx.handle, R.RMP_TUNE_CELL_SKIP, -1)
