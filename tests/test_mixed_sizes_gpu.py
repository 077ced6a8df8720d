"""Primitives of very different size in one call: the large ones are counted and emitted apart from the
groups that share a warp, in one window, in several and in a batch."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2604_13191_gb300 as vx  # noqa: E402

DEV = torch.device("cuda", 0)
FIELDS = ("keys", "mask", "mass", "moment", "occ", "proj", "lobes")


def _small(kind, n, R, rng):
    p = rng.uniform(0.05, 0.95, (n, 1, 3)) + rng.uniform(-0.4, 0.4, (n, 3 if kind == "tri" else 2, 3)) / R
    out = np.zeros((*p.shape[:2], 4), np.float32)
    out[..., :3] = p
    if kind == "cap":
        out[..., 3] = 0.3 / R
    return out


def _mixed(kind, n, large, at, R, rng):
    """n small primitives with the `large` (triangles [., 3, 3] or capsules [., 2, 4], in voxels) from place `at`."""
    p = _small(kind, n, R, rng)
    p[at:at + len(large), :, :large.shape[2]] = large / R
    return p


def _geom(kind, p):
    t = torch.from_numpy(np.ascontiguousarray(p)).to(DEV)
    if kind == "tri":
        return dict(tri_verts=t)
    return dict(ctrl=t.reshape(-1, 4), fiber_offsets=torch.arange(p.shape[0] + 1, device=DEV) * 2)


def _oracle(kind, p, grid):
    if kind == "tri":
        return oracle.voxelize(synth.Workload("mixed", "triangles", grid, tri_verts=p, K=1))
    return oracle.voxelize(synth.Workload("mixed", "fibers", grid, ctrl=p.reshape(-1, 4), K=1,
                                          fiber_offsets=np.arange(p.shape[0] + 1, dtype=np.int64) * 2))


def _large(kind, n, R, extent, rng):
    """n primitives whose ranges are about `extent` voxels wide on each axis."""
    c = rng.uniform(extent / 2, R - extent / 2, (n, 1, 3))
    if kind == "tri":
        corner = np.array([[-1, -1, -1], [1, 0.2, 1], [-0.5, 1, 0.3]]) * (extent / 2 - 0.3)
        return c + corner * rng.choice([-1.0, 1.0], (n, 1, 3))
    out = np.zeros((n, 2, 4))
    out[:, 0, :3], out[:, 1, :3] = c[:, 0] - 0.2, c[:, 0] + 0.2
    out[..., 3] = extent / 2 - 1.0
    return out


@pytest.mark.parametrize("kind,n,R,extents,at", [
    ("tri", 14592, 32, [11, 12, 12, 13, 14, 20], 40),       # about the bound of a grouped range (2,048 voxels)
    ("cap", 14592, 32, [11, 12, 12, 13, 14, 20], 40),
    ("tri", 15001, 64, [45] * 3 + [10] * 30, 14968),        # above 65,536 voxels; the last, short group
    ("cap", 29185, 64, [45] * 2 + [14] * 31, 0),
    ("tri", 14591, 32, [14] * 32, 100),                     # a warp per primitive anyway
])
def test_large_among_small(kind, n, R, extents, at):
    rng = np.random.default_rng(n)
    p = _mixed(kind, n, np.concatenate([_large(kind, 1, R, e, rng) for e in extents]), at, R, rng)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ref = _oracle(kind, p, grid)
    ctx = vx.Context(DEV)
    geom = _geom(kind, p)
    got = ctx.voxelize(grid, **geom).host()
    for f in ("keys", "mask", "occ", "proj"):
        assert np.array_equal(got[f], ref[f]), f
    for f in ("mass", "moment"):
        assert np.array_equal(got[f].view(np.uint32), ref[f].view(np.uint32)), f
    # in windows, some with and some without large ranges
    ctx.set_max_pairs_per_pass(6 * n)
    parts = ctx.voxelize(grid, **geom).host()
    for f in FIELDS:
        assert np.array_equal(np.asarray(parts[f]).view(np.uint8), np.asarray(got[f]).view(np.uint8)), f
    ctx.close()
    # two instances of one group of a batch
    ctx = vx.Context(DEV)
    one = dict(kind="triangles" if kind == "tri" else "fibers", grid=grid, **geom)
    batch = ctx.batch([one, one], K=1)
    for _ in range(2):
        batch.run()
        for i in range(2):
            lv = batch.level(i, 0).host()
            for f in FIELDS:
                assert np.array_equal(np.asarray(lv[f]).view(np.uint8), np.asarray(got[f]).view(np.uint8)), f
    batch.close()
    ctx.close()


def _time(call):
    for _ in range(2):
        call()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


@pytest.mark.parametrize("kind,extent", [("cap", 50), ("tri", 90)])
def test_order_of_the_large_ones_costs_nothing(kind, extent):
    """32 large primitives in a row take no longer than the same ones far apart: each has a warp (one warp
    for all of them took 20 times as long)."""
    R, n = 256, 240000
    rng = np.random.default_rng(extent)
    large = _large(kind, 32, R, extent, rng)
    row = _mixed(kind, n, large, 64, R, rng)
    spread = row.copy()
    to = 64 + 7000 * np.arange(32)
    spread[64:96], spread[to] = row[to], row[64:96]
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    g_row, g_spread = _geom(kind, row), _geom(kind, spread)
    assert _time(lambda: ctx.voxelize(grid, **g_row)) < 1.5 * _time(lambda: ctx.voxelize(grid, **g_spread))
    ctx.close()
