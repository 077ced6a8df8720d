"""The adjoint with one lane per primitive (long arrays) against the same primitives in short arrays,
where a whole warp walks each: the voxels of many primitives pass through a warp's queue at once
in the one, those of a single primitive in the other."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2604_13191_gb300 as vx  # noqa: E402

DEV = torch.device("cuda", 0)


def _segments(n, R, rng, length):
    """n fibers of one segment, lengths (voxels) spread over `length`."""
    a = rng.uniform(0.0, 1.0, (n, 3))
    d = rng.standard_normal((n, 3))
    d *= (rng.uniform(*length, n) / R / np.linalg.norm(d, axis=1))[:, None]
    ctrl = np.zeros((n, 2, 4), np.float32)
    ctrl[:, 0, :3], ctrl[:, 1, :3] = a, a + d
    ctrl[..., 3] = rng.uniform(0.1, 0.4, (n, 1)) / R
    return ctrl


def _triangles(n, R, rng, size):
    v = np.zeros((n, 3, 4), np.float32)
    v[..., :3] = rng.uniform(0.0, 1.0, (n, 1, 3)) + rng.uniform(-0.5, 0.5, (n, 3, 3)) * (rng.uniform(*size, n) / R)[:, None, None]
    return v


def _geom(kind, prims, weights):
    t = torch.from_numpy(np.ascontiguousarray(prims)).to(DEV)
    w = torch.from_numpy(weights).to(DEV)
    if kind == "triangles":
        return dict(tri_verts=t, weights=w)
    return dict(ctrl=t.reshape(-1, 4), fiber_offsets=torch.arange(prims.shape[0] + 1, device=DEV) * 2, weights=w)


def _level_gradients(keys, levels, rng):
    gm, gM = [], []
    for l in range(levels + 1):
        n = int(torch.unique_consecutive(keys >> (3 * l)).numel())
        gm.append(torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).to(DEV))
        gM.append(torch.from_numpy(rng.uniform(-1, 1, (n, 6)).astype(np.float32)).to(DEV))
    return gm, gM


def _rows(kind, g):
    return g[0].reshape(-1, 12 if kind == "triangles" else 8).double(), g[1].double()


@pytest.mark.parametrize("kind,n,R,size", [
    ("fibers", 77824, 64, (0.1, 9.0)),      # one lane per segment: uneven walks, so uneven queues
    ("fibers", 80001, 16, (0.01, 1.5)),
    ("triangles", 77824, 64, (0.1, 6.0)),
    ("triangles", 80001, 16, (0.01, 1.5)),
])
def test_one_lane_per_primitive(kind, n, R, size):
    """Every primitive's gradients, against those of arrays of 2,000.  Both add the same FP64 terms, in
    orders that differ, and round once to FP32 (2^-24 of the value); the terms of one primitive cancel by
    far less than the 2^29 between the two precisions."""
    rng = np.random.default_rng(n + R)
    prims = _segments(n, R, rng, size) if kind == "fibers" else _triangles(n, R, rng, size)
    weights = rng.uniform(0.5, 2.0, n).astype(np.float32)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    geom = _geom(kind, prims, weights)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    gm, gM = _level_gradients(keys, 3, rng)
    whole = _rows(kind, ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **geom))
    parts = []
    for b in range(0, n, 2000):
        part = _geom(kind, prims[b:b + 2000], weights[b:b + 2000])
        parts.append(_rows(kind, ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **part)))
    for got, ref in zip(whole, [torch.cat(x) for x in zip(*parts)]):
        size = ref.abs().reshape(n, -1).amax(1).reshape(n, *[1] * (ref.dim() - 1))
        assert bool(((got - ref).abs() <= 2.0 ** -23 * size).all())
        assert int((size > 0).sum()) > n // 2
    ctx.close()


def _with_large(kind, n, R, rng, extent, count, at):
    """Small primitives with `count` large ones (`extent` voxels long or wide) from place `at`."""
    prims = _segments(n, R, rng, (0.1, 2.0)) if kind == "fibers" else _triangles(n, R, rng, (0.1, 2.0))
    lo, hi = extent / 2 / R + 0.01, 1.0 - extent / 2 / R - 0.01
    c = rng.uniform(lo, hi, (count, 3))
    h = rng.uniform(-0.5, 0.5, (count, 3, 3)) * extent / R
    h[:, 0], h[:, 1] = -0.5 * extent / R, 0.5 * extent / R
    prims[at:at + count, :, :3] = c[:, None, :] + h[:, :prims.shape[1]]
    return prims


@pytest.mark.parametrize("kind,n,extent,count,at", [
    ("fibers", 77824, 100.0, 40, 100),          # above 64 slabs, in a row, across two warps
    ("fibers", 30000, 63.5, 33, 29967),         # about 64 slabs; the last, short group
    ("triangles", 77824, 40.0, 40, 100),
    ("triangles", 20000, 13.0, 33, 19967),      # about 2,048 voxels
])
def test_large_among_small(kind, n, extent, count, at):
    """As above with primitives whose walk is left to a second launch."""
    R = 128
    rng = np.random.default_rng(n + 1)
    prims = _with_large(kind, n, R, rng, extent, count, at)
    weights = rng.uniform(0.5, 2.0, n).astype(np.float32)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    geom = _geom(kind, prims, weights)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    gm, gM = _level_gradients(keys, 4, rng)
    whole = _rows(kind, ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **geom))
    for b in (at, max(0, at - 1900), 0):
        part = _geom(kind, prims[b:b + 2000], weights[b:b + 2000])
        ref = _rows(kind, ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **part))
        for got, r in zip(whole, ref):
            m = r.shape[0]
            size = r.abs().reshape(m, -1).amax(1).reshape(m, *[1] * (r.dim() - 1))
            assert bool(((got[b:b + m] - r).abs() <= 2.0 ** -23 * size).all())
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


@pytest.mark.parametrize("kind,extent", [("fibers", 200.0), ("triangles", 100.0)])
def test_large_ones_do_not_wait_for_one_lane(kind, extent):
    """90,000 small primitives and 32 large ones take about as long as the two apart (one lane on a large
    triangle took 32 times as long as its warp)."""
    R, n, count = 256, 90000, 32
    rng = np.random.default_rng(3)
    prims = _with_large(kind, n, R, rng, extent, count, 500)
    weights = np.ones(n, np.float32)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    geom = _geom(kind, prims, weights)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    gm, gM = _level_gradients(keys, 0, rng)
    few = slice(500, 500 + count)
    rest = np.concatenate([prims[:500], prims[500 + count:]])
    times = [_time(lambda g=g: ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **g))
             for g in (geom, _geom(kind, rest, weights[count:]), _geom(kind, prims[few], weights[few]))]
    print(kind, times)
    assert times[0] < 2.0 * (times[1] + times[2])
    ctx.close()
