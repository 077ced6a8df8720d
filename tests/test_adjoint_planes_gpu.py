"""The adjoint where primitives meet voxel planes exactly: coordinates on planes, negative zeros."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2604_13191_gb300 as vx  # noqa: E402

DEV = torch.device("cuda", 0)


def _loss(keys, seed):
    rng = np.random.default_rng(seed)
    n = keys.shape[0]
    return (torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).to(DEV),
            torch.from_numpy(rng.uniform(-1, 1, (n, 6)).astype(np.float32)).to(DEV))


def _geom(kind, p, weights):
    t = torch.from_numpy(np.ascontiguousarray(p)).to(DEV)
    w = torch.from_numpy(weights).to(DEV)
    if kind == "triangles":
        return dict(tri_verts=t, weights=w)
    return dict(ctrl=t.reshape(-1, 4), fiber_offsets=torch.arange(p.shape[0] + 1, device=DEV) * 2, weights=w)


def _snapped(kind, n, R, snap, extent, seed, lo=0.0):
    """n primitives with coordinates that are multiples of 1 / snap voxels, from `lo` voxels on."""
    rng = np.random.default_rng(seed)
    k = 3 if kind == "triangles" else 2
    p = rng.uniform(lo, R - 1.0, (n, 1, 3)) + rng.uniform(-0.5, 0.5, (n, k, 3)) * extent
    out = np.zeros((n, k, 4), np.float32)
    out[..., :3] = np.round(p * snap) / snap / R
    if kind == "fibers":
        out[..., 3] = 0.3 / R
    return out, rng.uniform(0.5, 2.0, n).astype(np.float32)


@pytest.mark.parametrize("kind", ["triangles", "fibers"])
@pytest.mark.parametrize("snap", [1, 2, 8])
def test_negative_zeros(kind, snap):
    """A coordinate of -0 is one of +0 (the grid begins at 0, so both lie on its first planes)."""
    R, n = 8, 3000
    p, w = _snapped(kind, n, R, snap, 5.0, snap, lo=-2.0)
    neg = p.copy()
    neg[p == 0.0] = -0.0
    assert int((p[..., :3] == 0.0).sum()) > 100
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    keys = ctx.voxelize(grid, **_geom(kind, p, w)).keys.clone()
    gm, gM = _loss(keys, 3)
    got = []
    for x in (p, neg):
        g, gw = ctx.backward(grid, keys0=keys, grad_mass=[gm], grad_moment=[gM], **_geom(kind, x, w))
        got.append((g.cpu().numpy(), gw.cpu().numpy()))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0], got[1][0], equal_nan=True)
    ctx.close()
