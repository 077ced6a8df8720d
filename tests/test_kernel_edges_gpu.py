"""Kernels at the sizes and positions where their fast paths hand over to the definition, against
the CPU oracle.  Whole numbers and FP32 sums are compared bit for bit."""
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


def _same_level0(got, ref):
    g = got.host()
    for f, r in (("keys", "keys"), ("mask", "mask"), ("occ", "occ"), ("proj", "proj")):
        assert np.array_equal(g[f], ref[r]), f
    for f in ("mass", "moment"):
        assert np.array_equal(g[f].view(np.uint32), ref[f].view(np.uint32)), f


@pytest.mark.parametrize("n,R,size,snap", [
    (1, 8, (0.5, 0.5), 0),          # one triangle
    (300, 16, (0.2, 3.0), 8),       # vertices on sub-cell planes: every axis test at its boundary
    (300, 16, (0.2, 3.0), 16),      # vertices on sub-cell centres
    (60, 64, (8.0, 40.0), 8),       # triangles many voxels wide
    (400, 32, (0.001, 0.1), 0),     # far smaller than a sub-cell
    (900, 4, (0.3, 1.0), 0),        # voxels of several batches of 32 triangles
    (120, 4, (0.2, 0.5), 2),        # groups of voxels at the edge of 32, vertices on voxel planes
])
def test_triangle_masks_at_the_boundaries(n, R, size, snap):
    tris, grid = synth.random_triangles(n, R, seed=100 + n + R, size=size)
    if snap:
        tris[..., :3] = np.round(tris[..., :3] * (R * snap)) / (R * snap)
    tris[n // 2] = tris[n // 2, :1]                       # a triangle without area
    rng = np.random.default_rng(n)
    w = synth.Workload("tris", "triangles", grid, tri_verts=tris, K=1,
                       weights=rng.uniform(0.5, 2.0, n).astype(np.float32))
    ctx = vx.Context(DEV)
    got = ctx.voxelize(grid, tri_verts=torch.from_numpy(tris).to(DEV), weights=torch.from_numpy(w.weights).to(DEV))
    _same_level0(got, oracle.voxelize(w))
    ctx.close()


@pytest.mark.parametrize("n_fibers,pts,R,radius,step,snap", [
    (1, 2, 8, (0.3, 0.3), (0.5, 0.5), 0),         # one capsule
    (40, 20, 16, (0.4, 1.5), (0.1, 2.0), 8),      # ends on sub-cell planes
    (40, 20, 32, (2.0, 4.0), (0.1, 0.5), 0),      # radius of several voxels: covered voxels
    (60, 12, 16, (0.02, 0.2), (2.0, 9.0), 0),     # long and thin: most sub-cells go to step 3
    (30, 30, 4, (0.1, 0.4), (0.05, 0.4), 0),      # voxels of several batches of 32 capsules
    (20, 6, 64, (0.3, 0.9), (20.0, 60.0), 4),     # tens of voxels long, ends on sub-cell corners
    (25, 20, 8, (0.125, 0.125), (0.125, 0.5), 8), # radius and steps of whole sub-cells
])
def test_capsule_masks_at_the_boundaries(n_fibers, pts, R, radius, step, snap):
    ctrl, off, grid = synth.random_segments(n_fibers, pts, R, seed=300 + n_fibers + R, radius=radius, step=step)
    if snap:
        ctrl[:, :3] = np.round(ctrl[:, :3] * (R * snap)) / (R * snap)
    ctrl[1, :3] = ctrl[0, :3]                             # a segment without length
    rng = np.random.default_rng(n_fibers)
    n = synth.fiber_segment_count(off)
    w = synth.Workload("caps", "fibers", grid, ctrl=ctrl, fiber_offsets=off, K=1,
                       weights=rng.uniform(0.0, 2.0, n).astype(np.float32))
    ctx = vx.Context(DEV)
    got = ctx.voxelize(grid, ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV),
                       weights=torch.from_numpy(w.weights).to(DEV))
    _same_level0(got, oracle.voxelize(w))
    ctx.close()
