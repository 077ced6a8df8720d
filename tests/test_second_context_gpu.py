"""Two CUDA contexts in one process: what the library sets up for its kernels belongs to the device and the
CUDA context, as on a second GPU, and is set up again in the second one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import ctypes as C
import numpy as np
from paper_2604_13191_gb300 import api

lib = api.load()
cu = C.CDLL("libcuda.so.1")

def drv(name, *args):
    r = getattr(cu, name)(*args)
    assert r == 0, (name, r)

def upload(a):
    p = C.c_void_p()
    drv("cuMemAlloc_v2", C.byref(p), C.c_size_t(a.nbytes))
    drv("cuMemcpyHtoD_v2", p, C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes))
    return p.value

def voxelize(R):
    rng = np.random.default_rng(1)
    tris = np.zeros((4000, 3, 4), np.float32)
    tris[..., :3] = rng.uniform(0.1, 0.9, (4000, 1, 3)) + rng.uniform(-0.5, 0.5, (4000, 3, 3)) * 2.0 / R
    P, G, L, h = api.VxPrimitives(), api.VxGrid(), api.VxLevel(), C.c_void_p()
    P.kind, P.num_prims, P.tri_verts = api.VX_TRIANGLES, 4000, upload(tris)
    G.voxel_size, G.resolution, G.sub_res = 1.0 / R, R, 8
    assert lib.vx_context_create(None, C.byref(h)) == 0
    st = lib.vx_voxelize(h, C.byref(P), C.byref(G), None, C.byref(L))
    assert st == 0, (st, R)
    drv("cuCtxSynchronize")
    keys = np.empty(L.num_voxels, np.uint64)
    drv("cuMemcpyDtoH_v2", C.c_void_p(keys.ctypes.data), C.c_uint64(L.keys), C.c_size_t(keys.nbytes))
    lib.vx_context_destroy(h)
    return keys

drv("cuInit", 0)
dev = C.c_int()
drv("cuDeviceGet", C.byref(dev), 0)
runs = []
for _ in range(2):
    ctx = C.c_void_p()
    drv("cuCtxCreate_v2", C.byref(ctx), 0, dev)
    runs.append([voxelize(R) for R in (64, 256)])     # key digits of 9 bits and of 8
for a, b in zip(*runs):
    assert a.size > 4000 and np.array_equal(a, b)
print("same")
"""


def test_second_cuda_context():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]
