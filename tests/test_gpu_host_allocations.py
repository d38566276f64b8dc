"""The calls that promise to allocate nothing allocate no host memory either: a counting operator new
in front of the C++ library's, loaded by a process of its own before the CUDA library."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COUNTER = """
#include <atomic>
#include <cstdlib>
#include <new>
static std::atomic<long long> n{0};
void* operator new(std::size_t b) {
    ++n;
    if (void* p = std::malloc(b ? b : 1)) return p;
    throw std::bad_alloc();
}
void* operator new[](std::size_t b) { return operator new(b); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
void operator delete[](void* p, std::size_t) noexcept { std::free(p); }
extern "C" long long news() { return n.load(); }
"""

PROGRAM = """
import ctypes, json, sys
count = ctypes.CDLL(sys.argv[1], ctypes.RTLD_GLOBAL).news
count.restype = ctypes.c_longlong
import numpy as np, torch
import synth
from paper_2104_03989_gb300 import binding as B
from paper_2104_03989_gb300 import stages as ST

p, tri = synth.icosphere(3)
uv, tri_uv = synth.equirect_uv_corners(p, tri)
W, H = 64, 48
views = synth.sample_views(1, 0, 2, W, H)
pipe = ST.Pipeline(tri, uv, tri_uv, len(p), views, H, W)
pos = torch.tensor(p.astype(np.float32), device="cuda")
mesh, clip = pipe.mesh(pos), pipe.empty(2, pipe.V, 4)
keys, rast, db = pipe.empty(2, H, W, dtype=torch.int64), pipe.empty(2, H, W, 2), pipe.empty(2, H, W, 4)
tri32 = torch.tensor(np.ascontiguousarray(tri, dtype=np.int32), device="cuda")
calls = {
    "counts": lambda: B.adms_mesh_topology(np.ascontiguousarray(tri, dtype=np.int32), len(p)),
    "setup": lambda: B.adms_setup_fwd(mesh, pipe.views, 2, H, W, clip, pipe.work),
    "raster": lambda: B.adms_raster_fwd(mesh, pipe.views, 2, H, W, clip, keys, rast, db, pipe.work),
    "noalloc": lambda: B.adms_visibility_noalloc(pos, tri32, pipe.views, 2, H, W, keys, None),
}
out = {}
for name, call in calls.items():
    call()
    seen = []
    for _ in range(5):  # the least of several: other threads of the process may allocate meanwhile
        before = count()
        call()
        seen.append(count() - before)
    out[name] = min(seen)
torch.cuda.synchronize()
print(json.dumps(out))
"""


def test_calls_without_device_allocations_make_none_on_the_host(gpu_lib, tmp_path):
    src, lib = tmp_path / "count.cpp", tmp_path / "libcount.so"
    src.write_text(COUNTER)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out.pop("counts") > 0  # a call that does allocate is seen to
    assert out == {"setup": 0, "raster": 0, "noalloc": 0}
