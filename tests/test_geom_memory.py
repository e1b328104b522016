"""The safety lists of a geometry are an accelerator: a geometry for which they find no device memory
is created without them, and they are bounded.  Runs against a stand-in for the CUDA runtime's
allocation, copy and launch calls (preloaded into a child process, so that no GPU is used): its
cudaMalloc refuses requests above a limit and reports the largest one it granted."""
import os
import shutil
import subprocess
import sys

import pytest

import __graft_entry__
import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
static size_t largest = 0, refused = 0;
size_t shim_largest(void) { return largest; }
size_t shim_refused(void) { return refused; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaMalloc(void** p, size_t n) {
  const char* l = getenv("SHIM_LIMIT");
  if (l && n > strtoull(l, 0, 10)) { refused++; return 2; }
  if (n > largest) largest = n;
  *p = malloc(n < (1u << 20) ? n : (1u << 20));  /* the large ones are written by kernels only */
  return 0;
}
int cudaFree(void* p) { free(p); return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; if (n <= (1u << 20)) memcpy(d, s, n); return 0; }
int cudaGetLastError(void) { return 0; }
int cudaStreamSynchronize(void* s) { (void)s; return 0; }
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void) { return 0; }
int cudaLaunchKernel(void) { return 0; }
"""
CHILD = """
import ctypes, sys
import workloads as W
import paper_1512_06637_gb300 as gv
shim = ctypes.CDLL(sys.argv[1])
shim.shim_largest.restype = shim.shim_refused.restype = ctypes.c_size_t
geo = W.crowded_geometry(int(sys.argv[2]))
parts = int(sys.argv[3])
world = {"solid": 0, "parent": -1, "R": geo["nodes"][0]["R"], "t": geo["nodes"][0]["t"]}
nodes = list(geo["nodes"])
for k in range(1, parts):  # more volumes like the world inside it
    at = len(nodes)
    nodes.append(dict(world, parent=0))
    nodes += [dict(d, parent=at) for d in geo["nodes"][1:] if d["parent"] == 0]
G = gv.Geometry(geo["solids"], nodes)
print(G.voxel_count, shim.shim_largest(), shim.shim_refused())
"""


def _create(tmp_path, lattice, parts, limit=None):
    so = str(tmp_path / "shim.so")
    src = tmp_path / "shim.c"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", str(src), "-o", so], check=True)
    env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
    env.pop("SHIM_LIMIT", None)
    if limit is not None:
        env["SHIM_LIMIT"] = str(limit)
    r = subprocess.run([sys.executable, "-c", CHILD, so, str(lattice), str(parts)], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return [int(v) for v in r.stdout.split()]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no CUDA toolkit")
    __graft_entry__.build()


def test_geometry_without_memory_for_safety_lists(tmp_path):
    # lattice 10: 1000 daughters and at least as many cells of 512 bytes; every other table is below 400 kB
    grids, largest, refused = _create(tmp_path, 10, 1, limit=400_000)
    assert grids >= 1 and refused == 1 and largest <= 400_000


def test_safety_lists_are_bounded(tmp_path):
    # 400 volumes of 1000 daughters: lists for all of them would take more than 200 MB
    grids, largest, _ = _create(tmp_path, 10, 400)
    assert grids >= 400
    assert largest <= (1 << 18) * 512
