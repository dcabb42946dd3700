"""What is only faster is done without where the device has no room for it: a longer step graph that cannot
be recorded (the shorter ones go on, with the same bits), the partial sums of the one-pass update (two
passes), also where particles find no room beside them later.  The failures come from a build of the library in
which cudaGraphInstantiate or cudaGraphLaunch refuses graphs of more than a given number of nodes and cudaMalloc, while the
environment says so, every allocation or those past a number of bytes in all."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

REFUSE = r"""
#include <cuda_runtime.h>
#include <cstdlib>
#include <map>
static std::map<cudaGraphExec_t, size_t> nodes;
static inline cudaError_t refuse_long(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long flags) {
  size_t n = 0;
  cudaGraphGetNodes(g, nullptr, &n);
  const char *most = std::getenv("MOST_GRAPH_NODES");
  if (most && n > (size_t)std::atol(most)) return cudaErrorMemoryAllocation;
  const cudaError_t e = cudaGraphInstantiate(x, g, flags);
  if (e == cudaSuccess) nodes[*x] = n;
  return e;
}
static inline cudaError_t refuse_launch(cudaGraphExec_t x, cudaStream_t st) {
  const char *most = std::getenv("MOST_LAUNCHED_NODES");
  return most && nodes[x] > (size_t)std::atol(most) ? cudaErrorMemoryAllocation : cudaGraphLaunch(x, st);
}
static std::map<void *, size_t> held;
static size_t total = 0;
extern "C" size_t bytes_held() { return total; }
static inline cudaError_t refuse_malloc(void **p, size_t n) {
  const char *most = std::getenv("MOST_BYTES");
  if (std::getenv("REFUSE_MALLOC") || (most && total + n > (size_t)std::atoll(most)))
    return cudaMalloc(p, (size_t)1 << 60);  // as no memory: the last error is set
  const cudaError_t e = cudaMalloc(p, n);
  if (e == cudaSuccess) total += held[*p] = n;
  return e;
}
static inline cudaError_t counted_free(void *p) {
  total -= held[p];
  held.erase(p);
  return cudaFree(p);
}
#define cudaGraphInstantiate refuse_long
#define cudaGraphLaunch refuse_launch
#define cudaMalloc refuse_malloc
#define cudaFree counted_free
"""

CHILD = r"""
import hashlib, sys
import numpy as np
from paper_1306_0788_gb300 import lbmd as L
particles, steps = int(sys.argv[1]), [int(n) for n in sys.argv[2].split(",")]
rng = np.random.default_rng(1)
dims = (24, 20, 22)
ctx, _ = L.lbmd_create(L.params(dims, g_AB=0.8))
L.lbmd_set_types(ctx, [L.lbmd_ptype(0.0, 0.0, 0.0, 0.0, 1.0, 200.0)])
L.lbmd_init_fluid(ctx, *(rng.uniform(0.95, 1.05, dims[::-1]).astype(np.float32) for _ in range(2)))
L.lbmd_set_particles(ctx, rng.uniform(0, 1, (particles, 3)) * dims, np.zeros((particles, 3)),
                     np.zeros(particles, dtype=np.int32))
for n in steps:
    L.lbmd_step(ctx, n)
L.lbmd_sync(ctx)
f = [L.lbmd_get_populations(ctx, k, dims[::-1]) for k in range(2)]
assert all(np.isfinite(x).all() for x in f)
print(L.lbmd_step_count(ctx), L.lbmd_last_error(ctx) or "-",
      hashlib.sha256(b"".join(x.tobytes() for x in f + list(L.lbmd_get_particles(ctx, particles)))).hexdigest())
"""


@pytest.fixture(scope="module")
def refusing(tmp_path_factory):
    """A copy of the package with that library."""
    from paper_1306_0788_gb300 import build
    build.build()
    top = tmp_path_factory.mktemp("refusing")
    package = top / "paper_1306_0788_gb300"
    package.mkdir()
    for f in os.listdir(build.HERE):
        if f.endswith(".py"):
            shutil.copy(os.path.join(build.HERE, f), package)
    header = top / "refuse.h"
    header.write_text(REFUSE)
    obj = str(top / "lbmd_api.o")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-include", str(header), "-I", build.INCLUDE, "-I", build.CSRC,
                    "-c", os.path.join(build.CSRC, "lbmd_api.cu"), "-o", obj], check=True)
    others = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()
              if not s.endswith("lbmd_api.cu")]
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-cudart", "static", "-o", str(package / "liblbmd.so"), obj,
                    *others], check=True)
    return str(top)


def _child(path, code, *args, **env):
    r = subprocess.run([sys.executable, "-c", code, *args], env=dict(os.environ, PYTHONPATH=path, **env), cwd=path,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout.split()


def _run(path, particles, steps, **env):
    return _child(path, CHILD, str(particles), steps, **env)


# fluid alone: 3, 9 and 33 nodes in graphs of 2, 8 and 32 steps; with particles 11, 41 and 161
@pytest.mark.parametrize("particles,steps,most", [(0, "200,31", 5), (0, "4300,64", 20), (50, "170,20", 20),
                                                  (50, "4200,7", 100)])
@pytest.mark.parametrize("call", ["MOST_GRAPH_NODES", "MOST_LAUNCHED_NODES"])
def test_run_goes_on_with_shorter_graphs(refusing, particles, steps, most, call):
    got = _run(refusing, particles, steps, **{call: str(most)})
    assert got == _run(ROOT, particles, steps)
    assert got[0] == str(sum(int(n) for n in steps.split(",")))


NO_ROOM = r"""
import os
import numpy as np
from paper_1306_0788_gb300 import lbmd as L
rng = np.random.default_rng(1)
dims = (160, 160, 160)
rho = [rng.uniform(0.95, 1.05, dims[::-1]).astype(np.float32) for _ in range(2)]
mrt = dict(g_AB=0.8, kT=1e-5, collision=L.LBMD_COLLISION_MRT)

def steps(ctx, n):
    L.lbmd_init_fluid(ctx, *rho)
    L.lbmd_step(ctx, n)
    return [L.lbmd_get_populations(ctx, k, dims[::-1]) for k in range(2)]

ctx, _ = L.lbmd_create(L.params(dims, **mrt))
L.lbmd_set_graphs(ctx, False)
L.lbmd_init_fluid(ctx, *rho)
os.environ["REFUSE_MALLOC"] = "1"
assert L.lbmd_get_lattice_passes(ctx) == 2
without = steps(ctx, 3)
del os.environ["REFUSE_MALLOC"]
assert L.lbmd_get_lattice_passes(ctx) == 2
L.lbmd_set_lattice_passes(ctx, 2)
assert all(np.array_equal(a, b) for a, b in zip(without, steps(ctx, 3)))
L.lbmd_set_lattice_passes(ctx, 0)
assert L.lbmd_get_lattice_passes(ctx) == 1
steps(ctx, 3)
L.lbmd_sync(ctx)
print("done")
"""


def test_two_passes_where_there_is_no_room_for_the_partial_sums(refusing):
    assert _child(refusing, NO_ROOM) == ["done"]


NO_ROOM_BESIDE = r"""
import ctypes, os
import numpy as np
from paper_1306_0788_gb300 import lbmd as L
held = L._lib.bytes_held
held.restype = ctypes.c_size_t
rng = np.random.default_rng(1)
dims, n = (160, 160, 160), 20000
rho = [rng.uniform(0.95, 1.05, dims[::-1]).astype(np.float32) for _ in range(2)]
x = rng.uniform(0, 160, (n, 3))

def context():
    ctx, _ = L.lbmd_create(L.params(dims, g_AB=0.8, kT=1e-5, collision=L.LBMD_COLLISION_MRT))
    L.lbmd_set_types(ctx, [L.lbmd_ptype(0.0, 0.0, 0.0, 0.0, 0.1, 200.0)])
    L.lbmd_init_fluid(ctx, *rho)
    return ctx

def with_particles(ctx):
    before = held()
    L.lbmd_set_particles(ctx, x, np.zeros_like(x), np.zeros(n, dtype=np.int32))
    return held() - before

def steps(ctx):
    L.lbmd_init_fluid(ctx, *rho)
    L.lbmd_step(ctx, 3)
    return [L.lbmd_get_populations(ctx, k, dims[::-1]) for k in range(2)] + list(L.lbmd_get_particles(ctx, n))

two = context()
L.lbmd_set_lattice_passes(two, 2)
size = with_particles(two)
want = steps(two)
L.lbmd_destroy(two)
for short in (1, size // 2, size):  # rows, then particle arrays, find no room
    ctx = context()
    L.lbmd_step(ctx, 2)
    assert L.lbmd_get_lattice_passes(ctx) == 1
    os.environ["MOST_BYTES"] = str(held() + size - short)
    with_particles(ctx)
    del os.environ["MOST_BYTES"]
    assert L.lbmd_get_lattice_passes(ctx) == 2
    assert all(np.array_equal(a, b) for a, b in zip(want, steps(ctx)))
    L.lbmd_destroy(ctx)
print("done")
"""


def test_particles_take_the_room_of_the_partial_sums(refusing):
    assert _child(refusing, NO_ROOM_BESIDE) == ["done"]
