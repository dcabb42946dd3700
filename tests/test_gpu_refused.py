"""What is only faster is done without where the device has no room for it: a longer step graph that cannot
be recorded (the shorter ones go on, with the same bits), the partial sums of the one-pass update (two
passes).  The failures come from a build of the library in which cudaGraphInstantiate refuses graphs of more
than a given number of nodes and cudaMalloc, while the environment says so, every allocation."""
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
static inline cudaError_t refuse_long(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long flags) {
  size_t n = 0;
  cudaGraphGetNodes(g, nullptr, &n);
  const char *most = std::getenv("MOST_GRAPH_NODES");
  return most && n > (size_t)std::atol(most) ? cudaErrorMemoryAllocation : cudaGraphInstantiate(x, g, flags);
}
static inline cudaError_t refuse_malloc(void **p, size_t n) {
  return cudaMalloc(p, std::getenv("REFUSE_MALLOC") ? (size_t)1 << 60 : n);  // (as no memory: the last error is set)
}
#define cudaGraphInstantiate refuse_long
#define cudaMalloc refuse_malloc
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
def test_run_goes_on_with_shorter_graphs(refusing, particles, steps, most):
    got = _run(refusing, particles, steps, MOST_GRAPH_NODES=str(most))
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
