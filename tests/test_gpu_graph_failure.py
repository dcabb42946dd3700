"""A longer step graph that cannot be recorded (no memory for it, say) is done without: the run goes on with
the shorter ones, with the same bits and no error.  The failure comes from a build of the library in which
cudaGraphInstantiate refuses graphs of more than a given number of nodes."""
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
#define cudaGraphInstantiate refuse_long
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
    """A copy of the package whose library refuses long graphs."""
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


def _run(path, particles, steps, most=None):
    env = dict(os.environ, PYTHONPATH=path)
    if most:
        env["MOST_GRAPH_NODES"] = str(most)
    r = subprocess.run([sys.executable, "-c", CHILD, str(particles), steps], env=env, cwd=path, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout.split()


# fluid alone: 3, 9 and 33 nodes in graphs of 2, 8 and 32 steps; with particles 11, 41 and 161
@pytest.mark.parametrize("particles,steps,most", [(0, "200,31", 5), (0, "4300,64", 20), (50, "170,20", 20),
                                                  (50, "4200,7", 100)])
def test_run_goes_on_with_shorter_graphs(refusing, particles, steps, most):
    got = _run(refusing, particles, steps, most)
    assert got == _run(ROOT, particles, steps)
    assert got[0] == str(sum(int(n) for n in steps.split(",")))
