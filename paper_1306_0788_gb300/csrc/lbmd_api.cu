// lbmd_api.cu -- the C ABI (include/lbmd.h): context, device memory, argument checks and the
// launch sequence of one coupled step.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "lbmd_internal.cuh"

using namespace lbmd;

namespace {
// Replayed graphs hold an even number of steps (both buffer pairs return to their start), of three
// lengths.  A replay costs about 5 us between one graph and the next: of 50 steps of 32^3 with 64
// particles 702 us with graphs of two steps, 579 of ten, 556 of fifty; of 45x37x29 fluid only 468,
// 356, 337; of 64^3 with 1000 particles 1273, 1122, 1092.  Recording takes 6 us per step of fluid
// alone and about 35 with particles (0.2 and 1.3 ms for 32 steps), so the longer graphs are recorded
// once a context has replayed as many steps as make up for it with particles: 8 steps save about 2.2 us a
// step, 280 us in 128 steps, 32 steps 0.4, 1.5 ms in 4096.  (Fluid alone would make up for it in about 22 and
// 500 steps.)
constexpr int kGraphLevels = 3;
constexpr int kGraphSteps[kGraphLevels] = {2, 8, 32};
constexpr int64_t kGraphAfter[kGraphLevels] = {0, 128, 4096};  // steps replayed since the last setter
constexpr int kShortGraph = kGraphSteps[0];

// A recorded sequence of coupled steps (lbmd_set_graphs).
struct StepGraph {
  cudaGraph_t graph = nullptr;  // kept for the event nodes' handles
  cudaGraphExec_t exec = nullptr;
  int64_t launches = 0;                            // kernels per replay
  cudaGraphNode_t ev_node[2 * kShortGraph] = {};  // k_collide timing events, retargeted per replay
  // the noisy MRT update of each step: its node and the counter offset it was recorded with
  // (its counter is patched per replay; see is_noisy_update)
  struct Update {
    cudaGraphNode_t node;
    unsigned long long off;
  };
  std::vector<Update> updates;
};
// What recording a graph returns where the steps can be taken without it: one by one, or by shorter graphs.
constexpr int kGraphUnavailable = 1, kGraphShorter = 2;
}  // namespace

struct lbmd_ctx {
  lbmd_params prm{};
  cudaStream_t st = nullptr;
  // the particle sort and the pair forces depend on the particles only, so they run on a side
  // stream: the pair forces beside the coupling; then, waiting for the coupling (ev_coupled), the
  // particle update and the sort of the updated particles for the next step, beside the lattice
  // update.  The sort writes the buffers of the step before (pa[1 - pcur], row_start[1 - pcur]),
  // whose last reader, that step's lattice update, the coupling came after.  st waits for the sort
  // (ev_sorted) at the end of a launch sequence or before the next coupling; sort_pending: it has
  // not yet.  ev_int forks side from st; with MD sub-stepping the substeps run on st, and the sort of
  // the particles starts when the substeps and the sort of their records are done (ev_sub).
  cudaStream_t side = nullptr;
  cudaEvent_t ev_int = nullptr, ev_sorted = nullptr, ev_coupled = nullptr, ev_sub = nullptr;
  bool sort_pending = false;
  bool onepass_no_room = false;  // the automatic choice found no device memory for the one-pass update
  // one pass with particles: the next step's corner j' (jc) is formed on side, at the sorted updated
  // particles, once the lattice update is done (ev_collided), beside the boundary densities on st
  cudaEvent_t ev_collided = nullptr;
  // the device-memory getters: the caller's stream's queued work before their writes (dev_in),
  // and their writes before what the caller queues next (dev_out); created on first use
  cudaEvent_t ev_dev_in = nullptr, ev_dev_out = nullptr;
  int dev = 0;
  StepParams P{};
  unsigned char *pop[2] = {nullptr, nullptr};  // population buffers, element type P.storage
  size_t pop_elem = 4;
  // 16-bit storage: FP32 rest populations [2][N], those of pop[cur] in rest[cur]; the same array twice
  // (they are local to a node) except on small lattices, whose update may read its neighbours' too
  float *rest[2] = {nullptr, nullptr};
  int cur = 0;
  // [N][2] interleaved rho_A, rho_B: rho_buf[cur] holds the densities of pop[cur] while
  // rho_valid (after init_fluid, set_populations and one-pass steps; the two-pass update
  // recomputes them at the start of its step)
  float *rho_buf[2] = {nullptr, nullptr};
  bool rho_valid = false;
  float *jp = nullptr;   // [3][N]
  // [cap][8] j' at the corners of each particle's cell (by particle id), for the coupling of the
  // one-pass update; jc_valid: formed from the current populations and positions
  float4 *jc = nullptr;
  bool jc_valid = false;
  // the lattice update: 0 = chosen by the lattice size, 1 = one pass (densities of the next step
  // formed by the update), 2 = two passes (density pass, then the update)
  int passes = 0;
  OnePassGeom op_geom{};
  int op_grid = 0;
  BoundaryRun *op_runs = nullptr;
  int op_nruns = 0;
  OnePassOut op_out{};     // partial sums (all buffers owned by the context)
  int *op_zslot = nullptr;  // [nz]: -1, or the chunk-edge plane's slot in op_out's z arrays
  // particles
  int np = 0, cap = 0;
  // pa[pcur], row_start[pcur]: the sorted particles of the current state; the other pair takes the
  // next step's; pt: the updated particles before their sort (in the order they had been in)
  ParticleArrays pa[2]{}, pt{};
  int pcur = 0;
  ParticleForces pf{};
  int *slot_of_id = nullptr;
  int *row_start[2] = {nullptr, nullptr};
  // CellIndex::node_bits: [b] those of pa[b] (with MD sub-stepping [0] those of the records, formed
  // anew each step)
  unsigned *node_bits[2] = {nullptr, nullptr};
  SortScratch sort{};
  int *bond_start = nullptr, *bond_other = nullptr;
  int nbonds = 0, bond_np = 0;  // bonds index particles 0..bond_np-1
  // MD sub-stepping: momentum-return records per (substep, particle), unsorted and sorted
  ReactionRecords rec[2]{};
  SortScratch rec_sort{};  // its counters are sort's
  int *rec_row_start = nullptr;
  long long rec_cap = 0;
  unsigned *err = nullptr;
  double *diag_partial = nullptr, *diag_out = nullptr;
  int diag_blocks = 0;
  // the FP64 drift check: reference totals [M_A, M_B, Px, Py, Pz] and the last check's
  // {step, drift A, drift B, momentum drift, checks} (device memory, 10 doubles)
  double *drift = nullptr;
  int64_t steps = 0, launches = 0;
  bool fluid_ready = false, types_set = false;
  unsigned sticky = 0;
  std::string msg;
  bool prof = false;
  std::vector<cudaEvent_t> ev;  // pairs (start, stop)
  size_t ev_used = 0;
  double prof_ms = 0.0;
  int64_t prof_launches = 0;
  // replayed step graphs: recorded on gst (never on the caller's stream, which may carry other
  // work), one per length and parity of (cur, pcur) at the replay's start, launched into st; the kernels
  // read their noise counter's base from step_base, which holds dev_step once the work
  // enqueued so far has run (-1: not known)
  bool graphs = true;
  cudaStream_t gst = nullptr;
  StepGraph graph[kGraphLevels][2][2];
  int64_t replayed = 0;  // steps replayed since the graphs were dropped
  int graph_levels = kGraphLevels;  // lengths in use: those past it could not be recorded
  unsigned long long *step_base = nullptr;
  int64_t dev_step = -1;
  cudaEvent_t ph[2 * kShortGraph] = {};  // stand-ins for the timing events while recording
};

namespace {

thread_local std::string g_create_error;

int fail(lbmd_ctx *c, int code, const std::string &m) {
  if (c)
    c->msg = m;
  else
    g_create_error = m;
  return code;
}

int cuda_fail(lbmd_ctx *c, cudaError_t e, const char *where) {
  return fail(c, LBMD_E_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define CK(call, where)                          \
  do {                                           \
    cudaError_t e_ = (call);                     \
    if (e_ != cudaSuccess) return cuda_fail(c, e_, where); \
  } while (0)

template <class T>
cudaError_t dalloc(T **p, size_t n) {
  *p = nullptr;
  if (n == 0) return cudaSuccess;
  return cudaMalloc((void **)p, n * sizeof(T));
}

template <class T>
void dfree(T *&p) {
  if (p) cudaFree((void *)p);
  p = nullptr;
}

int launched(lbmd_ctx *c, const char *where, int n = 1) {
  c->launches += n;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, where);
  return LBMD_OK;
}

int map_device_error(lbmd_ctx *c, unsigned bits) {
  if (bits & kErrNonFinite) return fail(c, LBMD_E_NONFINITE, "non-finite density or particle state");
  if (bits & kErrNegDensity) return fail(c, LBMD_E_NEGATIVE_DENSITY, "negative fluid density");
  if (bits & kErrBond) return fail(c, LBMD_E_BOND_BROKEN, "FENE bond stretched to or beyond R0");
  if (bits & kErrParticle) return fail(c, LBMD_E_NONFINITE, "particle position out of range");
  if (bits & kErrTooFast)
    return fail(c, LBMD_E_PARTICLE_TOO_FAST,
                "with md_substeps > 1 a particle moved more than one cell away within one lattice step");
  if (bits & kErrDrift) {
    double d[5] = {0, 0, 0, 0, 0};
    char m[256];
    if (cudaMemcpy(d, c->drift + 5, sizeof(d), cudaMemcpyDeviceToHost) != cudaSuccess) cudaGetLastError();
    std::snprintf(m, sizeof(m),
                  "FP64 drift check at step %.0f: mass drift A %.3e, B %.3e, momentum drift %.3e per unit mass "
                  "(tolerance %.3e)",
                  d[0], d[1], d[2], d[3], c->prm.drift_tol);
    return fail(c, LBMD_E_DRIFT, m);
  }
  return LBMD_OK;
}

int sync_and_check(lbmd_ctx *c) {
  CK(cudaStreamSynchronize(c->st), "cudaStreamSynchronize");
  unsigned bits = 0;
  CK(cudaMemcpy(&bits, c->err, sizeof(unsigned), cudaMemcpyDeviceToHost), "read error word");
  c->sticky |= bits;
  return map_device_error(c, c->sticky);
}

// The per-entry arrays of a sort of n entries (its counters belong to the context).
cudaError_t alloc_sort_entries(SortScratch &s, size_t n) {
  cudaError_t e;
  if ((e = dalloc(&s.row_of, n)) != cudaSuccess || (e = dalloc(&s.rank_of, n)) != cudaSuccess ||
      (e = dalloc(&s.perm, n)) != cudaSuccess || (e = dalloc(&s.row_at, n)) != cudaSuccess)
    return e;
  return dalloc(&s.key, n);
}

void free_sort_entries(SortScratch &s) {
  dfree(s.row_of); dfree(s.rank_of); dfree(s.perm); dfree(s.row_at); dfree(s.key);
}

void free_records(lbmd_ctx *c) {
  for (int b = 0; b < 2; ++b) {
    dfree(c->rec[b].cell); dfree(c->rec[b].frac); dfree(c->rec[b].key);
    dfree(c->rec[b].fric); dfree(c->rec[b].psA); dfree(c->rec[b].psB);
  }
  free_sort_entries(c->rec_sort);
  dfree(c->rec_row_start);
  c->rec_cap = 0;
}

int ensure_records(lbmd_ctx *c, long long n) {
  if (n <= c->rec_cap) return LBMD_OK;
  free_records(c);
  cudaError_t e = cudaSuccess;
  for (int b = 0; b < 2 && e == cudaSuccess; ++b) {
    ReactionRecords &r = c->rec[b];
    if ((e = dalloc(&r.cell, n)) != cudaSuccess || (e = dalloc(&r.frac, n)) != cudaSuccess ||
        (e = dalloc(&r.key, n)) != cudaSuccess || (e = dalloc(&r.fric, n)) != cudaSuccess ||
        (e = dalloc(&r.psA, n)) != cudaSuccess)
      break;
    e = dalloc(&r.psB, n);
  }
  if (e == cudaSuccess) e = alloc_sort_entries(c->rec_sort, (size_t)n);
  if (e == cudaSuccess) e = dalloc(&c->rec_row_start, (size_t)c->P.nrows + 1);
  // the first step clears the nodes of the cells here (with more particles than before, lbmd_set_particles
  // has cleared all): cells of the lattice, whatever it holds
  if (e == cudaSuccess) e = cudaMemsetAsync(c->rec[1].cell, 0, sizeof(int4) * (size_t)n, c->st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    free_records(c);
    return fail(c, LBMD_E_NOMEM, std::string("sub-stepping records: ") + cudaGetErrorString(e));
  }
  c->rec_cap = n;
  return LBMD_OK;
}

void free_particles(lbmd_ctx *c) {
  for (ParticleArrays *a : {&c->pa[0], &c->pa[1], &c->pt}) {
    dfree(a->cell);
    dfree(a->frac);
    dfree(a->vel);
    dfree(a->pid);
  }
  dfree(c->pf.fric); dfree(c->pf.psA); dfree(c->pf.psB); dfree(c->pf.fsr); dfree(c->pf.pair); dfree(c->pf.total);
  dfree(c->slot_of_id); dfree(c->jc);
  free_sort_entries(c->sort);
  c->jc_valid = false;
  c->cap = 0;
}

// One-pass update: BGK, or MRT in FP32 (by size only), one particle update per lattice step.  Chosen by
// the lattice size unless set (lbmd_set_lattice_passes); see onepass_pays and onepass_chunks.
constexpr int kOnePassChunkPlanes = 16;

bool onepass_allowed(const lbmd_ctx *c) {
  return (c->P.collision == LBMD_COLLISION_BGK || c->P.storage == LBMD_STORAGE_FP32) && c->P.substeps == 1;
}

// Whether one pass is the faster update, from what both took per step without particles (FP32,
// BGK, microseconds, two passes / one pass): 64^3 16.3 / 21.6, 80^3 33.9 / 38.8, 96^3 64.7 / 54.9,
// 100^3 75.8 / 74.8, 112^3 102 / 86, 128^3 150 / 119, 144^3 212 / 174, 192^3 476 / 382, 256^3
// 1124 / 886.  Two passes take about 72 ps per node there (less where the lattice stays in L2), one
// pass 8 us and 53 ps per lane of its 32 x 8 tiles, idle ones included: it loses where tiles are
// ragged (100 = 3 x 32 + 4 columns) and where the lattice is small.
// Fluctuating MRT, whose update is nearer to what the FMA pipes can do than to what HBM can: 96^3 71.2 /
// 74.0, 100 x 90 x 110 81.0 / 110.5, 128^3 162 / 160, 160^3 303 / 296, 192^3 514 / 502, 200 x 180 x 210 549 /
// 592, 256^3 1198 / 1143: 71 ps per node against 10 us more and 67 ps per lane.
bool onepass_pays(const StepParams &P) {
  const long long ntx = (P.nx + kOnePassCols - 1) / kOnePassCols, nty = (P.ny + kOnePassRows - 1) / kOnePassRows;
  const double lanes = (double)(ntx * nty * P.nz) * (kOnePassCols * kOnePassRows);
  if (P.collision == LBMD_COLLISION_MRT) return 67.0 * lanes + 10.0e6 < 71.0 * (double)P.N;
  return 53.0 * lanes + 8.0e6 < 72.0 * (double)P.N;
}

// The z-chunks of the one-pass update, a block for each column tile of a chunk: chunks of 16 planes,
// unless another count (8 to 32 planes: longer chunks let neighbouring blocks drift apart, and the
// sectors they share out of L2) fills the waves of the `slots` resident blocks better by 3 % or
// more, counting the 0.4 planes a block spends on its start and end.  With 16 planes, 128^3 has 512
// blocks on 456 slots and takes 138 us a step; with 7 chunks, 119 (a coupled step with 2500
// particles 184 -> 148 us).  Where there are many waves the count hardly matters: 886 to 901 us for 7
// to 32 chunks at 256^3.
int onepass_chunks(int tiles, int nz, int slots) {
  auto score = [&](int n) {
    const double waves = (double)tiles * n / slots, planes = (double)nz / n;
    return waves / std::ceil(waves) * planes / (planes + 0.4);
  };
  const int usual = std::max(1, (nz + kOnePassChunkPlanes / 2) / kOnePassChunkPlanes);
  int best = usual;
  double best_score = score(usual) * 1.03;
  const int least = (nz + 2 * kOnePassChunkPlanes - 1) / (2 * kOnePassChunkPlanes);
  const int most = std::min(2 * nz / kOnePassChunkPlanes, 64 * slots / tiles);  // past 64 waves: all alike
  for (int n = least; n <= most; ++n)
    if (score(n) > best_score) {
      best_score = score(n);
      best = n;
    }
  return best;
}

int onepass_full_grid(const lbmd_ctx *c) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev) != cudaSuccess || sms < 1) {
    cudaGetLastError();
    sms = 1;
  }
  return sms * onepass_blocks_per_sm();
}

bool uses_onepass(const lbmd_ctx *c) {
  if (!onepass_allowed(c) || c->passes == 2) return false;
  if (c->passes == 1) return true;
  return c->op_grid > 0;  // auto: prepare_onepass decided from the size
}

// Lattices without particles of up to kSmallNodes nodes take density pass and update in one launch
// (k_step_small has the figures on both sides of the line), unless two passes are set.
constexpr long long kSmallNodes = 65536;

bool small_lattice(const StepParams &P) { return P.N <= kSmallNodes; }

bool uses_one_launch(const lbmd_ctx *c) {
  return small_lattice(c->P) && c->np == 0 && c->passes == 0 && !uses_onepass(c);
}

void drop_graph(StepGraph &g) {
  if (g.exec) cudaGraphExecDestroy(g.exec);  // a launch in flight completes first
  if (g.graph) cudaGraphDestroy(g.graph);
  g = StepGraph{};
}

void drop_graphs(lbmd_ctx *c) {
  for (auto &level : c->graph)
    for (auto &row : level)
      for (StepGraph &g : row) drop_graph(g);
  c->replayed = 0;
}

// Frees what prepare_onepass set up.
void free_onepass(lbmd_ctx *c) {
  dfree(c->op_runs);
  dfree(c->op_out.edge);
  dfree(c->op_out.yedge);
  dfree(c->op_out.diag);
  dfree(c->op_out.zown);
  dfree(c->op_out.zedge);
  dfree(c->op_out.zyedge);
  dfree(c->op_zslot);
  c->op_nruns = 0;
  c->op_grid = 0;
}

// Sets up the one-pass update: its grid, chunks, partial sums and boundary runs.
int setup_onepass(lbmd_ctx *c) {
  const StepParams &P = c->P;
  free_onepass(c);  // what an earlier attempt that failed part-way left
  const int ntx = (P.nx + kOnePassCols - 1) / kOnePassCols, nty = (P.ny + kOnePassRows - 1) / kOnePassRows;
  // neighbouring column tiles of a chunk are launched together (they march in step, so the sectors
  // they share meet in L2)
  const int nchunks = onepass_chunks(ntx * nty, P.nz, onepass_full_grid(c));
  const int grid = ntx * nty * nchunks;
  std::vector<unsigned char> edge((size_t)ntx * nty * P.nz, 0);
  for (int col = 0; col < ntx * nty; ++col)
    for (int ch = 0; ch < nchunks; ++ch) {
      const int zs = (int)((long long)ch * P.nz / nchunks), ze = (int)((long long)(ch + 1) * P.nz / nchunks);
      if (ze <= zs) continue;
      edge[(size_t)col * P.nz + zs] = edge[(size_t)col * P.nz + ze - 1] = 1;
    }
  // edge rows from partial sums when every tile has at least 3 rows and 2 columns; chunk-edge
  // planes when the lattice is at least 2 planes deep
  const int ry = P.ny % kOnePassRows, rx = P.nx % kOnePassCols;
  const int ypart = (P.ny >= 3 && (ry == 0 || ry >= 3) && P.nx >= 2 && (rx == 0 || rx >= 2)) ? 1 : 0;
  const int zpart = P.nz >= 2 ? 1 : 0;
  std::vector<BoundaryRun> runs;
  for (int col = 0; col < ntx * nty; ++col) {
    const int tx = col % ntx, ty = col / ntx;
    const int x0 = tx * kOnePassCols, nown = std::min(kOnePassCols, P.nx - x0);
    const int y0 = ty * kOnePassRows, rows = std::min(kOnePassRows, P.ny - y0);
    for (int z = 0; z < P.nz; ++z)
      for (int w = 0; w < rows; ++w)
        if ((!zpart && edge[(size_t)col * P.nz + z]) || (!ypart && (w == 0 || w == rows - 1)))
          runs.push_back(BoundaryRun{z * P.ny + y0 + w, x0, nown});
  }
  if (runs.size() > 0x7fffffffull) return fail(c, LBMD_E_INVALID_ARG, "too many boundary runs");
  CK(dalloc(&c->op_out.edge, (size_t)P.nz * P.ny * ntx * 4), "edge sums");
  {
    // slot 2 b (plane zs - 1) and 2 b + 1 (plane zs) of the boundary below chunk b
    std::vector<int> zslot((size_t)P.nz, -1);
    for (int ch = 0; ch < nchunks; ++ch) {
      const int zs = (int)((long long)ch * P.nz / nchunks);
      zslot[(size_t)(zs == 0 ? P.nz - 1 : zs - 1)] = 2 * ch;
      zslot[(size_t)zs] = 2 * ch + 1;
    }
    CK(dalloc(&c->op_zslot, zslot.size()), "plane table");
    CK(cudaMemcpy(c->op_zslot, zslot.data(), sizeof(int) * zslot.size(), cudaMemcpyHostToDevice), "plane table");
  }
  // the kernels index the sums in 32 bits: at most 32 / 3 N entries here, with N < 2^32 / 19
  static_assert(kOnePassCols <= 3 * kQ, "2 nz nty ntx kOnePassCols < 2^32 for nx >= 2, ny >= 3");
  if (ypart) {
    CK(dalloc(&c->op_out.yedge, (size_t)2 * P.nz * nty * ntx * kOnePassCols * 2), "edge sums");
    CK(dalloc(&c->op_out.diag, (size_t)P.nz * nty * ntx * 4 * 2), "edge sums");
  }
  if (zpart) {
    CK(dalloc(&c->op_out.zown, (size_t)2 * nchunks * P.ny * P.nx * 2), "chunk-edge sums");
    CK(dalloc(&c->op_out.zedge, (size_t)2 * nchunks * P.ny * ntx * 4), "chunk-edge sums");
    if (ypart) CK(dalloc(&c->op_out.zyedge, (size_t)2 * 2 * nchunks * nty * ntx * kOnePassCols * 2), "chunk-edge sums");
  }
  CK(dalloc(&c->op_runs, runs.size()), "boundary runs");
  CK(cudaMemcpy(c->op_runs, runs.data(), sizeof(BoundaryRun) * runs.size(), cudaMemcpyHostToDevice), "boundary runs");
  c->op_nruns = (int)runs.size();
  c->op_geom = OnePassGeom{ntx, nty, nchunks, ypart, zpart};
  c->op_grid = grid;
  return LBMD_OK;
}

// Gives the one-pass update's partial sums back where the automatic choice took them, for another allocation
// that finds no room: two passes from the next step on.  Whether there were any.
bool release_onepass(lbmd_ctx *c) {
  if (c->passes != 0 || c->op_grid == 0) return false;
  drop_graphs(c);
  free_onepass(c);
  c->onepass_no_room = true;
  c->jc_valid = false;
  return true;
}

// setup_onepass once per context, where the next step takes one pass.  Allocates: call it before any
// capture.
int prepare_onepass(lbmd_ctx *c) {
  // set up already (op_grid; the run list may be empty: every node finished from partial sums)
  if (!onepass_allowed(c) || c->passes == 2 || c->op_grid > 0) return LBMD_OK;
  if (c->passes == 1) return setup_onepass(c);
  // automatic: one pass for FP32 storage where it pays (the 16-bit update is bound by instruction
  // issue, and the one-pass update's extra instructions cost it more than the second pass over half
  // the bytes) and where there is room for its partial sums
  if (c->onepass_no_room || c->P.storage != LBMD_STORAGE_FP32 || !onepass_pays(c->P)) return LBMD_OK;  // two passes
  const int r = setup_onepass(c);
  if (!r || cudaGetLastError() != cudaErrorMemoryAllocation) return r;
  free_onepass(c);
  c->onepass_no_room = true;
  return LBMD_OK;
}

// The densities of the current state into rho_buf[cur] (a density pass), if not there already.
int ensure_densities(lbmd_ctx *c) {
  if (c->rho_valid) return LBMD_OK;
  launch_moments(c->P, c->pop[c->cur], c->rest[c->cur], c->rho_buf[c->cur], nullptr, nullptr, c->st);
  const int r = launched(c, "moments");
  if (!r) c->rho_valid = true;
  return r;
}

// One pass with particles (one particle update per step): the corner j' of the current state
// into jc, if not there already.
int ensure_corner_j(lbmd_ctx *c) {
  if (c->jc_valid || c->np == 0 || c->P.substeps > 1 || !uses_onepass(c)) return LBMD_OK;
  if (c->sort_pending) {  // the arrays read here are the ones the pending sort writes
    CK(cudaStreamWaitEvent(c->st, c->ev_sorted, 0), "stream wait");
    c->sort_pending = false;
  }
  launch_corner_jprime(c->P, c->pa[c->pcur], c->np, c->pop[c->cur], c->jc, c->st);
  const int r = launched(c, "corner j'");
  if (!r) c->jc_valid = true;
  return r;
}

// Sorts the unsorted particles pt into pa[1 - pcur] and row_start[1 - pcur] on st, and makes these
// the current ones.  update: pt is first formed from pa[pcur] by the particle update.
int sort_particles(lbmd_ctx *c, bool update, cudaStream_t st) {
  const StepParams &P = c->P;
  const ParticleArrays &from = c->pa[c->pcur], &to = c->pa[1 - c->pcur];
  int *start = c->row_start[1 - c->pcur];
  unsigned *bits = P.substeps > 1 ? nullptr : c->node_bits[1 - c->pcur];
  c->pcur = 1 - c->pcur;
  if (sort_fits_one_block(P.nrows, P.np)) {
    launch_sort_small(P, update ? &from : nullptr, c->pt, c->pf, to, start, c->slot_of_id, bits, c->err, st);
    return launched(c, "particle sort");
  }
  if (update)
    launch_integrate_bin(P, from, c->pt, c->pf, c->sort, to.cell, bits, c->err, st);
  else
    launch_bin(P, c->pt, c->sort, c->err, st);
  launch_place(P, c->sort, c->pt, to, start, c->slot_of_id, bits, st);
  return launched(c, "particle sort", 4);  // bin, scan, scatter, place
}

// FP64 totals of the current state into diag_out: [M_A, M_B, Px, Py, Pz] of the fluid and,
// with particles, [5..7] = sum m v (K9 of the step; appendix and Sec. 2 for what they conserve).
int enqueue_totals(lbmd_ctx *c) {
  launch_fluid_sums(c->P, c->pop[c->cur], c->rest[c->cur], c->diag_partial, c->diag_blocks, c->st);
  launch_finish_sums(c->diag_partial, c->diag_blocks, 5, c->diag_out, c->st);
  int r = launched(c, "fluid sums", 2);
  if (r || c->np == 0) return r;
  StepParams P = c->P;
  P.np = c->np;
  const int nb = std::min(c->diag_blocks, (c->np + 255) / 256);
  double *part = c->diag_partial + (size_t)5 * c->diag_blocks - 3 * (size_t)nb;
  launch_particle_momentum(P, c->pa[c->pcur], part, nb, c->st);
  launch_finish_sums(part, nb, 3, c->diag_out + 5, c->st);
  return launched(c, "particle momentum", 2);
}

// The drift check on the device (set_ref: take the totals as the reference instead).
// The drift table before any reference: no reference, no check yet (step -1, no checks).
const double kDriftNone[10] = {0, 0, 0, 0, 0, -1, 0, 0, 0, 0};

int enqueue_drift(lbmd_ctx *c, int set_ref) {
  int r = enqueue_totals(c);
  if (r) return r;
  launch_drift_check(c->diag_out, c->np > 0 ? c->diag_out + 5 : nullptr, c->drift, c->drift + 5, c->err,
                     (long long)c->steps, c->prm.drift_tol, set_ref, c->st);
  return launched(c, "drift check");
}

}  // namespace

namespace {

// MD sub-stepping of one lattice step (K = P.substeps > 1): the sorted particles S of the step's
// start stay frozen (cell list, fluid-side solvation force); each of the K substeps, one launch,
// reads the particles' positions from one buffer and writes them to another: coupling forces (one
// momentum-return record per particle and substep), pair forces over S's rows with one more cell
// of reach, updates of dt / K.  The records are then sorted by row for the update's node-side
// gather.  On return pt is the particle state and (pa, pf, ci) describe the records.
int substep_particles(lbmd_ctx *c, ParticleArrays &pa, ParticleForces &pf, CellIndex &ci) {
  const StepParams &P = c->P;
  const int K = P.substeps, np = P.np;
  const long long nrec = (long long)K * np;
  if (nrec > 0x7fffffffLL) return fail(c, LBMD_E_INVALID_ARG, "md_substeps x particles exceeds 2^31");
  int r = ensure_records(c, nrec);
  if (r) return r;
  const ParticleArrays &S = c->pa[c->pcur];
  // the substeps alternate between pt, which takes the last one, and the buffer the particles' sort
  // overwrites later; the order is S's throughout, and so are the ids until pt gets its own
  const ParticleArrays &other = c->pa[1 - c->pcur];
  const ParticleArrays work[2] = {{c->pt.cell, c->pt.frac, c->pt.vel, S.pid},
                                  {other.cell, other.frac, other.vel, S.pid}};
  const CellIndex rows{c->row_start[c->pcur], nullptr};
  SortScratch rs = c->rec_sort;
  rs.row_count = c->sort.row_count;
  rs.block_count = c->sort.block_count;
  for (int sub = 0; sub < K; ++sub) {
    StepParams Q = P;
    Q.step = P.step * (unsigned long long)K + (unsigned long long)sub;
    Q.step_mul = (unsigned long long)K;
    Q.dt = P.dt / (float)K;
    const ParticleArrays &from = sub == 0 ? S : work[(K - sub) & 1];
    const ParticleArrays &to = sub == K - 1 ? c->pt : work[(K - 1 - sub) & 1];
    // (pair reach: particles may have left their row by one cell)
    launch_substep(Q, from, to, S, rows, P.reach > 0 ? P.reach + 1 : 0, c->rho_buf[c->cur], c->jp,
                   c->nbonds ? c->bond_start : nullptr, c->bond_other, c->slot_of_id, c->pf, sub, c->rec[0], rs,
                   c->rec[1].cell, c->node_bits[0], c->err, c->st);
    if ((r = launched(c, "particle substep"))) return r;
  }
  // sort the (binned) records by (row, x cell, substep * np + id): the same counting sort as particles
  launch_rec_place(P, (int)nrec, rs, c->rec[0], c->rec[1], c->rec_row_start, c->node_bits[0], c->st);
  if ((r = launched(c, "record sort", 3))) return r;
  pa = ParticleArrays{c->rec[1].cell, c->rec[1].frac, nullptr, nullptr};
  pf = c->pf;
  pf.fric = c->rec[1].fric;
  pf.psA = c->rec[1].psA;
  pf.psB = c->rec[1].psB;
  ci = CellIndex{c->rec_row_start, c->node_bits[0]};
  return LBMD_OK;
}

// Timing events of k_collide (lbmd_profile_enable): the pool holds at least n unused ones.
int reserve_events(lbmd_ctx *c, size_t n) {
  while (c->ev.size() < c->ev_used + n) {
    cudaEvent_t e;
    CK(cudaEventCreate(&e), "event");
    c->ev.push_back(e);
  }
  return LBMD_OK;
}

// st waits for a sort still pending on side.
int join_sort(lbmd_ctx *c) {
  if (!c->sort_pending) return LBMD_OK;
  CK(cudaStreamWaitEvent(c->st, c->ev_sorted, 0), "stream wait");
  c->sort_pending = false;
  return LBMD_OK;
}

// From this size on j' is stored at the marked nodes only, which needs the sort of the particles before
// the density pass.  Ten steps at 256^3: FP16 8575 -> 8529 us, fluctuating MRT 15000 -> 14857; twenty of
// 100x90x110, whose update is too short to hide the sort, 2087 -> 2153.
constexpr long long kMarkedFrom = 1 << 22;  // nodes

// One coupled step on st and side.  `step` is the noise counter the kernels get: the lattice
// step, or, while a graph is recorded, the step's offset in it (the kernels add the base).
// t0, t1 (or null): events recorded around the lattice update, with `flags`.
// The particles are kept sorted between steps: every step updates and sorts them for the next one
// on the side stream, beside the lattice update.  (The sort used to wait for the lattice update,
// whose particle arrays it overwrote, and the next coupling for the sort: with 2500 particles on
// 128^3, 199 us a step against 184; with 1000 on 100 x 90 x 110 and noise, 131 against 115.)
// join: st waits for that sort before returning (else the next step does, before its particle
// coupling).
int one_step(lbmd_ctx *c, unsigned long long step, cudaEvent_t t0, cudaEvent_t t1, unsigned flags, bool join) {
  StepParams &P = c->P;
  P.step = step;
  const CellIndex ci{c->row_start[c->pcur], c->node_bits[c->pcur]};
  const void *fin = c->pop[c->cur];
  void *fout = c->pop[1 - c->cur];
  float *rho = c->rho_buf[c->cur];
  int r;
  const bool sub = P.np > 0 && P.substeps > 1;
  const bool onepass = uses_onepass(c), small = uses_one_launch(c);
  const float *rest_in = c->rest[c->cur];
  float *rest_out = c->rest[1 - c->cur];
  if (P.np > 0 && !sub && !c->sort_pending) {
    // fork the side stream from the step's start (while st records a graph, this is also what
    // makes the side stream's work part of the graph); after a sort still pending there, the side
    // stream is already at this step
    CK(cudaEventRecord(c->ev_int, c->st), "event");
    CK(cudaStreamWaitEvent(c->side, c->ev_int, 0), "stream wait");
  }
  if (onepass) {
    if (!c->rho_valid) return fail(c, LBMD_E_STATE, "one-pass update without the densities of the current state");
  } else if (!small) {
    // densities (and j' for the particle coupling) of this step's populations; on large lattices j'
    // only at the nodes the sorted particles mark, whose sort the lattice update before has hidden
    // (with MD sub-stepping at every node: the particles move on within the step)
    const bool marked = P.np > 0 && !sub && P.N >= kMarkedFrom;
    if (marked && (r = join_sort(c))) return r;
    launch_moments(P, fin, rest_in, rho, P.np > 0 ? c->jp : nullptr, marked ? ci.node_bits : nullptr, c->st);
    if ((r = launched(c, "moments"))) return r;
  }
  if ((r = join_sort(c))) return r;
  ParticleArrays gpa = c->pa[c->pcur];  // what the update gathers the momentum return from
  ParticleForces gpf = c->pf;
  CellIndex gci = ci;
  if (sub) {
    if ((r = substep_particles(c, gpa, gpf, gci))) return r;
    // the working copy that took the substeps is the state
    CK(cudaEventRecord(c->ev_sub, c->st), "event");
    CK(cudaStreamWaitEvent(c->side, c->ev_sub, 0), "stream wait");
    if ((r = sort_particles(c, false, c->side))) return r;
    CK(cudaEventRecord(c->ev_sorted, c->side), "event");
    c->sort_pending = true;
  } else if (P.np > 0) {
    if (onepass) {  // no density pass stored j': the previous step formed it at the corners
      if (!c->jc_valid) return fail(c, LBMD_E_STATE, "one-pass coupling without the corner j' of the current state");
      launch_couple_jc(P, c->pa[c->pcur], ci, rho, c->jc, c->pf, c->st);
    } else
      launch_couple(P, c->pa[c->pcur], ci, rho, c->jp, c->pf, c->st);
    CK(cudaEventRecord(c->ev_coupled, c->st), "event");
    launch_pairs(P, c->pa[c->pcur], ci, c->nbonds ? c->bond_start : nullptr, c->bond_other, c->slot_of_id, c->pf,
                 c->err, c->side);
    if ((r = launched(c, "particle forces", 2))) return r;
    CK(cudaStreamWaitEvent(c->side, c->ev_coupled, 0), "stream wait");
    if ((r = sort_particles(c, true, c->side))) return r;
    CK(cudaEventRecord(c->ev_sorted, c->side), "event");
    c->sort_pending = true;
  }
  if (t0) CK(cudaEventRecordWithFlags(t0, c->st, flags), "event");
  if (onepass)
    launch_collide_onepass(P, fin, fout, rest_in, rest_out, rho, c->rho_buf[1 - c->cur],
                           c->op_out, gpa, gpf, gci, c->err, c->op_geom,
                           c->op_grid, c->st);
  else if (small)
    launch_step_small(P, fin, fout, rest_in, rest_out, c->err, c->st);
  else
    launch_collide(P, fin, fout, rest_in, rest_out, rho, gpa, gpf, gci, c->err, c->st);
  if ((r = launched(c, "collide"))) return r;
  if (t1) CK(cudaEventRecordWithFlags(t1, c->st, flags), "event");
  const bool corner_j = onepass && P.np > 0 && !sub;
  if (corner_j) {  // the next step's jc, at the sorted particles
    CK(cudaEventRecord(c->ev_collided, c->st), "event");
    CK(cudaStreamWaitEvent(c->side, c->ev_collided, 0), "stream wait");
    launch_corner_jprime(P, c->pa[c->pcur], P.np, fout, c->jc, c->side);
    if ((r = launched(c, "corner j'"))) return r;
    CK(cudaEventRecord(c->ev_sorted, c->side), "event");
  }
  if (onepass) {
    launch_boundary_densities(P, c->op_geom, fout, rest_out, c->rho_buf[1 - c->cur], c->op_runs, c->op_nruns,
                              c->op_out, c->op_zslot, c->st);
    if ((r = launched(c, "boundary densities"))) return r;
  }
  if (join && (r = join_sort(c))) return r;
  c->cur = 1 - c->cur;
  c->steps++;
  c->rho_valid = onepass;  // the two-pass update leaves the new state's densities to its next step
  c->jc_valid = corner_j;
  return LBMD_OK;
}

// Records nsteps steps from the current buffers into g: on the private stream gst, with
// the noise counters relative to the device-resident step base, the base advanced at the end.
// Nothing runs; the context's host state is left as it was.  (Profiled steps are recorded kShortGraph
// at a time.)
int record_steps(lbmd_ctx *c, StepGraph &g, int nsteps) {
  const StepParams &P = c->P;
  int r;
  if (P.np > 0 && P.substeps > 1 && (r = ensure_records(c, (long long)P.substeps * P.np)))
    return r;  // no allocation while recording
  if ((r = prepare_onepass(c))) return r;
  if (!c->gst) CK(cudaStreamCreateWithFlags(&c->gst, cudaStreamNonBlocking), "graph stream");
  if (!c->step_base) CK(dalloc(&c->step_base, 1), "alloc step base");
  if (c->prof)
    for (cudaEvent_t &e : c->ph)
      if (!e) CK(cudaEventCreate(&e), "event");
  const int cur0 = c->cur, pcur0 = c->pcur;
  const bool rho_valid0 = c->rho_valid, sort_pending0 = c->sort_pending, jc_valid0 = c->jc_valid;
  const int64_t steps0 = c->steps, launches0 = c->launches;
  cudaStream_t user = c->st;
  CK(cudaStreamBeginCapture(c->gst, cudaStreamCaptureModeThreadLocal), "begin capture");
  c->st = c->gst;
  c->P.step_base = c->step_base;
  r = LBMD_OK;
  for (int j = 0; j < nsteps && !r; ++j)
    r = one_step(c, (unsigned long long)j, c->prof ? c->ph[2 * j] : nullptr, c->prof ? c->ph[2 * j + 1] : nullptr,
                 cudaEventRecordExternal, j == nsteps - 1);
  if (!r) {
    launch_advance_step(c->step_base, nsteps, c->gst);
    r = launched(c, "step counter");
  }
  cudaGraph_t graph = nullptr;
  const cudaError_t e = cudaStreamEndCapture(c->gst, &graph);
  const bool back = c->cur == cur0 && c->pcur == pcur0;
  c->st = user;
  c->P.step_base = nullptr;
  c->cur = cur0;
  c->pcur = pcur0;
  c->rho_valid = rho_valid0;
  c->sort_pending = sort_pending0;
  c->jc_valid = jc_valid0;
  c->steps = steps0;
  g.launches = c->launches - launches0;
  c->launches = launches0;
  if (r || e != cudaSuccess || !back) {
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    if (r) return r;
    if (e != cudaSuccess) return cuda_fail(c, e, "graph capture");
    return fail(c, LBMD_E_STATE, "recorded steps do not return to their buffers");
  }
  g.graph = graph;
  cudaError_t ei = cudaGraphInstantiate(&g.exec, graph, 0);
  const bool noisy = c->P.collision == LBMD_COLLISION_MRT && c->P.fluct;
  if (ei == cudaSuccess && (c->prof || noisy)) {  // find the timing stand-ins and the noisy updates
    size_t n = 0;
    ei = cudaGraphGetNodes(graph, nullptr, &n);
    std::vector<cudaGraphNode_t> nodes(n);
    if (ei == cudaSuccess) ei = cudaGraphGetNodes(graph, nodes.data(), &n);
    for (size_t k = 0; k < n && ei == cudaSuccess; ++k) {
      cudaGraphNodeType t;
      if ((ei = cudaGraphNodeGetType(nodes[k], &t)) != cudaSuccess) break;
      if (t == cudaGraphNodeTypeEventRecord) {
        cudaEvent_t ev = nullptr;
        if ((ei = cudaGraphEventRecordNodeGetEvent(nodes[k], &ev)) != cudaSuccess) break;
        for (int q = 0; q < 2 * kShortGraph; ++q)
          if (ev == c->ph[q]) g.ev_node[q] = nodes[k];
      } else if (t == cudaGraphNodeTypeKernel && noisy) {
        cudaKernelNodeParams kp;
        if ((ei = cudaGraphKernelNodeGetParams(nodes[k], &kp)) != cudaSuccess) break;
        if (!is_noisy_update(kp.func) || !kp.kernelParams) continue;
        StepParams Q;
        std::memcpy(&Q, kp.kernelParams[0], sizeof(Q));
        g.updates.push_back({nodes[k], Q.step});
      }
    }
    for (int q = 0; q < 2 * kShortGraph && ei == cudaSuccess && c->prof; ++q)
      if (!g.ev_node[q]) ei = cudaErrorInvalidValue;
  }
  if (ei != cudaSuccess) {
    drop_graph(g);
    cudaGetLastError();
    return cuda_fail(c, ei, "graph instantiation");
  }
  if (noisy && g.updates.size() != (size_t)nsteps) {  // the update's nodes were not recognised
    drop_graphs(c);
    c->graphs = false;
    return kGraphUnavailable;
  }
  return LBMD_OK;
}

// The graph length for the next of n steps: the longest that fits and is recorded, or due for it.
int graph_level(const lbmd_ctx *c, int n) {
  int level = 0;
  for (int k = 1; k < c->graph_levels && !c->prof; ++k)
    if (kGraphSteps[k] <= n && c->replayed >= kGraphAfter[k]) level = k;
  return level;
}

// kGraphSteps[level] steps by one launch of the graph recorded for the current buffers; or none, and
// kGraphShorter, where a longer graph cannot be recorded or finds no memory.
int replay_steps(lbmd_ctx *c, int level) {
  StepGraph &g = c->graph[level][c->cur][c->pcur];
  const int nsteps = kGraphSteps[level];
  int r;
  if ((r = prepare_onepass(c))) return r;
  if (uses_onepass(c) && ((r = ensure_densities(c)) || (r = ensure_corner_j(c))))
    return r;  // before recording: not in the graph
  if (!g.exec) {
    const std::string msg = c->msg;
    r = record_steps(c, g, nsteps);
    if (level > 0 && r && r != kGraphUnavailable) {
      // (no memory for it, say) the graphs in use go on; an error of the device shows at their launch
      c->msg = msg;
      c->graph_levels = level;
      return kGraphShorter;
    }
    if (r) return r;
  }
  if (c->dev_step != c->steps) {  // steps were taken without the graph since it last ran
    launch_set_step(c->step_base, (unsigned long long)c->steps, c->st);
    if ((r = launched(c, "step counter"))) return r;
  }
  if (c->prof) {
    if ((r = reserve_events(c, 2 * kShortGraph))) return r;
    for (int q = 0; q < 2 * kShortGraph; ++q)
      CK(cudaGraphExecEventRecordNodeSetEvent(g.exec, g.ev_node[q], c->ev[c->ev_used + q]), "timing event");
  }
  for (const StepGraph::Update &u : g.updates)
    CK(set_update_step(g.exec, u.node, (unsigned long long)c->steps + u.off), "update counter");
  // (the first launch of a graph allocates; uploading it when it is recorded made every later launch whose
  // counters are patched 3 us slower)
  const cudaError_t launch = cudaGraphLaunch(g.exec, c->st);
  if (launch == cudaErrorMemoryAllocation && level > 0) {
    cudaGetLastError();
    drop_graph(g);
    c->graph_levels = level;
    return kGraphShorter;
  }
  CK(launch, "graph launch");
  if (c->prof) c->ev_used += 2 * kShortGraph;
  c->launches += g.launches;
  c->steps += nsteps;
  c->replayed += nsteps;
  c->dev_step = c->steps;
  c->rho_valid = uses_onepass(c);
  c->jc_valid = c->rho_valid && c->np > 0 && c->P.substeps == 1;
  return LBMD_OK;
}

}  // namespace

void lbmd::set_context_free_error(const std::string &m) { g_create_error = m; }

extern "C" {

const char *lbmd_last_error(const lbmd_ctx *c) { return c ? c->msg.c_str() : g_create_error.c_str(); }

int lbmd_create(const lbmd_params *prm, void *stream, lbmd_ctx **out, unsigned *warnings) {
  lbmd_ctx *c = nullptr;
  if (!prm || !out) return fail(c, LBMD_E_INVALID_ARG, "null argument");
  *out = nullptr;
  if (warnings) *warnings = 0;
  {
    std::string why;
    const int r = check_params(prm, why);
    if (r) return fail(c, r, why);
  }
  c = new lbmd_ctx();
  c->prm = *prm;
  c->st = (cudaStream_t)stream;
  cudaGetDevice(&c->dev);
  StepParams &P = c->P;
  fill_step_params(prm, P);
  c->pop_elem = prm->storage == LBMD_STORAGE_FP32 ? 4 : 2;
  cudaError_t e = cudaSuccess;
  const size_t npop = (size_t)2 * kQ * P.N * c->pop_elem;  // bytes; >= 19 N floats of staging
  if ((e = dalloc(&c->pop[0], npop)) != cudaSuccess || (e = dalloc(&c->pop[1], npop)) != cudaSuccess ||
      (e = dalloc(&c->rho_buf[0], (size_t)2 * P.N)) != cudaSuccess ||
      (e = dalloc(&c->rho_buf[1], (size_t)2 * P.N)) != cudaSuccess || (e = dalloc(&c->jp, (size_t)3 * P.N)) != cudaSuccess ||
      (e = dalloc(&c->err, 1)) != cudaSuccess ||
      (c->pop_elem == 2 && (e = dalloc(&c->rest[0], (size_t)2 * P.N)) != cudaSuccess) ||
      (c->pop_elem == 2 && small_lattice(P) && (e = dalloc(&c->rest[1], (size_t)2 * P.N)) != cudaSuccess)) {
    cudaGetLastError();
    lbmd_destroy(c);
    return fail(nullptr, e == cudaErrorMemoryAllocation ? LBMD_E_NOMEM : LBMD_E_CUDA,
                std::string("device allocation: ") + cudaGetErrorString(e));
  }
  if ((e = cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&c->ev_int, cudaEventDisableTiming)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&c->ev_sorted, cudaEventDisableTiming)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&c->ev_coupled, cudaEventDisableTiming)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&c->ev_sub, cudaEventDisableTiming)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&c->ev_collided, cudaEventDisableTiming)) != cudaSuccess) {
    cudaGetLastError();
    lbmd_destroy(c);
    return fail(nullptr, LBMD_E_CUDA, std::string("stream / event creation: ") + cudaGetErrorString(e));
  }
  if (!c->rest[1]) c->rest[1] = c->rest[0];
  c->diag_blocks = fluid_sum_blocks(P);
  if ((e = dalloc(&c->diag_partial, (size_t)5 * c->diag_blocks)) != cudaSuccess ||
      (e = dalloc(&c->diag_out, 8)) != cudaSuccess || (e = dalloc(&c->drift, 10)) != cudaSuccess ||
      (e = cudaMemcpy(c->drift, kDriftNone, sizeof(kDriftNone), cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(c->err, 0, sizeof(unsigned))) != cudaSuccess) {
    cudaGetLastError();
    lbmd_destroy(c);
    return fail(nullptr, LBMD_E_NOMEM, std::string("device allocation: ") + cudaGetErrorString(e));
  }
  const unsigned w = param_warnings(prm);
  if (warnings) *warnings = w;
  *out = c;
  return LBMD_OK;
}

void lbmd_destroy(lbmd_ctx *c) {
  if (!c) return;
  cudaSetDevice(c->dev);
  if (c->st) cudaStreamSynchronize(c->st);
  if (c->side) {
    cudaStreamSynchronize(c->side);
    cudaStreamDestroy(c->side);
  }
  if (c->ev_int) cudaEventDestroy(c->ev_int);
  if (c->ev_sorted) cudaEventDestroy(c->ev_sorted);
  if (c->ev_coupled) cudaEventDestroy(c->ev_coupled);
  if (c->ev_sub) cudaEventDestroy(c->ev_sub);
  if (c->ev_collided) cudaEventDestroy(c->ev_collided);
  if (c->ev_dev_in) cudaEventDestroy(c->ev_dev_in);
  if (c->ev_dev_out) cudaEventDestroy(c->ev_dev_out);
  drop_graphs(c);
  if (c->gst) cudaStreamDestroy(c->gst);
  for (cudaEvent_t e : c->ph)
    if (e) cudaEventDestroy(e);
  dfree(c->step_base);
  dfree(c->pop[0]); dfree(c->pop[1]); dfree(c->rho_buf[0]); dfree(c->rho_buf[1]); dfree(c->jp); dfree(c->err);
  if (c->rest[1] == c->rest[0]) c->rest[1] = nullptr;
  dfree(c->rest[0]); dfree(c->rest[1]);
  free_onepass(c);
  dfree(c->diag_partial); dfree(c->diag_out); dfree(c->drift);
  free_particles(c);
  free_records(c);
  dfree(c->sort.row_count); dfree(c->sort.block_count); dfree(c->row_start[0]); dfree(c->row_start[1]);
  dfree(c->node_bits[0]); dfree(c->node_bits[1]);
  dfree(c->bond_start); dfree(c->bond_other);
  for (cudaEvent_t ev : c->ev) cudaEventDestroy(ev);
  delete c;
}

int lbmd_set_types(lbmd_ctx *c, int ntypes, const lbmd_ptype *types, int npairs, const lbmd_pair *pairs,
                   unsigned *warnings) {
  if (!c) return LBMD_E_INVALID_ARG;
  drop_graphs(c);  // every setter: the recorded steps hold the old parameters and buffers
  if (warnings) *warnings = 0;
  unsigned w = 0;
  std::string why;
  const int r = apply_types(c->P, c->prm.kT, c->prm.dt, ntypes, types, npairs, pairs, w, why);
  if (r) return fail(c, r, why);
  c->types_set = true;
  if (warnings) *warnings = w;
  return LBMD_OK;
}

int lbmd_set_debye_hueckel(lbmd_ctx *c, double lB, double kappa_D, double rc) {
  if (!c) return LBMD_E_INVALID_ARG;
  drop_graphs(c);
  std::string why;
  const int r = apply_debye_hueckel(c->P, lB, kappa_D, rc, why);
  return r ? fail(c, r, why) : LBMD_OK;
}

int lbmd_init_fluid(lbmd_ctx *c, const float *rhoA, const float *rhoB, const float *u) {
  if (!c || !rhoA || !rhoB) return c ? fail(c, LBMD_E_INVALID_ARG, "null density") : LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  drop_graphs(c);
  const long long N = c->P.N;
  if (!densities_valid(rhoA, rhoB, N))
    return fail(c, LBMD_E_INVALID_ARG, "densities must be finite and > 0");
  // stage through the (not yet used) second population buffer
  float *stage = reinterpret_cast<float *>(c->pop[1 - c->cur]);
  const size_t bytes = sizeof(float) * (size_t)N;
  CK(cudaMemcpyAsync(stage, rhoA, bytes, cudaMemcpyHostToDevice, c->st), "upload rhoA");
  CK(cudaMemcpyAsync(stage + N, rhoB, bytes, cudaMemcpyHostToDevice, c->st), "upload rhoB");
  const float *du = nullptr;
  if (u) {
    CK(cudaMemcpyAsync(stage + 2 * N, u, 3 * bytes, cudaMemcpyHostToDevice, c->st), "upload u");
    du = stage + 2 * N;
  }
  launch_init_equilibrium(c->P, stage, stage + N, du, c->pop[c->cur], c->rest[c->cur], c->st);
  int r = launched(c, "init_equilibrium");
  if (r) return r;
  c->steps = 0;
  c->rho_valid = false;
  c->jc_valid = false;
  if ((r = ensure_densities(c))) return r;
  // the drift check's reference (a context that never checks takes it only when asked)
  if (c->prm.diag_every > 0 && (r = enqueue_drift(c, 1))) return r;
  CK(cudaStreamSynchronize(c->st), "sync");
  c->fluid_ready = true;
  return LBMD_OK;
}

int lbmd_set_populations(lbmd_ctx *c, int comp, const float *f) {
  if (!c || !f || comp < 0 || comp > 1) return c ? fail(c, LBMD_E_INVALID_ARG, "bad arguments") : LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  drop_graphs(c);
  float *stage = reinterpret_cast<float *>(c->pop[1 - c->cur]);
  CK(cudaMemcpyAsync(stage, f, sizeof(float) * kQ * (size_t)c->P.N, cudaMemcpyHostToDevice, c->st), "upload f");
  launch_restream(c->P, stage, comp, c->pop[c->cur], c->rest[c->cur], c->st);
  int r = launched(c, "restream");
  if (r) return r;
  c->rho_valid = false;
  c->jc_valid = false;
  if ((r = ensure_densities(c))) return r;
  CK(cudaStreamSynchronize(c->st), "sync");
  c->fluid_ready = true;
  return LBMD_OK;
}

int lbmd_get_populations(lbmd_ctx *c, int comp, float *f) {
  if (!c || !f || comp < 0 || comp > 1) return c ? fail(c, LBMD_E_INVALID_ARG, "bad arguments") : LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  float *stage = reinterpret_cast<float *>(c->pop[1 - c->cur]);
  launch_unstream(c->P, c->pop[c->cur], c->rest[c->cur], comp, stage, c->st);
  int r = launched(c, "unstream");
  if (r) return r;
  CK(cudaMemcpyAsync(f, stage, sizeof(float) * kQ * (size_t)c->P.N, cudaMemcpyDeviceToHost, c->st), "download f");
  return sync_and_check(c);
}

int lbmd_set_particles(lbmd_ctx *c, int n, const double *x, const double *v, const int *type, const double *q) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (n < 0 || (n > 0 && (!x || !v || !type))) return fail(c, LBMD_E_INVALID_ARG, "bad particle arrays");
  if (n > 0 && !c->types_set) return fail(c, LBMD_E_STATE, "set the particle types first");
  cudaSetDevice(c->dev);
  drop_graphs(c);
  StepParams &P = c->P;
  std::vector<int4> hc;
  std::vector<float4> hf, hv;
  std::vector<int> hid;
  {
    std::string why;
    const int r = convert_particles(P, n, x, v, type, q, hc, hf, hv, hid, why);
    if (r) return fail(c, r, why);
  }
  // an allocation, again without the one-pass update's partial sums if there is no room beside them
  auto with_room = [c](auto alloc) {
    cudaError_t e = alloc();
    if (e == cudaErrorMemoryAllocation && release_onepass(c)) {
      cudaGetLastError();
      e = alloc();
    }
    return e;
  };
  if (n > c->cap) {
    auto alloc = [c, n] {
      free_particles(c);
      cudaError_t e = cudaSuccess;
      for (ParticleArrays *a : {&c->pa[0], &c->pa[1], &c->pt}) {
        if (e != cudaSuccess || (e = dalloc(&a->cell, n)) != cudaSuccess ||
            (e = dalloc(&a->frac, n)) != cudaSuccess || (e = dalloc(&a->vel, n)) != cudaSuccess)
          break;
        e = dalloc(&a->pid, n);
      }
      if (e == cudaSuccess) e = dalloc(&c->pf.fric, n);
      if (e == cudaSuccess) e = dalloc(&c->pf.psA, n);
      if (e == cudaSuccess) e = dalloc(&c->pf.psB, n);
      if (e == cudaSuccess) e = dalloc(&c->pf.fsr, n);
      if (e == cudaSuccess) e = dalloc(&c->pf.pair, n);
      if (e == cudaSuccess) e = dalloc(&c->pf.total, n);
      if (e == cudaSuccess) e = dalloc(&c->slot_of_id, n);
      if (e == cudaSuccess) e = alloc_sort_entries(c->sort, (size_t)n);
      if (e == cudaSuccess) e = dalloc(&c->jc, (size_t)n * 8);
      return e;
    };
    const cudaError_t e = with_room(alloc);
    if (e != cudaSuccess) {
      cudaGetLastError();
      free_particles(c);
      c->np = 0;
      P.np = 0;
      return fail(c, LBMD_E_NOMEM, std::string("particle allocation: ") + cudaGetErrorString(e));
    }
    c->cap = n;
  }
  if (!c->sort.row_count) {  // rows are needed by the lattice kernels' gather even without particles
    const size_t nb = (size_t)scan_blocks(P.nrows);
    auto alloc = [c, &P, nb] {
      cudaError_t e = cudaSuccess;
      for (int *&start : c->row_start)
        if (e == cudaSuccess && !start) e = dalloc(&start, (size_t)P.nrows + 1);
      for (unsigned *&bits : c->node_bits)
        if (e == cudaSuccess && !bits) e = dalloc(&bits, node_words(P.nx) * (size_t)P.nrows);
      if (e == cudaSuccess && !c->sort.block_count) e = dalloc(&c->sort.block_count, nb);
      return e == cudaSuccess ? dalloc(&c->sort.row_count, (size_t)P.nrows) : e;
    };
    CK(with_room(alloc), "alloc rows");
    CK(cudaMemsetAsync(c->sort.block_count, 0, sizeof(int) * nb, c->st), "clear rows");
    CK(cudaMemsetAsync(c->sort.row_count, 0, sizeof(int) * (size_t)P.nrows, c->st), "clear rows");
  }
  c->np = n;
  P.np = n;
  c->pcur = 0;
  c->jc_valid = false;
  if (n > 0) {
    CK(cudaMemcpyAsync(c->pt.cell, hc.data(), sizeof(int4) * n, cudaMemcpyHostToDevice, c->st), "upload");
    CK(cudaMemcpyAsync(c->pt.frac, hf.data(), sizeof(float4) * n, cudaMemcpyHostToDevice, c->st), "upload");
    CK(cudaMemcpyAsync(c->pt.vel, hv.data(), sizeof(float4) * n, cudaMemcpyHostToDevice, c->st), "upload");
    CK(cudaMemcpyAsync(c->pt.pid, hid.data(), sizeof(int) * n, cudaMemcpyHostToDevice, c->st), "upload");
    // as after a step, the buffer the sort does not take holds the order of the (zero) total forces
    // and, its nodes cleared below, cells of the lattice
    for (unsigned *bits : c->node_bits)
      CK(cudaMemsetAsync(bits, 0, sizeof(unsigned) * node_words(P.nx) * (size_t)P.nrows, c->st), "clear nodes");
    CK(cudaMemcpyAsync(c->pa[0].cell, hc.data(), sizeof(int4) * n, cudaMemcpyHostToDevice, c->st), "upload");
    CK(cudaMemcpyAsync(c->pa[0].pid, hid.data(), sizeof(int) * n, cudaMemcpyHostToDevice, c->st), "upload");
    CK(cudaMemsetAsync(c->pf.total, 0, sizeof(float4) * n, c->st), "memset");
    int r = sort_particles(c, false, c->st);
    if (r) return r;
  }
  c->sort_pending = false;
  if (c->fluid_ready && c->prm.diag_every > 0) {  // the drift check's reference includes the new particles' momentum
    const int r = enqueue_drift(c, 1);
    if (r) return r;
  }
  CK(cudaStreamSynchronize(c->st), "sync");
  return LBMD_OK;
}

int lbmd_set_bonds(lbmd_ctx *c, int nb, const int *pairs, int kind, double k, double r) {
  if (!c) return LBMD_E_INVALID_ARG;
  drop_graphs(c);
  if (nb < 0 || (nb > 0 && !pairs)) return fail(c, LBMD_E_INVALID_ARG, "bad bond list");
  if (kind != LBMD_BOND_FENE && kind != LBMD_BOND_HARMONIC) return fail(c, LBMD_E_INVALID_ARG, "unknown bond kind");
  if (nb > 0 && (!(k >= 0.0) || !(r > 0.0 || kind == LBMD_BOND_HARMONIC)))
    return fail(c, LBMD_E_INVALID_ARG, "bad bond parameters");
  cudaSetDevice(c->dev);
  dfree(c->bond_start);
  dfree(c->bond_other);
  c->nbonds = 0;
  if (nb == 0) return LBMD_OK;
  const int n = c->np;
  std::vector<int> deg(n + 1, 0), other(2 * (size_t)nb);
  for (int b = 0; b < nb; ++b) {
    const int i = pairs[2 * b], j = pairs[2 * b + 1];
    if (i < 0 || i >= n || j < 0 || j >= n || i == j) return fail(c, LBMD_E_INVALID_ARG, "bond index out of range");
    deg[i + 1]++;
    deg[j + 1]++;
  }
  for (int i = 0; i < n; ++i) deg[i + 1] += deg[i];
  std::vector<int> fill(deg.begin(), deg.end() - 1);
  for (int b = 0; b < nb; ++b) {
    const int i = pairs[2 * b], j = pairs[2 * b + 1];
    other[fill[i]++] = j;
    other[fill[j]++] = i;
  }
  CK(dalloc(&c->bond_start, (size_t)n + 1), "alloc bonds");
  CK(dalloc(&c->bond_other, 2 * (size_t)nb), "alloc bonds");
  CK(cudaMemcpy(c->bond_start, deg.data(), sizeof(int) * (n + 1), cudaMemcpyHostToDevice), "upload bonds");
  CK(cudaMemcpy(c->bond_other, other.data(), sizeof(int) * 2 * nb, cudaMemcpyHostToDevice), "upload bonds");
  c->nbonds = nb;
  c->bond_np = n;
  c->P.bond_kind = kind;
  c->P.bond_k = (float)k;
  c->P.bond_r = (float)r;
  return LBMD_OK;
}

int lbmd_step(lbmd_ctx *c, int nsteps) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (nsteps < 0) return fail(c, LBMD_E_INVALID_ARG, "nsteps < 0");
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  if (c->nbonds > 0 && c->bond_np != c->np)
    return fail(c, LBMD_E_STATE, "bonds refer to a different particle set; call lbmd_set_bonds again");
  c->P.np = c->np;
  const int64_t K = c->prm.diag_every;
  int left = nsteps, r;
  while (left > 0) {
    // steps up to the next multiple of diag_every (the drift check runs after it), or all
    int n = left;
    if (K > 0) n = (int)std::min<int64_t>(left, K - c->steps % K);
    left -= n;
    int s = 0;
    if (c->graphs)
      while (s + kShortGraph <= n) {
        const int level = graph_level(c, n - s);
        r = replay_steps(c, level);
        if (r == kGraphShorter) continue;
        if (r == kGraphUnavailable) break;
        if (r) return r;
        s += kGraphSteps[level];
      }
    if (s < n) {
      if ((r = prepare_onepass(c))) return r;
      if (uses_onepass(c) && ((r = ensure_densities(c)) || (r = ensure_corner_j(c)))) return r;
    }
    for (; s < n; ++s) {
      cudaEvent_t t0 = nullptr, t1 = nullptr;
      if (c->prof) {
        if ((r = reserve_events(c, 2))) return r;
        t0 = c->ev[c->ev_used];
        t1 = c->ev[c->ev_used + 1];
      }
      if ((r = one_step(c, (unsigned long long)c->steps, t0, t1, cudaEventRecordDefault, true))) return r;
      if (c->prof) c->ev_used += 2;
    }
    if (K > 0 && c->steps % K == 0 && (r = enqueue_drift(c, 0))) return r;
  }
  return LBMD_OK;
}

int lbmd_set_graphs(lbmd_ctx *c, int on) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  drop_graphs(c);
  c->graphs = on != 0;
  c->graph_levels = kGraphLevels;
  return LBMD_OK;
}

int lbmd_set_lattice_passes(lbmd_ctx *c, int passes) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (passes < 0 || passes > 2) return fail(c, LBMD_E_INVALID_ARG, "passes must be 0 (by size), 1 or 2");
  if (passes == 1 && (c->P.collision != LBMD_COLLISION_BGK || !onepass_allowed(c)))
    return fail(c, LBMD_E_INVALID_ARG, "the one-pass update takes the BGK collision with md_substeps = 1");
  cudaSetDevice(c->dev);
  drop_graphs(c);
  if (passes != c->passes) {
    c->onepass_no_room = false;
    free_onepass(c);  // set up again for the new choice at the next step
    c->jc_valid = false;
  }
  c->passes = passes;
  return LBMD_OK;
}

int lbmd_get_lattice_passes(lbmd_ctx *c) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  const int r = prepare_onepass(c);
  if (r) return r;
  return uses_onepass(c) ? 1 : 2;
}

int lbmd_sync(lbmd_ctx *c) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  return sync_and_check(c);
}

int lbmd_clear_error(lbmd_ctx *c) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  CK(cudaStreamSynchronize(c->st), "sync");
  CK(cudaMemset(c->err, 0, sizeof(unsigned)), "clear error word");
  c->sticky = 0;
  c->msg.clear();
  return LBMD_OK;
}

int lbmd_get_fields(lbmd_ctx *c, float *rhoA, float *rhoB, float *u) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  const long long N = c->P.N;
  float *stage = reinterpret_cast<float *>(c->pop[1 - c->cur]);
  int r = ensure_densities(c);
  if (r) return r;
  launch_fields(c->P, c->pop[c->cur], c->rest[c->cur], c->rho_buf[c->cur], stage, stage + N, u ? stage + 2 * N : nullptr, c->st);
  if ((r = launched(c, "fields"))) return r;
  const size_t bytes = sizeof(float) * (size_t)N;
  if (rhoA) CK(cudaMemcpyAsync(rhoA, stage, bytes, cudaMemcpyDeviceToHost, c->st), "download");
  if (rhoB) CK(cudaMemcpyAsync(rhoB, stage + N, bytes, cudaMemcpyDeviceToHost, c->st), "download");
  if (u) CK(cudaMemcpyAsync(u, stage + 2 * N, 3 * bytes, cudaMemcpyDeviceToHost, c->st), "download");
  return sync_and_check(c);
}

int lbmd_get_particles(lbmd_ctx *c, double *x, double *v, double *f) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  const int n = c->np;
  if (n == 0) return sync_and_check(c);
  std::vector<int4> hc(n);
  std::vector<float4> hf(n), hv(n), ht(n);
  std::vector<int> hid(n), htid(n);
  const ParticleArrays &pa = c->pa[c->pcur];
  // the total forces are in the order of the copy the particle update wrote, which the sort for
  // the next step leaves in the other buffer
  const ParticleArrays &pt = c->pa[1 - c->pcur];
  CK(cudaMemcpyAsync(hc.data(), pa.cell, sizeof(int4) * n, cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaMemcpyAsync(hf.data(), pa.frac, sizeof(float4) * n, cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaMemcpyAsync(hv.data(), pa.vel, sizeof(float4) * n, cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaMemcpyAsync(ht.data(), c->pf.total, sizeof(float4) * n, cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaMemcpyAsync(hid.data(), pa.pid, sizeof(int) * n, cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaMemcpyAsync(htid.data(), pt.pid, sizeof(int) * n, cudaMemcpyDeviceToHost, c->st), "download");
  int r = sync_and_check(c);
  for (int j = 0; j < n; ++j) {
    const int id = hid[j], tid = htid[j];
    if (id < 0 || id >= n || tid < 0 || tid >= n) return fail(c, LBMD_E_CUDA, "corrupt particle ids");
    if (x) {
      x[3 * id] = hc[j].x + (double)hf[j].x;
      x[3 * id + 1] = hc[j].y + (double)hf[j].y;
      x[3 * id + 2] = hc[j].z + (double)hf[j].z;
    }
    if (v) {
      v[3 * id] = hv[j].x; v[3 * id + 1] = hv[j].y; v[3 * id + 2] = hv[j].z;
    }
    if (f) {
      f[3 * tid] = ht[j].x; f[3 * tid + 1] = ht[j].y; f[3 * tid + 2] = ht[j].z;
    }
  }
  return r;
}

// The device-memory getters write into caller buffers on the context's stream, ordered after the
// work already queued on the caller's stream and before the work the caller queues there next.
static int dev_getter_begin(lbmd_ctx *c, cudaStream_t caller) {
  if (!c->ev_dev_in) CK(cudaEventCreateWithFlags(&c->ev_dev_in, cudaEventDisableTiming), "event");
  if (!c->ev_dev_out) CK(cudaEventCreateWithFlags(&c->ev_dev_out, cudaEventDisableTiming), "event");
  if (caller != c->st) {
    CK(cudaEventRecord(c->ev_dev_in, caller), "event");
    CK(cudaStreamWaitEvent(c->st, c->ev_dev_in, 0), "stream wait");
  }
  return LBMD_OK;
}

static int dev_getter_end(lbmd_ctx *c, cudaStream_t caller) {
  if (caller != c->st) {
    CK(cudaEventRecord(c->ev_dev_out, c->st), "event");
    CK(cudaStreamWaitEvent(caller, c->ev_dev_out, 0), "stream wait");
  }
  return LBMD_OK;
}

static int dev_buffers_ok(lbmd_ctx *c, const char *name, const void *p, size_t bytes) {
  if (p && !device_buffer_ok(p, bytes))
    return fail(c, LBMD_E_INVALID_ARG,
                std::string(name) + " is not device memory of this context's device holding " +
                    std::to_string(bytes) + " bytes");
  return LBMD_OK;
}

int lbmd_get_fields_dev(lbmd_ctx *c, float *rhoA, float *rhoB, float *u, void *stream) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  const long long N = c->P.N;
  const size_t bytes = sizeof(float) * (size_t)N;
  int r;
  if ((r = dev_buffers_ok(c, "rhoA_dev", rhoA, bytes)) || (r = dev_buffers_ok(c, "rhoB_dev", rhoB, bytes)) ||
      (r = dev_buffers_ok(c, "u_dev", u, 3 * bytes)))
    return r;
  if (!rhoA && !rhoB && !u) return LBMD_OK;
  const cudaStream_t caller = static_cast<cudaStream_t>(stream);
  if ((r = dev_getter_begin(c, caller))) return r;
  if ((r = ensure_densities(c))) return r;
  launch_fields(c->P, c->pop[c->cur], c->rest[c->cur], c->rho_buf[c->cur], rhoA, rhoB, u, c->st);
  if ((r = launched(c, "fields"))) return r;
  return dev_getter_end(c, caller);
}

int lbmd_get_populations_dev(lbmd_ctx *c, int comp, float *f, void *stream) {
  if (!c || !f || comp < 0 || comp > 1) return c ? fail(c, LBMD_E_INVALID_ARG, "bad arguments") : LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  int r;
  if ((r = dev_buffers_ok(c, "f_dev", f, sizeof(float) * kQ * (size_t)c->P.N))) return r;
  const cudaStream_t caller = static_cast<cudaStream_t>(stream);
  if ((r = dev_getter_begin(c, caller))) return r;
  launch_unstream(c->P, c->pop[c->cur], c->rest[c->cur], comp, f, c->st);
  if ((r = launched(c, "unstream"))) return r;
  return dev_getter_end(c, caller);
}

int lbmd_get_particles_dev(lbmd_ctx *c, double *x, double *v, double *f, void *stream) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  const int n = c->np;
  const size_t bytes = sizeof(double) * 3 * (size_t)n;
  int r;
  if ((r = dev_buffers_ok(c, "x_dev", x, bytes)) || (r = dev_buffers_ok(c, "v_dev", v, bytes)) ||
      (r = dev_buffers_ok(c, "f_dev", f, bytes)))
    return r;
  if (n == 0 || (!x && !v && !f)) return LBMD_OK;
  const cudaStream_t caller = static_cast<cudaStream_t>(stream);
  if ((r = dev_getter_begin(c, caller))) return r;
  if (c->sort_pending) {  // the arrays read here are the ones the pending sort writes
    CK(cudaStreamWaitEvent(c->st, c->ev_sorted, 0), "stream wait");
    c->sort_pending = false;
  }
  // the total forces are in the order of the copy the particle update wrote (as in lbmd_get_particles)
  launch_particles_out(n, c->pa[c->pcur], c->pa[1 - c->pcur].pid, c->pf.total, x, v, f, c->st);
  if ((r = launched(c, "particles out"))) return r;
  return dev_getter_end(c, caller);
}

int lbmd_diagnostics(lbmd_ctx *c, double out[8]) {
  if (!c || !out) return c ? fail(c, LBMD_E_INVALID_ARG, "null output") : LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  int r = enqueue_totals(c);
  if (r) return r;
  double h[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  CK(cudaMemcpyAsync(h, c->diag_out, sizeof(double) * (c->np > 0 ? 8 : 5), cudaMemcpyDeviceToHost, c->st),
     "download");
  r = sync_and_check(c);
  std::memcpy(out, h, sizeof(h));
  return r;
}

int lbmd_set_drift_reference(lbmd_ctx *c) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  return enqueue_drift(c, 1);
}

int lbmd_get_drift(lbmd_ctx *c, double out[5]) {
  if (!c || !out) return c ? fail(c, LBMD_E_INVALID_ARG, "null output") : LBMD_E_INVALID_ARG;
  if (!c->fluid_ready) return fail(c, LBMD_E_STATE, "fluid not initialised");
  cudaSetDevice(c->dev);
  double h[5];
  CK(cudaMemcpyAsync(h, c->drift + 5, sizeof(h), cudaMemcpyDeviceToHost, c->st), "download");
  CK(cudaStreamSynchronize(c->st), "sync");
  std::memcpy(out, h, sizeof(h));
  return LBMD_OK;
}

int64_t lbmd_step_count(const lbmd_ctx *c) { return c ? c->steps : -1; }
int64_t lbmd_launch_count(const lbmd_ctx *c) { return c ? c->launches : -1; }

int lbmd_profile_enable(lbmd_ctx *c, int on) {
  if (!c) return LBMD_E_INVALID_ARG;
  if (c->prof != (on != 0)) drop_graphs(c);  // profiled graphs carry the timing events
  c->prof = on != 0;
  return LBMD_OK;
}

int lbmd_profile_read(lbmd_ctx *c, double *ms, int64_t *nl, int reset) {
  if (!c) return LBMD_E_INVALID_ARG;
  cudaSetDevice(c->dev);
  CK(cudaStreamSynchronize(c->st), "sync");
  for (size_t k = 0; k + 1 < c->ev_used; k += 2) {
    float t = 0.f;
    CK(cudaEventElapsedTime(&t, c->ev[k], c->ev[k + 1]), "event time");
    c->prof_ms += t;
    c->prof_launches++;
  }
  c->ev_used = 0;
  if (ms) *ms = c->prof_ms;
  if (nl) *nl = c->prof_launches;
  if (reset) {
    c->prof_ms = 0.0;
    c->prof_launches = 0;
  }
  return LBMD_OK;
}

}  // extern "C"
