// lb_particles.cu -- particle kernels of the coupled Shan-Chen LB / MD step (sm_103a):
// deterministic counting sort by lattice row, coupling forces (Eqs. NEWTON,
// solvation_kappa, solvation_lambda with trilinear interpolation), short-range pair and
// bonded forces (owner computes, no atomics), and the particle update.
#include "lb_site.cuh"

namespace lbmd {

namespace {

constexpr int kPBlock = 128;

inline unsigned pgrid(long long n) { return (unsigned)((n + kPBlock - 1) / kPBlock); }

// ------------------------------------------------------------------ particle sort
//
// Particles (and the reaction records of MD sub-stepping) are kept sorted by lattice row (z, y),
// then x cell, then id: a counting sort by row whose order within a row comes from ranks.
//   bin      the row of each particle, its rank of arrival in the row (the histogram's counter
//            before it), and the histogram summed over the kScanRows rows of each scan block
//   scan     rows -> first sorted slot: a block scans its rows from the sum of the block totals
//            before it (one launch; a total for 2048 rows), and clears the counters for the next sort:
//            21 us for 2 M rows, 547 for 67 M (a lattice of one column), beside updates of 186 and 3033
//   scatter  each particle's sort key to a slot of its row, in arrival order
//   place    a particle's slot in its row is the number of smaller keys there; it moves
// The keys of a row are distinct, so the order, and every gather after it, is deterministic
// whatever the order of arrival.  Every pass is bound by latency.  Placing by rank reads a row's
// keys from one contiguous run, a thread per particle: the insertion sort it replaces (a thread per
// row, each move a chain of dependent loads) took 80-90 us on the records of ten substeps of 800
// chain beads on 80^3, and a coupled step there 923 us where it now takes 450.
using site::block_exclusive_scan;
using site::kScanPerThread;
using site::kScanRows;
using site::kScanThreads;

using SortKey = unsigned long long;

__device__ __forceinline__ SortKey sort_key(int cx, int id) {
  return ((SortKey)(unsigned)cx << 32) | (unsigned)id;
}

// Counts particle p (in cell c) in its row, if `valid`.  Every thread of the warp calls it.
__device__ __forceinline__ void bin_particle(const StepParams &P, int p, bool valid, int4 c, const SortScratch &S) {
  const int row = valid ? c.z * P.ny + c.y : -1;
  if (valid) {
    S.row_of[p] = row;
    S.rank_of[p] = atomicAdd(S.row_count + row, 1);
  }
  // one addition per scan block a warp's particles fall in (they come nearly sorted: mostly one)
  const int blk = valid ? row / kScanRows : -1;
  const unsigned same = __match_any_sync(0xffffffffu, blk);
  if (valid && (int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(S.block_count + blk, __popc(same));
}

__global__ void __launch_bounds__(kPBlock) k_bin(StepParams P, ParticleArrays pa, SortScratch S, unsigned *err) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = p < P.np;
  int4 c = make_int4(0, 0, 0, 0);
  if (valid) {
    c = pa.cell[p];
    if (c.x < 0 || c.x >= P.nx || c.y < 0 || c.y >= P.ny || c.z < 0 || c.z >= P.nz) {
      atomicOr(err, kErrParticle);  // cannot happen for states written by this library
      c.x = wrapi(c.x, P.nx); c.y = wrapi(c.y, P.ny); c.z = wrapi(c.z, P.nz);
      pa.cell[p] = c;
    }
  }
  bin_particle(P, p, valid, c, S);
}

__device__ __forceinline__ void set_node_bits(const StepParams &P, int4 c, unsigned *node_bits) {
  site::for_corner_bits(P, c, [&](long long w, unsigned bits) { atomicOr(node_bits + w, bits); });
}
__device__ __forceinline__ void clear_node_bits(const StepParams &P, int4 c, unsigned *node_bits) {
  site::for_corner_bits(P, c, [&](long long w, unsigned) { node_bits[w] = 0u; });
}

// Particle update (site::integrate) from src into dst, in the same order, and the bin pass of the
// sort that follows it.  The nodes of the cells `marked` are cleared in node_bits.
__global__ void __launch_bounds__(kPBlock) k_integrate_bin(StepParams P, ParticleArrays src, ParticleArrays dst,
                                                           ParticleForces pf, SortScratch S,
                                                           const int4 *__restrict__ marked,
                                                           unsigned *__restrict__ node_bits, unsigned *err) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = p < P.np;
  if (valid) clear_node_bits(P, marked[p], node_bits);
  bin_particle(P, p, valid, valid ? site::integrate(P, p, src, dst, pf, err) : make_int4(0, 0, 0, 0), S);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_rows(int nrows, SortScratch S, int *__restrict__ start) {
  __shared__ int wt[kScanThreads / 32];
  int total;
  int before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += S.block_count[b];
  block_exclusive_scan(before, wt, total);
  before = total;  // particles in the rows of the blocks before this one
  __syncthreads();
  const int base = blockIdx.x * kScanRows + threadIdx.x * kScanPerThread;
  int c[kScanPerThread];
  int sum = 0;
#pragma unroll
  for (int k = 0; k < kScanPerThread; ++k) {
    c[k] = base + k < nrows ? S.row_count[base + k] : 0;
    sum += c[k];
  }
  int run = before + block_exclusive_scan(sum, wt, total);
#pragma unroll
  for (int k = 0; k < kScanPerThread; ++k)
    if (base + k < nrows) {
      start[base + k] = run;
      S.row_count[base + k] = 0;
      run += c[k];
    }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) start[nrows] = before + total;
}

__global__ void __launch_bounds__(kPBlock) k_scatter(int np, int nblocks, SortScratch S, const int *__restrict__ start,
                                                     const int4 *__restrict__ cell, const int *__restrict__ id) {
  if (blockIdx.x == 0)  // the block totals have been read: cleared for the next sort
    for (int b = threadIdx.x; b < nblocks; b += kPBlock) S.block_count[b] = 0;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const int row = S.row_of[p];
  const int j = start[row] + S.rank_of[p];
  S.perm[j] = p;
  S.row_at[j] = row;
  S.key[j] = sort_key(cell[p].x, id[p]);
}

// The slot of the entry scattered to j: the first slot of its row plus its rank there.
__device__ __forceinline__ int placed_slot(int j, const SortScratch &S, const int *__restrict__ start) {
  const int row = S.row_at[j];
  const SortKey key = S.key[j];
  const int b = start[row], e = start[row + 1];
  int slot = b;
  for (int q = b; q < e; ++q) slot += S.key[q] < key;
  return slot;
}

__device__ __forceinline__ void move_particle(const StepParams &P, const ParticleArrays &src, int p,
                                              const ParticleArrays &dst, int slot, int *__restrict__ slot_of_id,
                                              unsigned *__restrict__ node_bits) {
  const int id = src.pid[p];
  const int4 c = src.cell[p];
  if (node_bits) set_node_bits(P, c, node_bits);
  dst.cell[slot] = c;
  dst.frac[slot] = src.frac[p];
  dst.vel[slot] = src.vel[p];
  dst.pid[slot] = id;
  slot_of_id[id] = slot;
}

__global__ void __launch_bounds__(kPBlock) k_place(StepParams P, SortScratch S, const int *__restrict__ start,
                                                   ParticleArrays src, ParticleArrays dst,
                                                   int *__restrict__ slot_of_id, unsigned *__restrict__ node_bits) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= P.np) return;
  move_particle(P, src, S.perm[j], dst, placed_slot(j, S, start), slot_of_id, node_bits);
}

// The particle update (kUpdate) and the whole sort of a small system in one block, the counters,
// keys and slots in shared memory: one launch instead of four that a step of a small lattice would
// wait for.  The order is unique, so the result is that of the chain.  With 256 threads, insertion
// sorts per row and the update in a kernel before it, 1000 particles on 64^3 took 23 + 4 us and a
// coupled step 45 us; now the step takes 29.  The limits are what one block's shared memory holds
// with room to spare (112 KB); a step of 100 x 90 x 110 (9900 rows, 1000 particles) hides the four
// launches of the chain behind its lattice update.
constexpr int kSmallThreads = 1024;
constexpr int kSmallRows = 8192, kSmallNp = 4096;

inline size_t small_smem(int nrows, int np) { return sizeof(int) * (size_t)(nrows + 1) + (size_t)np * 20 + 16; }

template <bool kUpdate>
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(StepParams P, ParticleArrays src, ParticleArrays mid,
                                                              ParticleForces pf, ParticleArrays dst,
                                                              int *__restrict__ start, int *__restrict__ slot_of_id,
                                                              unsigned *__restrict__ node_bits, unsigned *err) {
  extern __shared__ SortKey small_keys[];
  __shared__ int wt[kSmallThreads / 32];
  const int np = P.np, nrows = P.nrows;
  SortKey *key = small_keys;                            // [np] by particle
  int *row_of = reinterpret_cast<int *>(key + np);      // [np]
  int *rank_of = row_of + np;                           // [np]
  int *list = rank_of + np;                             // [np] the particles of each row, in arrival order
  int *row = list + np;                                 // [nrows + 1] counters, then first slots
  for (int r = threadIdx.x; r <= nrows; r += kSmallThreads) row[r] = 0;
  __syncthreads();
  for (int p = threadIdx.x; p < np; p += kSmallThreads) {
    int4 c;
    if (kUpdate) {
      // dst still holds the particles whose nodes are set; it and the bits are written after the
      // barriers below
      clear_node_bits(P, dst.cell[p], node_bits);
      c = site::integrate(P, p, src, mid, pf, err);
    } else {
      c = mid.cell[p];
      if (c.x < 0 || c.x >= P.nx || c.y < 0 || c.y >= P.ny || c.z < 0 || c.z >= P.nz) {
        atomicOr(err, kErrParticle);  // cannot happen for states written by this library
        c.x = wrapi(c.x, P.nx); c.y = wrapi(c.y, P.ny); c.z = wrapi(c.z, P.nz);
        mid.cell[p] = c;
      }
    }
    const int r = c.z * P.ny + c.y;
    row_of[p] = r;
    rank_of[p] = atomicAdd(&row[r], 1);
    key[p] = sort_key(c.x, (kUpdate ? src : mid).pid[p]);
  }
  __syncthreads();
  const int per = (nrows + kSmallThreads - 1) / kSmallThreads;  // consecutive rows of a thread
  const int b0 = threadIdx.x * per;
  int sum = 0;
  for (int k = 0; k < per; ++k)
    if (b0 + k < nrows) sum += row[b0 + k];
  int total;
  int run = block_exclusive_scan<kSmallThreads>(sum, wt, total);
  for (int k = 0; k < per; ++k)
    if (b0 + k < nrows) {
      const int n = row[b0 + k];
      row[b0 + k] = run;
      start[b0 + k] = run;
      run += n;
    }
  if (threadIdx.x == 0) row[nrows] = start[nrows] = total;
  __syncthreads();
  for (int p = threadIdx.x; p < np; p += kSmallThreads) list[row[row_of[p]] + rank_of[p]] = p;
  __syncthreads();
  for (int p = threadIdx.x; p < np; p += kSmallThreads) {
    const int b = row[row_of[p]], e = row[row_of[p] + 1];
    const SortKey mine = key[p];
    int slot = b;
    for (int q = b; q < e; ++q) slot += key[list[q]] < mine;
    move_particle(P, mid, p, dst, slot, slot_of_id, node_bits);  // (this thread wrote entry p of mid)
  }
}

// Coupling forces of every particle (site::couple).
__global__ void __launch_bounds__(kPBlock) k_couple(StepParams P, ParticleArrays pa, CellIndex ci,
                                                    const float *__restrict__ rho, const float *__restrict__ jp,
                                                    ParticleForces pf) {
  // 8 lanes per particle (site::couple8): the group of a particle returns together
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = (int)(t >> 3), k = (int)(t & 7);
  if (p >= P.np) return;
  site::couple8(P, noise_step(P, P.step), p, k, 0xFFu << (threadIdx.x & 24), pa, ci, rho, jp, pf);
}

// k_couple with j' at each corner already formed (jc, 8 float4 per particle id).
__global__ void __launch_bounds__(kPBlock) k_couple_jc(StepParams P, ParticleArrays pa, CellIndex ci,
                                                       const float *__restrict__ rho, const float4 *__restrict__ jc,
                                                       ParticleForces pf) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = (int)(t >> 3), k = (int)(t & 7);
  if (p >= P.np) return;
  site::couple8(P, noise_step(P, P.step), p, k, 0xFFu << (threadIdx.x & 24), pa, ci, rho, nullptr, pf, jc);
}

// j' = sum_z sum_i f_zi c_i of the populations `store` at the 8 corners of every particle's cell,
// into jc[pid * 8 + corner] (the values k_couple_jc reads).
template <class T>
__global__ void __launch_bounds__(kPBlock) k_corner_jprime(StepParams P, ParticleArrays pa, int np,
                                                           const T *__restrict__ store, float4 *__restrict__ jc) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 8LL * np) return;
  const int p = (int)(t >> 3), k = (int)(t & 7);
  const site::Coord cc = site::cell_corner(P, __ldg(pa.cell + p), k);
  const float3 j = site::jprime_at<T>(P, store, cc.x, cc.y, cc.z);
  jc[(long long)__ldg(pa.pid + p) * 8 + k] = make_float4(j.x, j.y, j.z, 0.f);
}

// Pair and bonded forces of every particle (site::pairs).
__global__ void __launch_bounds__(kPBlock) k_pairs(StepParams P, ParticleArrays pa, CellIndex ci,
                                                   const int *__restrict__ bond_start,
                                                   const int *__restrict__ bond_other,
                                                   const int *__restrict__ slot_of_id, ParticleForces pf,
                                                   unsigned *err) {
  // 8 lanes per particle (site::pairs8): the group of a particle returns together
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = (int)(t >> 3), k = (int)(t & 7);
  if (p >= P.np) return;
  site::pairs8(P, p, k, 0xFFu << (threadIdx.x & 24), pa, ci, bond_start, bond_other, slot_of_id, pf, err);
}

// ------------------------------------------------------------------ MD sub-stepping

// One particle substep: the coupling and the pair forces at the particles' positions C (in the order
// of the step's sorted list S, whose rows and fluid-side solvation force stay frozen), the substep's
// reaction record -- position, friction and solvation forces over K, and the substep index in the
// cell's w (the fluid-side solvation force is taken from substep 0's records only) -- binned for the
// records' sort, and the update by P.dt = dt / K into D, with the check that each particle is still
// within one cell of where the step started (the rows of the step rely on it).
// A block takes 8 particles, 8 lanes each for the coupling (its first two warps) and for the pair
// forces (the others), which meet in shared memory.  Bound by latency: as three launches on two
// streams, working in place on a copy of S, a substep of 800 chain beads on 80^3 took 45 us and a
// lattice step with ten of them 450; this launch takes 18.5 and the step 245.
constexpr int kSubParticles = 8;
static_assert(kPBlock == 2 * 8 * kSubParticles, "two groups of 8 lanes per particle");

__global__ void __launch_bounds__(kPBlock) k_substep(StepParams P, ParticleArrays C, ParticleArrays D,
                                                     ParticleArrays S, CellIndex ci, int pair_reach,
                                                     const float *__restrict__ rho, const float *__restrict__ jp,
                                                     const int *__restrict__ bond_start,
                                                     const int *__restrict__ bond_other,
                                                     const int *__restrict__ slot_of_id, ParticleForces pf, int sub,
                                                     ReactionRecords rec, SortScratch rs,
                                                     const int4 *__restrict__ marked,
                                                     unsigned *__restrict__ node_bits, unsigned *err) {
  __shared__ float3 pair[kSubParticles];
  __shared__ site::CoupleForces coupled[kSubParticles];
  const int g = (threadIdx.x >> 3) & (kSubParticles - 1), k = threadIdx.x & 7;
  const int p = blockIdx.x * kSubParticles + g;
  const unsigned mask = 0xFFu << (threadIdx.x & 24);
  if (p < P.np) {  // the same for the 8 lanes of a group
    if (threadIdx.x < 8 * kSubParticles) {
      const site::CoupleForces F = site::couple_forces(P, noise_step(P, P.step), p, k, mask, C, S, ci, rho, jp, pf,
                                                       sub == 0, nullptr);
      if (k == 0) coupled[g] = F;
    } else {
      const float3 F = site::pair_forces(P, p, k, mask, C, ci, pair_reach, bond_start, bond_other, slot_of_id, err);
      if (k == 0) pair[g] = F;
    }
  }
  __syncthreads();
  if (threadIdx.x >= 32) {
    // the nodes that as many of the last step's records marked, by lanes with nothing else left to do; the
    // placing of this step's records, which sets theirs, follows the last substep.  (Clearing the lattice's
    // words in the first substep took the few blocks of few particles the longer: 8 on 2 x 1024 x 2048 with
    // four substeps 481 us a step for 353, on 256^3 with ten 1236 for 1204; 800 chain beads on 80^3 alike.)
    const int c = threadIdx.x - 32, m = blockIdx.x * kSubParticles + c;
    if (c < kSubParticles && m < P.np) clear_node_bits(P, marked[sub * P.np + m], node_bits);
    return;
  }
  const int q = blockIdx.x * kSubParticles + threadIdx.x;  // lane t of the first warp finishes particle t
  const bool valid = threadIdx.x < kSubParticles && q < P.np;
  int4 c = make_int4(0, 0, 0, 0);
  const int r = sub * P.np + q;
  if (valid) {
    const site::CoupleForces &F = coupled[threadIdx.x];
    const float invK = 1.f / (float)P.substeps;
    c = C.cell[q];
    rec.cell[r] = make_int4(c.x, c.y, c.z, c.w | (sub << 8));
    rec.frac[r] = C.frac[q];
    rec.key[r] = sub * P.np + C.pid[q];
    rec.fric[r] = make_float4(F.fric.x * invK, F.fric.y * invK, F.fric.z * invK, 0.f);
    rec.psA[r] = make_float4(F.psA.x * invK, F.psA.y * invK, F.psA.z * invK, 0.f);
    rec.psB[r] = make_float4(F.psB.x * invK, F.psB.y * invK, F.psB.z * invK, 0.f);
    float4 fsr = F.fsr;
    if (sub == 0)
      pf.fsr[q] = fsr;
    else
      fsr = pf.fsr[q];
    const float3 f = pair[threadIdx.x];
    const float3 total = site::total_force(F.fric, F.psA, F.psB, fsr, make_float4(f.x, f.y, f.z, 0.f));
    if (sub == P.substeps - 1) pf.total[q] = make_float4(total.x, total.y, total.z, 0.f);
    const int4 a = site::move_by(P, q, C, D, total, err), b = S.cell[q];
    const int dx = site::min_image_cells(a.x - b.x, P.nx), dy = site::min_image_cells(a.y - b.y, P.ny),
              dz = site::min_image_cells(a.z - b.z, P.nz);
    if (dx > 1 || dx < -1 || dy > 1 || dy < -1 || dz > 1 || dz < -1) atomicOr(err, kErrTooFast);
  }
  bin_particle(P, r, valid, c, rs);
}

__global__ void __launch_bounds__(kPBlock) k_rec_place(StepParams P, int n, SortScratch S,
                                                       const int *__restrict__ start, ReactionRecords src,
                                                       ReactionRecords dst, unsigned *__restrict__ node_bits) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int p = S.perm[j];
  const int4 c = src.cell[p];
  const float4 fr = src.frac[p], a = src.fric[p], b = src.psA[p], d = src.psB[p];
  const int slot = placed_slot(j, S, start);
  set_node_bits(P, c, node_bits);
  dst.cell[slot] = c;
  dst.frac[slot] = fr;
  dst.fric[slot] = a;
  dst.psA[slot] = b;
  dst.psB[slot] = d;
}

constexpr int kMomBlock = 256;
__global__ void __launch_bounds__(kMomBlock) k_particle_momentum(StepParams P, ParticleArrays pa,
                                                                 double *__restrict__ partial) {
  double acc[3] = {0.0, 0.0, 0.0};
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.np; p += gridDim.x * blockDim.x) {
    const float4 v = pa.vel[p];
    const double m = (double)P.types[pa.cell[p].w].mass;
    acc[0] += m * v.x;
    acc[1] += m * v.y;
    acc[2] += m * v.z;
  }
  __shared__ double sh[3][kMomBlock];
  for (int k = 0; k < 3; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = kMomBlock / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int k = 0; k < 3; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 3; ++k) partial[(long long)blockIdx.x * 3 + k] = sh[k][0];
}

// Particle state in the caller's order: entry j of the sorted arrays is particle pa.pid[j], and
// total force j is that of particle tid_of[j].  The ids are a permutation of 0..n-1; an id out of
// range (which no step writes) is skipped rather than written out of bounds.
__global__ void __launch_bounds__(kPBlock) k_particles_out(int n, ParticleArrays pa, const int *__restrict__ tid_of,
                                                           const float4 *__restrict__ total, double *__restrict__ x,
                                                           double *__restrict__ v, double *__restrict__ f) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int id = pa.pid[j];
  if (id >= 0 && id < n) {
    if (x) {
      const int4 c = pa.cell[j];
      const float4 q = pa.frac[j];
      x[3LL * id] = c.x + (double)q.x;  // exact: an integer plus an FP32 fraction fits FP64
      x[3LL * id + 1] = c.y + (double)q.y;
      x[3LL * id + 2] = c.z + (double)q.z;
    }
    if (v) {
      const float4 w = pa.vel[j];
      v[3LL * id] = w.x;
      v[3LL * id + 1] = w.y;
      v[3LL * id + 2] = w.z;
    }
  }
  if (f) {
    const int t = tid_of[j];
    if (t >= 0 && t < n) {
      const float4 g = total[j];
      f[3LL * t] = g.x;
      f[3LL * t + 1] = g.y;
      f[3LL * t + 2] = g.z;
    }
  }
}

}  // namespace

int scan_blocks(int nrows) { return (nrows + kScanRows - 1) / kScanRows; }

void launch_bin(const StepParams &P, const ParticleArrays &pa, const SortScratch &S, unsigned *err, cudaStream_t st) {
  k_bin<<<pgrid(P.np), kPBlock, 0, st>>>(P, pa, S, err);
}
void launch_integrate_bin(const StepParams &P, const ParticleArrays &src, const ParticleArrays &dst,
                          const ParticleForces &pf, const SortScratch &S, const int4 *marked, unsigned *node_bits,
                          unsigned *err, cudaStream_t st) {
  k_integrate_bin<<<pgrid(P.np), kPBlock, 0, st>>>(P, src, dst, pf, S, marked, node_bits, err);
}
// The scan and scatter passes of np binned entries.
static void scan_scatter(const StepParams &P, int np, const SortScratch &S, int *row_start, const int4 *cell,
                         const int *id, cudaStream_t st) {
  const int nb = scan_blocks(P.nrows);
  k_scan_rows<<<nb, kScanThreads, 0, st>>>(P.nrows, S, row_start);
  k_scatter<<<pgrid(np), kPBlock, 0, st>>>(np, nb, S, row_start, cell, id);
}
void launch_place(const StepParams &P, const SortScratch &S, const ParticleArrays &src, const ParticleArrays &dst,
                  int *row_start, int *slot_of_id, unsigned *node_bits, cudaStream_t st) {
  scan_scatter(P, P.np, S, row_start, src.cell, src.pid, st);
  k_place<<<pgrid(P.np), kPBlock, 0, st>>>(P, S, row_start, src, dst, slot_of_id, node_bits);
}
void launch_rec_place(const StepParams &P, int n, const SortScratch &S, const ReactionRecords &src,
                      const ReactionRecords &dst, int *row_start, unsigned *node_bits, cudaStream_t st) {
  scan_scatter(P, n, S, row_start, src.cell, src.key, st);
  k_rec_place<<<pgrid(n), kPBlock, 0, st>>>(P, n, S, row_start, src, dst, node_bits);
}

bool sort_fits_one_block(int nrows, int np) { return nrows <= kSmallRows && np <= kSmallNp; }

void launch_sort_small(const StepParams &P, const ParticleArrays *update_from, const ParticleArrays &mid,
                       const ParticleForces &pf, const ParticleArrays &dst, int *row_start, int *slot_of_id,
                       unsigned *node_bits, unsigned *err, cudaStream_t st) {
  const size_t smem = small_smem(P.nrows, P.np);
  const int most = (int)small_smem(kSmallRows, kSmallNp);
  if (update_from) {
    cudaFuncSetAttribute(k_sort_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    k_sort_small<true><<<1, kSmallThreads, smem, st>>>(P, *update_from, mid, pf, dst, row_start, slot_of_id, node_bits,
                                                             err);
  } else {
    cudaFuncSetAttribute(k_sort_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    k_sort_small<false><<<1, kSmallThreads, smem, st>>>(P, mid, mid, pf, dst, row_start, slot_of_id, node_bits, err);
  }
}

void launch_couple(const StepParams &P, const ParticleArrays &pa, CellIndex ci, const float *rho, const float *jp,
                   const ParticleForces &pf, cudaStream_t st) {
  k_couple<<<pgrid(8LL * P.np), kPBlock, 0, st>>>(P, pa, ci, rho, jp, pf);
}
void launch_couple_jc(const StepParams &P, const ParticleArrays &pa, CellIndex ci, const float *rho,
                      const float4 *jc, const ParticleForces &pf, cudaStream_t st) {
  k_couple_jc<<<pgrid(8LL * P.np), kPBlock, 0, st>>>(P, pa, ci, rho, jc, pf);
}
void launch_corner_jprime(const StepParams &P, const ParticleArrays &pa, int np, const void *store, float4 *jc,
                          cudaStream_t st) {
  if (np <= 0) return;
  switch (P.storage) {
    case LBMD_STORAGE_FP16_SHIFTED:
      k_corner_jprime<__half><<<pgrid(8LL * np), kPBlock, 0, st>>>(P, pa, np, static_cast<const __half *>(store), jc);
      break;
    case LBMD_STORAGE_BF16_SHIFTED:
      k_corner_jprime<__nv_bfloat16><<<pgrid(8LL * np), kPBlock, 0, st>>>(
          P, pa, np, static_cast<const __nv_bfloat16 *>(store), jc);
      break;
    default:
      k_corner_jprime<float><<<pgrid(8LL * np), kPBlock, 0, st>>>(P, pa, np, static_cast<const float *>(store), jc);
  }
}
void launch_pairs(const StepParams &P, const ParticleArrays &pa, CellIndex ci, const int *bond_start,
                  const int *bond_other, const int *slot_of_id, const ParticleForces &pf, unsigned *err,
                  cudaStream_t st) {
  k_pairs<<<pgrid(8LL * P.np), kPBlock, 0, st>>>(P, pa, ci, bond_start, bond_other, slot_of_id, pf, err);
}
void launch_substep(const StepParams &P, const ParticleArrays &C, const ParticleArrays &D, const ParticleArrays &S,
                    CellIndex ci, int pair_reach, const float *rho, const float *jp, const int *bond_start,
                    const int *bond_other, const int *slot_of_id, const ParticleForces &pf, int sub,
                    const ReactionRecords &rec, const SortScratch &rs, const int4 *marked, unsigned *node_bits,
                    unsigned *err, cudaStream_t st) {
  k_substep<<<(P.np + kSubParticles - 1) / kSubParticles, kPBlock, 0, st>>>(
      P, C, D, S, ci, pair_reach, rho, jp, bond_start, bond_other, slot_of_id, pf, sub, rec, rs, marked, node_bits,
      err);
}
void launch_particle_momentum(const StepParams &P, const ParticleArrays &pa, double *partial, int nblocks,
                              cudaStream_t st) {
  k_particle_momentum<<<nblocks, kMomBlock, 0, st>>>(P, pa, partial);
}
void launch_particles_out(int n, const ParticleArrays &pa, const int *tid_of, const float4 *total, double *x,
                          double *v, double *f, cudaStream_t st) {
  k_particles_out<<<pgrid(n), kPBlock, 0, st>>>(n, pa, tid_of, total, x, v, f);
}

}  // namespace lbmd
