// lb_fluid.cu -- lattice kernels of the coupled Shan-Chen LB / MD step (sm_103a).
//
// Storage: populations of both components in one buffer [19][nz][ny][nx][2] (structure of
// arrays over directions and sites, x fastest, the (A, B) pair of a direction at a node side by
// side, loaded and stored as one word).  The buffer holds the post-collision values f*(r, t-1)
// at their source node; a kernel "pulls" f_i(r, t) = f*_i(r - c_i, t-1), so reads are
// coalesced along x (shifted by at most one node) and writes are fully coalesced.  Element
// type: FP32, or a 16-bit type (FP16, BF16) holding the shifted value f_i - w_i rho0_z with the
// rest populations apart in FP32; all arithmetic is FP32.
#include <type_traits>

#include "lb_site.cuh"

namespace lbmd {

namespace {

constexpr int kBlock = 256;
// Blocks of the density pass and of the two-pass update, which wait for nothing within a block: small
// ones on large lattices, whose warps' slots are free again sooner (with 256 threads the slots of an
// update block stayed taken until its last warp was done: 17.7 of 24 warps active at 160^3).  Ten steps
// at 256^3 with the update in blocks of 256 / 128 / 64 / 32 threads: FP16 9.29 / 8.70 / 8.61 / 8.68 ms,
// fluctuating MRT 15.37 / 15.07 / 15.01 / 15.39; twenty of 100x90x110 MRT 2133 / 2101 / 2095 / 2155 us;
// 64 threads and the density pass in 256 / 128 / 64: FP16 8.61 / 8.58 / 8.58 ms.  A small lattice is
// launched in few waves, and starting more blocks costs it more: fifty steps of 64^3 1120 / 1111 / 1123 us,
// of 32^3 573 in 256 and 603 in 64; with the update of reaction records, whose blocks share the rows they
// search, ten steps of 80^3 take 14 % longer in 64 than in 256.  (More than 24 update warps an SM leave
// too few registers: 26 take 8.78 and 15.29 ms.)
constexpr long long kSmallBlocksFrom = 1 << 19;  // nodes
constexpr int kMomentsBlock = 128;
constexpr int kCollideBlock = 64;
constexpr int kUpdateThreads = 768;  // threads of the update per SM, 80 registers each

using namespace site;

// 8- and 4-byte asynchronous copies global -> shared (cp.async), their commit and wait.
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all_but_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

template <class T>
__global__ void __launch_bounds__(kBlock) k_init_equilibrium(StepParams P, const float *__restrict__ rhoA,
                                                             const float *__restrict__ rhoB,
                                                             const float *__restrict__ u, T *__restrict__ store,
                                                             float *__restrict__ rest) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  const Coord c = site_coord(P, s);
  const float ux = u ? u[3 * s] : 0.f, uy = u ? u[3 * s + 1] : 0.f, uz = u ? u[3 * s + 2] : 0.f;
  const float usq15 = 1.5f * (ux * ux + uy * uy + uz * uz);
  const float rc[2] = {rhoA[s], rhoB[s]};
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    // the post-streaming value at r is pulled from r - c_i: store it there
    const long long dst = site_index(P, wrapi(c.x - kCx[i], P.nx), wrapi(c.y - kCy[i], P.ny), wrapi(c.z - kCz[i], P.nz));
    const float cu = kCx[i] * ux + kCy[i] * uy + kCz[i] * uz;
    const float poly = 1.f + 3.f * cu + 4.5f * cu * cu - usq15;
#pragma unroll
    for (int z = 0; z < 2; ++z) pop_write(P, store, rest, z, i, dst, kW[i] * rc[z] * poly);
  }
}

template <class T>
__global__ void __launch_bounds__(kBlock) k_restream(StepParams P, const float *__restrict__ post, int comp,
                                                     T *__restrict__ store, float *__restrict__ rest) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  const Coord c = site_coord(P, s);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const long long dst = site_index(P, wrapi(c.x - kCx[i], P.nx), wrapi(c.y - kCy[i], P.ny), wrapi(c.z - kCz[i], P.nz));
    pop_write(P, store, rest, comp, i, dst, post[(long long)i * P.N + s]);
  }
}

template <class T>
__global__ void __launch_bounds__(kBlock) k_unstream(StepParams P, const T *__restrict__ store,
                                                     const float *__restrict__ rest, int comp,
                                                     float *__restrict__ post) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  const Coord c = site_coord(P, s);
  int xs[3], ys[3], zs[3];
  neighbours(P, c, xs, ys, zs);
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    post[(long long)i * P.N + s] = pop_read(P, store, rest, comp, i, pull_source(P, i, xs, ys, zs));
}

// Densities and j' of every site (site::moments).
template <class T>
__global__ void __launch_bounds__(kBlock) k_moments(StepParams P, const T *__restrict__ fin,
                                                    const float *__restrict__ rest, float *__restrict__ rho,
                                                    float *__restrict__ jp, const unsigned *__restrict__ node_bits) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  moments(P, s, fin, rest, rho, jp, node_bits);
}

// The lattice update of one step at every site (site::collide; with kMRT the fluctuating MRT
// collision, whose mode transforms spill a few registers at this budget of 24 warps per SM
// but run faster than without spills at 16; with kBisect the gather over the sub-stepping
// reaction records).
template <class T, bool kParticles, bool kMRT, bool kBisect = false, int kThreads = kBlock>
__global__ void __launch_bounds__(kThreads, kUpdateThreads / kThreads) k_collide(StepParams P, const T *__restrict__ fin,
                                                                  T *__restrict__ fout, const float *__restrict__ rho,
                                                                  ParticleArrays pa, ParticleForces pf, CellIndex ci,
                                                                  unsigned *err, const float *__restrict__ rest_in,
                                                                  float *__restrict__ rest_out) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  collide<T, kParticles, kMRT, kBisect>(P, s, P.step, fin, fout, rho, pa, pf, ci, err, rest_in, rest_out);
}

// ------------------------------------------------------------------ small lattices
//
// Density pass and update of a lattice without particles in one launch: a block forms the densities
// of its tile of 16 x 4 x 4 nodes and of the nodes around it (up to 648 for 256: the populations are
// read 2.5 times more than by a density pass, from L2 and L1, where a small lattice lives) in shared
// memory, then updates its nodes.  What bounds a small lattice is the chain of dependent launches; this
// halves it.  The same sums in the same order as the two kernels, so the same bits.  A step in two
// launches / one, us: 32^3 5.64 / 4.87, 45x37x29 6.92 / 6.42, 40^3 6.67 / 6.16, 48^3 8.06 / 9.48; 32^3 in
// FP16 5.03 / 4.62, with the fluctuating MRT collision 7.70 / 7.00.  (With particles the chain of
// coupling, particle update and sort bounds the step, and this form gains nothing.)
constexpr int kTileX = 16, kTileY = 4, kTileZ = 4;
static_assert(kTileX * kTileY * kTileZ == kBlock, "a thread per node of the tile");

struct TileRho {
  static constexpr bool kStaged = true;
  const float2 (*rho)[kTileY + 2][kTileX + 2];
  int x, y, z;  // this node in the tile, counted from the layer around it
  __device__ float2 operator()(int cx, int cy, int cz) const { return rho[z + cz][y + cy][x + cx]; }
};

// (the parameters of k_collide; rho, pa, pf and ci are not used)
template <class T, bool kMRT>
__global__ void __launch_bounds__(kBlock, 2) k_step_small(StepParams P, const T *__restrict__ fin,
                                                          T *__restrict__ fout, const float *__restrict__,
                                                          ParticleArrays pa, ParticleForces pf, CellIndex ci,
                                                          unsigned *err, const float *__restrict__ rest_in,
                                                          float *__restrict__ rest_out) {
  __shared__ float2 rho[kTileZ + 2][kTileY + 2][kTileX + 2];
  const int ntx = (P.nx + kTileX - 1) / kTileX, nty = (P.ny + kTileY - 1) / kTileY;
  const int tz = blockIdx.x / (ntx * nty), txy = blockIdx.x - tz * (ntx * nty), ty = txy / ntx;
  const int x0 = (txy - ty * ntx) * kTileX, y0 = ty * kTileY, z0 = tz * kTileZ;
  const int vx = min(kTileX, P.nx - x0), vy = min(kTileY, P.ny - y0), vz = min(kTileZ, P.nz - z0);
  constexpr int kAround = (kTileX + 2) * (kTileY + 2) * (kTileZ + 2);
#pragma unroll
  for (int r = 0; r < (kAround + kBlock - 1) / kBlock; ++r) {
    const int e = r * kBlock + threadIdx.x;
    const int hz = e / ((kTileX + 2) * (kTileY + 2)), hxy = e - hz * ((kTileX + 2) * (kTileY + 2));
    const int hy = hxy / (kTileX + 2), hx = hxy - hy * (kTileX + 2);
    if (hx > vx + 1 || hy > vy + 1 || hz > vz + 1) continue;
    const bool in_x = hx != 0 && hx != vx + 1, in_y = hy != 0 && hy != vy + 1, in_z = hz != 0 && hz != vz + 1;
    if (!in_x && !in_y && !in_z) continue;  // no neighbour of a node of the tile
    Coord c{x0 + hx - 1, y0 + hy - 1, z0 + hz - 1};
    c.x += c.x < 0 ? P.nx : c.x >= P.nx ? -P.nx : 0;
    c.y += c.y < 0 ? P.ny : c.y >= P.ny ? -P.ny : 0;
    c.z += c.z < 0 ? P.nz : c.z >= P.nz ? -P.nz : 0;
    const NodeMoments n = node_moments(P, c, (unsigned)site_index(P, c.x, c.y, c.z), fin, rest_in);
    rho[hz][hy][hx] = make_float2(n.rA, n.rB);
  }
  __syncthreads();
  const int x = threadIdx.x % kTileX, y = threadIdx.x / kTileX % kTileY, z = threadIdx.x / (kTileX * kTileY);
  if (x >= vx || y >= vy || z >= vz) return;
  const Coord c{x0 + x, y0 + y, z0 + z};
  const long long s = site_index(P, c.x, c.y, c.z);
  float fA[kQ], fB[kQ], rA, rB;
  collide_core_at<T, false, kMRT, false, TileRho>(P, c, s, P.step, fin, nullptr, pa, pf, ci, err, rest_in, fA, fB, rA,
                                                  rB, TileRho{rho, x + 1, y + 1, z + 1});
  store_node<T, kMRT>(P, (unsigned)s, fout, rest_out, fA, fB, rA, rB);
}

// ------------------------------------------------------------------ one-pass update
//
// Streaming carries f*_i(r) to r + c_i, so the next density of a node is the sum of the
// post-collision values arriving from its 19 sources: the update can form it from the values it
// has just computed instead of a second pass pulling every population again.  Each warp of a
// block owns one row y of an 8-row column tile and its 32 nodes x0 .. x0 + 31 (one per lane), and
// the block marches along z through one chunk of planes; the blocks of one chunk cover
// neighbouring tiles and are launched together, so that they march in step and the sectors they
// share meet in L2.  Per plane, for each of the 9 (c_y, c_z) groups of directions, a lane adds
// the values arriving at its node from c_x = 0, +1 (lane below) and -1 (lane above); the groups
// with c_y = +-1 go to the neighbouring rows through shared memory (double buffered: one barrier
// per plane), and each row adds what arrives at it into three accumulators, for the planes z - 1,
// z and z + 1.  After plane z the plane z - 1 is complete and is written.  What leaves the tile
// along x -- from lane 0 with c_x = -1, from the last lane with c_x = +1 -- is summed the same way
// into edge partials for the neighbouring tiles' edge nodes, which k_boundary_densities adds.  Every
// sum has a fixed order.  Nodes with sources in another block along y or z -- the first and last
// row of the tile, the first and last plane of the chunk -- get the same treatment: the block
// writes its part (across the tile's bottom and top rows per lane; for the planes below and at
// the chunk's start, and at and above its end, what its accumulators hold), and
// k_boundary_densities adds the parts of the two blocks.  Where a lattice is too thin for the
// partial sums (tiles of fewer than 3 rows or 2 columns; one plane), k_boundary_densities pulls
// those nodes' populations as the density pass does.
constexpr int kOPThreads = kOnePassRows * 32;
// the densities a block's stencils read in one plane: rows y0 - 1 .. y0 + 8, columns x0 - 1 ..
// x0 + 32
constexpr int kRhoRows = kOnePassRows + 2, kRhoCols = kOnePassCols + 2, kRhoSlots = 4;
static_assert(kOnePassCols == 32 && kRhoCols - 32 <= 32, "a warp stages a ring row with one or two copies per lane");
static_assert(kOnePassRows - 1 <= 15, "pair barriers 1 .. kOnePassRows - 1");

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// Named barrier `id` (1 .. 15; 0 is __syncthreads) for `n` threads of the block, all of whose
// warps take it convergently.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }

// The staged densities of a block's stencil: a ring of kRhoSlots planes.
struct StagedRho {
  static constexpr bool kStaged = true;
  const float2 (*ring)[kRhoRows][kRhoCols];
  int sm, s0, sp;  // slots of the planes z - 1, z, z + 1
  int k, j;        // this node's row and column in a plane
  __device__ float2 operator()(int cx, int cy, int cz) const {
    return ring[cz < 0 ? sm : (cz > 0 ? sp : s0)][k + cy][j + cx];
  }
};

// The elements of a staged plane: element e of the kRhoRows x kRhoCols rows y0 - 1 + e / kRhoCols,
// columns x0 - 1 + e % kRhoCols (both wrapped periodically) has the offset src[e] = y nx + x within
// a plane.  The same for every plane of a march: computed once per block, kept in shared memory
// (not in registers, which the update needs).
__device__ __forceinline__ void stage_sources(const StepParams &P, int x0, int y0, int *src) {
  for (int e = threadIdx.x; e < kRhoRows * kRhoCols; e += kOPThreads) {
    const int r = e / kRhoCols, j = e - r * kRhoCols;
    const int y = ((y0 - 1 + r) % P.ny + P.ny) % P.ny, x = ((x0 - 1 + j) % P.nx + P.nx) % P.nx;
    src[e] = y * P.nx + x;
  }
}

// The part of plane z's staged densities warp w copies (cp.async) into ring slot `slot_index` % 4:
// ring row w + 1, and the halo rows 0 (warp 0) and kRhoRows - 1 (the last warp).  The stencils
// of warp w read ring rows w .. w + 2, which warps w - 1 .. w + 1 copy.
__device__ __forceinline__ void stage_rows(const StepParams &P, const float *__restrict__ rho,
                                           float2 (*ring)[kRhoRows][kRhoCols], int slot_index, int z,
                                           const int *src, int w, int lane) {
  const float2 *plane = reinterpret_cast<const float2 *>(rho) + (long long)z * P.ny * P.nx;
  float2 *slot = &ring[slot_index & (kRhoSlots - 1)][0][0];
  auto row = [&](int r) {
    const int e = r * kRhoCols + lane;
    cp_async8(slot + e, plane + src[e]);
    if (lane < kRhoCols - 32) cp_async8(slot + e + 32, plane + src[e + 32]);
  };
  row(w + 1);
  if (w == 0) row(0);
  if (w == kOnePassRows - 1) row(kRhoRows - 1);
  cp_async_commit();
}

// Copies (cp.async) the densities of plane z into ring slot `slot_index` % 4 (the elements of
// stage_sources); every thread of the block takes part.  The slot follows the unwrapped plane
// index (z - 1 .. z + 2 of a march take four distinct slots even where the lattice is shorter than
// four planes).
__device__ __forceinline__ void stage_plane(const StepParams &P, const float *__restrict__ rho,
                                            float2 (*ring)[kRhoRows][kRhoCols], int slot_index, int z,
                                            const int *src) {
  const float2 *plane = reinterpret_cast<const float2 *>(rho) + (long long)z * P.ny * P.nx;
  float2 *slot = &ring[slot_index & (kRhoSlots - 1)][0][0];
  for (int e = threadIdx.x; e < kRhoRows * kRhoCols; e += kOPThreads) cp_async8(slot + e, plane + src[e]);
  cp_async_commit();
}

// The one-pass update of the tile and chunk of the block.  kMRT (FP32 storage): the fluctuating MRT collision,
// 1147 us at 256^3 with 20,000 particles for the two-pass update's 884 and its density pass's 376: bound by its
// arithmetic, 52.5 warp instructions per node.
template <class T, bool kParticles, bool kMRT = false>
__global__ void __launch_bounds__(kOPThreads, 3)
    k_collide_onepass(StepParams P, const T *__restrict__ fin, T *__restrict__ fout, const float *__restrict__ rho,
                      float *__restrict__ rho_next, OnePassOut out, ParticleArrays pa, ParticleForces pf,
                      CellIndex ci, unsigned *err, const float *__restrict__ rest_in, float *__restrict__ rest_out,
                      OnePassGeom G) {
  // groups handed to the neighbouring rows: [0..2] c_y = +1 with c_z = -1, 0, +1; [3..5] c_y = -1;
  // row w at index w + 1, indices 0 and kOnePassRows + 1 always 0 (the rows beyond the tile, whose
  // parts arrive as partial sums), so that a row adds its neighbours' without a select
  __shared__ float2 xch[2][6][kOnePassRows + 2][32];
  // the same for what leaves the tile along x: [side][c_y = +1, -1][row] (side 0: from lane 0
  // towards x0 - 1; side 1: from the last lane towards x0 + 32)
  __shared__ float2 xedge[2][2][2][kOnePassRows];
  // each thread's arrivals at its node, and each row's edge partials, in planes p with slot p % 3
  // (in shared memory rather than registers: they live across the whole update of a node)
  __shared__ float2 acc[3][kOPThreads];
  __shared__ float2 accE[3][2][kOnePassRows];
  // what leaves the tile across its bottom (0) and top (1) row, per lane
  __shared__ float2 accY[3][2][32];
  // the stencils' densities, read from global memory once per block and plane
  __shared__ float2 ring[kRhoSlots][kRhoRows][kRhoCols];
  __shared__ int stage_src[kRhoRows * kRhoCols];  // where each staged element comes from (stage_sources)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr unsigned kFull = 0xffffffffu;
  const int ncols = G.ntx * G.nty, chunk = blockIdx.x / ncols, col = blockIdx.x - chunk * ncols;
  const int zs = (int)((long long)chunk * P.nz / G.nchunks), ze = (int)((long long)(chunk + 1) * P.nz / G.nchunks);
  if (ze <= zs) return;  // block-uniform
  const int tx = col % G.ntx, ty = col / G.ntx;
  const int x0 = tx * kOnePassCols, nown = min(kOnePassCols, P.nx - x0);
  const bool own = lane < nown;
  const int x = own ? x0 + lane : x0;
  const int y0 = ty * kOnePassRows, rows = min(kOnePassRows, P.ny - y0);
  const int y = y0 + w;
  const bool inner_row = w >= 1 && w <= rows - 2;  // the sources along y are in the block
  const bool left = lane == 0, right = lane == nown - 1;  // the tile's x edges (both when nown = 1)
  acc[0][threadIdx.x] = acc[1][threadIdx.x] = acc[2][threadIdx.x] = make_float2(0.f, 0.f);
  for (int e = threadIdx.x; e < 2 * 6 * 2 * 32; e += kOPThreads) {
    const int r = (e >> 5) & 1, pg = e >> 6;
    xch[pg / 6][pg % 6][r ? kOnePassRows + 1 : 0][e & 31] = make_float2(0.f, 0.f);
  }
  if (threadIdx.x < 3 * 2 * kOnePassRows) (&accE[0][0][0])[threadIdx.x] = make_float2(0.f, 0.f);
  if (threadIdx.x < 3 * 2 * 32) (&accY[0][0][0])[threadIdx.x] = make_float2(0.f, 0.f);
  // rows whose partial sums the block forms: the inner ones, and with y partials the edge rows too
  // (lacking what arrives from the neighbouring tile's row, which that tile sends)
  const bool summed_row = w < rows && (G.ypart || inner_row);
  const bool lo = w > 0, hi = w < rows - 1;  // the rows below / above are in the block
  stage_sources(P, x0, y0, stage_src);
  __syncthreads();
  for (int dz = -1; dz <= 1; ++dz)
    stage_plane(P, rho, ring, zs + dz + kRhoSlots, (zs + dz + P.nz) % P.nz, stage_src);
  cp_async_wait_all();
  __syncthreads();
  int parity = 0;
  for (int z = zs; z < ze; ++z, parity ^= 1) {
    const int z2 = z + 2 < P.nz ? z + 2 : (z + 2) % P.nz;
    stage_rows(P, rho, ring, z + 2, z2, stage_src, w, lane);  // for the next plane; its slot is free
    float fA[kQ], fB[kQ];
    if (own && w < rows) {
      const long long s = ((long long)z * P.ny + y) * P.nx + x;
      float rA, rB;
      const StagedRho st{ring, (z + kRhoSlots - 1) & (kRhoSlots - 1), z & (kRhoSlots - 1),
                         (z + 1) & (kRhoSlots - 1), w + 1, lane + 1};
      collide_core_at<T, kParticles, kMRT, false, StagedRho>(P, Coord{x, y, z}, s, P.step, fin, rho, pa, pf, ci,
                                                              err, rest_in, fA, fB, rA, rB, st);
      store_node<T, kMRT, true, true>(P, (unsigned)s, fout, rest_out, fA, fB, rA, rB);
    } else {
#pragma unroll
      for (int i = 0; i < kQ; ++i) fA[i] = fB[i] = 0.f;
    }
    // arrivals of one (c_y, c_z) group at this lane's node: c_x = 0, +1 (from the lane below, none
    // for lane 0), -1 (from the lane above, none for the last lane)
    auto group = [&](int i0, int ip, int im) {
      float pA = __shfl_up_sync(kFull, fA[ip], 1), pB = __shfl_up_sync(kFull, fB[ip], 1);
      float mA = __shfl_down_sync(kFull, fA[im], 1), mB = __shfl_down_sync(kFull, fB[im], 1);
      if (lane == 0) pA = pB = 0.f;
      if (lane + 1 >= nown) mA = mB = 0.f;
      return add2(add2(make_float2(fA[i0], fB[i0]), make_float2(pA, pB)), make_float2(mA, mB));
    };
    float2(*X)[kOnePassRows + 2][32] = xch[parity];
    X[0][w + 1][lane] = make_float2(fA[17], fB[17]);  // (c_y, c_z) = (+1, -1)
    X[1][w + 1][lane] = group(3, 7, 10);              // (+1, 0)
    X[2][w + 1][lane] = make_float2(fA[15], fB[15]);  // (+1, +1)
    X[3][w + 1][lane] = make_float2(fA[16], fB[16]);  // (-1, -1)
    X[4][w + 1][lane] = group(4, 9, 8);               // (-1, 0)
    X[5][w + 1][lane] = make_float2(fA[18], fB[18]);  // (-1, +1)
    if (left) {  // leaving towards x0 - 1 with c_y = +1, -1
      xedge[parity][0][0][w] = make_float2(fA[10], fB[10]);
      xedge[parity][0][1][w] = make_float2(fA[8], fB[8]);
    }
    if (right) {  // leaving towards x0 + 32 with c_y = +1, -1
      xedge[parity][1][0][w] = make_float2(fA[7], fB[7]);
      xedge[parity][1][1][w] = make_float2(fA[9], fB[9]);
    }
    const float2 g0m = group(6, 13, 12), g00 = group(0, 1, 2), g0p = group(5, 11, 14);
    cp_async_wait_all();  // this warp's rows of the next plane's densities (issued above) have landed
    // The exchange with the rows below and above, and the staged rows they read: a barrier with
    // each neighbouring warp only (pair (w - 1, w) is barrier w), taken in that order.  A warp
    // passes plane z's barriers after its neighbours have written plane z's exchange and staged
    // rows, and writes the same buffers again (plane z + 2) only after they have passed plane
    // z + 1's, i.e. after they have read plane z's.
    if (w > 0) bar_sync(w, 64);
    if (w < kOnePassRows - 1) bar_sync(w + 1, 64);
    const int km = (z + 2) % 3, k0 = z % 3, kp = (z + 1) % 3;
    // plane z - 1 has all its sources (z - 2 .. z) in the chunk, or (with z partial sums) it is the
    // first plane of the chunk or the one below it, and this is the upper chunk's part
    const bool write = G.zpart || z >= zs + 2;
    const int zm = z == 0 ? P.nz - 1 : z - 1;
    const float2 zero = make_float2(0.f, 0.f);
    if (own && summed_row) {
      // from the row below (c_y = +1), this row (c_y = 0), the row above (c_y = -1), into the
      // planes z - 1, z, z + 1 (rows beyond the block and the rows of a ragged tile's absent
      // warps hold 0)
      const float2 am = add2(add2(add2(acc[km][threadIdx.x], X[0][w][lane]), g0m), X[3][w + 2][lane]);
      acc[k0][threadIdx.x] = add2(add2(add2(acc[k0][threadIdx.x], X[1][w][lane]), g00), X[4][w + 2][lane]);
      acc[kp][threadIdx.x] = add2(add2(add2(acc[kp][threadIdx.x], X[2][w][lane]), g0p), X[5][w + 2][lane]);
      if (write)
        reinterpret_cast<float2 *>(rho_next)[((long long)zm * P.ny + y) * P.nx + x] =
            add2(am, make_float2(shift_sum(P, 0), shift_sum(P, 1)));
      acc[km][threadIdx.x] = zero;  // becomes plane z + 2
    }
    if (summed_row && (left || right)) {
      // what leaves the tile along x, for the neighbouring tiles' edge nodes in this row: the
      // side-0 sums from lane 0 (c_x = -1: directions 2, 10, 8, 14, 12), the side-1 sums from the
      // last lane (c_x = +1: 1, 7, 9, 11, 13)
      float2 *edge2 = reinterpret_cast<float2 *>(out.edge);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 0 ? !left : !right) continue;
        const int i00 = side ? 1 : 2, i0p = side ? 11 : 14, i0m = side ? 13 : 12;
        const float2 em = add2(accE[km][side][w], make_float2(fA[i0m], fB[i0m]));
        accE[k0][side][w] = add2(add2(add2(accE[k0][side][w], lo ? xedge[parity][side][0][w - 1] : zero),
                                      make_float2(fA[i00], fB[i00])),
                                 hi ? xedge[parity][side][1][w + 1] : zero);
        accE[kp][side][w] = add2(accE[kp][side][w], make_float2(fA[i0p], fB[i0p]));
        if (write) edge2[(((long long)zm * P.ny + y) * G.ntx + tx) * 2 + side] = em;
        accE[km][side][w] = zero;
      }
    }
    if (G.ypart && own && (w == 0 || w == rows - 1)) {
      // what leaves the tile across its bottom row (the c_y = -1 groups of row 0) or its top row
      // (the c_y = +1 groups of the last row), for the neighbouring tile's edge row
      const int sy = w == 0 ? 0 : 1, g = sy ? 0 : 3;
      const float2 ym = add2(accY[km][sy][lane], X[g][w + 1][lane]);
      accY[k0][sy][lane] = add2(accY[k0][sy][lane], X[g + 1][w + 1][lane]);
      accY[kp][sy][lane] = add2(accY[kp][sy][lane], X[g + 2][w + 1][lane]);
      if (write)
        reinterpret_cast<float2 *>(out.yedge)[(((long long)sy * P.nz + zm) * G.nty + ty) * (G.ntx * kOnePassCols) +
                                              x0 + lane] = ym;
      accY[km][sy][lane] = zero;
      // the value leaving each corner diagonally (c_z = 0: it arrives in this plane)
      if ((left || right) && (G.zpart || (z >= zs + 1 && z <= ze - 2))) {
        const int k = (sy << 1) | (right ? 1 : 0);  // 0: bottom-left ... 3: top-right
        // directions 8, 9, 10, 7 (constant indices: the arrays stay in registers)
        const float2 d = sy ? (right ? make_float2(fA[7], fB[7]) : make_float2(fA[10], fB[10]))
                            : (right ? make_float2(fA[9], fB[9]) : make_float2(fA[8], fB[8]));
        reinterpret_cast<float2 *>(out.diag)[(((long long)z * G.nty + ty) * G.ntx + tx) * 4 + k] = d;
      }
    }
  }
  if (G.zpart) {
    // this chunk's part of the planes ze - 1 and ze, the first two planes of the boundary with the
    // next chunk (slots 2 b, 2 b + 1): what the last iteration left in the accumulators
    const int b = chunk + 1 == G.nchunks ? 0 : chunk + 1;
    const int k0 = (ze - 1) % 3, kp = ze % 3;
    if (own && summed_row) {
      float2 *zo = reinterpret_cast<float2 *>(out.zown);
      zo[((long long)(2 * b) * P.ny + y) * P.nx + x] = acc[k0][threadIdx.x];
      zo[((long long)(2 * b + 1) * P.ny + y) * P.nx + x] = acc[kp][threadIdx.x];
    }
    if (summed_row && (left || right)) {
      float2 *ze2 = reinterpret_cast<float2 *>(out.zedge);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 0 ? !left : !right) continue;
        ze2[(((long long)(2 * b) * P.ny + y) * G.ntx + tx) * 2 + side] = accE[k0][side][w];
        ze2[(((long long)(2 * b + 1) * P.ny + y) * G.ntx + tx) * 2 + side] = accE[kp][side][w];
      }
    }
    if (G.ypart && own && (w == 0 || w == rows - 1)) {
      const int sy = w == 0 ? 0 : 1;
      float2 *zy = reinterpret_cast<float2 *>(out.zyedge);
      const long long stride = (long long)G.nty * G.ntx * kOnePassCols;
      zy[((long long)sy * 2 * G.nchunks + 2 * b) * stride + (long long)ty * G.ntx * kOnePassCols + x0 + lane] =
          accY[k0][sy][lane];
      zy[((long long)sy * 2 * G.nchunks + 2 * b + 1) * stride + (long long)ty * G.ntx * kOnePassCols + x0 + lane] =
          accY[kp][sy][lane];
    }
  }
  cp_async_wait_all();  // no copy outlives the block
}

// The nodes the one-pass update leaves unfinished, in one launch of four block ranges:
//  1. the boundary runs, a warp per run: their densities from the new populations, as the density
//     pass computes them (without y partials the first and last row of each tile; without z
//     partials the first and last plane of each chunk);
//  2. the x-edge nodes of the inner rows: own partial (in rho_next) plus what arrives from the
//     neighbouring tile -- from the left one's side-1 sums at x0, from the right one's side-0 sums
//     at x0 + nown - 1 (both, in that order, when a tile has one column);
//  3. with y partials, the edge rows: own partial plus what the tile below (for the bottom row) or
//     above (for the top row) sends across, and at the two corners also the x-neighbour's edge-row
//     sums and the value the diagonal neighbour sends, in that order;
//  4. with z partials, the other nodes of the chunk-edge planes: own partial plus the lower
//     chunk's.
// In ranges 2 and 3 a chunk-edge plane's node adds the lower chunk's part after each term.  The
// sets of nodes are disjoint, and every node's sum has a fixed order.
// Bound by latency and by its scattered sectors: ranges 3 and 4 take kVec neighbouring nodes a thread (2
// where rows start on 16 bytes, nx even), indices by multiplication.  At 256^3: 45 us, with a node a thread and
// divisions 66; the next step's corner j' (33 us) runs on the side stream beside it, with it in one launch the two
// took 95.
template <int kVec>
struct NodeRun {
  float2 v[kVec];
  __device__ __forceinline__ void load(const float2 *p) {
    if constexpr (kVec == 2) {
      const float4 w = *reinterpret_cast<const float4 *>(p);
      v[0] = make_float2(w.x, w.y);
      v[1] = make_float2(w.z, w.w);
    } else {
      v[0] = *p;
    }
  }
  __device__ __forceinline__ void store(float2 *p) const {
    if constexpr (kVec == 2)
      *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    else
      *p = v[0];
  }
  __device__ __forceinline__ void add(const NodeRun &o) {
#pragma unroll
    for (int k = 0; k < kVec; ++k) v[k] = add2(v[k], o.v[k]);
  }
};

struct BoundaryBlocks {
  unsigned runs, edge, row;  // blocks of the ranges 1, 2 and 3 (the rest: 4)
  FastDiv by_ntx, by_nty, by_run;  // by the column tiles along x and y, and by nx / kVec
};

template <class T, int kVec>
__global__ void __launch_bounds__(kBlock) k_boundary_densities(StepParams P, OnePassGeom G, BoundaryBlocks D,
                                                               const T *__restrict__ store,
                                                               const float *__restrict__ rest,
                                                               float *__restrict__ rho_next,
                                                               const BoundaryRun *__restrict__ runs, int nruns,
                                                               OnePassOut out, const int *__restrict__ zslot) {
  unsigned bid = blockIdx.x;
  if (bid < D.runs) {
    const int r = (int)bid * (kBlock / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= nruns) return;
    const BoundaryRun b = runs[r];
    if (lane >= b.n) return;
    moments(P, (long long)b.row * P.nx + b.x0 + lane, store, rest, rho_next, nullptr);
    return;
  }
  bid -= D.runs;
  const float2 *e2 = reinterpret_cast<const float2 *>(out.edge);
  const float2 *zo = reinterpret_cast<const float2 *>(out.zown);
  const float2 *ze2 = reinterpret_cast<const float2 *>(out.zedge);
  float2 *rho2 = reinterpret_cast<float2 *>(rho_next);
  const unsigned nx = (unsigned)P.nx, ny = (unsigned)P.ny, ntx = (unsigned)G.ntx, nty = (unsigned)G.nty;
  // 32-bit index arithmetic: 19 N < 2^32.  The longest array, the y-edge sums padded to whole tiles along x, has
  // 2 nz nty 32 ntx entries, with at least 2 columns and 3 rows (ypart) at most 32 / 3 of N
  if (bid < D.edge) {
    const unsigned t = bid * kBlock + threadIdx.x;
    if (t >= (unsigned)P.nz * ny * ntx) return;
    const unsigned r = fast_div(t, D.by_ntx), tx = t - r * ntx;  // r = z * ny + y
    const unsigned z = fast_div(r, P.divy), y = r - z * ny;
    const int w = (int)(y % kOnePassRows), rows = min(kOnePassRows, P.ny - (int)(y - w));
    if (w < 1 || w > rows - 2) return;  // tile edge rows: runs, or range 3
    const int q = zslot[z];             // chunk-edge plane: its slot in the z arrays
    if (q >= 0 && !G.zpart) return;     // runs
    const unsigned x0 = tx * kOnePassCols, nown = min((unsigned)kOnePassCols, nx - x0);
    const unsigned txl = tx == 0 ? ntx - 1 : tx - 1, txr = tx == ntx - 1 ? 0 : tx + 1;
    const unsigned base = r * nx;
    const unsigned zr = (unsigned)q * ny + y, zb = zr * nx;  // this row in the z arrays (q >= 0)
    const unsigned xr = x0 + nown - 1;
    float2 v = rho2[base + x0], vr = rho2[base + xr];
    const float2 el = e2[(r * ntx + txl) * 2 + 1];  // from the left tile's last lane
    const float2 er = e2[(r * ntx + txr) * 2 + 0];  // and from the right tile's lane 0
    if (q >= 0) v = add2(v, zo[zb + x0]);
    v = add2(v, el);
    if (q >= 0) v = add2(v, ze2[(zr * ntx + txl) * 2 + 1]);
    if (nown == 1)
      vr = v;
    else if (q >= 0)
      vr = add2(vr, zo[zb + xr]);
    vr = add2(vr, er);
    if (q >= 0) vr = add2(vr, ze2[(zr * ntx + txr) * 2 + 0]);
    if (nown > 1) rho2[base + x0] = v;
    rho2[base + xr] = vr;
    return;
  }
  bid -= D.edge;
  const unsigned run = nx / kVec;  // threads per row
  if (bid < D.row) {
    // 3: edge rows (y partials): thread per (z, tile row, bottom / top, kVec nodes)
    const unsigned t = bid * kBlock + threadIdx.x;
    if (t >= (unsigned)P.nz * nty * 2 * run) return;
    const unsigned qq = fast_div(t, D.by_run), x = (t - qq * run) * kVec, sy = qq & 1u;
    const unsigned zt = qq >> 1, z = fast_div(zt, D.by_nty), ty = zt - z * nty;
    const int q = zslot[z];
    if (q >= 0 && !G.zpart) return;  // runs
    const unsigned y0 = ty * kOnePassRows, rows = min((unsigned)kOnePassRows, ny - y0), y = sy ? y0 + rows - 1 : y0;
    const unsigned tx = x / kOnePassCols, x0 = tx * kOnePassCols, nown = min((unsigned)kOnePassCols, nx - x0);
    const unsigned txl = tx == 0 ? ntx - 1 : tx - 1, txr = tx == ntx - 1 ? 0 : tx + 1;
    const unsigned tyn = sy ? (ty == nty - 1 ? 0 : ty + 1) : (ty == 0 ? nty - 1 : ty - 1);  // the tile sending across
    const float2 *y2 = reinterpret_cast<const float2 *>(out.yedge);
    const float2 *zy = reinterpret_cast<const float2 *>(out.zyedge);
    const float2 *d2 = reinterpret_cast<const float2 *>(out.diag);
    const unsigned er = z * ny + y, zr = (unsigned)q * ny + y, node = er * nx + x;
    const unsigned ystride = ntx * kOnePassCols;
    NodeRun<kVec> v, part;
    v.load(rho2 + node);
    // the bottom row gets what the tile below sends up (its side 1), the top row what the tile
    // above sends down (its side 0)
    part.load(y2 + (((1 - sy) * (unsigned)P.nz + z) * nty + tyn) * ystride + x);
    if (q >= 0) {
      NodeRun<kVec> below;
      below.load(zo + zr * nx + x);
      v.add(below);
    }
    v.add(part);
    if (q >= 0) {
      part.load(zy + (((1 - sy) * 2 * (unsigned)G.nchunks + (unsigned)q) * nty + tyn) * ystride + x);
      v.add(part);
    }
    if (x == x0) {  // corner: the left tile's side-1 sums of this row, the diagonal value
      float2 &c = v.v[0];
      c = add2(c, e2[(er * ntx + txl) * 2 + 1]);
      if (q >= 0) c = add2(c, ze2[(zr * ntx + txl) * 2 + 1]);
      c = add2(c, d2[((z * nty + tyn) * ntx + txl) * 4 + (sy ? 1 : 3)]);
    }
    if (x + kVec - 1 == x0 + nown - 1) {  // corner: the right tile's side-0 sums of this row, the diagonal value
      float2 &c = v.v[kVec - 1];
      c = add2(c, e2[(er * ntx + txr) * 2 + 0]);
      if (q >= 0) c = add2(c, ze2[(zr * ntx + txr) * 2 + 0]);
      c = add2(c, d2[((z * nty + tyn) * ntx + txr) * 4 + (sy ? 0 : 2)]);
    }
    v.store(rho2 + node);
    return;
  }
  bid -= D.row;
  // 4: the other nodes of the chunk-edge planes (z partials): thread per (slot, y, kVec nodes)
  const unsigned t = bid * kBlock + threadIdx.x;
  if (t >= 2u * (unsigned)G.nchunks * ny * run) return;
  const unsigned qy = fast_div(t, D.by_run), x = (t - qy * run) * kVec;
  const unsigned q = fast_div(qy, P.divy), y = qy - q * ny;
  const int w = (int)(y % kOnePassRows), rows = min(kOnePassRows, P.ny - (int)(y - w));
  if (w < 1 || w > rows - 2) return;  // tile edge rows: runs, or range 3
  const unsigned xt = x % kOnePassCols, nown = min((unsigned)kOnePassCols, nx - (x - xt));
  // x edges: range 2 (which stores them; they are not written here)
  const bool first = xt != 0, last = xt + kVec - 1 != nown - 1;
  if (kVec == 1 && (!first || !last)) return;
  // the plane of slot q: zs - 1 (q even) or zs (q odd) of chunk q / 2
  const unsigned zs = (unsigned)((unsigned long long)(q >> 1) * P.nz / G.nchunks);
  const unsigned z = (q & 1) ? zs : (zs == 0 ? P.nz - 1 : zs - 1);
  const unsigned at = y * nx + x, node = z * ny * nx + at;
  if (first && last) {
    NodeRun<kVec> v, part;
    v.load(rho2 + node);
    part.load(zo + q * ny * nx + at);
    v.add(part);
    v.store(rho2 + node);
  } else if (kVec == 2 && first) {
    rho2[node] = add2(rho2[node], zo[q * ny * nx + at]);
  } else if (kVec == 2 && last) {
    rho2[node + 1] = add2(rho2[node + 1], zo[q * ny * nx + at + 1]);
  }
}

// rho_A, rho_B and u = (j' + g^SC/2)/rho at the current step (for readback; any output may be null:
// without u the populations are not read).  Bound by HBM: 152 B of populations, 8 of densities and 20
// of results per node in FP32: 467 us at 256^3, 6.5 TB/s (578 with a load for each component and 64-bit
// neighbour addresses).
template <class T>
__global__ void __launch_bounds__(kBlock) k_fields(StepParams P, const T *__restrict__ store,
                                                   const float *__restrict__ rest,
                                                   const float *__restrict__ rho, float *__restrict__ oA,
                                                   float *__restrict__ oB, float *__restrict__ ou) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= P.N) return;
  const unsigned s32 = (unsigned)s;
  const float2 *rho2 = reinterpret_cast<const float2 *>(rho);
  const float2 r0 = __ldg(rho2 + s32);
  if (oA) oA[s] = r0.x;
  if (oB) oB[s] = r0.y;
  if (!ou) return;
  const NOff o = neighbour_offsets(P, site_coord(P, s));
  float2 f[kQ];
#pragma unroll
  for (int i = 1; i < kQ; ++i)  // (the rest populations carry no momentum)
    f[i] = pop_pair<T>(P, store, rest, i, (unsigned)((int)s32 + shift(o, -kCx[i], -kCy[i], -kCz[i])));
  float jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    const float a = f[i].x + f[i].y;
    jx += kCx[i] * a; jy += kCy[i] * a; jz += kCz[i] * a;
  }
  const float rA = r0.x, rB = r0.y;
  float SAx = 0.f, SAy = 0.f, SAz = 0.f, SBx = 0.f, SBy = 0.f, SBz = 0.f;
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    const float2 r = __ldg(rho2 + (unsigned)((int)s32 + shift(o, kCx[i], kCy[i], kCz[i])));
    const float a = kW[i] * r.x, b = kW[i] * r.y;
    SAx += kCx[i] * a; SAy += kCy[i] * a; SAz += kCz[i] * a;
    SBx += kCx[i] * b; SBy += kCy[i] * b; SBz += kCz[i] * b;
  }
  const float gx = -P.gAB * rA * SBx - P.gBA * rB * SAx;
  const float gy = -P.gAB * rA * SBy - P.gBA * rB * SAy;
  const float gz = -P.gAB * rA * SBz - P.gBA * rB * SAz;
  const float rinv = 1.f / (rA + rB);
  ou[3 * s] = (jx + 0.5f * gx) * rinv;
  ou[3 * s + 1] = (jy + 0.5f * gy) * rinv;
  ou[3 * s + 2] = (jz + 0.5f * gz) * rinv;
}

// FP64 block partial sums of [M_A, M_B, Px, Py, Pz] over the stored buffer (site::TotalSums).
// Bound by HBM once enough loads are in flight: with loads into registers the compiler kept a few
// per thread at a time (2 TB/s, 1008 us at 256^3, whatever the arithmetic).  Each thread copies its
// next node's values into a slot of its own in shared memory (cp.async, no barriers) while it adds
// the present one's: 497 us, 5.1 TB/s.  Five blocks fit an SM.
constexpr int kSumBlock = 128;
constexpr int kSumGrid = 5 * 152;
template <class T>
__global__ void __launch_bounds__(kSumBlock) k_fluid_sums(StepParams P, const T *__restrict__ store,
                                                          const float *__restrict__ rest,
                                                          double *__restrict__ partial) {
  // FP32: the (A, B) pair of each direction; 16-bit: its word, the rest pair in two more
  using Word = std::conditional_t<kSplitRest<T>, unsigned, float2>;
  constexpr int kWords = kSplitRest<T> ? kQ + 1 : kQ;
  __shared__ Word stage[2][kWords][kSumBlock];
  const unsigned N32 = (unsigned)P.N, stride = gridDim.x * kSumBlock;
  auto fetch = [&](int k, unsigned s) {
    const Word *src = reinterpret_cast<const Word *>(store) + s;
    if constexpr (kSplitRest<T>) {
#pragma unroll
      for (int i = 1; i < kQ; ++i) cp_async4(&stage[k][i][threadIdx.x], src + (size_t)i * N32);
      cp_async4(&stage[k][0][threadIdx.x], rest + s);
      cp_async4(&stage[k][kQ][threadIdx.x], rest + N32 + s);
    } else {
#pragma unroll
      for (int i = 0; i < kQ; ++i) cp_async8(&stage[k][i][threadIdx.x], src + (size_t)i * N32);
    }
  };
  TotalSums sums;
  unsigned s = blockIdx.x * kSumBlock + threadIdx.x;
  if (s < N32) fetch(0, s);
  cp_async_commit();
  for (int k = 0; s < N32; k ^= 1) {
    const unsigned next = s + stride;  // N + stride < 2^32: 19 N is
    if (next < N32) fetch(k ^ 1, next);
    cp_async_commit();
    cp_async_wait_all_but_one();
    sums.add([&](int i) {
      if constexpr (kSplitRest<T>) {
        if (i == 0)
          return make_float2(__uint_as_float(stage[k][0][threadIdx.x]), __uint_as_float(stage[k][kQ][threadIdx.x]));
        const float2 v = Pair16<T>::dec(stage[k][i][threadIdx.x]);
        return make_float2(v.x + pop_shift(P, 0, i), v.y + pop_shift(P, 1, i));
      } else {
        return stage[k][i][threadIdx.x];
      }
    });
    s = next;
  }
  cp_async_wait_all();
  sums.flush();
  const double *acc = sums.acc;
  __shared__ double sh[5][kSumBlock];
#pragma unroll
  for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = kSumBlock / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < 5; ++k) partial[(long long)blockIdx.x * 5 + k] = sh[k][0];
}

__global__ void k_finish_sums(const double *__restrict__ partial, int nblocks, int nvals, double *__restrict__ out) {
  // one warp per value: lane l adds the blocks l, l + 32, ... in order, then a fixed shuffle tree
  // (deterministic; 32 chains instead of one long chain of dependent FP64 additions)
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (k >= nvals) return;  // warp-uniform
  double a = 0.0;
  for (int b = lane; b < nblocks; b += 32) a += partial[(long long)b * nvals + k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if (lane == 0) out[k] = a;
}

// The drift check of the conserved totals (appendix: the collision and the forcing term keep
// each component's mass; Sec. 2: the momentum of fluid and particles together).
__global__ void k_drift_check(const double *__restrict__ sums, const double *__restrict__ psum, double *ref,
                              double *last, unsigned *err, long long step, double tol, int set_ref) {
  double t[5];
  for (int k = 0; k < 5; ++k) t[k] = sums[k] + (k >= 2 && psum ? psum[k - 2] : 0.0);
  if (set_ref) {
    for (int k = 0; k < 5; ++k) ref[k] = t[k];
    last[0] = -1.0;
    last[1] = last[2] = last[3] = 0.0;
    last[4] = 0.0;
    return;
  }
  const double dA = fabs(t[0] - ref[0]) / fabs(ref[0]), dB = fabs(t[1] - ref[1]) / fabs(ref[1]);
  const double px = t[2] - ref[2], py = t[3] - ref[3], pz = t[4] - ref[4];
  const double dP = sqrt(px * px + py * py + pz * pz) / (fabs(ref[0]) + fabs(ref[1]));
  last[0] = (double)step;
  last[1] = dA;
  last[2] = dB;
  last[3] = dP;
  last[4] += 1.0;
  // NaN drifts fail the comparison below as well
  if (!(dA <= tol) || !(dB <= tol) || !(dP <= tol)) atomicOr(err, kErrDrift);
}

inline unsigned grid_for(long long n, int block = kBlock) { return (unsigned)((n + block - 1) / block); }

}  // namespace

// Run `f` with a typed null pointer of the storage element type of P.
template <class F>
void with_storage(const StepParams &P, F f) {
  switch (P.storage) {
    case LBMD_STORAGE_FP16_SHIFTED: f((__half *)nullptr); break;
    case LBMD_STORAGE_BF16_SHIFTED: f((__nv_bfloat16 *)nullptr); break;
    default: f((float *)nullptr); break;
  }
}

void launch_init_equilibrium(const StepParams &P, const float *rhoA, const float *rhoB, const float *u,
                             void *store, float *rest, cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    k_init_equilibrium<T><<<grid_for(P.N), kBlock, 0, st>>>(P, rhoA, rhoB, u, static_cast<T *>(store), rest);
  });
}
void launch_restream(const StepParams &P, const float *post, int comp, void *store, float *rest, cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    k_restream<T><<<grid_for(P.N), kBlock, 0, st>>>(P, post, comp, static_cast<T *>(store), rest);
  });
}
void launch_unstream(const StepParams &P, const void *store, const float *rest, int comp, float *post,
                     cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    k_unstream<T><<<grid_for(P.N), kBlock, 0, st>>>(P, static_cast<const T *>(store), rest, comp, post);
  });
}
void launch_moments(const StepParams &P, const void *store, const float *rest, float *rho, float *jp,
                    const unsigned *node_bits, cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    const int block = P.N >= kSmallBlocksFrom ? kMomentsBlock : kBlock;
    k_moments<T><<<grid_for(P.N, block), block, 0, st>>>(P, static_cast<const T *>(store), rest, rho, jp, node_bits);
  });
}
void launch_step_small(const StepParams &P, const void *fin, void *fout, const float *rest_in, float *rest_out,
                       unsigned *err, cudaStream_t st) {
  auto tiles = [](int n, int edge) { return (unsigned)((n + edge - 1) / edge); };
  const unsigned grid = tiles(P.nx, kTileX) * tiles(P.ny, kTileY) * tiles(P.nz, kTileZ);
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    auto *kernel = P.collision == LBMD_COLLISION_MRT ? k_step_small<T, true> : k_step_small<T, false>;
    kernel<<<grid, kBlock, 0, st>>>(P, static_cast<const T *>(fin), static_cast<T *>(fout), nullptr, ParticleArrays{},
                                    ParticleForces{}, CellIndex{}, err, rest_in, rest_out);
  });
}

void launch_collide(const StepParams &P, const void *fin, void *fout, const float *rest_in, float *rest_out,
                    const float *rho, const ParticleArrays &pa, const ParticleForces &pf, CellIndex ci, unsigned *err,
                    cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    const T *a = static_cast<const T *>(fin);
    T *b = static_cast<T *>(fout);
    const bool mrt = P.collision == LBMD_COLLISION_MRT;
    const bool records = P.np > 0 && P.substeps > 1, parts = P.np > 0;
    constexpr int kC = kCollideBlock;
    const bool large = P.N >= kSmallBlocksFrom && !records;
    const int block = large ? kC : kBlock;
    auto *kernel = records ? (mrt ? k_collide<T, true, true, true> : k_collide<T, true, false, true>)
                   : large ? (parts ? (mrt ? k_collide<T, true, true, false, kC> : k_collide<T, true, false, false, kC>)
                                    : (mrt ? k_collide<T, false, true, false, kC> : k_collide<T, false, false, false, kC>))
                           : (parts ? (mrt ? k_collide<T, true, true> : k_collide<T, true, false>)
                                    : (mrt ? k_collide<T, false, true> : k_collide<T, false, false>));
    kernel<<<grid_for(P.N, block), block, 0, st>>>(P, a, b, rho, pa, pf, ci, err, rest_in, rest_out);
  });
}

void launch_collide_onepass(const StepParams &P, const void *fin, void *fout, const float *rest_in, float *rest_out,
                            const float *rho, float *rho_next, OnePassOut out, const ParticleArrays &pa, const ParticleForces &pf,
                            CellIndex ci, unsigned *err, OnePassGeom G, int grid, cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    const T *a = static_cast<const T *>(fin);
    T *b = static_cast<T *>(fout);
    auto *kernel = P.np > 0 ? k_collide_onepass<T, true> : k_collide_onepass<T, false>;
    if constexpr (!kSplitRest<T>)
      if (P.collision == LBMD_COLLISION_MRT)
        kernel = P.np > 0 ? k_collide_onepass<T, true, true> : k_collide_onepass<T, false, true>;
    kernel<<<grid, kOPThreads, 0, st>>>(P, a, b, rho, rho_next, out, pa, pf, ci, err, rest_in, rest_out, G);
  });
}

void launch_boundary_densities(const StepParams &P, OnePassGeom G, const void *store, const float *rest,
                               float *rho_next, const BoundaryRun *runs, int nruns, OnePassOut out,
                               const int *zslot, cudaStream_t st) {
  const int vec = P.nx % 2 == 0 ? 2 : 1;
  auto blocks = [](long long threads) { return (unsigned)((threads + kBlock - 1) / kBlock); };
  BoundaryBlocks D;
  D.runs = blocks(32LL * nruns);
  D.edge = blocks((long long)P.nz * P.ny * G.ntx);
  D.row = G.ypart ? blocks((long long)P.nz * G.nty * 2 * (P.nx / vec)) : 0;
  const unsigned plane = G.zpart ? blocks((long long)2 * G.nchunks * P.ny * (P.nx / vec)) : 0;
  D.by_ntx = make_fastdiv((uint32_t)G.ntx);
  D.by_nty = make_fastdiv((uint32_t)G.nty);
  D.by_run = make_fastdiv((uint32_t)(P.nx / vec));
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    auto *kernel = vec == 2 ? k_boundary_densities<T, 2> : k_boundary_densities<T, 1>;
    kernel<<<D.runs + D.edge + D.row + plane, kBlock, 0, st>>>(P, G, D, static_cast<const T *>(store), rest, rho_next,
                                                               runs, nruns, out, zslot);
  });
}

int onepass_blocks_per_sm() {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_collide_onepass<float, true>, kOPThreads, 0) !=
          cudaSuccess ||
      b < 1) {
    cudaGetLastError();
    b = 1;
  }
  return b;
}

template <class T>
bool is_noisy_update_of(const void *fn) {
  auto is = [fn](auto *kernel) { return fn == reinterpret_cast<const void *>(kernel); };
  return is(&k_collide<T, true, true, true>) || is(&k_collide<T, true, true>) || is(&k_collide<T, false, true>) ||
         is(&k_collide<T, true, true, false, kCollideBlock>) || is(&k_collide<T, false, true, false, kCollideBlock>) ||
         is(&k_step_small<T, true>);
}

bool is_noisy_onepass(const void *fn) {
  return fn == reinterpret_cast<const void *>(&k_collide_onepass<float, true, true>) ||
         fn == reinterpret_cast<const void *>(&k_collide_onepass<float, false, true>);
}

bool is_noisy_update(const void *fn) {
  return is_noisy_onepass(fn) || is_noisy_update_of<float>(fn) || is_noisy_update_of<__half>(fn) ||
         is_noisy_update_of<__nv_bfloat16>(fn);
}

template <class... A>
constexpr int arity(void (*)(A...)) {
  return (int)sizeof...(A);
}

cudaError_t set_update_step(cudaGraphExec_t exec, cudaGraphNode_t node, unsigned long long step) {
  constexpr int kArgs = arity(&k_collide<float, false, true>), kOnePassArgs = arity(&k_collide_onepass<float, false, true>);
  static_assert(kArgs == arity(&k_step_small<float, true>), "these noisy updates take the same parameters");
  cudaKernelNodeParams kp;
  cudaError_t e = cudaGraphKernelNodeGetParams(node, &kp);
  if (e != cudaSuccess) return e;
  if (!is_noisy_update(kp.func) || !kp.kernelParams) return cudaErrorInvalidValue;
  StepParams P;
  std::memcpy(&P, kp.kernelParams[0], sizeof(P));  // the node's own copy of the parameters
  P.step = step;
  const int nargs = is_noisy_onepass(kp.func) ? kOnePassArgs : kArgs;
  void *args[kArgs > kOnePassArgs ? kArgs : kOnePassArgs];
  for (int k = 0; k < nargs; ++k) args[k] = kp.kernelParams[k];
  args[0] = &P;
  kp.kernelParams = args;
  kp.extra = nullptr;
  return cudaGraphExecKernelNodeSetParams(exec, node, &kp);  // copies the values
}

void launch_fields(const StepParams &P, const void *store, const float *rest, const float *rho, float *rhoA,
                   float *rhoB, float *u, cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    k_fields<T><<<grid_for(P.N), kBlock, 0, st>>>(P, static_cast<const T *>(store), rest, rho, rhoA, rhoB, u);
  });
}
int fluid_sum_blocks(const StepParams &P) {
  const long long b = (P.N + kSumBlock - 1) / kSumBlock;
  return (int)(b < kSumGrid ? b : kSumGrid);
}
void launch_fluid_sums(const StepParams &P, const void *store, const float *rest, double *partial, int nblocks,
                       cudaStream_t st) {
  with_storage(P, [&](auto t) {
    using T = std::remove_pointer_t<decltype(t)>;
    k_fluid_sums<T><<<nblocks, kSumBlock, 0, st>>>(P, static_cast<const T *>(store), rest, partial);
  });
}
void launch_finish_sums(const double *partial, int nblocks, int nvals, double *out, cudaStream_t st) {
  k_finish_sums<<<1, 32 * nvals, 0, st>>>(partial, nblocks, nvals, out);
}
void launch_drift_check(const double *sums, const double *psum, double *ref, double *last, unsigned *err,
                        long long step, double tol, int set_ref, cudaStream_t st) {
  k_drift_check<<<1, 1, 0, st>>>(sums, psum, ref, last, err, step, tol, set_ref);
}

// The step base of replayed step graphs (one thread: a write, or an increment at the end of a
// replay, ordered after every launch of the replay that reads it).
__global__ void k_set_step(unsigned long long *base, unsigned long long value) { *base = value; }
__global__ void k_advance_step(unsigned long long *base, unsigned long long n) { *base += n; }

void launch_set_step(unsigned long long *base, unsigned long long value, cudaStream_t st) {
  k_set_step<<<1, 1, 0, st>>>(base, value);
}

void launch_advance_step(unsigned long long *base, unsigned long long n, cudaStream_t st) {
  k_advance_step<<<1, 1, 0, st>>>(base, n);
}

}  // namespace lbmd
