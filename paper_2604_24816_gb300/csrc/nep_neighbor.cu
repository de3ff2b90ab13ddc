// nep_neighbor.cu -- cell binning, cell sort and banded half/full neighbour lists on sm_103a.
//
// Rebuild pipeline (every kernel takes the control block and returns at once when the current step
// does not rebuild, so the whole MD step can be replayed as one CUDA graph):
//   k_cell_assign   wrap x into the box (float64), cell = floor(x / l) per dimension, histogram
//   k_scan_*        exclusive scan of the histogram -> cell_start (1 kernel for one tile of cells, else 3;
//                   integer, deterministic), which also clears the histogram for the next build
//   k_scatter       slot within the cell (arbitrary order), then
//   k_permute       rank of each atom in its cell by original id: the sorted order is a pure function of
//                   the positions, independent of launch timing and of the previous order; gathers x, v,
//                   id into it and forms the cell-relative float32 coordinates
//   k_copy_back     copy the gathered arrays back (fixed device pointers for graph replay)
//   k_rebuild_small, k_rebuild_cluster   all of the above in one block or one cluster, for small systems; these can
//                   also take the rebuild decision themselves
//   k_neighbors     for each atom, every j with |r_ij| < rc_R + skin among the 27 neighbouring cell
//                   images, split into the pairs this atom owns (one owner per unordered pair) and the
//                   rest, each part grouped by distance band so that the per-pair branches of the
//                   force kernels stay warp-uniform.
// Distances use cell-relative float32 coordinates plus the image offset of the neighbouring cell, so
// their error does not grow with the box size (float64 appears only in the wrap and cell assignment).
#include "nep_common.cuh"
#include "nep_control.cuh"

#include <algorithm>

namespace nep {

// Box edges, cell edges, cells per dimension (float64 side of the cell sort), and the reciprocal edges that index
// them.  The sort divides each cell into 2^ssh slices along x: a slice row (fixed y and z) is contiguous, so that
// the neighbour scan reads only the slices that its atom can reach.  ilx: slices per Angstrom.
struct CellGrid {
  double Lx, Ly, Lz, lx, ly, lz, ilx, ily, ilz;
  int ncx, ncy, ncz, ssh;
};

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// GB300's FP64 pipe is narrow and a float64 division is a chain of some ten dependent operations on it, so
// the divisions are kept out of the common path: an atom already inside the box is not wrapped, and the
// cell index multiplies by the reciprocal edge (an atom within rounding of a cell face may fall on either
// side of it; its cell-relative coordinate is then 0 or the edge, and the lists hold the same pairs): k_cell_assign
// 137 -> 39 us at 1,048,576 atoms, 7.8 -> 4.4 us at 16,384 (six divisions per atom before).
__device__ __forceinline__ double wrap_coord(double x, double L) {
  if (x >= 0.0 && x < L) return x;
  double y = x - L * floor(x / L);
  if (y >= L) y -= L;
  if (y < 0.0) y = 0.0;
  return y;
}
// Position of atom s wrapped into the box (a non-finite one becomes 0 and raises ST_NAN) and its cell
// coordinates.
struct CellOf {
  double x, y, z;
  int cx, cy, cz;
  int slice;             // index of its slice of cell in the sorted order
};
__device__ __forceinline__ CellOf cell_of_atom(double px, double py, double pz, const CellGrid &g, int *status) {
  if (!(isfinite(px) && isfinite(py) && isfinite(pz))) {
    atomicOr(status, ST_NAN);
    px = py = pz = 0.0;
  }
  CellOf c;
  c.x = wrap_coord(px, g.Lx); c.y = wrap_coord(py, g.Ly); c.z = wrap_coord(pz, g.Lz);
  const int sx = min((int)(c.x * g.ilx), (g.ncx << g.ssh) - 1);
  c.cx = sx >> g.ssh;
  c.cy = min((int)(c.y * g.ily), g.ncy - 1);
  c.cz = min((int)(c.z * g.ilz), g.ncz - 1);
  c.slice = (c.cz * g.ncy + c.cy) * (g.ncx << g.ssh) + sx;
  return c;
}
// Cell-relative float32 coordinates: the same expression as the drift and upload kernels (nep_md.cu), so
// that a position uploaded unchanged gives bitwise the same coordinates.
__device__ __forceinline__ float4 cell_relative(double px, double py, double pz, int cx, int cy, int cz,
                                                const CellGrid &g) {
  return make_float4((float)fma(-(double)cx, g.lx, px), (float)fma(-(double)cy, g.ly, py),
                     (float)fma(-(double)cz, g.lz, pz), __int_as_float(cx | (cy << 10) | (cz << 20)));
}

__global__ void k_cell_assign(int n, double *__restrict__ x, double *__restrict__ y, double *__restrict__ z,
                              const CellGrid g, int *__restrict__ cell_of, int *__restrict__ count, Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
    const double px = x[s], py = y[s], pz = z[s];
    const CellOf a = cell_of_atom(px, py, pz, g, &ctrl->status);
    if (a.x != px || a.y != py || a.z != pz) {          // also true for NaN: the wrapped position replaces it
      x[s] = a.x; y[s] = a.y; z[s] = a.z;
    }
    cell_of[s] = a.slice;
    atomicAdd(count + a.slice, 1);
  }
}

// Exclusive scan over the block of one int per thread (SCAN_THREADS threads); warp_tot: scratch.
__device__ __forceinline__ int block_scan_excl(int run, int *warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int t = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int u = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += u;
  }
  if (lane == 31) warp_tot[warp] = t;
  __syncthreads();
  if (warp == 0) {
    int w = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    warp_tot[lane] = w;
  }
  __syncthreads();
  return t - run + (warp > 0 ? warp_tot[warp - 1] : 0);
}

// Exclusive scan of count[0..m) into start[0..m], start[m] = total, and a copy in cursor (the running slots
// of k_scatter); count is cleared.  One tile (m <= SCAN_TILE): k_scan_tiles alone; else tile scan + carry
// pass + add.
__global__ void __launch_bounds__(SCAN_THREADS)
k_scan_tiles(int m, int *__restrict__ count, int *__restrict__ start, int *__restrict__ cursor,
             int *__restrict__ tile_sums, Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->nb_next = 0;   // the neighbour scan's work counter
  __shared__ int warp_tot[SCAN_THREADS / 32];
  const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
  int v[SCAN_ITEMS], run = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    v[k] = 0;
    if (base + k < m) {
      v[k] = count[base + k];
      count[base + k] = 0;
    }
    run += v[k];
  }
  int excl = block_scan_excl(run, warp_tot);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    if (base + k < m) {
      start[base + k] = excl;
      cursor[base + k] = excl;                                  // final when there is one tile
    }
    excl += v[k];
  }
  if (threadIdx.x == SCAN_THREADS - 1) {
    tile_sums[blockIdx.x] = excl;
    if (gridDim.x == 1) start[m] = excl;
  }
}

// Exclusive scan of the tile sums by one block, SCAN_THREADS at a time.
__global__ void __launch_bounds__(SCAN_THREADS)
k_scan_carry(int ntiles, int *__restrict__ tile_sums, int m, int *__restrict__ start, const Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  __shared__ int warp_tot[SCAN_THREADS / 32];
  int carry = 0;
  for (int b0 = 0; b0 < ntiles; b0 += SCAN_THREADS) {
    const int b = b0 + (int)threadIdx.x;
    const int s = b < ntiles ? tile_sums[b] : 0;
    const int excl = block_scan_excl(s, warp_tot);
    if (b < ntiles) tile_sums[b] = carry + excl;
    carry += warp_tot[SCAN_THREADS / 32 - 1];
    __syncthreads();                                            // warp_tot is reused by the next chunk
  }
  if (threadIdx.x == 0) start[m] = carry;
}

__global__ void k_scan_add(int m, int *__restrict__ start, int *__restrict__ cursor, const int *__restrict__ tile_sums,
                           const Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < m; idx += gridDim.x * blockDim.x) {
    const int s = start[idx] + tile_sums[idx / SCAN_TILE];
    start[idx] = s;
    cursor[idx] = s;
  }
}

// slot t of a cell (in order of arrival) holds atom perm[t].x, whose original id is perm[t].y.
__global__ void k_scatter(int n, const int *__restrict__ cell_of, const int *__restrict__ id, int *__restrict__ cursor,
                          int2 *__restrict__ perm, const Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
    perm[atomicAdd(cursor + cell_of[s], 1)] = make_int2(s, id[s]);
}

// One thread per slot: its atom's place in the cell is the number of the cell's atoms with a smaller
// original id (ids are unique), counted over the cell's slots, which neighbouring threads read too (L1
// hits).  The former pass, one thread per cell sorting its ~18 slots in global memory, was a chain of
// dependent loads: 41 us from 1,000 to 100,000 atoms, 51 us at 1,048,576; counting ranks here leaves that
// launch out and adds nothing measurable to this one.
__global__ void k_permute(int n, const int2 *__restrict__ perm, const int *__restrict__ start,
                          const double *__restrict__ x, const double *__restrict__ y,
                          const double *__restrict__ z, const double *__restrict__ vx, const double *__restrict__ vy,
                          const double *__restrict__ vz, const int *__restrict__ cell_of,
                          double *__restrict__ xb, double *__restrict__ yb, double *__restrict__ zb,
                          double *__restrict__ vxb, double *__restrict__ vyb, double *__restrict__ vzb,
                          int *__restrict__ idb, float4 *__restrict__ pos, float4 *__restrict__ pos_ref,
                          const CellGrid g, const Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const int2 sp = perm[q];
    const int s = sp.x;
    const int c = cell_of[s];
    const int b = start[c], e = start[c + 1];
    int t = b;
    for (int k = b; k < e; ++k) t += perm[k].y < sp.y ? 1 : 0;
    const double px = x[s], py = y[s], pz = z[s];
    xb[t] = px; yb[t] = py; zb[t] = pz;
    vxb[t] = vx[s]; vyb[t] = vy[s]; vzb[t] = vz[s];
    idb[t] = sp.y;
    const int nsx = g.ncx << g.ssh;
    const int cx = (c % nsx) >> g.ssh, cy = (c / nsx) % g.ncy, cz = c / (nsx * g.ncy);
    const float4 p = cell_relative(px, py, pz, cx, cy, cz, g);
    pos[t] = p;
    pos_ref[t] = p;
  }
}

__global__ void k_copy_back(int n, double *__restrict__ x, double *__restrict__ y, double *__restrict__ z,
                            double *__restrict__ vx, double *__restrict__ vy, double *__restrict__ vz,
                            int *__restrict__ id, const double *__restrict__ xb, const double *__restrict__ yb,
                            const double *__restrict__ zb, const double *__restrict__ vxb,
                            const double *__restrict__ vyb, const double *__restrict__ vzb,
                            const int *__restrict__ idb, const Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    x[t] = xb[t]; y[t] = yb[t]; z[t] = zb[t];
    vx[t] = vxb[t]; vy[t] = vyb[t]; vz[t] = vzb[t];
    id[t] = idb[t];
  }
}

// The whole cell sort of a small system (n <= SMALL_ATOMS, ncell <= SMALL_CELLS) in one block: histogram,
// scan, slots and ranks in shared memory, the state in registers between reading the old order and writing
// the new one (no second buffer).  The same order and coordinates as the kernels above.  At this size every
// kernel of the chain is a launch and a few dependent loads: 6.2 us at 862 atoms, and 1.7 us on a step that
// does not rebuild, the decision included, against nine launches (26 us and 13 us) and a control kernel.
constexpr int SMALL_ATOMS = 2048, SMALL_CELLS = 2048;
constexpr int SMALL_ITEMS = SMALL_ATOMS / SCAN_THREADS;
static_assert(SMALL_ATOMS % SCAN_THREADS == 0 && SMALL_CELLS == 2 * SCAN_THREADS, "two cells per thread");
__global__ void __launch_bounds__(SCAN_THREADS)
k_rebuild_small(int n, int ncell, double *__restrict__ x, double *__restrict__ y, double *__restrict__ z,
                double *__restrict__ vx, double *__restrict__ vy, double *__restrict__ vz, int *__restrict__ id,
                int *__restrict__ start, float4 *__restrict__ pos, float4 *__restrict__ pos_ref, const CellGrid g,
                Control *ctrl, int decide) {
  __shared__ int go;
  if (threadIdx.x == 0) go = decide_rebuild(ctrl, decide);
  __syncthreads();
  if (!go) return;
  __shared__ int cnt[SMALL_CELLS];                 // histogram, then the running slots
  __shared__ int first[SMALL_CELLS + 1];           // cell_start
  __shared__ int sid[SMALL_ATOMS];                 // original ids by slot
  __shared__ int warp_tot[SCAN_THREADS / 32];
  const int t = threadIdx.x;
  if (t == 0) ctrl->nb_next = 0;
  cnt[2 * t] = 0;
  cnt[2 * t + 1] = 0;
  __syncthreads();
  CellOf a[SMALL_ITEMS];
  double u[SMALL_ITEMS][3];
  int oid[SMALL_ITEMS], cell[SMALL_ITEMS];
#pragma unroll
  for (int k = 0; k < SMALL_ITEMS; ++k) {
    const int s = k * SCAN_THREADS + t;
    cell[k] = -1;
    if (s < n) {
      a[k] = cell_of_atom(x[s], y[s], z[s], g, &ctrl->status);
      u[k][0] = vx[s]; u[k][1] = vy[s]; u[k][2] = vz[s];
      oid[k] = id[s];
      cell[k] = a[k].slice;
      atomicAdd(&cnt[cell[k]], 1);
    }
  }
  __syncthreads();
  const int c0 = cnt[2 * t], c1 = cnt[2 * t + 1];
  const int excl = block_scan_excl(c0 + c1, warp_tot);
  first[2 * t] = cnt[2 * t] = excl;
  first[2 * t + 1] = cnt[2 * t + 1] = excl + c0;
  if (t == SCAN_THREADS - 1) first[SMALL_CELLS] = excl + c0 + c1;
  __syncthreads();
  // cells past ncell are empty, so first[ncell] is the total
  for (int c = t; c <= ncell; c += SCAN_THREADS) start[c] = first[c];
#pragma unroll
  for (int k = 0; k < SMALL_ITEMS; ++k)
    if (cell[k] >= 0) sid[atomicAdd(&cnt[cell[k]], 1)] = oid[k];
  __syncthreads();                                 // every old value has been read, every slot is filled
#pragma unroll
  for (int k = 0; k < SMALL_ITEMS; ++k) {
    if (cell[k] < 0) continue;
    const int b = first[cell[k]], e = first[cell[k] + 1];
    int d = b;
    for (int q = b; q < e; ++q) d += sid[q] < oid[k] ? 1 : 0;
    x[d] = a[k].x; y[d] = a[k].y; z[d] = a[k].z;
    vx[d] = u[k][0]; vy[d] = u[k][1]; vz[d] = u[k][2];
    id[d] = oid[k];
    const float4 p = cell_relative(a[k].x, a[k].y, a[k].z, a[k].cx, a[k].cy, a[k].cz, g);
    pos[d] = p;
    pos_ref[d] = p;
  }
}

// The same for up to CLUSTER_ATOMS atoms and CLUSTER_CELLS cells by a cluster of eight blocks: the phases meet at
// cluster barriers (hardware barriers; the blocks of a cluster are always resident together), cell counts, scan
// and slots go through global memory, each thread keeps its atoms' old state in registers until every block has
// read its share.  The histogram's own atomic gives each atom its slot, so there is no scatter counter.  One launch
// instead of five per rebuild (25 us at 16,384 atoms: eight SMs' narrow FP64 pipes and six barriers, against 17 us
// and four gaps) and, on the other steps, 1.9 us instead of the 8 us of a conditional graph node or five early
// exits: a 10-step block of 16,384 atoms 789 -> 771 us.
constexpr int CLUSTER_BLOCKS = 8;
constexpr int CLUSTER_THREADS = CLUSTER_BLOCKS * SCAN_THREADS;
constexpr int CLUSTER_ITEMS = 2;
constexpr int CLUSTER_ATOMS = CLUSTER_THREADS * CLUSTER_ITEMS, CLUSTER_CELLS = CLUSTER_THREADS * 2;

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __cluster_dims__(CLUSTER_BLOCKS, 1, 1) __launch_bounds__(SCAN_THREADS)
k_rebuild_cluster(int n, int ncell, double *__restrict__ x, double *__restrict__ y, double *__restrict__ z,
                  double *__restrict__ vx, double *__restrict__ vy, double *__restrict__ vz, int *__restrict__ id,
                  int *__restrict__ count, int *__restrict__ start, int *__restrict__ tile_sums,
                  int *__restrict__ slot_id, float4 *__restrict__ pos, float4 *__restrict__ pos_ref, const CellGrid g,
                  Control *ctrl, int decide) {
  __shared__ int warp_tot[SCAN_THREADS / 32];
  const int t = threadIdx.x, b = blockIdx.x;
  if (b == 0 && t == 0) decide_rebuild(ctrl, decide);
  __threadfence();
  cluster_barrier();
  if (!__ldcg(&ctrl->do_rebuild)) return;
  if (b == 0 && t == 0) ctrl->nb_next = 0;
  CellOf a[CLUSTER_ITEMS];
  double u[CLUSTER_ITEMS][3];
  int oid[CLUSTER_ITEMS], cell[CLUSTER_ITEMS], ord[CLUSTER_ITEMS];
#pragma unroll
  for (int k = 0; k < CLUSTER_ITEMS; ++k) {
    const int s = (k * CLUSTER_BLOCKS + b) * SCAN_THREADS + t;
    cell[k] = -1;
    if (s < n) {
      a[k] = cell_of_atom(x[s], y[s], z[s], g, &ctrl->status);
      u[k][0] = vx[s]; u[k][1] = vy[s]; u[k][2] = vz[s];
      oid[k] = id[s];
      cell[k] = a[k].slice;
      ord[k] = atomicAdd(count + cell[k], 1);
    }
  }
  __threadfence();
  cluster_barrier();                               // every atom is counted
  // two cells per thread; reads past L1, where another block wrote
  const int c = (b * SCAN_THREADS + t) * 2;
  const int c0 = c < ncell ? __ldcg(count + c) : 0, c1 = c + 1 < ncell ? __ldcg(count + c + 1) : 0;
  if (c < ncell) count[c] = 0;
  if (c + 1 < ncell) count[c + 1] = 0;
  const int excl = block_scan_excl(c0 + c1, warp_tot);
  if (t == SCAN_THREADS - 1) tile_sums[b] = excl + c0 + c1;
  __threadfence();
  cluster_barrier();
  int first = 0;
  for (int k = 0; k < b; ++k) first += __ldcg(tile_sums + k);
  if (c < ncell) start[c] = first + excl;
  if (c + 1 < ncell) start[c + 1] = first + excl + c0;
  if (b == CLUSTER_BLOCKS - 1 && t == SCAN_THREADS - 1) start[ncell] = first + excl + c0 + c1;
  __threadfence();
  cluster_barrier();
  int lo[CLUSTER_ITEMS], hi[CLUSTER_ITEMS];
#pragma unroll
  for (int k = 0; k < CLUSTER_ITEMS; ++k) {
    if (cell[k] < 0) continue;
    lo[k] = __ldcg(start + cell[k]);
    hi[k] = __ldcg(start + cell[k] + 1);
    slot_id[lo[k] + ord[k]] = oid[k];
  }
  __threadfence();
  cluster_barrier();                               // every slot is filled, every old value has been read
#pragma unroll
  for (int k = 0; k < CLUSTER_ITEMS; ++k) {
    if (cell[k] < 0) continue;
    int d = lo[k];
    for (int q = lo[k]; q < hi[k]; ++q) d += __ldcg(slot_id + q) < oid[k] ? 1 : 0;
    x[d] = a[k].x; y[d] = a[k].y; z[d] = a[k].z;
    vx[d] = u[k][0]; vy[d] = u[k][1]; vz[d] = u[k][2];
    id[d] = oid[k];
    const float4 p = cell_relative(a[k].x, a[k].y, a[k].z, a[k].cx, a[k].cy, a[k].cz, g);
    pos[d] = p;
    pos_ref[d] = p;
  }
}

// One warp per atom over the candidates of the 27 neighbouring cell images (below).
//
// Segments: the pair (i, j) is "owned" by i when r_ij lies in the upper half-space (see owns_pair;
// exactly one of r_ij and r_ji = -r_ij is owned, so every unordered pair has one owner), and the row
// is laid out as [owned | not owned], each part grouped by build-time distance band:
// [0, rc_A), [rc_A, rc_A + skin), [rc_A + skin, rc_R), [rc_R, rc_R + e), [rc_R + e, rc_R + skin) with
// e = FAR_EDGE skin, in stencil order inside a band.  The half-list force kernels walk only the owned part (each pair once,
// Newton's third law); the other walks take the whole row.  The last ("far") band of each part can
// only hold a pair inside rc_R after some atom moved more than e/2 since the build, so while the
// largest displacement stays below that the walks leave both far bands out (their counts go to
// nfar).  Because every atom of a lattice owns exactly half of each shell and the bands follow the
// shells, the per-pair branches stay warp-uniform without a full sort.
// The placement's 4-byte stores into the neighbour-major list are scattered across rows; L2 merges
// them into full sectors before they reach DRAM.
constexpr int NB_WARPS = 8;            // atoms (one warp each) per block
// Atoms from which a block takes four groups of NB_WARPS atoms at a time: fewer barriers, but too coarse for small
// systems.  One and four groups per take: 16,384 atoms 32 and 47 us, 55,296 80 and 86, 131,072 170 and 172, 157,216 205
// and 205, 262,400 336 and 330, 500,000 627 and 602, 1,048,576 1,360 and 1,311 (eight: 1,309).
constexpr int NB_TAKE_MIN = 160000;
constexpr int NB_STAGE = 128;          // staged entries per atom (lists longer than this are an overflow)
constexpr float OWN_EPS = 0.5f;        // Angstrom; lattice-vector components are either ~0 or >= a/2

struct Bands {
  float b0, b1, b2, b3, b4;  // squared band edges: rc_A^2, (rc_A+skin)^2, rc_R^2, (rc_R+e)^2, (rc_R+skin)^2
};
constexpr int NB_SEG = 10;             // segments of a row: [owned | not owned] x 5 distance bands

// Upper half-space test, exactly antisymmetric: owns_pair(d) != owns_pair(-d) for d != 0.  The
// tolerance makes near-zero components of lattice vectors (thermal noise) defer to the next axis, so
// each fcc shell splits into two equal halves for every atom.
__device__ __forceinline__ bool owns_pair(float dx, float dy, float dz) {
  if (dz > OWN_EPS) return true;
  if (dz < -OWN_EPS) return false;
  if (dy > OWN_EPS) return true;
  if (dy < -OWN_EPS) return false;
  if (dx != 0.f) return dx > 0.f;
  if (dy != 0.f) return dy > 0.f;
  return dz > 0.f;
}

// Squared distance with an explicit operation order, so that both passes classify a pair identically.
__device__ __forceinline__ float nb_r2(float a, float b, float c) { return fmaf(a, a, fmaf(b, b, c * c)); }

// Segment of an accepted pair: owned by i (0..4) or not (5..9), by build-time distance band.
__device__ __forceinline__ int segment_of(float dx, float dy, float dz, float r2, const Bands &B) {
  const int bd = (int)(r2 >= B.b0) + (int)(r2 >= B.b1) + (int)(r2 >= B.b2) + (int)(r2 >= B.b3);   // edges below r2
  return owns_pair(dx, dy, dz) ? bd : 5 + bd;
}

// This chunk's entries of segment `lane % 5` (lanes 0..4) or `5 + lane % 5` (lanes 5..9); key NB_SEG
// marks an empty slot.  fsh = 6 (lane % 5).
__device__ __forceinline__ int segment_counts(int key, int lane, unsigned fsh) {
  const unsigned lo = key < 5 ? 1u << (6 * key) : 0u;
  const unsigned hi = key >= 5 && key < NB_SEG ? 1u << (6 * (key - 5)) : 0u;
  const unsigned slo = __reduce_add_sync(0xffffffffu, lo), shi = __reduce_add_sync(0xffffffffu, hi);
  return (int)(((lane < 5 ? slo : shi) >> fsh) & 63u);
}

// The candidate scan and segment placement of atom i by one warp (see k_neighbors).
__device__ __forceinline__ void neighbors_of_atom(int i, int n, const float4 *__restrict__ pos,
                                                  const int *__restrict__ cell_start, const Geom &geom, int ssh,
                                                  float slices, const Bands &B, int limit, float4 *stage, float4 *tab,
                                                  int lane, int32_t *__restrict__ nbr,
                                                  int32_t *__restrict__ nnum, int32_t *__restrict__ nang,
                                                  int32_t *__restrict__ nown, int32_t *__restrict__ nband0,
                                                  int32_t *__restrict__ nfar, Control *ctrl) {
  const unsigned lower = (1u << lane) - 1u;
  const float4 pi = pos[i];
  const int cx = cell_x(pi.w), cy = cell_y(pi.w), cz = cell_z(pi.w);
  const bool xwrap = cx == 0 || cx == geom.ncx - 1;
  int acc = 0;                                         // accepted so far (warp-uniform)
  // The candidate ranges in stencil order (dz, dy, then the x part), set up one per lane L = 9 (dz + 1)
  // + 3 (dy + 1) + part: a row of three cells that does not wrap around x is one range (part 0), a row that wraps is
  // three; rows whose (y, z) slab lies beyond the list radius are empty.  A range holds the x slices within the reach
  // left after the row's (y, z) gap: every candidate outside is at least that far away in x.  The 1e-4 margin
  // (0.0036 Angstrom^2) keeps every candidate a float32 distance test could accept, so the lists are unchanged.
  int rb = 0, rlen = 0;
  float roy = 0.f, roz = 0.f;
  int rcode = 0;                                       // shift-table base (dy, dz) | x part << 8
  if (lane < 27) {
    const int dz = lane / 9 - 1, dy = (lane / 3) % 3 - 1, part = lane % 3;
    roz = dz < 0 ? -geom.lz : (dz > 0 ? geom.lz : 0.f);   // the shift table's offsets
    roy = dy < 0 ? -geom.ly : (dy > 0 ? geom.ly : 0.f);
    rcode = (3 * (dy + 1) + 9 * (dz + 1)) | (part << 8);
    int zz = cz + dz;
    zz += zz < 0 ? geom.ncz : (zz >= geom.ncz ? -geom.ncz : 0);
    int yy = cy + dy;
    yy += yy < 0 ? geom.ncy : (yy >= geom.ncy ? -geom.ncy : 0);
    const int sub = 1 << ssh, row = (zz * geom.ncy + yy) * (geom.ncx << ssh);
    const float gy = dy < 0 ? pi.y : (dy > 0 ? geom.ly - pi.y : 0.f);
    const float gz = dz < 0 ? pi.z : (dz > 0 ? geom.lz - pi.z : 0.f);
    const float reach2 = B.b4 * 1.0001f - (gy * gy + gz * gz);
    if (reach2 >= 0.f) {
      // slices from this cell's first: s0..s1 within the three cells
      const float reach = sqrtf(reach2);
      int s0 = max(__float2int_rd((pi.x - reach) * slices), -sub), s1 = min(__float2int_rd((pi.x + reach) * slices), 2 * sub - 1);
      int at = cx;                                     // the cell that s0 is counted from
      if (xwrap) {
        const int o = (part - 1) * sub;
        s0 = max(s0, o) - o;
        s1 = min(s1, o + sub - 1) - o;
        at = cx + part - 1;
        at += at < 0 ? geom.ncx : (at >= geom.ncx ? -geom.ncx : 0);
      }
      if ((xwrap || part == 0) && s1 >= s0) {
        rb = cell_start[row + at * sub + s0];
        rlen = cell_start[row + at * sub + s1 + 1] - rb;
      }
    }
  }
  // The non-empty ranges form one sequence, walked 32 candidates at a time (8.4 turns per atom of an fcc crystal; range
  // by range it takes 13.2, half of the ranges needing a second, mostly empty one).  A lane finds its range as the
  // number of range starts up to its place: one bit per start inside the turn, combined over the warp.  Each candidate
  // is tested without a branch (the load index clamped), and an accepted pair's displacement and entry go to the
  // stage as one 16-byte record in candidate order.
  int incl = rlen;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31), first = incl - rlen;
  const unsigned ne = __ballot_sync(0xffffffffu, rlen > 0);
  if (rlen > 0) tab[__popc(ne & lower)] = make_float4(__int_as_float(rb - first), roy, roz, __int_as_float(rcode));
  __syncwarp();
  const unsigned upto = lower | (1u << lane);
  int started = 0;                                     // ranges that began before this turn (warp-uniform)
  for (int c0 = 0; c0 < total; c0 += 32) {
    const unsigned rel = (unsigned)(first - c0);
    const unsigned starts = __reduce_or_sync(0xffffffffu, rlen > 0 && rel < 32u ? 1u << rel : 0u);
    const float4 t = tab[started + __popc(starts & upto) - 1];
    started += __popc(starts);
    const bool inr = c0 + lane < total;
    const int j = __float_as_int(t.x) + c0 + lane;     // past the end of the last range when !inr
    const int code = __float_as_int(t.w);
    const float4 pj = pos[inr ? j : i];
    const int dx = xwrap ? (code >> 8) - 1 : cell_x(pj.w) - cx;
    const float ox = (float)dx * geom.lx;              // exact: dx is -1, 0 or 1
    const float ddx = pj.x - pi.x + ox, ddy = pj.y - pi.y + t.y, ddz = pj.z - pi.z + t.z;
    const bool ok = inr && j != i && nb_r2(ddx, ddy, ddz) < B.b4;
    const uint32_t ent = (uint32_t)j | ((uint32_t)((dx + 1) + (code & 255)) << J_BITS);
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    const int slot = acc + __popc(m & lower);
    if (ok && slot < NB_STAGE) stage[slot] = make_float4(ddx, ddy, ddz, __uint_as_float(ent));
    acc += __popc(m);
  }
  __syncwarp();
  // Segments of the staged entries (classified here, 32 accepted pairs at a time, rather than in the
  // sparse candidate loop; the same float32 arithmetic as the acceptance test): each entry's rank among the
  // turn's entries of its segment, and per lane g < NB_SEG the segment's count (two warp reductions of one-hot
  // 6-bit fields, segments 0..4 and 5..9: at most 32 per field, no carries) before and after the turn.  Then the
  // segments' offsets, and placement in candidate order within each segment.
  constexpr int TURNS = NB_STAGE / 32;
  const int ms = min(acc, NB_STAGE);
  const unsigned fsh = 6u * (unsigned)(lane % 5);
  int mycnt = 0;
  int keyrank[TURNS], before[TURNS];
#pragma unroll
  for (int t = 0; t < TURNS; ++t) {
    keyrank[t] = NB_SEG;
    before[t] = 0;
    if (32 * t >= ms) continue;                        // warp-uniform
    int key = NB_SEG;
    if (32 * t + lane < ms) {
      const float4 sd = stage[32 * t + lane];
      key = segment_of(sd.x, sd.y, sd.z, nb_r2(sd.x, sd.y, sd.z), B);
    }
    keyrank[t] = key | (__popc(__match_any_sync(0xffffffffu, key) & lower) << 8);
    before[t] = mycnt;
    mycnt += segment_counts(key, lane, fsh);
  }
  if (lane >= NB_SEG) mycnt = 0;
  incl = mycnt;                                        // inclusive prefix over lanes 0..NB_SEG-1
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
#pragma unroll
  for (int t = 0; t < TURNS; ++t) {
    if (32 * t >= ms) continue;
    const int k = __shfl_sync(0xffffffffu, incl - mycnt + before[t], keyrank[t] & 255) + (keyrank[t] >> 8);
    if (32 * t + lane < ms && k < limit)
      nbr[(size_t)k * n + i] = (int32_t)__float_as_uint(stage[32 * t + lane].w);
  }
  const int c0 = __shfl_sync(0xffffffffu, mycnt, 0), c1 = __shfl_sync(0xffffffffu, mycnt, 1);
  const int c4 = __shfl_sync(0xffffffffu, mycnt, 4), c5 = __shfl_sync(0xffffffffu, mycnt, 5);
  const int c6 = __shfl_sync(0xffffffffu, mycnt, 6), c9 = __shfl_sync(0xffffffffu, mycnt, 9);
  const int n_own = __shfl_sync(0xffffffffu, incl, 4);
  if (lane == 0) {
    const int kept = min(acc, limit);
    if (acc > kept || acc > NB_STAGE) atomicOr(&ctrl->status, ST_OVERFLOW);
    nnum[i] = kept;
    nown[i] = min(n_own, kept);
    nang[i] = c0 + c1 + c5 + c6;
    nband0[i] = min(c0, kept);
    // far bands (each part's last): skippable while no atom moved far enough to bring them in range;
    // zero when the row overflowed (the evaluation then reports the overflow)
    nfar[i] = acc > kept ? 0 : (c4 | (c9 << 16));
  }
}

// One warp per atom i.  The lanes test 32 candidates at a time (coalesced position loads, the atom's
// own position broadcast): for each of the 9 (dy, dz) rows of the 27-cell stencil the x slices within reach
// are consecutive in the sorted arrays, so the row is one contiguous range and a
// candidate's x offset comes from its packed cell coordinate (rows that wrap around the periodic x
// boundary are walked cell by cell; the bounds of all ranges are read up front, one lane each), and the ranges are
// walked as one sequence.  Accepted entries go to a per-warp shared-memory stage in
// candidate order (ballot + popc), then are placed by segment: [owned | not owned] x band, candidate
// order inside a segment -- the same row as the thread-per-atom formulation, with 32-wide work
// instead of divergent per-thread cell loops.  The kernel is bound by issue slots (85 % busy), so what counts is the
// number of turns and what each costs.  1,048,576 atoms: 1,608 us per build over whole cells, range by range; 1,500
// with four x slices per cell (269 candidates per atom instead of 385; eight slices 2 % less again, for twice the
// cells); 1,353 with the ranges as one sequence; 1,331 with segment ranks kept in registers between counting and
// placement; 1,299 with four groups per take.  Two candidates per lane and turn in float2 pairs: no gain.
__global__ void __launch_bounds__(NB_WARPS * 32, 6)   // 40 registers at most: 6 resident blocks
k_neighbors(int n, const float4 *__restrict__ pos, const int *__restrict__ cell_start, const Geom geom, int ssh,
            float slices, int take, int cap, Bands B, int32_t *__restrict__ nbr, int32_t *__restrict__ nnum, int32_t *__restrict__ nang,
            int32_t *__restrict__ nown, int32_t *__restrict__ nband0, int32_t *__restrict__ nfar, Control *ctrl) {
  if (!ctrl->do_rebuild) return;
  __shared__ float4 stage[NB_WARPS][NB_STAGE];         // staged (displacement, entry)
  __shared__ float4 tab[NB_WARPS][28];                 // candidate ranges
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // The grid is capped at the resident blocks (a launch on a step without a rebuild then costs a few
  // microseconds whatever the atom count); each block takes the next `take` groups of NB_WARPS consecutive
  // atoms from a counter, which keeps the order of the hardware's own block scheduling (a static
  // stride over the atoms measured 25 % slower).
  __shared__ int group;
  for (;;) {
    if (threadIdx.x == 0) group = atomicAdd(&ctrl->nb_next, 1);
    __syncthreads();
    const int g = group;
    __syncthreads();                                   // read by every warp before the next take
    if ((long long)g * (NB_WARPS * take) >= n) break;   // block-uniform
    for (int k = 0; k < take; ++k) {
      const int i = (g * take + k) * NB_WARPS + w;  // warp-uniform
      if (i >= n) break;
      neighbors_of_atom(i, n, pos, cell_start, geom, ssh, slices, B, min(cap, NB_STAGE), stage[w], tab[w], lane, nbr, nnum,
                        nang, nown, nband0, nfar, ctrl);
      __syncwarp();                                    // the stage is reused by the warp's next atom
    }
  }
}

// ---------------------------------------------------------------------------------------------------
// Host launcher for the whole rebuild chain.


static int blocks_for(long long m, int b) { return (int)((m + b - 1) / b); }

// Grid of the rebuild-chain kernels: enough blocks for m items, at most what is resident at once (the
// occupancy calculator's blocks per SM x the SM count); the kernels loop over the rest.  Every step
// launches the chain and the kernels return at once when it does not rebuild, so the grid size is
// what such a step pays for.
template <class K>
static int resident_grid(K kernel, long long m, int per_block, int threads) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm <= 0)
    per_sm = 1;
  return (int)std::min<long long>(blocks_for(m, per_block), (long long)sm_count() * per_sm);
}

// Slices per cell along x as a shift, for n atoms in ncell cells: four, unless the box is sparse (no gain, and four
// times the cells to clear and scan).
int slice_shift(int n, int64_t ncell) { return ncell <= n ? 2 : 0; }

// The forms of the cell sort: one block, one cluster, or the chain of kernels.
static bool small_system(int n, int ncell) { return n <= SMALL_ATOMS && ncell <= SMALL_CELLS; }
static bool cluster_system(int n, int ncell) { return n <= CLUSTER_ATOMS && ncell <= CLUSTER_CELLS; }
// Whether the sort is a single kernel, which can also take the rebuild decision.
bool cell_sort_decides(int n, int ncell) { return cluster_system(n, ncell); }
// Kernels that launch_cell_sort enqueues for a system of n atoms in ncell cells.
int cell_sort_launches(int n, int ncell) {
  if (n <= 0) return 0;
  return cluster_system(n, ncell) ? 1 : (ncell <= SCAN_TILE ? 5 : 7);
}

// a.count is zero on entry and on exit.  decide (nep_control.cuh): a decision that the sort's only kernel takes
// first (cell_sort_decides); DECIDE_DONE otherwise.
cudaError_t launch_cell_sort(const RebuildArgs &a, int decide, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  const CellGrid g{a.L[0], a.L[1], a.L[2], a.l[0], a.l[1], a.l[2], (1 << a.ssh) / a.l[0], 1.0 / a.l[1], 1.0 / a.l[2],
                   a.nc[0], a.nc[1], a.nc[2], a.ssh};
  if (small_system(a.n, a.ncell)) {
    k_rebuild_small<<<1, SCAN_THREADS, 0, st>>>(a.n, a.ncell, a.x, a.y, a.z, a.vx, a.vy, a.vz, a.id, a.start, a.pos,
                                                a.pos_ref, g, a.ctrl, decide);
    return cudaGetLastError();
  }
  if (cluster_system(a.n, a.ncell)) {
    k_rebuild_cluster<<<CLUSTER_BLOCKS, SCAN_THREADS, 0, st>>>(a.n, a.ncell, a.x, a.y, a.z, a.vx, a.vy, a.vz, a.id,
                                                               a.count, a.start, a.tile_sums, a.cell_of, a.pos,
                                                               a.pos_ref, g, a.ctrl, decide);
    return cudaGetLastError();
  }
  if (decide != DECIDE_DONE) return cudaErrorInvalidValue;
  k_cell_assign<<<resident_grid(k_cell_assign, a.n, 256, 256), 256, 0, st>>>(a.n, a.x, a.y, a.z, g, a.cell_of, a.count,
                                                                            a.ctrl);
  const int ntiles = blocks_for(a.ncell, SCAN_TILE);
  k_scan_tiles<<<ntiles, SCAN_THREADS, 0, st>>>(a.ncell, a.count, a.start, a.cursor, a.tile_sums, a.ctrl);
  if (ntiles > 1) {
    k_scan_carry<<<1, SCAN_THREADS, 0, st>>>(ntiles, a.tile_sums, a.ncell, a.start, a.ctrl);
    k_scan_add<<<resident_grid(k_scan_add, a.ncell, 256, 256), 256, 0, st>>>(a.ncell, a.start, a.cursor, a.tile_sums,
                                                                            a.ctrl);
  }
  k_scatter<<<resident_grid(k_scatter, a.n, 256, 256), 256, 0, st>>>(a.n, a.cell_of, a.id, a.cursor, a.perm, a.ctrl);
  k_permute<<<resident_grid(k_permute, a.n, 256, 256), 256, 0, st>>>(a.n, a.perm, a.start, a.x, a.y, a.z, a.vx, a.vy, a.vz,
                                                                    a.cell_of, a.xb, a.yb, a.zb, a.vxb, a.vyb, a.vzb,
                                                                    a.idb, a.pos, a.pos_ref, g, a.ctrl);
  k_copy_back<<<resident_grid(k_copy_back, a.n, 256, 256), 256, 0, st>>>(a.n, a.x, a.y, a.z, a.vx, a.vy, a.vz, a.id, a.xb, a.yb, a.zb,
                                                    a.vxb, a.vyb, a.vzb, a.idb, a.ctrl);
  return cudaGetLastError();
}

cudaError_t launch_neighbors(const RebuildArgs &a, cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  Geom g;
  g.lx = (float)a.l[0]; g.ly = (float)a.l[1]; g.lz = (float)a.l[2];
  g.ncx = a.nc[0]; g.ncy = a.nc[1]; g.ncz = a.nc[2];
  Bands B;
  B.b0 = a.ba2; B.b1 = a.ra2; B.b2 = a.br2; B.b3 = std::min(a.fs2, a.rl2); B.b4 = a.rl2;
  k_neighbors<<<resident_grid(k_neighbors, a.n, NB_WARPS, NB_WARPS * 32), NB_WARPS * 32, 0, st>>>(
      a.n, a.pos, a.start, g, a.ssh, (float)((1 << a.ssh) / a.l[0]), a.n >= NB_TAKE_MIN ? 4 : 1, a.cap, B, a.nbr, a.nnum, a.nang, a.nown, a.nband0, a.nfar, a.ctrl);
  return cudaGetLastError();
}

int scan_tiles(int ncell) { return std::max(CLUSTER_BLOCKS, blocks_for(ncell, SCAN_TILE)); }

}  // namespace nep
