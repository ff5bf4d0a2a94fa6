// Domain assignment and cell list (arXiv:1502.06447, Sec. II.A).
//
// Per sweep: the tile shift o in [0,T)^3 is drawn from Philox (tag 2,
// counter (2, sweep, 0, 0)); along each axis tile k covers
// [o + kT, o + (k+1)T - w) and the remaining width w is joint, whose beads
// cannot move this sweep.  The same pass bins every bead into the global
// cell grid (counting sort: count with atomics, exclusive scan, scatter of
// positions/ids/tiles into cell order).  The order of beads inside one cell
// is not fixed; nothing downstream depends on it (the EC kernel sorts what
// it stages by bead id).  With bead springs a bead whose bonded bead is
// motile in another tile is made immotile too (a spring has no longest
// bond, so only this keeps tiles apart).
#include <cuda_runtime.h>
#include <limits.h>

#include "ecmc_dev.cuh"
#include "ecmc_internal.h"

namespace ecmc {
namespace {

constexpr int SCAN_BLOCK = 1024;
constexpr int SCAN_ITEMS = 4;  // elements per thread
constexpr int SCAN_TILE = SCAN_BLOCK * SCAN_ITEMS;
// A call of ecmc_observables on 4,096 beads (GB300) whose blocks add the sums
// up / with k_scan_sums: 4,242 tiles 150 / 152 us, 16,950 447 / 459, 33,934
// 840 / 850, 68,607 1,753 / 1,647, 271,469 10,850 / 6,313, 442,234 24,038 /
// 10,249.
constexpr int64_t SCAN_DIRECT = 32768;

// Cell and tile of one coordinate.  FP32 decides both unless the coordinate
// lies within its error (C.tol) of a boundary; those few take the FP64
// expressions of the definition, so the result is always theirs.  (In FP64
// alone a bead took some 40 FP64 and conversion instructions: 150 us per
// sweep of 1e6 beads.)
__device__ __forceinline__ int cell_axis(const CellParams &C, int a, double r, float rf) {
  const float q = rf * C.cinv_f[a];
  int k = (int)q;
  const float f = q - (float)k, e = C.tol * C.cinv_f[a];
  if (f < e || f > 1.f - e) k = (int)div_rn(r, C.cs[a]);
  return k < 0 ? 0 : (k >= C.nc[a] ? C.nc[a] - 1 : k);
}

// o: the tile shift of the axis; false: in the joint
__device__ __forceinline__ bool tile_axis(const CellParams &C, int a, double r, float rf, double o, float of, int &k) {
  const float L = C.Lf[a], T = C.Tf[a], e = C.tol;
  float u = rf - of;
  const bool edge = fabsf(u) < e || L - fabsf(u) < e;
  if (u < 0.f) u += L;
  k = (int)(u * C.tinv_f[a]);
  const float loc = u - (float)k * T;
  if (edge || loc < e || loc > T - e || fabsf(loc - C.Wf[a]) < e) {
    double v = r - o;
    if (neg_bits(v)) v = v + C.L[a];
    if (!less_pos(v, C.L[a])) v = v - C.L[a];
    k = (int)div_rn(v, C.T[a]);
    if (k > C.D[a] - 1) k = C.D[a] - 1;
    return v - (double)k * C.T[a] < C.W[a];
  }
  if (k > C.D[a] - 1) k = C.D[a] - 1;
  return loc < C.Wf[a];
}

// the sweep's tile shift (threads 0..2 of a block, axis each)
__device__ __forceinline__ void sweep_shift(const CellParams &C, double *o) {
  if (threadIdx.x < 3) {
    const int64_t sweep = C.sweep_dev ? *C.sweep_dev : C.sweep;
    const u64x4 w = philox(TAG_SHIFT, (uint64_t)sweep, 0, 0, C.seed, C.replica);
    o[threadIdx.x] = unit53(threadIdx.x == 0 ? w.v[0] : (threadIdx.x == 1 ? w.v[1] : w.v[2])) * C.T[threadIdx.x];
  }
}

// tag and cell of bead b; returns the cell
__device__ __forceinline__ int tag_and_cell(const CellParams &C, int64_t b, const double *o) {
  const double r[3] = {C.r[3 * b], C.r[3 * b + 1], C.r[3 * b + 2]};
  int c[3], k[3];
  bool in = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float rf = f32_trunc(r[a]);
    c[a] = cell_axis(C, a, r[a], rf);
    k[a] = 0;
    if (C.domain) in = tile_axis(C, a, r[a], rf, o[a], f32_trunc(o[a]), k[a]) && in;
  }
  C.tag[b] = in ? (k[2] * C.D[1] + k[1]) * C.D[0] + k[0] : -1;
  const int cell = (c[2] * C.nc[1] + c[1]) * C.nc[0] + c[0];
  C.cell[b] = cell;
  return cell;
}

__global__ void k_tag_count(const CellParams C) {
  __shared__ double o[3];
  if (C.domain) sweep_shift(C, o);
  if (C.counters && blockIdx.x == 0 && threadIdx.x < 3) C.counters[threadIdx.x] = 0;
  __syncthreads();
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b < C.n) C.rank[b] = atomicAdd(&C.count[tag_and_cell(C, b, o)], 1);
}

// block-wide exclusive scan of SCAN_TILE ints; returns the tile total
__device__ int block_scan(int (&v)[SCAN_ITEMS], int *sh) {
  int local = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    const int t = v[i];
    v[i] = local;
    local += t;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int inc = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += y;
  }
  if (lane == 31) sh[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    int w = lane < (SCAN_BLOCK / 32) ? sh[lane] : 0;
    int wi = w;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, wi, off);
      if (lane >= off) wi += y;
    }
    if (lane < (SCAN_BLOCK / 32)) sh[lane] = wi - w;
    if (lane == 31) sh[32] = wi;
  }
  __syncthreads();
  const int base = sh[wid] + inc - local;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) v[i] += base;
  const int total = sh[32];
  __syncthreads();
  return total;
}

// (clears the counts it has read, for the next pass)
__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_tiles(int *in, int64_t n, int *out, int *block_sums) {
  __shared__ int sh[33];
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int v[SCAN_ITEMS];
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = (base + i < n) ? in[base + i] : 0;
  const int total = block_scan(v, sh);
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i)
    if (base + i < n) {
      out[base + i] = v[i];
      in[base + i] = 0;
    }
  if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

// adds to every tile of SCAN_TILE starts the sums of the tiles before it:
// each block adds those up itself, or, of more than SCAN_DIRECT tiles (what
// the blocks read grows with their square), takes the one that k_scan_sums left
__global__ void __launch_bounds__(256) k_scan_add(int *out, int64_t n, const int *sums, int64_t tiles, bool summed) {
  __shared__ int sh[8];
  int before = 0;
  if (summed) {
    before = sums[blockIdx.x];
  } else {
    int part = 0;
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += 256) part += sums[i];
    part = __reduce_add_sync(0xffffffffu, part);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = part;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) before += sh[i];
    if (blockIdx.x == tiles - 1 && threadIdx.x == 0) out[n] = before + sums[tiles - 1];
  }
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  for (int64_t i = base + threadIdx.x; i < base + SCAN_TILE && i < n; i += 256) out[i] += before;
}

// exclusive scan of the tile sums in place, and the total (one block)
__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_sums(int *sums, int64_t tiles, int *total) {
  __shared__ int sh[33];
  int carry = 0;
  for (int64_t t0 = 0; t0 < tiles; t0 += SCAN_TILE) {
    const int64_t base = t0 + (int64_t)threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = base + i < tiles ? sums[base + i] : 0;
    const int chunk = block_scan(v, sh);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i)
      if (base + i < tiles) sums[base + i] = v[i] + carry;
    carry += chunk;
  }
  if (threadIdx.x == 0) *total = carry;
}

// counts -> starts (ncell + 1), the counts cleared
void launch_scan(int *count, int64_t ncell, int *start, int *sums, cudaStream_t s) {
  const int64_t tiles = (ncell + SCAN_TILE - 1) / SCAN_TILE;
  const bool summed = tiles > SCAN_DIRECT;
  k_scan_tiles<<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(count, ncell, start, sums);
  if (summed) k_scan_sums<<<1, SCAN_BLOCK, 0, s>>>(sums, tiles, start + ncell);
  k_scan_add<<<(unsigned)tiles, 256, 0, s>>>(start, ncell, sums, tiles, summed);
}

// Tag of a joint bead in cell order: whose tile its bonded beads are motile
// in (staging takes a joint bead beyond the hard-sphere halo only for those):
// -1 several tiles, -2 - k tile k, INT_MIN none
__device__ __forceinline__ int32_t joint_tag(int32_t tp, int32_t tn) {
  if (tp >= 0 && tn >= 0 && tp != tn) return -1;
  const int32_t k = tp >= 0 ? tp : tn;
  return k >= 0 ? -2 - k : INT_MIN;
}

__device__ __forceinline__ void scatter_bead(const CellParams &C, int64_t b, int64_t pos) {
  const double x = C.r[3 * b], y = C.r[3 * b + 1], z = C.r[3 * b + 2];
  const float fx = (float)x, fy = (float)y, fz = (float)z;
  C.cr[3 * pos] = x;
  C.cr[3 * pos + 1] = y;
  C.cr[3 * pos + 2] = z;
  C.crf[3 * pos] = fx;
  C.crf[3 * pos + 1] = fy;
  C.crf[3 * pos + 2] = fz;
  C.rf[3 * b] = fx;
  C.rf[3 * b + 1] = fy;
  C.rf[3 * b + 2] = fz;
  C.cid[pos] = (int32_t)b;
  int32_t t = C.tag[b];
  const int64_t c = b % C.N;
  const int32_t tp = c != 0 ? C.tag[b - 1] : -1;
  const int32_t tn = c != C.N - 1 ? C.tag[b + 1] : -1;
  // bead-spring chains: a bead whose bonded bead is motile in another
  // tile waits for a later sweep (the tags of both are the ones
  // k_tag_count assigned, before any is dropped)
  if (C.spring && t >= 0 && ((tp >= 0 && tp != t) || (tn >= 0 && tn != t))) t = -1;
  C.ctag[pos] = t >= 0 ? t : joint_tag(tp, tn);
  if (C.ftag) C.ftag[b] = t;
}

__global__ void k_scatter(const CellParams C) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b < C.n) scatter_bead(C, b, (int64_t)C.start[C.cell[b]] + C.rank[b]);
}

// The whole pass of a small melt in one block, counts in shared memory: a
// small melt's sweep takes as long as its launches, and four of them become
// one.  One block / four kernels: us per sweep (27 tiles, next to no events)
// of 512 beads 28 / 39, 1,728 38 / 44, 4,096 50 / 51, 5,832 64 / 58, 8,000
// 84 / 70; us per call of ecmc_observables on 512 beads 47 / 53, 4,096 59 / 63,
// 6,859 62 / 63, 8,000 73 / 63.  The line at 8,192 beads is older than these
// figures: even are some 4,300 beads for sweeps, 6,900 for observables.
constexpr int SMALL_BEADS = 8192, SMALL_CELLS = 16 * SCAN_BLOCK;
__global__ void __launch_bounds__(SCAN_BLOCK) k_cells_small(const CellParams C, int ncell) {
  extern __shared__ int cnt[];  // [ncell]
  __shared__ int sh[33];
  __shared__ double o[3];
  for (int i = threadIdx.x; i < ncell; i += SCAN_BLOCK) cnt[i] = 0;
  if (C.domain) sweep_shift(C, o);
  if (C.counters && threadIdx.x < 3) C.counters[threadIdx.x] = 0;
  __syncthreads();
  const int n = (int)C.n;
  for (int b = threadIdx.x; b < n; b += SCAN_BLOCK) C.rank[b] = atomicAdd(&cnt[tag_and_cell(C, b, o)], 1);
  __syncthreads();
  int carry = 0;
  for (int c0 = 0; c0 < ncell; c0 += SCAN_TILE) {
    const int base = c0 + threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = base + i < ncell ? cnt[base + i] : 0;
    const int total = block_scan(v, sh);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i)
      if (base + i < ncell) {
        cnt[base + i] = v[i] + carry;
        C.start[base + i] = v[i] + carry;
      }
    carry += total;
  }
  if (threadIdx.x == 0) C.start[ncell] = carry;
  __syncthreads();
  for (int b = threadIdx.x; b < n; b += SCAN_BLOCK) scatter_bead(C, b, cnt[C.cell[b]] + C.rank[b]);
}

__global__ void k_tag_count_b(const CellBatch C) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x == 0 && threadIdx.x < 3) C.counters[threadIdx.x] = 0;
  if (b >= C.n) return;
  const RepParams &R = C.reps[C.rep_of[b]];
  const double rr[3] = {C.r[3 * b], C.r[3 * b + 1], C.r[3 * b + 2]};
  const u64x4 w = philox(TAG_SHIFT, (uint64_t)*C.sweep_dev, 0, 0, C.seed, R.replica);
  int k[3], c[3];
  bool in = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double o = unit53(w.v[a]) * R.T[a];
    double u = rr[a] - o;
    if (u < 0.0) u = u + R.L[a];
    if (u >= R.L[a]) u = u - R.L[a];
    int t = (int)(u / R.T[a]);
    if (t > R.D[a] - 1) t = R.D[a] - 1;
    const double loc = u - (double)t * R.T[a];
    in = in && (loc < R.W[a]);
    k[a] = t;
    int q = (int)(rr[a] / R.cs[a]);
    if (q >= R.nc[a]) q = R.nc[a] - 1;
    if (q < 0) q = 0;
    c[a] = q;
  }
  C.tag[b] = in ? (k[2] * R.D[1] + k[1]) * R.D[0] + k[0] : -1;
  const int64_t cell = R.cell_off + (c[2] * R.nc[1] + c[1]) * R.nc[0] + c[0];
  C.cell[b] = (int32_t)cell;
  C.rank[b] = atomicAdd(&C.count[cell], 1);
}

__global__ void k_scatter_b(const CellBatch C) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= C.n) return;
  const int64_t pos = (int64_t)C.start[C.cell[b]] + C.rank[b];
  const double x = C.r[3 * b], y = C.r[3 * b + 1], z = C.r[3 * b + 2];
  C.crf[3 * pos] = (float)x;
  C.crf[3 * pos + 1] = (float)y;
  C.crf[3 * pos + 2] = (float)z;
  C.rf[3 * b] = (float)x;
  C.rf[3 * b + 1] = (float)y;
  C.rf[3 * b + 2] = (float)z;
  const RepParams &R = C.reps[C.rep_of[b]];
  const int64_t id = b - R.bead_off;
  C.cid[pos] = (int32_t)id;
  const int32_t t = C.tag[b];
  if (t >= 0) {
    C.ctag[pos] = t;
  } else {
    const int64_t c = id % R.N;
    C.ctag[pos] = joint_tag(c != 0 ? C.tag[b - 1] : -1, c != R.N - 1 ? C.tag[b + 1] : -1);
  }
}

__global__ void k_sweep_advance(int64_t *sweep) { *sweep += 1; }

}  // namespace

cudaError_t launch_cells_batch(const CellBatch &C, int64_t ncell, cudaStream_t s) {
  const int T = 256;
  const int64_t nb = (C.n + T - 1) / T;
  if (C.n > 0) k_tag_count_b<<<(unsigned)nb, T, 0, s>>>(C);
  launch_scan(C.count, ncell, C.start, C.block_sums, s);
  if (C.n > 0) k_scatter_b<<<(unsigned)nb, T, 0, s>>>(C);
  return cudaGetLastError();
}

cudaError_t launch_sweep_advance(int64_t *sweep_dev, cudaStream_t s) {
  k_sweep_advance<<<1, 1, 0, s>>>(sweep_dev);
  return cudaGetLastError();
}

size_t cells_scratch_ints(int64_t ncell) { return (size_t)((ncell + SCAN_TILE - 1) / SCAN_TILE) + 1; }

cudaError_t launch_cells(const CellParams &C0, int64_t ncell, cudaStream_t s) {
  CellParams C = C0;
  float Lmax = 0.f;
  for (int a = 0; a < 3; ++a) {
    C.Lf[a] = (float)C.L[a];
    C.cinv_f[a] = (float)(1.0 / C.cs[a]);
    C.Tf[a] = (float)C.T[a];
    C.Wf[a] = (float)C.W[a];
    C.tinv_f[a] = C.T[a] > 0.0 ? (float)(1.0 / C.T[a]) : 0.f;
    Lmax = C.Lf[a] > Lmax ? C.Lf[a] : Lmax;
  }
  // error of a coordinate (truncated to FP32, less a truncated shift, wrapped,
  // less k T): below 8 L / 2^23, taken twice
  C.tol = 16.f * Lmax / 8388608.f;
  if (C.n > 0 && C.n <= SMALL_BEADS && ncell <= SMALL_CELLS) {
    const cudaError_t e = cudaFuncSetAttribute(k_cells_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(int) * SMALL_CELLS);
    if (e != cudaSuccess) return e;
    k_cells_small<<<1, SCAN_BLOCK, sizeof(int) * (size_t)ncell, s>>>(C, (int)ncell);
    return cudaGetLastError();
  }
  const int T = 256;
  const int64_t nb = (C.n + T - 1) / T;
  if (C.n > 0) k_tag_count<<<(unsigned)nb, T, 0, s>>>(C);
  launch_scan(C.count, ncell, C.start, C.block_sums, s);
  if (C.n > 0) k_scatter<<<(unsigned)nb, T, 0, s>>>(C);
  return cudaGetLastError();
}

}  // namespace ecmc
