// Fused observables over the current state and the initial lattice.
//
//   R_e^2 per chain from minimum-image bonds (end-to-end distance, Sec. IV
//   and the ideal-chain law <R^2> = c N sigma^2); bond lengths and tether
//   violations (b > b_max); hard-sphere overlaps (Eq. 1) from the cell list;
//   g1, the mean-square displacement of the middle bead N/2 (Eq. for g1 in
//   Sec. IV) against a reference snapshot of unwrapped positions; pair and
//   bond counts in thin shells at contact (sigma, b_max) for the
//   contact-value pressure.
#include <cuda_runtime.h>

#include "ecmc_dev.cuh"
#include "ecmc_internal.h"

namespace ecmc {
namespace {

__device__ __forceinline__ void atomic_max_pos(double *a, double v) {
  atomicMax((unsigned long long *)a, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void atomic_min_pos(double *a, double v) {
  atomicMin((unsigned long long *)a, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ double warp_sum(double v, int width = 32) {
  for (int off = width / 2; off > 0; off >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Bonds of every chain: g threads per chain (a power of two up to a warp, or
// the whole block), one bond per thread and round; sums over threads, then one
// set of atomics per warp.
// One thread per chain took 1.75 ms on 1000 chains of 1000 beads (1000
// threads on the chip, each a chain of dependent loads and FP64 operations);
// spread over the bonds the FP64 units bound it: 13 instructions per bond,
// 20 us there.
// out_d: [0] sum R_e^2, [1] max bond, [2] min bond, [3] sum g1, [4] sum of bond lengths
// out_u: [0] overlaps, [1] tether violations, [4] [5] bonds in the shells
// (t1, t0] and (t2, t1] below b_max
__global__ void __launch_bounds__(128) k_chains(const ObsParams O, int g) {
  __shared__ double Rs[3][4];
  const int lane = threadIdx.x & 31, gl = threadIdx.x & (g - 1);
  const int64_t ch = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / g;
  const int64_t nch = O.n / O.N;
  const bool live = ch < nch;
  double R0 = 0.0, R1 = 0.0, R2 = 0.0, bsum = 0.0;
  double dmax = 0.0, dmin = 1e300;  // squared bond lengths
  unsigned viol = 0, tb0 = 0, tb1 = 0;
  const double lim = O.b2 * (1.0 + 1e-10);
  for (int j = gl; live && j + 1 < O.N; j += g) {
    const double *q = O.r + 3 * (ch * O.N + j);
    const double d0 = wrap_bits(q[3] - q[0], O.L[0], O.half[0]);
    const double d1 = wrap_bits(q[4] - q[1], O.L[1], O.half[1]);
    const double d2 = wrap_bits(q[5] - q[2], O.L[2], O.half[2]);
    R0 += d0;
    R1 += d1;
    R2 += d2;
    const double dd = d0 * d0 + d1 * d1 + d2 * d2;
    viol += less_pos(lim, dd);
    tb0 += less_pos(O.c_t1, dd) && !less_pos(O.c_t0, dd);
    tb1 += less_pos(O.c_t2, dd) && !less_pos(O.c_t1, dd);
    bsum += sqrt_rn(dd);
    if (less_pos(dmax, dd)) dmax = dd;
    if (less_pos(dd, dmin)) dmin = dd;
  }
  const int gw = g < 32 ? g : 32;
  R0 = warp_sum(R0, gw);
  R1 = warp_sum(R1, gw);
  R2 = warp_sum(R2, gw);
  if (g > 32) {
    if (lane == 0) {
      Rs[0][threadIdx.x >> 5] = R0;
      Rs[1][threadIdx.x >> 5] = R1;
      Rs[2][threadIdx.x >> 5] = R2;
    }
    __syncthreads();
    R0 = (Rs[0][0] + Rs[0][1]) + (Rs[0][2] + Rs[0][3]);
    R1 = (Rs[1][0] + Rs[1][1]) + (Rs[1][2] + Rs[1][3]);
    R2 = (Rs[2][0] + Rs[2][1]) + (Rs[2][2] + Rs[2][3]);
  }
  double re2 = 0.0, g1 = 0.0;
  if (live && gl == 0) {
    re2 = R0 * R0 + R1 * R1 + R2 * R2;
    if (O.g1ref) {
      const int64_t b = ch * O.N + O.N / 2;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double u = O.r[3 * b + a] + (double)O.img[3 * b + a] * O.L[a];
        const double d = u - O.g1ref[3 * ch + a];
        g1 += d * d;
      }
    }
  }
  re2 = warp_sum(re2);
  bsum = warp_sum(bsum);
  if (O.g1ref) g1 = warp_sum(g1);
  for (int off = 16; off > 0; off >>= 1) {
    const double a = __shfl_xor_sync(0xffffffffu, dmax, off), b = __shfl_xor_sync(0xffffffffu, dmin, off);
    if (less_pos(dmax, a)) dmax = a;
    if (less_pos(b, dmin)) dmin = b;
  }
  viol = __reduce_add_sync(0xffffffffu, viol);
  tb0 = __reduce_add_sync(0xffffffffu, tb0);
  tb1 = __reduce_add_sync(0xffffffffu, tb1);
  if (lane != 0 || !live) return;
  atomicAdd(&O.out_d[0], re2);
  if (O.N > 1) {
    atomicAdd(&O.out_d[4], bsum);
    // (the square root is monotone: the longest bond is that of the largest square)
    atomic_max_pos(&O.out_d[1], sqrt_rn(dmax));
    atomic_min_pos(&O.out_d[2], sqrt_rn(dmin));
  }
  if (viol) atomicAdd(&O.out_u[1], (unsigned long long)viol);
  if (tb0) atomicAdd(&O.out_u[4], (unsigned long long)tb0);
  if (tb1) atomicAdd(&O.out_u[5], (unsigned long long)tb1);
  if (O.g1ref) atomicAdd(&O.out_d[3], g1);
}

__global__ void k_snapshot(const ObsParams O, double *ref) {
  const int64_t ch = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nch = O.n / O.N;
  if (ch >= nch) return;
  const int64_t b = ch * O.N + O.N / 2;
#pragma unroll
  for (int a = 0; a < 3; ++a) ref[3 * ch + a] = O.r[3 * b + a] + (double)O.img[3 * b + a] * O.L[a];
}

// the beads of the cells x = cx + x0 .. cx + x1 of row (y, z): one or two
// contiguous ranges of the cell-ordered arrays
template <class F>
__device__ __forceinline__ void row_ranges(const ObsParams &O, int cx, int x0, int x1, int y, int z, F f) {
  const int nx = O.nc[0];
  const int *const st = O.cstart + (z * O.nc[1] + y) * nx;
  int a = cx + x0, b = cx + x1;  // inclusive
  if (a < 0) {
    f(st[a + nx], st[nx]);
    a = 0;
  } else if (b >= nx) {
    f(st[0], st[b - nx + 1]);
    b = nx - 1;
  }
  f(st[a], st[b + 1]);
}

// pairs closer than sigma (1 - 1e-10)^(1/2), and pairs in the shells
// [lo, s1) and [s1, s2) above sigma, through the cell list (cell side >=
// sqrt(s2), at least 3 cells per axis).  A thread takes a bead in cell order
// and the half of its neighbourhood ahead of it (its own cell past itself,
// the next cell, three rows' worth of the rest), so that every pair is seen
// once.  FP32 positions classify a pair; only one within their error of a
// bound is measured in FP64.
__global__ void __launch_bounds__(128) k_overlaps(const ObsParams O) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned cnt = 0, cs0 = 0, cs1 = 0;
  if (t < O.n) {
    const int c = O.cell[O.cid[t]];
    const int cx = c % O.nc[0], cy = (c / O.nc[0]) % O.nc[1], cz = c / (O.nc[0] * O.nc[1]);
    const float p0 = O.crf[3 * t], p1 = O.crf[3 * t + 1], p2 = O.crf[3 * t + 2];
    const float L0 = O.Lf[0], L1 = O.Lf[1], L2 = O.Lf[2];
    const double lim = O.sig2 * (1.0 - 1e-10);
    auto one = [&](int j) {
      float d0 = p0 - O.crf[3 * (int64_t)j], d1 = p1 - O.crf[3 * (int64_t)j + 1],
            d2 = p2 - O.crf[3 * (int64_t)j + 2];
      d0 = fabsf(d0);
      d1 = fabsf(d1);
      d2 = fabsf(d2);
      d0 = fminf(d0, L0 - d0);
      d1 = fminf(d1, L1 - d1);
      d2 = fminf(d2, L2 - d2);
      const float f = __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, d0 * d0));
      if (f > O.f_s2 + O.f_err) return;
      if (fabsf(f - O.f_lo) > O.f_err && fabsf(f - O.f_s1) > O.f_err && fabsf(f - O.f_s2) > O.f_err) {
        cnt += f < O.f_lo;
        cs0 += f > O.f_lo && f < O.f_s1;
        cs1 += f > O.f_s1 && f < O.f_s2;
        return;
      }
      const double e0 = wrap_bits(O.cr[3 * t] - O.cr[3 * (int64_t)j], O.L[0], O.half[0]);
      const double e1 = wrap_bits(O.cr[3 * t + 1] - O.cr[3 * (int64_t)j + 1], O.L[1], O.half[1]);
      const double e2 = wrap_bits(O.cr[3 * t + 2] - O.cr[3 * (int64_t)j + 2], O.L[2], O.half[2]);
      const double dd = e0 * e0 + e1 * e1 + e2 * e2;
      cnt += less_pos(dd, lim);
      cs0 += !less_pos(dd, O.c_lo) && less_pos(dd, O.c_s1);
      cs1 += !less_pos(dd, O.c_s1) && less_pos(dd, O.c_s2);
    };
    auto range = [&](int j0, int j1) {
      for (int j = j0; j < j1; ++j) one(j);
    };
    range((int)t + 1, O.cstart[c + 1]);
    row_ranges(O, cx, 1, 1, cy, cz, range);
    const int yn = cy + 1 == O.nc[1] ? 0 : cy + 1;
    row_ranges(O, cx, -1, 1, yn, cz, range);
    const int zn = cz + 1 == O.nc[2] ? 0 : cz + 1;
    const int yp = cy == 0 ? O.nc[1] - 1 : cy - 1;
    row_ranges(O, cx, -1, 1, yp, zn, range);
    row_ranges(O, cx, -1, 1, cy, zn, range);
    row_ranges(O, cx, -1, 1, yn, zn, range);
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  cs0 = __reduce_add_sync(0xffffffffu, cs0);
  cs1 = __reduce_add_sync(0xffffffffu, cs1);
  if ((threadIdx.x & 31) != 0) return;
  if (cnt) atomicAdd(&O.out_u[0], (unsigned long long)cnt);
  if (cs0) atomicAdd(&O.out_u[2], (unsigned long long)cs0);
  if (cs1) atomicAdd(&O.out_u[3], (unsigned long long)cs1);
}

__global__ void k_lattice(int n0, int n1, int n2, double a, double jitter, uint64_t seed,
                          uint64_t replica, double *r, int64_t n) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const int64_t plane = (int64_t)n0 * n1;
  const int z = (int)(b / plane);
  const int64_t rem = b % plane;
  const int yy = (int)(rem / n0), xx = (int)(rem % n0);
  const int y = (z % 2 == 0) ? yy : n1 - 1 - yy;
  const int row = z * n1 + yy;
  const int x = (row % 2 == 0) ? xx : n0 - 1 - xx;
  const int site[3] = {x, y, z};
  u64x4 w;
  w.v[0] = w.v[1] = w.v[2] = w.v[3] = 0;
  if (jitter != 0.0) w = philox(TAG_JITTER, 0, (uint64_t)b, 0, seed, replica);
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    double p = ((double)site[ax] + 0.5) * a;
    if (jitter != 0.0) p = p + jitter * (2.0 * unit53(w.v[ax]) - 1.0);
    r[3 * b + ax] = p;
  }
}

// beads that overlap another bead (|d|^2 < thr, minimum image, squared
// length (d0 d0 + d1 d1) + d2 d2) through the cell list: flag 0/1 per bead
// and their number (the push-off's start beads, Sec. II.B).  A warp per
// bead, one of the 27 cells per lane: a push-off has a few thousand beads, and
// one thread per bead left most of the chip idle (180 us on 2,400 beads).
// FP32 positions decide unless the square lies within their error of thr.
__global__ void __launch_bounds__(128) k_po_flags(const ObsParams O, double thr, float thr_f, float err,
                                                  uint8_t *flag, unsigned long long *count) {
  const int lane = threadIdx.x & 31;
  const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (t >= O.n) return;
  const int i = O.cid[t];
  bool f = false;
  if (lane < 27) {
    const int c = O.cell[i];
    int x = c % O.nc[0] + lane % 3 - 1, y = (c / O.nc[0]) % O.nc[1] + (lane / 3) % 3 - 1,
        z = c / (O.nc[0] * O.nc[1]) + lane / 9 - 1;
    x += x < 0 ? O.nc[0] : (x >= O.nc[0] ? -O.nc[0] : 0);
    y += y < 0 ? O.nc[1] : (y >= O.nc[1] ? -O.nc[1] : 0);
    z += z < 0 ? O.nc[2] : (z >= O.nc[2] ? -O.nc[2] : 0);
    const int cc = (z * O.nc[1] + y) * O.nc[0] + x;
    const float p0 = O.crf[3 * t], p1 = O.crf[3 * t + 1], p2 = O.crf[3 * t + 2];
    for (int j = O.cstart[cc]; j < O.cstart[cc + 1] && !f; ++j) {
      if (j == (int)t) continue;
      float d0 = fabsf(p0 - O.crf[3 * (int64_t)j]), d1 = fabsf(p1 - O.crf[3 * (int64_t)j + 1]),
            d2 = fabsf(p2 - O.crf[3 * (int64_t)j + 2]);
      d0 = fminf(d0, O.Lf[0] - d0);
      d1 = fminf(d1, O.Lf[1] - d1);
      d2 = fminf(d2, O.Lf[2] - d2);
      const float q = __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, d0 * d0));
      if (q > thr_f + err) continue;
      if (q < thr_f - err) {
        f = true;
        break;
      }
      const double e0 = wrap_bits(O.cr[3 * t] - O.cr[3 * (int64_t)j], O.L[0], O.half[0]);
      const double e1 = wrap_bits(O.cr[3 * t + 1] - O.cr[3 * (int64_t)j + 1], O.L[1], O.half[1]);
      const double e2 = wrap_bits(O.cr[3 * t + 2] - O.cr[3 * (int64_t)j + 2], O.L[2], O.half[2]);
      f = less_pos((e0 * e0 + e1 * e1) + e2 * e2, thr);
    }
  }
  f = __any_sync(0xffffffffu, f);
  if (lane == 0) {
    flag[i] = f ? 1 : 0;
    if (f) atomicAdd(count, 1ull);
  }
}

// Phantom chains (Sec. II.B, first stage of the initial configuration):
// one thread per chain walks N beads with bond length `bond`, the first bead
// uniform in the box, the first bond uniform on the sphere, every next bond
// uniform on the cap t_j . t_{j+1} >= ct around the one before (cos theta =
// 1 - u (1 - ct); the azimuth from the first point of the unit disc drawn
// as (2u - 1, 2u' - 1), at most 256 attempts; the orthonormal pair of t_j
// after Duff et al., "Building an orthonormal basis, revisited", JCGT 2017);
// Philox4x64-10 key (seed, 0), counter (TAG_PHANTOM, chain, bead, attempt).
// Writes unwrapped positions; launch_wrap folds them into the box.
__global__ void k_phantom(int64_t nch, int N, double L0, double L1, double L2, double bond,
                          double ct, uint64_t seed, double *r, unsigned long long *bad) {
  const int64_t ch = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (ch >= nch) return;
  u64x4 w = philox(TAG_PHANTOM, (uint64_t)ch, 0, 0, seed, 0);
  double p0 = unit53(w.v[0]) * L0, p1 = unit53(w.v[1]) * L1, p2 = unit53(w.v[2]) * L2;
  double t0 = 0.0, t1 = 0.0, t2 = 1.0;
  double *rc = r + 3 * ch * N;
  rc[0] = p0;
  rc[1] = p1;
  rc[2] = p2;
  for (int j = 1; j < N; ++j) {
    const double ctj = j == 1 ? -1.0 : ct;
    w = philox(TAG_PHANTOM, (uint64_t)ch, (uint64_t)j, 0, seed, 0);
    const double cth = 1.0 - unit53(w.v[0]) * (1.0 - ctj);
    double x = 2.0 * unit53(w.v[1]) - 1.0, y = 2.0 * unit53(w.v[2]) - 1.0;
    double s = x * x + y * y;
    for (uint64_t att = 1; !(s > 0.0 && s <= 1.0); ++att) {
      if (att == 256) {
        atomicAdd(bad, 1ull);
        return;
      }
      w = philox(TAG_PHANTOM, (uint64_t)ch, (uint64_t)j, att, seed, 0);
      x = 2.0 * unit53(w.v[0]) - 1.0;
      y = 2.0 * unit53(w.v[1]) - 1.0;
      s = x * x + y * y;
    }
    const double sq = sqrt(s);
    const double cph = x / sq, sph = y / sq;
    const double sth = sqrt(1.0 - cth * cth);
    const double sg = t2 >= 0.0 ? 1.0 : -1.0;
    const double aa = -1.0 / (sg + t2);
    const double bb = t0 * t1 * aa;
    const double e10 = 1.0 + sg * t0 * t0 * aa, e11 = sg * bb, e12 = -sg * t0;
    const double e20 = bb, e21 = sg + t1 * t1 * aa, e22 = -t1;
    const double n0 = cth * t0 + sth * (cph * e10 + sph * e20);
    const double n1 = cth * t1 + sth * (cph * e11 + sph * e21);
    const double n2 = cth * t2 + sth * (cph * e12 + sph * e22);
    const double q = sqrt(n0 * n0 + n1 * n1 + n2 * n2);
    t0 = n0 / q;
    t1 = n1 / q;
    t2 = n2 / q;
    p0 = p0 + bond * t0;
    p1 = p1 + bond * t1;
    p2 = p2 + bond * t2;
    rc[3 * j] = p0;
    rc[3 * j + 1] = p1;
    rc[3 * j + 2] = p2;
  }
}

// wrap caller positions into [0, L) and fold whole boxes into the image
// counters (the host-side rule, same FP64 operations); counts non-finite
// coordinates
__global__ void k_wrap(double *r, int32_t *img, int64_t n3, double L0, double L1, double L2,
                       unsigned long long *bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  const int a = (int)(i % 3);
  const double L = a == 0 ? L0 : (a == 1 ? L1 : L2);
  double x = r[i];
  if (!isfinite(x)) {
    atomicAdd(bad, 1ull);
    return;
  }
  const double f = floor(x / L);
  x -= f * L;
  if (x >= L) x -= L;
  if (x < 0) x = 0;
  r[i] = x;
  img[i] += (int32_t)f;
}

// g1 table, one block: thread (k, j) adds the squared displacements of the
// middle beads over the lag j P^k (chains in order, (d0 d0 + d1 d1) + d2 d2)
// when sweep t is an origin multiple of P^k and the earlier snapshot exists;
// then every level whose period divides t stores the current snapshot in
// slot (t / P^k) mod P, which no lag of this sweep reads
__global__ void k_g1_track(const G1Track G) {
  const int64_t nch = G.n / G.N;
  const int nlag = G.K * (G.P - 1);
  for (int q = threadIdx.x; q < nlag; q += blockDim.x) {
    const int k = q / (G.P - 1), j = q % (G.P - 1) + 1;
    const int64_t pk = G.Pk[k];
    if (G.t % pk != 0 || G.t / pk < j) continue;
    const int64_t slot = (G.t / pk - j) % G.P;
    const double *old = G.ring + (k * (int64_t)G.P + slot) * nch * 3;
    double s = 0.0;
    for (int64_t ch = 0; ch < nch; ++ch) {
      const int64_t b = ch * G.N + G.N / 2;
      const double u0 = G.r[3 * b] + (double)G.img[3 * b] * G.L[0];
      const double u1 = G.r[3 * b + 1] + (double)G.img[3 * b + 1] * G.L[1];
      const double u2 = G.r[3 * b + 2] + (double)G.img[3 * b + 2] * G.L[2];
      const double d0 = u0 - old[3 * ch], d1 = u1 - old[3 * ch + 1], d2 = u2 - old[3 * ch + 2];
      s = s + ((d0 * d0 + d1 * d1) + d2 * d2);
    }
    G.sum[q] = G.sum[q] + s;
    G.cnt[q] += 1ull;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < (int64_t)G.K * nch; i += blockDim.x) {
    const int k = (int)(i / nch);
    const int64_t ch = i % nch;
    const int64_t pk = G.Pk[k];
    if (G.t % pk != 0) continue;
    const int64_t slot = (G.t / pk) % G.P;
    double *dst = G.ring + ((k * (int64_t)G.P + slot) * nch + ch) * 3;
    const int64_t b = ch * G.N + G.N / 2;
#pragma unroll
    for (int a = 0; a < 3; ++a) dst[a] = G.r[3 * b + a] + (double)G.img[3 * b + a] * G.L[a];
  }
}

__global__ void k_po_advance(const unsigned long long *count, int64_t *ctr) {
  if (*count) {
    ctr[0] += 1;
    ctr[1] += 1;
  }
}

}  // namespace

cudaError_t launch_po_advance(const unsigned long long *count, int64_t *ctr, cudaStream_t s) {
  k_po_advance<<<1, 1, 0, s>>>(count, ctr);
  return cudaGetLastError();
}

cudaError_t launch_g1_track(const G1Track &G, cudaStream_t s) {
  k_g1_track<<<1, 256, 0, s>>>(G);
  return cudaGetLastError();
}

cudaError_t launch_wrap(double *r, int32_t *img, int64_t n, const double L[3],
                        unsigned long long *bad, cudaStream_t s) {
  const int64_t n3 = 3 * n;
  if (n3 > 0) k_wrap<<<(unsigned)((n3 + 255) / 256), 256, 0, s>>>(r, img, n3, L[0], L[1], L[2], bad);
  return cudaGetLastError();
}

// Error of a squared separation near r^2 from FP32 positions in [0, L), with
// u = 2^-24: a difference is off by 2 L u (two positions rounded), one that is
// wrapped by 4 L u (its own rounding near L and the FP32 side of the box), and
// r u; the square by 2 sqrt(3) r times that and 3 r^2 u: at most
// (13.9 L + 6.5 r) r u.  The bound is 16 (L + r) r u and 17 r^2 u more.
static float f32_square_error(const ObsParams &O, double r) {
  double L = O.L[0] > O.L[1] ? O.L[0] : O.L[1];
  L = L > O.L[2] ? L : O.L[2];
  return round_up_f32(16.0 * r * (L + r) / 16777216.0 + 1e-6 * r * r);
}

cudaError_t launch_po_flags(const ObsParams &O, double thr, uint8_t *flag,
                            unsigned long long *count, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  if (O.n > 0)
    k_po_flags<<<(unsigned)((O.n + 3) / 4), 128, 0, s>>>(O, thr, (float)thr, f32_square_error(O, sqrt(thr)), flag,
                                                        count);
  return cudaGetLastError();
}

cudaError_t launch_phantom(int64_t nch, int N, const double L[3], double bond, double ct,
                           uint64_t seed, double *r, unsigned long long *bad, cudaStream_t s) {
  if (nch > 0) k_phantom<<<(unsigned)((nch + 127) / 128), 128, 0, s>>>(nch, N, L[0], L[1], L[2], bond, ct, seed, r, bad);
  return cudaGetLastError();
}

cudaError_t launch_obs(const ObsParams &O0, cudaStream_t s) {
  ObsParams O = O0;
  const int64_t nch = O.n / O.N;
  // A block per chain once it has a few rounds of bonds for one.  Whole call,
  // a warp / a block per chain: 64,000 beads, N = 160: 65.6 / 68.1 us, 320:
  // 75.3 / 65.4, 1000: 87.6 / 67.4; 1e6 beads, N = 160: 151 / 198, 250: 149 /
  // 174, 500: 149 / 161, 1000: 150 / 150, 2000: 186 / 149.
  int g = 1;
  while (g < 32 && g < O.N - 1) g *= 2;
  if (O.N > 256) g = 128;
  if (nch > 0) k_chains<<<(unsigned)((nch * g + 127) / 128), 128, 0, s>>>(O, g);
  O.f_lo = (float)O.c_lo;
  O.f_s1 = (float)O.c_s1;
  O.f_s2 = (float)O.c_s2;
  O.f_err = f32_square_error(O, sqrt(O.c_s2));
  if (O.n > 0 && O.cr) k_overlaps<<<(unsigned)((O.n + 127) / 128), 128, 0, s>>>(O);
  return cudaGetLastError();
}

cudaError_t launch_g1_snapshot(const ObsParams &O, double *g1ref, cudaStream_t s) {
  const int64_t nch = O.n / O.N;
  if (nch > 0) k_snapshot<<<(unsigned)((nch + 127) / 128), 128, 0, s>>>(O, g1ref);
  return cudaGetLastError();
}

cudaError_t launch_lattice(const int32_t dims[3], double a, double jitter, uint64_t seed,
                           uint64_t replica, double *r, int64_t n, cudaStream_t s) {
  if (n > 0)
    k_lattice<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(dims[0], dims[1], dims[2], a, jitter,
                                                         seed, replica, r, n);
  return cudaGetLastError();
}

}  // namespace ecmc
