// Chain structure of the current state (arXiv:1502.06447, Sec. IV: radius
// of gyration and the relative MSD g2 of the middle bead; Appendix A: the
// moment of inertia tensor of a chain, its shape descriptors, and the
// end-to-end distance distribution W(R); Sec. II.B: mean-square internal
// distances R^2(n)).
//
// Positions along a chain come from minimum-image bonds: u_0 = 0,
// u_{j+1} = u_j + minimg(r_{j+1} - r_j).  The gyration tensor
// S = (1/N) sum_j (u_j - U)(u_j - U)^T with U = (1/N) sum_j u_j; the
// moment of inertia tensor is N (Tr S 1 - S), so its eigenvalue
// combinations follow from those of S.  Every sum runs in index order
// (beads, then chains), so all sums, S, R^2(n) and W(R) are reproducible
// bit for bit; the eigenvalues come from a cyclic Jacobi iteration.
#include <cuda_runtime.h>

#include "ecmc_dev.cuh"
#include "ecmc_internal.h"

namespace ecmc {
namespace {

// Eigenvalues of a symmetric 3x3 matrix, ascending: cyclic Jacobi rotations
// (Rutishauser's formulation: t = sgn(theta) / (|theta| + sqrt(theta^2 + 1)),
// theta = (a_qq - a_pp) / (2 a_pq)), until the off-diagonal part is below
// 1e-18 of the diagonal or after 12 sweeps.
__device__ void sym3_eigen(double a00, double a01, double a02, double a11, double a12, double a22,
                           double &l0, double &l1, double &l2) {
  for (int sweep = 0; sweep < 12; ++sweep) {
    const double off = fabs(a01) + fabs(a02) + fabs(a12);
    if (off <= 1e-18 * (fabs(a00) + fabs(a11) + fabs(a22)) || off == 0.0) break;
#pragma unroll
    for (int pq = 0; pq < 3; ++pq) {
      // (p, q) = (0, 1), (0, 2), (1, 2); r is the third index
      double &app = pq == 2 ? a11 : a00;
      double &aqq = pq == 0 ? a11 : a22;
      double &apq = pq == 0 ? a01 : (pq == 1 ? a02 : a12);
      double &arp = pq == 0 ? a02 : (pq == 1 ? a01 : a01);  // a_rp
      double &arq = pq == 0 ? a12 : (pq == 1 ? a12 : a02);  // a_rq
      if (apq == 0.0) continue;
      const double theta = div_rn(aqq - app, 2.0 * apq);
      double t;
      if (fabs(theta) > 1e150) {
        t = 0.5 / theta;
      } else {
        t = div_rn(1.0, fabs(theta) + sqrt_rn(theta * theta + 1.0));
        if (theta < 0.0) t = -t;
      }
      const double c = div_rn(1.0, sqrt_rn(t * t + 1.0)), s = t * c;
      app = app - t * apq;
      aqq = aqq + t * apq;
      apq = 0.0;
      const double xp = arp, xq = arq;
      arp = c * xp - s * xq;
      arq = s * xp + c * xq;
    }
  }
  // ascending order of the diagonal
  double x = a00, y = a11, z = a22, w;
  if (x > y) { w = x; x = y; y = w; }
  if (y > z) { w = y; y = z; z = w; }
  if (x > y) { w = x; x = y; y = w; }
  l0 = x;
  l1 = y;
  l2 = z;
}

// Positions along the chains (into u), the gyration tensor and its shape
// values, the middle bead relative to the centre of mass, g2's summand,
// |R_e|^2 and the end-to-end bin.
//
// Every sum runs in bead order, one dependent FP64 addition (64 cycles) per
// bead, so a chain's time is set by how many additions stand in that line.
// One thread per chain had 17 FP64 instructions and its own uncoalesced
// loads per bead (1.69 ms on 1000 chains of 1000).  A warp now takes five
// chains: all lanes load a chunk of beads and do what is independent (bond
// vectors; differences to the centre and their products) into shared memory,
// then a lane per sum adds its column in order (three axes of u and of its
// sum, later the six components of S).
constexpr int SC_CHAINS = 5, SC_CHUNK = 32;
__global__ void __launch_bounds__(32) k_struct_chain(const StructParams S) {
  __shared__ double sh[SC_CHAINS][SC_CHUNK][6];  // first pass: bond vectors, then u, in [0..2]
  const int lane = threadIdx.x;
  const int64_t nch = S.n / S.N;
  const int64_t ch0 = (int64_t)blockIdx.x * SC_CHAINS;
  const int nc = nch - ch0 < SC_CHAINS ? (int)(nch - ch0) : SC_CHAINS;
  const int N = S.N;
  const double *const r = S.r + 3 * ch0 * N;
  double *const u = S.u + 3 * ch0 * N;
  // lane 3 q + a: chain q, axis a
  const int q3 = lane / 3, a3 = lane % 3;
  const bool on3 = q3 < nc;
  double x = 0.0, t = 0.0, mid = 0.0;
  const int h = N / 2;
  if (on3) u[3 * (int64_t)q3 * N + a3] = 0.0;
  // element lane + 32 m of a chain's chunk (m = 0, 1, 2): bead ib[m], axis ia[m]
  int ib[3], ia[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    ib[m] = (lane + 32 * m) / 3;
    ia[m] = (lane + 32 * m) % 3;
  }
  // the next chunk's coordinates are loaded while this one's sums are taken
  double lo[3 * SC_CHAINS], hi[3 * SC_CHAINS];
  auto fetch = [&](int j0) {
    const int left = 3 * (N - 1 - j0);
#pragma unroll
    for (int k = 0; k < 3 * SC_CHAINS; ++k) {
      const int i = lane + 32 * (k % 3);
      if (k / 3 < nc && i < left) {
        const double *const p = r + 3 * ((int64_t)(k / 3) * N + j0) + i;
        lo[k] = p[0];
        hi[k] = p[3];
      }
    }
  };
  fetch(0);
  for (int j0 = 0; j0 + 1 < N; j0 += SC_CHUNK) {
    const int cnt = N - 1 - j0 < SC_CHUNK ? N - 1 - j0 : SC_CHUNK;  // bonds of the chunk
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 3 * SC_CHAINS; ++k)
      if (k / 3 < nc && lane + 32 * (k % 3) < 3 * cnt)
        sh[k / 3][ib[k % 3]][ia[k % 3]] = wrap_bits(hi[k] - lo[k], S.L[ia[k % 3]], S.half[ia[k % 3]]);
    __syncwarp();
    if (j0 + SC_CHUNK + 1 < N) fetch(j0 + SC_CHUNK);
    if (on3) {
      for (int j = 0; j < cnt; ++j) {
        x = x + sh[q3][j][a3];
        t = t + x;
        sh[q3][j][a3] = x;
        if (j0 + j + 1 == h) mid = x;
      }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 3 * SC_CHAINS; ++k)
      if (k / 3 < nc && lane + 32 * (k % 3) < 3 * cnt)
        u[3 * ((int64_t)(k / 3) * N + j0 + 1) + lane + 32 * (k % 3)] = sh[k / 3][ib[k % 3]][ia[k % 3]];
  }
  const double U = div_rn(t, (double)N);
  // the six components of S: lane 6 q + k, (0 0) (0 1) (0 2) (1 1) (1 2) (2 2)
  const int q6 = lane / 6, k6 = lane % 6;
  double s = 0.0;
  __threadfence_block();
  __syncwarp();
  auto fetch_u = [&](int j0) {
#pragma unroll
    for (int q = 0; q < SC_CHAINS; ++q)
      if (q < nc && j0 + lane < N) {
        const double *const p = u + 3 * ((int64_t)q * N + j0 + lane);
        lo[3 * q] = p[0];
        lo[3 * q + 1] = p[1];
        lo[3 * q + 2] = p[2];
      }
  };
  fetch_u(0);
  for (int j0 = 0; j0 < N; j0 += SC_CHUNK) {
    const int cnt = N - j0 < SC_CHUNK ? N - j0 : SC_CHUNK;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < SC_CHAINS; ++q) {
      const double U0 = __shfl_sync(0xffffffffu, U, 3 * q), U1 = __shfl_sync(0xffffffffu, U, 3 * q + 1),
                   U2 = __shfl_sync(0xffffffffu, U, 3 * q + 2);
      if (q < nc && lane < cnt) {
        const double d0 = lo[3 * q] - U0, d1 = lo[3 * q + 1] - U1, d2 = lo[3 * q + 2] - U2;
        sh[q][lane][0] = d0 * d0;
        sh[q][lane][1] = d0 * d1;
        sh[q][lane][2] = d0 * d2;
        sh[q][lane][3] = d1 * d1;
        sh[q][lane][4] = d1 * d2;
        sh[q][lane][5] = d2 * d2;
      }
    }
    __syncwarp();
    if (j0 + SC_CHUNK < N) fetch_u(j0 + SC_CHUNK);
    if (q6 < nc)
      for (int j = 0; j < cnt; ++j) s = s + sh[q6][j][k6];
  }
  s = div_rn(s, (double)N);
  // one lane per chain finishes it
  const int q = lane < nc ? lane : 0;
  const double s00 = __shfl_sync(0xffffffffu, s, 6 * q), s01 = __shfl_sync(0xffffffffu, s, 6 * q + 1),
               s02 = __shfl_sync(0xffffffffu, s, 6 * q + 2), s11 = __shfl_sync(0xffffffffu, s, 6 * q + 3),
               s12 = __shfl_sync(0xffffffffu, s, 6 * q + 4), s22 = __shfl_sync(0xffffffffu, s, 6 * q + 5);
  const double u0 = __shfl_sync(0xffffffffu, x, 3 * q), u1 = __shfl_sync(0xffffffffu, x, 3 * q + 1),
               u2 = __shfl_sync(0xffffffffu, x, 3 * q + 2);
  mid = mid - U;
  const double m0 = __shfl_sync(0xffffffffu, mid, 3 * q), m1 = __shfl_sync(0xffffffffu, mid, 3 * q + 1),
               m2 = __shfl_sync(0xffffffffu, mid, 3 * q + 2);
  if (lane >= nc) return;
  const int64_t ch = ch0 + lane;
  const double T = (s00 + s11) + s22;
  const double P = ((s00 * s11 - s01 * s01) + (s00 * s22 - s02 * s02)) + (s11 * s22 - s12 * s12);
  double l0, l1, l2;
  sym3_eigen(s00, s01, s02, s11, s12, s22, l0, l1, l2);
  double g2 = 0.0;
  if (S.mref) {
    const double e0 = m0 - S.mref[3 * ch], e1 = m1 - S.mref[3 * ch + 1], e2 = m2 - S.mref[3 * ch + 2];
    g2 = (e0 * e0 + e1 * e1) + e2 * e2;
  }
  const double re2 = (u0 * u0 + u1 * u1) + u2 * u2;
  if (S.hist && S.nbins > 0) {
    int64_t b = (int64_t)floor(sqrt(re2) / S.dR);
    if (b >= S.nbins) b = S.nbins - 1;
    atomicAdd(&S.hist[b], 1ull);
  }
  double *o = S.rec + STRUCT_REC * ch;
  o[0] = T;
  o[1] = l0;
  o[2] = l1;
  o[3] = l2;
  o[4] = l2 - 0.5 * (l0 + l1);     // asphericity
  o[5] = l1 - l0;                  // acylindricity
  o[6] = 1.0 - 3.0 * P / (T * T);  // shape anisotropy
  o[7] = 4.0 * (T * T - 3.0 * P);  // 4 b^2 + 3 c^2
  o[8] = g2;
  o[9] = re2;
  o[10] = m0;
  o[11] = m1;
  o[12] = m2;
}

// ---------------------------------------------------------------- R^2(n)
// A pair term of R^2(n) is nine FP64 operations, and an FP64 warp instruction
// takes its unit 64 cycles: 576 cycles per term.  The three squares are done
// in integer arithmetic beside it (square_rn, the same bits).

// R^2(n) partial sums: thread (chain, n) adds |u_{j+n} - u_j|^2 over j
__global__ void k_struct_r2n(const StructParams S) {
  const int N = S.N;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nch = S.n / N;
  if (t >= nch * (N - 1)) return;
  const int64_t ch = t / (N - 1);
  const int n = 1 + (int)(t % (N - 1));
  const double *uc = S.u + 3 * ch * N;
  double part = 0.0;
  for (int j = 0; j + n < N; ++j) {
    const double d0 = uc[3 * (j + n)] - uc[3 * j];
    const double d1 = uc[3 * (j + n) + 1] - uc[3 * j + 1];
    const double d2 = uc[3 * (j + n) + 2] - uc[3 * j + 2];
    part = part + ((square_rn(d0) + square_rn(d1)) + square_rn(d2));
  }
  S.part[ch * N + n] = part;
}

// The same with a block per chain, its positions in shared memory: thread i
// takes the lags 1 + i and N - 1 - i, N terms together, so all threads of a
// block finish at the same time.
__global__ void __launch_bounds__(512) k_struct_r2n_chain(const StructParams S) {
  extern __shared__ double su[];  // [3][N]
  const int N = S.N;
  const int64_t ch = blockIdx.x;
  const double *const uc = S.u + 3 * ch * N;
  for (int i = threadIdx.x; i < 3 * N; i += blockDim.x) su[(i % 3) * N + i / 3] = uc[i];
  __syncthreads();
  const double *const x = su, *const y = su + N, *const z = su + 2 * N;
  for (int i = threadIdx.x; 2 * i < N - 1; i += blockDim.x) {
    const int na = 1 + i, nb = N - 1 - i;
    // first the terms of lag na, then those of lag nb
    int n = na, j = 0;
    double part = 0.0;
    const int terms = na == nb ? N - na : N;
    for (int k = 0; k < terms; ++k) {
      const double d0 = x[j + n] - x[j], d1 = y[j + n] - y[j], d2 = z[j + n] - z[j];
      part = part + ((square_rn(d0) + square_rn(d1)) + square_rn(d2));
      ++j;
      if (j + n == N) {
        S.part[ch * N + n] = part;
        part = 0.0;
        n = nb;
        j = 0;
      }
    }
  }
}

// sums over chains in chain order: the record columns (last block) and
// R^2(n) (one thread per n, a warp per block).  Eight loads ahead of the additions, which
// have to follow one another.
__global__ void __launch_bounds__(32) k_struct_sum(const StructParams S) {
  const int64_t nch = S.n / S.N;
  auto column = [&](const double *p, int64_t stride) {
    double s = 0.0;
    int64_t ch = 0;
    for (; ch + 8 <= nch; ch += 8) {
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = p[(ch + k) * stride];
#pragma unroll
      for (int k = 0; k < 8; ++k) s = s + v[k];
    }
    for (; ch < nch; ++ch) s = s + p[ch * stride];
    return s;
  };
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x < STRUCT_SUMS) S.sums[threadIdx.x] = column(S.rec + threadIdx.x, STRUCT_REC);
    return;
  }
  const int n = blockIdx.x * 32 + threadIdx.x;
  if (n >= S.N) return;
  S.r2n[n] = n == 0 ? 0.0 : column(S.part + n, S.N) / ((double)nch * (double)(S.N - n));
}

}  // namespace

cudaError_t launch_struct(const StructParams &S, cudaStream_t s) {
  const int64_t nch = S.n / S.N;
  if (nch <= 0 || S.N < 2) return cudaErrorInvalidValue;
  if (S.hist && S.nbins > 0) {
    cudaError_t e = cudaMemsetAsync(S.hist, 0, sizeof(unsigned long long) * (size_t)S.nbins, s);
    if (e != cudaSuccess) return e;
  }
  k_struct_chain<<<(unsigned)((nch + SC_CHAINS - 1) / SC_CHAINS), 32, 0, s>>>(S);
  if (S.r2n) {
    // a block per chain once a chain's lags fill most of a warp; longer chains
    // than fit shared memory read it from the global array.  Whole call on 1e6
    // beads, a thread per lag / a block per chain: N = 16 3.38 / 3.65 ms, 32
    // 2.11 / 2.14, 40 2.01 / 1.92, 50 1.87 / 1.66, 64 1.84 / 1.47.
    const size_t smem = sizeof(double) * 3 * (size_t)S.N;
    if (S.N >= 48 && smem <= 96 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(k_struct_r2n_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
      if (e != cudaSuccess) return e;
      const int want = ((S.N - 1 + 1) / 2 + 31) / 32 * 32;
      k_struct_r2n_chain<<<(unsigned)nch, want < 512 ? want : 512, smem, s>>>(S);
    } else {
      const int64_t work = nch * (S.N - 1);
      k_struct_r2n<<<(unsigned)((work + 255) / 256), 256, 0, s>>>(S);
    }
  }
  k_struct_sum<<<(S.r2n ? (S.N + 31) / 32 : 0) + 1, 32, 0, s>>>(S);
  return cudaGetLastError();
}

}  // namespace ecmc
