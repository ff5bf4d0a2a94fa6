// Device helpers shared by the EC kernels (arXiv:1502.06447, Sec. II, II.A,
// II.C): FP64 comparisons on bit patterns, the minimum image, the contact and
// tether distances (Eq. 1), the reflection (Fig. 2c), candidate keys and the
// tie rule, the shared-memory staging of one tile with its slab masks, and
// the FP32 screen.  Included by the kernel translation units only.
#pragma once
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>

#include "ecmc_dev.cuh"
#include "ecmc_internal.h"

namespace ecmc {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// ---------------------------------------------------------------- FP64 bits
__device__ __forceinline__ uint64_t dbits(double x) { return bits_of(x); }
// x < 0.0 (false for -0.0)
__device__ __forceinline__ bool neg(double x) {
  const uint64_t b = dbits(x);
  return (int64_t)b < 0 && (b << 1) != 0;
}
// x > 0.0
__device__ __forceinline__ bool posv(double x) { return (int64_t)dbits(x) > 0; }
// y >= L for L > 0
__device__ __forceinline__ bool ge_pos(double y, double L) {
  return (int64_t)dbits(y) >= (int64_t)dbits(L);
}
__device__ __forceinline__ bool nonzero(double x) { return (dbits(x) << 1) != 0; }
// 2 x, exact (|x| zero or normal and below 2^1022)
__device__ __forceinline__ double twice(double x) { return from_bits(dbits(x) + (nonzero(x) ? 1ull << 52 : 0ull)); }

// y = r + x v on one axis back into [0, L); returns the image change
__device__ __forceinline__ int wrap_step(double &y, double L) {
  int di = 0;
  if (ge_pos(y, L)) {
    y = add_fp64(y, flip(L));
    di = 1;
  } else if (neg(y)) {
    y = add_fp64(y, L);
    di = -1;
    if (ge_pos(y, L)) {
      y = 0.0;
      di = 0;
    }
  }
  return di;
}

// Hard-sphere contact (Eq. 1, R2 = sigma^2) or tether limit (R2 = b_max^2)
// of a pivot moving along v, d = pivot - partner.  Returns x >= 0, or -1 when
// a contact candidate misses; dv = d.v.
// (skip_overlap: a hard sphere the pivot overlaps is no obstacle, the
// push-off rule of Sec. II.B)
__device__ __forceinline__ double quad_x(bool tether, double d0, double d1, double d2, double v0,
                                         double v1, double v2, double R2, double &dv,
                                         bool skip_overlap = false) {
  // (straight-line: the lanes of a warp hold different candidates, and some
  // lane needs every instruction as a rule)
  dv = __fma_rn(d2, v2, __fma_rn(d1, v1, d0 * v0));
  const double dd = __fma_rn(d2, d2, __fma_rn(d1, d1, d0 * d0));
  double rad = R2 - __fma_rn(-dv, dv, dd);
  const bool hit = tether || (neg(dv) && posv(rad) && !(skip_overlap && dbits(dd) < dbits(R2)));
  if (tether && neg(rad)) rad = 0.0;
  const double q = sqrt_rn(hit ? rad : 1.0);
  const double x = -dv + (tether ? q : flip(q));
  return hit ? (neg(x) ? 0.0 : x) : -1.0;
}

template <int G>
__device__ __forceinline__ float group_minf(float v) {
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, off));
  return v;
}

// FP32 minimum image (serial mode only; tile-local shadows need none)
__device__ __forceinline__ float wrapf(float d, float L) {
  return d > 0.5f * L ? d - L : (d < -0.5f * L ? d + L : d);
}

// ---------------------------------------------------------------- staging
// Shared memory of one group: FP32 shadow (tile-local) and id of every
// staged bead (16 B, one load); FP64 positions of the first M64 slots (M64 =
// 0: they are read from the global array, where every move is written
// through); bond-partner words of the first MNB slots (the motile beads);
// the slab masks; a header.
//
// Slab masks.  Every axis of the tile's box is cut into nsl slabs; row k + 1
// of an axis is the set of obstacle slots in slabs <= k (row 0 is empty), so
// the obstacles in slabs [a, b] are row[b + 1] & ~row[a], and those in a box
// the AND over the axes: six loads give the beads a path can reach, where a
// grid of cells has to visit, count and gather up to 27 of them.  Slot s is
// bit (s / G) of lane s % G: a lane reads and keeps current its own words and
// no others, so the masks need no synchronisation.
constexpr int LIST_CAP = 32;
constexpr int HDR_BYTES = 32 + 4 * LIST_CAP;

// The accepted tile sizes count an overflow list of max(64, S / 4) slots per
// tile, rounded up to a multiple of 8 (staging_budget in ecmc_internal.h).
constexpr int OVF_CAP = 64;
__host__ __device__ __forceinline__ int ovf_cap_for(int S) {
  return S / 4 > OVF_CAP ? (S / 4 + 7) / 8 * 8 : OVF_CAP;
}

struct Stage {
  float4 *sh;       // [S] x, y, z, id (bits)
  double *pos;      // [3][M64]
  uint2 *nb;        // [MNB] x: bond partner slots, 16 + 16 bits (0xFFFF = none);
                    // y: slabs of the stored shadow, 10 bits per axis
  unsigned *mask;   // [3][nsl + 1][W][G]
  int *lst;         // [LIST_CAP] candidates dealt to the lanes
  int *hdr;         // [0] staged beads (springs: with the far partners)
#ifdef ECMC_CHECKED
  int cap;          // S (slots)
  long long nglob;  // beads of the system (ids), set by the kernel
  int *status;
#endif
};

// 16-byte units of a group's slab masks (G is a multiple of 4)
__host__ __device__ __forceinline__ int mask_quads(int S, int G, int nsl) {
  const int W = (S + 32 * G - 1) / (32 * G);
  return 3 * (nsl + 1) * W * (G / 4);
}

// S, M64 and MNB are multiples of 8 and the masks whole 16-byte units, so
// every array starts 16-byte aligned and group_bytes is a multiple of 16
__host__ __device__ __forceinline__ size_t group_bytes(int S, int M64, int MNB, int MQ) {
  return (size_t)S * 16 + (size_t)M64 * 24 + (size_t)MNB * 8 + (size_t)MQ * 16 + HDR_BYTES;
}

__device__ __forceinline__ Stage carve(unsigned char *base, int S, int M64, int MNB, int MQ) {
  Stage s;
  s.sh = (float4 *)base;
  s.pos = (double *)(s.sh + S);
  s.nb = (uint2 *)(s.pos + 3 * M64);
  s.mask = (unsigned *)(s.nb + MNB);
  s.hdr = (int *)(s.mask + 4 * MQ);
  s.lst = s.hdr + 8;
#ifdef ECMC_CHECKED
  s.cap = S;
  s.nglob = 0x7fffffffffffffffll;
  s.status = nullptr;
#endif
  return s;
}

__device__ __forceinline__ int nb_prev(unsigned w) { return (w & 0xFFFF) == 0xFFFF ? -1 : (int)(w & 0xFFFF); }
__device__ __forceinline__ int nb_next(unsigned w) { return (w >> 16) == 0xFFFF ? -1 : (int)(w >> 16); }
__device__ __forceinline__ unsigned nb_pack(int prev, int next) {
  return ((unsigned)(next < 0 ? 0xFFFF : next) << 16) | (unsigned)(prev < 0 ? 0xFFFF : prev);
}

// binary search of id in the sorted range [lo, hi); -1 if absent
__device__ __forceinline__ int find_id(const int *ids, int lo, int hi, int id) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    const int v = ids[mid];
    if (v == id) return mid;
    if (v < id) lo = mid + 1;
    else hi = mid;
  }
  return -1;
}

__device__ __forceinline__ void set_status(int *st, int code) { atomicCAS(st, 0, code); }

// Bounds checks of the checked build (-DECMC_CHECKED): CHK(i, n, site, st)
// is true when 0 <= i < n; otherwise it records DEV_BOUNDS | site << 8 in
// the status word st (first failure wins) and is false, and the caller
// skips the access.  CI(i, ...) is i, or 0 after a failed check; it
// evaluates i once (the index can be an atomic's result).  In the normal
// build CHK is the constant true and CI the index itself.
#ifdef ECMC_CHECKED
__device__ __forceinline__ bool chk_range(long long i, long long n, int site, int *st) {
  if (i >= 0 && i < n) return true;
  atomicCAS(st, 0, DEV_BOUNDS | (site << 8));
  return false;
}
template <class T>
__device__ __forceinline__ T chk_index(T i, long long n, int site, int *st) {
  return chk_range((long long)i, n, site, st) ? i : T(0);
}
#define CHK(i, n, site, st) chk_range((long long)(i), (long long)(n), (site), (st))
#define CI(i, n, site, st) chk_index((i), (long long)(n), (site), (st))
#else
#define CHK(i, n, site, st) true
#define CI(i, n, site, st) (i)
#endif

// ---------------------------------------------------------------- slabs
// Slab of a tile-local coordinate: rint(f inv) - base, clamped to the nsl
// slabs (domain) or taken modulo nsl (serial, the slabs go around the box).
// Both steps are monotone in f, so a bead between two coordinates lies in a
// slab between theirs.  The rounding is the one of adding 1.5 2^23.
struct Slabs {
  float inv0, inv1, inv2;
  int base;  // magic bits + rint(origin inv)
  int nsl;
};
constexpr float SLAB_MAGIC = 12582912.f;
__device__ __forceinline__ int slab_raw(float f, float inv, int base) {
  return __float_as_int(__fmaf_rn(f, inv, SLAB_MAGIC)) - base;
}
template <bool DOM>
__device__ __forceinline__ int slab_of(float f, float inv, int base, int nsl) {
  const int k = slab_raw(f, inv, base);
  if (DOM) return min(max(k, 0), nsl - 1);
  return k < 0 ? k + nsl : (k >= nsl ? k - nsl : k);
}

// FP32 screen of one hard-sphere obstacle k for the pivot shadow pf moving
// along vf: updates the upper bound ubl and keeps the slot when its lower
// bound can reach it (two kept per lane, more -> ovf)
struct Screen {
  float sig2f, eps_v, eps_d;
};

__device__ __forceinline__ void screen_hs(const Screen &Z, float d0, float d1, float d2, float vf0,
                                          float vf1, float vf2, int k, float &ubl, int &ks0,
                                          float &kl0, int &ks1, float &kl1, bool &ovf) {
  const float dd = __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, d0 * d0));
  const float dv = __fmaf_rn(d2, vf2, __fmaf_rn(d1, vf1, d0 * vf0));
  const float disc = Z.sig2f - (dd - dv * dv);
  if (!(dv < Z.eps_v && disc > -Z.eps_d)) return;
  // bounds on sqrt(disc +- eps_d) from one reciprocal square root: with
  // dm = max(disc, eps_d) and s = sqrt(dm), sqrt(dm + eps_d) <= s + eps_d / (2 s)
  // and, for disc > eps_d, sqrt(disc - eps_d) >= s - eps_d / s
  const float dm = fmaxf(disc, Z.eps_d);
  const float rs = rsqrtf(dm);
  const float q = dm * rs, t = Z.eps_d * rs;
  const float lb = -dv - Z.eps_v - (q + 0.5f * t) * 1.000001f;
  if (lb > ubl) return;
  if (dv < -Z.eps_v && disc > Z.eps_d)
    ubl = fminf(ubl, fmaxf(0.f, -dv + Z.eps_v - (q - t) * 0.999999f) + 1e-6f);
  const float INF = __int_as_float(0x7f800000);
  if (kl0 > ubl) {
    ks0 = -1;
    kl0 = INF;
  }
  if (kl1 > ubl) {
    ks1 = -1;
    kl1 = INF;
  }
  if (ks0 < 0) {
    ks0 = k;
    kl0 = lb;
  } else if (ks1 < 0) {
    ks1 = k;
    kl1 = lb;
  } else {
    ovf = true;
  }
}

__device__ __forceinline__ float screen_lb(const Screen &Z, float d0, float d1, float d2,
                                           float vf0, float vf1, float vf2, bool &possible) {
  const float dd = __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, d0 * d0));
  const float dv = __fmaf_rn(d2, vf2, __fmaf_rn(d1, vf1, d0 * vf0));
  const float disc = Z.sig2f - (dd - dv * dv);
  possible = dv < Z.eps_v && disc > -Z.eps_d;
  const float dm = fmaxf(disc, Z.eps_d), rs = rsqrtf(dm);
  return -dv - Z.eps_v - (dm * rs + 0.5f * (Z.eps_d * rs)) * 1.000001f;
}

// FP64 position of staged slot k (bead id) on one axis: shared memory for
// the first M64 slots, otherwise the global position array (a joint bead,
// static this sweep, or a motile one, written through by every move)
__device__ __forceinline__ double pos64(const Stage &st, const double *r, int k, int id, int axis, int M64) {
#ifdef ECMC_CHECKED
  if (st.status && !CHK(k, st.cap, 1, st.status)) return 0.0;
  if (k >= M64 && st.status && !CHK(id, st.nglob, 2, st.status)) return 0.0;
#endif
  return k < M64 ? st.pos[axis * M64 + k] : r[3 * (int64_t)id + axis];
}

// ---------------------------------------------------------------- staging
// Stage one tile (domain) or the whole system (serial) into the group's
// shared memory: the lanes in `mask` call this together (one group of G
// lanes, or all groups of a warp that take a tile at the same time).
// Returns the motile count m, the hard-sphere joint count j1 and the staged
// count ns; clears `live` when the tile does not fit its capacity.
#define SYS(f) (BATCH ? rp->f : P.f)
template <int G, bool DOM, bool SPRING, bool BATCH>
__device__ __forceinline__ void stage_tile(const ECParams &P, const RepParams *rp, const Stage &st,
                                           int gl, bool &live, int unit, double ca, double *Rr, const int32_t *Rstart, int S,
                                           int M64, int MNB, int W, const Slabs &SL, int &m,
                                           int &j1, int &ns, unsigned mask, bool *overflow) {
  // a tile that does not fit its capacities sets the device status, or, when
  // the caller passes `overflow`, only that flag (the caller stages the tile
  // again later with larger capacities)
  auto capacity = [&]() {
    if (overflow) *overflow = true;
    else if (gl == 0) set_status(P.status, DEV_CAPACITY);
  };
  if (overflow) *overflow = false;
  const int nsl = SL.nsl;
  m = 0;
  j1 = 0;
  ns = 0;
  if (!DOM) {
    // serial: every bead, slot = id, all motile
    const int n = (int)P.n;
    for (int b = gl; b < n; b += G) {
      const double x = Rr[3 * (int64_t)b], y = Rr[3 * (int64_t)b + 1], z = Rr[3 * (int64_t)b + 2];
      if (b < M64) {
        st.pos[b] = x;
        st.pos[M64 + b] = y;
        st.pos[2 * M64 + b] = z;
      }
      st.sh[b] = make_float4(f32_trunc(x), f32_trunc(y), f32_trunc(z), __int_as_float(b));
      const int c = b % SYS(N);
      st.nb[b].x = nb_pack(c == 0 ? -1 : b - 1, c == SYS(N) - 1 ? -1 : b + 1);
    }
    m = n;
    j1 = 0;
    ns = n;
  } else {
    // cell window covering the tether halo of the tile: lane a works out
    // axis a (corner ca) and the group shares it
    int c_lo[3], c_n[3];
    float cf[3];
    {
      const int ax = (gl & 3) < 3 ? (gl & 3) : 0;
      const double lo = ca - P.halo_te, hi = ca + SYS(W)[ax] + P.halo_te;
      int l = (int)floor(div_rn(lo, SYS(cs)[ax]));
      const int h = (int)floor(div_rn(hi, SYS(cs)[ax]));
      int cnt = h - l + 1;
      if (cnt >= SYS(nc)[ax]) {
        l = 0;
        cnt = SYS(nc)[ax];
      }
      const float cfa = f32_trunc(ca);
      const int first = (threadIdx.x & 31) & ~(G - 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        c_lo[a] = __shfl_sync(mask, l, first + a);
        c_n[a] = __shfl_sync(mask, cnt, first + a);
        cf[a] = __shfl_sync(mask, cfa, first + a);
      }
    }
    // halo membership in FP32 from FP32 copies of the positions, widened by
    // 1e-3 sigma plus four FP32 ulps of the box: a superset of the exact
    // sets (an extra obstacle beyond reach is never hit; a bond partner is
    // always within the tether halo)
    float Lf[3], Lhf[3], Wf[3];
    float Lmax = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Lf[a] = SYS(Lf)[a];
      Lhf[a] = 0.5f * Lf[a];
      Wf[a] = SYS(Wf)[a];
      Lmax = fmaxf(Lmax, Lf[a]);
    }
    const float widen = 1e-3f * P.sigma_f + 4.8e-7f * Lmax;
    const float hs_f = P.halo_hs_f + widen, te_f = P.halo_te_f + widen;
    const int nc0 = SYS(nc)[0], nc1 = SYS(nc)[1], nc2 = SYS(nc)[2];
    const int nrows = c_n[1] * c_n[2];
    int cx = c_lo[0] % nc0;
    if (cx < 0) cx += nc0;
    const int len0 = c_n[0] < nc0 - cx ? c_n[0] : nc0 - cx;
    const unsigned below = (1u << gl) - 1u;
    const int g0 = (threadIdx.x & 31) & ~(G - 1);
    auto votes = [&](bool v) {
      const unsigned b = __ballot_sync(mask, v) >> g0;
      return G == 32 ? b : b & ((1u << (G & 31)) - 1u);
    };
    // pass 1: collect (cell-order index, flag | category | id), motile beads
    // from the front, joint beads from the back; the shadow array serves as
    // scratch until pass 3.  Obstacles are the joint beads of the hard-sphere
    // halo; beyond it, in the tether halo, only the bonded beads of motile
    // ones are wanted, and the tag of a joint bead tells whose tile those are
    // in (-1: of several, -2 - k: of tile k, else none).  The cells of one row
    // of the window (consecutive x) are one contiguous range of the
    // cell-ordered arrays (two when the row wraps around the box); each lane
    // takes whole rows and loads four beads at a time; votes give the places.
    int2 *scr = (int2 *)st.sh;
    int nj = 0;
    for (int r0 = 0; r0 < nrows; r0 += G) {
      const int r = r0 + gl;
      int a0 = 0, a1 = 0, n0 = 0, nt = 0;
      if (r < nrows) {
        const int qy = r % c_n[1], qz = r / c_n[1];
        int cy = (c_lo[1] + qy) % nc1;
        int cz = (c_lo[2] + qz) % nc2;
        if (cy < 0) cy += nc1;
        if (cz < 0) cz += nc2;
        const int base = (cz * nc1 + cy) * nc0;
        a0 = Rstart[base + cx];
        n0 = Rstart[base + cx + len0] - a0;
        nt = n0;
        if (len0 < c_n[0]) {
          a1 = Rstart[base];
          nt += Rstart[base + c_n[0] - len0] - a1;
        }
      }
      int most = nt;
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) most = max(most, __shfl_xor_sync(mask, most, off));
      for (int k0 = 0; k0 < most; k0 += 4) {
        int tg[4], jj[4], idv[4];
        float px[4], py[4], pz[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = k0 + u;
          jj[u] = k < n0 ? a0 + k : a1 + (k - n0);
          tg[u] = INT_MAX;
          idv[u] = 0;
          px[u] = py[u] = pz[u] = 0.f;
          if (k < nt) {
            const int64_t j = jj[u];
            tg[u] = P.ctag[j];
            idv[u] = P.cid[j];
            px[u] = P.crf[3 * j];
            py[u] = P.crf[3 * j + 1];
            pz[u] = P.crf[3 * j + 2];
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          int cat = tg[u] == unit ? 0 : -1;
          const bool bonded = tg[u] == -1 || tg[u] == -2 - unit;
          if (tg[u] < 0) {
            const float pp[3] = {px[u], py[u], pz[u]};
            bool in_hs = true, in_te = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              float sa = pp[a] - cf[a];
              sa = sa > Lhf[a] ? sa - Lf[a] : (sa < -Lhf[a] ? sa + Lf[a] : sa);
              in_hs = in_hs && (sa >= -hs_f) && (sa <= Wf[a] + hs_f);
              in_te = in_te && (sa >= -te_f) && (sa <= Wf[a] + te_f);
            }
            cat = in_hs ? 1 : (in_te && bonded ? 2 : -1);
          }
          const unsigned bm = votes(cat == 0), bj = votes(cat > 0);
          const int q = cat == 0 ? m + __popc(bm & below) : nj + __popc(bj & below);
          if (cat >= 0 && q < S)
            scr[cat == 0 ? q : S - 1 - q] =
                make_int2(jj[u], (int)((bonded && cat > 0 ? 0x80000000u : 0u) | ((unsigned)cat << 29) | (unsigned)idv[u]));
          m += __popc(bm);
          nj += __popc(bj);
          j1 += __popc(votes(cat == 1));
        }
      }
    }
    __syncwarp(mask);
    ns = m + nj;
    // (a list that ran into the other one holds no valid entries)
    if (ns > S || m > MNB) {
      capacity();
      live = false;
      m = j1 = ns = nj = 0;
    }
    // pass 2: slots.  Motile beads take their rank by id (the start bead of
    // an EC is the u-th motile bead in id order); joint beads take the next
    // free slot of their category (their order matters to nothing).  The ids
    // go to the mask area (nsl >= 10 makes it as large as S words), those of
    // joint beads with the flag of a bonded one.
    int *idt = (int *)st.mask;
    for (int s = gl; s < m; s += G) {
      const int id = scr[s].y;
      int rank = 0;
      for (int t = 0; t < m; ++t) rank += (scr[t].y < id);
      if (CHK(rank, S, 3, P.status)) idt[rank] = id;
    }
    {
      int n1 = 0, n2 = 0;
      for (int s0 = 0; s0 < nj; s0 += G) {
        const int s = s0 + gl;
        const unsigned e = s < nj ? (unsigned)scr[S - 1 - s].y : 0u;
        const int cat = (int)(e >> 29) & 3;
        const unsigned b1 = votes(cat == 1), b2 = votes(cat == 2);
        const int slot = cat == 1 ? m + n1 + __popc(b1 & below) : m + j1 + n2 + __popc(b2 & below);
        if (cat != 0 && CHK(slot, S, 33, P.status)) idt[slot] = (int)(e & 0x9FFFFFFFu);
        n1 += __popc(b1);
        n2 += __popc(b2);
      }
    }
    __syncwarp(mask);
    // pass 2b: bond partners among the motile beads (sorted, so id - 1 can
    // only be the slot before)
    const int Nc = SYS(N);
    for (int s = gl; s < m; s += G) {
      const int id = idt[s], c = id % Nc;
      const int prev = c != 0 && s > 0 && idt[s - 1] == id - 1 ? s - 1 : -1;
      const int next = c != Nc - 1 && s + 1 < m && idt[s + 1] == id + 1 ? s + 1 : -1;
      st.nb[s].x = nb_pack(prev, next);
    }
    __syncwarp(mask);
    // pass 3: shadows (FP32 position minus FP32 corner, the form the moved
    // pivot's shadow takes too), FP64 positions, and a bonded joint bead
    // announces itself to its motile neighbours.  Four slots at a time
    // (independent loads).
    const float *const Rf = P.rf + (BATCH ? 3 * rp->bead_off : 0);
    const int32_t *const Rtag = P.tag + (BATCH ? rp->bead_off : 0);
    unsigned short *const nbh = (unsigned short *)st.nb;
    auto fill = [&](int from, int to) {
      for (int s0 = from; s0 < to; s0 += 4 * G) {
        float x[4], y[4], z[4];
        int idv[4], up[4], dn[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int s = s0 + u * G + gl;
          idv[u] = 0;
          up[u] = dn[u] = -1;
          if (s < to) {
            const int e = idt[s];
            const int64_t b = CI(e & 0x7FFFFFFF, BATCH ? rp->n_beads : P.n, 5, P.status);
            idv[u] = (int)b;
            x[u] = Rf[3 * b];
            y[u] = Rf[3 * b + 1];
            z[u] = Rf[3 * b + 2];
            if (e < 0) {
              const int c = (int)b % Nc;
              if (c != Nc - 1) up[u] = Rtag[b + 1];
              if (c != 0) dn[u] = Rtag[b - 1];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int s = s0 + u * G + gl;
          if (s >= to) continue;
          float f0 = x[u] - cf[0], f1 = y[u] - cf[1], f2 = z[u] - cf[2];
          f0 = f0 > Lhf[0] ? f0 - Lf[0] : (f0 < -Lhf[0] ? f0 + Lf[0] : f0);
          f1 = f1 > Lhf[1] ? f1 - Lf[1] : (f1 < -Lhf[1] ? f1 + Lf[1] : f1);
          f2 = f2 > Lhf[2] ? f2 - Lf[2] : (f2 < -Lhf[2] ? f2 + Lf[2] : f2);
          st.sh[s] = make_float4(f0, f1, f2, __int_as_float(idv[u]));
          if (up[u] == unit) {
            const int t = find_id(idt, 0, m, idv[u] + 1);
            if (t >= 0) nbh[4 * t] = (unsigned short)s;
          }
          if (dn[u] == unit) {
            const int t = find_id(idt, 0, m, idv[u] - 1);
            if (t >= 0) nbh[4 * t + 1] = (unsigned short)s;
          }
        }
      }
#pragma unroll 3
      for (int s = from + gl; s < to && s < M64; s += G) {
        const double *const x = Rr + 3 * (int64_t)CI(idt[s] & 0x7FFFFFFF, BATCH ? rp->n_beads : P.n, 6, P.status);
        const double X = x[0], Y = x[1], Z = x[2];
        st.pos[s] = X;
        st.pos[M64 + s] = Y;
        st.pos[2 * M64 + s] = Z;
      }
    };
    fill(0, ns);
    if (gl == 0) st.hdr[0] = ns;
    __syncwarp(mask);
    for (int s = gl; s < m; s += G) {
      const int id = idt[s], c = id % Nc;
#pragma unroll
      for (int dir = 0; dir < 2; ++dir) {
        if (nbh[4 * s + dir] != 0xFFFF) continue;
        const int q = dir == 0 ? (c != 0 ? id - 1 : -1) : (c != Nc - 1 ? id + 1 : -1);
        if (q < 0) continue;
        if (!SPRING) {
          set_status(P.status, DEV_TILE);
          continue;
        }
        // a spring has no longest bond, so the bonded beads of motile beads
        // are staged wherever they are; one outside the tether halo (a joint
        // bead, static this sweep) is appended after the staged beads (two
        // motile beads may append the same bead twice; both copies are
        // read-only and equal)
        if (!CHK(q, BATCH ? rp->n_beads : P.n, 4, P.status)) continue;
        const int slot = atomicAdd(&st.hdr[0], 1);
        if (slot < S) {
          idt[slot] = q;
          nbh[4 * s + dir] = (unsigned short)slot;
        }
      }
    }
    if (SPRING) {
      __syncwarp(mask);
      const int all = st.hdr[0];
      if (all > S) {
        if (live) capacity();
        live = false;
        m = j1 = ns = 0;
      } else {
        fill(ns, all);
        ns = all;
      }
    }
  }
  __syncwarp(mask);
  // pass 4: the slab masks of the obstacle slots; every lane builds its own
  // words: the beads of each slab, then the running union
  const int nhs = m + j1;
  const int row = W * G;
  for (int i = 0; i < 3 * (nsl + 1) * W; ++i) st.mask[i * G + gl] = 0u;
  for (int s = gl; s < nhs; s += G) {
    const float4 f = st.sh[s];
    const int b = s / G;
    unsigned *const w = st.mask + (b >> 5) * G + gl;
    const unsigned bit = 1u << (b & 31);
    const int k0 = slab_of<DOM>(f.x, SL.inv0, SL.base, nsl), k1 = slab_of<DOM>(f.y, SL.inv1, SL.base, nsl),
              k2 = slab_of<DOM>(f.z, SL.inv2, SL.base, nsl);
    if (s < m) st.nb[s].y = (unsigned)(k0 | (k1 << 10) | (k2 << 20));
    w[(k0 + 1) * row] |= bit;
    w[(nsl + 1 + k1 + 1) * row] |= bit;
    w[(2 * (nsl + 1) + k2 + 1) * row] |= bit;
  }
  for (int w = 0; w < W; ++w) {
    unsigned *const q = st.mask + w * G + gl;
    unsigned acc0 = 0u, acc1 = 0u, acc2 = 0u;
#pragma unroll 4
    for (int k = 1; k <= nsl; ++k) {
      unsigned *const p = q + k * row;
      const unsigned x = p[0], y = p[(nsl + 1) * row], z = p[2 * (nsl + 1) * row];
      p[0] = acc0 |= x;
      p[(nsl + 1) * row] = acc1 |= y;
      p[2 * (nsl + 1) * row] = acc2 |= z;
    }
  }
  __syncwarp(mask);
  if (!live) m = 0;
}
#undef SYS

// The obstacle in slot k went from slabs (o0, o1, o2) to (n0, n1, n2): its
// bit flips in the rows between (called by lane k % G alone)
__device__ __forceinline__ void slab_move(const Stage &st, int G, int W, int nsl, int k, int o0, int o1,
                                          int o2, int n0, int n1, int n2) {
  const int gl = k % G, b = k / G, row = W * G;
  const unsigned bit = 1u << (b & 31);
  unsigned *const w = st.mask + (b >> 5) * G + gl + row;
  for (int i = min(o0, n0); i < max(o0, n0); ++i) w[i * row] ^= bit;
  for (int i = min(o1, n1); i < max(o1, n1); ++i) w[(nsl + 1 + i) * row] ^= bit;
  for (int i = min(o2, n2); i < max(o2, n2); ++i) w[(2 * (nsl + 1) + i) * row] ^= bit;
}

}  // namespace
}  // namespace ecmc
