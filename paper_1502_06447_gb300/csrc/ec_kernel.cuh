// Event-chain kernel (arXiv:1502.06447, Sec. II: EC move, with hard tethers
// or harmonic bead springs; Sec. II.A: tile-joint decomposition with
// reflections; Sec. II.B: push-off; Sec. II.C: swap move).  Included by the
// translation units that instantiate it.
//
// One group of G lanes (G = 32, 16, 8 or 4) runs the ECs of one tile, one
// event per step; the 32 / G groups of a warp step together, and no warp
// waits for another: there is no block barrier.  A group whose tile has run
// its ECs takes the next unit of the launch from a device counter and stages
// it while the warp's other groups wait.
//
// What bounds it: the latency of one step, a chain of dependent instructions
// (a warp issues one every 6.4 cycles, of which 2.4 are fixed latencies, 1.2
// shuffles and shared memory, 0.7 branches), with 12 warps per SM to hide it
// (registers; about 4.7 KB of shared memory per tile).  The dearest of them
// are FP64 instructions: GB300's FP64 unit takes a warp instruction every 64
// cycles per SM sub-partition whatever its active mask and dependences
// (conversions and comparisons 80-110).  Hence:
//   - the lanes of a quad hold one axis each (lane 3: what is left of ell),
//     and the three axes of a difference, a move or a reflection are one
//     instruction; d.v and d.d are one chain of three on two lanes; the move,
//     the rest of ell and the projection of a lift come from one multiply-add;
//   - square roots and quotients are integer code (ecmc_dev.cuh), as are
//     comparisons, sign changes and conversions to FP32.
// A step with one contact takes 9 FP64 instructions, a reflection 5 more.
//
// A step:
//   A  the obstacles the flight can reach come from the slab masks
//      (ec_device.cuh), each lane its own words.  In the screened form (F32)
//      a lane bounds its obstacles, a tether or a wall in FP32 and keeps
//      those whose lower bound can reach the group's smallest upper bound U;
//      in the plain form every reachable obstacle is kept;
//   B  what was kept is evaluated in FP64 (exactly the definition's
//      expressions), one candidate per quad in the screened form, one per
//      lane in the plain form; the group takes the smallest x under the tie
//      rule;
//   D  the lanes move the pivot, lift, reflect or swap.
// A candidate left out by the screen cannot win: the winner's exact x is <= U
// and every lower bound is <= its candidate's exact x, so both forms produce
// the same events.
//
// Measured (cycles per warp step): 9,700 with 48 tiles of 8 lanes per SM on
// 1e6 beads, 5,200 for a warp alone with one tile of 32 lanes; the kernel
// that exchanged requests between the tiles of a block over block barriers
// took 21,100 and some 14,000.  One sweep of 1e6 beads, eight ECs per tile
// of 4.2 sigma: 91 -> 41 ms; a serial run of 640 beads in FP64, 400 ECs: 529
// -> 58 ms (2.4 us per event); 64 replicas, four sweeps: 475 -> 181 ms.  A
// bound of 128 registers with half the mask bytes (64 tiles per SM) lengthens
// every step by as much as it adds tiles: 1e6 beads 1 % faster, 64 replicas
// 11 % and lone warps 4 % slower.
#pragma once
#include "ec_device.cuh"

namespace ecmc {

namespace {

// A group's candidates: x (bits), kind << 28 | slot, d.v before the flight and
// the partner's position on this lane's axis.  In a quad all lanes hold the
// same x, code and d.v.
struct Cand {
  uint64_t x;
  int code;
  double dv, pos;
};
constexpr int CAND_NONE = -1;

#define SYS(f) (BATCH ? rp->f : P.f)

// DOM: domain mode (else serial: one unit, the whole periodic box);
// SPRING: harmonic bonds; PO: push-off (start beads and overlap rule)
template <int G, bool F32, bool BATCH, bool DOM, bool SPRING, bool PO>
__global__ void __launch_bounds__(128, 3) ec_kernel(const ECParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  // push-off run from the device: nothing to do once no bead overlaps
  if (PO && P.po_count && *P.po_count == 0ull) return;
  const int lane = threadIdx.x & 31;
  const int gl = lane & (G - 1);
  const int gbase = lane & ~(G - 1);
  const int qbase = lane & ~3;
  const int ax = lane & 3;            // this lane's axis; 3: what is left of ell
  const int axc = ax < 3 ? ax : 0;
  constexpr int NQ = G / 4;           // quads of the group
  const int qd = gl >> 2;             // this lane's quad
  // the lane whose move instruction gives the projection of a lift, and
  // whose lift and reflection sums count
  constexpr int AL = G >= 8 ? 7 : 0;
  const unsigned gmask = (G == 32) ? FULL : (((1u << G) - 1) << gbase);
  const int gib = threadIdx.x / G;
  const int64_t sweep = P.sweep_dev ? *P.sweep_dev : P.sweep;
  const int S = P.stage_cap, MNB = P.m_cap, M64 = P.m64, nsl = P.nsl;
  const int W = (S + 32 * G - 1) / (32 * G);
  const int row = W * G;
  const int MQ = mask_quads(S, G, nsl);
  Stage st = carve(smem + (size_t)gib * group_bytes(S, M64, MNB, MQ), S, M64, MNB, MQ);
#ifdef ECMC_CHECKED
  st.status = P.status;
  st.nglob = P.n;
#endif

  // ------------------------------------------------------------ tile state
  enum : int { TILE_NEED = 0, EC_NEED = 1, EC_RUN = 2, TILE_DONE = 3 };
  int state = TILE_NEED;
  const RepParams *rp = BATCH ? P.reps : nullptr;
  int unit = 0, gunit = 0;
  int m = 0, j1 = 0;
  double *Rr = P.r;
  int32_t *Ri = P.img;
  uint64_t Rkey = P.replica;
  const Slabs SL{P.sinv[0], P.sinv[1], P.sinv[2], slab_raw(P.sorg, P.sinv[0], 0), nsl};
  // this lane's axis: tile corner (FP64, FP32), tile side, whether positions
  // of the tile can wrap (a tile whose halo lies inside (0, L) on an axis
  // never needs the minimum image or a wrap there)
  double ca = 0.0;
  float cfa = 0.f, Wfa = 0.f;
  bool wra = !DOM && ax < 3;
  int n_ec = P.ecs_per_tile;

  // ------------------------------------------------------------ EC state
  int e = 0, p = 0, pid = 0;
  unsigned nbw = 0xFFFFFFFFu;
  int oslab = 0;  // slabs of the pivot's stored shadow, 10 bits per axis
  double qa = 0.0;             // pivot position on this lane's axis; lane 3: what is left of ell
  double va = 0.0;             // direction on this lane's axis; lane 3: -1
  double v0 = 0.0, v1 = 0.0, v2 = 0.0, xrem = 0.0;  // the same, on every lane
  double lift = 0.0, refl_all = 0.0;                // (lane AL)
  float pf0 = 0.f, pf1 = 0.f, pf2 = 0.f, vf0 = 0.f, vf1 = 0.f, vf2 = 0.f;
  float rb0 = 0.f, rb1 = 0.f, rb2 = 0.f;  // per-axis reach of a contact against the direction
  unsigned nev = 0;
  unsigned pmask = ~0u;  // this lane's first mask word without the pivot
  unsigned ncontact = 0, swgo = 0;  // swap proposals of this and the next contacts, one bit each
  uint64_t h = 0;
  // springs: 2 dE / k of the next G / 2 events, drawn together
  double dEk = 0.0;
  int dE_at = 0;

  double lift_all = 0.0;
  unsigned long long nev_all = 0;
  unsigned tried = 0, confirmed = 0, ecs_done = 0, exh = 0;
  // events by outcome: lane k of a group (of 4 lanes: lane k % 4, two counts)
  // counts outcome k
  unsigned ev_lo = 0, ev_hi = 0;
  const unsigned event_cap = P.event_cap < 0xFFFFFFFFll ? (unsigned)P.event_cap : 0xFFFFFFFFu;

  Screen Z;
  Z.sig2f = P.sig2_f;
  Z.eps_v = P.eps_v;
  Z.eps_d = P.eps_d;
  const float eps_v = P.eps_v, eps_d = P.eps_d;
  const float reach_hs = P.sigma_f + 2.f * eps_v;  // per-axis reach of a contact
  // A contact partner lies ahead, within the half sphere of radius sigma
  // around v from the path: against the direction of v_a it reaches no more
  // than sigma sqrt(1 - v_a^2).  The box of a flight holds a third fewer
  // obstacles than one with sigma on both sides.
  auto reach_back = [&](float v) { return P.sigma_f * sqrt_hi(fmaxf(1.f - v * v, 0.f) + 1e-6f) + 2.f * eps_v; };
  auto new_direction = [&]() {
    vf0 = f32_trunc(v0);
    vf1 = f32_trunc(v1);
    vf2 = f32_trunc(v2);
    rb0 = reach_back(vf0);
    rb1 = reach_back(vf1);
    rb2 = reach_back(vf2);
  };
  const float INF = __int_as_float(0x7f800000);
  const uint64_t r1 = DOM ? (uint64_t)sweep : 0;

  auto slabs_at = [&](float f0, float f1, float f2) {
    return slab_of<DOM>(f0, SL.inv0, SL.base, nsl) | (slab_of<DOM>(f1, SL.inv1, SL.base, nsl) << 10) |
           (slab_of<DOM>(f2, SL.inv2, SL.base, nsl) << 20);
  };
  // minimum image on this lane's axis (identity where it cannot be needed)
  auto wrap_a = [&](double d, bool on) {
    return wrap_bits(d, SYS(L)[axc], SYS(half)[axc], on);
  };
  // the FP32 shadow of the position x on this lane's axis, for every lane:
  // FP32 position minus FP32 corner
  auto shadows = [&](double x, float &f0, float &f1, float &f2) {
    float f = f32_trunc(x) - cfa;
    if (DOM && wra) {
      const float Lf = SYS(Lf)[axc], Lh = 0.5f * Lf;
      f = f > Lh ? f - Lf : (f < -Lh ? f + Lf : f);
    }
    f0 = __shfl_sync(gmask, f, gbase);
    f1 = __shfl_sync(gmask, f, gbase + 1);
    f2 = __shfl_sync(gmask, f, gbase + 2);
  };
  // d.v and d.d of a separation whose components the quad's lanes hold
  // (lane 3's is not used): one chain of three FP64 instructions, d.v on the
  // quad's first lane, d.d on the others
  auto dots = [&](unsigned mask, double d, double &dv, double &dd) {
    const double d0 = __shfl_sync(mask, d, qbase), d1 = __shfl_sync(mask, d, qbase + 1),
                 d2 = __shfl_sync(mask, d, qbase + 2);
    const bool first = ax == 0;
    double s = d0 * (first ? v0 : d0);
    s = __fma_rn(d1, (first ? v1 : d1), s);
    s = __fma_rn(d2, (first ? v2 : d2), s);
    dv = __shfl_sync(mask, s, qbase);
    dd = __shfl_sync(mask, s, qbase + 1);
  };
  // The bead in slot k sits at x (this lane's axis) now: FP64 position
  // (write-through), shadow and slab masks.  A pivot never screens itself, so
  // its copies are brought up to date only when it stops being the pivot.
  auto settle = [&](int k, int id, double x, float f0, float f1, float f2, int os) {
    if (gl < 3) {
      Rr[3 * (int64_t)id + gl] = x;
      if (k < M64) st.pos[gl * M64 + k] = x;
    }
    if (gl == (k & (G - 1))) {
      st.sh[k] = make_float4(f0, f1, f2, __int_as_float(id));
      const int nw = slabs_at(f0, f1, f2);
      if (nw != os) {
        st.nb[k].y = (unsigned)nw;
        slab_move(st, G, W, nsl, k, os & 1023, (os >> 10) & 1023, os >> 20, nw & 1023,
                  (nw >> 10) & 1023, nw >> 20);
      }
    }
  };

  // take the next unit and stage it (group-collective); false when none left
  auto take_tile = [&]() -> bool {
    int u = 0;
    if (gl == 0) {
      u = atomicAdd(P.unit_next, 1);
      if (P.defer_mode == 2) u = u < *P.n_deferred ? P.deferred[u] : P.n_units;
    }
    u = __shfl_sync(gmask, u, gbase);
    if (u >= P.n_units) return false;
    gunit = u;
    unit = u;
    if (BATCH) {
      int lo = 0, hi = P.n_reps - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.reps[mid].unit_off <= u) lo = mid;
        else hi = mid - 1;
      }
      rp = P.reps + lo;
      unit = u - (int)rp->unit_off;
      Rr = P.r + 3 * rp->bead_off;
      Ri = P.img + 3 * rp->bead_off;
      Rkey = rp->replica;
#ifdef ECMC_CHECKED
      st.nglob = rp->n_beads;
#endif
    }
    const int32_t *const Rstart = BATCH ? P.cstart + rp->cell_off : P.cstart;
    if (DOM) {
      const int D0 = SYS(D)[0], D1 = SYS(D)[1];
      const int tk = ax == 0 ? unit % D0 : (ax == 1 ? (unit / D0) % D1 : unit / (D0 * D1));
      const u64x4 w = philox(TAG_SHIFT, (uint64_t)sweep, 0, 0, P.seed, Rkey);
      const double T = SYS(T)[axc], L = SYS(L)[axc];
      ca = unit53(ax == 0 ? w.v[0] : (ax == 1 ? w.v[1] : w.v[2])) * T + (double)tk * T;
      cfa = f32_trunc(ca);
      Wfa = SYS(Wf)[axc];
      wra = ax < 3 && !(ca - P.halo_te > 0.0 && ca + SYS(W)[axc] + P.halo_te < L);
    }
    bool live = true, over = false;
    int ns = 0;
    stage_tile<G, DOM, SPRING, BATCH>(P, rp, st, gl, live, unit, ca, Rr, Rstart, S, M64, MNB, W, SL, m,
                                      j1, ns, gmask, P.defer_mode == 1 ? &over : nullptr);
    if (over && gl == 0) {
      const int at = atomicAdd(P.n_deferred, 1);
      P.deferred[CI(at, P.n_units, 32, P.status)] = gunit;
    }
    if (PO) {
      // push-off: one EC from every flagged motile bead, in id order
      int f = 0;
      for (int s = gl; s < m; s += G) f += P.po_flag[__float_as_int(st.sh[s].w)] ? 1 : 0;
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) f += __shfl_xor_sync(gmask, f, off);
      n_ec = f;
    }
    e = 0;
    return true;
  };

  // start EC e of the tile: start bead and direction (Sec. II, R6)
  auto start_ec = [&]() {
    const uint64_t r0 = DOM ? (TAG_START | ((uint64_t)e << 8)) : TAG_START;
    const uint64_t r2 = DOM ? (uint64_t)unit : (uint64_t)(sweep + e);
    u64x4 w = philox(r0, r1, r2, 0, P.seed, Rkey);
    p = (int)scale_below(w.v[0], (uint64_t)m);
    if (PO) {
      // the e-th flagged motile slot (slots are in id order)
      int before = 0;
      for (int s0 = 0; s0 < m; s0 += G) {
        const int s = s0 + gl;
        const bool f = s < m && P.po_flag[__float_as_int(st.sh[s].w)];
        unsigned bal = (__ballot_sync(gmask, f) & gmask) >> gbase;
        const int c = __popc(bal);
        if (e < before + c) {
          for (int i = before; i < e; ++i) bal &= bal - 1;
          p = s0 + __ffs(bal) - 1;
          break;
        }
        before += c;
      }
    }
    if (P.dir_mode == ECMC_DIR_CART3) {
      va = ax == (int)scale_below(w.v[1], 3) ? 1.0 : 0.0;
    } else {
      // one component per lane
      double t = 2.0 * unit53(ax == 0 ? w.v[1] : (ax == 1 ? w.v[2] : w.v[3])) - 1.0;
      uint64_t att = 0;
      for (;;) {
        const double t2 = t * t;
        const double s = __shfl_sync(gmask, t2, gbase) + __shfl_sync(gmask, t2, gbase + 1) +
                         __shfl_sync(gmask, t2, gbase + 2);
        // s > 1e-6 && s <= 1
        if (dbits(s) > dbits(1e-6) && dbits(s) <= dbits(1.0)) {
          va = div_rn(t, sqrt_rn(s));
          break;
        }
        ++att;
        w = philox(r0, r1, r2, att, P.seed, Rkey);
        t = 2.0 * unit53(ax == 0 ? w.v[0] : (ax == 1 ? w.v[1] : w.v[2])) - 1.0;
      }
    }
    v0 = __shfl_sync(gmask, va, gbase);
    v1 = __shfl_sync(gmask, va, gbase + 1);
    v2 = __shfl_sync(gmask, va, gbase + 2);
    p = CI(p, m, 10, P.status);
    const float4 f = st.sh[p];
    pid = CI(__float_as_int(f.w), BATCH ? rp->n_beads : P.n, 11, P.status);
    qa = pos64(st, Rr, p, pid, axc, M64);
    if (ax == 3) {
      qa = P.ell;
      va = -1.0;
    }
    xrem = P.ell;
    const uint2 nb = st.nb[p];
    nbw = nb.x;
    oslab = (int)nb.y;
    pmask = gl == (p & (G - 1)) && p / G < 32 ? ~(1u << ((p / G) & 31)) : ~0u;
    pf0 = f.x;
    pf1 = f.y;
    pf2 = f.z;
    new_direction();
    lift = 0.0;
    nev = 0;
    ncontact = 0;
    if (SPRING) dE_at = G / 2;  // draw at the first event
    h = 0xCBF29CE484222325ull;
  };

  // ------------------------------------------------------------ steps
  for (;;) {
    if (__any_sync(FULL, state != EC_RUN)) {
      if (state == TILE_NEED) {
        // (tiles without motile beads have no ECs and are passed over)
        for (;;) {
          if (!take_tile()) {
            state = TILE_DONE;
            break;
          }
          if (m > 0 && n_ec > 0) {
            state = EC_NEED;
            break;
          }
        }
      }
      if (state == EC_NEED) {
        start_ec();
        state = EC_RUN;
      }
      __syncwarp();
      if (!__any_sync(FULL, state == EC_RUN)) break;
    }
    const bool act = state == EC_RUN;

    // ---------------------------------------------------------- A: screen
    // what the flight ends with at the latest
    const bool pass = dbits(P.s_cap) < dbits(xrem);
    const float xc = act ? (pass ? P.s_cap_f : f32_above(xrem)) : 0.f;
    float ubl = xc;
    Cand best{~0ull, CAND_NONE, 0.0, 0.0};  // this lane's best evaluated candidate
    // (x, kind, partner id) order: an exact tie in x goes to the smaller kind,
    // then to the smaller id (wall: axis)
    auto beats = [&](uint64_t xb, int code) {
      if (xb != best.x || best.code == CAND_NONE) return xb < best.x;
      const int k0 = code >> 28, k1 = best.code >> 28;
      if (k0 != k1 || k0 == KIND_WALL) return code < best.code;
      return __float_as_int(st.sh[code & 0xFFFFFFF].w) < __float_as_int(st.sh[best.code & 0xFFFFFFF].w);
    };
    auto keep = [&](double x, int code, double dv, double pos) {
      if (beats(dbits(x), code)) best = Cand{dbits(x), code, dv, pos};
    };
    if (SPRING) {
      // energies for the next G / 2 events of every group's EC: lane
      // 2 i + j draws bond j of event nev + i, so that the draw and the
      // logarithm (some 50 FP64 instructions) are paid for once per G / 2
      // events.  All groups draw when one has used up its own.
      if (__any_sync(FULL, act && dE_at == G / 2)) {
        const uint64_t r2 = DOM ? (uint64_t)unit : (uint64_t)(sweep + e);
        const u64x4 w = philox(TAG_SPRING | ((uint64_t)(DOM ? e : 0) << 8), r1, r2,
                               (uint64_t)(nev + (gl >> 1)), P.seed, Rkey);
        dEk = div_rn(2.0 * spring_dE((gl & 1) ? w.v[1] : w.v[0]), P.k_spring);
        dE_at = 0;
      }
      // quad j evaluates bond j (0: to the previous bead, 1: to the next)
#pragma unroll
      for (int j0 = 0; j0 < 2; j0 += NQ) {
        const int j = j0 + qd;
        const int t = j >= 2 || !act ? -1 : (j == 0 ? nb_prev(nbw) : nb_next(nbw));
        const double bE = __shfl_sync(FULL, dEk, gbase + 2 * (dE_at & (G / 2 - 1)) + (j & 1));
        // (a spring partner may lie beyond the tile's halo, across the
        // periodic boundary: always the minimum image)
        double d = 0.0, dv, dd, pos = 0.0;
        if (t >= 0 && ax < 3) {
          pos = pos64(st, Rr, CI(t, S, 20, P.status), __float_as_int(st.sh[t].w), ax, M64);
          d = wrap_a(qa - pos, true);
        }
        dots(FULL, d, dv, dd);
        if (t >= 0) {
          const double x = spring_flight(dv, dd, P.sigma, bE);
          ubl = fminf(ubl, f32_above(x));
          if (F32 || ax == 0) keep(x, (KIND_TETHER << 28) | t, dv, pos);
        }
      }
      ++dE_at;
    }
    // the slabs of the box that holds every obstacle in reach of the path
    // [pf, pf + xc vf]
    const float e0 = xc * vf0, e1 = xc * vf1, e2 = xc * vf2;
    const unsigned *wa0, *wa1, *wa2, *wb0, *wb1, *wb2;
    bool fl0 = false, fl1 = false, fl2 = false;  // serial: the range goes around the box
    {
      const bool u0 = signbit(vf0), u1 = signbit(vf1), u2 = signbit(vf2);
      const float l0 = pf0 + (u0 ? e0 - reach_hs : -rb0), h0 = pf0 + (u0 ? rb0 : e0 + reach_hs);
      const float l1 = pf1 + (u1 ? e1 - reach_hs : -rb1), h1 = pf1 + (u1 ? rb1 : e1 + reach_hs);
      const float l2 = pf2 + (u2 ? e2 - reach_hs : -rb2), h2 = pf2 + (u2 ? rb2 : e2 + reach_hs);
      int a0 = slab_raw(l0, SL.inv0, SL.base), b0 = slab_raw(h0, SL.inv0, SL.base);
      int a1 = slab_raw(l1, SL.inv1, SL.base), b1 = slab_raw(h1, SL.inv1, SL.base);
      int a2 = slab_raw(l2, SL.inv2, SL.base), b2 = slab_raw(h2, SL.inv2, SL.base);
      if (DOM) {
        a0 = min(max(a0, 0), nsl - 1);
        b0 = min(max(b0, 0), nsl - 1);
        a1 = min(max(a1, 0), nsl - 1);
        b1 = min(max(b1, 0), nsl - 1);
        a2 = min(max(a2, 0), nsl - 1);
        b2 = min(max(b2, 0), nsl - 1);
      } else {
        // the range [a, b] of slabs around the box; nsl or more: all of them
        auto around = [&](int &a, int &b, bool &fl) {
          if (b - a >= nsl - 1) {
            a = 0;
            b = nsl - 1;
            return;
          }
          if (a < 0) a += nsl;
          else if (a >= nsl) a -= nsl;
          if (b < 0) b += nsl;
          else if (b >= nsl) b -= nsl;
          fl = a > b;
        };
        around(a0, b0, fl0);
        around(a1, b1, fl1);
        around(a2, b2, fl2);
      }
      const unsigned *const mk = st.mask + gl;
      wa0 = mk + a0 * row;
      wb0 = mk + (b0 + 1) * row;
      wa1 = mk + (nsl + 1 + a1) * row;
      wb1 = mk + (nsl + 2 + b1) * row;
      wa2 = mk + (2 * (nsl + 1) + a2) * row;
      wb2 = mk + (2 * (nsl + 1) + b2 + 1) * row;
    }
    // this lane's word w of the obstacles in the box, the pivot left out
    auto cand_word = [&](int w) -> unsigned {
      const int o = w * G;
      unsigned c;
      if (DOM) {
        c = (wb0[o] & ~wa0[o]) & (wb1[o] & ~wa1[o]) & (wb2[o] & ~wa2[o]);
      } else {
        const unsigned all = st.mask[gl + nsl * row + o];
        c = (fl0 ? wb0[o] | ~wa0[o] : wb0[o] & ~wa0[o]) & (fl1 ? wb1[o] | ~wa1[o] : wb1[o] & ~wa1[o]) &
            (fl2 ? wb2[o] | ~wa2[o] : wb2[o] & ~wa2[o]) & all;
      }
      if (w == 0) c &= pmask;
      else if (gl == (p & (G - 1)) && (p / G) >> 5 == w) c &= ~(1u << ((p / G) & 31));
      return act ? c : 0u;
    };
    // lane-wise exact evaluation of a contact or tether with slot k (the
    // pivot's position on every lane: bq0..2)
    double bq0 = 0.0, bq1 = 0.0, bq2 = 0.0;
    auto all_axes = [&]() {
      bq0 = __shfl_sync(FULL, qa, gbase);
      bq1 = __shfl_sync(FULL, qa, gbase + 1);
      bq2 = __shfl_sync(FULL, qa, gbase + 2);
    };
    bool wrg0 = false, wrg1 = false, wrg2 = false;  // wrap flags of the group's axes
    auto wrap_flags = [&]() {
      const unsigned wb = __ballot_sync(FULL, wra) >> gbase;
      wrg0 = wb & 1;
      wrg1 = wb & 2;
      wrg2 = wb & 4;
    };
    auto exact = [&](int k, bool te) {
      const int kid = __float_as_int(st.sh[k].w);
      const double k0 = pos64(st, Rr, k, kid, 0, M64), k1 = pos64(st, Rr, k, kid, 1, M64),
                   k2 = pos64(st, Rr, k, kid, 2, M64);
      double dv;
      const double x = quad_x(te, wrap_bits(bq0 - k0, SYS(L)[0], SYS(half)[0], wrg0),
                              wrap_bits(bq1 - k1, SYS(L)[1], SYS(half)[1], wrg1),
                              wrap_bits(bq2 - k2, SYS(L)[2], SYS(half)[2], wrg2), v0, v1, v2,
                              (te ? P.b2 : P.sig2), dv, PO);
      if (F32) ++confirmed;
      if (!neg(x)) keep(x, ((te ? KIND_TETHER : KIND_HS) << 28) | k, dv, 0.0);
    };

    // walls: lane a < 3 of the group, axis a; tethers: lanes TL and TL + 1
    constexpr int TL = G >= 8 ? 4 : 0;
    bool sw = DOM && gl < 3 && act && nonzero(va);
    bool sth = false;
    int ts = 0;
    if (!SPRING && act && (gl == TL || gl == TL + 1)) {
      const int t = gl == TL ? nb_prev(nbw) : nb_next(nbw);
      sth = t >= 0;
      if (sth) ts = CI(t, S, 20, P.status);
    }
    // Which lanes may hold the winner: `quads`, more than one quad of a group;
    // `lanes`, single lanes (walls, lane-wise evaluation: no Cand::pos)
    bool quads, lanes = false;
    if (F32) {
      int ks0 = -1, ks1 = -1;
      float kl0 = INF, kl1 = INF;
      bool kovf = false;
      int nscr = 0;
      // the FP32 numbers of this lane's tether and wall
      float tdv = 0.f, trad = 0.f;
      if (sth) {
        const float4 f = st.sh[ts];
        float d0 = pf0 - f.x, d1 = pf1 - f.y, d2 = pf2 - f.z;
        if (!DOM) {
          d0 = wrapf(d0, P.Lf[0]);
          d1 = wrapf(d1, P.Lf[1]);
          d2 = wrapf(d2, P.Lf[2]);
        }
        const float dd = __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, d0 * d0));
        tdv = __fmaf_rn(d2, vf2, __fmaf_rn(d1, vf1, d0 * vf0));
        trad = P.b2_f - (dd - tdv * tdv) - eps_d;
      }
      const float vfa = ax == 0 ? vf0 : (ax == 1 ? vf1 : vf2);
      const float pfa = ax == 0 ? pf0 : (ax == 1 ? pf1 : pf2);
      const float wdist = (signbit(vfa) ? pfa : Wfa - pfa) - eps_v, wav = fabsf(vfa) * 1.000002f;
      // screen up to two obstacles, so that their loads overlap
      auto screen2 = [&](int ka, int kb, bool two) {
        const float4 fa = st.sh[ka], fb = st.sh[kb];
        float a0 = pf0 - fa.x, a1 = pf1 - fa.y, a2 = pf2 - fa.z;
        float b0 = pf0 - fb.x, b1 = pf1 - fb.y, b2 = pf2 - fb.z;
        if (!DOM) {
          a0 = wrapf(a0, P.Lf[0]);
          a1 = wrapf(a1, P.Lf[1]);
          a2 = wrapf(a2, P.Lf[2]);
          b0 = wrapf(b0, P.Lf[0]);
          b1 = wrapf(b1, P.Lf[1]);
          b2 = wrapf(b2, P.Lf[2]);
        }
        screen_hs(Z, a0, a1, a2, vf0, vf1, vf2, ka, ubl, ks0, kl0, ks1, kl1, kovf);
        if (two) screen_hs(Z, b0, b1, b2, vf0, vf1, vf2, kb, ubl, ks0, kl0, ks1, kl1, kovf);
      };
      bool listed = false;
      int total = 0;  // obstacles in the list
      if (G <= 4) {
        // With few lanes a group's obstacles spread unevenly over them, and
        // the warp would go round as often as its fullest lane asks: deal
        // them out through a list.
        for (int w = 0; w < W; ++w) nscr += __popc(cand_word(w));
        int incl = nscr;
#pragma unroll
        for (int off = 1; off < G; off <<= 1) {
          const int t = __shfl_up_sync(FULL, incl, off, G);
          if (gl >= off) incl += t;
        }
        total = __shfl_sync(FULL, incl, gbase + G - 1);
        listed = !__any_sync(FULL, total > LIST_CAP);
        if (listed) {
          int at = incl - nscr;
          for (int w = 0; w < W; ++w) {
            unsigned c = cand_word(w);
            while (c) {
              st.lst[at++] = ((w << 5) + __ffs(c) - 1) * G + gl;
              c &= c - 1;
            }
          }
          __syncwarp();
          for (int j = gl; j < total; j += 2 * G) {
            const bool two = j + G < total;
            screen2(CI(st.lst[j], S, 21, P.status), CI(st.lst[two ? j + G : j], S, 21, P.status), two);
          }
        }
        nscr = gl == 0 ? total : 0;
      }
      if (!listed) {
        for (int w = 0; w < W; ++w) {
          unsigned c = cand_word(w);
          if (G > 4) nscr += __popc(c);
          while (c) {
            const int ka = CI(((w << 5) + __ffs(c) - 1) * G + gl, S, 21, P.status);
            c &= c - 1;
            const bool two = c != 0;
            const int kb = two ? CI(((w << 5) + __ffs(c) - 1) * G + gl, S, 21, P.status) : ka;
            c &= c - 1;
            screen2(ka, kb, two);
          }
        }
      }
      const float U = G == 32 ? __uint_as_float(__reduce_min_sync(FULL, __float_as_uint(ubl))) : group_minf<G>(ubl);
      // A wall or a tether can win only when its lower bound reaches U:
      // (dist - eps) / |v| <= U, and -dv - eps + sqrt(rad - eps_d) <= U.
      sw = sw && wdist <= U * wav;
      const bool bonded = sth;
      {
        const float q = U + tdv + eps_v;
        sth = sth && q >= 0.f && trad <= q * q * 1.000002f;
      }
      bool h0 = ks0 >= 0 && kl0 <= U, h1 = ks1 >= 0 && kl1 <= U;
      bool all_fp64 = false;  // evaluate every obstacle in the box
      if (P.rq_per_tile < 6) {
        // a small request_cap sends tiles with more survivors than that (or
        // more than 4 per request in reach) to the exhaustive evaluation
        int ns = sth + sw + h0 + h1;
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) {
          ns += __shfl_xor_sync(FULL, ns, off);
          nscr += __shfl_xor_sync(FULL, nscr, off);
        }
        all_fp64 = act && (ns > P.rq_per_tile || nscr > 4 * P.rq_per_tile);
        if (all_fp64) {
          if (gl == 0) ++exh;
          h0 = h1 = kovf = false;
          sth = bonded;
          sw = DOM && gl < 3 && nonzero(va);
        }
      }
      // ---------------------------------------------------------- B: FP64
      // The quads of a group take its survivors, one each per round
      // (rarely more than one survives).
      quads = SPRING && NQ > 1;
      for (;;) {
        const int code = sth ? (KIND_TETHER << 28) | ts : (h0 ? (KIND_HS << 28) | ks0 : (h1 ? (KIND_HS << 28) | ks1 : 0));
        const unsigned mine = (__ballot_sync(FULL, code != 0) & gmask) >> gbase;
        unsigned left = mine;
#pragma unroll
        for (int i = 0; i < NQ - 1; ++i)
          if (i < qd) left &= left - 1u;
        const int qcode = __shfl_sync(FULL, code, gbase + __ffs(left) - 1);
        const bool on = left != 0u;
        const bool te = (qcode >> 28) == KIND_TETHER;
        const int k = on ? CI(qcode & 0xFFFFFFF, S, 24, P.status) : 0;
        const int kid = __float_as_int(st.sh[k].w);
        double d = 0.0, dv, dd, pos = 0.0;
        if (on && ax < 3) {
          pos = pos64(st, Rr, k, kid, ax, M64);
          d = wrap_a(qa - pos, wra);
        }
        dots(FULL, d, dv, dd);
        const double R2 = (te ? P.b2 : P.sig2);
        double rad = R2 - __fma_rn(-dv, dv, dd);
        const bool hit = on && (te || (neg(dv) && posv(rad) && !(PO && dbits(dd) < dbits(R2))));
        if (te && neg(rad)) rad = 0.0;
        const double q = sqrt_rn(hit ? rad : 1.0);
        double x = -dv + (te ? q : flip(q));
        if (neg(x)) x = 0.0;
        if (hit) keep(x, qcode, dv, pos);
        if (on && ax == 0) ++confirmed;
        // survivors that did not get a quad, or share a lane with one that did
        bool more = code != 0 && __popc(mine & ((1u << gl) - 1u)) >= NQ;
        if (code != 0 && !more) {
          more = sth ? h0 || h1 : h0 && h1;
          if (sth) sth = false;
          else if (h0) h0 = false;
          else h1 = false;
        }
        quads = quads || (mine & (mine - 1u)) != 0u;
        if (!__any_sync(FULL, more)) break;
        quads = true;
      }
      lanes = __any_sync(FULL, kovf || all_fp64 || sw);
      if (lanes && __any_sync(FULL, kovf || all_fp64)) {
        wrap_flags();
        all_axes();
        if (act && (kovf || all_fp64)) {
          // more than two possible winners in this lane: screen its obstacles
          // again against the group's U and evaluate every one that can reach
          // it (exhaustive evaluation: all of them)
          auto again = [&](int k) {
            if (!all_fp64) {
              if (k == ks0 || k == ks1) return;
              const float4 f = st.sh[k];
              float d0 = pf0 - f.x, d1 = pf1 - f.y, d2 = pf2 - f.z;
              if (!DOM) {
                d0 = wrapf(d0, P.Lf[0]);
                d1 = wrapf(d1, P.Lf[1]);
                d2 = wrapf(d2, P.Lf[2]);
              }
              bool possible;
              const float lb = screen_lb(Z, d0, d1, d2, vf0, vf1, vf2, possible);
              if (!possible || lb > U) return;
            }
            exact(k, false);
          };
          if (listed) {  // (the obstacles dealt to this lane)
            for (int j = gl; j < total; j += G) again(CI(st.lst[j], S, 22, P.status));
          } else {
            for (int w = 0; w < W; ++w) {
              unsigned c = cand_word(w);
              while (c) {
                const int k = CI(((w << 5) + __ffs(c) - 1) * G + gl, S, 22, P.status);
                c &= c - 1;
                again(k);
              }
            }
          }
        }
        __syncwarp();
      }
      quads = __any_sync(FULL, quads || kovf || all_fp64);
    } else {
      // plain form: the tethers, the walls in reach and every obstacle in the
      // box.  A lane's words hold an uneven share of them and an evaluation
      // costs the warp the same for one lane as for all, so they are dealt out
      // through a list: as a rule one round instead of as many as the fullest
      // lane would take.
      wrap_flags();
      all_axes();
      if (sw) {
        const float vfa = ax == 0 ? vf0 : (ax == 1 ? vf1 : vf2);
        const float pfa = ax == 0 ? pf0 : (ax == 1 ? pf1 : pf2);
        sw = (signbit(vfa) ? pfa : Wfa - pfa) - eps_v <= xc * fabsf(vfa) * 1.000002f;
      }
      int total = 0;
      for (int from = 0; from == 0 || __any_sync(FULL, from < total); from += LIST_CAP) {
        total = 0;
        auto deal = [&](bool have, int code) {
          const unsigned b = (__ballot_sync(FULL, have) & gmask) >> gbase;
          const int at = total + __popc(b & ((1u << gl) - 1u)) - from;
          if (have && at >= 0 && at < LIST_CAP) st.lst[at] = code;
          total += __popc(b);
        };
        deal(sth, (KIND_TETHER << 28) | ts);
        for (int w = 0; w < W; ++w) {
          unsigned c = cand_word(w);
          while (__any_sync(FULL, c != 0u)) {
            deal(c != 0u, (KIND_HS << 28) | (((w << 5) + __ffs(c) - 1) * G + gl));
            c &= c - 1u;
          }
        }
        __syncwarp();
        const int n = total - from < LIST_CAP ? total - from : LIST_CAP;
        for (int j = gl; j < n; j += G) {
          const int code = st.lst[j];
          exact(CI(code & 0xFFFFFFF, S, 23, P.status), (code >> 28) == KIND_TETHER);
        }
        __syncwarp();
      }
      lanes = true;
      quads = NQ > 1;
    }
    if (DOM && lanes) {
      if (__any_sync(FULL, sw)) {
        if (sw) {
          const double loc = wrap_a(qa - ca, wra);
          double x = div_rn((posv(va) ? SYS(W)[axc] : 0.0) - loc, va);
          if (neg(x)) x = 0.0;
          if (F32) ++confirmed;
          // A bead on its tile's lower wall, moving out, meets it after
          // -0.0: bits that order above every candidate.  It competes as 0;
          // d.v, which a wall does not have, keeps the zero's sign for the
          // records.
          keep(from_bits(dbits(x) & 0x7FFFFFFFFFFFFFFFull), (KIND_WALL << 28) | ax, x, 0.0);
        }
        __syncwarp();
      }
    }
    // ---------------- winner of the group and its pre-flight d.v
    auto exchange = [&](int off) {
      const uint64_t ox = __shfl_xor_sync(FULL, best.x, off);
      const int oc = __shfl_xor_sync(FULL, best.code, off);
      const double odv = __shfl_xor_sync(FULL, best.dv, off);
      const double op = __shfl_xor_sync(FULL, best.pos, off);
      if (oc != CAND_NONE && oc != best.code && beats(ox, oc)) {
        best.x = ox;
        best.code = oc;
        best.dv = odv;
        best.pos = op;
      }
    };
    bool done = false;
    if (!F32) {
      // single lanes hold the candidates: the smallest upper half of x settles
      // it unless two share it
      const unsigned hi = best.code == CAND_NONE ? ~0u : (unsigned)(best.x >> 32);
      unsigned mn = hi;
      if (G == 32) {
        mn = __reduce_min_sync(FULL, hi);
      } else {
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) mn = min(mn, __shfl_xor_sync(FULL, mn, off));
      }
      const unsigned own = __ballot_sync(FULL, hi == mn) & gmask;
      done = !__any_sync(FULL, mn != ~0u && (own & (own - 1u)) != 0u);
      if (done) {
        const int src = __ffs(own) - 1;
        best.x = __shfl_sync(FULL, best.x, src);
        best.code = __shfl_sync(FULL, best.code, src);
        best.dv = __shfl_sync(FULL, best.dv, src);
      }
    }
    if (lanes && !done) {
      // (a lane-wise candidate carries no position: it is read again below)
      exchange(1);
      exchange(2);
    }
    if (done) {
    } else if (NQ > 1 && quads) {
#pragma unroll
      for (int off = 4; off < G; off <<= 1) exchange(off);
    } else if (NQ > 1) {
      // one candidate at most, the first quad's
      best.x = __shfl_sync(FULL, best.x, gbase + ax);
      best.code = __shfl_sync(FULL, best.code, gbase + ax);
      best.dv = __shfl_sync(FULL, best.dv, gbase + ax);
      best.pos = __shfl_sync(FULL, best.pos, gbase + ax);
    }

    // ---------------------------------------------------------- D: move
    if (act && nev >= event_cap) {
      if (gl == 0) set_status(P.status, DEV_STUCK);
      settle(p, pid, qa, pf0, pf1, pf2, oslab);
      state = EC_NEED;
    }
    if (state == EC_RUN) {
      double x = pass ? P.s_cap : xrem;
      int kind = pass ? KIND_PASS : KIND_END, slot = 0, partner = -1;
      if (best.x < dbits(x)) {  // (END and PASS win ties)
        x = from_bits(best.x);
        kind = best.code >> 28;
        slot = best.code & 0xFFFFFFF;
        partner = slot;
      }
      const bool bead = kind >= KIND_HS;
      double ka = best.pos;  // the partner's position on this lane's axis
      if (bead) {
        slot = CI(slot, S, 30, P.status);
        partner = __float_as_int(st.sh[slot].w);
        if (lanes && ax < 3) ka = pos64(st, Rr, slot, partner, ax, M64);
      }
      // r + x v on the axes, what is left of ell on lane 3, and on lane AL
      // (of G >= 8) the projection (r_target - r_pivot).v = -(d.v) - x
      double y = __fma_rn(x, va, (G >= 8 && gl == AL ? flip(best.dv) : qa));
      const double proj = G >= 8 ? y : -best.dv - x;
      if (wra) {
        const int di = wrap_step(y, SYS(L)[axc]);
        if (di && gl < 3) Ri[3 * (int64_t)pid + gl] += di;
      }
      qa = y;
      xrem = __shfl_sync(gmask, qa, gbase + 3);
      if (G >= 8 && gl == AL) qa = xrem;
      ++nev;
      int out = kind == KIND_END ? ECMC_EV_END : (kind == KIND_PASS ? ECMC_EV_PASS : ECMC_EV_WALL);
      int np = p;
      bool swapped = false;
      if (bead) {
        const bool hs = kind == KIND_HS;
        const bool motile = slot < m;
        out = hs ? (motile ? ECMC_EV_HS_LIFT : ECMC_EV_HS_REFLECT)
                 : (motile ? ECMC_EV_TE_LIFT : ECMC_EV_TE_REFLECT);
        const double acc = (motile ? lift : refl_all) + proj;
        if (motile) lift = acc;
        else refl_all = acc;
        if (!motile) {
          // v <- v - (2 v.d / d.d) d: reflection at the plane normal to d
          // (Fig. 2c)
          double d = 0.0, vd, dd;
          if (ax < 3) d = wrap_a(qa - ka, wra || (SPRING && !hs));
          dots(gmask, d, vd, dd);
          const double t = twice(div_rn(vd, dd));
          va = __fma_rn(-t, d, va);  // (lane 3: d = 0)
          v0 = __shfl_sync(gmask, va, gbase);
          v1 = __shfl_sync(gmask, va, gbase + 1);
          v2 = __shfl_sync(gmask, va, gbase + 2);
          new_direction();
        } else {
          np = slot;
          if (!SPRING && !PO && hs && P.swap_mode) {
            bool go = true;
            if (P.swap_mode != 1) {
              // the proposals of the next 4 min(G, 8) contacts, drawn
              // together: lane j draws the four of counter word ncontact/4 + j
              constexpr int NB = G < 8 ? 16 : 32;
              if ((ncontact & (NB - 1)) == 0) {
                const uint64_t r2 = DOM ? (uint64_t)unit : (uint64_t)(sweep + e);
                const u64x4 w = philox(TAG_SWAP | ((uint64_t)(DOM ? e : 0) << 8), r1, r2,
                                       (uint64_t)((ncontact >> 2) + (gl & (NB / 4 - 1))), P.seed, Rkey);
                unsigned g4 = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) g4 |= ((w.v[i] >> 11) < P.swap_thr ? 1u : 0u) << i;
                swgo = 0;
#pragma unroll
                for (int j = 0; j < NB / 4; ++j) swgo |= __shfl_sync(gmask, g4, gbase + j) << (4 * j);
              }
              go = (swgo >> (ncontact & (NB - 1))) & 1u;
              ++ncontact;
            }
            if (go) {
              if (gl == 0) ++tried;
              // every bond of both beads, positions exchanged, within b_max:
              // bond j (pivot to previous, next; partner to previous, next)
              // on quad j
              bool ok = true;
              const uint2 nb2 = st.nb[slot];
              const unsigned nbs = nb2.x;
#pragma unroll
              for (int j0 = 0; j0 < 4; j0 += NQ) {
                const int j = j0 + qd;
                const unsigned nbv = (j & 2) ? nbs : nbw;
                const int b = j >= 4 ? -1 : ((j & 1) ? nb_next(nbv) : nb_prev(nbv));
                double d = 0.0, dv, dd;
                if (b >= 0 && ax < 3) {
                  const double pa = (j & 2) ? qa : ka;
                  const double ba = b == p ? ka : (b == slot ? qa : pos64(st, Rr, b, __float_as_int(st.sh[b].w), ax, M64));
                  d = wrap_a(pa - ba, wra);
                }
                dots(gmask, d, dv, dd);
                ok = ok && !(b >= 0 && dbits(dd) > dbits(P.b2));
              }
              ok = (__ballot_sync(gmask, ok) & gmask) == gmask;
              if (ok) {
                swapped = true;
                out = ECMC_EV_SWAP;
                np = p;
                const int kid = __float_as_int(st.sh[slot].w);
                float g0, g1, g2;
                shadows(qa, g0, g1, g2);
                settle(slot, kid, qa, g0, g1, g2, (int)nb2.y);
                if (gl < 3) {
                  const int ti = Ri[3 * (int64_t)pid + gl];
                  Ri[3 * (int64_t)pid + gl] = Ri[3 * (int64_t)kid + gl];
                  Ri[3 * (int64_t)kid + gl] = ti;
                }
                if (ax < 3) qa = ka;
              }
            }
          }
        }
      } else if (kind == KIND_WALL) {
        // (negation is exact in both precisions)
        const int wa = partner;
        if (ax == wa) va = flip(va);
        if (wa == 0) {
          v0 = flip(v0);
          vf0 = -vf0;
        } else if (wa == 1) {
          v1 = flip(v1);
          vf1 = -vf1;
        } else {
          v2 = flip(v2);
          vf2 = -vf2;
        }
      }
      ev_lo += gl == (G >= 8 ? out : out & 3) && (G >= 8 || out < 4) ? 1u : 0u;
      if (G < 8) ev_hi += out >= 4 && gl == (out & 3) ? 1u : 0u;
      __syncwarp(gmask);
      shadows(qa, pf0, pf1, pf2);
      // (x as recorded)
      auto flight = [&]() { return kind == KIND_WALL ? best.dv : x; };
      if (P.rec_digest) {
        fnv_mix(h, (uint64_t)pid);
        fnv_mix(h, ((uint64_t)(uint32_t)out << 32) | (uint64_t)(uint32_t)partner);
        fnv_mix(h, dbits(flight()));
      }
      if (P.log && gl == 0) {
        const unsigned long long at = atomicAdd(P.log_n, 1ull);
        if ((int64_t)at < P.log_cap) {
          ecmc_event ev;
          ev.unit = P.rec_offset + (P.sweep_dev ? (sweep - P.rec_sweep0) * P.n_units * P.ecs_per_tile : 0) +
                    (DOM ? (int64_t)gunit * P.ecs_per_tile + e : (int64_t)e);
          ev.seq = (int32_t)(nev - 1);
          ev.pivot = pid;
          ev.kind = out;
          ev.pad = 0;
          ev.partner = partner;
          ev.x = flight();
          P.log[at] = ev;
        }
      }
      if (out == ECMC_EV_END || np != p) settle(p, pid, qa, pf0, pf1, pf2, oslab);
      if (out == ECMC_EV_END) state = EC_NEED;
      if (np != p) {
        // lift: the partner (motile, unmoved this event) becomes the pivot
        p = np;
        const float4 f = st.sh[p];
        pid = CI(__float_as_int(f.w), BATCH ? rp->n_beads : P.n, 31, P.status);
        const uint2 nb = st.nb[p];
        nbw = nb.x;
        oslab = (int)nb.y;
        pmask = gl == (p & (G - 1)) && p / G < 32 ? ~(1u << ((p / G) & 31)) : ~0u;
        if (ax < 3) qa = ka;
        pf0 = f.x;
        pf1 = f.y;
        pf2 = f.z;
      }
    }
    if (act && state == EC_NEED) {
      // end of an EC: records, then the tile's next EC or a new tile
      lift_all = lift_all + lift;
      nev_all += (unsigned long long)nev;
      ++ecs_done;
      if (gl == AL && P.rec_digest) {
        const int64_t idx = P.rec_offset +
                            (P.sweep_dev ? (sweep - P.rec_sweep0) * P.n_units * P.ecs_per_tile : 0) +
                            (DOM ? (int64_t)gunit * P.ecs_per_tile + e : (int64_t)e);
        if (idx < P.rec_cap) {
          P.rec_digest[idx] = h;
          P.rec_lift[idx] = lift;
          P.rec_events[idx] = (int64_t)nev;
        }
      }
      ++e;
      if (e >= n_ec) state = TILE_NEED;
    }
    __syncwarp();
  }

  // ------------------------------------------------------------ counters
  if (F32) {
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) confirmed += __shfl_xor_sync(FULL, confirmed, off);
  }
  if (gl == 0 && ecs_done) {
    atomicAdd(&P.counters[CNT_EVENTS], nev_all);
    if (tried) atomicAdd(&P.counters[CNT_SWAP_TRIED], (unsigned long long)tried);
    if (confirmed) atomicAdd(&P.counters[CNT_CONFIRMED], (unsigned long long)confirmed);
    if (exh) atomicAdd(&P.counters[CNT_EXHAUSTIVE], (unsigned long long)exh);
    atomicAdd(&P.counters[CNT_ECS], (unsigned long long)ecs_done);
    atomicAdd(&P.sums[SUM_DISP], (double)ecs_done * P.ell);  // an EC's flights add up to ell
  }
  if (gl < ECMC_NEV && ev_lo) atomicAdd(&P.counters[gl], (unsigned long long)ev_lo);
  if (G < 8 && ev_hi) atomicAdd(&P.counters[(gl & 3) + 4], (unsigned long long)ev_hi);
  if (gl == AL && ecs_done) {
    atomicAdd(&P.sums[SUM_LIFT], lift_all);
    atomicAdd(&P.sums[SUM_REFL], refl_all);
  }
}
#undef SYS


// Shared memory of one tile for G lanes and S staged beads: the slab side is
// 0.3 sigma (a reach box then holds about 12 obstacles at phi = 0.45, 9 with
// infinitely thin slabs) and grows while the masks of a tile would take
// more than `budget` bytes; at least 10 slabs (staging keeps S ids in the
// masks' area).  The launch gives 2 KB to tiles of 4 and 8 lanes, 192 bytes
// per lane to the others; with half / with twice that, a pass of the 1e6-bead
// melt takes 44.1 / 47.0 ms (43.6), 262k beads in FP64 5.29 / 5.12 (5.00), 64
// replicas 207 / 205 (205), 48,000 beads on springs 10.90 / 10.97 (10.92).
struct SlabPick {
  float inv;
  int nsl;
};
inline SlabPick pick_slabs(double e_max, double sigma, int S, int G, size_t budget) {
  SlabPick k{};
  for (double side = 0.3 * sigma;; side *= 1.1) {
    k.inv = (float)(1.0 / side);
    const double ns = floor(e_max / side) + 3.0;
    k.nsl = ns < 10.0 ? 10 : (ns > 1000.0 ? 1001 : (int)ns);
    if (k.nsl <= 1000 && (k.nsl == 10 || (size_t)mask_quads(S, G, k.nsl) * 16 <= budget)) return k;
  }
}

// the staging capacity, at most S and at least M, that fits `room` bytes with
// the fewest slabs
inline int fit_stage(int S, int M, int G, size_t room) {
  while (S - 32 >= M && group_bytes(S, 0, M, mask_quads(S, G, 10)) > room) S -= 32;
  return S;
}

template <int G, bool F32, bool BATCH, bool DOM, bool SPRING, bool PO>
cudaError_t launch_ec_t(const ECParams &P0, cudaStream_t s) {
  auto kern = ec_kernel<G, F32, BATCH, DOM, SPRING, PO>;
  // the device's limits, asked again when the thread has changed its device
  static thread_local int sms = 0, smem_max = 0, device = -1;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess && dev != device) {
    device = -1;
    err = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err == cudaSuccess) device = dev;
  }
  if (err == cudaSuccess) err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (err != cudaSuccess) return err;
  // tiles per block and resident blocks of the last shapes asked for
  struct Shape {
    int S, M64, M, nsl, bt, nt, blocks, units, dev;
    float inv;
    size_t smem;
  };
  static thread_local Shape memo[4];
  static thread_local int memo_at = 0;
  auto shape = [&](int S, int M, Shape *out) -> cudaError_t {
    ECParams const &P = P0;
    const int step = 32 / G;
    const size_t room = (size_t)smem_max / step;  // one warp's tiles must fit a block
    SlabPick k{};
    // (the capacity counts every bead of the tether halo, with long tethers
    // many times what is staged: where even one tile of it would not fit, the
    // tile takes what fits)
    if (DOM && G == 32) S = fit_stage(S, M, G, room);
    if (DOM) {
      k = pick_slabs(P.e_max, P.s_len, S, G, (size_t)(G <= 8 ? 2048 : 192 * G));
      if (group_bytes(S, 0, M, mask_quads(S, G, k.nsl)) > room)
        k = pick_slabs(P.e_max, P.s_len, S, G, 0);
    } else {
      // the box's own slabs, nsl of them around every axis
      k.nsl = 30;
      while (k.nsl > 3 && group_bytes(S, 0, M, mask_quads(S, G, k.nsl)) > room) --k.nsl;
      k.inv = 1.f;
    }
    for (const Shape &h : memo)
      if (h.nt && h.S == S && h.M == M && h.bt == P.block_tiles && h.nsl == k.nsl && h.inv == k.inv &&
          h.units == P.n_units && h.dev == dev) {
        *out = h;
        return cudaSuccess;
      }
    Shape w{};
    w.S = S;
    w.M = M;
    w.bt = P.block_tiles;
    w.units = P.n_units;
    w.dev = dev;
    w.nsl = k.nsl;
    w.inv = k.inv;
    const int MQ = mask_quads(S, G, w.nsl);
    // FP64 positions in shared memory: the plain form reads many of them per
    // event; the screened form one (an L2 round trip less on every event),
    // and keeps them there only while all tiles stay resident
    size_t per = 0;
    for (int want = S;; want = 0) {
    w.M64 = want;
    w.nt = w.blocks = 0;
    per = group_bytes(S, want, M, MQ);
    int best = -1;
    for (int t = step; t <= 128 / G; t += step) {
      if (P.block_tiles > 0 && t != P.block_tiles && per * P.block_tiles <= (size_t)smem_max &&
          P.block_tiles % step == 0 && P.block_tiles <= 128 / G)
        continue;
      if (per * t > (size_t)smem_max) break;
      int blocks = 0;
      cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kern, t * G, per * t);
      if (e != cudaSuccess) return e;
      if (blocks * t > best) {
        best = blocks * t;
        w.nt = t;
        w.blocks = blocks;
      }
    }
    if (want == 0 || (w.nt > 0 && (!F32 || (long long)w.blocks * w.nt * sms >= P.n_units))) break;
    }
    if (w.nt == 0 || w.blocks < 1) return cudaErrorInvalidValue;
    w.smem = per * w.nt;
    memo[memo_at] = w;
    memo_at = (memo_at + 1) & 3;
    *out = w;
    return cudaSuccess;
  };
  // persistent groups: as many as stay resident, each taking tiles from the
  // unit counter until none are left
  auto run = [&](const Shape &h, int mode) -> cudaError_t {
    ECParams P = P0;
    P.stage_cap = h.S;
    P.m_cap = h.M;
    P.m64 = h.M64;
    P.nsl = h.nsl;
    P.sorg = DOM ? P.lorg : 0.f;
    for (int a = 0; a < 3; ++a) {
      P.sinv[a] = DOM ? h.inv : (float)(h.nsl / P.L[a]);
      P.Lf[a] = (float)P.L[a];
      P.Wf[a] = (float)P.W[a];
    }
    P.sigma_f = round_up_f32(P.sigma);
    P.sig2_f = (float)P.sig2;
    P.b2_f = (float)P.b2;
    P.halo_hs_f = round_up_f32(P.halo_hs);
    P.halo_te_f = round_up_f32(P.halo_te);
    P.defer_mode = mode;
    const long long want = (P.n_units + h.nt - 1) / h.nt;
    const long long room = (long long)h.blocks * sms;
    const int blocks = (int)(want < room ? want : room);
    // (the cell pass before a domain launch clears the unit counters)
    if (!DOM) {
      const cudaError_t e = cudaMemsetAsync(P.unit_next, 0, sizeof(int32_t), s);
      if (e != cudaSuccess) return e;
    }
    if (mode == 2) P.unit_next += 1;
    if (blocks > 0) kern<<<blocks, h.nt * G, h.smem, s>>>(P);
    return cudaGetLastError();
  };
  Shape full{};
  cudaError_t e = shape(P0.stage_cap, P0.m_cap, &full);
  if (e != cudaSuccess) return e;
  // A first pass with tight capacities keeps more tiles resident; the tiles
  // that do not fit run in a second one.  When all tiles are resident with
  // the full capacities anyway, one pass does it.
  const bool two = P0.stage_tight > 0 && P0.m_tight > 0 && P0.deferred && P0.n_deferred &&
                   (P0.stage_tight < P0.stage_cap || P0.m_tight < P0.m_cap) &&
                   (long long)full.blocks * full.nt * sms < P0.n_units;
  if (!two) return run(full, 0);
  Shape tight{};
  e = shape(P0.stage_tight, P0.m_tight, &tight);
  if (e == cudaSuccess) e = run(tight, 1);
  if (e == cudaSuccess) e = run(full, 2);
  return e;
}

}  // namespace
}  // namespace ecmc
