// Mid pass of the fused FFT iteration: forward length-N1 FFTs along the rows
// of the N2 x N1 exchange array (with the four-step twiddle), the spectrum
// operator over every (k, N - k) pair, and the inverse FFTs.
// Included by cs_mid.cu (run-time and large static shapes) and cs_mid8.cu
// (radix-8 shapes).
#pragma once

#include "cs_passes.cuh"

namespace csk {

namespace {

// ---------------------------------------------------------------- mid pass

// w_N^(j1 k2) from the two-level table: w_N^p = w_N^(p mod N1) * w_N2^(p div N1)
__device__ __forceinline__ float2 tw4(const Geo& g, int p) {
  return cmul(__ldg(g.twl + (p & (g.N1 - 1))), __ldg(g.tw2 + (p >> g.lgN1)));
}

__device__ __forceinline__ int slot_row(const Geo& g, int u, int second) {
  if (u == 0) return second ? (g.N2 >> 1) : 0;
  return second ? g.N2 - u : u;
}

// Global source / sink of the first forward and last inverse FFT stages of
// the static shapes: row `vec` of the tile is row slot_row(u0 + vec/2,
// vec & 1) of the N2 x N1 exchange array.
struct MidIO {
  static constexpr bool kGlobal = true;
  float2* W;
  int u0, lgN1, N2;
  __device__ __forceinline__ float2* at(int vec, int idx) const {
    const int u = u0 + (vec >> 1);
    const int k2 = u == 0 ? ((vec & 1) ? (N2 >> 1) : 0) : ((vec & 1) ? N2 - u : u);
    return W + ((size_t)k2 << lgN1) + idx;
  }
  __device__ __forceinline__ float2 load(int vec, int idx) const { return __ldcg(at(vec, idx)); }
  __device__ __forceinline__ void store(int vec, int idx, float2 v) const { __stcg(at(vec, idx), v); }
};

// Four-step twiddle as FFT hooks: w_N^(j1 k2) on the values the first
// forward stage loads, its conjugate on the values the last inverse stage
// produces (k2 = the tile row's index in the N2 x N1 array).  With
// j1 = j + r L/R:  w_N^(j1 k2) = w_N^(j k2) * w_N^(r (L/R) k2); the second
// factor comes from a per-CTA table rt[row][r] in shared memory.
constexpr int MID_MAX_ROWS = 64;   // 2U <= min(N2, TILE/N1) <= 64 rows, as N2 <= N1

// Static shapes: w_N^(j1 k2) = lo[j1 mod LO] * hi[j1 div LO], LO = 2^LOB = 16
// (8 for 64-point rows in radix 8), two per-row tables of LO and N1/LO
// entries (both exact FP64-rounded values).  With j1 = j + r L/R and
// L/R >= LO, lo depends on the thread only and hi is read at
// (j div LO) + r (L/R)/LO.
template <bool PRE, int LOB>
struct MidTwHookS {
  static constexpr bool kPre = PRE, kPost = !PRE;
  const float2* lo;   // [rows][LO]
  const float2* hi;   // [rows][N1/LO]
  int lgN1;
  float2 wl;
  __device__ __forceinline__ void begin(int vec, int j, int) { wl = lo[(vec << LOB) + (j & ((1 << LOB) - 1))]; }
  __device__ __forceinline__ float2 tw(int vec, int j, int r, int lgLR) const {
    return cmul(wl, hi[(vec << (lgN1 - LOB)) + (j >> LOB) + (r << (lgLR - LOB))]);
  }
  __device__ __forceinline__ float2 pre(int vec, int j, int r, int lgLR, float2 v) const {
    return cmul(v, tw(vec, j, r, lgLR));
  }
  __device__ __forceinline__ float2 post(int vec, int j, int r, int lgLR, float2 v) {
    return cmulc(v, tw(vec, j, r, lgLR));
  }
};

template <bool PRE>
struct MidTwHook {
  static constexpr bool kPre = PRE, kPost = !PRE;
  const Geo& g;
  int u0;
  const float2* rt;   // [2U][16]
  float2 wj;
  __device__ __forceinline__ void begin(int vec, int j, int) {
    wj = tw4(g, j * slot_row(g, u0 + (vec >> 1), vec & 1));
  }
  __device__ __forceinline__ float2 pre(int vec, int, int r, int, float2 v) const {
    return cmul(v, cmul(wj, rt[vec * 16 + r]));
  }
  __device__ __forceinline__ float2 post(int vec, int, int r, int, float2 v) {
    return cmulc(v, cmul(wj, rt[vec * 16 + r]));
  }
};
// Real-FFT spectrum operator (products with C and C^T on the packed vector).
// For the pair (k, N - k) of the packed spectrum Z, with H the real-signal
// spectrum of the product (H = chat for C^T, conj(chat) for C):
//   Z'_k   = a  Z_k   + b  conj(Z_{N-k})
//   Z'_N-k = a' Z_N-k + b' conj(Z_k),   b' = -conj(b)
// with, for H = chat, P = (H_k + H_{k+N})/2N, Q = (H_k - H_{k+N})/2N (the
// table, FP64-rounded once) and the packing phase w = exp(-i theta),
// theta = 2 pi k / 2N:  a = P - Q sin(theta), a' = conj(P + Q sin(theta)),
// b = i Q cos(theta).  H = conj(chat) conjugates a and a' and maps
// b -> -conj(b).  w = w_2N^k is the product of two small tables (1D:
// twr[k2] tw1[k1]; 2D, where the phase is that of the packed axis only:
// tw1[k1]).
template <bool ADJ>
__device__ __forceinline__ void op_real(const float4 t, float2 w, float2& za, float2& zb) {
  const float2 P = make_float2(t.x, t.y), Q = make_float2(t.z, t.w);
  // sin(theta) = -w.y, cos(theta) = w.x
  float2 al = make_float2(fmaf(w.y, Q.x, P.x), fmaf(w.y, Q.y, P.y));
  float2 al2 = make_float2(fmaf(-w.y, Q.x, P.x), -fmaf(-w.y, Q.y, P.y));
  float2 be = make_float2(-w.x * Q.y, w.x * Q.x);
  float2 be2 = make_float2(-be.x, be.y);
  if (!ADJ) {
    al = cconj(al);
    al2 = cconj(al2);
    const float2 tb = be;
    be = make_float2(-tb.x, tb.y);
    be2 = tb;
  }
  const float2 a2 = za, b2 = zb;
  za = cadd(cmul(al, a2), cmul(be, cconj(b2)));
  zb = cadd(cmul(al2, b2), cmul(be2, cconj(a2)));
}

// Complex-n ADMM operator for the pair (k, N - k) of Z = FFT((v) + i (z - nu)):
//   V = (Z_k + conj Z_{N-k}) / 2,  Wk = (Z_k - conj Z_{N-k}) / 2i
//   X = bhat (rho chat V + sigma Wk) / N            (x-update, Algorithm 3)
//   Pc = conj(chat) X                                 (spectrum of C x)
//   Z'_k = X + i Pc,  Z'_{N-k} = conj(X) + i conj(Pc)
__device__ __forceinline__ void op_admm(const float2 ch, const float bb, float rho, float sigma, float2& za,
                                        float2& zb) {
  const float2 V = make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y));
  const float2 Wk = make_float2(0.5f * (za.y + zb.y), -0.5f * (za.x - zb.x));
  const float2 cv = cmul(ch, V);
  const float2 X = make_float2(bb * fmaf(rho, cv.x, sigma * Wk.x),
                               bb * fmaf(rho, cv.y, sigma * Wk.y));
  const float2 Pc = cmulc(X, ch);
  za = make_float2(X.x - Pc.y, X.y + Pc.x);
  zb = make_float2(X.x + Pc.y, Pc.x - X.y);
}

// SHAPE 0: any geometry; SHAPE s > 0 fixes (log2 N1, log2 U) at compile time
// for the geometries of N = 2^20 (1024 x 1024, U = 2), 2^21 (2048 x 1024,
// U = 1) and 2^22 (4096 x 1024, U = 1).
// SHAPE 4..6: the same for a 2D DFT (no four-step twiddle; see Geo::twod):
// 4 any geometry, 5 and 6 fix (log2 N1, log2 U) = (11, 0) and (12, 0), the
// packed and the complex geometry of a 4096 x 4096 image.
// SHAPE 10 + LGN1 (1D) and 30 + LGN1 (2D), LGN1 = 6 .. 10: radix-8 tiles of
// one row pair (two for LGN1 = 6), 8 values per thread.
// SHAPE 50 + LGN1 (1D, LGN1 = 7 .. 11): 4096-value tiles, 16 values per thread
// (grouped launches).
template <int SHAPE> struct MidShape {
  static_assert((SHAPE >= 16 && SHAPE <= 20) || (SHAPE >= 36 && SHAPE <= 40) || (SHAPE >= 57 && SHAPE <= 61),
                "mid shapes");
  static constexpr bool kTwoD = SHAPE >= 30 && SHAPE <= 40, kR8 = SHAPE < 50;
  static constexpr int kLgN1 = SHAPE - (kTwoD ? 30 : kR8 ? 10 : 50);
  static constexpr int kLgU = kR8 ? (kLgN1 == 6 ? 1 : 0) : 11 - kLgN1;
  static constexpr int kLgR = kR8 ? 3 : 4, kVpt = kR8 ? VPT8 : EPT;
  static constexpr bool kTwFull = true;
  using Lay = StaticLayout<kLgN1, kLgU + 1, false, kLgR>;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgN1(const Geo&) { return kLgN1; }
  __device__ static constexpr int lgU(const Geo&) { return kLgU; }
};
template <> struct MidShape<0> {
  using Lay = DynLayout;
  static constexpr bool kTwoD = false, kTwFull = false;
  static constexpr int kLgR = 4, kVpt = EPT;
  __device__ static Lay lay(const Geo& g) { return Lay{g.lgN1, g.lgU + 1, false}; }
  __device__ static int lgN1(const Geo& g) { return g.lgN1; }
  __device__ static int lgU(const Geo& g) { return g.lgU; }
};
template <int LGN1, int LGU, bool TWOD = false> struct MidShapeS {
  using Lay = StaticLayout<LGN1, LGU + 1, false, 4, false>;
  static constexpr bool kTwoD = TWOD, kTwFull = false;
  static constexpr int kLgR = 4, kVpt = EPT;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgN1(const Geo&) { return LGN1; }
  __device__ static constexpr int lgU(const Geo&) { return LGU; }
};
template <> struct MidShape<1> : MidShapeS<10, 1> {};
template <> struct MidShape<2> : MidShapeS<11, 0> {};
template <> struct MidShape<3> : MidShapeS<12, 0> {};
template <> struct MidShape<4> : MidShape<0> { static constexpr bool kTwoD = true; };
template <> struct MidShape<5> : MidShapeS<11, 0, true> {};
template <> struct MidShape<6> : MidShapeS<12, 0, true> {};

// The mid pass of tile `blk` (row-pair units blk U .. blk U + U - 1).
template <int KIND, int TILE, int SHAPE>
__device__ __forceinline__ void mid_body(const KParams& kp, const int blk) {
  using S = MidShape<SHAPE>;
  constexpr bool R8 = S::kVpt == VPT8;
  constexpr int NT = Cfg<TILE, S::kVpt>::NT;
  constexpr int NLD = Cfg<TILE, S::kVpt>::NLD;
  extern __shared__ float2 sm[];
  pdl_trigger();
  const Geo& g = kp.geo;
  const int lgU = S::lgU(g), U = 1 << lgU;
  const int u0 = blk << lgU;
  const int lgN1 = S::lgN1(g), N1 = 1 << lgN1;
  const int tot = (2 * U) << lgN1;
  const auto lay = S::lay(g);
  float2* W = kp.pp.W;
  const float2* Wi = kp.pp.Wi;   // may be W
  constexpr bool TWS = S::Lay::kStatic;   // static shape: twiddles in shared memory
  constexpr bool TWOD = S::kTwoD;         // 2D DFT: no four-step twiddle hooks
  constexpr int LGN1S = TWS ? S::lgN1(Geo{}) : 4;
  constexpr int ROWS = TWS ? (2 << S::lgU(Geo{})) : MID_MAX_ROWS;
  constexpr int LOB = LGN1S - S::kLgR < 4 ? LGN1S - S::kLgR : 4;   // see MidTwHookS
  constexpr int TW_N = TWS ? stage_tw_count(LGN1S, S::kLgR, S::kTwFull) : 2;
  __shared__ __align__(16) float2 tws[TW_N];
  // static shapes: per-row lo[] and hi[]; dynamic: rt (see MidTwHook)
  constexpr int LOHI = (TWS && !TWOD) ? ROWS * ((1 << LOB) + (1 << (LGN1S - LOB))) : 2;
  __shared__ float2 lohi[LOHI];
  __shared__ float2 rt[2][(TWS || TWOD) ? 2 : MID_MAX_ROWS * 16];
  if (TWS) copy_table<NT>(tws, g.tws1, TW_N);
  if constexpr (TWOD) {
  } else if (TWS) {
    constexpr int LO = 1 << LOB, HI = 1 << (LGN1S - LOB);
    for (int t = threadIdx.x; t < ROWS * (LO + HI); t += NT) {
      const bool is_lo = t < ROWS * LO;
      const int tt = is_lo ? t : t - ROWS * LO;
      const int vec = is_lo ? (tt >> LOB) : (tt >> (LGN1S - LOB));
      const int q = is_lo ? (tt & (LO - 1)) : (tt & (HI - 1)) << LOB;
      const int k2 = slot_row(g, u0 + (vec >> 1), vec & 1);
      lohi[t] = tw4(g, (q * k2) & (g.N - 1));
    }
  } else {
    // rt[0][row][r] = w_N^(r (L/R) k2) for R the radix of the first stage (the
    // forward pre-hook), rt[1] for the radix of the last stage (inverse post-hook)
    const int lgRf = lgN1 >= 4 ? 4 : lgN1;
    const int lgRl = (lgN1 & 3) ? (lgN1 & 3) : 4;
    for (int t = threadIdx.x; t < 2 * 2 * U * 16; t += NT) {
      const int which = t / (2 * U * 16);
      const int tt = t - which * (2 * U * 16);
      const int vec = tt >> 4, r = tt & 15;
      const int lgR = which ? lgRl : lgRf;
      const int k2 = slot_row(g, u0 + (vec >> 1), vec & 1);
      rt[which][tt] = r < (1 << lgR) ? tw4(g, ((r << (lgN1 - lgR)) * k2) & (g.N - 1)) : make_float2(1.f, 0.f);
    }
  }
  // Pair slot t of this CTA: elements ea (frequency k = k2 + N2 k1) and eb
  // (frequency N - k) of the tile, table index tidx.
  const int nslots = (U << lgN1) + (u0 == 0 ? (TWOD ? 2 : 1) : 0);
  const int base_u1 = ((g.N2 >> 1) - 1) << lgN1;   // table offset of unit 0
  auto slot_at = [&](int t, int& ea, int& eb, int& k2, int& k1, int& tidx) {
    int ul, q;
    if (t < (U << lgN1)) { ul = t >> lgN1; q = t & (N1 - 1); }
    else { ul = 0; q = N1 + (t - (U << lgN1)); }
    const int u = u0 + ul;
    if constexpr (TWOD) {
      // 2D partner of (k2, k1): (-k2, -k1); unit 0: rows 0 and N2/2, each
      // with N1/2 + 1 slots q -> (q, (N1 - q) mod N1)
      if (u > 0) {
        k2 = u; k1 = q;
        ea = ((2 * ul) << lgN1) + q;
        eb = ((2 * ul + 1) << lgN1) + ((N1 - q) & (N1 - 1));
        tidx = ((u - 1) << lgN1) + q;
      } else {
        const bool hi = q > (N1 >> 1);
        const int qq = hi ? q - (N1 >> 1) - 1 : q;
        k2 = hi ? (g.N2 >> 1) : 0; k1 = qq;
        ea = ((2 * ul + (hi ? 1 : 0)) << lgN1) + qq;
        eb = ((2 * ul + (hi ? 1 : 0)) << lgN1) + ((N1 - qq) & (N1 - 1));
        tidx = base_u1 + q;
      }
      return;
    }
    if (u > 0) {
      k2 = u; k1 = q;
      ea = ((2 * ul) << lgN1) + q;
      eb = ((2 * ul + 1) << lgN1) + (N1 - 1 - q);
      tidx = ((u - 1) << lgN1) + q;
    } else if (q <= (N1 >> 1)) {
      k2 = 0; k1 = q;
      ea = ((2 * ul) << lgN1) + q;
      eb = ((2 * ul) << lgN1) + ((N1 - q) & (N1 - 1));
      tidx = base_u1 + q;
    } else {
      const int qq = q - (N1 >> 1) - 1;
      k2 = g.N2 >> 1; k1 = qq;
      ea = ((2 * ul + 1) << lgN1) + qq;
      eb = ((2 * ul + 1) << lgN1) + (N1 - 1 - qq);
      tidx = base_u1 + q;
    }
  };
  auto phase_at = [&](int k2, int k1) {
    return TWOD ? __ldg(g.tw1 + k1) : cmul(__ldg(g.twr + k2), __ldg(g.tw1 + k1));
  };
  // radix-8 tiles: the spectrum tables and phases of the thread's pair slots
  // (plan constants) are loaded while the pass before this one still runs
  constexpr bool PRET = R8 && (KIND == MID_FWD || KIND == MID_ADJ || KIND == MID_ADMM);
  constexpr int SL = PRET ? VPT8 / 2 : 1;
  float4 pt[SL];
  float2 pw[SL];
  if constexpr (PRET) {
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      int ea, eb, k2, k1, tidx;
      slot_at(threadIdx.x + i * NT, ea, eb, k2, k1, tidx);
      if constexpr (KIND == MID_ADMM) {
        pw[i] = __ldg(kp.pp.tab_admm_c + tidx);
        pt[i].x = __ldcg(kp.pp.tab_admm_b + tidx);   // re-tabulated between calls
      } else {
        pt[i] = __ldg(kp.pp.tab_ista + tidx);
        pw[i] = phase_at(k2, k1);
      }
    }
  }
  pdl_wait();   // everything above reads plan constants; W is not one
  const float a_rho = kp.ca->rho, a_sigma = kp.ca->sigma;   // ADMM only
  auto load_tile = [&](float2* dst, const float2* src) {
    float4 buf[NLD];
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = 2 * (threadIdx.x + i * NT);
      if (e < tot) {
        const int slot = e >> lgN1, j1 = e & (N1 - 1);
        const int k2 = slot_row(g, u0 + (slot >> 1), slot & 1);
        buf[i] = __ldcg(reinterpret_cast<const float4*>(src + ((size_t)k2 << lgN1) + j1));
      }
    }
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = 2 * (threadIdx.x + i * NT);
      if (e < tot) {
        dst[pad(e)] = make_float2(buf[i].x, buf[i].y);
        dst[pad(e + 1)] = make_float2(buf[i].z, buf[i].w);
      }
    }
    __syncthreads();
  };
  // static shapes: the first forward stage reads the rows from W itself
  // (after a barrier: its hook reads the twiddle tables written above)
  auto fwd_rows_from_global = [&]() {
    if constexpr (TWS) {
      __syncthreads();
      const MidIO io{const_cast<float2*>(Wi), u0, lgN1, g.N2};
      if constexpr (TWOD) {
        NoHook nh;
        tile_fft<-1, TILE, NT, true>(sm, lay, tws, lgN1, nh, io, SmemIO{});
      } else {
        MidTwHookS<true, LOB> h{lohi, lohi + (ROWS << LOB), LGN1S, make_float2(1.f, 0.f)};
        tile_fft<-1, TILE, NT, true>(sm, lay, tws, lgN1, h, io, SmemIO{});
      }
    }
  };
  auto fwd_rows = [&](float2* buf) {
    if constexpr (TWOD) {
      if constexpr (TWS) tile_fft<-1, TILE, NT, true>(buf, lay, tws, lgN1);
      else tile_fft<-1, TILE, NT, false>(buf, lay, g.tw1h, lgN1);
    } else if constexpr (TWS) {
      MidTwHookS<true, LOB> h{lohi, lohi + (ROWS << LOB), LGN1S, make_float2(1.f, 0.f)};
      tile_fft<-1, TILE, NT, true>(buf, lay, tws, lgN1, h);
    } else {
      MidTwHook<true> h{g, u0, rt[0], make_float2(1.f, 0.f)};
      tile_fft<-1, TILE, NT, false>(buf, lay, g.tw1, lgN1 + 1, h);
    }
  };
  if constexpr (KIND == MID_FWD_CORR || KIND == MID_ADJ_CORR) {
    // The product of the vector in W (as MID_FWD, MID_ADJ) and its correlation
    // with the vector in W2, both packed real.  From the pair (Z_k, Z_{N-k})
    // of a packed spectrum: E = (Z_k + conj Z_{N-k}) / 2,
    // O = (Z_k - conj Z_{N-k}) / 2i, and the length-2N real spectrum is
    // a^_k = E + w O, a^_{k+N} = E - w O, w = exp(-2 pi i k / 2N).
    constexpr bool ADJ = KIND == MID_ADJ_CORR;
    float2* sm2 = sm + smem_slots(TILE);
    load_tile(sm2, kp.pp.W2);
    fwd_rows(sm2);
    if constexpr (TWS) {
      fwd_rows_from_global();
    } else {
      load_tile(sm, Wi);
      fwd_rows(sm);
    }
    for (int t = threadIdx.x; t < nslots; t += NT) {
      int ea, eb, k2, k1, tidx;
      slot_at(t, ea, eb, k2, k1, tidx);
      const float2 w = phase_at(k2, k1);
      const float4 tab = __ldg(kp.pp.tab_ista + tidx);
      float4 acc = kp.pp.gacc[tidx];
      float2 sp[2][2];   // [W, W2][k, k + N]
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const float2* bufv = v ? sm2 : sm;
        const float2 za = bufv[pad(ea)], zb = bufv[pad(eb)];
        const float2 E = make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y));
        const float2 O = make_float2(0.5f * (za.y + zb.y), -0.5f * (za.x - zb.x));
        const float2 wo = cmul(w, O);
        sp[v][0] = cadd(E, wo);
        sp[v][1] = csub(E, wo);
      }
      // + conj(r^) w^ (W: w, W2: r), - conj(q^) x^ (W: q, W2: x)
      const float sgn = ADJ ? -1.f : 1.f;
      const float2 p0 = ADJ ? cmulc(sp[1][0], sp[0][0]) : cmulc(sp[0][0], sp[1][0]);
      const float2 p1 = ADJ ? cmulc(sp[1][1], sp[0][1]) : cmulc(sp[0][1], sp[1][1]);
      acc.x = fmaf(sgn, p0.x, acc.x);
      acc.y = fmaf(sgn, p0.y, acc.y);
      acc.z = fmaf(sgn, p1.x, acc.z);
      acc.w = fmaf(sgn, p1.y, acc.w);
      kp.pp.gacc[tidx] = acc;
      float2 za = sm[pad(ea)], zb = sm[pad(eb)];
      op_real<ADJ>(tab, w, za, zb);
      sm[pad(eb)] = zb;   // self-pairs (ea == eb) keep the k-side value
      sm[pad(ea)] = za;
    }
    __syncthreads();
  } else if constexpr (KIND == MID_ADMM_REV) {
    // Reverse of the x-update of one Algorithm 3 iteration.  W holds the
    // column transform of p' + i x', W2 that of the iteration's forward pair
    // v + i (z - nu).  Per pair slot, with the k-side spectra P', X'l, V0, Wf
    // of the four real vectors: Xs = bhat (rho chat V0 + sigma Wf) and
    // Bs = bhat (chat P' + X'l) are the spectra of x and b' = B (C^T p' + x')
    // divided by N (bhat holds 1/N).  The spectrum of this iteration's dL/dc
    // divided by N,
    //   A = conj(P') Xs + rho conj(V0) Bs - 2 rho N chat Re(conj(Xs) Bs),
    // is added to gacc_a (DFT of sum_i a_i b_{i+k} = conj(a^) b^; the B-term
    // pairs C x with b' and C b' with x, whose sum is real times chat), and
    // Bs + i conj(chat) Bs goes back for the inverse: b' + i C b'.
    float2* sm2 = sm + smem_slots(TILE);
    load_tile(sm, Wi);
    fwd_rows(sm);
    load_tile(sm2, kp.pp.W2);
    fwd_rows(sm2);
    const float rho = kp.ca->rho, sigma = kp.ca->sigma;
    const float nN = (float)g.N;
    for (int t = threadIdx.x; t < nslots; t += NT) {
      int ea, eb, k2, k1, tidx;
      slot_at(t, ea, eb, k2, k1, tidx);
      const float2 za = sm[pad(ea)], zb = sm[pad(eb)];
      const float2 fa = sm2[pad(ea)], fb = sm2[pad(eb)];
      const float2 Pb = make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y));
      const float2 Xl = make_float2(0.5f * (za.y + zb.y), -0.5f * (za.x - zb.x));
      const float2 V0 = make_float2(0.5f * (fa.x + fb.x), 0.5f * (fa.y - fb.y));
      const float2 Wf = make_float2(0.5f * (fa.y + fb.y), -0.5f * (fa.x - fb.x));
      const float2 ch = __ldg(kp.pp.tab_admm_c + tidx);
      const float bb = __ldg(kp.pp.tab_admm_b + tidx);
      const float2 cv = cmul(ch, V0);
      const float2 Xs = make_float2(bb * fmaf(rho, cv.x, sigma * Wf.x), bb * fmaf(rho, cv.y, sigma * Wf.y));
      const float2 cp = cmul(ch, Pb);
      const float2 Bs = make_float2(bb * (cp.x + Xl.x), bb * (cp.y + Xl.y));
      const float2 t1 = cmulc(Xs, Pb);
      const float2 t2 = cmulc(Bs, V0);
      const float sc = -2.f * rho * nN * fmaf(Xs.x, Bs.x, Xs.y * Bs.y);
      const float2 acc = kp.pp.gacc_a[tidx];
      kp.pp.gacc_a[tidx] = make_float2(acc.x + fmaf(rho, t2.x, fmaf(sc, ch.x, t1.x)),
                                       acc.y + fmaf(rho, t2.y, fmaf(sc, ch.y, t1.y)));
      const float2 Pc = cmulc(Bs, ch);
      sm[pad(eb)] = make_float2(Bs.x + Pc.y, Pc.x - Bs.y);   // self-pairs keep the k-side value
      sm[pad(ea)] = make_float2(Bs.x - Pc.y, Bs.y + Pc.x);
    }
    __syncthreads();
  } else if constexpr (KIND == MID_ADMM_FROM_ACC) {
    // dL/dc = the inverse transform of the accumulated Hermitian spectrum
    for (int t = threadIdx.x; t < nslots; t += NT) {
      int ea, eb, k2, k1, tidx;
      slot_at(t, ea, eb, k2, k1, tidx);
      const float2 A = kp.pp.gacc_a[tidx];
      sm[pad(eb)] = cconj(A);
      sm[pad(ea)] = A;
    }
    __syncthreads();
  } else if constexpr (KIND == MID_FROM_ACC) {
    // The packed spectrum of the real vector d whose length-2N spectrum is
    // gacc (D_k, D_{k+N} per slot), times tau / N for the unnormalised
    // inverse:  E' = (D_k + D_{k+N}) / 2,  O' = conj(w) (D_k - D_{k+N}) / 2,
    // Z'_k = E' + i O',  Z'_{N-k} = conj(E') + i conj(O').
    const float sc = kp.ca->tau / (float)g.N;
    for (int t = threadIdx.x; t < nslots; t += NT) {
      int ea, eb, k2, k1, tidx;
      slot_at(t, ea, eb, k2, k1, tidx);
      const float2 w = cmul(__ldg(g.twr + k2), __ldg(g.tw1 + k1));
      const float4 d = kp.pp.gacc[tidx];
      const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
      const float2 E = cscale(cadd(d0, d1), 0.5f);
      const float2 O = cscale(cmulc(csub(d0, d1), w), 0.5f);
      const float2 za = make_float2(E.x - O.y, E.y + O.x);
      const float2 zb = make_float2(E.x + O.y, O.x - E.y);
      sm[pad(eb)] = cscale(zb, sc);   // self-pairs (ea == eb): both sides agree
      sm[pad(ea)] = cscale(za, sc);
    }
    __syncthreads();
  } else {
    if constexpr (TWS) {
      fwd_rows_from_global();
    } else {
      load_tile(sm, Wi);
      fwd_rows(sm);
    }
    // spectrum operator over all (k, N-k) pairs held by this CTA (unrolled so
    // that the table loads of several slots are in flight together)
    if constexpr (PRET) {
#pragma unroll
      for (int i = 0; i < SL; ++i) {
        int ea, eb, k2, k1, tidx;
        slot_at(threadIdx.x + i * NT, ea, eb, k2, k1, tidx);
        float2 za = sm[pad(ea)], zb = sm[pad(eb)];
        if (KIND == MID_ADMM) op_admm(pw[i], pt[i].x, a_rho, a_sigma, za, zb);
        else op_real<KIND == MID_ADJ>(pt[i], pw[i], za, zb);
        sm[pad(eb)] = zb;   // self-pairs (ea == eb) keep the k-side value
        sm[pad(ea)] = za;
      }
    }
    // (radix-8 tiles: only unit 0's one or two extra slots remain)
#pragma unroll 8
    for (int t = threadIdx.x + (PRET ? (U << lgN1) : 0); t < nslots; t += NT) {
      int ea, eb, k2, k1, tidx;
      slot_at(t, ea, eb, k2, k1, tidx);
      float2 za = sm[pad(ea)], zb = sm[pad(eb)];
      if (KIND == MID_ADMM) {
        op_admm(__ldg(kp.pp.tab_admm_c + tidx), __ldg(kp.pp.tab_admm_b + tidx), a_rho, a_sigma, za, zb);
      } else {
        op_real<KIND == MID_ADJ>(__ldg(kp.pp.tab_ista + tidx), phase_at(k2, k1), za, zb);
      }
      sm[pad(eb)] = zb;   // self-pairs (ea == eb) keep the k-side value
      sm[pad(ea)] = za;
    }
    __syncthreads();
  }
  if constexpr (TWS) {
    // static shapes: the last inverse stage writes the rows to W itself
    const MidIO io{W, u0, lgN1, g.N2};
    if constexpr (TWOD) {
      NoHook nh;
      tile_fft<+1, TILE, NT, true>(sm, lay, tws, lgN1, nh, SmemIO{}, io);
    } else {
      MidTwHookS<false, LOB> h{lohi, lohi + (ROWS << LOB), LGN1S, make_float2(1.f, 0.f)};
      tile_fft<+1, TILE, NT, true>(sm, lay, tws, lgN1, h, SmemIO{}, io);
    }
    return;
  } else {
    if constexpr (TWOD) {
      tile_fft<+1, TILE, NT, false>(sm, lay, g.tw1h, lgN1);
    } else {
      MidTwHook<false> h{g, u0, rt[1], make_float2(1.f, 0.f)};
      tile_fft<+1, TILE, NT, false>(sm, lay, g.tw1, lgN1 + 1, h);
    }
  }

#pragma unroll
  for (int i = 0; i < NLD; ++i) {
    const int e = 2 * (threadIdx.x + i * NT);
    if (e < tot) {
      const int slot = e >> lgN1, j1 = e & (N1 - 1);
      const int k2 = slot_row(g, u0 + (slot >> 1), slot & 1);
      const float2 lo = sm[pad(e)], hi = sm[pad(e + 1)];
      __stcg(reinterpret_cast<float4*>(W + ((size_t)k2 << lgN1) + j1), make_float4(lo.x, lo.y, hi.x, hi.y));
    }
  }
}

template <int KIND, int TILE, int SHAPE>
__global__ void __launch_bounds__(Cfg<TILE, MidShape<SHAPE>::kVpt>::NT, Cfg<TILE, MidShape<SHAPE>::kVpt>::MINB)
    mid_kernel(const KParams kp) {
  mid_body<KIND, TILE, SHAPE>(kp, blockIdx.x);
}

}  // namespace

#define CS_MID_KINDS(X, T, S)                                                                    \
  X(MID_FWD, T, S) X(MID_ADJ, T, S) X(MID_ADMM, T, S) X(MID_FWD_CORR, T, S) X(MID_ADJ_CORR, T, S) X(MID_FROM_ACC, T, S)       \
  X(MID_ADMM_REV, T, S) X(MID_ADMM_FROM_ACC, T, S)
#define CS_MID_KINDS_2D(X, T, S) X(MID_FWD, T, S) X(MID_ADJ, T, S) X(MID_ADMM, T, S)

// the reverse passes that correlate hold two tiles in shared memory
constexpr int mid_smem_mult(int kind) {
  return (kind == MID_FWD_CORR || kind == MID_ADJ_CORR || kind == MID_ADMM_REV) ? 2 : 1;
}

}  // namespace csk
