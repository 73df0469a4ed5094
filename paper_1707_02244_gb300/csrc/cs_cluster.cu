// Whole solves and products of one instance of middle size (ISTA n = 2^14 and
// 2^15, ADMM n = 2^13 .. 2^15) by one cluster of 16 CTAs in one launch.
//
// The transform is the passes' four-step split, N = N1 x N2, but the exchange
// array lives in the CTAs' shared memory: CTA c holds N1/16 columns (column
// phase) and N2/16 rows as row pairs (row phase).  The last stage of each
// phase stores its outputs straight into the shared memory of the CTA that
// needs them next (st.shared::cluster), and a cluster barrier takes the place
// of the launch boundary: two per product.  The solver's state stays in
// registers for all iterations, 8 elements per thread.
//
// A pass of these lengths is bound by its latency: launch gap, the round trip
// of W, x and y through L2, table fills.  Here an exchange costs the SM-to-SM
// latency and one fence, and tables are filled once per solve.  Measured, us
// an iteration, passes -> cluster: ADMM n = 2^13 5.7 -> 3.5, 2^14 6.5 -> 4.8,
// 2^15 6.7 -> 5.8, 2^16 7.1 -> 14.6; ISTA 2^14 11.4 -> 9.2, 2^15 12.2 -> 11.3,
// 2^16 11.9 -> 17.0: beyond 2048 values a CTA the exchange through 16 SMs is
// slower than the passes on all of them, so the lengths end there.  At
// n = 2^15 an ADMM iteration issues in 31 % of its cycles; the fence of the
// cluster barrier waits for the remote stores (20 % of the stalls).
#include "cs_mid.cuh"

namespace csk {

namespace {

constexpr int CL_LG = 4, CL = 1 << CL_LG;   // CTAs per cluster (non-portable size)

template <int LGN> struct ClShape {
  static constexpr int kLgN2 = LGN / 2, kLgN1 = LGN - kLgN2;   // as make_geo
  static constexpr int kLgG = kLgN1 - CL_LG;                   // columns per CTA
  static constexpr int kLgRows = kLgN2 - CL_LG;                // rows per CTA (two per unit)
  static constexpr int T = 1 << (LGN - CL_LG), NT = T / VPT8;
  using ColLay = LoopLayout<StaticLayout<kLgN2, kLgG, true, 3>>;
  using RowLay = LoopLayout<StaticLayout<kLgN1, kLgRows, false, 3>>;
  static constexpr int kLob = kLgN1 - 3 < 4 ? kLgN1 - 3 : 4;
  static constexpr int kTw1 = stage_tw_count(kLgN1, 3, true), kTw2 = stage_tw_count(kLgN2, 3, true);
  static constexpr int kLo = 1 << kLob, kHi = 1 << (kLgN1 - kLob);
  static constexpr int kLohi = (1 << kLgRows) * (kLo + kHi);
  // float2 of dynamic shared memory: FFT scratch, row and column inputs, tables
  static constexpr int kSmem = T + T / 16 + 2 * T + kTw1 + kTw2 + kLohi;
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t remote_addr(uint32_t a, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// Column phase: inputs from this CTA's column buffer; outputs (row k2 of
// column c) to the row buffer of the CTA that holds row k2.
template <int LGN> struct ClColIn {
  static constexpr bool kGlobal = true;
  const float2* cb;
  __device__ __forceinline__ float2 load(int c, int j2) const { return cb[(j2 << ClShape<LGN>::kLgG) + c]; }
};
template <int LGN> struct ClColOut {
  static constexpr bool kGlobal = true;
  uint32_t rb;   // shared address of the row buffer
  int col0;
  __device__ __forceinline__ void store(int c, int k2, float2 v) const {
    using S = ClShape<LGN>;
    constexpr int N2 = 1 << S::kLgN2;
    // row k2 is the first (k2 < N2/2) or second row of unit min(k2, N2 - k2);
    // row N2/2 is the second of unit 0
    const int second = k2 >= N2 / 2, u = second ? (N2 - k2) & (N2 / 2 - 1) : k2;
    const int slot = 2 * u + second;
    const int rank = slot >> S::kLgRows, vec = slot & ((1 << S::kLgRows) - 1);
    st_remote(remote_addr(rb + (uint32_t)sizeof(float2) * ((vec << S::kLgN1) + col0 + c), rank), v);
  }
};
template <int LGN> struct ClRowIn {
  static constexpr bool kGlobal = true;
  const float2* rb;
  __device__ __forceinline__ float2 load(int vec, int j) const { return rb[(vec << ClShape<LGN>::kLgN1) + j]; }
};
template <int LGN> struct ClRowOut {
  static constexpr bool kGlobal = true;
  uint32_t cb;
  int slot0;   // first row slot of this CTA
  __device__ __forceinline__ void store(int vec, int j1, float2 v) const {
    using S = ClShape<LGN>;
    constexpr int N2 = 1 << S::kLgN2;
    const int slot = slot0 + vec, u = slot >> 1;
    const int k2 = (slot & 1) ? (u == 0 ? N2 / 2 : N2 - u) : u;
    const int rank = j1 >> S::kLgG, c = j1 & ((1 << S::kLgG) - 1);
    st_remote(remote_addr(cb + (uint32_t)sizeof(float2) * ((k2 << S::kLgG) + c), rank), v);
  }
};

// Elements of this thread after the last inverse column stage, in the order
// of its butterflies and slots: spatial index p of element i.
template <int LGN>
__device__ __forceinline__ int cl_elem(int i, int col0) {
  using S = ClShape<LGN>;
  constexpr int LGR = S::kLgN2 % 3 ? S::kLgN2 % 3 : 3, R = 1 << LGR;
  const int b = threadIdx.x + (i / R) * S::NT;
  const int c = b & ((1 << S::kLgG) - 1), j2 = (b >> S::kLgG) + ((i % R) << (S::kLgN2 - LGR));
  return col0 + c + (j2 << S::kLgN1);
}
// ... and its place in the padded scratch tile.
template <int LGN>
__device__ __forceinline__ int cl_slot(int p, int col0) {
  using S = ClShape<LGN>;
  return pad(((p >> S::kLgN1) << S::kLgG) + (p & ((1 << S::kLgN1) - 1)) - col0);
}

// Hook of the last inverse stage: f(i, value) for the thread's element i.
template <int R, class F> struct ClEpi {
  static constexpr bool kPre = false, kPost = true;
  F& f;
  int bi = 0;
  __device__ __forceinline__ void begin(int, int, int i) { bi = i; }
  __device__ __forceinline__ float2 pre(int, int, int, int, float2 v) const { return v; }
  __device__ __forceinline__ float2 post(int, int, int r, int, float2 v) { return f(bi * R + r, v); }
};

template <int LGN> struct ClCtx {
  float2 *sm, *rb, *cb, *tw1, *tw2, *lohi;
  int rank, col0;
  const volatile int* zero;   // see LoopLayout
};

template <int LGN>
__device__ __forceinline__ ClCtx<LGN> cl_begin(const ClusterArgs& a, float2* base) {
  using S = ClShape<LGN>;
  const Geo& g = a.geo;
  __shared__ int zero;
  if (threadIdx.x == 0) zero = 0;   // read behind the first barrier
  ClCtx<LGN> x;
  x.zero = &zero;
  x.sm = base;
  x.rb = x.sm + S::T + S::T / 16;
  x.cb = x.rb + S::T;
  x.tw1 = x.cb + S::T;
  x.tw2 = x.tw1 + S::kTw1;
  x.lohi = x.tw2 + S::kTw2;
  x.rank = blockIdx.x;   // one cluster per grid
  x.col0 = x.rank << S::kLgG;
  copy_table<S::NT>(x.tw1, g.tws1, S::kTw1);
  copy_table<S::NT>(x.tw2, g.tws2, S::kTw2);
  for (int t = threadIdx.x; t < S::kLohi; t += S::NT) {
    constexpr int NLO = (1 << S::kLgRows) * S::kLo;
    const bool is_lo = t < NLO;
    const int tt = is_lo ? t : t - NLO;
    const int vec = is_lo ? tt / S::kLo : tt / S::kHi;
    const int q = is_lo ? tt % S::kLo : (tt % S::kHi) << S::kLob;
    const int slot = (x.rank << S::kLgRows) + vec;
    // one rounded value (the passes' tw4 is a product of two): the 128-point
    // transforms have a stage more here than radix 16 gives them, and with tw4
    // an ADMM solve at n = 2^14, 2^15 rounded 3 % more than by the passes
    x.lohi[t] = __ldg(a.twn + ((q * slot_row(g, slot >> 1, slot & 1)) & (g.N - 1)));
  }
  return x;
}

// Pair slots of this CTA's rows: as the mid pass (t < U N1, unit u0 + t / N1;
// CTA 0 has one more).
template <int LGN>
__device__ __forceinline__ void cl_pair(int t, int u0, int& ea, int& eb, int& k2, int& k1, int& tidx) {
  using S = ClShape<LGN>;
  constexpr int N1 = 1 << S::kLgN1, N2 = 1 << S::kLgN2, UN = 1 << (S::kLgRows - 1 + S::kLgN1);
  const int ul = t < UN ? t >> S::kLgN1 : 0, q = t < UN ? t & (N1 - 1) : N1 + t - UN;
  const int u = u0 + ul;
  if (u > 0) {
    k2 = u;
    k1 = q;
    ea = 2 * ul * N1 + q;
    eb = (2 * ul + 1) * N1 + N1 - 1 - q;
    tidx = (u - 1) * N1 + q;
  } else {
    const bool hi = q > N1 / 2;
    const int qq = hi ? q - N1 / 2 - 1 : q;
    k2 = hi ? N2 / 2 : 0;
    k1 = qq;
    ea = (hi ? N1 : 0) + qq;
    eb = hi ? 2 * N1 - 1 - qq : (N1 - qq) & (N1 - 1);
    tidx = (N2 / 2 - 1) * N1 + q;
  }
}

// Row phase: forward FFTs of the rows, op(i, k2, k1, tidx, za, zb) on the
// pairs (i: the thread's pair number, 4 for the extra slot), inverse FFTs, to
// the column buffers.
template <int LGN, class OP>
__device__ __forceinline__ void cl_rows(const ClCtx<LGN>& x, const OP& op) {
  using S = ClShape<LGN>;
  constexpr int NLO = (1 << S::kLgRows) * S::kLo;
  const int z = *x.zero;
  const typename S::RowLay lay(z);
  MidTwHookS<true, S::kLob> hf{x.lohi, x.lohi + NLO, S::kLgN1, make_float2(1.f, 0.f)};
  tile_fft<-1, S::T, S::NT, true>(x.sm, lay, x.tw1, S::kLgN1, hf, ClRowIn<LGN>{x.rb}, SmemIO{});
  const int u0 = x.rank << (S::kLgRows - 1), t0 = threadIdx.x + z;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int ea, eb, k2, k1, tidx;
    cl_pair<LGN>(t0 + i * S::NT, u0, ea, eb, k2, k1, tidx);
    float2 za = x.sm[pad(ea)], zb = x.sm[pad(eb)];
    op(i, k2, k1, tidx, za, zb);
    x.sm[pad(eb)] = zb;   // self-pairs (ea == eb) keep the k-side value
    x.sm[pad(ea)] = za;
  }
  if (x.rank == 0 && threadIdx.x == 0) {
    int ea, eb, k2, k1, tidx;
    cl_pair<LGN>(4 * S::NT + z, u0, ea, eb, k2, k1, tidx);
    float2 za = x.sm[pad(ea)], zb = x.sm[pad(eb)];
    op(4, k2, k1, tidx, za, zb);
    x.sm[pad(eb)] = zb;
    x.sm[pad(ea)] = za;
  }
  __syncthreads();
  MidTwHookS<false, S::kLob> hi{x.lohi, x.lohi + NLO, S::kLgN1, make_float2(1.f, 0.f)};
  tile_fft<+1, S::T, S::NT, true>(x.sm, lay, x.tw1, S::kLgN1, hi, SmemIO{},
                                  ClRowOut<LGN>{smem_addr(x.cb), x.rank << S::kLgRows});
}

// Inverse column FFTs with f(i, value) on the thread's elements; the results
// f returns are left in the scratch tile.
template <int LGN, class F>
__device__ __forceinline__ void cl_cols_inv(const ClCtx<LGN>& x, F&& f) {
  using S = ClShape<LGN>;
  constexpr int R = S::kLgN2 % 3 ? 1 << (S::kLgN2 % 3) : 8;
  const typename S::ColLay lay(*x.zero);
  ClEpi<R, F> h{f};
  tile_fft<+1, S::T, S::NT, true>(x.sm, lay, x.tw2, S::kLgN2, h, ClColIn<LGN>{x.cb}, SmemIO{});
}
// Forward column FFTs of the scratch tile, to the row buffers.
template <int LGN>
__device__ __forceinline__ void cl_cols_fwd(const ClCtx<LGN>& x) {
  using S = ClShape<LGN>;
  const typename S::ColLay lay(*x.zero);
  NoHook nh;
  tile_fft<-1, S::T, S::NT, true>(x.sm, lay, x.tw2, S::kLgN2, nh, SmemIO{}, ClColOut<LGN>{smem_addr(x.rb), x.col0});
}

// The real product's operator, its table entries and phases of the thread's
// pairs kept in registers for the whole launch.
template <int LGN> struct ClOpReal {
  float4 pt[4];
  float2 pw[4];
  __device__ __forceinline__ void load(const ClusterArgs& a, int rank) {
    using S = ClShape<LGN>;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int ea, eb, k2, k1, tidx;
      cl_pair<LGN>(threadIdx.x + i * S::NT, rank << (S::kLgRows - 1), ea, eb, k2, k1, tidx);
      pt[i] = __ldg(a.tab_i + tidx);
      pw[i] = cmul(__ldg(a.geo.twr + k2), __ldg(a.geo.tw1 + k1));
    }
  }
  template <bool ADJ>
  __device__ __forceinline__ void op(const ClusterArgs& a, int i, int k2, int k1, int tidx, float2& za,
                                     float2& zb) const {
    if (i < 4) op_real<ADJ>(pt[i & 3], pw[i & 3], za, zb);
    else op_real<ADJ>(__ldg(a.tab_i + tidx), cmul(__ldg(a.geo.twr + k2), __ldg(a.geo.tw1 + k1)), za, zb);
  }
};

__device__ __forceinline__ int plan_tile(const Geo& g, int p) {   // spatial index -> the plan's tile order
  const int j1 = p & (g.N1 - 1), j2 = p >> g.lgN1;
  return ((j1 >> g.lgG) << (g.lgG + g.lgN2)) + (j2 << g.lgG) + (j1 & (g.G - 1));
}

constexpr int CL_SLOTS_ISTA = (1 << ST_ERR2) | (1 << ST_DX2) | (1 << ST_X2) | (1 << ST_L1) | (1 << ST_R2) |
                              (1 << ST_NONFIN);

template <int LGN>
__global__ void __launch_bounds__(ClShape<LGN>::NT, 1) cluster_ista_k(const ClusterArgs a) {
  using S = ClShape<LGN>;
  extern __shared__ float2 smem[];
  const ClCtx<LGN> x = cl_begin<LGN>(a, smem);
  ClOpReal<LGN> tab;
  tab.load(a, x.rank);
  // the thread's elements: x, the kept rows' y
  float2 xv[VPT8], yv[VPT8];
  uint32_t mb = 0;
  float2* xg = reinterpret_cast<float2*>(a.x);
  RowSel rs{a.mask, a.prefix, 0};
#pragma unroll
  for (int i = 0; i < VPT8; ++i) {
    const int p = cl_elem<LGN>(i, x.col0);
    xv[i] = xg[p];
    int i0;
    const uint32_t mm = rs.get2(plan_tile(a.geo, p), i0);
    yv[i].x = (mm & 1u) ? __ldg(a.ys + i0) : 0.f;
    yv[i].y = (mm & 2u) ? __ldg(a.ys + i0 + (int)(mm & 1u)) : 0.f;
    mb |= mm << (2 * i);
    x.sm[cl_slot<LGN>(p, x.col0)] = xv[i];
  }
  __syncthreads();
  cluster_sync();   // every CTA of the cluster is running
  cl_cols_fwd<LGN>(x);
  cluster_sync();
  Acc acc;
  acc.zero();
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const bool end = it + 1 == a.iters, st = a.stats && end;
    cl_rows<LGN>(x, [&](int i, int k2, int k1, int ti, float2& za, float2& zb) {
      tab.template op<false>(a, i, k2, k1, ti, za, zb);
    });
    cluster_sync();
    cl_cols_inv<LGN>(x, [&](int i, float2 v) {
      const float r0 = ((mb >> (2 * i)) & 1u) ? yv[i].x - v.x : 0.f;
      const float r1 = ((mb >> (2 * i)) & 2u) ? yv[i].y - v.y : 0.f;
      if (st) acc.v[ST_R2] = fmaf(r0, r0, fmaf(r1, r1, acc.v[ST_R2]));
      return make_float2(r0, r1);
    });
    cl_cols_fwd<LGN>(x);
    cluster_sync();
    cl_rows<LGN>(x, [&](int i, int k2, int k1, int ti, float2& za, float2& zb) {
      tab.template op<true>(a, i, k2, k1, ti, za, zb);
    });
    cluster_sync();
    cl_cols_inv<LGN>(x, [&](int i, float2 g) {
      const float2 xo = xv[i];
      const float2 xn = make_float2(soft(fmaf(a.tau, g.x, xo.x), a.thr), soft(fmaf(a.tau, g.y, xo.y), a.thr));
      xv[i] = xn;
      if (st) {
        const float d0 = xn.x - xo.x, d1 = xn.y - xo.y;
        acc.v[ST_DX2] = fmaf(d0, d0, fmaf(d1, d1, acc.v[ST_DX2]));
        acc.v[ST_X2] = fmaf(xn.x, xn.x, fmaf(xn.y, xn.y, acc.v[ST_X2]));
        acc.v[ST_L1] += fabsf(xo.x) + fabsf(xo.y);
        if (a.xtrue) {
          const float2 xs = ld2(a.xtrue, plan_tile(a.geo, cl_elem<LGN>(i, x.col0 + *x.zero)));
          const float e0 = xn.x - xs.x, e1 = xn.y - xs.y;
          acc.v[ST_ERR2] = fmaf(e0, e0, fmaf(e1, e1, acc.v[ST_ERR2]));
        }
        if (!isfinite(xn.x) || !isfinite(xn.y)) acc.v[ST_NONFIN] += 1.f;
      }
      return xn;
    });
    if (!end) {
      cl_cols_fwd<LGN>(x);
      cluster_sync();
    }
  }
#pragma unroll
  for (int i = 0; i < VPT8; ++i) xg[cl_elem<LGN>(i, x.col0 + *x.zero)] = xv[i];
  if (a.stats) block_stats<CL_SLOTS_ISTA, S::NT>(acc, a.partials, x.rank);
}

template <int LGN>
__global__ void __launch_bounds__(ClShape<LGN>::NT, 1) cluster_admm_k(const ClusterArgs a) {
  using S = ClShape<LGN>;
  extern __shared__ float2 smem[];
  const ClCtx<LGN> x = cl_begin<LGN>(a, smem);
  float2 tc[4];
  float tb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int ea, eb, k2, k1, tidx;
    cl_pair<LGN>(threadIdx.x + i * S::NT, x.rank << (S::kLgRows - 1), ea, eb, k2, k1, tidx);
    tc[i] = __ldg(a.tab_c + tidx);
    tb[i] = __ldg(a.tab_b + tidx);
  }
  float mu[VPT8], nu[VPT8], yv[VPT8];
  uint32_t mb = 0;
  RowSel rs{a.mask, a.prefix, 0};
#pragma unroll
  for (int i = 0; i < VPT8; ++i) {
    const int p = cl_elem<LGN>(i, x.col0);
    int i0;
    const bool on = rs.get(plan_tile(a.geo, p), i0);
    yv[i] = on ? __ldg(a.ys + i0) : 0.f;
    mb |= (on ? 1u : 0u) << i;
    mu[i] = a.warm ? a.mu[p] : 0.f;
    nu[i] = a.warm ? a.nu[p] : 0.f;
    x.sm[cl_slot<LGN>(p, x.col0)] = a.warm ? make_float2(a.v[p], a.z[p] - nu[i]) : make_float2(0.f, 0.f);
  }
  __syncthreads();
  cluster_sync();
  cl_cols_fwd<LGN>(x);
  cluster_sync();
  Acc acc;
  acc.zero();
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const bool end = it + 1 == a.iters, st = a.stats && end;
    cl_rows<LGN>(x, [&](int i, int, int, int ti, float2& za, float2& zb) {
      if (i < 4) op_admm(tc[i & 3], tb[i & 3], a.rho, a.sigma, za, zb);
      else op_admm(__ldg(a.tab_c + ti), __ldg(a.tab_b + ti), a.rho, a.sigma, za, zb);
    });
    cluster_sync();
    cl_cols_inv<LGN>(x, [&](int i, float2 xc) {
      const bool on = (mb >> i) & 1u;
      const float xx = xc.x, cx = xc.y;
      const float v = (on ? a.d_on : a.d_off) * fmaf(a.rho, cx - mu[i], yv[i]);
      const float z = soft(xx + nu[i], a.thr);
      mu[i] = fmaf(a.tau1, v - cx, mu[i]);
      nu[i] = fmaf(a.tau2, xx - z, nu[i]);
      const float vf = v + mu[i];
      if (end) {
        const int p = cl_elem<LGN>(i, x.col0 + *x.zero);
        if (a.z) a.z[p] = z;
        if (a.v) a.v[p] = vf;
        if (a.mu) a.mu[p] = mu[i];
        if (a.nu) a.nu[p] = nu[i];
        if (a.x) a.x[p] = xx;
        if (st) {
          if (a.xtrue) {
            const float e = z - __ldg(a.xtrue + plan_tile(a.geo, p));
            acc.v[ST_ERR2] = fmaf(e, e, acc.v[ST_ERR2]);
          }
          acc.v[ST_DX2] = fmaf(xx - z, xx - z, acc.v[ST_DX2]);
          acc.v[ST_X2] = fmaf(z, z, acc.v[ST_X2]);
          acc.v[ST_L1] += fabsf(z);
          const float r = on ? yv[i] - cx : 0.f;
          acc.v[ST_R2] = fmaf(r, r, acc.v[ST_R2]);
          if (!isfinite(z) || !isfinite(vf)) acc.v[ST_NONFIN] += 1.f;
        }
      }
      return make_float2(vf, z - nu[i]);
    });
    if (!end) {
      cl_cols_fwd<LGN>(x);
      cluster_sync();
    }
  }
  if (a.stats) block_stats<CL_SLOTS_ISTA, S::NT>(acc, a.partials, x.rank);
}

// Power iteration on A^T A from a.x (natural order): stats as the pass form.
template <int LGN>
__global__ void __launch_bounds__(ClShape<LGN>::NT, 1) cluster_power_k(const ClusterArgs a) {
  using S = ClShape<LGN>;
  extern __shared__ float2 smem[];
  __shared__ double red[S::NT / 32][2], part[CL][2], tot[2];
  const ClCtx<LGN> x = cl_begin<LGN>(a, smem);
  ClOpReal<LGN> tab;
  tab.load(a, x.rank);
  float2 w[VPT8], u[VPT8];
  uint32_t mb = 0;
  const float2* xg = reinterpret_cast<const float2*>(a.x);
  RowSel rs{a.mask, a.prefix, 0};
  // sums over the cluster in a fixed order; every CTA gets both
  auto cluster_sum = [&](double s0, double s1) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_down_sync(0xffffffffu, s0, o);
      s1 += __shfl_down_sync(0xffffffffu, s1, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[threadIdx.x >> 5][0] = s0;
      red[threadIdx.x >> 5][1] = s1;
    }
    __syncthreads();
    if (threadIdx.x < CL * 2) {   // thread (rank r, value k) sends this CTA's sum k to CTA r
      const int k = threadIdx.x & 1, r = threadIdx.x >> 1;
      double s = 0.0;
      for (int q = 0; q < S::NT / 32; ++q) s += red[q][k];
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote_addr(smem_addr(&part[x.rank][k]), r)), "d"(s)
                   : "memory");
    }
    cluster_sync();
    if (threadIdx.x < 2) {
      double s = 0.0;
      for (int r = 0; r < CL; ++r) s += part[r][threadIdx.x];
      tot[threadIdx.x] = s;
    }
    __syncthreads();
  };
  double n2 = 0.0;
#pragma unroll
  for (int i = 0; i < VPT8; ++i) {
    const int p = cl_elem<LGN>(i, x.col0);
    w[i] = xg[p];
    int i0;
    mb |= rs.get2(plan_tile(a.geo, p), i0) << (2 * i);
    n2 += (double)w[i].x * w[i].x + (double)w[i].y * w[i].y;
  }
  __syncthreads();
  cluster_sync();   // every CTA is running before the first remote store
  cluster_sum(n2, 0.0);
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const float s = (float)rsqrt(tot[0]);
#pragma unroll
    for (int i = 0; i < VPT8; ++i) {
      u[i] = cscale(w[i], s);
      const int c0 = x.col0 + *x.zero;
      x.sm[cl_slot<LGN>(cl_elem<LGN>(i, c0), c0)] = u[i];
    }
    __syncthreads();
    cl_cols_fwd<LGN>(x);
    cluster_sync();
    cl_rows<LGN>(x, [&](int i, int k2, int k1, int ti, float2& za, float2& zb) {
      tab.template op<false>(a, i, k2, k1, ti, za, zb);
    });
    cluster_sync();
    cl_cols_inv<LGN>(x, [&](int i, float2 v) {
      return make_float2(((mb >> (2 * i)) & 1u) ? v.x : 0.f, ((mb >> (2 * i)) & 2u) ? v.y : 0.f);
    });
    cl_cols_fwd<LGN>(x);
    cluster_sync();
    cl_rows<LGN>(x, [&](int i, int k2, int k1, int ti, float2& za, float2& zb) {
      tab.template op<true>(a, i, k2, k1, ti, za, zb);
    });
    cluster_sync();
    float x2 = 0.f, uw = 0.f;
    cl_cols_inv<LGN>(x, [&](int i, float2 v) {
      w[i] = v;
      x2 = fmaf(v.x, v.x, fmaf(v.y, v.y, x2));
      uw = fmaf(u[i].x, v.x, fmaf(u[i].y, v.y, uw));
      return v;
    });
    cluster_sum((double)x2, (double)uw);
  }
  if (x.rank == 0 && threadIdx.x == 0) {
    a.stats[ST_X2] = tot[0];
    a.stats[ST_DX2] = tot[1];
  }
}

// One product in natural order: a.z = C a.x (ADJ: C^T a.x).
template <int LGN, bool ADJ>
__global__ void __launch_bounds__(ClShape<LGN>::NT, 1) cluster_product_k(const ClusterArgs a) {
  extern __shared__ float2 smem[];
  const ClCtx<LGN> x = cl_begin<LGN>(a, smem);
  ClOpReal<LGN> tab;
  tab.load(a, x.rank);
  const float2* src = reinterpret_cast<const float2*>(a.x);
  float2* dst = reinterpret_cast<float2*>(a.z);
#pragma unroll
  for (int i = 0; i < VPT8; ++i) {
    const int p = cl_elem<LGN>(i, x.col0);
    x.sm[cl_slot<LGN>(p, x.col0)] = src[p];
  }
  __syncthreads();
  cluster_sync();
  cl_cols_fwd<LGN>(x);
  cluster_sync();
  cl_rows<LGN>(x, [&](int i, int k2, int k1, int ti, float2& za, float2& zb) {
    tab.template op<ADJ>(a, i, k2, k1, ti, za, zb);
  });
  cluster_sync();
  cl_cols_inv<LGN>(x, [&](int i, float2 v) {
    dst[cl_elem<LGN>(i, x.col0)] = v;
    return v;
  });
}

template <int LGN>
const void* cluster_kernel(ClusterKind k) {
  if (k == CLUSTER_ADMM) return (const void*)cluster_admm_k<LGN>;
  if constexpr (LGN <= 14) switch (k) {
    case CLUSTER_ISTA: return (const void*)cluster_ista_k<LGN>;
    case CLUSTER_POWER: return (const void*)cluster_power_k<LGN>;
    case CLUSTER_FWD: return (const void*)cluster_product_k<LGN, false>;
    case CLUSTER_ADJ: return (const void*)cluster_product_k<LGN, true>;
    default: break;
  }
  return nullptr;
}

struct ClLaunch {
  const void* fn = nullptr;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
};

template <int LGN>
bool cluster_config(ClusterKind k, ClLaunch& l) {
  l.fn = cluster_kernel<LGN>(k);
  l.cfg.gridDim = dim3(CL);
  l.cfg.blockDim = dim3(ClShape<LGN>::NT);
  l.cfg.dynamicSmemBytes = sizeof(float2) * ClShape<LGN>::kSmem;
  l.attr[0].id = cudaLaunchAttributeClusterDimension;
  l.attr[0].val.clusterDim.x = CL;
  l.attr[0].val.clusterDim.y = 1;
  l.attr[0].val.clusterDim.z = 1;
  l.cfg.attrs = l.attr;
  l.cfg.numAttrs = 1;
  return true;
}

// N = 2^13 and 2^14 for all, 2^15 for ADMM (2048 values a CTA).
bool cluster_config(ClusterKind k, int lgN, ClLaunch& l) {
  switch (lgN) {
    case 13: return cluster_config<13>(k, l);
    case 14: return cluster_config<14>(k, l);
    case 15: return k == CLUSTER_ADMM && cluster_config<15>(k, l);
  }
  return false;
}

}  // namespace

// Whether the device can run one cluster of every kernel of this length, and
// their attributes.  False (and no error left behind) sends the plan's calls
// to the passes.
bool cluster_init(const Geo& g, bool admm) {
  if (!g.col_r8 || !g.mid_r8 || g.twod) return false;
  for (ClusterKind k : {CLUSTER_ISTA, CLUSTER_ADMM, CLUSTER_POWER, CLUSTER_FWD, CLUSTER_ADJ}) {
    if ((k == CLUSTER_ADMM) != admm) continue;
    ClLaunch l;
    if (!cluster_config(k, g.lgN, l)) return false;
    int n = 0;
    if (cudaFuncSetAttribute(l.fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(l.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.cfg.dynamicSmemBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, l.fn, &l.cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return false;
    }
  }
  return true;
}

cudaError_t launch_cluster(ClusterKind kind, const ClusterArgs& a, cudaStream_t s) {
  ClLaunch l;
  if (!cluster_config(kind, a.geo.lgN, l)) return cudaErrorInvalidValue;
  l.cfg.stream = s;
  void* args[] = {const_cast<ClusterArgs*>(&a)};
  return cudaLaunchKernelExC(&l.cfg, l.fn, args);
}

int cluster_ctas() { return CL; }

}  // namespace csk
