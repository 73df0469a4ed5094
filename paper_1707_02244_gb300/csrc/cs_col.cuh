// Column pass of the fused FFT iteration: inverse length-N2 FFTs down G
// columns of the N2 x N1 exchange array, the method's elementwise step
// (residual on the kept rows, soft threshold, ADMM updates) as the hook of
// the last inverse stage, then the forward FFTs of the next product.
// Included by cs_col.cu (run-time and large static shapes) and cs_col8*.cu
// (radix-8 shapes), one translation unit each so that they compile in
// parallel.
#pragma once

#include "cs_passes.cuh"

namespace csk {

namespace {

// ---------------------------------------------------------------- column pass

// The column pass uses 4096-value tiles (4 CTAs per SM; 1D: N2 <= 1024
// gives G >= 4 columns), and 16384-value tiles of four 4096-long columns for
// 2D arrays of 4096 rows (1 CTA per SM): four columns make each row of the
// exchange buffer a full 32-byte sector (two would use half of it).
constexpr int COL_TILE = 4096;
constexpr int COL_MINB = 4;
constexpr int COL_TILE4 = 16384;
constexpr int COL_MINB4 = 1;
// 2048-long columns (2D) the same way: 8192-value tiles of four, 2 CTAs per SM
// (run-time shapes of two columns used half of each sector: 2048 x 2048 image,
// 10 + 10 iterations, 2.40 ms, now 1.48 with the other static shapes).
constexpr int COL_TILE2 = 8192;
constexpr int COL_MINB2 = 2;

// Epilogue as the post hook of the inverse column FFT: runs on each value as
// the last stage produces it, so the elementwise step costs no extra pass
// over shared memory.
// NPRE > 0: the epilogue's inputs of the thread's NPRE elements were loaded
// ahead (in the order of the last stage's butterflies and slots).
template <int KIND, int NPRE = 0, int RLAST = 1>
struct EpiHook {
  static constexpr bool kPre = false, kPost = true;
  using E = Epi<KIND>;
  const KParams& kp;
  const CallArgs& a;
  int col0, lgN1;
  Acc& acc;
  int tbase;   // tile-order index of this CTA's first element: col0 * N2
  int lgG;
  int bi = 0;
  typename PreOf<E>::T q[NPRE ? NPRE : 1];
  __device__ __forceinline__ void begin(int, int, int i) { bi = i; }
  __device__ __forceinline__ float2 pre(int, int, int, int, float2 v) const { return v; }
  __device__ __forceinline__ float2 post(int vec, int j, int r, int lgLR, float2 v) {
    const int idx = j + (r << lgLR);
    const int p = col0 + vec + (idx << lgN1), t = tbase + (idx << lgG) + vec;
    if constexpr (HasPre<E>::value) {
      if constexpr (NPRE > 0) return E::apply(kp, a, v, p, t, acc, q[bi * RLAST + r]);
      else return E::apply(kp, a, v, p, t, acc, E::load(kp, a, p, t, acc));
    } else {
      return E::apply(kp, a, v, p, t, acc);
    }
  }
};

// SHAPE 0: any geometry (shape read at run time); SHAPE 1: N2 = 1024 and
// G = 4 columns, the geometry of every N >= 2^20, fixed at compile time.
// SHAPE 10 + LGN2 (LGN2 = 5 .. 9): radix-8 tiles of 4 columns (8 for
// LGN2 = 5), 8 values per thread.
// SHAPE 40 + LGN2 (LGN2 = 6 .. 10): 4096-value tiles, 16 values per thread
// (grouped launches).
template <int SHAPE> struct ColShape {
  static_assert((SHAPE >= 15 && SHAPE <= 19) || (SHAPE >= 46 && SHAPE <= 50), "column shapes");
  static constexpr bool kR8 = SHAPE < 40;
  static constexpr int kLgN2 = SHAPE % (kR8 ? 10 : 40), kLgG = kR8 ? (kLgN2 == 5 ? 3 : 2) : 12 - kLgN2;
  using Lay = StaticLayout<kLgN2, kLgG, true, kR8 ? 3 : 4>;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgG(const Geo&) { return kLgG; }
  __device__ static constexpr int lgN2(const Geo&) { return kLgN2; }
};
template <> struct ColShape<0> {
  using Lay = DynLayout;
  __device__ static Lay lay(const Geo& g) { return Lay{g.lgN2, g.lgG, true}; }
  __device__ static int lgG(const Geo& g) { return g.lgG; }
  __device__ static int lgN2(const Geo& g) { return g.lgN2; }
};
template <> struct ColShape<1> {
  using Lay = StaticLayout<10, 2, true, 4, false>;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgG(const Geo&) { return 2; }
  __device__ static constexpr int lgN2(const Geo&) { return 10; }
};

// SHAPE 3: N2 = 4096 and G = 4, 16384-value tiles (1024 threads).
template <> struct ColShape<3> {
  using Lay = StaticLayout<12, 2, true, 4, false>;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgG(const Geo&) { return 2; }
  __device__ static constexpr int lgN2(const Geo&) { return 12; }
};

// SHAPE 5: N2 = 2048 and G = 4, 8192-value tiles (512 threads).
template <> struct ColShape<5> {
  using Lay = StaticLayout<11, 2, true>;
  __device__ static Lay lay(const Geo&) { return Lay{}; }
  __device__ static constexpr int lgG(const Geo&) { return 2; }
  __device__ static constexpr int lgN2(const Geo&) { return 11; }
};

// Global source / sink of the tile's first and last FFT stages (static
// shapes): element (column c, row j2) of the tile is W[col0 + c + j2 N1].
struct ColIO {
  static constexpr bool kGlobal = true;
  float2* W;
  int col0, lgN1;
  __device__ __forceinline__ float2 load(int c, int j2) const {
    return __ldcg(W + col0 + c + ((size_t)j2 << lgN1));
  }
  __device__ __forceinline__ void store(int c, int j2, float2 v) const {
    __stcg(W + col0 + c + ((size_t)j2 << lgN1), v);
  }
};

template <int SHAPE> struct ColTile {
  static constexpr bool kR8 = SHAPE >= 10 && SHAPE < 40;
  static constexpr int kVpt = kR8 ? VPT8 : EPT;
  static constexpr int kLgN2 = kR8 ? SHAPE - 10 : SHAPE > 40 ? SHAPE - 40 : SHAPE == 3 ? 12 : SHAPE == 5 ? 11 : 10;   // static shapes
  static constexpr int kTile = kR8 ? (kLgN2 == 5 ? 256 : 4 << kLgN2)
                               : SHAPE == 3 ? COL_TILE4 : SHAPE == 5 ? COL_TILE2 : COL_TILE;
  static constexpr int kMinB = kR8 ? Cfg<kTile, kVpt>::MINB : SHAPE == 3 ? COL_MINB4 : SHAPE == 5 ? COL_MINB2 : COL_MINB;
  static constexpr int kCarve = kR8 ? 0 : kMinB;
  static constexpr int kLgR = kR8 ? 3 : 4;
  static constexpr bool kTwFull = SHAPE != 1 && SHAPE != 3;   // as the shape's layout
};

// The column pass of tile `blk` (columns blk G .. blk G + G - 1).
template <int KIND, int SHAPE>
__device__ __forceinline__ void col_body(const KParams& kp, const int blk) {
  constexpr int TILE = ColTile<SHAPE>::kTile;
  constexpr int NT = Cfg<TILE, ColTile<SHAPE>::kVpt>::NT;
  constexpr int NLD = Cfg<TILE, ColTile<SHAPE>::kVpt>::NLD;
  using E = Epi<KIND>;
  using S = ColShape<SHAPE>;
  extern __shared__ float2 sm[];
  pdl_trigger();
  const Geo& g = kp.geo;
  const int lgG = S::lgG(g), lgN2 = S::lgN2(g);
  const int G = 1 << lgG;
  const int col0 = blk << lgG;
  const int tot = G << lgN2;
  const auto lay = S::lay(g);
  constexpr bool TWS = SHAPE != 0;   // static shape: stage-major twiddles in shared memory
  constexpr int TW_N = TWS ? stage_tw_count(ColTile<SHAPE>::kLgN2, ColTile<SHAPE>::kLgR, ColTile<SHAPE>::kTwFull) : 2;
  __shared__ __align__(16) float2 tws[TW_N];
  const float2* tw = TWS ? tws : g.tw2;
  if (TWS) copy_table<NT>(tws, g.tws2, TW_N);   // plan constant
  // the tile's row-mask and prefix words (plan constants): 2 bits per element
  // in the packed geometry, 1 in complex-n
  constexpr int MB = UsesMask<KIND>::kBits;
  constexpr int MW = MB ? TILE * MB / 32 : 1;
  __shared__ uint32_t smask[MW], spref[MW];
  const int wbase = MB ? (((col0 << lgN2) * MB) >> 5) : 0;
  if (MB) {
    const int words = (tot * MB) >> 5;
    for (int w = threadIdx.x; w < words; w += NT) {
      smask[w] = __ldg(kp.pp.mask + wbase + w);
      spref[w] = __ldg(kp.pp.prefix + wbase + w);
    }
  }
  pdl_wait();                                   // everything below may depend on earlier kernels
  const CallArgs a = *kp.ca;
  float2* W = kp.pp.W;
  const float2* Wi = kp.pp.Wi;   // may be W
  Acc acc;
  acc.zero();
  acc.smask = smask;
  acc.spref = spref;
  acc.wbase = wbase;

  if constexpr (E::kRead && ColTile<SHAPE>::kR8 && HasPre<E>::value) {
    // radix-8 tiles: the epilogue's inputs are loaded ahead of the inverse FFT
    constexpr int LGN2 = ColTile<SHAPE>::kLgN2, LGR = LGN2 % 3 ? LGN2 % 3 : 3, R = 1 << LGR;   // last stage
    EpiHook<KIND, VPT8, R> hook{kp, a, col0, g.lgN1, acc, col0 << lgN2, lgG};
    if (MB) __syncthreads();   // the mask words
#pragma unroll
    for (int i = 0; i < VPT8 / R; ++i) {
      const int b = threadIdx.x + i * NT;
      const int vec = b & ((1 << lgG) - 1), j = b >> lgG;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int idx = j + (r << (LGN2 - LGR));
        hook.q[i * R + r] = E::load(kp, a, col0 + vec + (idx << g.lgN1), (col0 << lgN2) + (idx << lgG) + vec, acc);
      }
    }
    tile_fft<+1, TILE, NT, TWS>(sm, lay, tw, lgN2, hook, ColIO{const_cast<float2*>(Wi), col0, g.lgN1}, SmemIO{});
  } else if constexpr (E::kRead && SHAPE != 0) {
    // static shapes: the first inverse stage reads the exchange buffer itself
    EpiHook<KIND> hook{kp, a, col0, g.lgN1, acc, col0 << lgN2, lgG};
    tile_fft<+1, TILE, NT, TWS>(sm, lay, tw, lgN2, hook, ColIO{const_cast<float2*>(Wi), col0, g.lgN1}, SmemIO{});
  } else if constexpr (E::kRead) {
    float4 buf[NLD];
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = 2 * (threadIdx.x + i * NT);
      if (e < tot) {
        const int j2 = e >> lgG, c = e & (G - 1);
        buf[i] = __ldcg(reinterpret_cast<const float4*>(Wi + col0 + c + ((size_t)j2 << g.lgN1)));
      }
    }
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = 2 * (threadIdx.x + i * NT);
      if (e < tot) {
        sm[pad(e)] = make_float2(buf[i].x, buf[i].y);
        sm[pad(e + 1)] = make_float2(buf[i].z, buf[i].w);
      }
    }
    __syncthreads();
    EpiHook<KIND> hook{kp, a, col0, g.lgN1, acc, col0 << lgN2, lgG};
    tile_fft<+1, TILE, NT, TWS>(sm, lay, tw, lgN2, hook);
  } else {
    for (int e = threadIdx.x; e < tot; e += NT) {
      const int j2 = e >> lgG, c = e & (G - 1);
      sm[pad(e)] = E::apply(kp, a, make_float2(0.f, 0.f), col0 + c + (j2 << g.lgN1), (col0 << lgN2) + e, acc);
    }
    __syncthreads();
  }
  if constexpr (KIND == COL_GRAD_W || KIND == COL_GRAD_GW || KIND == COL_ADMM_REV) block_accum<NT>(acc.v[0], kp.pp.gpart, blk);
  if (kp.flags & FL_STATS) {
    constexpr int kSlots =
        KIND == COL_RESIDUAL ? (1 << ST_R2)
        : KIND == COL_POWER_OUT ? ((1 << ST_DX2) | (1 << ST_X2))
        : (KIND == COL_ISTA || KIND == COL_ISTA_LAST)
            ? ((1 << ST_ERR2) | (1 << ST_DX2) | (1 << ST_X2) | (1 << ST_L1) | (1 << ST_NONFIN))
        : (KIND == COL_ADMM || KIND == COL_ADMM_LAST) ? ((1 << ST_ERR2) | (1 << ST_DX2) | (1 << ST_X2) |
                                                         (1 << ST_L1) | (1 << ST_R2) | (1 << ST_NONFIN))
        : 0;
    if (kSlots) block_stats<kSlots, NT>(acc, kp.pp.partials, blk);
  }
  if constexpr (E::kFwd && SHAPE != 0) {
    // static shapes: the last forward stage writes the exchange buffer itself
    NoHook nh;
    tile_fft<-1, TILE, NT, TWS>(sm, lay, tw, lgN2, nh, SmemIO{}, ColIO{W, col0, g.lgN1});
  } else if constexpr (E::kFwd) {
    tile_fft<-1, TILE, NT, TWS>(sm, lay, tw, lgN2);
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = 2 * (threadIdx.x + i * NT);
      if (e < tot) {
        const int j2 = e >> lgG, c = e & (G - 1);
        const float2 lo = sm[pad(e)], hi = sm[pad(e + 1)];
        __stcg(reinterpret_cast<float4*>(W + col0 + c + ((size_t)j2 << g.lgN1)),
               make_float4(lo.x, lo.y, hi.x, hi.y));
      }
    }
  }
}

template <int KIND, int SHAPE>
__global__ void __launch_bounds__(ColTile<SHAPE>::kTile / ColTile<SHAPE>::kVpt, ColTile<SHAPE>::kMinB) col_kernel(const KParams kp) {
  col_body<KIND, SHAPE>(kp, blockIdx.x);
}

}  // namespace

// kinds of the 2D solves (no gradient)
#define CS_COL_KINDS_2D(X, S)                                                                  \
  X(COL_LOAD, S) X(COL_LOAD_SCALED, S) X(COL_STORE, S) X(COL_MASK, S) X(COL_RESIDUAL, S)         \
  X(COL_ISTA, S) X(COL_ISTA_LAST, S) X(COL_POWER_OUT, S) X(COL_ADMM_INIT, S) X(COL_ADMM, S)       \
  X(COL_ADMM_LAST, S)

#define CS_COL_KINDS(X, S)                                                                     \
  X(COL_LOAD, S) X(COL_LOAD_SCALED, S) X(COL_STORE, S) X(COL_MASK, S) X(COL_RESIDUAL, S)         \
  X(COL_ISTA, S) X(COL_ISTA_LAST, S) X(COL_POWER_OUT, S) X(COL_ADMM_INIT, S) X(COL_ADMM, S)       \
  X(COL_ADMM_LAST, S) X(COL_LOADT, S) X(COL_ISTA_SEG, S) X(COL_GRAD_W, S)           \
  X(COL_GRAD_MASK, S) X(COL_GRAD_G, S) X(COL_GRAD_GW, S) X(COL_ADMM_SEG, S) X(COL_ADMM_REV, S) X(COL_STORE_RE, S)

}  // namespace csk
