// One CTA holds the whole FFT of a short transform: building blocks of the
// solvers for n <= 8192 (cs_small.cu).
//
// N = 2^LG complex values, E per thread, kept in registers between the
// stages.  A product with C is  forward FFT -> operator on the pairs
// (k, N - k) -> inverse FFT, with radices R1 = E first and RL = E/2 last in
// the forward direction and the same in reverse order on the way back:
//   - the last inverse stage leaves elements tid + r N/R1 with thread tid,
//     which are the inputs of its first forward stage, so the solver's
//     element-wise step and the turn to the next product need no exchange;
//   - thread tid runs butterflies j = tid and M - tid (M = N/RL; thread 0:
//     0 and M/2) of the last forward stage.  Output r of butterfly j is
//     frequency j + r M and its mirror is output RL-1-r of butterfly M - j
//     (butterfly 0: RL - r of itself), so both members of every pair are
//     in one thread and the operator and the first inverse stage (the same
//     butterflies) work in registers.
// A product then costs one exchange through shared memory per stage boundary
// that is left: 2 (NS - 1) for NS stages, one barrier each (two buffers).
#pragma once

#include "cs_fft.cuh"

namespace csk {

// Shape of the transform.  8 values per thread up to N = 2048 (more threads
// hide more latency: 4.4 us an ISTA iteration at n = 4096 against 5.7 with
// 16), 16 above (fewer exchanges, and 8 would need a third middle stage).
template <int LG> struct SmallShape {
  static constexpr int kLgE = LG <= 11 ? 3 : 4;
  static constexpr int E = 1 << kLgE;
  static constexpr int N = 1 << LG;
  static constexpr int NA = N / E;                     // threads that hold values
  static constexpr int NT = NA < 32 ? 32 : NA;         // threads launched
  static constexpr int kLg1 = kLgE, kLgL = kLgE - 1;   // first and last forward radix
  static constexpr int kLgM = LG - kLg1 - kLgL;        // what is left for the middle stages
  static constexpr int kLgM1 = kLgM > kLgE ? (kLgM + 1) / 2 : kLgM;
  static constexpr int kLgM2 = kLgM - kLgM1;
  static_assert(kLgM >= 0 && kLgM1 <= kLgE && kLgM2 <= kLgE, "radices");
};

// Twiddle blocks: forward middle 1, middle 2, last; inverse middle 2, middle
// 1, last (radix R1 = 2 RL).
//
// FULL: every twiddle is a table value rounded once.  The two last stages take
// the same roots w_N^(r k), so the inverse one reads the forward one's rows:
// r < RL directly, an even r >= RL as row r / 2 at 2k; its own block holds the
// odd r > RL only (8192-long transforms fit the CTA's shared memory this way).
// Otherwise the higher powers are products of two table values (see
// stage_twiddle).
//
// The batch's size classes take FULL: the solver they replaced did too, and
// with products their ADMM error against 64 bits was 10 to 15 % larger (20
// iterations, n = 1024 .. 8192; ISTA 1 to 2 %), within 2 % with FULL.  50
// iterations of 200 instances each of n = 8192, 4096 and 2048 take 0.93 ms
// (ISTA) and 0.92 ms (ADMM), with products 0.85 and 0.91 ms.
// One instance of a plan takes products: bound by one SM's shared-memory pipe,
// it is 10 % slower with FULL (500 ISTA iterations at n = 4096: 2.04 against
// 2.25 ms), and either way it rounds less than the four-step passes it replaced
// (n = 1024 .. 4096: products 0.79 .. 0.84 of a product's error, ISTA 0.95, ADMM
// 0.9; FULL 0.75 .. 0.80, 0.94, 0.8).
template <int LG, bool FULL> struct SmallTw {
  using S = SmallShape<LG>;
  static constexpr int kF1 = 0;
  static constexpr int kF2 = kF1 + (S::kLgM1 ? tw_rows(S::kLgM1, FULL) << S::kLg1 : 0);
  static constexpr int kFL = kF2 + (S::kLgM2 ? tw_rows(S::kLgM2, FULL) << (S::kLg1 + S::kLgM1) : 0);
  static constexpr int kI2 = kFL + (tw_rows(S::kLgL, FULL) << (LG - S::kLgL));
  static constexpr int kI1 = kI2 + (S::kLgM2 ? tw_rows(S::kLgM2, FULL) << S::kLgL : 0);
  static constexpr int kIL = kI1 + (S::kLgM1 ? tw_rows(S::kLgM1, FULL) << (S::kLgL + S::kLgM2) : 0);
  static constexpr int kTw = kIL + ((FULL ? S::E / 4 : tw_rows(S::kLg1, false)) << (LG - S::kLg1));
};

// The same description for the host and the table kernel: row `row` of stage b
// holds w_{Ls R}^(r k) at off + row Ls + k, r = small_tw_r(stages, b, row).
struct SmallTwStages {
  int count;
  int off[6], lgLs[6], lgR[6];
  int total;
  bool full;
};
__host__ __device__ inline int small_tw_r(const SmallTwStages& d, int b, int row) {
  if (d.full && b + 1 == d.count) return (1 << (d.lgR[b] - 1)) + 1 + 2 * row;   // last inverse stage: odd r > RL
  return tw_row_r(d.lgR[b], row, d.full);
}
template <int LG, bool FULL> SmallTwStages small_tw_stages() {
  using S = SmallShape<LG>;
  using T = SmallTw<LG, FULL>;
  SmallTwStages d{};
  d.full = FULL;
  auto add = [&](int off, int lgLs, int lgR) {
    if (lgR == 0) return;
    d.off[d.count] = off;
    d.lgLs[d.count] = lgLs;
    d.lgR[d.count++] = lgR;
  };
  add(T::kF1, S::kLg1, S::kLgM1);
  add(T::kF2, S::kLg1 + S::kLgM1, S::kLgM2);
  add(T::kFL, LG - S::kLgL, S::kLgL);
  add(T::kI2, S::kLgL, S::kLgM2);
  add(T::kI1, S::kLgL + S::kLgM2, S::kLgM1);
  add(T::kIL, LG - S::kLg1, S::kLg1);
  d.total = T::kTw;
  return d;
}

// padP(a + b) = padP(a) + padP(b) for every base and offset of a stage: the
// strides are powers of two, so the parts below 16 never carry.
__host__ __device__ constexpr int padP(int i) { return i + (i >> 4); }

template <int LG> __host__ __device__ constexpr int small_buf() { return padP(1 << LG); }   // float2 per exchange buffer

// One middle stage (span 2^LGLS, radix 2^LGR) from buffer a to buffer b.
template <int LG, bool FULL, int LGLS, int LGR, int DIR>
__device__ __forceinline__ void small_mid(const float2* a, float2* b, const float2* tw) {
  using S = SmallShape<LG>;
  constexpr int R = 1 << LGR, LS = 1 << LGLS, B = S::E / R, ST = S::N / R;
  if (threadIdx.x < S::NA) {
    float2 v[B][R];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const float2* q = a + padP(threadIdx.x + i * S::NA);
#pragma unroll
      for (int r = 0; r < R; ++r) v[i][r] = q[padP(r * ST)];
    }
#pragma unroll
    for (int i = 0; i < B; ++i) {
      const int j = threadIdx.x + i * S::NA, k = j & (LS - 1);
      stage_twiddle<R, DIR, FULL>(v[i], tw, LS, k);
      dft<R, DIR>(v[i]);
      float2* q = b + padP(((j - k) << LGR) + k);
#pragma unroll
      for (int r = 0; r < R; ++r) q[padP(r * LS)] = v[i][out_slot<R>(r)];
    }
  }
  __syncthreads();
}

// Twiddles of the last inverse stage, butterfly k.
template <int LG, bool FULL>
__device__ __forceinline__ void small_twiddle_last(float2* v, const float2* tw, int k) {
  using S = SmallShape<LG>;
  using T = SmallTw<LG, FULL>;
  constexpr int R1 = S::E, RL = S::E / 2, M = S::N / RL, ST1 = S::N / R1;
  if constexpr (FULL) {
#pragma unroll
    for (int r = 1; r < R1; ++r) {
      const float2 w = r < RL        ? tw[T::kFL + (r - 1) * M + k]
                       : (r & 1) == 0 ? tw[T::kFL + (r / 2 - 1) * M + 2 * k]
                                      : tw[T::kIL + (r - RL) / 2 * ST1 + k];
      v[r] = cmulc(v[r], w);
    }
  } else {
    stage_twiddle<R1, +1, false>(v, tw + T::kIL, ST1, k);
  }
}

// v (element tid + r N/R1 in v[r]) -> inverse FFT of op(forward FFT of v),
// unnormalised, in the same order.  op(k, za, zb) is applied to every pair
// (k, N - k), k <= N/2; for the self-pairs k = 0 and N/2 za and zb hold the
// same value and za is kept.  S0, S1: exchange buffers; on return S0 and S1
// may still be read by other threads of the CTA only in the way the next call
// allows (it writes S0 first, whose last reader is behind a barrier).
template <int LG, bool FULL, class OP>
__device__ __forceinline__ void small_conv(float2 (&v)[SmallShape<LG>::E], float2* S0, float2* S1,
                                           const float2* tw, const OP& op) {
  using S = SmallShape<LG>;
  using T = SmallTw<LG, FULL>;
  constexpr int N = S::N, R1 = S::E, RL = S::E / 2, M = N / RL, ST1 = N / R1;
  const int tid = threadIdx.x;
  const bool act = tid < S::NA;
  float2 *a = S0, *b = S1;
  if (act) {
    dft<R1, -1>(v);
    float2* q = a + padP(tid * R1);
#pragma unroll
    for (int r = 0; r < R1; ++r) q[r] = v[out_slot<R1>(r)];   // padP(tid R1 + r): r stays below the next pad slot
  }
  __syncthreads();
  if constexpr (S::kLgM1 > 0) {
    small_mid<LG, FULL, S::kLg1, S::kLgM1, -1>(a, b, tw + T::kF1);
    float2* t = a; a = b; b = t;
  }
  if constexpr (S::kLgM2 > 0) {
    small_mid<LG, FULL, S::kLg1 + S::kLgM1, S::kLgM2, -1>(a, b, tw + T::kF2);
    float2* t = a; a = b; b = t;
  }
  if (act) {
    const int j0 = tid, j1 = tid == 0 ? M / 2 : M - tid;
    float2 x[RL], y[RL];
    const float2 *q0 = a + padP(j0), *q1 = a + padP(j1);
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      x[r] = q0[padP(r * M)];
      y[r] = q1[padP(r * M)];
    }
    stage_twiddle<RL, -1, FULL>(x, tw + T::kFL, M, j0);
    stage_twiddle<RL, -1, FULL>(y, tw + T::kFL, M, j1);
    dft<RL, -1>(x);
    dft<RL, -1>(y);
    float2 p[RL], w[RL];   // frequency order
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      p[r] = x[out_slot<RL>(r)];
      w[r] = y[out_slot<RL>(r)];
    }
    // pairs (j0 + r M, its mirror) and (j1 + r M, its mirror), r < RL/2; the
    // mirrors are the other butterfly's outputs, but thread 0's butterflies
    // are their own mirrors: its partner is selected, as a branch would run
    // the operator twice in its warp
    const bool self = tid == 0;
#pragma unroll
    for (int r = 0; r < RL / 2; ++r) {
      float2 z = self ? p[r == 0 ? 0 : RL - r] : w[RL - 1 - r];
      op(j0 + r * M, p[r], z);
      if (r > 0) p[RL - r] = self ? z : p[RL - r];
      w[RL - 1 - r] = self ? w[RL - 1 - r] : z;
    }
#pragma unroll
    for (int r = 0; r < RL / 2; ++r) {
      float2 z = self ? w[RL - 1 - r] : p[RL - 1 - r];
      op(j1 + r * M, w[r], z);
      w[RL - 1 - r] = self ? z : w[RL - 1 - r];
      p[RL - 1 - r] = self ? p[RL - 1 - r] : z;
    }
    if (self) {
      float2 z = p[RL / 2];
      op(N / 2, p[RL / 2], z);
    }
    dft<RL, +1>(p);
    dft<RL, +1>(w);
    float2 *o0 = b + padP(j0 * RL), *o1 = b + padP(j1 * RL);
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      o0[r] = p[out_slot<RL>(r)];
      o1[r] = w[out_slot<RL>(r)];
    }
  }
  __syncthreads();
  { float2* t = a; a = b; b = t; }
  if constexpr (S::kLgM2 > 0) {
    small_mid<LG, FULL, S::kLgL, S::kLgM2, +1>(a, b, tw + T::kI2);
    float2* t = a; a = b; b = t;
  }
  if constexpr (S::kLgM1 > 0) {
    small_mid<LG, FULL, S::kLgL + S::kLgM2, S::kLgM1, +1>(a, b, tw + T::kI1);
    float2* t = a; a = b; b = t;
  }
  if (act) {
    const float2* q = a + padP(tid);
    float2 u[R1];
#pragma unroll
    for (int r = 0; r < R1; ++r) u[r] = q[padP(r * ST1)];
    small_twiddle_last<LG, FULL>(u, tw, tid);
    dft<R1, +1>(u);
#pragma unroll
    for (int r = 0; r < R1; ++r) v[r] = u[out_slot<R1>(r)];
  }
}

}  // namespace csk
