// Whole solves and products of one instance with n <= 8192 (ADMM: n <= 4096)
// by one CTA: a solve is one launch, and an iteration passes through shared
// memory only between FFT stages (cs_small.cuh).
//
// The pass kernels spend 4 (ADMM 2) launches an iteration on transforms that
// fill one to 32 CTAs for a few microseconds each; here the state (x, or mu
// and nu) stays in registers and y in shared memory for all iterations.  What
// bounds it is the latency of one SM: barriers and FP32 issue.
#include "cs_small.cuh"

#include "cs_internal.h"

namespace csk {

namespace {

__device__ __forceinline__ float soft(float u, float g) { return u > g ? u - g : (u < -g ? u + g : 0.f); }

// Product operator on a pair of the packed spectrum (a, a', b in tA, tB; see
// the table kernel below): C^T for ADJ, else C.
//   C^T: Z_k' = a Z_k + b conj(Z_{N-k}), Z_{N-k}' = a' Z_{N-k} - conj(b) conj(Z_k)
//   C:   a, a' conjugated and b -> -conj(b)
template <bool ADJ>
struct OpReal {
  const float4* tA;
  const float2* tB;
  __device__ __forceinline__ void operator()(int k, float2& za, float2& zb) const {
    const float4 t = __ldg(tA + k);
    const float2 be = __ldg(tB + k);
    const float2 al = make_float2(t.x, ADJ ? t.y : -t.y), al2 = make_float2(t.z, ADJ ? t.w : -t.w);
    const float2 b1 = ADJ ? be : make_float2(-be.x, be.y);
    const float2 b2 = make_float2(-b1.x, b1.y);
    const float2 a0 = za, c0 = zb;
    za = cadd(cmul(al, a0), cmul(b1, cconj(c0)));
    zb = cadd(cmul(al2, c0), cmul(b2, cconj(a0)));
  }
};

// Algorithm 3's x-update on a pair (see the mid pass's operator).
struct OpAdmm {
  const float2* tc;
  const float* tb;
  float rho, sigma;
  __device__ __forceinline__ void operator()(int k, float2& za, float2& zb) const {
    const float2 ch = __ldg(tc + k);
    const float bb = __ldg(tb + k);
    const float2 V = make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y));
    const float2 Wk = make_float2(0.5f * (za.y + zb.y), -0.5f * (za.x - zb.x));
    const float2 cv = cmul(ch, V);
    const float2 X = make_float2(bb * fmaf(rho, cv.x, sigma * Wk.x), bb * fmaf(rho, cv.y, sigma * Wk.y));
    const float2 Pc = cmulc(X, ch);
    za = make_float2(X.x - Pc.y, X.y + Pc.x);
    zb = make_float2(X.x + Pc.y, Pc.x - X.y);
  }
};

template <int LG, bool FULL>
__device__ __forceinline__ void load_tw(float2* dst, const float2* __restrict__ src) {
  for (int i = threadIdx.x; i < SmallTw<LG, FULL>::kTw; i += SmallShape<LG>::NT) dst[i] = __ldg(src + i);
}

// Sum over the CTA in a fixed order; every thread gets it.
template <int NT>
__device__ double block_sum(double d, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  __syncthreads();   // red may still be read from the call before
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) s += red[w];
  return s;
}

// y (caller's order) into the dense shared vector yd by row, with the row
// mask; a non-finite y latches STS_NONFINITE.  Ends with a barrier.
template <int NT>
__device__ __forceinline__ void stage_y(const SmallArgs& a, int n, float* yd, uint32_t* mk) {
  for (int i = threadIdx.x; i < n; i += NT) yd[i] = 0.f;
  for (int i = threadIdx.x; i < n / 32; i += NT) mk[i] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < a.m; i += NT) {
    const float v = __ldg(a.y + i);
    const int r = __ldg(a.rows + i);
    if (!isfinite(v)) atomicOr(a.status, STS_NONFINITE);
    yd[r] = v;
    atomicOr(mk + (r >> 5), 1u << (r & 31));
  }
  __syncthreads();
}

// ISTA (Algorithm 1): n = 2 N packed, x (natural order, any 4-byte boundary)
// in and out.
template <int LG, bool FULL>
__device__ __forceinline__ void small_ista(const SmallArgs& a) {
  using S = SmallShape<LG>;
  constexpr int N = S::N, E = S::E, ST = N / E, NT = S::NT;
  extern __shared__ float2 sm[];
  float2 *S0 = sm, *S1 = S0 + small_buf<LG>(), *tw = S1 + small_buf<LG>();
  float2* yd = tw + ((SmallTw<LG, FULL>::kTw + 1) & ~1);
  __shared__ uint32_t mk[2 * N / 32];
  __shared__ double red[NT / 32];
  load_tw<LG, FULL>(tw, a.tw);
  stage_y<NT>(a, 2 * N, reinterpret_cast<float*>(yd), mk);
  const int tid = threadIdx.x;
  const bool act = tid < S::NA;
  float2 x[E], v[E];
  uint32_t mb = 0;
  if (act) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int p = tid + r * ST;
      x[r] = v[r] = make_float2(a.x[2 * p], a.x[2 * p + 1]);
      mb |= ((mk[p >> 4] >> ((2 * p) & 31)) & 3u) << (2 * r);
    }
  }
  const OpReal<false> opf{a.tA, a.tB};
  const OpReal<true> opa{a.tA, a.tB};
  // (one copy of the transform with the product's sign as a run-time factor
  // was slower, 4.7 against 4.0 us an iteration at n = 4096)
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const bool st = a.stats != nullptr && it + 1 == a.iters;
    float r2 = 0.f;
    small_conv<LG, FULL>(v, S0, S1, tw, opf);
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const float2 y = yd[tid + r * ST];
        const float r0 = ((mb >> (2 * r)) & 1u) ? y.x - v[r].x : 0.f;
        const float r1 = ((mb >> (2 * r)) & 2u) ? y.y - v[r].y : 0.f;
        if (st) r2 = fmaf(r0, r0, fmaf(r1, r1, r2));
        v[r] = make_float2(r0, r1);
      }
    }
    small_conv<LG, FULL>(v, S0, S1, tw, opa);
    float dx2 = 0.f, x2 = 0.f, l1 = 0.f, er = 0.f, nf = 0.f;
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const float2 xo = x[r];
        x[r].x = soft(fmaf(a.tau, v[r].x, xo.x), a.thr);
        x[r].y = soft(fmaf(a.tau, v[r].y, xo.y), a.thr);
        v[r] = x[r];
        if (st) {
          const float d0 = x[r].x - xo.x, d1 = x[r].y - xo.y;
          dx2 = fmaf(d0, d0, fmaf(d1, d1, dx2));
          x2 = fmaf(x[r].x, x[r].x, fmaf(x[r].y, x[r].y, x2));
          l1 += fabsf(xo.x) + fabsf(xo.y);
          if (a.xtrue) {   // tile order of the plan's packed geometry
            const int p = tid + r * ST, j1 = p & ((1 << a.lgN1) - 1), j2 = p >> a.lgN1;
            const int t = ((j1 >> a.lgG) << (a.lgG + a.lgN2)) + (j2 << a.lgG) + (j1 & ((1 << a.lgG) - 1));
            const float e0 = x[r].x - a.xtrue[2 * t], e1 = x[r].y - a.xtrue[2 * t + 1];
            er = fmaf(e0, e0, fmaf(e1, e1, er));
          }
          if (!isfinite(x[r].x) || !isfinite(x[r].y)) nf += 1.f;
        }
      }
    }
    if (st) {
      const float s[6] = {er, dx2, x2, l1, r2, nf};   // order of the ST_ slots
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double d = block_sum<NT>((double)s[k], red);
        if (tid == 0) a.stats[k] = d;
      }
    }
  }
  if (act) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int p = tid + r * ST;
      a.x[2 * p] = x[r].x;
      a.x[2 * p + 1] = x[r].y;
    }
  }
}

// Algorithm 3, n = N (complex): state (v, z, mu, nu) in natural order, in
// when a.warm (else zero), out where the pointer is not null.
template <int LG, bool FULL>
__device__ __forceinline__ void small_admm(const SmallArgs& a) {
  using S = SmallShape<LG>;
  constexpr int N = S::N, E = S::E, ST = N / E, NT = S::NT;
  extern __shared__ float2 sm[];
  float2 *S0 = sm, *S1 = S0 + small_buf<LG>(), *tw = S1 + small_buf<LG>();
  float* yd = reinterpret_cast<float*>(S1);   // only until the registers hold it
  __shared__ uint32_t mk[N / 32];
  __shared__ double red[NT / 32];
  load_tw<LG, FULL>(tw, a.tw);
  stage_y<NT>(a, N, yd, mk);
  const int tid = threadIdx.x;
  const bool act = tid < S::NA;
  float2 v[E];
  float mu[E], nu[E], y[E];
  uint32_t mb = 0;
  if (act) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int p = tid + r * ST;
      mb |= ((mk[p >> 5] >> (p & 31)) & 1u) << r;
      y[r] = yd[p];
      mu[r] = a.warm ? a.mu[p] : 0.f;
      nu[r] = a.warm ? a.nu[p] : 0.f;
      v[r] = a.warm ? make_float2(a.v[p], a.z[p] - nu[r]) : make_float2(0.f, 0.f);
    }
  }
  const OpAdmm op{a.tc, a.tb, a.rho, a.sigma};
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const bool end = it + 1 == a.iters, st = a.stats != nullptr && end;
    float r2 = 0.f, dx2 = 0.f, x2 = 0.f, l1 = 0.f, er = 0.f, nf = 0.f;
    small_conv<LG, FULL>(v, S0, S1, tw, op);
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const bool on = (mb >> r) & 1u;
        const float x = v[r].x, cx = v[r].y;
        const float vv = (on ? a.d_on : a.d_off) * fmaf(a.rho, cx - mu[r], y[r]);
        const float z = soft(x + nu[r], a.thr);
        mu[r] = fmaf(a.tau1, vv - cx, mu[r]);
        nu[r] = fmaf(a.tau2, x - z, nu[r]);
        const float vf = vv + mu[r];
        v[r] = make_float2(vf, z - nu[r]);
        if (end) {
          const int p = tid + r * ST;
          if (a.z) a.z[p] = z;
          if (a.v) a.v[p] = vf;
          if (a.mu) a.mu[p] = mu[r];
          if (a.nu) a.nu[p] = nu[r];
          if (a.x) a.x[p] = x;
          if (st) {
            if (a.xtrue) {
              const int j1 = p & ((1 << a.lgN1) - 1), j2 = p >> a.lgN1;
              const float e = z - a.xtrue[((j1 >> a.lgG) << (a.lgG + a.lgN2)) + (j2 << a.lgG) +
                                          (j1 & ((1 << a.lgG) - 1))];
              er = fmaf(e, e, er);
            }
            dx2 = fmaf(x - z, x - z, dx2);
            x2 = fmaf(z, z, x2);
            l1 += fabsf(z);
            const float rr = on ? y[r] - cx : 0.f;
            r2 = fmaf(rr, rr, r2);
            if (!isfinite(z) || !isfinite(vf)) nf += 1.f;
          }
        }
      }
    }
    if (st) {
      const float s[6] = {er, dx2, x2, l1, r2, nf};
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double d = block_sum<NT>((double)s[k], red);
        if (tid == 0) a.stats[k] = d;
      }
    }
  }
}

template <int LG>
__global__ void __launch_bounds__(SmallShape<LG>::NT) small_ista_k(const SmallArgs a) { small_ista<LG, false>(a); }
template <int LG>
__global__ void __launch_bounds__(SmallShape<LG>::NT) small_admm_k(const SmallArgs a) { small_admm<LG, false>(a); }

// Instance blockIdx.x of a size class of a batch: its constants, its scalars
// of this call, and the call's concatenated vectors.
__device__ __forceinline__ SmallArgs class_args(const SmallInst& d, const SmallScalars& s, const float* y, int iters) {
  SmallArgs a{};
  a.tA = d.tA;
  a.tB = d.tB;
  a.tc = d.tc;
  a.tb = d.tb;
  a.tw = d.tw;
  a.rows = d.rows;
  a.m = d.m;
  a.y = y + d.moff;
  a.status = d.status;
  a.iters = iters;
  a.thr = s.thr;
  a.tau = s.tau;
  a.rho = s.rho;
  a.sigma = s.sigma;
  a.tau1 = s.tau1;
  a.tau2 = s.tau2;
  a.d_on = s.d_on;
  a.d_off = s.d_off;
  return a;
}
template <int LG>
__global__ void __launch_bounds__(SmallShape<LG>::NT)
    class_ista_k(const SmallInst* __restrict__ inst, const SmallScalars* __restrict__ sc, const float* __restrict__ y,
                 float* __restrict__ x, int iters) {
  SmallInst d = inst[blockIdx.x];
  d.tw = d.tw_i;
  SmallArgs a = class_args(d, sc[d.id], y, iters);
  a.x = x + d.noff;
  small_ista<LG, true>(a);
}
template <int LG>
__global__ void __launch_bounds__(SmallShape<LG>::NT)
    class_admm_k(const SmallInst* __restrict__ inst, const SmallScalars* __restrict__ sc, const float* __restrict__ y,
                 float* __restrict__ z, int iters) {
  SmallInst d = inst[blockIdx.x];
  d.tw = d.tw_a;
  SmallArgs a = class_args(d, sc[d.id], y, iters);
  a.z = z + d.noff;
  small_admm<LG, true>(a);
}

// Power iteration on A^T A from the fixed start vector in a.x (natural
// order): per iteration u = w / ||w||, w = A^T A u; stats[ST_DX2] = <u, w> and
// stats[ST_X2] = ||w||^2 of the last.
template <int LG>
__global__ void __launch_bounds__(SmallShape<LG>::NT) small_power_k(const SmallArgs a) {
  using S = SmallShape<LG>;
  constexpr int N = S::N, E = S::E, ST = N / E, NT = S::NT;
  extern __shared__ float2 sm[];
  float2 *S0 = sm, *S1 = S0 + small_buf<LG>(), *tw = S1 + small_buf<LG>();
  __shared__ uint32_t mk[2 * N / 32];
  __shared__ double red[NT / 32];
  load_tw<LG, false>(tw, a.tw);
  for (int i = threadIdx.x; i < 2 * N / 32; i += NT) mk[i] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < a.m; i += NT) {
    const int r = __ldg(a.rows + i);
    atomicOr(mk + (r >> 5), 1u << (r & 31));
  }
  __syncthreads();
  const int tid = threadIdx.x;
  const bool act = tid < S::NA;
  const float2* xg = reinterpret_cast<const float2*>(a.x);
  float2 u[E], v[E];
  uint32_t mb = 0;
  double s2 = 0.0;
  if (act) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int p = tid + r * ST;
      v[r] = xg[p];
      mb |= ((mk[p >> 4] >> ((2 * p) & 31)) & 3u) << (2 * r);
      s2 += (double)v[r].x * v[r].x + (double)v[r].y * v[r].y;
    }
  }
  double x2 = block_sum<NT>(s2, red), dot = 0.0;
  const OpReal<false> opf{a.tA, a.tB};
  const OpReal<true> opa{a.tA, a.tB};
#pragma unroll 1
  for (int it = 0; it < a.iters; ++it) {
    const float s = (float)rsqrt(x2);
#pragma unroll
    for (int r = 0; r < E; ++r) u[r] = v[r] = act ? cscale(v[r], s) : make_float2(0.f, 0.f);
    small_conv<LG, false>(v, S0, S1, tw, opf);
#pragma unroll
    for (int r = 0; r < E; ++r)
      v[r] = make_float2(((mb >> (2 * r)) & 1u) ? v[r].x : 0.f, ((mb >> (2 * r)) & 2u) ? v[r].y : 0.f);
    small_conv<LG, false>(v, S0, S1, tw, opa);
    float n2 = 0.f, uw = 0.f;
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        n2 = fmaf(v[r].x, v[r].x, fmaf(v[r].y, v[r].y, n2));
        uw = fmaf(u[r].x, v[r].x, fmaf(u[r].y, v[r].y, uw));
      }
    }
    x2 = block_sum<NT>((double)n2, red);
    dot = block_sum<NT>((double)uw, red);
  }
  if (tid == 0) {
    a.stats[ST_X2] = x2;
    a.stats[ST_DX2] = dot;
  }
}

// One product.  FWD: y = A x (rows gathered in the caller's order); else
// x = A^T y.
template <int LG, bool FWD>
__global__ void __launch_bounds__(SmallShape<LG>::NT) small_product_k(const SmallArgs a) {
  using S = SmallShape<LG>;
  constexpr int N = S::N, E = S::E, ST = N / E, NT = S::NT;
  extern __shared__ float2 sm[];
  float2 *S0 = sm, *S1 = S0 + small_buf<LG>(), *tw = S1 + small_buf<LG>();
  float2* d = tw + ((SmallTw<LG, false>::kTw + 1) & ~1);
  const int tid = threadIdx.x;
  const bool act = tid < S::NA;
  float2 v[E];
  float2* xg = reinterpret_cast<float2*>(a.x);
  if (FWD) {
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = __ldg(xg + tid + r * ST);
    }
    load_tw<LG, false>(tw, a.tw);   // read behind the product's first barrier
    small_conv<LG, false>(v, S0, S1, tw, OpReal<false>{a.tA, a.tB});
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) d[tid + r * ST] = v[r];
    }
    __syncthreads();
    const float* df = reinterpret_cast<const float*>(d);
    for (int i = tid; i < a.m; i += NT) a.yo[i] = df[__ldg(a.rows + i)];
  } else {
    load_tw<LG, false>(tw, a.tw);
    for (int i = tid; i < N; i += NT) d[i] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int i = tid; i < a.m; i += NT) reinterpret_cast<float*>(d)[__ldg(a.rows + i)] = __ldg(a.y + i);
    __syncthreads();
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = d[tid + r * ST];
    }
    small_conv<LG, false>(v, S0, S1, tw, OpReal<true>{a.tA, a.tB});
    if (act) {
#pragma unroll
      for (int r = 0; r < E; ++r) xg[tid + r * ST] = v[r];
    }
  }
}

// ------------------------------------------------------------- plan time

__global__ void small_tw_k(float2* dst, SmallTwStages d) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= d.total) return;
  int b = 0;
  while (b + 1 < d.count && t >= d.off[b + 1]) ++b;
  const int q = t - d.off[b], r = small_tw_r(d, b, q >> d.lgLs[b]), k = q & ((1 << d.lgLs[b]) - 1);
  double sn, cs;
  sincospi(-2.0 * (double)(r * k) / (double)(1 << (d.lgLs[b] + d.lgR[b])), &sn, &cs);
  dst[t] = make_float2((float)cs, (float)sn);
}

// Packed real geometry, pairs (k, N - k) of k in [0, N/2] in natural order:
// P = (c^_k + c^_{k+N}) / 2N, Q = (c^_k - c^_{k+N}) / 2N, theta = pi k / N,
// a = P - Q sin(theta), a' = conj(P + Q sin(theta)), b = i Q cos(theta).
__global__ void small_tab_ista_k(const double2* __restrict__ chat, int64_t n, float4* __restrict__ tA,
                                 float2* __restrict__ tB) {
  const int64_t N = n >> 1;
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k > (N >> 1)) return;
  double2 a = chat[k], b = chat[k + N];
  if (k == 0) { a.y = 0.0; b.y = 0.0; }
  const double s = 0.5 / (double)N;
  const double Px = (a.x + b.x) * s, Py = (a.y + b.y) * s, Qx = (a.x - b.x) * s, Qy = (a.y - b.y) * s;
  double sn, cs;
  sincospi((double)k / (double)N, &sn, &cs);
  tA[k] = make_float4((float)(Px - Qx * sn), (float)(Py - Qy * sn), (float)(Px + Qx * sn), (float)(-(Py + Qy * sn)));
  tB[k] = make_float2((float)(-Qy * cs), (float)(Qx * cs));
}

__global__ void small_tab_admm_k(const double2* __restrict__ chat, int64_t n, float2* __restrict__ tc,
                                 double* __restrict__ abs2) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k > (n >> 1)) return;
  double2 a = chat[k];
  if (k == 0 || k == (n >> 1)) a.y = 0.0;
  tc[k] = make_float2((float)a.x, (float)a.y);
  abs2[k] = a.x * a.x + a.y * a.y;
}

template <int LG, bool FULL>
constexpr size_t small_smem(bool dense) {
  return sizeof(float2) * (2 * small_buf<LG>() + ((SmallTw<LG, FULL>::kTw + 1) & ~1)) +
         (dense ? sizeof(float2) << LG : 0);
}

cudaError_t opt_in_smem(const void* fn, size_t smem) {
  return smem > 48 * 1024 ? cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                          : cudaSuccess;
}

// LG = 13 (64 values of padding per 1024 and 84 KiB of twiddles: 220 KiB)
// fits without a dense y, so only ADMM takes it.
template <int LG>
cudaError_t class_run(bool admm, const SmallInst* inst, int count, const SmallScalars* sc, const float* y, float* xz,
                      int iters, cudaStream_t s) {
  const void* fn = nullptr;
  size_t smem = small_smem<LG, true>(!admm);
  if (admm) fn = (const void*)class_admm_k<LG>;
  else if constexpr (LG <= SMALL_LG_MAX) fn = (const void*)class_ista_k<LG>;
  if (!fn) return cudaErrorInvalidValue;
  const cudaError_t e = opt_in_smem(fn, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&inst, &sc, &y, &xz, &iters};
  return cudaLaunchKernel(fn, dim3((unsigned)count), dim3(SmallShape<LG>::NT), args, smem, s);
}

template <int LG>
cudaError_t class_wave(int* instances) {
  const void* fn = (const void*)class_admm_k<LG>;
  const size_t smem = small_smem<LG, true>(false);
  int dev = 0, sms = 0, ctas = 0;
  cudaError_t e = opt_in_smem(fn, smem);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, fn, SmallShape<LG>::NT, smem);
  *instances = sms * ctas > 0 ? sms * ctas : 1;
  return e;
}

template <int LG>
cudaError_t small_run(SmallKind kind, const SmallArgs& a, cudaStream_t s) {
  using S = SmallShape<LG>;
  const void* fn = nullptr;
  size_t smem = 0;
  switch (kind) {
    case SMALL_ISTA: fn = (const void*)small_ista_k<LG>; smem = small_smem<LG, false>(true); break;
    case SMALL_ADMM: fn = (const void*)small_admm_k<LG>; smem = small_smem<LG, false>(false); break;
    case SMALL_POWER: fn = (const void*)small_power_k<LG>; smem = small_smem<LG, false>(false); break;
    case SMALL_FWD: fn = (const void*)small_product_k<LG, true>; smem = small_smem<LG, false>(true); break;
    case SMALL_ADJ: fn = (const void*)small_product_k<LG, false>; smem = small_smem<LG, false>(true); break;
  }
  const cudaError_t e = opt_in_smem(fn, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<SmallArgs*>(&a)};
  return cudaLaunchKernel(fn, dim3(1), dim3(S::NT), args, smem, s);
}

}  // namespace

#define CS_SMALL_LG(X) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12)

cudaError_t launch_small(SmallKind kind, int lgN, const SmallArgs& a, cudaStream_t s) {
  switch (lgN) {
#define CS_X(L) case L: return small_run<L>(kind, a, s);
    CS_SMALL_LG(CS_X)
#undef CS_X
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_small_class(bool admm, int lgN, const SmallInst* inst, int count, const SmallScalars* sc,
                               const float* y, float* xz, int iters, cudaStream_t s) {
  switch (lgN) {
#define CS_X(L) case L: return class_run<L>(admm, inst, count, sc, y, xz, iters, s);
    CS_SMALL_LG(CS_X)
    CS_X(13)
#undef CS_X
  }
  return cudaErrorInvalidValue;
}

cudaError_t small_class_wave(int lgn, int* instances) {
  switch (lgn) {
#define CS_X(L) case L: return class_wave<L>(instances);
    CS_SMALL_LG(CS_X)
    CS_X(13)
#undef CS_X
  }
  return cudaErrorInvalidValue;
}

static SmallTwStages tw_stages(int lgN, bool full) {
  switch (lgN) {
    case 13: return small_tw_stages<13, true>();   // size classes only
#define CS_X(L) case L: return full ? small_tw_stages<L, true>() : small_tw_stages<L, false>();
    CS_SMALL_LG(CS_X)
#undef CS_X
  }
  return SmallTwStages{};
}

int small_tw_count(int lgN, bool full) { return tw_stages(lgN, full).total; }

cudaError_t launch_small_tw(int lgN, bool full, float2* tw, cudaStream_t s) {
  const SmallTwStages d = tw_stages(lgN, full);
  small_tw_k<<<(unsigned)((d.total + 255) / 256), 256, 0, s>>>(tw, d);
  return cudaGetLastError();
}

cudaError_t launch_small_tables(const double2* chat, int64_t n, float4* tA, float2* tB, float2* tc, double* abs2,
                                cudaStream_t s) {
  auto nb = [](int64_t c) { return (unsigned)((c + 255) / 256); };
  small_tab_ista_k<<<nb(n / 4 + 1), 256, 0, s>>>(chat, n, tA, tB);
  if (tc) small_tab_admm_k<<<nb(n / 2 + 1), 256, 0, s>>>(chat, n, tc, abs2);
  return cudaGetLastError();
}

}  // namespace csk
