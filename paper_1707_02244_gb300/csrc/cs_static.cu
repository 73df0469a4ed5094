// Allocation-free circulant product: y = C x or C^T x for one generating
// vector, with its FFT work space in a fixed device array of this library
// instead of memory from cudaMalloc.
//
// Some callers cannot call cudaMalloc: code whose device memory is owned
// entirely by another allocator (a framework's caching allocator, or a fixed
// pool reserved up front), and latency-critical loops that cannot afford the
// implicit device synchronisation an allocation may cause.  This entry point
// serves them: the caller passes the inputs and the output, and the work
// space is the file-scope array below.
#include <cuda_runtime.h>

#include <mutex>

#include "../../include/cs.h"
#include "cs_internal.h"

namespace csk {

namespace {

constexpr int64_t kStaticMaxN = CS_STATIC_MAX_N;

// The packed transforms of c and x, n/2 FP64 complex values each, at the
// largest supported length (256 KiB).
// Every GPU that loads the library holds this array until the process exits.
// All calls share it: calls that overlap on the GPU race on it.
static __device__ __align__(256) double2 g_static_scratch[kStaticMaxN];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
struct ScratchAddr {
  void* ctx = nullptr;        // CUDA context the address belongs to
  double2* addr = nullptr;
};
ScratchAddr g_scratch_addr[kMaxDevices];

// cuCtxGetCurrent from the driver, fetched through the runtime so that the
// library needs no link against libcuda.
using CtxGetCurrentFn = int (*)(void**);
CtxGetCurrentFn ctx_get_current() {
  static CtxGetCurrentFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<CtxGetCurrentFn>(f);
  }();
  return fn;
}

// Device address of the array in the current context.  In host code the
// array's name is only a host-side stand-in, so the address comes from
// cudaGetSymbolAddress, looked up once per device with that device current.
// The lookup is repeated when the device's current context is another one
// than at the last lookup (after cudaDeviceReset the module, and with it the
// array, can be loaded at another address).
cudaError_t scratch_address(double2** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  CtxGetCurrentFn get = ctx_get_current();
  if (!get) return cudaErrorInitializationError;
  // null before the runtime has made a context current on this thread
  void* ctx = nullptr;
  if (get(&ctx) != 0) return cudaErrorInitializationError;
  std::lock_guard<std::mutex> lock(g_mu);
  ScratchAddr& sa = g_scratch_addr[dev];
  if (!sa.addr || !ctx || sa.ctx != ctx) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);   // makes the device's primary context current if none is
    if (e != cudaSuccess) return e;
    if (get(&ctx) != 0 || !ctx) return cudaErrorInitializationError;
    sa.addr = static_cast<double2*>(p);
    sa.ctx = ctx;
  }
  *out = sa.addr;
  return cudaSuccess;
}

// ------------------------------------------------------------ the product
//
// c and x are real: each is packed as N = n/2 complex values (v_2p + i
// v_2p+1) and transformed four-step, N = N1 x N2 (element p = j1 + N1 j2,
// frequency k = k2 + N2 k1), in three launches:
//   1  length-N2 FFTs of the columns of both, and the twiddle w_N^(j1 k2);
//   2  length-N1 FFTs of the rows k2 and N2 - k2 of both, so that every
//      frequency meets its mirror N - k; the product of the two real
//      spectra; the length-N1 inverse and the twiddle on the way back;
//   3  the length-N2 inverse FFTs of the columns, rounded to y.
// FP64 runs at about 2 FMA per clock and SM, so what bounds a call is the
// arithmetic of the busiest SM and the latency of three small launches:
// one column or one row pair per CTA spreads 16384 values over 64 to 128 SMs,
// and the roots of unity come from a table instead of sincospi.
// Radix-2 stages over global memory took 45 launches and 275 us a call at
// n = 16384; this takes 25 us.

constexpr int kMaxLgN = 13;                      // log2 of the largest N
constexpr int kRoots = 128;                      // w_128^q and w_16384^q, q < 128

struct Cplx { double x, y; };
struct RootTab { Cplx v[2 * kRoots]; };

// cos / sin of 2 pi q / m (m a multiple of 8) by their Taylor series on the
// first octant, the angle reduced exactly in integers.
constexpr double taylor_sin(double t) {
  double s = 0.0;
  for (int k = 10; k >= 0; --k) s = 1.0 - s * t * t / ((2.0 * k + 2.0) * (2.0 * k + 3.0));
  return t * s;
}
constexpr double taylor_cos(double t) {
  double s = 0.0;
  for (int k = 10; k >= 0; --k) s = 1.0 - s * t * t / ((2.0 * k + 1.0) * (2.0 * k + 2.0));
  return s;
}
constexpr Cplx root(int q, int m) {   // exp(-2 pi i q / m), 0 <= q < m
  const int oct = q / (m / 8), rem = q % (m / 8);
  const int f = (oct & 1) ? m / 8 - rem : rem;   // angle to the nearest axis
  const double t = 6.283185307179586476925286766559 * f / m;
  const double cs = taylor_cos(t), sn = taylor_sin(t);
  double c = 0.0, s = 0.0;                       // cos, sin of 2 pi q / m
  switch (oct) {
    case 0: c = cs; s = sn; break;
    case 1: c = sn; s = cs; break;
    case 2: c = -sn; s = cs; break;
    case 3: c = -cs; s = sn; break;
    case 4: c = -cs; s = -sn; break;
    case 5: c = -sn; s = -cs; break;
    case 6: c = sn; s = -cs; break;
    default: c = cs; s = -sn; break;
  }
  return Cplx{c, -s};
}
constexpr RootTab make_roots() {
  RootTab r{};
  for (int q = 0; q < kRoots; ++q) {
    r.v[q] = root(q, kRoots);
    r.v[kRoots + q] = root(q, kRoots * kRoots);
  }
  return r;
}
__device__ const RootTab g_roots = make_roots();

__device__ __forceinline__ double2 dmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 dadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 dsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 dconj(double2 a) { return make_double2(a.x, -a.y); }

__device__ __forceinline__ void load_roots(double2* rt) {
  for (int i = threadIdx.x; i < 2 * kRoots; i += blockDim.x) rt[i] = make_double2(g_roots.v[i].x, g_roots.v[i].y);
}
// w_16384^p, p < 16384
__device__ __forceinline__ double2 root_at(const double2* rt, int p) {
  return dmul(rt[p >> 7], rt[kRoots + (p & (kRoots - 1))]);
}

// FFTs of `vecs` length-2^lgL vectors (element e of vector v at v L + e) in
// shared memory, radix 4 with a closing radix 2, between two buffers; DIR as
// elsewhere (-1 forward).  Returns the buffer that holds the result; starts
// and ends with a barrier.
template <int DIR>
__device__ double2* fft64_tile(double2* a, double2* b, int lgL, int vecs, const double2* rt) {
  const int L = 1 << lgL;
  int lgLs = 0;
  __syncthreads();
  while (lgLs < lgL) {
    const int lgR = lgL - lgLs >= 2 ? 2 : 1;
    const int lgB = lgL - lgR, Ls = 1 << lgLs;
    for (int t = threadIdx.x; t < vecs << lgB; t += blockDim.x) {
      const int base = (t >> lgB) << lgL, j = t & ((1 << lgB) - 1), k = j & (Ls - 1);
      const int o = base + ((j - k) << lgR) + k;
      const int step = kRoots >> (lgLs + lgR);   // w_{Ls R}^k = w_128^(k step): L <= 128
      auto tw = [&](double2 v, int r) {
        double2 w = rt[r * k * step];
        if (DIR > 0) w.y = -w.y;
        return dmul(v, w);
      };
      if (lgR == 2) {
        const int h = L >> 2;
        double2 v0 = a[base + j], v1 = a[base + j + h], v2 = a[base + j + 2 * h], v3 = a[base + j + 3 * h];
        if (k) {
          v1 = tw(v1, 1);
          v2 = tw(v2, 2);
          v3 = tw(v3, 3);
        }
        const double2 s02 = dadd(v0, v2), d02 = dsub(v0, v2), s13 = dadd(v1, v3), d = dsub(v1, v3);
        const double2 d13 = DIR > 0 ? make_double2(-d.y, d.x) : make_double2(d.y, -d.x);
        b[o] = dadd(s02, s13);
        b[o + Ls] = dadd(d02, d13);
        b[o + 2 * Ls] = dsub(s02, s13);
        b[o + 3 * Ls] = dsub(d02, d13);
      } else {
        const int h = L >> 1;
        const double2 v0 = a[base + j];
        double2 v1 = a[base + j + h];
        if (k) v1 = tw(v1, 1);
        b[o] = dadd(v0, v1);
        b[o + Ls] = dsub(v0, v1);
      }
    }
    __syncthreads();
    double2* t = a;
    a = b;
    b = t;
    lgLs += lgR;
  }
  return a;
}

__device__ __forceinline__ void dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int kColNt = 32, kMidNt = 128;

// Launch 1: column blockIdx.x of c (blockIdx.y = 0) or x (1).  Row k2 of the
// N2 x N1 result at k2 N1.
__global__ void __launch_bounds__(kColNt) static_fwd_k(const double* __restrict__ c, const float* __restrict__ x,
                                                       double2* __restrict__ w, int lgN1, int lgN2) {
  __shared__ double2 rt[2 * kRoots], A[kRoots], B[kRoots];
  dep_trigger();
  const int N2 = 1 << lgN2, j1 = blockIdx.x;
  const bool isx = blockIdx.y != 0;
  for (int j2 = threadIdx.x; j2 < N2; j2 += kColNt) {
    const int p = j1 + (j2 << lgN1);
    A[j2] = isx ? make_double2((double)x[2 * p], (double)x[2 * p + 1]) : make_double2(c[2 * p], c[2 * p + 1]);
  }
  load_roots(rt);
  const double2* r = fft64_tile<-1>(A, B, lgN2, 1, rt);
  double2* o = w + ((int64_t)blockIdx.y << (lgN1 + lgN2));
  const int sh = kMaxLgN + 1 - (lgN1 + lgN2);   // w_N^q = w_16384^(q << sh)
  for (int k2 = threadIdx.x; k2 < N2; k2 += kColNt) o[(k2 << lgN1) + j1] = dmul(r[k2], root_at(rt, (j1 * k2) << sh));
}

// Launch 2: rows (u, N2 - u), or 0 and N2/2 for u = 0.
__global__ void __launch_bounds__(kMidNt) static_mid_k(double2* w, int lgN1, int lgN2, int transpose) {
  __shared__ double2 rt[2 * kRoots], A[4 * kRoots / 2], B[4 * kRoots / 2];   // N1 <= 64
  dep_trigger();
  const int N1 = 1 << lgN1, N2 = 1 << lgN2, lgN = lgN1 + lgN2, u = blockIdx.x;
  const int row[2] = {u, u == 0 ? N2 / 2 : N2 - u};
  load_roots(rt);
  dep_wait();
  // vectors 0, 1: the rows of c; 2, 3: of x
  for (int t = threadIdx.x; t < 4 << lgN1; t += kMidNt) {
    const int v = t >> lgN1, q = t & (N1 - 1);
    A[t] = __ldcg(w + ((int64_t)(v >> 1) << lgN) + ((int64_t)row[v & 1] << lgN1) + q);
  }
  double2* r = fft64_tile<-1>(A, B, lgN1, 4, rt);
  double2* o = r == A ? B : A;
  const double sc = 1.0 / (double)(1 << lgN);
  const int sh = kMaxLgN + 1 - (lgN + 1);   // w_2N^k = w_16384^(k << sh)
  // pairs: u > 0: (u, q) ~ (N2 - u, N1 - 1 - q), N1 of them; u = 0: row 0
  // q ~ (N1 - q) mod N1, row N2/2 q ~ N1 - 1 - q
  const int cnt = u ? N1 : N1 + 1;
  for (int t = threadIdx.x; t < cnt; t += kMidNt) {
    int ea, eb, k;
    if (u) {
      ea = t;
      eb = N1 + N1 - 1 - t;
      k = u + (t << lgN2);
    } else if (t <= N1 / 2) {
      ea = t;
      eb = (N1 - t) & (N1 - 1);
      k = t << lgN2;
    } else {
      const int q = t - N1 / 2 - 1;
      ea = N1 + q;
      eb = N1 + N1 - 1 - q;
      k = N2 / 2 + (q << lgN2);
    }
    const double2 ph = root_at(rt, k << sh);
    double2 F[2][2];   // [c, x][bin k, bin k + N] of the real spectra
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const double2 za = r[(2 * v << lgN1) + ea], zb = r[(2 * v << lgN1) + eb];
      const double2 E = make_double2(0.5 * (za.x + zb.x), 0.5 * (za.y - zb.y));
      const double2 O = make_double2(0.5 * (za.y + zb.y), -0.5 * (za.x - zb.x));
      const double2 wo = dmul(ph, O);
      F[v][0] = dadd(E, wo);
      F[v][1] = dsub(E, wo);
    }
    double2 Y[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) Y[b] = dmul(transpose ? F[0][b] : dconj(F[0][b]), F[1][b]);
    const double2 E = make_double2(0.5 * (Y[0].x + Y[1].x), 0.5 * (Y[0].y + Y[1].y));
    const double2 D = make_double2(0.5 * (Y[0].x - Y[1].x), 0.5 * (Y[0].y - Y[1].y));
    const double2 O = dmul(dconj(ph), D);
    // self-pairs (ea == eb) agree on both sides
    o[eb] = make_double2(sc * (E.x + O.y), sc * (O.x - E.y));
    o[ea] = make_double2(sc * (E.x - O.y), sc * (E.y + O.x));
  }
  r = fft64_tile<+1>(o, r, lgN1, 2, rt);
  const int sh4 = kMaxLgN + 1 - lgN;
  for (int t = threadIdx.x; t < 2 << lgN1; t += kMidNt) {
    const int k2 = row[t >> lgN1], j1 = t & (N1 - 1);
    w[((int64_t)k2 << lgN1) + j1] = dmul(r[t], dconj(root_at(rt, (j1 * k2) << sh4)));
  }
}

// Launch 3: column blockIdx.x of the result.
// (w is read through L2: a read-only load could be moved above the wait for
// the launch that writes it)
__global__ void __launch_bounds__(kColNt) static_inv_k(const double2* w, float* __restrict__ y, int lgN1, int lgN2) {
  __shared__ double2 rt[2 * kRoots], A[kRoots], B[kRoots];
  dep_trigger();
  const int N2 = 1 << lgN2, j1 = blockIdx.x;
  load_roots(rt);
  dep_wait();
  for (int k2 = threadIdx.x; k2 < N2; k2 += kColNt) A[k2] = __ldcg(w + (k2 << lgN1) + j1);
  const double2* r = fft64_tile<+1>(A, B, lgN2, 1, rt);
  for (int j2 = threadIdx.x; j2 < N2; j2 += kColNt) {
    const int p = j1 + (j2 << lgN1);
    y[2 * p] = (float)r[j2].x;
    y[2 * p + 1] = (float)r[j2].y;
  }
}

// Programmatic dependent launch: the roots are in shared memory when the
// launch in front ends.
template <typename K, typename... A>
cudaError_t launch_dep(K kern, int grid, int nt, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(nt);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace
}  // namespace csk

using namespace csk;

extern "C" cs_status cs_circulant_apply_static(int64_t n, const double* c, const float* x, float* y,
                                               int transpose, void* stream) {
  if (!c || !x || !y) return CS_ERR_ARG;
  if (n < 64 || n > kStaticMaxN || (n & (n - 1)) != 0) return CS_ERR_UNSUPPORTED;
  // An error the caller left pending on this thread is not this call's: leave
  // it in place (peek does not clear it) and launch nothing.
  if (cudaPeekAtLastError() != cudaSuccess) return CS_ERR_CUDA;
  double2* base = nullptr;
  cudaError_t e = scratch_address(&base);
  if (e != cudaSuccess) return CS_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int lgN = 0;
  while ((int64_t(2) << lgN) < n) ++lgN;
  const int lgN1 = lgN / 2, lgN2 = lgN - lgN1;
  static_fwd_k<<<dim3(1u << lgN1, 2), kColNt, 0, s>>>(c, x, base, lgN1, lgN2);
  if (cudaGetLastError() != cudaSuccess) return CS_ERR_CUDA;
  if (launch_dep(static_mid_k, 1 << (lgN2 - 1), kMidNt, s, base, lgN1, lgN2, transpose ? 1 : 0) != cudaSuccess ||
      launch_dep(static_inv_k, 1 << lgN1, kColNt, s, (const double2*)base, y, lgN1, lgN2) != cudaSuccess) {
    cudaGetLastError();   // this call's own error, reported by its status
    return CS_ERR_CUDA;
  }
  return CS_OK;
}
