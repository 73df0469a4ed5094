// Internal declarations shared by the host runtime and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct cs_plan_s;

namespace csk {

// Four-step geometry of one complex FFT of length N = N1 * N2, stored as an
// N2 x N1 row-major array (element p = j1 + N1 * j2).
//   column pass: length-N2 FFTs down the columns, G columns per CTA
//   mid pass:    length-N1 FFTs along the rows, U row pairs per CTA; row
//                pair unit u holds rows (u, N2 - u) for u >= 1 and rows
//                (0, N2/2) for u = 0, so every frequency k meets its mirror
//                N - k inside one CTA.
struct Geo {
  int N, lgN, N1, lgN1, N2, lgN2;
  int G, lgG, col_ctas;
  int U, lgU, mid_ctas;
  int tile;            // mid pass: complex values per CTA; threads = tile / 16 (tile / 8 with mid_r8)
  int col_tile;        // column pass: complex values per CTA; threads = col_tile / 16 (/ 8 with col_r8)
  int col_r8, mid_r8;  // 1: the pass runs 8 values per thread and radix-8 stages (small tiles, see make_geo)
  int tw1_full, tw2_full;   // 1: tws1 / tws2 hold every stage twiddle (see make_geo)
  int twod;            // 1: 2D DFT of the N2 x N1 array (no four-step twiddle; pairs (k2, k1) ~ (-k2, -k1))
  const float2* tw1;   // exp(-2 pi i q / (2 N1)), q < 2 N1
  const float2* tw2;   // exp(-2 pi i q / N2),     q < N2
  const float2* twl;   // exp(-2 pi i q / N),      q < N1
  const float2* twr;   // exp(-2 pi i q / (2 N)),  q < N2
  const float2* tw1h;  // exp(-2 pi i q / N1),     q < N1
  const float2* tws1;  // stage-major twiddles of the length-N1 FFT
  const float2* tws2;  // stage-major twiddles of the length-N2 FFT
};

constexpr int NSTAT = 8;

// Statistic slots (partials[block * NSTAT + slot]).
enum : int {
  ST_ERR2 = 0,   // ||x - x*||^2           (ISTA: x_t, ADMM: z_t)
  ST_DX2 = 1,    // ISTA ||x_t - x_{t-1}||^2, ADMM ||x_t - z_t||^2
  ST_X2 = 2,     // ||x_t||^2 (ADMM ||z_t||^2)
  ST_L1 = 3,     // ISTA ||x_{t-1}||_1, ADMM ||z_t||_1
  ST_R2 = 4,     // ||y - A x||^2 (ISTA at x_{t-1}, ADMM at x_t)
  ST_NONFIN = 5  // count of non-finite iterate values
};

// Plan-constant device pointers, passed by value to every pass kernel.
struct PlanPtrs {
  const float2* Wi;          // exchange buffer a pass reads (W unless a pass keeps its input)
  float2* W;                 // exchange buffer, complex[n]
  const uint32_t* mask;      // rows of Omega, one bit per row in tile order, [n/32]
  const uint32_t* prefix;    // set bits before word w, [n/32]
  const float* ys;           // y in tile order of its rows, [m]
  double* partials;          // [max_ctas * NSTAT]
  double* stats;             // [NSTAT] finalised sums
  const float4* tab_ista;    // (P, Q) per pair slot, real-FFT geometry (see op_real)
  const float2* tab_admm_c;  // chat_k per pair slot, complex-n geometry
  const float* tab_admm_b;   // 1 / (n (rho |chat_k|^2 + sigma)) per pair slot
  int* status;               // device status word
  // unrolled-ISTA gradient (cs_grad) only
  const float2* W2;          // column transform of the vector a reverse mid pass correlates with
  float4* gacc;              // per pair slot: accumulated spectrum at (k, k + N)
  double* gpart;             // per column CTA: accumulated dL/dtheta
  // unrolled-ADMM gradient (cs_grad_admm) only
  float2* gacc_a;            // per pair slot of the complex-n geometry: accumulated spectrum of dL/dc at k
};

// Per-call arguments, resident in device memory and written by a one-thread
// kernel at the start of each call (kernel parameters are captured when the
// launch is enqueued, so this is safe while earlier work is in flight).
struct CallArgs {
  const float* src;     // load source (x, scattered r, power vector)
  float* dst;           // store target
  float* aux;           // power iteration: normalised u
  const float* xtrue;   // monitor ground truth or null
  float* x;             // ISTA iterate / ADMM x output (may be null)
  float* z;
  float* mu;
  float* nu;
  float* v;
  float thr;            // ISTA tau*lambda, ADMM lambda/sigma
  float tau;            // ISTA step
  float rho, sigma, tau1, tau2, d_on, d_off;
};

struct KParams {
  Geo geo;
  PlanPtrs pp;
  const CallArgs* ca;
  int flags;
};

enum : int { FL_STATS = 1, FL_WRITE_STATE = 2, FL_POWER_SCALE = 4 };

// Column-pass epilogues and mid-pass spectrum operators.
enum ColKind : int {
  COL_LOAD = 0,        // forward FFT of src (real-FFT geometry: src float[2N])
  COL_LOAD_SCALED,     // same, times 1/sqrt(stats[ST_X2]); copies it to aux
  COL_STORE,           // inverse FFT, store to dst
  COL_MASK,            // inverse, keep rows of Omega, forward
  COL_RESIDUAL,        // inverse, r = M (y - Cx), forward
  COL_ISTA,            // inverse, x <- eta(x + tau g), forward
  COL_ISTA_LAST,       // same without the forward FFT
  COL_POWER_OUT,       // inverse, w -> dst, stats <u, w>, ||w||^2
  COL_ADMM_INIT,       // complex-n geometry: forward FFT of (v) + i (z - nu)
  COL_ADMM,            // inverse, Algorithm 3 elementwise steps, forward
  COL_ADMM_LAST,       // same without the forward FFT
  // unrolled-ISTA gradient (real-FFT geometry, vectors in tile order)
  COL_LOADT,           // forward FFT of x (tile order)
  COL_ISTA_SEG,        // inverse, z <- eta(x + tau g) (x kept), forward
  COL_GRAD_W,          // w = dst on the support of z -> mu, dtheta partials, forward
  COL_GRAD_MASK,       // inverse, q = M C w, aux += tau P C w, forward
  COL_GRAD_G,          // inverse, dst = mu - tau C^T q
  COL_GRAD_GW,         // COL_GRAD_G of one step and COL_GRAD_W of the one before it
  // unrolled-ADMM gradient (complex-n geometry, vectors in tile order)
  COL_ADMM_SEG,        // as COL_ADMM (no state written), and s = x + nu -> aux
  COL_ADMM_REV,        // inverse (b' + i C b'), reverse of one Algorithm 3 iteration, forward FFT of (p' + i x')
  COL_STORE_RE         // inverse FFT, real part -> dst
};
enum MidKind : int {
  MID_FWD = 0, MID_ADJ, MID_ADMM,
  MID_FWD_CORR,        // MID_FWD of w, and gacc += conj(r^) w^ with r's column transform in W2
  MID_ADJ_CORR,        // MID_ADJ of q, and gacc -= conj(q^) x^ with x's in W2
  MID_FROM_ACC,        // tau / N times the packed spectrum of gacc -> inverse FFT -> W
  // unrolled-ADMM gradient (complex-n geometry)
  MID_ADMM_REV,        // FFTs of W (p' + i x') and W2 (the forward pair): b' = B (C^T p' + x'), dL/dc spectrum
                       // -> gacc_a, inverse FFT of b' + i C b' -> W
  MID_ADMM_FROM_ACC    // the Hermitian spectrum of gacc_a -> inverse FFT -> W
};

// Launchers (cs_passes.cu).  Return cudaGetLastError() of the launch.
cudaError_t launch_col(ColKind kind, const KParams& kp, cudaStream_t s);
cudaError_t launch_mid(MidKind kind, const KParams& kp, cudaStream_t s);
size_t pass_smem_bytes(int tile);
// Shared-memory attributes of the pass kernels that geometry g launches.
cudaError_t init_col_kernels(const Geo& g);
cudaError_t init_mid_kernels(const Geo& g);
// Grouped launches over many plans of one length (batched solves, cs_group.cu;
// 4096-value tiles): CTA b runs tile map[b].y of the plan whose parameters are
// kps[map[b].x] (both device arrays), g their common geometry.
cudaError_t launch_col_multi(ColKind kind, const Geo& g, const KParams* kps, const int2* map, int nctas,
                             cudaStream_t s);
cudaError_t launch_mid_multi(MidKind kind, const Geo& g, const KParams* kps, const int2* map, int nctas,
                             cudaStream_t s);
cudaError_t init_multi_kernels(const Geo& g);

// Small kernels (cs_aux.cu).
cudaError_t launch_set_args(const CallArgs& a, CallArgs* dst, cudaStream_t s);
enum : int { SEQ_X = 1, SEQ_Z = 2, SEQ_AUX = 4 };
cudaError_t launch_set_args_seq(const CallArgs& a, int adv, int64_t stride, int count, CallArgs* dst, cudaStream_t s);
cudaError_t launch_finalize(const double* partials, int nblk, double* stats, cudaStream_t s);
cudaError_t launch_twiddle(float2* dst, int count, int64_t M, cudaStream_t s);
cudaError_t launch_fft64(const double* c, double2* a, double2* b, int64_t n, double2** out,
                         cudaStream_t s);
cudaError_t launch_tab_ista(const double2* chat, const Geo& g, int64_t n, float4* tabA, cudaStream_t s);
// 2D: chat2 is the n0 x n1 FP64 spectrum (row-major); g the 2D geometry.
cudaError_t launch_tab_ista2d(const double2* chat2, const Geo& g, int64_t n0, int64_t n1, float4* tabA,
                              cudaStream_t s);
cudaError_t launch_tab_admm2d(const double2* chat2, const Geo& g, int64_t n0, int64_t n1, float2* tabc,
                              double* abs2, cudaStream_t s);
// FP64 2D DFT of the real n0 x n1 array c2 (row-major); a, b work space of
// n0 n1 values each; *out is whichever holds the result.
cudaError_t launch_fft64_2d(const double* c2, double2* a, double2* b, int64_t n0, int64_t n1, double2** out,
                            cudaStream_t s);
// Pair slots of the mid pass (spectrum tables' length).
inline int64_t tab_count(const Geo& g) { return ((int64_t)(g.N2 >> 1) << g.lgN1) + (g.twod ? 2 : 1); }
cudaError_t launch_stage_tw(float2* dst, int lgL, int lgRmax, bool full, cudaStream_t s);
cudaError_t launch_tab_admm(const double2* chat, const Geo& g, int64_t n, float2* tabc,
                            double* abs2, cudaStream_t s);
cudaError_t launch_tab_admm_b(const double* abs2, int count, int64_t n, double rho,
                              double sigma, float* tabb, cudaStream_t s);
// Row mask of Omega in the tile order of geometry g (packed: two spatial rows
// per complex element, the real-FFT geometry).
cudaError_t launch_build_mask(const int64_t* rows, int64_t m, int64_t n, const Geo& g, int packed,
                              uint32_t* mask, int* status, cudaStream_t s);
// Natural order <-> tile order of the column pass (float2 elements when
// complex_elems, else float), g.N elements.
cudaError_t launch_to_tile(const void* nat, void* tiled, const Geo& g, int complex_elems, cudaStream_t s);
cudaError_t launch_from_tile(const void* tiled, void* nat, const Geo& g, int complex_elems, cudaStream_t s);
cudaError_t launch_prefix(const uint32_t* mask, int64_t words, uint32_t* prefix,
                          cudaStream_t s);
cudaError_t launch_row_pos(const int64_t* rows, int64_t m, const Geo& g, int packed,
                           const uint32_t* mask, const uint32_t* prefix, int32_t* pos,
                           int32_t* rows32, cudaStream_t s);
cudaError_t launch_scatter_y(const float* y, const int32_t* pos, int64_t m, float* ys,
                             int* status, cudaStream_t s);
cudaError_t launch_gather_rows(const float* dense, const int32_t* rows32, int64_t m,
                               float* y, cudaStream_t s);
cudaError_t launch_scatter_rows(const float* r, const int32_t* rows32, int64_t m,
                                float* dense, cudaStream_t s);
cudaError_t launch_norm2(const float* x, int64_t n, double* partials, double* out,
                         cudaStream_t s);
cudaError_t launch_power_init(float* u, int64_t n, cudaStream_t s);
// out[0] = scale * sum(v[0 .. count)), summed in a fixed order in FP64.
cudaError_t launch_sum_scaled(const double* v, int count, float scale, float* out, cudaStream_t s);

// Single-CTA solves and products of short transforms (cs_small.cu): packed
// length N = n/2 for ISTA, the power iteration and the products, N = n for
// ADMM, N = 2^lgN <= 4096.  All vectors in natural order.
constexpr int SMALL_LG_MAX = 12;
enum SmallKind : int { SMALL_ISTA, SMALL_ADMM, SMALL_POWER, SMALL_FWD, SMALL_ADJ };
struct SmallArgs {
  const float4* tA;        // pair operator of the packed geometry, k in [0, N/2] (tA, tB)
  const float2* tB;
  const float2* tc;        // ADMM: c^_k and b^_k / n, k in [0, n/2]
  const float* tb;
  const float2* tw;        // stage twiddles
  const int32_t* rows;     // rows of Omega in the caller's order
  int m;
  const float* y;          // y (solves), r (A^T r)
  float* yo;               // A x
  float *x, *z, *mu, *nu, *v;   // ISTA: x; ADMM: the state (null: not returned)
  const float* xtrue;      // monitor ground truth in the plan's tile order, or null
  int lgN1, lgN2, lgG;     // of the geometry xtrue is tiled for
  double* stats;           // NSTAT sums of the last iteration, or null
  int* status;
  int iters, warm;
  float thr, tau, rho, sigma, tau1, tau2, d_on, d_off;
};
cudaError_t launch_small(SmallKind kind, int lgN, const SmallArgs& a, cudaStream_t s);
// Stage twiddles, small_tw_count values: `full` for the size classes, else for
// the solves and products of a plan (see SmallTw).
int small_tw_count(int lgN, bool full);
cudaError_t launch_small_tw(int lgN, bool full, float2* tw, cudaStream_t s);
// Pair-operator tables of one instance from its FP64 spectrum: tA, tB n/4 + 1
// values, tc, abs2 n/2 + 1 (null: no ADMM).
cudaError_t launch_small_tables(const double2* chat, int64_t n, float4* tA, float2* tB, float2* tc, double* abs2,
                                cudaStream_t s);

// Size classes of a batch: one CTA per instance (ISTA lgN = lgn - 1, ADMM
// lgN = lgn; n <= 8192 for both).
struct SmallInst {
  const float4* tA;
  const float2 *tB, *tc;
  const float* tb;
  const float2 *tw_i, *tw_a, *tw;
  const int32_t* rows;
  int* status;
  int64_t noff, moff;      // x / z and y in the caller's concatenated vectors
  int m, id;               // id: the instance's scalars
};
struct SmallScalars {      // per call and instance
  float thr, tau, rho, sigma, tau1, tau2, d_on, d_off;
};
// Instances of n = 2^lgn whose ADMM CTAs the device holds at a time (>= 1).
cudaError_t small_class_wave(int lgn, int* instances);
cudaError_t launch_small_class(bool admm, int lgN, const SmallInst* inst, int count, const SmallScalars* sc,
                               const float* y, float* xz, int iters, cudaStream_t s);

// Solves and products of middle-sized instances by one cluster of CTAs
// (cs_cluster.cu); geo the radix-8 geometry (packed, or complex-n for ADMM).
enum ClusterKind : int { CLUSTER_ISTA, CLUSTER_ADMM, CLUSTER_POWER, CLUSTER_FWD, CLUSTER_ADJ };
struct ClusterArgs {
  Geo geo;
  const float2* twn;               // exp(-2 pi i q / N), q < N
  const uint32_t *mask, *prefix;   // rows of Omega and compact y in the plan's tile order
  const float* ys;
  const float4* tab_i;
  const float2* tab_c;
  const float* tab_b;
  float *x, *z, *mu, *nu, *v;      // natural order (ISTA: x; ADMM: the state, null not returned; products: x -> z)
  const float* xtrue;              // tile order, or null
  double* partials;                // per CTA, with stats
  double* stats;                   // null: no statistics (power iteration: the sums themselves)
  int iters, warm;
  float thr, tau, rho, sigma, tau1, tau2, d_on, d_off;
};
bool cluster_init(const Geo& g, bool admm);
cudaError_t launch_cluster(ClusterKind kind, const ClusterArgs& a, cudaStream_t s);
int cluster_ctas();

// One plan of a grouped (batched) solve: what the grouped element-wise
// kernels need of it.
struct GroupDesc {
  Geo gi, ga;                  // real-FFT and complex-n geometry
  int64_t noff, moff, m;       // offsets of its x / z and y in the concatenated vectors; rows kept
  const int32_t* pos_i;        // compact position of y[i], real-FFT geometry
  float* ys_i;
  const int32_t* pos_a;        // the same, complex-n geometry
  float* ys_a;
  float* xi_t;                 // ISTA iterate (tile order of gi, float2[n/2])
  float *av, *az, *amu, *anu;  // ADMM state (tile order of ga)
};

// The plan's parameters of the pass kernels (flags 0, its own CallArgs), its
// geometries and buffers, for grouped launches (cs_api.cu).
struct PlanView {
  KParams kp_i, kp_a;          // real-FFT and complex-n geometry
  GroupDesc desc;
};
PlanView plan_view(cs_plan_s* p);
// A 1D plan whose passes use 4096-value tiles at every size (cs_plan's own
// argument checks apply): the geometry of the grouped launches.
int plan_for_group(cs_plan_s** out, int64_t n, int64_t m, const int64_t* rows, const double* c, void* stream);
// Re-tabulate the plan's ADMM inverse spectrum for (rho, sigma) when it holds
// another pair.
cudaError_t plan_admm_table(cs_plan_s* p, double rho, double sigma, cudaStream_t s);

// Grouped element-wise kernels over `count` plans (cs_aux.cu): compact y of
// every plan (geometry: 0 real-FFT, 1 complex-n; non-finite values latch
// STS_NONFINITE in *status); x (natural order) to and from the ISTA iterates;
// the zero ADMM state; z from the ADMM state.
cudaError_t launch_group_scatter_y(const GroupDesc* d, int count, const float* y, int geo, int* status,
                                   cudaStream_t s);
cudaError_t launch_group_ista_in(const GroupDesc* d, int count, const float* x, cudaStream_t s);
cudaError_t launch_group_ista_out(const GroupDesc* d, int count, float* x, cudaStream_t s);
cudaError_t launch_group_admm_zero(const GroupDesc* d, int count, cudaStream_t s);
cudaError_t launch_group_admm_out(const GroupDesc* d, int count, float* z, cudaStream_t s);

// Device status bits.
enum : int { STS_NONFINITE = 1, STS_TIMEOUT = 2, STS_BAD_ROW = 4, STS_DUP_ROW = 8 };

// Batched instances whose n is 7-smooth but not a power of two (cs_smooth.cu):
// mixed-radix FFTs, one persistent launch per solve.  smooth_plan takes the
// batch's arrays and the `count` instances ids[] (rows and c as the batch
// plan's; noff / moff their offsets); status is the batch's status word.
struct SmoothSet;
bool smooth_size(int64_t n);
int smooth_plan(SmoothSet** out, const int* ids, int count, const int64_t* n, const int64_t* m,
                const int64_t* noff, const int64_t* moff, const int64_t* rows, const double* c, int* status,
                cudaStream_t s);
cudaError_t smooth_ista(SmoothSet* q, const float* y, const float* lambda, const float* tau, int iters, float* x,
                        cudaStream_t s);
cudaError_t smooth_admm(SmoothSet* q, const float* y, const float* lambda, const float* rho, int iters, float* z,
                        cudaStream_t s);
void smooth_free(SmoothSet* q);

}  // namespace csk
