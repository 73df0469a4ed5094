// Batched solver: many independent instances A_i = P_i C(c_i) of uneven size.
// Every instance with n <= CS_BATCH_MAX_N is solved by one CTA that keeps its
// iterate on chip for all iterations (cs_small.cu), one launch per
// power-of-two size class.  Larger instances have their own plan's buffers
// and tables but are iterated together: each pass of an iteration is one
// grouped launch over the tiles of all instances of one length (cs_group.cu),
// and the lengths run side by side as branches of one captured CUDA graph.
// Instances whose n is 7-smooth but not a power of two go to the mixed-radix
// solver of cs_smooth.cu (one persistent launch per solve over all of them).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <map>
#include <new>
#include <numeric>
#include <vector>

#include "../../include/cs.h"
#include "cs_fft.cuh"
#include "cs_internal.h"

namespace csk {
namespace {

constexpr int NSIDE_MAX = 4;    // side streams of the size-class launches (within CUDA's default 8 queues)

struct BatchDesc {
  int n, lgn, m;
  int pad0;
  int64_t noff;   // offset of x / z / state in the concatenated n-vectors
  int64_t moff;   // offset of y in the concatenated m-vectors
  int64_t itab;   // ISTA table offset (n/4 + 1 entries)
  int64_t atab;   // ADMM table offset (n/2 + 1 entries)
};

// ---------------------------------------------------------------- plan time

__global__ void tab_admm1_b_k(const double* __restrict__ abs2, int64_t count, const int* __restrict__ inst,
                              const BatchDesc* __restrict__ descs, const double* __restrict__ rho,
                              const double* __restrict__ sigma, float* __restrict__ tb) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count) return;
  const int i = inst[t];
  tb[t] = (float)(1.0 / ((double)descs[i].n * (rho[i] * abs2[t] + sigma[i])));
}

// rows of one instance as int32, range and repeats checked (mask: n bits, zero)
__global__ void batch_rows_k(const int64_t* __restrict__ rows, int64_t m, int64_t n, uint32_t* mask,
                             int32_t* __restrict__ rows32, int* status) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int64_t r = rows[i];
  if (r < 0 || r >= n) { atomicOr(status, STS_BAD_ROW); return; }
  const uint32_t bit = 1u << (r & 31);
  if (atomicOr(mask + (r >> 5), bit) & bit) atomicOr(status, STS_DUP_ROW);
  rows32[i] = (int32_t)r;
}

inline unsigned nb256(int64_t c) { return (unsigned)((c + 255) / 256); }

}  // namespace
}  // namespace csk

using namespace csk;

struct cs_batch_s {
  int count = 0;
  cudaStream_t stream = nullptr;
  std::vector<int64_t> n, m, noff, moff;
  std::vector<int> small;           // instances solved by the single-CTA kernels, largest first
  std::vector<int> large;           // instances solved by their own plan
  std::vector<int> smooth_ids;      // 7-smooth, not power-of-two n: the mixed-radix solver
  SmoothSet* smooth = nullptr;
  std::vector<cs_plan_t> plans;     // per large instance
  // grouped launches over the large instances (in the order of `large`,
  // which is by length): one chain of passes per length
  struct Chain {
    Geo gi, ga;
    int col_i0, n_col_i, mid_i0, n_mid_i, col_a0, n_col_a, mid_a0, n_mid_a;   // ranges of the maps
    cudaStream_t cap;             // capture-only stream of this chain (the first uses Group::cap)
    cudaEvent_t done;
  };
  struct Group {
    int count = 0;
    std::vector<GroupDesc> hdesc;
    std::vector<Chain> chains;
    GroupDesc* desc = nullptr;
    KParams *kps_i = nullptr, *kps_a0 = nullptr, *kps_a1 = nullptr;
    CallArgs* ca = nullptr;
    int2 *map_col_i = nullptr, *map_mid_i = nullptr, *map_col_a = nullptr, *map_mid_a = nullptr;
    cudaStream_t cap = nullptr;
    cudaEvent_t fork = nullptr;
    std::map<uint64_t, cudaGraphExec_t> graphs;
  } grp;
  struct Class {
    int lgn, start, count, side;    // instances order[start, start + count) have n = 2^lgn
  };
  std::vector<Class> classes;
  int nside = NSIDE_MAX;
  cudaStream_t side[NSIDE_MAX] = {};
  cudaEvent_t side_done[NSIDE_MAX] = {};
  cudaEvent_t fork = nullptr;
  BatchDesc* descs = nullptr;
  SmallInst* insts = nullptr;       // in the order of `small`
  SmallScalars* sc = nullptr;
  float4* tA = nullptr;
  float2* tB = nullptr;
  float2* tc = nullptr;
  double* abs2 = nullptr;
  float* tb = nullptr;
  int* tb_inst = nullptr;           // instance of every ADMM table entry
  double* drho = nullptr;
  double* dsigma = nullptr;
  int32_t* rows32 = nullptr;
  float2* tw = nullptr;             // stage twiddles of every transform length in use
  int* status = nullptr;
  int64_t ntot = 0, mtot = 0, atab_tot = 0;
  std::vector<double> host_rho, host_sigma;
};

namespace {

void batch_free(cs_batch_s* b) {
  if (!b) return;
  for (cs_plan_t p : b->plans)
    if (p) cs_plan_destroy(p);
  smooth_free(b->smooth);
  void* bufs[] = {b->descs, b->insts, b->sc,     b->tA,     b->tB, b->tc,   b->abs2,
                  b->tb,    b->tb_inst, b->drho, b->dsigma, b->rows32, b->tw, b->status};
  for (void* q : bufs)
    if (q) cudaFree(q);
  for (int k = 0; k < NSIDE_MAX; ++k) {
    if (b->side[k]) cudaStreamDestroy(b->side[k]);
    if (b->side_done[k]) cudaEventDestroy(b->side_done[k]);
  }
  if (b->fork) cudaEventDestroy(b->fork);
  auto& G = b->grp;
  for (auto& kv : G.graphs) cudaGraphExecDestroy(kv.second);
  void* gb[] = {G.desc, G.kps_i, G.kps_a0, G.kps_a1, G.ca, G.map_col_i, G.map_mid_i, G.map_col_a, G.map_mid_a};
  for (void* q : gb)
    if (q) cudaFree(q);
  for (auto& ch : G.chains) {
    if (ch.cap && ch.cap != G.cap) cudaStreamDestroy(ch.cap);
    if (ch.done) cudaEventDestroy(ch.done);
  }
  if (G.fork) cudaEventDestroy(G.fork);
  if (G.cap) cudaStreamDestroy(G.cap);
  delete b;
}

template <typename T>
cudaError_t balloc(T** p, size_t count) {
  return cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(T) + 256);
}

cs_status cstat(cudaError_t e) {
  return e == cudaSuccess ? CS_OK : (e == cudaErrorMemoryAllocation ? CS_ERR_NOMEM : CS_ERR_CUDA);
}

bool pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }

int ilog2(int64_t v) {
  int l = 0;
  while ((int64_t(1) << l) < v) ++l;
  return l;
}

// Side streams wait for the work already on the batch's stream ...
cudaError_t fork_sides(cs_batch_s* b) {
  cudaError_t e = cudaEventRecord(b->fork, b->stream);
  for (int k = 0; k < b->nside && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->side[k], b->fork, 0);
  return e;
}

// ... and the batch's stream waits for all of theirs.
cudaError_t join_sides(cs_batch_s* b) {
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < b->nside && e == cudaSuccess; ++k) {
    e = cudaEventRecord(b->side_done[k], b->side[k]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->side_done[k], 0);
  }
  return e;
}

// Run `enqueue` on the batch's stream as a cached CUDA graph under `key`.
template <class F>
cudaError_t run_group_graph(cs_batch_s* b, uint64_t key, F&& enqueue) {
  auto& G = b->grp;
  auto it = G.graphs.find(key);
  if (it == G.graphs.end()) {
    cudaError_t e = cudaStreamBeginCapture(G.cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    cudaError_t e2 = enqueue(G.cap);
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(G.cap, &graph);
    if (e2 != cudaSuccess || e != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      return e2 != cudaSuccess ? e2 : e;
    }
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return e;
    it = G.graphs.emplace(key, exec).first;
  }
  return cudaGraphLaunch(it->second, b->stream);
}

// T iterations of Algorithm 1 on the instances of one length: per iteration
// four grouped passes (C x, residual, C^T r, update).
cudaError_t enqueue_chain_ista(const cs_batch_s::Group& G, const cs_batch_s::Chain& c, int T, cudaStream_t s) {
  auto col = [&](ColKind k) { return launch_col_multi(k, c.gi, G.kps_i, G.map_col_i + c.col_i0, c.n_col_i, s); };
  auto mid = [&](MidKind k) { return launch_mid_multi(k, c.gi, G.kps_i, G.map_mid_i + c.mid_i0, c.n_mid_i, s); };
  cudaError_t e = col(COL_LOAD);
  for (int t = 0; t < T && e == cudaSuccess; ++t) {
    e = mid(MID_FWD);
    if (e == cudaSuccess) e = col(COL_RESIDUAL);
    if (e == cudaSuccess) e = mid(MID_ADJ);
    if (e == cudaSuccess) e = col(t + 1 < T ? COL_ISTA : COL_ISTA_LAST);
  }
  return e;
}

// T iterations of Algorithm 3 on the instances of one length: per iteration
// the grouped x-update (mid pass) and elementwise steps (column pass); the
// last one writes z.
cudaError_t enqueue_chain_admm(const cs_batch_s::Group& G, const cs_batch_s::Chain& c, int T, cudaStream_t s) {
  auto col = [&](ColKind k, const KParams* kps) {
    return launch_col_multi(k, c.ga, kps, G.map_col_a + c.col_a0, c.n_col_a, s);
  };
  cudaError_t e = col(COL_ADMM_INIT, G.kps_a0);
  for (int t = 0; t < T && e == cudaSuccess; ++t) {
    e = launch_mid_multi(MID_ADMM, c.ga, G.kps_a0, G.map_mid_a + c.mid_a0, c.n_mid_a, s);
    const bool last = t + 1 == T;
    if (e == cudaSuccess) e = col(last ? COL_ADMM_LAST : COL_ADMM, last ? G.kps_a1 : G.kps_a0);
  }
  return e;
}

// Every length's chain as a branch of the captured graph, forked from `s` and
// joined back.  Lengths are independent, and a chain's passes only fill the
// chip where it has many instances: side by side they fill each other's
// partial waves, and a short length does not wait for a long one's passes.
template <class F>
cudaError_t enqueue_chains(cs_batch_s* b, cudaStream_t s, F&& chain) {
  auto& G = b->grp;
  cudaError_t e = cudaEventRecord(G.fork, s);
  for (auto& c : G.chains) {
    if (e == cudaSuccess && c.cap != s) e = cudaStreamWaitEvent(c.cap, G.fork, 0);
    if (e == cudaSuccess) e = chain(c, c.cap);
    if (c.cap == s) continue;
    if (e == cudaSuccess) e = cudaEventRecord(c.done, c.cap);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, c.done, 0);
  }
  return e;
}

}  // namespace

extern "C" {

cs_status cs_batch_plan(cs_batch_t* out, int count, const int64_t* n, const int64_t* m, const int64_t* rows,
                        const double* c, void* stream) {
  if (!out || count < 1 || !n || !m || !rows || !c) return CS_ERR_ARG;
  *out = nullptr;
  for (int i = 0; i < count; ++i) {
    const bool p2 = pow2(n[i]) && n[i] >= 64 && n[i] <= (int64_t(1) << 21);
    if (!p2 && !smooth_size(n[i])) return CS_ERR_UNSUPPORTED;
    if (m[i] < 1 || m[i] > n[i]) return CS_ERR_ARG;
  }
  cs_batch_s* b = new (std::nothrow) cs_batch_s();
  if (!b) return CS_ERR_NOMEM;
  b->count = count;
  b->stream = static_cast<cudaStream_t>(stream);

  cudaStream_t s = b->stream;
  b->n.assign(n, n + count);
  b->m.assign(m, m + count);
  b->noff.resize(count);
  b->moff.resize(count);
  std::vector<BatchDesc> hd(count);
  int64_t no = 0, mo = 0, it = 0, at = 0;
  for (int i = 0; i < count; ++i) {
    b->noff[i] = no;
    b->moff[i] = mo;
    BatchDesc& d = hd[i];
    d.n = (int)n[i];
    d.lgn = ilog2(n[i]);
    d.m = (int)m[i];
    d.pad0 = 0;
    d.noff = no;
    d.moff = mo;
    d.itab = it;
    d.atab = at;
    no += n[i];
    mo += m[i];
    if (!pow2(n[i])) {
      b->smooth_ids.push_back(i);
    } else if (n[i] <= CS_BATCH_MAX_N) {
      b->small.push_back(i);
      it += n[i] / 4 + 1;
      at += n[i] / 2 + 1;
    } else {
      b->large.push_back(i);
    }
  }
  b->ntot = no;
  b->mtot = mo;
  b->atab_tot = at;
  std::stable_sort(b->small.begin(), b->small.end(), [&](int a, int c2) { return n[a] > n[c2]; });
  std::stable_sort(b->large.begin(), b->large.end(), [&](int a, int c2) { return n[a] > n[c2]; });
  // The size-class launches of the small instances go to the side streams
  // longest first, each to the stream with the least work so far (cost ~ n
  // per iteration and wave; a wave is what the chip holds of the class's ADMM
  // CTAs, one per SM at n = 8192 and more below); the grouped launches of the
  // large instances run on the batch's stream.
  for (size_t j = 0; j < b->small.size();) {
    const int lg = hd[b->small[j]].lgn;
    size_t e = j;
    while (e < b->small.size() && hd[b->small[e]].lgn == lg) ++e;
    b->classes.push_back({lg, (int)j, (int)(e - j), 0});
    j = e;
  }
  {
    struct Item { double cost; int kind, idx; };
    std::vector<Item> items;
    for (size_t j = 0; j < b->classes.size(); ++j) {
      const auto& cl = b->classes[j];
      int wave = 0;
      const cudaError_t e = small_class_wave(cl.lgn, &wave);
      if (e != cudaSuccess) {
        batch_free(b);
        return cstat(e);
      }
      items.push_back({(double)(int64_t(1) << cl.lgn) * (double)((cl.count + wave - 1) / wave), 0, (int)j});
    }
    std::stable_sort(items.begin(), items.end(), [](const Item& a, const Item& c2) { return a.cost > c2.cost; });
    double load[NSIDE_MAX] = {};
    for (const Item& itm : items) {
      const int k = (int)(std::min_element(load, load + b->nside) - load);
      load[k] += itm.cost;
      b->classes[itm.idx].side = k;
    }
  }
  auto fail = [&](cs_status e) {
    batch_free(b);
    return e;
  };
#define CS_B_TRY(expr)                          \
  do {                                          \
    cs_status e_ = cstat(expr);                 \
    if (e_ != CS_OK) return fail(e_);           \
  } while (0)
  for (int k = 0; k < b->nside; ++k) {
    CS_B_TRY(cudaStreamCreateWithFlags(&b->side[k], cudaStreamNonBlocking));
    CS_B_TRY(cudaEventCreateWithFlags(&b->side_done[k], cudaEventDisableTiming));
  }
  CS_B_TRY(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming));
  // large instances: their own plans (buffers, tables, masks) on the batch's
  // stream, and the parameters of the grouped launches over all of them
  for (size_t j = 0; j < b->large.size(); ++j) {
    const int i = b->large[j];
    cs_plan_t p = nullptr;
    const cs_status st = (cs_status)plan_for_group(&p, n[i], m[i], rows + b->moff[i], c + b->noff[i], s);
    if (st != CS_OK) return fail(st);
    b->plans.push_back(p);
  }
  if (!b->large.empty()) {
    auto& G = b->grp;
    G.count = (int)b->large.size();
    CS_B_TRY(cudaStreamCreateWithFlags(&G.cap, cudaStreamNonBlocking));
    CS_B_TRY(cudaEventCreateWithFlags(&G.fork, cudaEventDisableTiming));
    CS_B_TRY(balloc(&G.desc, G.count));
    CS_B_TRY(balloc(&G.kps_i, G.count));
    CS_B_TRY(balloc(&G.kps_a0, G.count));
    CS_B_TRY(balloc(&G.kps_a1, G.count));
    CS_B_TRY(balloc(&G.ca, G.count));
    std::vector<KParams> ki(G.count), ka0(G.count), ka1(G.count);
    std::vector<int2> mci, mmi, mca, mma;
    for (int j = 0; j < G.count; ++j) {
      const int i = b->large[j];
      const PlanView v = plan_view(b->plans[j]);
      GroupDesc d = v.desc;
      d.noff = b->noff[i];
      d.moff = b->moff[i];
      G.hdesc.push_back(d);
      ki[j] = v.kp_i;
      ka0[j] = v.kp_a;
      ki[j].ca = ka0[j].ca = G.ca + j;
      ka1[j] = ka0[j];
      ka1[j].flags = FL_WRITE_STATE;
      // grouped launches take 4096-value tiles of a fixed set of shapes
      if (j == 0 || n[i] != n[b->large[j - 1]]) {
        cs_batch_s::Chain ch{};
        ch.gi = d.gi;
        ch.ga = d.ga;
        ch.col_i0 = (int)mci.size();
        ch.mid_i0 = (int)mmi.size();
        ch.col_a0 = (int)mca.size();
        ch.mid_a0 = (int)mma.size();
        G.chains.push_back(ch);
        auto& c = G.chains.back();
        if (G.chains.size() == 1) c.cap = G.cap;
        else CS_B_TRY(cudaStreamCreateWithFlags(&c.cap, cudaStreamNonBlocking));
        CS_B_TRY(cudaEventCreateWithFlags(&c.done, cudaEventDisableTiming));
        for (const Geo* g : {&d.gi, &d.ga}) {
          const cudaError_t eg = init_multi_kernels(*g);
          if (eg == cudaErrorInvalidValue) return fail(CS_ERR_UNSUPPORTED);
          CS_B_TRY(eg);
        }
      }
      auto& ch = G.chains.back();
      ch.n_col_i += d.gi.col_ctas;
      ch.n_mid_i += d.gi.mid_ctas;
      ch.n_col_a += d.ga.col_ctas;
      ch.n_mid_a += d.ga.mid_ctas;
      for (int t = 0; t < d.gi.col_ctas; ++t) mci.push_back(make_int2(j, t));
      for (int t = 0; t < d.gi.mid_ctas; ++t) mmi.push_back(make_int2(j, t));
      for (int t = 0; t < d.ga.col_ctas; ++t) mca.push_back(make_int2(j, t));
      for (int t = 0; t < d.ga.mid_ctas; ++t) mma.push_back(make_int2(j, t));
    }
    CS_B_TRY(balloc(&G.map_col_i, mci.size()));
    CS_B_TRY(balloc(&G.map_mid_i, mmi.size()));
    CS_B_TRY(balloc(&G.map_col_a, mca.size()));
    CS_B_TRY(balloc(&G.map_mid_a, mma.size()));
    CS_B_TRY(cudaMemcpyAsync(G.desc, G.hdesc.data(), G.count * sizeof(GroupDesc), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.kps_i, ki.data(), G.count * sizeof(KParams), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.kps_a0, ka0.data(), G.count * sizeof(KParams), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.kps_a1, ka1.data(), G.count * sizeof(KParams), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.map_col_i, mci.data(), mci.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.map_mid_i, mmi.data(), mmi.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.map_col_a, mca.data(), mca.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaMemcpyAsync(G.map_mid_a, mma.data(), mma.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    CS_B_TRY(cudaStreamSynchronize(s));
  }
  if (!b->small.empty()) {
    // stage twiddles of the lengths in use (ISTA 2^(lgn-1), ADMM 2^lgn)
    std::map<int, int64_t> twoff;
    int64_t twn = 0;
    for (int i : b->small)
      for (int lg : {hd[i].lgn - 1, hd[i].lgn})
        if (twoff.emplace(lg, twn).second) twn += (small_tw_count(lg, true) + 1) & ~1;
    const int ns = (int)b->small.size();
    int64_t ms = 0;
    for (int i : b->small) ms += m[i];
    CS_B_TRY(balloc(&b->descs, count));
    CS_B_TRY(balloc(&b->insts, ns));
    CS_B_TRY(balloc(&b->sc, count));
    CS_B_TRY(balloc(&b->tA, it));
    CS_B_TRY(balloc(&b->tB, it));
    CS_B_TRY(balloc(&b->tc, at));
    CS_B_TRY(balloc(&b->abs2, at));
    CS_B_TRY(balloc(&b->tb, at));
    CS_B_TRY(balloc(&b->tb_inst, at));
    CS_B_TRY(balloc(&b->drho, count));
    CS_B_TRY(balloc(&b->dsigma, count));
    CS_B_TRY(balloc(&b->rows32, ms));
    CS_B_TRY(balloc(&b->tw, twn));
    CS_B_TRY(balloc(&b->status, 1));
    CS_B_TRY(cudaMemsetAsync(b->status, 0, sizeof(int), s));
    CS_B_TRY(cudaMemcpyAsync(b->descs, hd.data(), count * sizeof(BatchDesc), cudaMemcpyHostToDevice, s));
    for (const auto& kv : twoff) CS_B_TRY(launch_small_tw(kv.first, true, b->tw + kv.second, s));
    std::vector<SmallInst> hs_inst(ns);
    ms = 0;
    for (int k = 0; k < ns; ++k) {
      const BatchDesc& d = hd[b->small[k]];
      SmallInst& q = hs_inst[k];
      q = SmallInst{};
      q.tA = b->tA + d.itab;
      q.tB = b->tB + d.itab;
      q.tc = b->tc + d.atab;
      q.tb = b->tb + d.atab;
      q.tw_i = b->tw + twoff[d.lgn - 1];
      q.tw_a = b->tw + twoff[d.lgn];
      q.rows = b->rows32 + ms;
      q.status = b->status;
      q.noff = d.noff;
      q.moff = d.moff;
      q.m = d.m;
      q.id = b->small[k];
      ms += d.m;
    }
    CS_B_TRY(cudaMemcpyAsync(b->insts, hs_inst.data(), ns * sizeof(SmallInst), cudaMemcpyHostToDevice, s));
    std::vector<int> inst(at);
    int64_t nmax = 0, mmax = 0;
    for (int i : b->small) {
      nmax = std::max(nmax, n[i]);
      mmax = std::max(mmax, m[i]);
      std::fill(inst.begin() + hd[i].atab, inst.begin() + hd[i].atab + n[i] / 2 + 1, i);
    }
    CS_B_TRY(cudaMemcpyAsync(b->tb_inst, inst.data(), at * sizeof(int), cudaMemcpyHostToDevice, s));
    double* dc = nullptr;
    double2 *fa = nullptr, *fb = nullptr;
    int64_t* drows = nullptr;
    uint32_t* dmask = nullptr;
    CS_B_TRY(balloc(&dmask, nmax / 32));
    CS_B_TRY(balloc(&dc, nmax));
    CS_B_TRY(balloc(&fa, nmax));
    CS_B_TRY(balloc(&fb, nmax));
    CS_B_TRY(balloc(&drows, mmax));
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < ns; ++k) {
      const int i = b->small[k];
      const BatchDesc& d = hd[i];
      if (e == cudaSuccess) e = cudaMemcpyAsync(dc, c + d.noff, n[i] * sizeof(double), cudaMemcpyHostToDevice, s);
      if (e == cudaSuccess) e = cudaMemcpyAsync(drows, rows + d.moff, m[i] * sizeof(int64_t), cudaMemcpyHostToDevice, s);
      if (e == cudaSuccess) e = cudaMemsetAsync(dmask, 0, n[i] / 32 * sizeof(uint32_t), s);
      double2* chat = nullptr;
      if (e == cudaSuccess) e = launch_fft64(dc, fa, fb, n[i], &chat, s);
      if (e == cudaSuccess)
        e = launch_small_tables(chat, n[i], b->tA + d.itab, b->tB + d.itab, b->tc + d.atab, b->abs2 + d.atab, s);
      if (e == cudaSuccess) {
        batch_rows_k<<<nb256(m[i]), 256, 0, s>>>(drows, m[i], n[i], dmask, const_cast<int32_t*>(hs_inst[k].rows),
                                                  b->status);
        e = cudaGetLastError();
      }
      // the staging buffers are reused by the next instance: keep the order
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    cudaFree(dmask);
    cudaFree(dc);
    cudaFree(fa);
    cudaFree(fb);
    cudaFree(drows);
    CS_B_TRY(e);
    int hs = 0;
    CS_B_TRY(cudaMemcpy(&hs, b->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (hs & (STS_BAD_ROW | STS_DUP_ROW)) return fail(CS_ERR_ARG);
    b->host_rho.assign(count, -1.0);
    b->host_sigma.assign(count, -1.0);
  }
  if (!b->status) {
    CS_B_TRY(balloc(&b->status, 1));
    CS_B_TRY(cudaMemsetAsync(b->status, 0, sizeof(int), s));
  }
  if (!b->smooth_ids.empty()) {
    const cs_status st = (cs_status)smooth_plan(&b->smooth, b->smooth_ids.data(), (int)b->smooth_ids.size(), n, m,
                                                b->noff.data(), b->moff.data(), rows, c, b->status, s);
    if (st != CS_OK) return fail(st);
  }
  CS_B_TRY(cudaStreamSynchronize(s));
  for (int k = 0; k < b->nside; ++k) CS_B_TRY(cudaStreamSynchronize(b->side[k]));
#undef CS_B_TRY
  *out = b;
  return CS_OK;
}

cs_status cs_batch_destroy(cs_batch_t b) {
  if (!b) return CS_ERR_ARG;
  cudaStreamSynchronize(b->stream);
  for (int k = 0; k < b->nside; ++k)
    if (b->side[k]) cudaStreamSynchronize(b->side[k]);
  batch_free(b);
  return CS_OK;
}

cs_status cs_batch_ista(cs_batch_t b, const float* y, const float* lambda, const float* tau, int iters, float* x) {
  if (!b || !y || !lambda || !tau || !x || iters < 0) return CS_ERR_ARG;
  for (int i = 0; i < b->count; ++i)
    if (!(lambda[i] >= 0.f) || !(tau[i] > 0.f) || !std::isfinite(lambda[i]) || !std::isfinite(tau[i])) return CS_ERR_ARG;
  cudaStream_t s = b->stream;
  if (!b->small.empty() && iters > 0) {
    std::vector<SmallScalars> h(b->count);
    for (int i = 0; i < b->count; ++i) {
      h[i] = SmallScalars{};
      h[i].thr = (float)((double)tau[i] * (double)lambda[i]);
      h[i].tau = tau[i];
    }
    const cs_status st = cstat(cudaMemcpyAsync(b->sc, h.data(), b->count * sizeof(SmallScalars),
                                               cudaMemcpyHostToDevice, s));
    if (st != CS_OK) return st;
  }
  cs_status st = cstat(fork_sides(b));
  if (!b->large.empty() && st == CS_OK) {
    auto& G = b->grp;
    std::vector<CallArgs> h(G.count);
    for (int j = 0; j < G.count; ++j) {
      const int i = b->large[j];
      h[j] = CallArgs{};
      h[j].src = x + b->noff[i];   // COL_LOAD transforms x(0) in natural order
      h[j].x = G.hdesc[j].xi_t;    // the iterate lives in tile order during the solve
      h[j].thr = (float)((double)tau[i] * (double)lambda[i]);
      h[j].tau = tau[i];
    }
    st = cstat(cudaMemcpyAsync(G.ca, h.data(), G.count * sizeof(CallArgs), cudaMemcpyHostToDevice, s));
    if (st == CS_OK) st = cstat(launch_group_scatter_y(G.desc, G.count, y, 0, b->status, s));
    if (st == CS_OK && iters > 0) {
      st = cstat(launch_group_ista_in(G.desc, G.count, x, s));
      if (st == CS_OK)
        st = cstat(run_group_graph(b, (uint64_t(1) << 40) | (uint32_t)iters,
                                   [&](cudaStream_t cs) {
                                     return enqueue_chains(b, cs, [&](const cs_batch_s::Chain& c, cudaStream_t t) {
                                       return enqueue_chain_ista(G, c, iters, t);
                                     });
                                   }));
      if (st == CS_OK) st = cstat(launch_group_ista_out(G.desc, G.count, x, s));
    }
  }
  if (iters > 0) {
    for (const auto& cl : b->classes) {
      if (st != CS_OK) break;
      st = cstat(launch_small_class(false, cl.lgn - 1, b->insts + cl.start, cl.count, b->sc, y, x, iters,
                                    b->side[cl.side]));
    }
  }
  const cs_status sj = cstat(join_sides(b));
  if (st == CS_OK && sj == CS_OK && b->smooth) st = cstat(smooth_ista(b->smooth, y, lambda, tau, iters, x, s));
  return st != CS_OK ? st : sj;
}

cs_status cs_batch_admm(cs_batch_t b, const float* y, const float* lambda, const float* rho, int iters, float* z) {
  if (!b || !y || !lambda || !rho || !z || iters < 0) return CS_ERR_ARG;
  for (int i = 0; i < b->count; ++i)
    if (!(lambda[i] >= 0.f) || !(rho[i] > 0.f) || !std::isfinite(lambda[i]) || !std::isfinite(rho[i])) return CS_ERR_ARG;
  cudaStream_t s = b->stream;
  cs_status st = CS_OK;
  if (!b->small.empty() && iters == 0) {
    for (int i : b->small) {
      st = cstat(cudaMemsetAsync(z + b->noff[i], 0, b->n[i] * sizeof(float), s));
      if (st != CS_OK) return st;
    }
  }
  if (!b->small.empty() && iters > 0) {
    // sigma = rho, tau1 = tau2 = 1 (as cs_admm); B's spectrum re-tabulated when rho changes
    bool changed = false;
    std::vector<SmallScalars> h(b->count);
    for (int i = 0; i < b->count; ++i) {
      const double r = rho[i];
      if (r != b->host_rho[i]) changed = true;
      b->host_rho[i] = r;
      b->host_sigma[i] = r;
      h[i] = SmallScalars{};
      h[i].thr = (float)((double)lambda[i] / r);
      h[i].rho = (float)r;
      h[i].sigma = (float)r;
      h[i].tau1 = 1.f;
      h[i].tau2 = 1.f;
      h[i].d_on = (float)(1.0 / (1.0 + r));
      h[i].d_off = (float)(1.0 / r);
    }
    st = cstat(cudaMemcpyAsync(b->sc, h.data(), b->count * sizeof(SmallScalars), cudaMemcpyHostToDevice, s));
    if (st != CS_OK) return st;
    if (changed) {
      st = cstat(cudaMemcpyAsync(b->drho, b->host_rho.data(), b->count * sizeof(double), cudaMemcpyHostToDevice, s));
      if (st == CS_OK)
        st = cstat(cudaMemcpyAsync(b->dsigma, b->host_sigma.data(), b->count * sizeof(double),
                                   cudaMemcpyHostToDevice, s));
      if (st != CS_OK) return st;
      tab_admm1_b_k<<<nb256(b->atab_tot), 256, 0, s>>>(b->abs2, b->atab_tot, b->tb_inst, b->descs, b->drho,
                                                        b->dsigma, b->tb);
    }
  }
  st = cstat(fork_sides(b));
  if (!b->large.empty() && st == CS_OK) {
    // sigma = rho, tau1 = tau2 = 1 (as cs_admm), zero start
    auto& G = b->grp;
    std::vector<CallArgs> h(G.count);
    for (int j = 0; j < G.count && st == CS_OK; ++j) {
      const int i = b->large[j];
      const double r = rho[i];
      st = cstat(plan_admm_table(b->plans[j], r, r, s));
      h[j] = CallArgs{};
      h[j].z = G.hdesc[j].az;
      h[j].mu = G.hdesc[j].amu;
      h[j].nu = G.hdesc[j].anu;
      h[j].v = G.hdesc[j].av;
      h[j].thr = (float)((double)lambda[i] / r);
      h[j].rho = (float)r;
      h[j].sigma = (float)r;
      h[j].tau1 = 1.f;
      h[j].tau2 = 1.f;
      h[j].d_on = (float)(1.0 / (1.0 + r));
      h[j].d_off = (float)(1.0 / r);
    }
    if (st == CS_OK) st = cstat(cudaMemcpyAsync(G.ca, h.data(), G.count * sizeof(CallArgs), cudaMemcpyHostToDevice, s));
    if (st == CS_OK) st = cstat(launch_group_admm_zero(G.desc, G.count, s));
    if (st == CS_OK) st = cstat(launch_group_scatter_y(G.desc, G.count, y, 1, b->status, s));
    if (st == CS_OK && iters > 0)
      st = cstat(run_group_graph(b, (uint64_t(2) << 40) | (uint32_t)iters,
                                 [&](cudaStream_t cs) {
                                   return enqueue_chains(b, cs, [&](const cs_batch_s::Chain& c, cudaStream_t t) {
                                     return enqueue_chain_admm(G, c, iters, t);
                                   });
                                 }));
    if (st == CS_OK) st = cstat(launch_group_admm_out(G.desc, G.count, z, s));
  }
  if (iters > 0) {
    for (const auto& cl : b->classes) {
      if (st != CS_OK) break;
      st = cstat(launch_small_class(true, cl.lgn, b->insts + cl.start, cl.count, b->sc, y, z, iters,
                                    b->side[cl.side]));
    }
  }
  const cs_status sj = cstat(join_sides(b));
  if (st == CS_OK && sj == CS_OK && b->smooth) st = cstat(smooth_admm(b->smooth, y, lambda, rho, iters, z, s));
  return st != CS_OK ? st : sj;
}

cs_status cs_batch_status_sync(cs_batch_t b) {
  if (!b) return CS_ERR_ARG;
  cs_status st = cstat(cudaStreamSynchronize(b->stream));
  if (st != CS_OK) return st;
  for (cs_plan_t p : b->plans) {
    const cs_status ps = cs_status_sync(p);
    if (ps != CS_OK) return ps;
  }
  if (b->status) {
    int hs = 0;
    st = cstat(cudaMemcpy(&hs, b->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st != CS_OK) return st;
    st = cstat(cudaMemset(b->status, 0, sizeof(int)));   // reported once, as cs_status_sync
    if (st != CS_OK) return st;
    if (hs & STS_TIMEOUT) return CS_ERR_TIMEOUT;
    if (hs & STS_NONFINITE) return CS_ERR_NONFINITE;
  }
  return CS_OK;
}

}  // extern "C"
