// select.cu -- Eq. 2 and Eq. 3 on materialised log-probabilities (the unfused
// path behind pced_contrastive_select).
//   shat_k(v) = (1 + beta_k) lp_k(v) - beta_k lp_0(v) + gamma log r_k,  k = 1..N
//   y = argmax_v max_k shat_k(v)
// Pass 1: a cluster of SEL_CLUSTER CTAs per (SEL_CHUNK tokens, query) takes the
// max over experts per token and the chunk's best token; pass 2: one warp per
// query reduces the chunk records.  Ties: highest score, then lowest token id,
// then lowest expert index (the amateur, row 0, never competes).
//
// What bounds it: a few MB per query, so latency until the rows are tens of
// MB and the loads after that.  One CTA per 4096 tokens left most SMs idle
// (32 CTAs at V = 128256, one query) and each thread waited for one load at a
// time: 28.6 us + 2.8 us of a second launch for 9 rows, 128 us for 16 x 17
// rows.  Now a thread has SEL_TOK tokens of SEL_ROWS experts in flight, four
// CTAs share a chunk (their bests meet in the first one's shared memory, so
// the workspace still holds one record per SEL_CHUNK tokens), and the second
// kernel's launch is set up beside the first (programmatic launch).  Neither
// this kernel nor adacad.cu's triggers its dependents early; with a trigger at
// their start beta, select and relevance in a graph took longer, us: 33 rows of
// V = 128256 34.4 against 25.1, 9 rows 16.3 against 15.7, 4 x 9 rows of V = 50000
// 18.8 against 16.3 (the dependents start once every CTA is running and then
// share the SMs with them; what of that costs the time was not taken apart).
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"

namespace pced {

namespace cg = cooperative_groups;

constexpr int SEL_THREADS = 256;
constexpr int SEL_TOK = 4;      // tokens of a thread
constexpr int SEL_ROWS = 4;     // expert rows loaded at a time
constexpr int SEL_CLUSTER = 4;  // CTAs per chunk record
constexpr int SEL_CHUNK = SEL_CLUSTER * SEL_THREADS * SEL_TOK;
constexpr int SEL_MAX_N = 255;
constexpr int SEL_NONE = 0x7fffffff;

struct Cand {
  float s;
  int v, k;
};
__device__ __forceinline__ bool cand_better(const Cand& x, const Cand& y) {
  return x.s > y.s || (x.s == y.s && (x.v < y.v || (x.v == y.v && x.k < y.k)));
}
__device__ __forceinline__ Cand warp_best(Cand c) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Cand d;
    d.s = __shfl_xor_sync(0xffffffffu, c.s, o);
    d.v = __shfl_xor_sync(0xffffffffu, c.v, o);
    d.k = __shfl_xor_sync(0xffffffffu, c.k, o);
    if (cand_better(d, c)) c = d;
  }
  return c;
}

// lp, beta and r are plain pointers, as in adacad.cu: the launch before may
// still be writing them when this one starts.
__global__ void __cluster_dims__(SEL_CLUSTER, 1, 1) __launch_bounds__(SEL_THREADS)
    select_dense_kernel(const float* lp, const float* beta, const float* r, float gamma, int N, int V, Cand* rec) {
  cg::cluster_group cluster = cg::this_cluster();
  const int b = blockIdx.y, tid = threadIdx.x, n1 = N + 1;
  __shared__ float bt[SEL_MAX_N], bias[SEL_MAX_N];
  __shared__ Cand wbest[SEL_THREADS / 32], cbest[SEL_CLUSTER];
  cluster.barrier_arrive();  // waited for before the first CTA's shared memory is written
  pdl_wait();
  for (int k = tid; k < N; k += SEL_THREADS) {
    bt[k] = beta[b * N + k];
    bias[k] = gamma * logf(fminf(fmaxf(r[b * N + k], 1e-8f), 1.0f));
  }
  const float* lp0 = lp + (int64_t)b * n1 * V;
  const int v0 = blockIdx.x * (SEL_THREADS * SEL_TOK) + tid;
  float a0[SEL_TOK], s[SEL_TOK];
  int kk[SEL_TOK];
#pragma unroll
  for (int j = 0; j < SEL_TOK; ++j) {
    const int v = v0 + j * SEL_THREADS;
    a0[j] = v < V ? lp0[v] : 0.f;
    s[j] = -INFINITY;
    kk[j] = SEL_NONE;
  }
  __syncthreads();
  for (int k0 = 1; k0 <= N; k0 += SEL_ROWS) {
    float x[SEL_ROWS][SEL_TOK];
#pragma unroll
    for (int u = 0; u < SEL_ROWS; ++u)
#pragma unroll
      for (int j = 0; j < SEL_TOK; ++j) {
        const int v = v0 + j * SEL_THREADS;
        x[u][j] = k0 + u <= N && v < V ? lp0[(int64_t)(k0 + u) * V + v] : 0.f;
      }
#pragma unroll
    for (int u = 0; u < SEL_ROWS; ++u) {
      const int k = k0 + u;
      if (k > N) break;
#pragma unroll
      for (int j = 0; j < SEL_TOK; ++j) {
        const float y = (1.f + bt[k - 1]) * x[u][j] - bt[k - 1] * a0[j] + bias[k - 1];
        if (y > s[j] || (y == s[j] && k < kk[j])) {  // k rises: a tie keeps the lower expert
          s[j] = y;
          kk[j] = k;
        }
      }
    }
  }
  Cand best{-INFINITY, SEL_NONE, SEL_NONE};
#pragma unroll
  for (int j = 0; j < SEL_TOK; ++j) {
    const int v = v0 + j * SEL_THREADS;
    const Cand c{s[j], v, kk[j]};
    if (v < V && kk[j] != SEL_NONE && cand_better(c, best)) best = c;
  }
  best = warp_best(best);
  if ((tid & 31) == 0) wbest[tid >> 5] = best;
  __syncthreads();
  if (tid < 32) {
    best = warp_best(tid < SEL_THREADS / 32 ? wbest[tid] : Cand{-INFINITY, SEL_NONE, SEL_NONE});
  }
  cluster.barrier_wait();
  if (tid == 0) *cluster.map_shared_rank(cbest + cluster.block_rank(), 0) = best;
  cluster.sync();
  if (tid == 0 && cluster.block_rank() == 0) {
#pragma unroll
    for (int i = 1; i < SEL_CLUSTER; ++i)
      if (cand_better(cbest[i], best)) best = cbest[i];
    rec[(int64_t)b * (gridDim.x / SEL_CLUSTER) + blockIdx.x / SEL_CLUSTER] = best;
  }
}

__global__ void __launch_bounds__(32)
    select_reduce_kernel(const Cand* rec, int nchunks, int32_t* token, int32_t* expert, float* score) {
  const int b = blockIdx.x;
  pdl_wait();
  Cand best{-INFINITY, SEL_NONE, SEL_NONE};
#pragma unroll 4
  for (int i = threadIdx.x; i < nchunks; i += 32) {
    const Cand c = rec[(int64_t)b * nchunks + i];
    if (cand_better(c, best)) best = c;
  }
  best = warp_best(best);
  if (threadIdx.x == 0) {
    token[b] = best.v;
    expert[b] = best.k;
    score[b] = best.s;
  }
}

}  // namespace pced

using namespace pced;
using namespace pced_host;

extern "C" size_t pced_contrastive_select_workspace_size(int32_t B, int32_t N, int32_t V) {
  if (B < 1 || N < 1 || V < 1) return 0;
  const int64_t nchunks = (V + SEL_CHUNK - 1) / SEL_CHUNK;
  Carver c(nullptr);
  c.take<Cand>((size_t)(B * nchunks));
  return 256 + c.used();
}

extern "C" pced_status pced_contrastive_select(const float* logprobs, const float* beta, const float* r, float gamma,
                                               int32_t B, int32_t N, int32_t V, int32_t* token, int32_t* expert,
                                               float* score, void* workspace, size_t workspace_bytes, void* stream) {
  if (!logprobs || !beta || !r || !token || !expert || !score || !workspace)
    return fail(PCED_ERR_INVALID_ARG, "pced_contrastive_select: null pointer");
  if (B < 1 || N < 1 || V < 1 || B > 65535) return fail(PCED_ERR_INVALID_ARG, "pced_contrastive_select: bad sizes");
  if (N > SEL_MAX_N) return fail(PCED_ERR_UNSUPPORTED, "pced_contrastive_select: N > %d", SEL_MAX_N);
  if (!isfinite(gamma)) return fail(PCED_ERR_INVALID_ARG, "pced_contrastive_select: gamma not finite");
  if (((uintptr_t)workspace) & 255u || workspace_bytes < pced_contrastive_select_workspace_size(B, N, V))
    return fail(PCED_ERR_WORKSPACE, "pced_contrastive_select: workspace too small or misaligned");
  if (num_sms() <= 0) return fail(PCED_ERR_NO_DEVICE, "pced_contrastive_select: no CUDA device");
  const int nchunks = (V + SEL_CHUNK - 1) / SEL_CHUNK;
  Carver cv((char*)workspace + 256);
  Cand* rec = cv.take<Cand>((size_t)B * nchunks);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = launch_pdl(select_dense_kernel, dim3(nchunks * SEL_CLUSTER, B), SEL_THREADS, 0, s, logprobs, beta, r,
                             gamma, N, V, rec);
  if (e != cudaSuccess) return cuda_status(e, "select launch");
  e = launch_pdl(select_reduce_kernel, dim3(B), 32, 0, s, (const Cand*)rec, nchunks, token, expert, score);
  if (e != cudaSuccess) return cuda_status(e, "select reduce launch");
  return PCED_OK;
}
