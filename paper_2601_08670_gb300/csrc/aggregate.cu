// aggregate.cu -- aggregation variants of the experts (appendix "Ablation of
// Expert Aggregation Rule": Mixture-of-Experts, a weighted sum, and
// Product-of-Experts, a weighted product, in probability space, with weights
// from the retrieval scores).  Reading (the paper prints no formula):
//   c_k(v) = (1 + beta_k) lp_k(v) - beta_k lp_0(v)      (Eq. 2 without the prior)
//   p_k = softmax_v c_k,  w_k = r~_k / sum_j r~_j       (r~: r clipped to [1e-8, 1])
//   MoE: agg(v) = log sum_k w_k p_k(v)     PoE: agg(v) = sum_k w_k log p_k(v)
//   token = argmax_v agg (lowest id on ties), score = agg(token),
//   expert = argmax_k w_k p_k(token) (lowest k on ties).
// Two launches over the materialised log-probabilities (S x V fp32): (1) a
// cluster of CTAs per (query, expert) forms the log-sum-exp of c_k; (2) per
// (query, chunk) the best aggregate and the best at another token; the last
// CTA of a query picks the token across chunks, attributes the expert and
// writes the step's results with both near-tie margins.  Every sum runs in a
// fixed order, so results do not depend on timing.
//
// What bounds them: latency for one query (a few MB in L2), the rows' bytes
// and one exp per entry and kernel for many.  (1) with a CTA, a fence and an
// arrival per 1024 entries and two exps per entry: 11-12 us for 8 experts of
// 128256 entries, 151 us for 16 x 16.  A thread now has AGG_UNROLL entries in
// flight and scales once per batch, and the cluster's sums meet in shared
// memory: 8.4 and 59 us.  (2) with one load in flight per thread: 13 and 65 us;
// with four tokens of four experts 9.4 and 37 us; the pick reads its chunk
// records four at a time instead of one after another (a step of 9 rows and
// four layers 238.5 -> 237.7 us).
#include <cooperative_groups.h>
#include <math.h>

#include "aggregate.cuh"
#include "select_key.cuh"

namespace pced {

namespace cg = cooperative_groups;

constexpr int AGG_THREADS = 256;     // selection kernel
constexpr int AGG_L_THREADS = 1024;  // log-sum-exp kernel
constexpr int AGG_FIN = 4;           // chunk records of a lane in flight (128 chunks: V = 128K)
constexpr int AGG_UNROLL = 8;        // entries of a thread in flight (log-sum-exp kernel)
constexpr int AGG_TOK = AGG_CHUNK / AGG_THREADS, AGG_ROWS = 4;  // tokens and expert rows in flight (selection)

__device__ __forceinline__ void agg_lse_merge(float& m, float& s, float m2, float s2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2;
    s = s2;
    return;
  }
  const float M = fmaxf(m, m2);
  s = s * expf(m - M) + s2 * expf(m2 - M);
  m = M;
}

// log-sum-exp over a warp of per-lane (m, s)
__device__ __forceinline__ void warp_lse(float& m, float& s) {
  const float M = warp_max(m);
  s = warp_sum(m == -INFINITY ? s : s * expf(m - M));
  m = M;
}

// (m, s) over the CTA's threads, in thread 0
__device__ __forceinline__ void block_lse(float& m, float& s, float2* red) {
  const int tid = threadIdx.x;
  warp_lse(m, s);
  __syncthreads();
  if ((tid & 31) == 0) red[tid >> 5] = make_float2(m, s);
  __syncthreads();
  if (tid < 32) {
    m = red[tid].x;
    s = red[tid].y;
    warp_lse(m, s);
  }
}

// grid (CTAs of a cluster, N, B): lse_k of (query b, expert k); with rec_stats also
// the rows' own log-sum-exps
__global__ void __launch_bounds__(AGG_L_THREADS) agg_partials_kernel(AggArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = blockIdx.x, nc = gridDim.x, k = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const int N = a.N, V = a.V;
  __shared__ float2 red[AGG_L_THREADS / 32], part[ROW_CLUSTER];
  cluster.barrier_arrive();  // waited for before the first CTA's shared memory is written
  pdl_launch_dependents();
  pdl_wait();
  const float* lp0 = a.lp + (int64_t)b * (N + 1) * V;
  const float* lpk = lp0 + (int64_t)(k + 1) * V;
  const float bt = a.beta[b * N + k];
  const int per = (V - 1) / nc + 1;
  const int64_t v0 = (int64_t)rank * per, v1 = min((int64_t)V, v0 + per);
  float m = -INFINITY, s = 0.f;
  for (int64_t v = v0 + tid; v < v1; v += AGG_UNROLL * AGG_L_THREADS) {
    float x[AGG_UNROLL], y[AGG_UNROLL];
#pragma unroll
    for (int u = 0; u < AGG_UNROLL; ++u) {
      const bool in = v + u * AGG_L_THREADS < v1;
      x[u] = in ? lpk[v + u * AGG_L_THREADS] : -INFINITY;
      y[u] = in ? lp0[v + u * AGG_L_THREADS] : 0.f;
    }
    float mn = m;
#pragma unroll
    for (int u = 0; u < AGG_UNROLL; ++u) {
      x[u] = (1.f + bt) * x[u] - bt * y[u];
      if (v + u * AGG_L_THREADS >= v1) x[u] = -INFINITY;  // whatever beta is
      mn = fmaxf(mn, x[u]);
    }
    if (m != -INFINITY) s *= expf(m - mn);
    m = mn;
#pragma unroll
    for (int u = 0; u < AGG_UNROLL; ++u)
      if (x[u] != -INFINITY) s += expf(x[u] - m);
  }
  block_lse(m, s, red);
  cluster.barrier_wait();
  if (tid == 0) *cluster.map_shared_rank(part + rank, 0) = make_float2(m, s);
  cluster.sync();
  if (rank == 0 && tid == 0) {
    for (int i = 1; i < nc; ++i) agg_lse_merge(m, s, part[i].x, part[i].y);
    a.lse_k[(int64_t)b * N + k] = m + logf(s);
  }
  // raw logits: the log-sum-exps of expert k's row and, for k = 0, the amateur's
  // (by other CTAs where there are some) from the LM head's tile records, in a fixed order
  for (int i = 0; a.rec_stats && i < (k == 0 ? 2 : 1); ++i) {
    if (rank != (i + 1) % nc) continue;
    const int64_t row = (int64_t)b * (N + 1) + (i == 0 ? k + 1 : 0);
    m = -INFINITY;
    s = 0.f;
    for (int j = tid; j < a.nrec; j += AGG_L_THREADS) {
      const float2 e = a.rec_stats[row * a.nrec + j];
      agg_lse_merge(m, s, e.x, e.y);
    }
    block_lse(m, s, red);
    if (tid == 0) a.lse_rows[row] = m + logf(s);
  }
}

// (value, token) order: larger value, then lower token
__device__ __forceinline__ bool agg_better(float v2, int t2, float v1, int t1) {
  return v2 > v1 || (v2 == v1 && t2 < t1);
}
// top-2 over disjoint token sets: (b1, t1) best, b2 best value at another token
__device__ __forceinline__ void agg_top2(float& b1, int& t1, float& b2, float r1, int rt, float r2) {
  if (agg_better(r1, rt, b1, t1)) {
    b2 = fmaxf(b1, r2);
    b1 = r1;
    t1 = rt;
  } else {
    b2 = fmaxf(b2, r1);
  }
}

// grid (nchunks, B).  rule 0 is Eq. 3 itself on the materialised
// log-probabilities: per token the best expert's score of Eq. 2 (the first
// step of a dynamic-beta decode selects this way, from the log-probabilities
// it has written for beta anyway); rules 1 and 2 are MoE and PoE.
template <int RULE>
__global__ void __launch_bounds__(AGG_THREADS) agg_select_kernel(AggArgs a) {
  const int c = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = a.N, V = a.V, n1 = N + 1;
  // w_s: r clipped; wn_s: normalised weights; lse_s: per-expert constants
  __shared__ float w_s[AGG_MAX_N], wn_s[AGG_MAX_N], lse_s[AGG_MAX_N], beta_s[AGG_MAX_N];
  __shared__ float wsum[AGG_THREADS / 32];
  __shared__ float bv_s[AGG_THREADS / 32], b2_s[AGG_THREADS / 32];
  __shared__ int bt_s[AGG_THREADS / 32];
  __shared__ int last;
  pdl_wait();
  if (c == 0 && b == 0 && tid == 0 && a.tile_ctr) *a.tile_ctr = 0;  // the next LM head claims its tiles from 0
  const float* lp0 = a.lp + (int64_t)b * n1 * V;
  const int v0 = c * AGG_CHUNK + tid;
  float l0[AGG_TOK], acc[AGG_TOK];
#pragma unroll
  for (int j = 0; j < AGG_TOK; ++j) {
    l0[j] = v0 + j * AGG_THREADS < V ? lp0[v0 + j * AGG_THREADS] : 0.f;
    acc[j] = RULE == 0 ? -INFINITY : 0.f;
  }
  float t = 0.f;
  for (int k = tid; k < N; k += AGG_THREADS) {
    const float w = fminf(fmaxf(a.r[b * N + k], 1e-8f), 1.0f);
    w_s[k] = w;
    t += w;
    beta_s[k] = a.beta[b * N + k];
    if (RULE == 0) {
      // the per-expert constant of Eq. 2: gamma log r_k (plus the log-sum-exps
      // when s_k are raw logits: z = lp + L)
      const float btk = beta_s[k];
      lse_s[k] = a.gamma * logf(w) + (a.raw_logits ? (1.f + btk) * a.lse[b * n1 + 1 + k] - btk * a.lse[b * n1] : 0.f);
    } else {
      lse_s[k] = a.lse_k[(int64_t)b * N + k];
    }
  }
  if (RULE != 0) {
    t = warp_sum(t);
    if (lane == 0) wsum[warp] = t;
    __syncthreads();
    t = 0.f;
    for (int w = 0; w < AGG_THREADS / 32; ++w) t += wsum[w];
    const float inv_w = 1.0f / t;
    for (int k = tid; k < N; k += AGG_THREADS) wn_s[k] = w_s[k] * inv_w;
  }
  __syncthreads();
  for (int k0 = 0; k0 < N; k0 += AGG_ROWS) {
    float x[AGG_ROWS][AGG_TOK];
#pragma unroll
    for (int u = 0; u < AGG_ROWS; ++u)
#pragma unroll
      for (int j = 0; j < AGG_TOK; ++j) {
        const int v = v0 + j * AGG_THREADS;
        x[u][j] = k0 + u < N && v < V ? lp0[(int64_t)(k0 + u + 1) * V + v] : 0.f;
      }
#pragma unroll
    for (int u = 0; u < AGG_ROWS; ++u) {
      const int k = k0 + u;
      if (k >= N) break;
      const float bk = beta_s[k], lk = lse_s[k], wk = RULE == 0 ? 0.f : wn_s[k];
#pragma unroll
      for (int j = 0; j < AGG_TOK; ++j) {
        const float ck = (1.f + bk) * x[u][j] - bk * l0[j];
        if (RULE == 0)
          acc[j] = fmaxf(acc[j], ck + lk);
        else if (RULE == 1)
          acc[j] += wk * expf(ck - lk);  // ck - lk = log p_k(v)
        else
          acc[j] += wk * (ck - lk);
      }
    }
  }
  // the chunk's best aggregate and token, and the best at another token
  float bv = -INFINITY, b2 = -INFINITY;
  int bt = 0x7fffffff;
#pragma unroll
  for (int j = 0; j < AGG_TOK; ++j)
    if (v0 + j * AGG_THREADS < V)
      agg_top2(bv, bt, b2, RULE == 1 ? logf(acc[j]) : acc[j], v0 + j * AGG_THREADS, -INFINITY);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, bv, o), s2 = __shfl_xor_sync(0xffffffffu, b2, o);
    const int t2 = __shfl_xor_sync(0xffffffffu, bt, o);
    agg_top2(bv, bt, b2, v2, t2, s2);
  }
  if (lane == 0) {
    bv_s[warp] = bv;
    bt_s[warp] = bt;
    b2_s[warp] = b2;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < AGG_THREADS / 32; ++w) agg_top2(bv, bt, b2, bv_s[w], bt_s[w], b2_s[w]);
    a.best[(int64_t)b * a.nchunks + c] = make_float2(bv, __int_as_float(bt));
    a.best2[(int64_t)b * a.nchunks + c] = b2;
    __threadfence();
    last = atomicAdd(a.qdone + b, 1) == a.nchunks - 1;
  }
  __syncthreads();
  if (!last || warp != 0) return;
  __threadfence();  // the other chunks' results of query b are visible
  const int t_step = a.step ? *a.step : 0;  // advances only once every query is through
  // best over the chunks (one warp, lanes over chunks, then a tree)
  float sv = -INFINITY, sv2 = -INFINITY;
  int st = 0x7fffffff;
  for (int j0 = lane; j0 < a.nchunks; j0 += 32 * AGG_FIN) {
    float2 e[AGG_FIN];
    float e2[AGG_FIN];
#pragma unroll
    for (int u = 0; u < AGG_FIN; ++u) {
      const int j = j0 + 32 * u;
      const bool in = j < a.nchunks;
      e[u] = in ? __ldcg(a.best + (int64_t)b * a.nchunks + j) : make_float2(-INFINITY, __int_as_float(0x7fffffff));
      e2[u] = in ? __ldcg(a.best2 + (int64_t)b * a.nchunks + j) : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < AGG_FIN; ++u) agg_top2(sv, st, sv2, e[u].x, __float_as_int(e[u].y), e2[u]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, sv, o), s2 = __shfl_xor_sync(0xffffffffu, sv2, o);
    const int t2 = __shfl_xor_sync(0xffffffffu, st, o);
    agg_top2(sv, st, sv2, v2, t2, s2);
  }
  if (st >= V) st = 0;  // no finite aggregate (degenerate rows): token 0
  // the expert: for Eq. 3 the best score at the token, for MoE / PoE the
  // one that puts the most weighted mass on it (log(w p)); lowest k on
  // ties, and the margin to the next one
  float bp = -INFINITY, bp2 = -INFINITY;
  int bk = 0x7fffffff;
  for (int k = lane; k < N; k += 32) {
    const float ck = (1.f + beta_s[k]) * lp0[(int64_t)(k + 1) * V + st] - beta_s[k] * lp0[st];
    agg_top2(bp, bk, bp2, RULE == 0 ? ck + lse_s[k] : logf(w_s[k]) + ck - lse_s[k], k, -INFINITY);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, bp, o), s2 = __shfl_xor_sync(0xffffffffu, bp2, o);
    const int t2 = __shfl_xor_sync(0xffffffffu, bk, o);
    agg_top2(bp, bk, bp2, v2, t2, s2);
  }
  if (bk >= N) bk = 0;
  if (a.lse_out)
    for (int j = lane; j < n1; j += 32) a.lse_out[b * n1 + j] = a.lse[b * n1 + j];
  if (lane != 0) return;
  a.qdone[b] = 0;
  if (a.key_out) {  // expert-partitioned step (rule 0): the reduction and the append come after
    a.key_out[b] = select_key(sv, st, a.expert_base + bk + 1);
    return;
  }
  if (a.token) a.token[b] = st;
  if (a.expert) a.expert[b] = bk + 1;
  if (a.score) a.score[b] = sv;
  if (a.step) {
    const int t = t_step;
    if (t >= 0 && t < a.max_steps) {
      a.history[(int64_t)b * a.max_steps + t] = st;
      if (a.expert_trace) a.expert_trace[(int64_t)b * a.max_steps + t] = bk + 1;
      if (a.score_trace) a.score_trace[(int64_t)b * a.max_steps + t] = sv;
      if (a.gap_trace) a.gap_trace[(int64_t)b * a.max_steps + t] = make_float2(sv - sv2, bp - bp2);
    } else {
      dev_flag(a.status, PCED_DEV_STEP_LIMIT);
    }
    __threadfence();
    if (atomicAdd(a.done_counter, 1) == a.B - 1) {
      if (t >= 0 && t < a.max_steps) *a.step = t + 1;  // at the limit t stays (as the commit does)
      *a.done_counter = 0;
      __threadfence();
    }
  }
}

cudaError_t agg_partials_launch(const AggArgs& a, bool pdl, cudaStream_t stream) {
  const int nc = pced_host::row_cluster((int64_t)a.B * a.N);
  return pced_host::launch_cluster(agg_partials_kernel, dim3(nc, a.N, a.B), nc, AGG_L_THREADS, 0, stream, pdl, a);
}

cudaError_t agg_select_launch(const AggArgs& a, bool pdl, cudaStream_t stream) {
  auto kernel = a.rule == 0 ? agg_select_kernel<0> : a.rule == 1 ? agg_select_kernel<1> : agg_select_kernel<2>;
  return pced_host::launch_kernel(kernel, dim3(a.nchunks, a.B), AGG_THREADS, 0, stream, pdl, a);
}

}  // namespace pced
