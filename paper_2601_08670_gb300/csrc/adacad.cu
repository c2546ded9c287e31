// adacad.cu -- dynamic contrast strength for the first generated token
// (paper Sec. 3 after Eq. 2: beta_0 is computed as in AdaCAD for the first
// generated token and kept fixed thereafter).  Reading: one beta per
// contextual expert, the Jensen-Shannon divergence in bits between the
// expert's next-token distribution p_k = exp(lp_k) and the amateur's
// p_0 = exp(lp_0):
//   beta[b][k-1] = 1/2 sum_v [ p_k log2(p_k / m) + p_0 log2(p_0 / m) ],  m = (p_k + p_0) / 2,
// in [0, 1].  With hi / lo the larger and smaller of the two log-probabilities
// the midpoint's is log m = hi + log1p(exp(lo - hi)) - log 2; terms in fp32.
//
// What bounds it: three exp and one log1p per entry and expert (and, past the
// L2, the rows).  A cluster of CTAs takes one (expert, query): the
// cluster's sums meet in the first CTA's shared memory, so there is no scratch,
// no counter to clear and no second pass.  (One CTA per 2048 entries left the
// last one to add 63 chunk sums one load after the other.  Experts of 128256
// entries, in a graph: 8 17.4 -> 9.8 us, 16 x 16 184 -> 110.)  A term without
// the midpoint's logarithm, exp(hi) (q + e (q + lo - hi)) with e = exp(lo - hi)
// and q = -log((1 + e) / 2), needs one exponential less (16 x 16: 86 us) and
// has half the error, but moves beta's last bit, which a score near zero
// magnifies to 2.5e-6 of itself.
//
// Sums are held as three fp32 numbers (sum3.cuh, no less exact than an fp64
// accumulator) and rounded once from fp64 at the end: this chip adds 64-bit
// numbers at 1/64 of the fp32 rate, so one fp64 conversion and addition per
// entry cost more than the entry's exponentials.  (Two fp32 numbers, 8.9 and 102
// us for the two sizes above, hold fewer bits than fp64.)  The order is fixed (thread,
// then xor trees over lanes and warps, then the CTAs in order), so the result
// does not depend on timing.
#include <cooperative_groups.h>
#include <math.h>

#include "adacad.cuh"
#include "sum3.cuh"

namespace pced {

namespace cg = cooperative_groups;

constexpr int ADA_THREADS = 1024;
constexpr int ADA_UNROLL = 4;  // entries of a thread in flight

__device__ __forceinline__ Sum3 warp_sum3(Sum3 p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    p = sum3_merge(p, Sum3{__shfl_xor_sync(0xffffffffu, p.s, o), __shfl_xor_sync(0xffffffffu, p.c, o),
                           __shfl_xor_sync(0xffffffffu, p.e, o)});
  return p;
}

__device__ __forceinline__ float jsd_term(float a, float b) {
  const float hi = fmaxf(a, b), lo = fminf(a, b);
  if (hi == -INFINITY) return 0.f;  // both probabilities are 0
  const float lm = hi + log1pf(expf(lo - hi)) - 0.69314718055994531f;  // log of the midpoint
  float t = 0.f;
  if (a > -INFINITY) t += expf(a) * (a - lm);
  if (b > -INFINITY) t += expf(b) * (b - lm);
  return t;
}

// grid (CTAs of a cluster, N, B), one cluster per (k - 1, b).  lp is a plain
// pointer: the launch before may still rewrite the rows when this one starts
// (the log-softmax pass does, in place), so its loads must not become
// non-coherent ones, which const __restrict__ allows.
__global__ void __launch_bounds__(ADA_THREADS)
    adacad_beta_kernel(const float* lp, int32_t N, int32_t V, float* beta) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = blockIdx.x, nc = gridDim.x, k = blockIdx.y + 1, b = blockIdx.z, tid = threadIdx.x;
  __shared__ Sum3 wsum[ADA_THREADS / 32], csum[ROW_CLUSTER];
  cluster.barrier_arrive();  // waited for before the first CTA's shared memory is written
  pdl_wait();  // dependents are launched when this ends: select.cu has the figures
  const float* l0 = lp + (int64_t)b * (N + 1) * V;
  const float* lk = l0 + (int64_t)k * V;
  const int per = (V - 1) / nc + 1;
  const int64_t v0 = (int64_t)rank * per, v1 = min((int64_t)V, v0 + per);
  Sum3 acc{0.f, 0.f, 0.f};
  int terms = 0;
  for (int64_t v = v0 + tid; v < v1; v += ADA_UNROLL * ADA_THREADS) {
    float x[ADA_UNROLL], y[ADA_UNROLL];
#pragma unroll
    for (int u = 0; u < ADA_UNROLL; ++u) {
      const bool in = v + u * ADA_THREADS < v1;
      x[u] = in ? lk[v + u * ADA_THREADS] : -INFINITY;
      y[u] = in ? l0[v + u * ADA_THREADS] : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < ADA_UNROLL; ++u) sum3_add(acc, jsd_term(x[u], y[u]));
    if ((terms += ADA_UNROLL) % SUM3_RUN == 0) sum3_settle(acc);
  }
  acc = warp_sum3(acc);
  if ((tid & 31) == 0) wsum[tid >> 5] = acc;
  __syncthreads();
  if (tid < 32) acc = warp_sum3(wsum[tid]);
  cluster.barrier_wait();
  if (tid == 0) *cluster.map_shared_rank(csum + rank, 0) = acc;
  cluster.sync();
  if (rank == 0 && tid == 0) {
    Sum3 t = csum[0];
    for (int i = 1; i < nc; ++i) t = sum3_merge(t, csum[i]);
    beta[(int64_t)b * N + k - 1] = (float)(sum3_value(t) * 0.72134752044448170);  // 1 / (2 ln 2)
  }
}

cudaError_t adacad_beta_launch(const float* lp, int32_t B, int32_t N, int32_t V, float* beta, bool pdl,
                               cudaStream_t stream) {
  const int nc = pced_host::row_cluster((int64_t)B * N);
  return pced_host::launch_cluster(adacad_beta_kernel, dim3(nc, N, B), nc, ADA_THREADS, 0, stream, pdl, lp, N, V,
                                   beta);
}

}  // namespace pced

using namespace pced;
using namespace pced_host;

extern "C" size_t pced_adacad_beta_workspace_size(int32_t B, int32_t N, int32_t V) {
  if (B < 1 || N < 1 || V < 1) return 0;
  // the kernel needs no scratch; the size that callers allocate by stays (8
  // bytes for each 2048 entries of an expert, 4 for each expert)
  Carver c(nullptr);
  c.take<double>((size_t)B * N * (((size_t)V + 2047) / 2048));
  c.take<int>((size_t)B * N);
  return c.used();
}

extern "C" pced_status pced_adacad_beta(const float* logprobs, int32_t B, int32_t N, int32_t V, float* beta,
                                        void* workspace, size_t workspace_bytes, void* stream) {
  if (!logprobs || !beta || !workspace) return fail(PCED_ERR_INVALID_ARG, "pced_adacad_beta: null pointer");
  if (B < 1 || N < 1 || V < 1 || B > 65535 || N > 65535)
    return fail(PCED_ERR_INVALID_ARG, "pced_adacad_beta: bad sizes (B=%d N=%d V=%d)", B, N, V);
  if (((uintptr_t)logprobs | (uintptr_t)beta) & 3u)
    return fail(PCED_ERR_INVALID_ARG, "pced_adacad_beta: pointers must be 4-byte aligned");
  if (((uintptr_t)workspace) & 255u || workspace_bytes < pced_adacad_beta_workspace_size(B, N, V))
    return fail(PCED_ERR_WORKSPACE, "pced_adacad_beta: workspace too small or misaligned");
  if (num_sms() <= 0) return fail(PCED_ERR_NO_DEVICE, "pced_adacad_beta: no CUDA device");
  cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e = adacad_beta_launch(logprobs, B, N, V, beta, true, s);
  if (e != cudaSuccess) return cuda_status(e, "pced_adacad_beta launch");
  return PCED_OK;
}
