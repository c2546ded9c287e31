// lm_head.cu -- per-expert vocabulary scores (paper Sec. 3, "per-expert logits
// s_k"; Eq. 2 mixes them as log-probabilities) on the 5th-generation tensor
// cores.
//
// Swap-AB skinny GEMM: Z^T[V x S] = W[V x d] * H^T[d x S].  The vocabulary is
// the UMMA M dimension (128-row tiles), the S hidden rows are the N dimension,
// so the bf16 unembedding matrix streams from HBM exactly once per step while
// the tiny H operand is re-read from L2 (from LM_PAIR_MIN_S rows on by pairs of
// CTAs, lm_head_pair.cu).  Persistent CTAs, one per SM:
//   warp 0  TMA producer (W tile 128x64 + H slab S_pad x 64 per stage, 128B swizzle)
//   warp 1  TMEM allocator and single-thread tcgen05.mma issuer (fp32 accumulators
//           in TMEM, double-buffered)
//   warps 2-9 epilogue: tcgen05.ld of the 128 x S accumulator (warp w reads TMEM lane
//           quarter w % 4; warps 2-5 take the first half of the columns, 6-9 the rest);
//           per column the tile's (max, sum exp) for the log-softmax and, for each
//           contextual expert k of query b, the tile's max and argmax of
//           u_k(v) = (1+beta_k) z_k(v) - beta_k z_0(v), reduced over the rows with
//           transposed butterflies (one shuffle per column and reduction).
// Because shat_k(v) = u_k(v) + c_k with c_k = -(1+beta_k) L_k + beta_k L_0 + gamma log r_k
// constant in v, Eq. 3 only needs these per-tile maxima and the log-sum-exps L:
// the [S x V] logits never reach HBM on the fused path.
#include <cooperative_groups.h>
#include <math.h>
#include <stdlib.h>

#include "lm_epilogue.cuh"
#include "lm_head.cuh"
#include "select_key.cuh"

namespace pced {

namespace cg = cooperative_groups;

constexpr int LM_PAIR_HSTAGES = 5;  // most stages of a pair's H ring

bool lm_geometry(int32_t S, int32_t d, int32_t V, LmGeom* g) {
  if (S < 1 || S > LM_MAX_S || d < LM_TILE_K || d % LM_TILE_K != 0 || V < 1) return false;
  g->S = S;
  g->d = d;
  g->V = V;
  g->pair = S >= LM_PAIR_MIN_S;
  if (g->pair) {
    // N of a pair's MMA is a multiple of 32 up to 256
    g->S_pad = (S + 31) / 32 * 32;
    if (g->S_pad <= 256) {
      g->chunk_n = g->S_pad;
      g->acc_bufs = 2;
    } else if (g->S_pad <= 384) {
      g->chunk_n = 512 - g->S_pad;  // double buffered; the rest, at most 256 columns, once
      g->acc_bufs = 2;
    } else {
      g->chunk_n = 256;
      g->acc_bufs = 1;
    }
    g->tmem_cols = 512;
  } else {
    g->chunk_n = g->S_pad = ((S < 16 ? 16 : S) + 15) / 16 * 16;
    g->acc_bufs = 2;
    uint32_t cols = 32;
    while (cols < (uint32_t)(2 * g->S_pad)) cols <<= 1;
    g->tmem_cols = cols;
  }
  g->ntiles = (V + LM_TILE_V - 1) / LM_TILE_V;
  g->nks = d / LM_TILE_K;
  const size_t fixed = 1024 + 80 * 8 + 16 + 4 * LM_TRING + (size_t)2 * 4 * g->S_pad * sizeof(float2) +
                       (size_t)2 * g->S_pad * sizeof(float2) + (size_t)g->S_pad * sizeof(float2) + 32 * 4 + 8 * 64 * 4 + 64 + 128;
  if (g->pair) {
    // W comes from HBM and H from L2: H has few stages, W what is left
    const size_t hslab = (size_t)g->S_pad * 64;
    g->slabs = 1;
    g->nst = g->nks;
    g->hstages = LM_PAIR_HSTAGES;
    while (g->hstages > 2 && fixed + g->hstages * (hslab + LM_A_BYTES) > LM_SMEM_BUDGET) --g->hstages;
    int st = (int)((LM_SMEM_BUDGET - fixed - g->hstages * hslab) / LM_A_BYTES);
    if (st > 12) st = 12;
    g->stages = st;
    g->smem = fixed + g->hstages * hslab + (size_t)st * LM_A_BYTES;
  } else {
    const size_t slab = LM_A_BYTES + (size_t)g->S_pad * 128;
    // several consecutive K-slabs per stage so each row is fetched in longer
    // runs and the tensor cores get longer bursts per stage; keep at least
    // three stages in flight
    g->slabs = 1;
    for (int sl = 4; sl >= 2; sl >>= 1)
      if (g->nks % sl == 0 && fixed + 3 * sl * slab <= LM_SMEM_BUDGET) {
        g->slabs = sl;
        break;
      }
    const size_t stage = (size_t)g->slabs * slab;
    int st = (int)((LM_SMEM_BUDGET - fixed) / stage);
    if (st > 8) st = 8;
    if (st < 2) return false;
    g->stages = st;
    g->hstages = 0;
    g->nst = g->nks / g->slabs;
    g->smem = fixed + (size_t)st * stage;
  }
  int sms = pced_host::num_sms();
  if (g->pair) {
    const int pairs = (g->ntiles + 1) / 2;
    g->grid = 2 * (pairs < sms / 2 ? pairs : sms / 2);
    if (g->grid < 2) g->grid = 2;
  } else {
    g->grid = g->ntiles < sms ? g->ntiles : sms;
    if (g->grid < 1) g->grid = 1;
  }
  return true;
}

pced_status lm_head_maps(const void* w_unembed, const void* hidden, const LmGeom& g, LmMaps* m) {
  using pced_host::make_tmap_2d;
  pced_status st = make_tmap_2d(&m->w, w_unembed, (uint64_t)g.V, (uint64_t)g.d, LM_TILE_V, LM_TILE_K, true);
  const int share = g.pair ? 2 : 1;  // a CTA of a pair loads half of a chunk's rows
  for (int c = 0; c < 2 && st == PCED_OK; ++c) {
    const int n = c == 0 || g.chunk_n == g.S_pad ? g.chunk_n : g.S_pad - g.chunk_n;
    st = make_tmap_2d(&m->h[c], hidden, (uint64_t)g.S, (uint64_t)g.d, (uint32_t)(n / share), LM_TILE_K, false);
    if (g.chunk_n == g.S_pad) {
      m->h[1] = m->h[0];
      break;
    }
  }
  return st;
}

LmArgs lm_args(const LmGeom& g) {
  LmArgs a = {};
  a.S = g.S;
  a.V = g.V;
  a.ntiles = g.ntiles;
  a.nks = g.nks;
  a.slabs = g.slabs;
  a.nst = g.nst;
  a.stages = g.stages;
  a.hstages = g.hstages;
  a.acc_bufs = g.acc_bufs;
  a.S_pad = g.S_pad;
  a.chunk_n = g.chunk_n;
  a.tmem_cols = g.tmem_cols;
  return a;
}

// The MMAs of one stage of SL K-slabs (single N chunk), fully unrolled: the
// start-address field of a K-major SW128 descriptor advances by 2 per 16-wide
// K-step and by the slab size >> 4 per slab.
template <int SL>
__device__ __forceinline__ void umma_slabs(uint32_t on, uint32_t dcol, uint64_t ad0, uint64_t bd0, uint32_t bstep, uint32_t idesc,
                                           bool first) {
#pragma unroll
  for (int j = 0; j < SL; ++j)
#pragma unroll
    for (int k = 0; k < LM_TILE_K / 16; ++k)
      umma_bf16(on, dcol, ad0 + (uint64_t)(j * (LM_A_BYTES >> 4) + 2 * k), bd0 + (uint64_t)(j * bstep + 2 * k), idesc,
                !(first && j == 0 && k == 0));
}

__global__ void __launch_bounds__(LM_THREADS, 1)
    lm_head_kernel(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap hmap, LmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const int SL = a.slabs, S_pad = a.S_pad;
  const uint32_t b_bytes = (uint32_t)S_pad * 128u;
  const uint32_t st_bytes = (uint32_t)SL * (LM_A_BYTES + b_bytes);  // SL A slabs, then SL B slabs
  const int stages = a.stages;
  // layout: stages | full | empty | tfull[2] | tempty[2] | tid[2] | epi | drain |
  //         tmem slot, tile ring, accumulator tiles | scratch
  const uint32_t bar_full = base + stages * st_bytes;
  const uint32_t bar_empty = bar_full + 8 * stages;
  const uint32_t bar_tfull = bar_empty + 8 * stages;
  const uint32_t bar_tempty = bar_tfull + 16;
  const uint32_t bar_tid = bar_tempty + 16;
  const uint32_t bar_epi = bar_tid + 16;
  const uint32_t bar_drain = bar_epi + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + (bar_drain + 8 - base));
  int32_t* tring = reinterpret_cast<int32_t*>(tmem_slot + 4);  // [LM_TRING] claimed tiles, producer -> MMA warp
  int32_t* acc_tile = tring + LM_TRING;                        // [2] tile of each accumulator, MMA warp -> epilogue
  float2* wst = reinterpret_cast<float2*>(gbase + (bar_drain + 8 - base) + 32 + 4 * LM_TRING);  // [4][S_pad] per-warp stats
  float2* wag = wst + 4 * S_pad;                                                  // [4][S_pad] per-warp argmax
  float* wu2 = reinterpret_cast<float*>(wag + 4 * S_pad);                         // [4][S_pad] per-warp runner-up
  float2* ccoef = wag + 6 * S_pad;                                 // [S_pad] (1 + beta, beta) per column
  uint32_t* cmask = reinterpret_cast<uint32_t*>(ccoef + S_pad);     // [2][16] amateur / expert column bits
  float* bc = reinterpret_cast<float*>(cmask + 32);                // [8][64] per-warp column broadcast

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_tfull + 8 * i, 1);
      mbar_init(bar_tempty + 8 * i, LM_EPI_THREADS);
      mbar_init(bar_tid + 8 * i, 1);
    }
    mbar_init(bar_epi, LM_EPI_THREADS);
    mbar_init(bar_drain, 1);
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&wmap);
    tma_prefetch_desc(&hmap);
  }
  if (a.mode == 1) pdl_launch_dependents();
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), a.tmem_cols);
    tmem_relinquish();
  }
  if (a.mode == 1) column_tables(a, tid, ccoef, cmask);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const int ntiles = a.ntiles, nst = a.nst;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    const uint32_t on = elect_one();
    const uint64_t pol_w = policy_evict_first(), pol_h = policy_evict_last();
    // Tiles are claimed from a global counter, so CTAs that start early (as
    // the previous kernel's CTAs leave their SMs) take more of them; without
    // a counter CTA c takes tiles c, c + CTAs, ...  The claimed ids reach the MMA warp through tring (written before the
    // arrive on the full barrier of the tile's first stage); -1 ends.
    int tile = -1, ks = 0;
    uint32_t tseq = 0;
    auto claim = [&]() {
      int t = -1;
      if (lane == 0) {
        t = a.tile_ctr ? atomicAdd(a.tile_ctr, 1) : (int)(blockIdx.x + tseq * gridDim.x);
        if (t >= ntiles) t = -1;
        tring[tseq % LM_TRING] = t;
      }
      tile = __shfl_sync(0xffffffffu, t, 0);
      ++tseq;
      ks = 0;
    };
    auto load_w = [&](uint32_t st) {
      const uint32_t fb = bar_full + 8 * st, sa = base + st * st_bytes;
      mbar_arrive_expect_tx_if(on, fb, st_bytes);
      // consecutive K-slabs of the same 128 rows back to back: longer runs per row
      for (int j = 0; j < SL; ++j)
        tma_load_2d(on, sa + j * LM_A_BYTES, &wmap, fb, (ks * SL + j) * LM_TILE_K, tile * LM_TILE_V, pol_w);
    };
    auto load_h = [&](uint32_t st, int kss) {
      const uint32_t fb = bar_full + 8 * st, sb = base + st * st_bytes + SL * LM_A_BYTES;
      for (int j = 0; j < SL; ++j)
        tma_load_2d(on, sb + j * b_bytes, &hmap, fb, (kss * SL + j) * LM_TILE_K, 0, pol_h);
    };
    if (a.pdl == LM_PDL_ALL) pdl_wait();
    claim();
    uint32_t it = 0;
    // With programmatic dependent launch the weights of the first stages
    // stream while the previous kernel (which writes H) finishes; a tile has
    // nst stages, so stage i of these belongs to stage i % nst of its tile.
    if (a.pdl == LM_PDL_H) {
      while (tile >= 0 && it < (uint32_t)stages) {
        load_w(it++);
        if (++ks == nst) claim();
      }
      pdl_wait();
      for (uint32_t i = 0; i < it; ++i) load_h(i, (int)(i % (uint32_t)nst));
    }
    bool ok = true;
    uint32_t st = it == (uint32_t)stages ? 0 : it, ph = it == (uint32_t)stages ? 1 : 0;
    while (tile >= 0) {
      if (!mbar_wait_warp(bar_empty + 8 * st, ph ^ 1u, a.status)) {
        ok = false;
        break;
      }
      load_w(st);
      load_h(st, ks);
      ++it;
      if (++st == (uint32_t)stages) {
        st = 0;
        ph ^= 1u;
      }
      if (++ks == nst) claim();
    }
    if (ok) {
      // end marker: a phase of the next stage's full barrier without data
      if (mbar_wait_warp(bar_empty + 8 * st, ph ^ 1u, a.status) && lane == 0) mbar_arrive(bar_full + 8 * st);
    } else {
      for (uint32_t j = (it >= (uint32_t)stages ? it - stages : 0); j < it; ++j)
        mbar_wait_warp(bar_full + 8 * (j % stages), (j / stages) & 1u, a.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    const uint32_t on = elect_one();
    const uint32_t idesc = umma_idesc_bf16(LM_TILE_V, a.chunk_n);
    uint32_t acc = 0, tseq = 0, st = 0, ph = 0;
    bool ok = true;
    for (;; ++acc) {
      const uint32_t buf = acc & 1u, aph = (acc >> 1) & 1u;
      // the next tile's first stage (or the end marker) tells which tile it is
      if (!mbar_wait_warp(bar_full + 8 * st, ph, a.status)) break;
      const int tile = __shfl_sync(0xffffffffu, tring[tseq % LM_TRING], 0);
      ++tseq;
      if (!mbar_wait_warp(bar_tempty + 8 * buf, aph ^ 1u, a.status)) break;
      if (lane == 0) {
        acc_tile[buf] = tile;
        mbar_arrive(bar_tid + 8 * buf);
      }
      __syncwarp();
      if (tile < 0) break;
      tc_fence_after();
      const uint32_t dcol = tmem_base + buf * S_pad;
      for (int ks = 0; ks < nst; ++ks) {
        if (ks > 0 && !mbar_wait_warp(bar_full + 8 * st, ph, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = base + st * st_bytes, sb = sa + SL * LM_A_BYTES;
        // descriptors are built once per stage; a K-step moves the start
        // address field (bytes >> 4) by 2, a slab by its size >> 4
        const uint64_t ad0 = umma_desc_sw128(sa), bd0 = umma_desc_sw128(sb);
        const uint32_t bstep = b_bytes >> 4;
        const bool first = ks == 0;
        if (SL == 4)
          umma_slabs<4>(on, dcol, ad0, bd0, bstep, idesc, first);
        else if (SL == 2)
          umma_slabs<2>(on, dcol, ad0, bd0, bstep, idesc, first);
        else
          umma_slabs<1>(on, dcol, ad0, bd0, bstep, idesc, first);
        umma_commit(on, bar_empty + 8 * st);
        if (++st == (uint32_t)stages) {
          st = 0;
          ph ^= 1u;
        }
      }
      if (!ok) break;
      umma_commit(on, bar_tfull + 8 * buf);
    }
    // all issued MMAs complete before TMEM is released
    umma_commit(on, bar_drain);
    mbar_wait_warp(bar_drain, 0, a.status);
    __syncwarp();
  } else {
    // ----------------------------------------------------------- epilogue
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    const int etid = tid - 64, half = (warp - 2) >> 2;
    const int S = a.S, n1 = a.N + 1;
    uint32_t ephase = 0;
    for (uint32_t acc = 0;; ++acc) {
      const uint32_t buf = acc & 1u, aph = (acc >> 1) & 1u;
      if (!mbar_wait(bar_tid + 8 * buf, aph, a.status)) break;
      const int tile = acc_tile[buf];
      if (tile < 0) break;
      if (!mbar_wait(bar_tfull + 8 * buf, aph, a.status)) break;
      tc_fence_after();
      const int v = tile * LM_TILE_V + 32 * q + lane;
      const bool valid = v < a.V;
      const uint32_t trow = tmem_base + ((uint32_t)(32 * q) << 16) + buf * S_pad;
      // column blocks of W = 32 (the last one may be 16 wide), or of S_pad / 2
      // when S_pad <= 32 so that both warp halves work; the first half of the
      // blocks goes to warps 2-5, the rest to warps 6-9
      const int W = S_pad <= 32 ? S_pad / 2 : 32;
      const int nb = (S + W - 1) / W, kb0 = half ? (nb + 1) / 2 : 0, kb1 = half ? nb : (nb + 1) / 2;
      float z_am = 0.f;
      if (a.mode == 1 && kb0 < kb1 && (W * kb0) % n1 != 0)
        z_am = tmem_ld1(trow + W * kb0 - (W * kb0) % n1);  // the row's amateur logit of the open query
      float* wbc = bc + 64 * (warp - 2);
      // the accumulator is free for the next tile's MMAs once this warp's last
      // columns are in its registers
      auto release = [&]() {
        tc_fence_before();
        mbar_arrive(bar_tempty + 8 * buf);
      };
      if (kb0 >= kb1) release();
      for (int kb = kb0; kb < kb1; ++kb) {
        const int c0 = W * kb;
        auto loaded = [&]() {
          if (kb + 1 == kb1) release();
        };
        if (W == 8)
          epi_block<8>(a, trow + c0, c0, v, valid, lane, q, wbc, wst, wag, wu2, ccoef, cmask, z_am, loaded);
        else if (c0 + 32 <= S_pad && W == 32)
          epi_block<32>(a, trow + c0, c0, v, valid, lane, q, wbc, wst, wag, wu2, ccoef, cmask, z_am, loaded);
        else
          epi_block<16>(a, trow + c0, c0, v, valid, lane, q, wbc, wst, wag, wu2, ccoef, cmask, z_am, loaded);
      }
      if (!bar_sync_bounded(bar_epi, ephase, a.status)) break;
      const bool tile_ok = PCED_IN_BOUNDS(tile < ntiles, a.status);
      if (tile_ok) fold_tile(a, tile, etid, wst, wag, wu2);
      if (!bar_sync_bounded(bar_epi, ephase, a.status)) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  // the log-softmax or aggregation kernels come at the end (at the start, a call
  // in a graph takes 250 us instead of 245 at S = 272, 24.4 instead of 23.0 at S =
  // 33, d = 1024, V = 50000); the selection's cluster, which starts later, comes
  // early (the 9-row step 538 us, 543 with a late one)
  if (a.mode == 0) pdl_launch_dependents();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, a.tmem_cols);
  }
}

cudaError_t lm_head_launch(const LmMaps& m, const LmGeom& g, const LmArgs& a, cudaStream_t stream) {
  if (g.pair) return lm_head_pair_launch(m, g, a, stream);
  // the shared-memory limit is an attribute of the kernel on each device
  static bool configured[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(lm_head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LM_SMEM_BUDGET);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  return pced_host::launch_kernel(lm_head_kernel, dim3(g.grid), LM_THREADS, g.smem, stream, a.pdl != 0,
                                  m.w, m.h[0], a);
}

// ------------------------------------------------------------ mode-0 finish
constexpr int LSE_THREADS = 256;

// log-sum-exp of row s from its tile records (fixed order), in every thread
__device__ __forceinline__ float row_lse(const float2* rec, int32_t nrec, float2* red, float* Ls) {
  const int tid = threadIdx.x;
  float M = -INFINITY, sum = 0.f;
  for (int t = tid; t < nrec; t += LSE_THREADS) {
    const float2 r = rec[t];
    lse_merge(M, sum, r.x, r.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, M, o), s2 = __shfl_xor_sync(0xffffffffu, sum, o);
    lse_merge(M, sum, m2, s2);
  }
  if ((tid & 31) == 0) red[tid >> 5] = make_float2(M, sum);
  __syncthreads();
  if (tid == 0) {
    float m = -INFINITY, su = 0.f;
    for (int w = 0; w < LSE_THREADS / 32; ++w) lse_merge(m, su, red[w].x, red[w].y);
    *Ls = m + logf(su);
  }
  __syncthreads();
  return *Ls;
}

__global__ void __launch_bounds__(LSE_THREADS) lm_lse_kernel(const float2* rec_stats, float* lse, int32_t nrec) {
  __shared__ float2 red[LSE_THREADS / 32];
  __shared__ float Ls;
  pdl_launch_dependents();
  pdl_wait();
  const float L = row_lse(rec_stats + (int64_t)blockIdx.x * nrec, nrec, red, &Ls);
  if (threadIdx.x == 0) lse[blockIdx.x] = L;
}

// CTA (chunk, row s), all rows of the last chunk first (the tiles written last
// are still in L2: the whole call, in a graph, 245 us instead of 261 at S = 272, V
// = 128256): chunk of logits -> log-probabilities in place.  FUSED: every CTA of
// row s also forms lse[s], one launch less (6.8 us instead of 7.2 at S = 3, d =
// 512, V = 8192, 23.0 instead of 23.7 at S = 33, d = 1024, V = 50000; not at S = 9,
// V = 128256: 162.9, 161.6); otherwise lm_lse_kernel has written it, so that a
// CTA's time is that of its loads and stores alone (245 us instead of 256 at S =
// 272, 185.6 instead of 190.4 at S = 128, 168.1 instead of 170.0 at S = 65).
template <bool FUSED, int CHUNK>
__global__ void __launch_bounds__(LSE_THREADS) lm_lse_finalize_kernel(float* logits, const float2* rec_stats, float* lse,
                                                                      int32_t S, int32_t V, int32_t nrec) {
  const int tid = threadIdx.x, s = blockIdx.x % S, c = (gridDim.x - 1 - blockIdx.x) / S;
  __shared__ float2 red[LSE_THREADS / 32];
  __shared__ float Ls;
  pdl_launch_dependents();
  float* row = logits + (int64_t)s * V + (int64_t)c * CHUNK;
  const int n = min(CHUNK, V - c * CHUNK);
  float x[CHUNK / LSE_THREADS];
  pdl_wait();
#pragma unroll
  for (int i = 0; i < CHUNK / LSE_THREADS; ++i)
    if (tid + i * LSE_THREADS < n) x[i] = row[tid + i * LSE_THREADS];
  float L;
  if (FUSED) {
    L = row_lse(rec_stats + (int64_t)s * nrec, nrec, red, &Ls);
    if (c == 0 && tid == 0) lse[s] = L;
  } else {
    L = lse[s];
  }
#pragma unroll
  for (int i = 0; i < CHUNK / LSE_THREADS; ++i)
    if (tid + i * LSE_THREADS < n) row[tid + i * LSE_THREADS] = x[i] - L;
}

constexpr int LSE_FUSED_CHUNK = 8192;  // (144 CTAs for 9 rows of 128K entries)
constexpr int LSE_CHUNK = 2048;

cudaError_t lm_lse_finalize_launch(float* logits, const float2* rec_stats, float* lse, int32_t S, int32_t V,
                                   int32_t nrec, bool fused, bool pdl, cudaStream_t stream) {
  const int chunk = fused ? LSE_FUSED_CHUNK : LSE_CHUNK;
  const dim3 grid((unsigned)((V + chunk - 1) / chunk) * (unsigned)S);
  using pced_host::launch_kernel;
  if (fused)
    return launch_kernel(lm_lse_finalize_kernel<true, LSE_FUSED_CHUNK>, grid, LSE_THREADS, 0, stream, pdl, logits,
                         rec_stats, lse, S, V, nrec);
  const cudaError_t e = launch_kernel(lm_lse_kernel, dim3(S), LSE_THREADS, 0, stream, pdl, rec_stats, lse, nrec);
  if (e != cudaSuccess) return e;
  return launch_kernel(lm_lse_finalize_kernel<false, LSE_CHUNK>, grid, LSE_THREADS, 0, stream, pdl, logits, rec_stats,
                       lse, S, V, nrec);
}

// ------------------------------------------- Eq. 2 + Eq. 3 from tile records
// One cluster of up to SEL_CLUSTER CTAs per query b; CTA c takes the rows j = c,
// c + CTAs, ... of the query: L_s from the row's tile records and, for an
// expert row (j > 0), the best tile record of u_k.  Every CTA gets every row's
// results and forms score_k = u_k* + c_k and the pick (score desc, token asc,
// expert asc); for the near-tie margins each recomputes z_s(token) of its own
// rows, and the first one finishes.  Every reduction runs in a fixed order (a
// row's threads take its records in turn, then xor trees over lanes, then the
// warps in order), so the result does not depend on timing.
//
// What bounds it: a chain of dependent steps (records, the rows' exchange, the
// chosen row of W, the exchange of the margins' products), all of latency.
// The exchanges go through shared memory of the cluster, without the fences,
// the arrival counter and the reloads of results in global memory that CTAs
// without a cluster need, and the recomputed products, 129 rows of H at 128
// experts, are spread over the cluster instead of one CTA.  A row's records are
// in flight together and their maximum is the thread's own first, so one pass
// does.  Measured (one CTA per row with an arrival counter -> this): 9 rows
// 12.4 -> 10.1 us, 33 rows 17.4 -> 10.6, 129 rows 35 -> 21, 16 x 17 rows 19.0 ->
// 13.2, 3 rows of d = 512 9.3 -> 8.4.  A row's warps meet in the lanes of its
// first one (each receiver used to add the sixteen results one after another),
// and beta and r are loaded while the cluster meets: a step of 3 rows and one
// layer 37.7 -> 36.7 us, of 9 rows and 32 layers 528.8 -> 527.6.  Loading them
// beside the records cost 16 x 17 rows 2 us; an L2 prefetch of each candidate's
// row of W gained nothing.
constexpr int SEL_R_THREADS = 512;
constexpr int SEL_R_WARPS = SEL_R_THREADS / 32;
constexpr int SEL_R_CLUSTER = 8;  // most CTAs per query
constexpr int SEL_RECS = 8;       // records of a thread in flight
constexpr int SEL_ZROWS = 8;      // rows of a thread group in flight in the near-tie products

__global__ void __launch_bounds__(SEL_R_THREADS) select_from_records_kernel(SelectArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  const int nc = gridDim.x, rank = blockIdx.x, b = blockIdx.y;  // one cluster per query
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = a.N, n1 = N + 1, T = a.nrec;
  __shared__ float row_L[LM_MAX_N1], row_u[LM_MAX_N1], row_u2[LM_MAX_N1];  // every row's results
  __shared__ int row_tok[LM_MAX_N1];
  __shared__ float zy[LM_MAX_N1];  // z_s(token) of the query's rows (first CTA)
  __shared__ float sm[SEL_R_WARPS], su[SEL_R_WARPS], sv[SEL_R_WARPS], sv2[SEL_R_WARPS];
  __shared__ int si[SEL_R_WARPS];
  __shared__ int pick[2];  // token, expert of the query
  __shared__ float zpart[SEL_R_WARPS][SEL_ZROWS];
  cluster.barrier_arrive();  // waited for before another CTA's shared memory is written
  if (a.pdl) pdl_wait();     // the LM head's records are complete and visible
  if (rank == 0 && b == 0 && tid == 0 && a.tile_ctr) *a.tile_ctr = 0;  // the next LM head claims its tiles from 0
  const int t_step = a.step && tid == 0 ? *a.step : 0;  // advances only once every query is through
  // ---- the CTA's rows, rf at a time, SEL_R_WARPS / rf warps each
  const int rows = (n1 - rank + nc - 1) / nc;
  int rf = 1;
  while (rf < rows && rf < 8) rf <<= 1;
  const int wpr = SEL_R_WARPS / rf, grp = warp / wpr, gt = tid - grp * wpr * 32, gn = wpr * 32;
  bool started = false;
  for (int q0 = 0; q0 < rows; q0 += rf) {
    const int q = q0 + grp, j = rank + nc * q, s = b * n1 + j;
    const bool on = q < rows && PCED_IN_BOUNDS(s < a.B * n1, a.status);
    // the row's (largest logit, sum of exp), its best u_k and its token, and the best u_k at any other token
    float m = -INFINITY, sum = 0.f, bu = -INFINITY, b2 = -INFINITY;
    int bv = 0x7fffffff;
    if (on) {
      const float2* rec = a.rec_stats + (int64_t)s * T;
      const float2* reca = a.rec_arg + (int64_t)s * T;
      const float* rec2 = a.rec_u2 + (int64_t)s * T;
      for (int t0 = gt; t0 < T; t0 += SEL_RECS * gn) {
        float2 st[SEL_RECS], ar[SEL_RECS];
        float u2[SEL_RECS];
#pragma unroll
        for (int i = 0; i < SEL_RECS; ++i) {
          const int t = t0 + i * gn;
          const bool in = t < T;
          st[i] = in ? __ldcg(rec + t) : make_float2(-INFINITY, 0.f);
          ar[i] = in && j > 0 ? __ldcg(reca + t) : make_float2(-INFINITY, __int_as_float(0x7fffffff));
          u2[i] = in && j > 0 ? __ldcg(rec2 + t) : -INFINITY;
        }
        float mn = m;
#pragma unroll
        for (int i = 0; i < SEL_RECS; ++i) mn = fmaxf(mn, st[i].x);
        if (m != -INFINITY) sum *= expf(m - mn);
#pragma unroll
        for (int i = 0; i < SEL_RECS; ++i) {
          if (st[i].x != -INFINITY) sum += st[i].y * expf(st[i].x - mn);
          top2_merge(bu, bv, b2, ar[i].x, __float_as_int(ar[i].y), u2[i]);
        }
        m = mn;
      }
      const float mw = warp_max(m);
      sum = warp_sum(m == -INFINITY ? sum : sum * expf(m - mw));
      m = mw;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float r1 = __shfl_xor_sync(0xffffffffu, bu, o), r2 = __shfl_xor_sync(0xffffffffu, b2, o);
        const int rt = __shfl_xor_sync(0xffffffffu, bv, o);
        top2_merge(bu, bv, b2, r1, rt, r2);
      }
    }
    if (lane == 0) {
      sm[warp] = m;
      su[warp] = sum;
      sv[warp] = bu;
      si[warp] = bv;
      sv2[warp] = b2;
    }
    __syncthreads();
    if (!started) cluster.barrier_wait();
    started = true;
    if (on && gt < 32) {  // the row's first warp: lane w takes warp w's results
      const int w = grp * wpr + lane;
      const bool in = lane < wpr;
      m = in ? sm[w] : -INFINITY;
      bu = in ? sv[w] : -INFINITY;
      b2 = in ? sv2[w] : -INFINITY;
      bv = in ? si[w] : 0x7fffffff;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float r1 = __shfl_xor_sync(0xffffffffu, bu, o), r2 = __shfl_xor_sync(0xffffffffu, b2, o);
        const int rt = __shfl_xor_sync(0xffffffffu, bv, o);
        top2_merge(bu, bv, b2, r1, rt, r2);
      }
      const float M = warp_max(m), e = !in ? 0.f : m == -INFINITY ? su[w] : su[w] * expf(m - M);
      float L = 0.f;
      for (int i = 0; i < wpr; ++i) L += __shfl_sync(0xffffffffu, e, i);  // the warps in order
      L = M + logf(L);
      if (lane < nc) {  // lane c writes to CTA c
        cluster.map_shared_rank(row_L, lane)[j] = L;
        cluster.map_shared_rank(row_u, lane)[j] = bu;
        cluster.map_shared_rank(row_u2, lane)[j] = b2;
        cluster.map_shared_rank(row_tok, lane)[j] = bv;
        if (lane == 0 && a.lse_out) a.lse_out[s] = L;
      }
    }
    if (q0 + rf < rows) __syncthreads();  // the partial results are used again
  }
  cluster.barrier_arrive();
  // warp 0's first experts' beta and relevance arrive while the cluster meets
  const float beta0 = warp == 0 && lane < N ? a.beta[b * N + lane] : 0.f;
  const float r0 = warp == 0 && lane < N ? a.r[b * N + lane] : 1.f;
  cluster.barrier_wait();
  float bs = -INFINITY;
  int bt = 0x7fffffff, bk = 0x7fffffff;
  // Eq. 2's per-expert constant (warp 0, k = lane + 32 i)
  auto beta_of = [&](int k) { return k < 32 ? beta0 : a.beta[b * N + k]; };
  auto bias = [&](int k) {
    const float btk = beta_of(k);
    const float rr = fminf(fmaxf(k < 32 ? r0 : a.r[b * N + k], 1e-8f), 1.0f);
    return (a.raw_logits ? 0.f : -(1.f + btk) * row_L[1 + k] + btk * row_L[0]) + a.gamma * logf(rr);
  };
  if (warp == 0) {
    for (int k = lane; k < N; k += 32) {
      const float sc = row_u[1 + k] + bias(k);
      const int tk = row_tok[1 + k];
      if (sc > bs || (sc == bs && (tk < bt || (tk == bt && k < bk)))) {
        bs = sc;
        bt = tk;
        bk = k;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float s2 = __shfl_xor_sync(0xffffffffu, bs, o);
      const int t2 = __shfl_xor_sync(0xffffffffu, bt, o), k2 = __shfl_xor_sync(0xffffffffu, bk, o);
      if (s2 > bs || (s2 == bs && (t2 < bt || (t2 == bt && k2 < bk)))) {
        bs = s2;
        bt = t2;
        bk = k2;
      }
    }
    if (lane == 0) {
      pick[0] = bt;
      pick[1] = bk;
    }
  }
  float2 gaps = make_float2(INFINITY, INFINITY);
  if (a.gap_trace && !a.key_out) {
    __syncthreads();
    const int y = pick[0] >= 0 && pick[0] < a.V ? pick[0] : 0;
    // z_s(y) = h_s . W[y] for the CTA's rows.  tpr threads take a row (16-byte
    // chunks i, i + tpr, ... of W[y] and of the row), SEL_ZROWS rows of each
    // group of tpr threads in flight together.  Per row the partial sums meet
    // in a fixed order (warp tree, then the group's warps in order).
    const int nv = a.d / 8;  // 16-byte chunks of a row (d % 64 == 0)
    int tpr = 32;
    while (tpr < nv && tpr < SEL_R_THREADS / (rows > 1 ? 2 : 1)) tpr <<= 1;
    const int ng = SEL_R_THREADS / tpr, g = tid / tpr, wpg = tpr / 32;
    const uint4* wy = reinterpret_cast<const uint4*>(a.w_unembed + (int64_t)y * a.d);
    const uint4* h0 = reinterpret_cast<const uint4*>(a.hidden + (int64_t)b * n1 * a.d);
    for (int q0 = 0; q0 < rows; q0 += ng * SEL_ZROWS) {
      float acc[SEL_ZROWS];
#pragma unroll
      for (int u = 0; u < SEL_ZROWS; ++u) acc[u] = 0.f;
      for (int i = tid % tpr; i < nv; i += tpr) {
        const uint4 wv = __ldg(wy + i);
        uint4 hv[SEL_ZROWS];
#pragma unroll
        for (int u = 0; u < SEL_ZROWS; ++u) {
          const int q = q0 + g + ng * u;
          hv[u] = q < rows ? __ldcg(h0 + (int64_t)(rank + nc * q) * nv + i) : make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t ww[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
        for (int u = 0; u < SEL_ZROWS; ++u) {
          const uint32_t hw[4] = {hv[u].x, hv[u].y, hv[u].z, hv[u].w};
          float p = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            p = fmaf(bf16_lo(hw[e]), bf16_lo(ww[e]), p);
            p = fmaf(bf16_hi(hw[e]), bf16_hi(ww[e]), p);
          }
          acc[u] += p;
        }
      }
#pragma unroll
      for (int u = 0; u < SEL_ZROWS; ++u) {
        const float t = warp_sum(acc[u]);
        if (lane == 0) zpart[warp][u] = t;
      }
      __syncthreads();
      if (tid < ng * SEL_ZROWS && q0 + tid < rows) {
        // row q0 + tid of the CTA: group tid % ng, slot tid / ng
        float z = 0.f;
        for (int w = 0; w < wpg; ++w) z += zpart[(tid % ng) * wpg + w][tid / ng];
        cluster.map_shared_rank(zy, 0)[rank + nc * (q0 + tid)] = z;
      }
      __syncthreads();
    }
    cluster.sync();
    if (warp == 0 && rank == 0) {
      // token gap: the best score at another token, over all experts
      float other = -INFINITY, se_best = -INFINITY, se_other = -INFINITY;
      for (int k = lane; k < N; k += 32) {
        const float c = bias(k), btk = beta_of(k);
        other = fmaxf(other, (row_tok[1 + k] != bt ? row_u[1 + k] : row_u2[1 + k]) + c);
        // expert gap: every expert's score at the chosen token, from the recomputed logits
        const float se = (1.f + btk) * zy[1 + k] - btk * zy[0] + c;
        if (k == bk) se_best = se;
        else se_other = fmaxf(se_other, se);
      }
      other = warp_max(other);
      se_best = warp_max(se_best);
      se_other = warp_max(se_other);
      gaps = make_float2(bs - other, se_best - se_other);
    }
  }
  if (rank != 0) return;
  if (warp != 0) return;
  if (lane == 0 && a.key_out) {
    // expert-partitioned step: this GPU's best, the reduction over GPUs and
    // the append come after
    a.key_out[b] = select_key(bs, bt, a.expert_base + bk + 1);
    return;
  }
  if (lane == 0) {
    if (a.token) a.token[b] = bt;
    if (a.expert) a.expert[b] = bk + 1;
    if (a.score) a.score[b] = bs;
    if (a.step) {
      const int t = t_step;
      if (t >= 0 && t < a.max_steps) {
        a.history[(int64_t)b * a.max_steps + t] = bt;
        if (a.expert_trace) a.expert_trace[(int64_t)b * a.max_steps + t] = bk + 1;
        if (a.score_trace) a.score_trace[(int64_t)b * a.max_steps + t] = bs;
        if (a.gap_trace) a.gap_trace[(int64_t)b * a.max_steps + t] = gaps;
      } else {
        dev_flag(a.status, PCED_DEV_STEP_LIMIT);
      }
      bool all = a.B == 1;
      if (!all) {
        __threadfence();
        all = atomicAdd(a.done_counter, 1) == a.B - 1;
        if (all) *a.done_counter = 0;
      }
      if (all && t >= 0 && t < a.max_steps) *a.step = t + 1;  // at the limit t stays (as the commit does)
    }
  }
}

cudaError_t select_from_records_launch(const SelectArgs& a, cudaStream_t stream) {
  int nc = 1;  // CTAs per query: a power of two, at most one per row
  while (2 * nc <= SEL_R_CLUSTER && 2 * nc <= a.N + 1) nc *= 2;
  return pced_host::launch_cluster(select_from_records_kernel, dim3(nc, a.B), nc, SEL_R_THREADS, 0, stream, a.pdl != 0,
                                   a);
}

}  // namespace pced

// ------------------------------------------------------------------ C ABI
using namespace pced;
using namespace pced_host;

extern "C" size_t pced_lm_head_workspace_size(int32_t S, int32_t V) {
  if (S < 1 || V < 1) return 0;
  const int64_t ntiles = (V + LM_TILE_V - 1) / LM_TILE_V;
  Carver c(nullptr);
  c.take<float2>((size_t)(S * ntiles));
  return 256 + c.used();
}

extern "C" pced_status pced_lm_head_logprobs(const void* hidden, const void* w_unembed, int32_t S, int32_t d,
                                             int32_t V, float* logprobs, float* lse, void* workspace,
                                             size_t workspace_bytes, void* stream) {
  if (!hidden || !w_unembed || !logprobs || !lse || !workspace)
    return fail(PCED_ERR_INVALID_ARG, "pced_lm_head_logprobs: null pointer");
  if (S < 1 || d < 1 || V < 1) return fail(PCED_ERR_INVALID_ARG, "pced_lm_head_logprobs: bad sizes");
  LmGeom g;
  if (!lm_geometry(S, d, V, &g) || d > 16384)
    return fail(PCED_ERR_UNSUPPORTED, "pced_lm_head_logprobs: S=%d d=%d (need S<=512, d%%64==0, d<=16384)", S, d);
  if ((((uintptr_t)hidden) | ((uintptr_t)w_unembed)) & 15u)
    return fail(PCED_ERR_INVALID_ARG, "pced_lm_head_logprobs: operands must be 16-byte aligned");
  if (((uintptr_t)workspace) & 255u || workspace_bytes < pced_lm_head_workspace_size(S, V))
    return fail(PCED_ERR_WORKSPACE, "pced_lm_head_logprobs: workspace too small or misaligned");
  if (num_sms() <= 0) return fail(PCED_ERR_NO_DEVICE, "pced_lm_head_logprobs: no CUDA device");
  LmMaps maps;
  const pced_status st = lm_head_maps(w_unembed, hidden, g, &maps);
  if (st != PCED_OK) return st;
  Carver cv((char*)workspace + 256);
  LmArgs a = lm_args(g);
  a.logits = logprobs;
  a.rec_stats = cv.take<float2>((size_t)S * g.ntiles);
  a.status = (int*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  // every CTA starts at the same time here, so the tiles need no counter, and
  // no clearing of one before the launch (S = 3, d = 512, V = 8192: 11.6 -> 7.2
  // us; S = 9, d = 4096, V = 128256: 164 -> 162; S = 200, d = 1792, V = 30000: 49 -> 43)
  a.pdl = LM_PDL_ALL;
  cudaError_t e = lm_head_launch(maps, g, a, s);
  if (e != cudaSuccess) return cuda_status(e, "lm head launch");
  e = lm_lse_finalize_launch(logprobs, a.rec_stats, lse, S, V, g.ntiles, S <= 64, true, s);
  if (e != cudaSuccess) return cuda_status(e, "lse finalize launch");
  return PCED_OK;
}
