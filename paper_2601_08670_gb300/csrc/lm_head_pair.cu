// lm_head_pair.cu -- the LM head of many hidden rows on CTA pairs: Z^T[V x S] =
// W[V x d] H^T[d x S] with tcgen05.mma over two SMs (cta_group::2).
//
// What bounds it: at S = 272 the MMAs take about 150 us (at the 1.65 GHz that
// this load runs at) and W's 1.05 GB 155 us, and one SM per tile (lm_head.cu's
// shape) cannot feed them: per 64 hidden elements 16 KB of W and 37 KB of H are
// written to shared memory and 70 KB read from it by the MMAs, 960 clocks
// against 576 of MMAs.  A pair takes 256 vocabulary rows: each CTA loads its own
// 128 rows of W and half of H's rows, and the tensor cores of both read both
// halves, so the L2 traffic of H and its part of the shared-memory traffic
// halve.
//
// TMEM (512 columns a CTA): up to 256 padded rows the accumulator is double
// buffered.  Past that the columns are two chunks, the first (n0 = 512 - S_pad
// columns) double buffered and the second (n1) single; the epilogue reads the
// second one first, so the next tile's MMAs wait for n1 columns of it only.
//
// W comes from HBM, H from L2, so they have rings of their own: five stages of
// H, and W in the rest of shared memory (S = 272, a call in a graph: two stages
// of H 285 us, three 256, four 248, five 245, six 246; one ring of both with three
// stages was 4 us slower than two rings).  An epilogue warp gives its columns back
// as soon as they are in its registers (8 us less).
//
// Measured (pced_lm_head_logprobs, d = 4096, V = 128256, in a graph; one CTA per
// tile -> pairs): S = 272 369 -> 245 us, S = 384 508 -> 344, S = 512 581 -> 456; a
// call among others, on new inputs, at S = 272 372 -> 263; the launch in a decode
// step of 272 sequences 358 -> 207-221 (by the clock that the power limit leaves).  About half of that came from issuing MMAs
// and copies in warp-uniform code (elect_one in common.cuh), which lm_head.cu
// has too; LM_PAIR_MIN_S in lm_head.cuh has both kernels where one CTA can do.
//
// Roles per CTA as in lm_head.cu.  CTA 0 of the pair claims tiles (both CTAs get
// them through a ring in shared memory), waits for the operands of both (its
// full barriers count both CTAs' bytes), and issues every MMA; commits arrive
// on the barriers of both; both epilogues release TMEM to CTA 0.
#include "lm_epilogue.cuh"
#include "lm_head.cuh"

namespace pced {

// CTA 0's full barriers for lm_pair_drain (a whole warp, `on` in one lane)
struct PairFull {
  uint32_t on, bar, bytes;  // bytes of one CTA's share of a slab
  int* status;
  __device__ void expect_one(uint32_t w) { mbar_arrive_expect_tx_if(on, bar + 8 * w, bytes); }
  __device__ void missing_one(uint32_t w) { mbar_complete_tx_if(on, bar + 8 * w, bytes); }
  __device__ bool wait(uint32_t w, uint32_t parity) { return mbar_wait_warp(bar + 8 * w, parity, status); }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(LM_THREADS, 1)
    lm_head_pair_kernel(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap hmap0,
                        const __grid_constant__ CUtensorMap hmap1, LmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const int S_pad = a.S_pad, n0 = a.chunk_n, nc1 = S_pad - a.chunk_n;
  const uint32_t b_bytes = (uint32_t)S_pad * 64u;  // this CTA's half of an H slab
  const uint32_t wst_n = a.stages, hst_n = a.hstages;
  // layout: W ring | H ring | full[W stages] | empty[W stages] | tfull[2] | tempty0[2] | tempty1 |
  //         claim[LM_TRING] | epi | drain | done | tmem slot, CTA 1's slabs, tile ring | scratch
  const uint32_t hbase = base + wst_n * LM_A_BYTES;
  const uint32_t bar_full = hbase + hst_n * b_bytes;
  const uint32_t bar_empty = bar_full + 8 * wst_n;
  const uint32_t bar_tfull = bar_empty + 8 * wst_n;
  const uint32_t bar_tempty0 = bar_tfull + 16;
  const uint32_t bar_tempty1 = bar_tempty0 + 16;
  const uint32_t bar_claim = bar_tempty1 + 8;
  const uint32_t bar_epi = bar_claim + 8 * LM_TRING;
  const uint32_t bar_drain = bar_epi + 8;
  const uint32_t bar_done = bar_drain + 8;  // CTA 0: CTA 1's producer has asked for its last slab
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + (bar_done + 8 - base));
  uint32_t* peer_slabs = tmem_slot + 1;     // CTA 0: how many that were
  int32_t* tring = reinterpret_cast<int32_t*>(tmem_slot + 4);  // [LM_TRING] claimed tiles
  float2* wst = reinterpret_cast<float2*>(gbase + ((bar_done + 8 - base + 16 + 4 * LM_TRING + 15) & ~15u));
  float2* wag = wst + 4 * S_pad;                           // [4][S_pad] per-warp argmax
  float* wu2 = reinterpret_cast<float*>(wag + 4 * S_pad);  // [4][S_pad] per-warp runner-up
  float2* ccoef = wag + 6 * S_pad;                         // [S_pad] (1 + beta, beta) per column
  uint32_t* cmask = reinterpret_cast<uint32_t*>(ccoef + S_pad);  // [2][16] amateur / expert column bits
  float* bc = reinterpret_cast<float*>(cmask + 32);        // [8][64] per-warp column broadcast

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  if (tid == 0) {
    for (uint32_t i = 0; i < wst_n; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_tfull + 8 * i, 1);
      mbar_init(bar_tempty0 + 8 * i, 2 * LM_EPI_THREADS / 32);
    }
    mbar_init(bar_tempty1, 2 * LM_EPI_THREADS / 32);
    for (int i = 0; i < LM_TRING; ++i) mbar_init(bar_claim + 8 * i, 1);
    mbar_init(bar_epi, LM_EPI_THREADS);
    mbar_init(bar_drain, 1);
    mbar_init(bar_done, 1);
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&wmap);
    tma_prefetch_desc(&hmap0);
    if (nc1) tma_prefetch_desc(&hmap1);
  }
  if (a.mode == 1) pdl_launch_dependents();
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), 512);
  if (a.mode == 1) column_tables(a, tid, ccoef, cmask);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are ready
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const int nks = a.nks, ntiles = (a.ntiles + 1) / 2;  // tiles of 256 vocabulary rows
  const bool dbl = a.acc_bufs == 2;
  const uint32_t col1 = (dbl ? 2u : 1u) * (uint32_t)n0;  // TMEM column of chunk 1

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    const uint32_t on = elect_one();
    const uint64_t pol_w = policy_evict_first(), pol_h = policy_evict_last();
    const uint32_t full0 = mapa(bar_full, 0);  // CTA 0's full barriers
    int tile = -1, ks = 0;
    uint32_t tseq = 0;
    bool ok = true;
    // tile tseq of the pair: claimed by CTA 0 from the global counter (without
    // one, the pairs' tiles in turn) and handed to both CTAs (-1 ends); a ring entry is used again LM_TRING
    // tiles later, when every role of both CTAs is past it
    auto claim = [&]() {
      const uint32_t i = tseq % LM_TRING;
      int t = -1;
      if (rank == 0) {
        if (lane == 0) {
          t = a.tile_ctr ? atomicAdd(a.tile_ctr, 1) : (int)((blockIdx.x >> 1) + tseq * (gridDim.x >> 1));
          if (t >= ntiles) t = -1;
          tring[i] = t;
          st_cluster_u32(mapa(smem_u32(tring + i), 1), (uint32_t)t);
          mbar_arrive_cluster(mapa(bar_claim + 8 * i, 1));
          mbar_arrive(bar_claim + 8 * i);
        }
      } else {
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(bar_claim + 8 * i, (tseq / LM_TRING) & 1u, a.status));
        if (ok) t = *(volatile int32_t*)(tring + i);
      }
      tile = __shfl_sync(0xffffffffu, t, 0);
      ++tseq;
      ks = 0;
    };
    // slab it of W (the tile's next) into stage w of its ring; its full barrier
    // counts the bytes of the slab's W and H of both CTAs
    auto load_w = [&](uint32_t w) {
      mbar_arrive_expect_tx_if(on & (rank ^ 1u), bar_full + 8 * w, 2 * (LM_A_BYTES + b_bytes));
      tma_load_2d_pair(on, base + w * LM_A_BYTES, &wmap, full0 + 8 * w, ks * LM_TILE_K,
                       (2 * tile + (int)rank) * LM_TILE_V, pol_w);
      if (++ks == nks) claim();
    };
    // H of the slab in W stage w into stage h of its ring
    int hks = 0;
    auto load_h = [&](uint32_t h, uint32_t w) {
      tma_load_2d_pair(on, hbase + h * b_bytes, &hmap0, full0 + 8 * w, hks * LM_TILE_K, (int)rank * (n0 / 2), pol_h);
      if (nc1)
        tma_load_2d_pair(on, hbase + h * b_bytes + n0 * 64, &hmap1, full0 + 8 * w, hks * LM_TILE_K,
                         n0 + (int)rank * (nc1 / 2), pol_h);
      if (++hks == nks) hks = 0;
    };
    if (a.pdl == LM_PDL_ALL) pdl_wait();
    claim();
    // first fill; with programmatic dependent launch W streams while the
    // previous kernel (which writes H) finishes
    uint32_t nw = 0, nh = 0;  // slabs of W and of H issued
    while (tile >= 0 && nw < wst_n) load_w(nw++);
    if (a.pdl == LM_PDL_H) pdl_wait();
    for (; nh < hst_n && nh < nw; ++nh) load_h(nh, nh);
    // with slab n consumed, its W stage takes slab n + wst_n and its H stage slab n + hst_n
    uint32_t w = 0, wph = 0, h = 0, hw = nh == wst_n ? 0 : nh;
    while (tile >= 0 || nh < nw) {
      if (!mbar_wait_warp(bar_empty + 8 * w, wph, a.status)) {
        ok = false;
        break;
      }
      if (tile >= 0) {
        load_w(w);
        ++nw;
      }
      load_h(h, hw);
      ++nh;
      if (++w == wst_n) {
        w = 0;
        wph ^= 1u;
      }
      if (++h == hst_n) h = 0;
      if (++hw == wst_n) hw = 0;
    }
    // a producer that gave up leaves whole slabs behind: their H follows their W
    while (nh < nw) {
      load_h(h, hw);
      ++nh;
      if (++h == hst_n) h = 0;
      if (++hw == wst_n) hw = 0;
    }
    if (rank == 1 && lane == 0) {
      st_cluster_u32(mapa(smem_u32(peer_slabs), 0), nw);
      mbar_arrive_cluster(mapa(bar_done, 0));
    }
    // CTA 0's commits arrive on the barriers of both CTAs, and an arrival must
    // not find its CTA gone: both producers see the last commit of every stage,
    // and CTA 1's the one after the last MMA too, which nothing else waits for
    // there (CTA 0's MMA warp does; the epilogues wait for the tiles' commits)
    for (uint32_t j = nw > wst_n ? nw - wst_n : 0; ok && j < nw; ++j)
      ok = mbar_wait_warp(bar_empty + 8 * (j % wst_n), (j / wst_n) & 1u, a.status);
    if (rank == 1) {
      mbar_wait_warp(bar_drain, 0, a.status);
    } else {
      // CTA 1 may be at a wait that runs out one limit later; then both CTAs'
      // copies land before either leaves the cluster barrier below (with every
      // stage's last commit seen there are none)
      const bool met = mbar_wait_cluster(bar_done, 0, a.status) || mbar_wait_cluster(bar_done, 0, a.status);
      const uint32_t n1 = met ? *(volatile uint32_t*)peer_slabs : nw;
      PairFull full{on, bar_full, LM_A_BYTES + b_bytes, a.status};
      if (!ok) lm_pair_drain(nw, __shfl_sync(0xffffffffu, n1, 0), wst_n, full);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    if (rank == 0) {
      const uint32_t on = elect_one();
      const uint32_t idesc0 = umma_idesc_bf16(2 * LM_TILE_V, n0), idesc1 = umma_idesc_bf16(2 * LM_TILE_V, nc1);
      const uint32_t coff = (uint32_t)(n0 * 64) >> 4;
      uint32_t st = 0, ph = 0, h = 0;
      bool ok = true;
      for (uint32_t acc = 0; ok; ++acc) {
        if (!mbar_wait_warp(bar_claim + 8 * (acc % LM_TRING), (acc / LM_TRING) & 1u, a.status)) break;
        if (__shfl_sync(0xffffffffu, *(volatile int32_t*)(tring + acc % LM_TRING), 0) < 0) break;
        // both CTAs' epilogues have read what these columns held
        const uint32_t b0 = dbl ? acc & 1u : 0u, use0 = dbl ? acc >> 1 : acc;
        bool free = mbar_wait_cluster(bar_tempty0 + 8 * b0, (use0 & 1u) ^ 1u, a.status);
        if (nc1) free = free && mbar_wait_cluster(bar_tempty1, (acc & 1u) ^ 1u, a.status);
        if (!__all_sync(0xffffffffu, free)) break;
        tc_fence_after();
        const uint32_t d0 = tmem_base + b0 * n0, d1 = tmem_base + col1;
        for (int ks = 0; ks < nks; ++ks) {
          if (!mbar_wait_warp(bar_full + 8 * st, ph, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = umma_desc_sw128(base + st * LM_A_BYTES), bd = umma_desc_sw128(hbase + h * b_bytes);
          if (nc1) {
#pragma unroll
            for (int k = 0; k < LM_TILE_K / 16; ++k) {
              umma_bf16_pair(on, d0, ad + 2 * k, bd + 2 * k, idesc0, (ks | k) != 0);
              umma_bf16_pair(on, d1, ad + 2 * k, bd + coff + 2 * k, idesc1, (ks | k) != 0);
            }
          } else {
#pragma unroll
            for (int k = 0; k < LM_TILE_K / 16; ++k)
              umma_bf16_pair(on, d0, ad + 2 * k, bd + 2 * k, idesc0, (ks | k) != 0);
          }
          umma_commit_pair(on, bar_empty + 8 * st);
          if (++st == wst_n) {
            st = 0;
            ph ^= 1u;
          }
          if (++h == hst_n) h = 0;
        }
        if (ok) umma_commit_pair(on, bar_tfull + 8 * (acc & 1u));
      }
      // all issued MMAs complete before TMEM is released
      umma_commit_pair(on, bar_drain);
      mbar_wait_warp(bar_drain, 0, a.status);
    }
    __syncwarp();
  } else {
    // ----------------------------------------------------------- epilogue
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    const int etid = tid - 64, half = (warp - 2) >> 2;
    const int S = a.S, n1 = a.N + 1;
    const int nb1 = S > n0 ? (S - n0 + 31) / 32 : 0, nb0 = ((S < n0 ? S : n0) + 31) / 32;  // 32-column blocks
    const uint32_t tempty0 = mapa(bar_tempty0, 0), tempty1 = mapa(bar_tempty1, 0);
    float* wbc = bc + 64 * (warp - 2);
    uint32_t ephase = 0;
    for (uint32_t acc = 0;; ++acc) {
      if (!mbar_wait_cluster(bar_claim + 8 * (acc % LM_TRING), (acc / LM_TRING) & 1u, a.status)) break;
      const int tile2 = *(volatile int32_t*)(tring + acc % LM_TRING);
      if (tile2 < 0) break;
      if (!mbar_wait(bar_tfull + 8 * (acc & 1u), (acc >> 1) & 1u, a.status)) break;
      tc_fence_after();
      const int tile = 2 * tile2 + (int)rank;  // this CTA's 128 rows
      const int v = tile * LM_TILE_V + 32 * q + lane;
      const bool valid = v < a.V;
      const uint32_t b0 = dbl ? acc & 1u : 0u;
      const uint32_t trow = tmem_base + ((uint32_t)(32 * q) << 16);
      auto tcol = [&](int c) { return trow + (c < n0 ? b0 * n0 + c : col1 + (c - n0)); };
      // a chunk's columns are free for the next tile's MMAs once this warp's
      // last ones of them are in its registers
      auto release = [&](uint32_t bar) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(bar);
      };
      auto blocks = [&](int cbase, int kb0, int nb, uint32_t bar) {
        if (kb0 >= nb) release(bar);
        for (int kb = kb0; kb < nb; kb += 2) {
          const int c0 = cbase + 32 * kb;
          float z_am = 0.f;
          if (a.mode == 1 && c0 % n1 != 0) z_am = tmem_ld1(tcol(c0 - c0 % n1));  // the open query's amateur logit
          epi_block<32>(a, tcol(c0), c0, v, valid, lane, q, wbc, wst, wag, wu2, ccoef, cmask, z_am, [&]() {
            if (kb + 2 >= nb) release(bar);
          });
        }
      };
      if (nc1) blocks(n0, half, nb1, tempty1);
      blocks(0, (nb1 & 1) ? 1 - half : half, nb0, tempty0 + 8 * b0);
      if (!bar_sync_bounded(bar_epi, ephase, a.status)) break;
      // the last pair's second half may hold no rows
      if (PCED_IN_BOUNDS(tile2 < ntiles, a.status) && tile < a.ntiles) fold_tile(a, tile, etid, wst, wag, wu2);
      if (!bar_sync_bounded(bar_epi, ephase, a.status)) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA's shared memory, barriers or TMEM is used by the other any more:
  // both have seen every arrival on a barrier of theirs (above)
  cluster_sync_all();
  if (a.mode == 0) pdl_launch_dependents();  // see lm_head.cu
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

cudaError_t lm_head_pair_launch(const LmMaps& m, const LmGeom& g, const LmArgs& a, cudaStream_t stream) {
  static bool configured[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(lm_head_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LM_SMEM_BUDGET);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  return pced_host::launch_kernel(lm_head_pair_kernel, dim3(g.grid), LM_THREADS, g.smem, stream, a.pdl != 0,
                                  m.w, m.h[0], m.h[1], a);
}

}  // namespace pced
