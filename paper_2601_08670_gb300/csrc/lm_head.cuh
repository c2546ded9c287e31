// lm_head.cuh -- unembedding GEMM with fused log-softmax statistics and the
// contrastive per-tile maxima, plus the cross-tile reductions.
#pragma once
#include "common.cuh"

namespace pced {

constexpr int LM_EPI_THREADS = 256;  // eight epilogue warps: two per TMEM lane quarter, each half of the columns
constexpr int LM_THREADS = 64 + LM_EPI_THREADS;  // warp 0 TMA, warp 1 MMA + TMEM owner, warps 2-9 epilogue
constexpr int LM_TILE_V = 128;   // vocabulary rows per tile (UMMA M)
constexpr int LM_TILE_K = 64;    // hidden elements per stage (one 128-byte swizzle row)
constexpr int LM_MAX_S = 512;
constexpr int LM_MAX_N1 = 256;   // experts + amateur per query in the selection kernels
constexpr int LM_TRING = 32;     // claimed-tile ring between the TMA and the other warps (> stages + 3 tiles in flight)

constexpr int LM_A_BYTES = LM_TILE_V * LM_TILE_K * 2;  // 16 KB
constexpr size_t LM_SMEM_BUDGET = 227 * 1024;
// From this many hidden rows on a tile is taken by a pair of CTAs
// (lm_head_pair.cu), below by one (lm_head.cu), which TMEM allows up to 256 rows.
// One CTA / pairs, us a call in a graph: d = 4096, V = 128256 185 / 185 at 128
// rows, 198 / 194 at 160, 209 / 203 at 192, 248 / 232 at 256; d = 4096, V = 8000
// 27.4 / 27.1, 28.5 / 29.4, 35.1 / 34.5 at 160, 192, 256; d = 1792, V = 30000 36.2 /
// 37.0 and 42.2 / 42.0 at 192 and 256.  The line is drawn for such rows; with
// shorter ones one CTA stays ahead up to 256 rows, which the rule leaves: d =
// 1024, V = 50000 40.8 / 44.4 and 50.1 / 52.2 at 192 and 256, d = 512, V = 8192 14.8 /
// 16.8 and 17.4 / 19.1, d = 64 at most 14 % more.
constexpr int LM_PAIR_MIN_S = 161;

struct LmGeom {
  bool pair;
  int32_t S, S_pad, chunk_n, d, V, ntiles, nks, slabs, nst, stages, hstages, acc_bufs, grid;
  uint32_t tmem_cols;
  size_t smem;
};
// returns false when the shape is unsupported
bool lm_geometry(int32_t S, int32_t d, int32_t V, LmGeom* g);

// Of the kernel that writes H: the weights are read, tiles claimed and beta's
// coefficients formed before it ends.  That kernel must write none of these, and
// must itself be launched in full stream order (att_step_launch is), so that
// the selection before it has reset the tile counter and any upload of beta has
// landed.
constexpr int LM_PDL_H = 1;
constexpr int LM_PDL_ALL = 2;  // of any kernel: nothing is read before it ends

struct LmArgs {
  int mode;  // 0: write logits[S][V]; 1: contrastive records (needs N, beta)
  int32_t S, N, V, ntiles, nks, slabs, nst, stages, acc_bufs, S_pad;
  int32_t hstages;    // pair: stages of the H ring (stages: of the W ring)
  int32_t chunk_n;    // accumulator columns of the first N chunk (pair: S_pad - chunk_n in a second one)
  uint32_t tmem_cols;
  float* logits;      // mode 0
  float2* rec_stats;  // [S][ntiles] (max z, sum exp(z - max)) of each vocabulary tile
  float2* rec_arg;    // [S][ntiles] (max u, argmax v as int bits) for expert columns, mode 1
  float* rec_u2;      // [S][ntiles] the tile's second-largest u (another token), mode 1
  int* tile_ctr;      // tiles claimed so far (zero at launch), or null: dealt out in turn
  const float* beta;  // [B][N]
  int pdl;            // launched as a programmatic dependent: LM_PDL_H, LM_PDL_ALL (0: not)
  int* status;
};

// The copies of a pair that are still on their way when a producer has given
// up.  n0, n1: slabs (of W and H) that CTA 0 and CTA 1 have asked for, whose
// bytes CTA 0's full barriers count; for a slab of its own CTA 0 has arrived on
// its stage's barrier with the bytes of both.  The two counts differ by at most
// `stages`: neither asks for slab n before slab n - stages has been consumed.
// Waits until every copy of both has landed; false if that wait runs out.
#pragma nv_exec_check_disable  // (the barriers are the device's, or a model of them on the host)
template <class Ring>
__host__ __device__ inline bool lm_pair_drain(uint32_t n0, uint32_t n1, uint32_t stages, Ring& ring) {
  const uint32_t n = n0 > n1 ? n0 : n1;
  for (uint32_t j = n0; j < n; ++j) ring.expect_one(j % stages);  // CTA 1 alone asked for it: its bytes
  for (uint32_t j = n1; j < n; ++j) ring.missing_one(j % stages);  // CTA 0 alone did: the other bytes never come
  for (uint32_t j = n > stages ? n - stages : 0; j < n; ++j)
    if (!ring.wait(j % stages, (j / stages) & 1u)) return false;
  return true;
}

struct LmMaps {
  CUtensorMap w, h[2];  // W tiles; H rows of the N chunks
};
pced_status lm_head_maps(const void* w_unembed, const void* hidden, const LmGeom& g, LmMaps* m);
LmArgs lm_args(const LmGeom& g);  // the geometry's fields; the others zero
cudaError_t lm_head_launch(const LmMaps& m, const LmGeom& g, const LmArgs& a, cudaStream_t stream);
cudaError_t lm_head_pair_launch(const LmMaps& m, const LmGeom& g, const LmArgs& a, cudaStream_t stream);
// mode-0 finish: lse[s] from the tile records, logits -> log-probs in place, in
// one launch (fused) or two (pdl: as programmatic dependents)
cudaError_t lm_lse_finalize_launch(float* logits, const float2* rec_stats, float* lse, int32_t S, int32_t V,
                                   int32_t nrec, bool fused, bool pdl, cudaStream_t stream);

// Selection from mode-1 records (Eq. 2 + Eq. 3), one cluster per query.
struct SelectArgs {
  const float2* rec_stats;
  const float2* rec_arg;
  const float* rec_u2;
  int32_t B, N, nrec;  // records per row (the LM head's vocabulary tiles)
  int32_t V;
  int* tile_ctr;       // optional: the LM head's tile counter, reset here for its next launch
  const float* beta;
  const float* r;
  float gamma;
  int32_t* token;     // optional [B]
  int32_t* expert;    // optional [B]
  float* score;       // optional [B]
  float* lse_out;     // optional [S]
  // step bookkeeping (optional): history[b][t] etc. with t = *step, then *step += 1
  int32_t* step;
  int32_t* history;
  int32_t* expert_trace;
  float* score_trace;
  int32_t max_steps;
  int32_t* done_counter;
  // near-tie margins of the choice (optional): gap_trace[b][t] = (token gap,
  // expert gap); the expert gap recomputes z_s(y) = h_s . W[y] for the
  // query's rows
  float2* gap_trace;
  int64_t* key_out;   // expert-partitioned step: packed choices [B], nothing appended
  int32_t expert_base;
  const __nv_bfloat16* hidden;     // [S][d]
  const __nv_bfloat16* w_unembed;  // [V][d]
  int32_t d;
  int pdl;            // launched as a programmatic dependent of the LM head
  int raw_logits;     // s_k of Eq. 2 are the raw logits: c_k = gamma log r_k alone
  int* status;
};
cudaError_t select_from_records_launch(const SelectArgs& a, cudaStream_t stream);

}  // namespace pced
