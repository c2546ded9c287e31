// lm_epilogue.cuh -- the LM head kernels' epilogue: per-column statistics of 32
// vocabulary rows held one per lane, and their fold into a tile's records.
#pragma once
#include "lm_head.cuh"

namespace pced {

// Top-2 over tokens of (value, token) candidates whose token sets are
// disjoint: (b1, t1) the best (larger value, then lower token), b2 the best
// value at another token; merges the candidate set (r1, rt, r2) into it.
__device__ __forceinline__ void top2_merge(float& b1, int& t1, float& b2, float r1, int rt, float r2) {
  if (r1 > b1 || (r1 == b1 && rt < t1)) {
    b2 = fmaxf(b1, r2);
    b1 = r1;
    t1 = rt;
  } else {
    b2 = fmaxf(b2, r1);
  }
}

struct FMax {
  __device__ __forceinline__ float operator()(float x, float y) const { return fmaxf(x, y); }
};
struct FAdd {
  __device__ __forceinline__ float operator()(float x, float y) const { return x + y; }
};

// Reduce NB columns held one per register over the 32 lanes (vocabulary rows)
// of a warp in transposed form: every exchange hands half of the columns still
// held to the partner lane, so NB columns cost NB - 1 shuffles instead of
// 5 NB.  The pairing (lane bit 4 first, bit 0 last) is that of a per-column
// xor tree, so sums round identically.  NB = 32: lane l ends with column l;
// NB = 16 or 8: full exchanges across the lane bits at and above NB first, so
// every lane l ends with column l & (NB - 1).
template <int NB, class Op>
__device__ __forceinline__ float bfly_reduce(float (&x)[NB], int lane, Op op) {
#pragma unroll
  for (int w = 16; w >= NB; w >>= 1) {
#pragma unroll
    for (int i = 0; i < NB; ++i) x[i] = op(x[i], __shfl_xor_sync(0xffffffffu, x[i], w));
  }
#pragma unroll
  for (int w = NB / 2; w >= 1; w >>= 1) {
    const bool hi = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = hi ? x[i] : x[i + w];
      const float keep = hi ? x[i + w] : x[i];
      x[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, w));
    }
  }
  return x[0];
}

// Top-2 over the 32 lanes (vocabulary rows) of NB columns held one per
// register, in the transposed form of bfly_reduce: (best value, its token,
// best value at another token) travel together, ties to the lower token.
// Lane l ends with column l & (NB - 1).  `tok` is this lane's token.
template <int NB>
__device__ __forceinline__ void bfly_top2(const float (&u)[NB], int tok, int lane, float& r1, int& rt, float& r2) {
  constexpr int K = NB == 32 ? 16 : NB;  // slots after the first level
  float b1[K], b2[K];
  int bt[K];
  const int ptok = tok + ((lane ^ 16) - lane);  // the row across lane bit 4
  const bool hi16 = (lane & 16) != 0;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    // NB = 32: the first halving level; NB <= 16: a full exchange
    const float send = NB == 32 ? (hi16 ? u[i] : u[(i + 16) % NB]) : u[i];
    const float keep = NB == 32 ? (hi16 ? u[(i + 16) % NB] : u[i]) : u[i];
    const float o = __shfl_xor_sync(0xffffffffu, send, 16);
    const bool take = o > keep || (o == keep && ptok < tok);
    b1[i] = take ? o : keep;
    bt[i] = take ? ptok : tok;
    b2[i] = take ? keep : o;
  }
  // NB = 8: one more full exchange, across lane bit 3
#pragma unroll
  for (int w = 8; w >= NB; w >>= 1) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const float o1 = __shfl_xor_sync(0xffffffffu, b1[i], w), o2 = __shfl_xor_sync(0xffffffffu, b2[i], w);
      const int ot = __shfl_xor_sync(0xffffffffu, bt[i], w);
      top2_merge(b1[i], bt[i], b2[i], o1, ot, o2);
    }
  }
#pragma unroll
  for (int w = (NB == 32 ? 8 : NB / 2); w >= 1; w >>= 1) {
    const bool hi = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float s1 = hi ? b1[i] : b1[i + w], s2 = hi ? b2[i] : b2[i + w];
      const int st = hi ? bt[i] : bt[i + w];
      float k1 = hi ? b1[i + w] : b1[i], k2 = hi ? b2[i + w] : b2[i];
      int kt = hi ? bt[i + w] : bt[i];
      const float o1 = __shfl_xor_sync(0xffffffffu, s1, w), o2 = __shfl_xor_sync(0xffffffffu, s2, w);
      const int ot = __shfl_xor_sync(0xffffffffu, st, w);
      top2_merge(k1, kt, k2, o1, ot, o2);
      b1[i] = k1;
      bt[i] = kt;
      b2[i] = k2;
    }
  }
  r1 = b1[0];
  rt = bt[0];
  r2 = b2[0];
}

// Epilogue of NB accumulator columns c0.. (c0 a multiple of NB) of one
// warp's 32 vocabulary rows: mode 0 stores the logits; both modes record the
// per-column (max, sum of exp) of the 32 rows; mode 1 also records per expert
// column the max of u_k = (1 + beta) z_k - beta z_0, its first (lowest)
// vocabulary index and the best value at another index.  `bc` is this warp's
// broadcast buffer; z_am carries the row's amateur logit from its query's
// first column to the expert columns; ccoef / cmask hold each column's
// (1 + beta, beta) and the amateur / expert column bits of each 32-column
// block (the same for every tile).  `loaded` runs once the accumulator's
// columns are in registers.
template <int NB, class F>
__device__ __forceinline__ void epi_block(const LmArgs& a, uint32_t taddr, int c0, int v, bool valid, int lane,
                                          int q, float* bc, float2* wst, float2* wag, float* wu2, const float2* ccoef,
                                          const uint32_t* cmask, float& z_am, F loaded) {
  const int S = a.S, S_pad = a.S_pad;
  float z[NB], t[NB];
  if (NB == 32)
    tmem_ld32(taddr, z);
  else if (NB == 16)
    tmem_ld16(taddr, z);
  else
    tmem_ld8(taddr, z);
  loaded();
  if (a.mode == 0 && valid) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (c0 + i < S) a.logits[(int64_t)(c0 + i) * a.V + v] = z[i];
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) t[i] = valid ? z[i] : -INFINITY;
  float u[NB];
  const uint32_t em = a.mode == 1 ? cmask[16 + (c0 >> 5)] >> (c0 & 31) : 0u;
  if (a.mode == 1) {
    const uint32_t am = cmask[c0 >> 5] >> (c0 & 31);
    float za = z_am;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if ((am >> i) & 1u) za = z[i];
      const float2 cf = ccoef[c0 + i];
      u[i] = valid && ((em >> i) & 1u) ? cf.x * z[i] - cf.y * za : -INFINITY;
    }
    z_am = za;
  }
  const float m = bfly_reduce<NB>(t, lane, FMax());
  float b1 = -INFINITY, b2 = -INFINITY;
  int bt = 0;
  if (a.mode == 1) bfly_top2<NB>(u, v, lane, b1, bt, b2);
  const int li = lane & (NB - 1), mycol = c0 + li;
  if (lane < NB) bc[lane] = m;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < NB; ++i) t[i] = valid ? __expf(z[i] - bc[i]) : 0.f;
  const float sm = bfly_reduce<NB>(t, lane, FAdd());
  if (lane < NB && mycol < S) {
    wst[q * S_pad + mycol] = make_float2(m, sm);
    if ((em >> li) & 1u) {
      wag[q * S_pad + mycol] = make_float2(b1, __int_as_float(bt));
      wu2[q * S_pad + mycol] = b2;
    }
  }
  __syncwarp();
}

// A tile's records: the four lane quarters' results folded in a fixed order,
// stored per tile so the cross-tile merge order does not depend on which CTA
// took the tile.
__device__ __forceinline__ void fold_tile(const LmArgs& a, int tile, int etid, const float2* wst, const float2* wag,
                                          const float* wu2) {
  const int n1 = a.N + 1, S_pad = a.S_pad;
  for (int col = etid; col < a.S; col += LM_EPI_THREADS) {
    float cm = -INFINITY, cs = 0.f;
#pragma unroll
    for (int qq = 0; qq < 4; ++qq) {
      const float2 r = wst[qq * S_pad + col];
      lse_merge(cm, cs, r.x, r.y);
    }
    a.rec_stats[(int64_t)col * a.ntiles + tile] = make_float2(cm, cs);
    if (a.mode == 1 && col % n1 != 0) {
      float bu = -INFINITY, b2 = -INFINITY;
      int bv = 0x7fffffff;
#pragma unroll
      for (int qq = 0; qq < 4; ++qq) {
        const float2 r = wag[qq * S_pad + col];
        top2_merge(bu, bv, b2, r.x, __float_as_int(r.y), wu2[qq * S_pad + col]);
      }
      a.rec_arg[(int64_t)col * a.ntiles + tile] = make_float2(bu, __int_as_float(bv));
      a.rec_u2[(int64_t)col * a.ntiles + tile] = b2;
    }
  }
}

// Per column: expert columns carry (1 + beta_k, beta_k); the amateur column of
// each query starts its group; bit i of block kb is column 32 kb + i.
__device__ __forceinline__ void column_tables(const LmArgs& a, int tid, float2* ccoef, uint32_t* cmask) {
  const int n1 = a.N + 1, lane = tid & 31;
  for (int c = tid; c < a.S_pad; c += LM_THREADS) {
    const int j = c % n1, bq = c / n1;
    const float bt = c < a.S && j > 0 ? a.beta[bq * a.N + j - 1] : 0.f;
    ccoef[c] = make_float2(1.f + bt, bt);
  }
  if (tid < 32)
    for (int kb = 0; kb < 16; ++kb) {
      const int c = 32 * kb + lane;
      const bool in = c < a.S;
      const uint32_t am = __ballot_sync(0xffffffffu, in && c % n1 == 0);
      const uint32_t em = __ballot_sync(0xffffffffu, in && c % n1 != 0);
      if (lane == 0) {
        cmask[kb] = am;
        cmask[16 + kb] = em;
      }
    }
}

}  // namespace pced
