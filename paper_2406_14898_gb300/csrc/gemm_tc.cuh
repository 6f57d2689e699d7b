// Persistent tcgen05 GEMM for sm_103a with fused epilogues.
//
// D[M,N] = epilogue(A . B^T): bf16 operands staged by TMA (128-byte swizzle) into a
// STAGES-deep shared-memory ring, one elected thread issues tcgen05.mma kind::f16
// (M=128, N=BN, K=16) into a double-buffered fp32 TMEM accumulator, and eight
// epilogue warps drain TMEM with tcgen05.ld while the next tile's main loop runs.
// An epilogue warp owns 32 rows of the tile (its TMEM lane quarter) and half of its columns;
// it moves each 32x64 fp32 chunk through 8 KB of
// shared memory so that, row by row, its lanes handle consecutive columns and every global
// load and store of the epilogue is coalesced.  The epilogue's own operands (residual,
// gradient accumulator, AdamW state) are read one batch of rows ahead of their use, across
// chunks and tiles, the first batch of a tile before its accumulator is complete.
//
// Operand majorness is a template parameter: K-major operands are [rows, K] row-major
// (one TMA box of 64 x rows per stage), MN-major operands are [K, rows] row-major
// (rows/64 boxes of 64 x BK per stage).  The three GEMM families of a transformer
// block map onto it as
//   forward  X[T,K]  . W[N,K]^T          A K-major,  B K-major
//   dgrad    dY[T,N] . W[N,K]            A K-major,  B MN-major
//   wgrad    dY[T,N]^T . X[T,K]          A MN-major, B MN-major  (fp32 accumulate)
//
// Warp roles (320 threads): warp 0 TMA producer, warp 1 TMEM owner + MMA issuer,
// warps 2..9 epilogue (warp w reads TMEM lanes 32*(w%4) .. +31, column half (w-2)/4).  The
// AdamW families have four epilogue warps (192 threads), see adamw_epilogue.
#pragma once
#include <cuda.h>
#include <atomic>
#include <cstdio>
#include <mutex>

#include "../../include/flglm_kernels.h"
#include "common.cuh"
#include "ptx.cuh"

namespace fl_gemm {

constexpr int BM = 128;
constexpr int BK = 64;  // one 128-byte swizzle row of bf16
constexpr int UMMA_K = 16;
// Bytes of operand panels kept resident per raster group: 32 MB while K <= 8192, 48 MB for
// the longer panels of K = 12288 / 16384 (measured on GB300 at the stack26 shapes: DRAM
// reads of the up-projection 827 -> 554 MB and the weight gradients 8-10 us faster at 32
// MB; the K = 16384 / 12288 data gradients and down-projection best at 48 MB).
constexpr double L2_GROUP_BUDGET = 48.0 * (1 << 20);
constexpr double L2_GROUP_BUDGET_SHORT_K = 32.0 * (1 << 20);

// Epilogue families: each kernel instantiation carries only its family's code, which keeps
// the kernel small enough for the instruction cache (the MMA-issuing warp shares it).
enum { FAM_PLAIN = 0, FAM_GELU = 1, FAM_RESID = 2, FAM_ROPE = 3, FAM_ADAMW = 4, FAM_ADAMW_LONG = 5, FAM_F32 = 6 };
__host__ __device__ constexpr int family_of(int mode) {
  return (mode == FL_EPI_BIAS_GELU || mode == FL_EPI_GELU_BWD) ? FAM_GELU
         : (mode == FL_EPI_BIAS_RESID || mode == FL_EPI_RESID) ? FAM_RESID
         : mode == FL_EPI_BIAS_ROPE                            ? FAM_ROPE
         : mode == FL_EPI_ADAMW                                ? FAM_ADAMW
                                                               : FAM_PLAIN;
}

// ------------------------------------------------------------------ AdamW epilogue
// The weight-gradient GEMMs' fused update moves 26 B per output element (w, m, v read; w, m,
// v and the bf16 copy written), which bounds the launch while the contraction (the call's
// tokens) is short.  Its operands therefore travel by TMA: each of four epilogue warps owns
// 32 rows of the tile and walks it in chunks of CC columns, the chunk's w, m and v loaded
// SLOTS - 1 chunks ahead (across tiles, before the accumulator they belong to is complete)
// into a ring slot of its own; a lane updates the CC elements of its row in place, the
// gradient read from TMEM straight into registers, and the slot leaves by TMA stores.
// Two 4096 x 16384 weights at 77 tokens: 630 us, 5.5 TB/s (1048 us, 3.3 TB/s with loads and
// stores from registers on four warps).  CC = 32 with two slots: 603 us, but three operand
// stages instead of four (770 against 730 us at 2048 tokens); CC = 16 with two: 800 us.
struct AdamRing {
  static constexpr int CC = 16;     // columns per chunk (64 B rows of fp32, 64-byte swizzle)
  static constexpr int SLOTS = 3;   // per warp
  static constexpr int WARPS = 4;
  static constexpr int TENSOR = 32 * CC * 4;                // one chunk of w, m or v
  static constexpr int SLOT = 3 * TENSOR + 32 * CC * 2;     // and the bf16 copy's
  static constexpr int BYTES = WARPS * SLOTS * SLOT;
};

// The fp32 gradients' epilogue (stored, or added to what is there) the same way, one tensor, chunks of
// whole 128-byte rows (128-byte swizzle).
struct F32Ring {
  static constexpr int CC = 32;
  static constexpr int SLOTS = 4;
  static constexpr int WARPS = 4;
  static constexpr int SLOT = 32 * CC * 4;
  static constexpr int BYTES = WARPS * SLOTS * SLOT;
};

// Epilogue warps of a family at tile width BN (64 columns give eight warps nothing to share)
// and the shared memory they work in: the AdamW ring, or one 32x64 fp32 chunk per warp.
template <int FAM, int BN>
struct EpiCfg {
  static constexpr int WARPS = FAM == FAM_ADAMW  ? AdamRing::WARPS
                               : FAM == FAM_F32 ? F32Ring::WARPS
                               : FAM == FAM_ADAMW_LONG || BN == 64 ? 4 : 8;
  static constexpr int THREADS = 64 + 32 * WARPS;
  static constexpr int BYTES = FAM == FAM_ADAMW ? AdamRing::BYTES : FAM == FAM_F32 ? F32Ring::BYTES : WARPS * 32 * 64 * 4;
  // barriers of its own: the rings', or the column sums' (written and read, per column half)
  static constexpr int BARS = FAM == FAM_ADAMW  ? WARPS * AdamRing::SLOTS
                              : FAM == FAM_F32  ? WARPS * F32Ring::SLOTS
                              : FAM == FAM_GELU ? 4 : 0;
  static constexpr int bar_count(int i) { return FAM == FAM_GELU && i % 2 == 0 ? 4 : 1; }
};
// Depth of the operand ring for stages of `bytes`: what fits beside the epilogue's shared
// memory, six stages at most (deeper gains nothing).
constexpr int SMEM_MAX = 227 * 1024;
constexpr int BAR_BYTES = 256;
constexpr int ring_stages(int bytes, int epi_bytes) {
  const int n = (SMEM_MAX - 1024 - BAR_BYTES - epi_bytes) / bytes;
  return n < 6 ? n : 6;
}

// k-blocks per stage: the products of one k-block of a 128 x 64 tile are shorter than a
// stage's barrier round trip, so a stage of that shape holds two (4096 columns, K = 16384, 77
// rows: 67 -> 51 us; the 256 x 128 pair tile, left three such stages, would lose: 63 -> 68 us).

template <int BN, int FAM>
struct Cfg {
  static constexpr int KSUB = BN == 64 ? 2 : 1;
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = KSUB * (A_BYTES + B_BYTES);
  static constexpr int STAGES = ring_stages(STAGE_BYTES, EpiCfg<FAM, BN>::BYTES);
  static constexpr int TMEM_COLS = 2 * BN;  // double-buffered accumulator
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EpiCfg<FAM, BN>::BYTES + BAR_BYTES + 1024 /*align*/;
  static_assert((2 * STAGES + 5 + EpiCfg<FAM, BN>::BARS) * 8 + 4 <= BAR_BYTES, "barriers");
};

struct Epi {
  int mode;
  const float* bias;
  const __nv_bfloat16* aux;
  int64_t ld_aux;
  float alpha;
  __nv_bfloat16* aux_out;
  int64_t ld_aux_out;
  void* D;
  int64_t ldd;
  const int32_t* pos;
  const int32_t* pos2;     // GLM block positions (second rotary half) or null
  const float2* rope_tab;  // [pos][rotary_dim/2]
  int rope_cols;           // 2*H: columns that hold q and k
  int head_dim, rotary_dim;
  int aux_f32, d_f32;
  const float *ln_mean, *ln_rstd, *ln_gamma, *ln_beta;  // residual = LayerNorm(aux) when ln_mean
  float *adam_m, *adam_v;
  float lr, b1, b2, eps, wd, inv_bc1, inv_bc2;
  float den_scale;  // power of two that keeps the AdamW denominator in div_nr's range
  float* colsum;  // GELU_BWD: column sums of D added here (bias gradient of the up-projection)
  // launch of several problems: element offsets of problem r's pointers from problem 0's
  // (entry 0 unused, always 0): D, aux, aux_out, bias / colsum, the per-row arrays (pos,
  // pos2, LayerNorm statistics), LayerNorm gain / shift, Adam moments
  int64_t o_d[FL_GEMM_MAX_BATCH], o_aux[FL_GEMM_MAX_BATCH], o_aux_out[FL_GEMM_MAX_BATCH],
      o_bias[FL_GEMM_MAX_BATCH], o_row[FL_GEMM_MAX_BATCH], o_lnp[FL_GEMM_MAX_BATCH], o_adam[FL_GEMM_MAX_BATCH];
};

// The operands of the problems of one launch: A and B of problem r with their leading
// dimensions (tensor maps are built from these on the host).
struct Problems {
  int n;
  const void* A[FL_GEMM_MAX_BATCH];
  const void* B[FL_GEMM_MAX_BATCH];
  int64_t lda[FL_GEMM_MAX_BATCH], ldb[FL_GEMM_MAX_BATCH];
};

// Tensor maps of the A and B operands of up to FL_GEMM_MAX_BATCH problems, and with the AdamW
// epilogue of the weights, moments and bf16 copies (a kernel parameter: TMA reads each map
// from parameter space).
template <int FAM>
struct GemmMaps {
  CUtensorMap a[FL_GEMM_MAX_BATCH];
  CUtensorMap b[FL_GEMM_MAX_BATCH];
};
template <>
struct GemmMaps<FAM_F32> {
  CUtensorMap a[FL_GEMM_MAX_BATCH];
  CUtensorMap b[FL_GEMM_MAX_BATCH];
  CUtensorMap w[FL_GEMM_MAX_BATCH];
};
template <>
struct GemmMaps<FAM_ADAMW> {
  CUtensorMap a[FL_GEMM_MAX_BATCH];
  CUtensorMap b[FL_GEMM_MAX_BATCH];
  CUtensorMap w[FL_GEMM_MAX_BATCH], m[FL_GEMM_MAX_BATCH], v[FL_GEMM_MAX_BATCH], h[FL_GEMM_MAX_BATCH];
};

FL_DEV float4 ld_quad(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
FL_DEV float4 ld_quad(const __nv_bfloat16* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  const float2 a = unpack_bf16x2(u.x), b = unpack_bf16x2(u.y);
  return make_float4(a.x, a.y, b.x, b.y);
}
FL_DEV void st_quad(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
FL_DEV void st_quad(__nv_bfloat16* p, float4 v) {
  *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
}

// AdamW of one weight with gradient g (the formula of adamw_kernel).
FL_DEV void adamw_update(const Epi& e, float g, float& w, float& m, float& v) {
  m = e.b1 * m + (1.f - e.b1) * g;
  v = e.b2 * v + (1.f - e.b2) * g * g;
  const float d = (sqrt_nr(v * e.inv_bc2) + e.eps) * e.den_scale;
  w = w - e.lr * (div_nr(m * e.inv_bc1, d) * e.den_scale + e.wd * w);
}

// Entry r of a per-problem offset array (constant indices only: no local copy of the
// parameter struct).
FL_DEV int64_t prob_off(const int64_t (&o)[FL_GEMM_MAX_BATCH], int r) {
  static_assert(FL_GEMM_MAX_BATCH == 4, "prob_off selects among four problems");
  return r == 0 ? 0 : r == 1 ? o[1] : r == 2 ? o[2] : o[3];
}

// Where a tile lies for one epilogue warp: its problem r, the warp's first row and valid rows,
// the tile's first column, and the problem's element offsets into the epilogue operands.
struct TilePos {
  int r, row0, rows, n0;
  int64_t od, oaux, oauxo, oad;
};
template <int FAM>
FL_DEV void tile_offsets(TilePos& t, const Epi& e) {
  t.od = prob_off(e.o_d, t.r);
  if (FAM == FAM_RESID || FAM == FAM_GELU) t.oaux = prob_off(e.o_aux, t.r);
  if (FAM == FAM_GELU || FAM == FAM_ADAMW_LONG) t.oauxo = prob_off(e.o_aux_out, t.r);
  if (FAM == FAM_ADAMW_LONG) t.oad = prob_off(e.o_adam, t.r);
}

// Batches of an epilogue family: RB row pairs each, DEPTH register sets (DEPTH - 1 batches
// are requested ahead of the one at work).  The sizes keep the loop nearly free of spills (a
// spilled value would be read back through an L1 that the epilogue's own streams evict).
template <int FAM>
struct EpiBatch {
  static constexpr int RB = FAM == FAM_RESID || FAM == FAM_PLAIN ? 2 : 4;
  static constexpr int DEPTH = FAM == FAM_ADAMW_LONG ? 2 : 4;
};
// The epilogue operands of one batch: residual, accumulator or weight, the Adam moments, the
// pre-activation, the rows' LayerNorm statistics or positions.
template <int FAM, int RB>
struct EpiRegs {
  float4 a[FAM == FAM_ROPE || FAM == FAM_GELU ? 1 : RB];
  float4 m[FAM == FAM_ADAMW_LONG ? RB : 1], v[FAM == FAM_ADAMW_LONG ? RB : 1];
  uint2 h[FAM == FAM_GELU ? RB : 1];
  float mu[FAM == FAM_RESID ? RB : 1], rs[FAM == FAM_RESID ? RB : 1];
  int pos[FAM == FAM_ROPE ? RB : 1];
};
// Per-column operands of a chunk.
struct EpiCols {
  float4 bias, g, b;
};

template <int FAM>
FL_DEV void epi_cols(EpiCols& c, const Epi& e, const TilePos& t, int n) {
  c.bias = e.bias ? ld_quad(e.bias + prob_off(e.o_bias, t.r) + n) : make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (FAM == FAM_RESID) {
    if (e.ln_mean) {
      c.g = ld_quad(e.ln_gamma + prob_off(e.o_lnp, t.r) + n);
      c.b = ld_quad(e.ln_beta + prob_off(e.o_lnp, t.r) + n);
    }
  }
}

// Rotary placement of this lane's four columns of the chunk at column n0.  Dims
// [0, rotary_dim) of a head turn by pos; with GLM block positions, dims [rotary_dim,
// 2 rotary_dim) turn by pos2 (same frequencies and pairing).  Each rotary region is 32 or 64
// columns aligned inside the 64-column chunk, so a column's partner is half / 4 lanes away.
struct RopePos {
  bool rope, rotated, first;
  int rcol, half;
  const int32_t* src;
};
FL_DEV RopePos rope_pos(const Epi& e, int n0, int cl) {
  RopePos p;
  const int hoff = n0 % e.head_dim;
  p.rope = n0 < e.rope_cols && (hoff == 0 || e.pos2 != nullptr);
  p.half = e.rotary_dim >> 1;
  const int region = (hoff + 4 * cl) / e.rotary_dim;  // 0: rotated by pos, 1: by pos2
  p.rcol = hoff + 4 * cl - region * e.rotary_dim;
  p.rotated = p.rope && (region == 0 || (region == 1 && e.pos2 != nullptr));
  p.src = region == 0 ? e.pos : e.pos2;
  p.first = p.rcol < p.half;
  return p;
}

// Requests the operands of row pairs pb .. pb + RB - 1 of a chunk (this lane: column n, row
// parity h).  Rows past the matrix read its last row, so that a batch is straight-line code;
// epi_apply stores nothing for them.
template <int FAM, int RB>
FL_DEV void epi_load(EpiRegs<FAM, RB>& q, const Epi& e, const TilePos& t, int n, int pb, int h) {
  const int r0 = 2 * pb + h;
  if constexpr (FAM == FAM_ROPE) {
    const RopePos p = rope_pos(e, n & ~63, (n & 63) >> 2);
    if (!p.rotated) return;
    const int32_t* src = p.src + prob_off(e.o_row, t.r) + t.row0;
#pragma unroll
    for (int i = 0; i < RB; ++i) q.pos[i] = __ldg(src + min(r0 + 2 * i, t.rows - 1));
  } else if constexpr (FAM == FAM_GELU) {
    if (e.mode != FL_EPI_GELU_BWD) return;
    const __nv_bfloat16* src = e.aux + t.oaux + n;
#pragma unroll
    for (int i = 0; i < RB; ++i)
      q.h[i] = __ldg(reinterpret_cast<const uint2*>(src + (int64_t)(t.row0 + min(r0 + 2 * i, t.rows - 1)) * e.ld_aux));
  } else if constexpr (FAM == FAM_RESID) {
    const int64_t orow = prob_off(e.o_row, t.r);
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int m = t.row0 + min(r0 + 2 * i, t.rows - 1);
      const int64_t o = t.oaux + (int64_t)m * e.ld_aux + n;
      q.a[i] = e.aux_f32 ? ld_quad(reinterpret_cast<const float*>(e.aux) + o) : ld_quad(e.aux + o);
      if (e.ln_mean) {
        q.mu[i] = __ldg(e.ln_mean + orow + m);
        q.rs[i] = __ldg(e.ln_rstd + orow + m);
      }
    }
  } else {
    if (FAM == FAM_PLAIN && e.mode != FL_EPI_ACCUM_F32) return;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int64_t o = (int64_t)(t.row0 + min(r0 + 2 * i, t.rows - 1)) * e.ldd + n;
      q.a[i] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(e.D) + t.od + o);
      if constexpr (FAM == FAM_ADAMW_LONG) {
        q.m[i] = *reinterpret_cast<const float4*>(e.adam_m + t.oad + o);
        q.v[i] = *reinterpret_cast<const float4*>(e.adam_v + t.oad + o);
      }
    }
  }
}

// Arithmetic and stores of row pairs pb .. pb + RB - 1 of a 32-row x 64-column chunk held in
// `stage` (row r, float4 slot j stored at slot j ^ (r & 15)).  Half-warp h = lane / 16 takes
// the rows of parity h; lane l handles columns n0 + 4 (l % 16) .. + 3, so every warp-wide
// access covers two 64-column rows (256 B of bf16 or 512 B of fp32).  cs: this lane's column
// sums over its rows of the chunk (GELU_BWD).
template <int FAM, int RB>
FL_DEV void epi_apply(const EpiRegs<FAM, RB>& q, const EpiCols& c, const Epi& e, const TilePos& t, const float* stage,
                      int n, int pb, int h, float (&cs)[4]) {
  const int cl = (n & 63) >> 2;
  const bool gelu_bwd = FAM == FAM_GELU && e.mode == FL_EPI_GELU_BWD;
  const bool accum = FAM == FAM_PLAIN && e.mode == FL_EPI_ACCUM_F32;
  const bool out_f32 = e.mode == FL_EPI_STORE_F32 || e.d_f32;
  RopePos p;
  if constexpr (FAM == FAM_ROPE) p = rope_pos(e, n & ~63, cl);
  int64_t off = (int64_t)(t.row0 + 2 * pb + h) * e.ldd + n;
  int64_t offo = FAM == FAM_GELU || FAM == FAM_ADAMW_LONG ? t.oauxo + (int64_t)(t.row0 + 2 * pb + h) * e.ld_aux_out + n : 0;
#pragma unroll
  for (int i = 0; i < RB; ++i, off += 2 * e.ldd, offo += 2 * e.ld_aux_out) {
    const int rr = 2 * (pb + i) + h;
    const float4 acc = *reinterpret_cast<const float4*>(stage + rr * 64 + 4 * (cl ^ (rr & 15)));
    float y[4] = {acc.x + c.bias.x, acc.y + c.bias.y, acc.z + c.bias.z, acc.w + c.bias.w};
    if constexpr (FAM == FAM_ROPE) {
      if (p.rope) {  // uniform across the warp: every lane takes part in the shuffles
        float z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = __shfl_xor_sync(0xffffffffu, y[k], p.half >> 2);
        if (p.rotated) {
          const float2* tab = e.rope_tab + (int64_t)q.pos[i] * p.half + (p.first ? p.rcol : p.rcol - p.half);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 w = __ldg(tab + k);
            y[k] = p.first ? y[k] * w.x - z[k] * w.y : y[k] * w.x + z[k] * w.y;
          }
        }
      }
    }
    const bool ok = rr < t.rows;
    if constexpr (FAM == FAM_RESID) {
      const float a4[4] = {q.a[i].x, q.a[i].y, q.a[i].z, q.a[i].w};
      const float g4[4] = {c.g.x, c.g.y, c.g.z, c.g.w}, b4[4] = {c.b.x, c.b.y, c.b.z, c.b.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float r = e.ln_mean ? (a4[k] - q.mu[i]) * q.rs[i] * g4[k] + b4[k] : a4[k];  // LayerNorm(aux) in fp32
        y[k] = fmaf(e.alpha, r, y[k]);
      }
    } else if constexpr (FAM == FAM_GELU) {
      if (gelu_bwd) {
        const float2 u0 = unpack_bf16x2(q.h[i].x), u1 = unpack_bf16x2(q.h[i].y);
        const float u[4] = {u0.x, u0.y, u1.x, u1.y};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          y[k] *= gelu_tanh_grad(u[k]);
          cs[k] += ok ? y[k] : 0.f;
        }
      } else {
        if (ok) st_quad(e.aux_out + offo, make_float4(y[0], y[1], y[2], y[3]));
#pragma unroll
        for (int k = 0; k < 4; ++k) y[k] = gelu_tanh(y[k]);
      }
    }
    if constexpr (FAM == FAM_ADAMW_LONG) {
      float w[4] = {q.a[i].x, q.a[i].y, q.a[i].z, q.a[i].w};
      float mm[4] = {q.m[i].x, q.m[i].y, q.m[i].z, q.m[i].w};
      float vv[4] = {q.v[i].x, q.v[i].y, q.v[i].z, q.v[i].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) adamw_update(e, y[k], w[k], mm[k], vv[k]);
      if (!ok) continue;
      st_quad(reinterpret_cast<float*>(e.D) + t.od + off, make_float4(w[0], w[1], w[2], w[3]));
      st_quad(e.adam_m + t.oad + off, make_float4(mm[0], mm[1], mm[2], mm[3]));
      st_quad(e.adam_v + t.oad + off, make_float4(vv[0], vv[1], vv[2], vv[3]));
      st_quad(e.aux_out + offo, make_float4(w[0], w[1], w[2], w[3]));
      continue;
    }
    if (accum) {
      y[0] += q.a[i].x;
      y[1] += q.a[i].y;
      y[2] += q.a[i].z;
      y[3] += q.a[i].w;
    }
    if (!ok) continue;
    if (accum || out_f32) st_quad(reinterpret_cast<float*>(e.D) + t.od + off, make_float4(y[0], y[1], y[2], y[3]));
    else st_quad(reinterpret_cast<__nv_bfloat16*>(e.D) + t.od + off, make_float4(y[0], y[1], y[2], y[3]));
  }
}

// The epilogue of one warp over its CTA's (or CTA pair's) tiles t0, t0 + step, ...: WCH
// 64-column chunks per tile, each in batches of RB row pairs.  Short contractions are bound by
// it: two 4096 x 16384 fp32 outputs at 77 tokens take 108 us stored (155 with four warps, each
// batch's operands read when it is reached and a cluster-scope release per tile), 232 us
// accumulated (335).  `place` gives a tile's
// position for this warp, `release` frees accumulator `acc` once the warp has read it.
template <int FAM, int BN, typename Place, typename Release>
FL_DEV void epilogue_loop(const Epi& e, float* stage, uint32_t tmem_base, int warp, int lane, int t0, int step,
                          int num_tiles, uint64_t* acc_full, uint64_t* cs_bars, int* status, Place place, Release release) {
  constexpr int RB = EpiBatch<FAM>::RB, DEPTH = EpiBatch<FAM>::DEPTH;
  constexpr int HALVES = EpiCfg<FAM, BN>::WARPS / 4;    // warps per lane quarter
  constexpr int WCH = BN / (64 * HALVES);           // chunks per warp and tile
  constexpr int NBC = 16 / RB;                      // batches per chunk
  static_assert(NBC % DEPTH == 0, "whole rounds of register sets per chunk");
  const int c_first = ((warp - 2) >> 2) * (BN / HALVES);  // first column of the warp's chunks
  const int h = lane >> 4, cl4 = 4 * (lane & 15);
  const uint32_t t_row = tmem_base + (uint32_t((warp & 3) * 32) << 16) + c_first;
  float4* my = reinterpret_cast<float4*>(stage + lane * 64);
  if (t0 >= num_tiles) return;
  TilePos t;
  place(t0, t);
  tile_offsets<FAM>(t, e);
  EpiRegs<FAM, RB> q[DEPTH];
  EpiCols c, cn;
  int n = t.n0 + c_first + cl4;
  epi_cols<FAM>(c, e, t, n);
#pragma unroll
  for (int s = 0; s < DEPTH - 1; ++s) epi_load<FAM, RB>(q[s], e, t, n, s * RB, h);
  int local = 0;
  uint32_t cs_par = 0;  // parity of the column sums' barriers
  for (int tile = t0; tile < num_tiles; tile += step, ++local) {
    const int acc = local & 1;
    if (!mbar_wait_warp(&acc_full[acc], (local >> 1) & 1)) {
      if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_FULL);
      return;
    }
    tc_fence_after();
    TilePos tn = t;
    const bool more = tile + step < num_tiles;
    if (more) {
      place(tile + step, tn);
      tile_offsets<FAM>(tn, e);
    }
#pragma unroll 1
    for (int ch = 0; ch < WCH; ++ch) {
      // this lane's row -> shared memory, float4 slot j at j ^ (row & 15), 32 columns at a
      // time (the prefetched operands need the registers)
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        uint32_t x[32];
        tmem_ld32(t_row + acc * BN + 64 * ch + 32 * s, x);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          my[(8 * s + j) ^ (lane & 15)] = make_float4(__uint_as_float(x[4 * j]), __uint_as_float(x[4 * j + 1]),
                                                      __uint_as_float(x[4 * j + 2]), __uint_as_float(x[4 * j + 3]));
      }
      const bool last = ch == WCH - 1;
      if (last) {  // the warp's accumulator part is read: the MMA may reuse it
        tc_fence_before();
        __syncwarp();
        release(acc);
      }
      __syncwarp();
      // the chunk after this one, of this tile or the next
      const int nx = last ? tn.n0 + c_first + cl4 : n + 64;
      const bool next = !last || more;
      float cs[4] = {0.f, 0.f, 0.f, 0.f};
      if (next) epi_cols<FAM>(cn, e, last ? tn : t, nx);
#pragma unroll 1
      for (int b0 = 0; b0 < NBC; b0 += DEPTH) {
#pragma unroll
        for (int s = 0; s < DEPTH; ++s) {
          const int j = b0 + s + DEPTH - 1;  // the batch requested now
          EpiRegs<FAM, RB>& qn = q[(s + DEPTH - 1) % DEPTH];
          if (j < NBC) epi_load<FAM, RB>(qn, e, t, n, j * RB, h);
          else if (next) epi_load<FAM, RB>(qn, e, last ? tn : t, nx, (j - NBC) * RB, h);
          epi_apply<FAM, RB>(q[s], c, e, t, stage, n, (b0 + s) * RB, h, cs);
        }
      }
      if (FAM == FAM_GELU && e.colsum != nullptr) {
        // the two half-warps hold the same columns for rows of either parity; the four warps of the
        // column half meet in their staging and one adds their sum, so that calls of up to two row
        // blocks sum a bias gradient in one order
#pragma unroll
        for (int k = 0; k < 4; ++k) cs[k] += __shfl_xor_sync(0xffffffffu, cs[k], 16);
        __syncwarp();
        if (h == 0) *reinterpret_cast<float4*>(stage + cl4) = make_float4(cs[0], cs[1], cs[2], cs[3]);
        __syncwarp();
        const int wi = (warp - 2) & 3;
        uint64_t* written = cs_bars + 2 * ((warp - 2) >> 2);
        if (lane == 0) mbar_arrive(written);
        if (wi == 0) {
          if (!mbar_wait_warp(written, cs_par)) {
            if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_FULL);
            return;
          }
          if (h == 0) {
            float4 t4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 q4 = *reinterpret_cast<const float4*>(stage + i * 32 * 64 + cl4);
              t4 = make_float4(t4.x + q4.x, t4.y + q4.y, t4.z + q4.z, t4.w + q4.w);
            }
            red_add_v4(e.colsum + prob_off(e.o_bias, t.r) + n, t4.x, t4.y, t4.z, t4.w);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(written + 1);
        } else if (!mbar_wait_warp(written + 1, cs_par)) {
          if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_FULL);
          return;
        }
        cs_par ^= 1;
      }
      __syncwarp();  // the chunk has been read
      c = cn;
      n = nx;
    }
    t = tn;
  }
}

template <int BN, typename Maps, typename Place, typename Release>
FL_DEV void adamw_epilogue(const Epi& e, const Maps& maps, uint8_t* ring, uint64_t* ring_full, uint32_t tmem_base,
                           int warp, int lane, int t0, int step, int num_tiles, uint64_t* acc_full, int* status,
                           Place place, Release release) {
  using R = AdamRing;
  constexpr int CC = R::CC, S = R::SLOTS, CPT = BN / CC;
  uint8_t* slots = ring + (warp - 2) * S * R::SLOT;
  uint64_t* full = ring_full + (warp - 2) * S;
  const int total = t0 < num_tiles ? ((num_tiles - t0 + step - 1) / step) * CPT : 0;
  const uint32_t t_row = tmem_base + (uint32_t((warp & 3) * 32) << 16);
  TilePos tl, t;  // the tile being loaded (lane 0), the tile at work
  auto issue = [&](int k) {
    if (k % CPT == 0) place(t0 + (k / CPT) * step, tl);
    const int s = k % S, x = tl.n0 + (k % CPT) * CC;
    uint8_t* p = slots + s * R::SLOT;
    mbar_arrive_expect_tx(full + s, 3 * R::TENSOR);
    tma_load_2d(p, &maps.w[tl.r], full + s, x, tl.row0);
    tma_load_2d(p + R::TENSOR, &maps.m[tl.r], full + s, x, tl.row0);
    tma_load_2d(p + 2 * R::TENSOR, &maps.v[tl.r], full + s, x, tl.row0);
  };
  int issued = 0;
  if (lane == 0)
    for (; issued < S - 1 && issued < total; ++issued) issue(issued);
  int k = 0;
  for (; k < total; ++k) {
    const int c = k % CPT, local = k / CPT, acc = local & 1, s = k % S;
    if (c == 0) {
      place(t0 + local * step, t);
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (local >> 1) & 1))) {
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_FULL);
        break;
      }
      tc_fence_after();
    }
    if (!__all_sync(0xffffffffu, mbar_wait(full + s, (k / S) & 1))) {
      if (lane == 0) report_status(status, FL_DEV_TIMEOUT_FULL);
      break;
    }
    uint32_t g[CC];
    tmem_ld16(t_row + acc * BN + c * CC, g);
    tmem_ld_wait();
    if (c == CPT - 1) {  // the warp's accumulator part is read: the MMA may reuse it
      tc_fence_before();
      __syncwarp();
      release(acc);
    }
    uint8_t* p = slots + s * R::SLOT;
    uint32_t hb[CC / 2];
#pragma unroll
    for (int j = 0; j < CC / 4; ++j) {
      // 16-byte piece j of the lane's row: 64-byte swizzle
      float4* q = reinterpret_cast<float4*>(p + lane * (CC * 4) + ((j ^ ((lane >> 1) & 3)) << 4));
      constexpr int T4 = R::TENSOR / 16;
      const float4 w4 = q[0], m4 = q[T4], v4 = q[2 * T4];
      float w[4] = {w4.x, w4.y, w4.z, w4.w}, mm[4] = {m4.x, m4.y, m4.z, m4.w}, vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) adamw_update(e, __uint_as_float(g[4 * j + i]), w[i], mm[i], vv[i]);
      q[0] = make_float4(w[0], w[1], w[2], w[3]);
      q[T4] = make_float4(mm[0], mm[1], mm[2], mm[3]);
      q[2 * T4] = make_float4(vv[0], vv[1], vv[2], vv[3]);
      hb[2 * j] = pack_bf16x2(w[0], w[1]);
      hb[2 * j + 1] = pack_bf16x2(w[2], w[3]);
    }
#pragma unroll
    for (int j = 0; j < CC / 8; ++j)  // 32-byte swizzle
      *reinterpret_cast<uint4*>(p + 3 * R::TENSOR + lane * (CC * 2) + ((j ^ ((lane >> 2) & 1)) << 4)) =
          make_uint4(hb[4 * j], hb[4 * j + 1], hb[4 * j + 2], hb[4 * j + 3]);
    fence_proxy_async_smem();  // the lane's updates, visible to the bulk stores
    __syncwarp();
    if (lane == 0) {
      bulk_wait_read();  // chunk k - 1's stores have read their slot: chunk k + S - 1 loads into it
      if (issued < total) issue(issued++);
      if (t.rows > 0) {
        const int x = t.n0 + c * CC;
        tma_store_2d(&maps.w[t.r], p, x, t.row0);
        tma_store_2d(&maps.m[t.r], p + R::TENSOR, x, t.row0);
        tma_store_2d(&maps.v[t.r], p + 2 * R::TENSOR, x, t.row0);
        tma_store_2d(&maps.h[t.r], p + 3 * R::TENSOR, x, t.row0);
        bulk_commit();
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    for (; k < issued; ++k) mbar_wait(full + k % S, (k / S) & 1);  // after a wait gave up: its copies land first
    bulk_wait_all();  // the stores are complete before the CTA leaves
  }
}

// D = acc or D += acc in fp32, see adamw_epilogue: bound by HBM while the contraction is short.  Two
// 4096 x 16384 gradients at 77 tokens: added 191 us, 5.6 TB/s (230 from registers on eight warps
// of the same tile), stored 97 us, 5.5 TB/s (102).  64 KB of ring leave five operand stages.
template <int BN, typename Maps, typename Place, typename Release>
FL_DEV void f32_epilogue(const Epi& e, const Maps& maps, uint8_t* ring, uint64_t* ring_full, uint32_t tmem_base,
                         int warp, int lane, int t0, int step, int num_tiles, uint64_t* acc_full, int* status,
                         Place place, Release release) {
  using R = F32Ring;
  constexpr int CC = R::CC, S = R::SLOTS, CPT = BN / CC;
  uint8_t* slots = ring + (warp - 2) * S * R::SLOT;
  uint64_t* full = ring_full + (warp - 2) * S;
  const bool add = e.mode == FL_EPI_ACCUM_F32;
  const int total = t0 < num_tiles ? ((num_tiles - t0 + step - 1) / step) * CPT : 0;
  const uint32_t t_row = tmem_base + (uint32_t((warp & 3) * 32) << 16);
  TilePos tl, t;  // the tile being loaded (lane 0), the tile at work
  auto issue = [&](int k) {
    if (k % CPT == 0) place(t0 + (k / CPT) * step, tl);
    const int s = k % S;
    mbar_arrive_expect_tx(full + s, R::SLOT);
    tma_load_2d(slots + s * R::SLOT, &maps.w[tl.r], full + s, tl.n0 + (k % CPT) * CC, tl.row0);
  };
  int issued = 0;
  if (lane == 0 && add)
    for (; issued < S - 1 && issued < total; ++issued) issue(issued);
  int k = 0;
  for (; k < total; ++k) {
    const int c = k % CPT, local = k / CPT, acc = local & 1, s = k % S;
    if (c == 0) {
      place(t0 + local * step, t);
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[acc], (local >> 1) & 1))) {
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_FULL);
        break;
      }
      tc_fence_after();
    }
    if (add) {
      if (!__all_sync(0xffffffffu, mbar_wait(full + s, (k / S) & 1))) {
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_FULL);
        break;
      }
    } else {  // the slot's last store has read it
      if (lane == 0) bulk_wait_read<S - 1>();
      __syncwarp();
    }
    uint32_t g[CC];
    tmem_ld32(t_row + acc * BN + c * CC, g);
    tmem_ld_wait();
    if (c == CPT - 1) {  // the warp's accumulator part is read: the MMA may reuse it
      tc_fence_before();
      __syncwarp();
      release(acc);
    }
    uint8_t* p = slots + s * R::SLOT;
#pragma unroll
    for (int j = 0; j < CC / 4; ++j) {
      float4* q = reinterpret_cast<float4*>(p + lane * (CC * 4) + ((j ^ (lane & 7)) << 4));
      float4 y = make_float4(__uint_as_float(g[4 * j]), __uint_as_float(g[4 * j + 1]), __uint_as_float(g[4 * j + 2]),
                             __uint_as_float(g[4 * j + 3]));
      if (add) {
        const float4 d = *q;
        y = make_float4(d.x + y.x, d.y + y.y, d.z + y.z, d.w + y.w);
      }
      *q = y;
    }
    fence_proxy_async_smem();  // the lane's values, visible to the bulk store
    __syncwarp();
    if (lane == 0) {
      if (add) {
        bulk_wait_read();  // chunk k - 1's store has read its slot: chunk k + S - 1 loads into it
        if (issued < total) issue(issued++);
      }
      if (t.rows > 0) tma_store_2d(&maps.w[t.r], p, t.n0 + c * CC, t.row0);
      bulk_commit();  // (a group per chunk, empty or not)
    }
    __syncwarp();
  }
  if (lane == 0) {
    for (; k < issued; ++k) mbar_wait(full + k % S, (k / S) & 1);  // after a wait gave up: its copies land first
    bulk_wait_all();  // the stores are complete before the CTA leaves
  }
}

// Tile order.  Tiles are taken in groups of `gsz` panels of one operand: along m
// (gsz m-blocks, m fastest) every group streams B once while its A panels stay in L2;
// along n the roles swap.  The host picks the side and size that minimise DRAM reads.
struct Raster {
  int gsz;
  int along_n;
};
// Problem r of a batched launch and the tile's coordinates inside it: the problems' tile
// ranges follow each other, each in its own raster order.
FL_DEV void batch_tile(int tile, int num_m, int num_n, Raster rs, int& r, int& mb, int& nb);

FL_DEV void tile_coords(int tile, int num_m, int num_n, Raster r, int& mb, int& nb) {
  if (!r.along_n) {
    const int group = r.gsz * num_n;
    const int g = tile / group;
    const int first = g * r.gsz;
    const int gm = min(num_m - first, r.gsz);
    const int local = tile - g * group;
    mb = first + local % gm;
    nb = local / gm;
  } else {
    const int group = r.gsz * num_m;
    const int g = tile / group;
    const int first = g * r.gsz;
    const int gn = min(num_n - first, r.gsz);
    const int local = tile - g * group;
    nb = first + local % gn;
    mb = local / gn;
  }
}

FL_DEV void batch_tile(int tile, int num_m, int num_n, Raster rs, int& r, int& mb, int& nb) {
  const int per = num_m * num_n;
  r = tile / per;
  tile_coords(tile - r * per, num_m, num_n, rs, mb, nb);
}

// Shared-memory descriptor of an operand stage, and its step from one 16-deep MMA to the next:
// K-major, the next 16 elements are 32 bytes further along the swizzled row; MN-major, the next
// 16 k-rows 16 * 128 bytes further (the descriptor counts 16-byte units).
template <bool MN>
FL_DEV uint64_t stage_desc(uint32_t base) {
  return MN ? smem_desc_sw128(base, BK * 128, 1024) : smem_desc_sw128(base, 16, 1024);
}
template <bool MN>
__host__ __device__ constexpr uint64_t kstep_desc() {
  return MN ? 128 : 2;
}

template <int BN, bool A_MN, bool B_MN, int FAM>
__global__ void __launch_bounds__(EpiCfg<FAM, BN>::THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ GemmMaps<FAM> maps, Epi epi, int M, int N, int K, int batch, Raster raster,
                   int* status) {
  using C = Cfg<BN, FAM>;
  constexpr int STAGES = C::STAGES, KSUB = C::KSUB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * KSUB * C::A_BYTES;
  uint8_t* epi_smem = smem + STAGES * C::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi_smem + EpiCfg<FAM, BN>::BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + STAGES;
  uint64_t* acc_full = bars + 2 * STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain = acc_empty + 2;
  uint64_t* epi_bars = drain + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(epi_bars + EpiCfg<FAM, BN>::BARS);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int num_m = (M + BM - 1) / BM;
  const int num_n = N / BN;
  const int num_tiles = batch * num_m * num_n;
  const int num_k = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], EpiCfg<FAM, BN>::WARPS);
    }
    mbar_init(drain, 1);
    for (int i = 0; i < EpiCfg<FAM, BN>::BARS; ++i) mbar_init(&epi_bars[i], EpiCfg<FAM, BN>::bar_count(i));
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    for (int r = 0; r < batch; ++r) {
      tma_prefetch_desc(&maps.a[r]);
      tma_prefetch_desc(&maps.b[r]);
    }
  }
  if (warp == 1) {
    tmem_alloc(tmem_holder, C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  pdl_wait();  // the previous kernel's outputs (operands, epilogue inputs) are complete
  pdl_trigger();

  // The producer and MMA loops are run by whole (converged) warps, one elected lane issuing: the
  // loop state stays in uniform registers, which the TMA and MMA instructions take directly.
  // With the loops inside one lane's branch a k-block cost at least 270 ns whatever the tile
  // (4096 columns, K = 16384, 77 rows on 256 x 128 pairs: 79 us; 63 us this way), and the full
  // 256 x 256 tiles at 2048 rows ran 5-8% slower (QKV projection 131 -> 123 us).
  if (warp == 0) {
    // -------------------------------------------------------------- TMA producer
    int stage = 0, used = 0;  // used: stages armed so far (up to STAGES), for the teardown drain
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int r, mb, nb;
      batch_tile(tile, num_m, num_n, raster, r, mb, nb);
      const CUtensorMap* tmA = &maps.a[r];
      const CUtensorMap* tmB = &maps.b[r];
      for (int kb = 0; kb < num_k; kb += KSUB) {
        if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
          if (lane == 0) report_status(status, FL_DEV_TIMEOUT_EMPTY);
          ok = false;
          break;
        }
        if (elect_one()) {
          mbar_arrive_expect_tx(&full[stage], C::STAGE_BYTES);
#pragma unroll
          for (int q = 0; q < KSUB; ++q) {  // a k-block past K reads zeros
            const int k0 = (kb + q) * BK;
            uint8_t* a_dst = sA + (stage * KSUB + q) * C::A_BYTES;
            uint8_t* b_dst = sB + (stage * KSUB + q) * C::B_BYTES;
            if (!A_MN) {
              tma_load_2d(a_dst, tmA, &full[stage], k0, mb * BM);
            } else {
#pragma unroll
              for (int j = 0; j < BM / 64; ++j) tma_load_2d(a_dst + j * 64 * BK * 2, tmA, &full[stage], mb * BM + 64 * j, k0);
            }
            if (!B_MN) {
              tma_load_2d(b_dst, tmB, &full[stage], k0, nb * BN);
            } else {
#pragma unroll
              for (int j = 0; j < BN / 64; ++j) tma_load_2d(b_dst + j * 64 * BK * 2, tmB, &full[stage], nb * BN + 64 * j, k0);
            }
          }
        }
        __syncwarp();
        if (used < STAGES) ++used;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    // Drain: every armed stage's copies must have landed before shared memory is released.
    // Stage s was last armed in the phase before the current one, or in it where s < stage.
    for (int s = 0; s < used; ++s)
      if (!mbar_wait_warp(&full[s], s < stage ? phase : phase ^ 1))
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_DRAIN);
  } else if (warp == 1) {
    // -------------------------------------------------------------- MMA issuer
    constexpr uint32_t IDESC = umma_idesc_bf16(BM, BN, A_MN, B_MN);
    int stage = 0;
    uint32_t phase = 0;
    int local = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++local) {
      const int acc = local & 1;
      const uint32_t acc_par = (local >> 1) & 1;
      if (!mbar_wait_warp(&acc_empty[acc], acc_par ^ 1)) {
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_EMPTY);
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * BN;
      for (int kb = 0; kb < num_k; kb += KSUB) {
        if (!mbar_wait_warp(&full[stage], phase)) {
          if (lane == 0) report_status(status, FL_DEV_TIMEOUT_FULL);
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int q = 0; q < KSUB; ++q) {
            if (KSUB > 1 && kb + q >= num_k) break;
            const uint64_t ad = stage_desc<A_MN>(smem_u32(sA + (stage * KSUB + q) * C::A_BYTES));
            const uint64_t bd = stage_desc<B_MN>(smem_u32(sB + (stage * KSUB + q) * C::B_BYTES));
#pragma unroll
            for (int kk = 0; kk < BK / UMMA_K; ++kk)
              umma_bf16(d_tmem, ad + kk * kstep_desc<A_MN>(), bd + kk * kstep_desc<B_MN>(), IDESC,
                        (kb | q | kk) != 0 ? 1u : 0u);
          }
          umma_commit(&empty[stage]);
          if (kb + KSUB >= num_k) umma_commit(&acc_full[acc]);
        }
        __syncwarp();
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    // Drain: all MMAs issued by this warp complete before TMEM is released.
    if (elect_one()) umma_commit(drain);
    __syncwarp();
    if (!mbar_wait_warp(drain, 0) && lane == 0) report_status(status, FL_DEV_TIMEOUT_DRAIN);
  } else {
    // -------------------------------------------------------------- epilogue warps
    auto place = [&](int tile, TilePos& t) {
      int mb, nb;
      batch_tile(tile, num_m, num_n, raster, t.r, mb, nb);
      t.row0 = mb * BM + (warp & 3) * 32;
      t.rows = M - t.row0 < 32 ? M - t.row0 : 32;  // may be <= 0 for the ragged last tile
      t.n0 = nb * BN;
    };
    auto release = [&](int acc) {
      if (lane == 0) mbar_arrive(&acc_empty[acc]);
    };
    if constexpr (FAM == FAM_ADAMW)
      adamw_epilogue<BN>(epi, maps, epi_smem, epi_bars, tmem_base, warp, lane, blockIdx.x, gridDim.x, num_tiles, acc_full,
                         status, place, release);
    else if constexpr (FAM == FAM_F32)
      f32_epilogue<BN>(epi, maps, epi_smem, epi_bars, tmem_base, warp, lane, blockIdx.x, gridDim.x, num_tiles, acc_full,
                         status, place, release);
    else
      epilogue_loop<FAM, BN>(epi, reinterpret_cast<float*>(epi_smem) + (warp - 2) * 32 * 64, tmem_base, warp, lane,
                             blockIdx.x, gridDim.x, num_tiles, acc_full, epi_bars, status, place, release);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ------------------------------------------------------------------ CTA-pair kernel
// A cluster of two CTAs on two SMs computes one 256 x PBN tile (PBN 256 or 128) with
// tcgen05.mma.cta_group::2.  Each CTA stages its own 128 rows of A and PBN / 2 columns of B
// (32 KB per k-block at PBN 256, against 48 KB for a 128 x 256 tile on one SM); the even CTA
// issues 256 x PBN x 16 MMAs that read both CTAs' stages and write accumulator rows 0..127
// into its own TMEM and rows 128..255 into the odd CTA's; each CTA's epilogue warps drain
// their own half exactly as in gemm_tc_kernel.
// Barriers: both producers' loads complete on the even CTA's full[s]; the MMA commits
// arrive on empty[s] and acc_full[a] of both CTAs; every epilogue warp of the pair
// arrives once on the even CTA's acc_empty[a].
constexpr int PAIR_BM = 256;
template <int PBN, int FAM>
struct CfgPair {
  static constexpr int A_BYTES = 128 * BK * 2;        // this CTA's 128 rows of A
  static constexpr int B_BYTES = (PBN / 2) * BK * 2;  // this CTA's columns of B
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = ring_stages(STAGE_BYTES, EpiCfg<FAM, PBN>::BYTES);
  static constexpr int TMEM_COLS = 2 * PBN;  // double-buffered accumulator
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EpiCfg<FAM, PBN>::BYTES + BAR_BYTES + 1024 /*align*/;
  static_assert((2 * STAGES + 5 + EpiCfg<FAM, PBN>::BARS) * 8 + 4 <= BAR_BYTES, "barriers");
};

template <int PBN, bool A_MN, bool B_MN, int FAM>
__global__ void __launch_bounds__(EpiCfg<FAM, PBN>::THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ GemmMaps<FAM> maps, Epi epi, int M, int N, int K, int batch, Raster raster,
                     int* status) {
  using C = CfgPair<PBN, FAM>;
  constexpr int STAGES = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * C::A_BYTES;
  uint8_t* epi_smem = smem + STAGES * C::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi_smem + EpiCfg<FAM, PBN>::BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + STAGES;
  uint64_t* acc_full = bars + 2 * STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* drain = acc_empty + 2;
  uint64_t* epi_bars = drain + 1;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(epi_bars + EpiCfg<FAM, PBN>::BARS);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int num_m = (M + PAIR_BM - 1) / PAIR_BM;
  const int num_n = N / PBN;
  const int num_tiles = batch * num_m * num_n;
  const int num_k = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);   // the even CTA's producer (expect_tx of both CTAs' bytes)
      mbar_init(&empty[s], 1);  // one MMA commit
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 2 * EpiCfg<FAM, PBN>::WARPS);  // the epilogue warps of both CTAs
    }
    mbar_init(drain, 1);
    for (int i = 0; i < EpiCfg<FAM, PBN>::BARS; ++i) mbar_init(&epi_bars[i], EpiCfg<FAM, PBN>::bar_count(i));
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    for (int r = 0; r < batch; ++r) {
      tma_prefetch_desc(&maps.a[r]);
      tma_prefetch_desc(&maps.b[r]);
    }
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_holder, C::TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers initialised and TMEM allocated
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  pdl_wait();  // the previous kernel's outputs (operands, epilogue inputs) are complete
  pdl_trigger();

  if (warp == 0) {
    // -------------------------------------------------------------- TMA producer (both CTAs)
    const uint32_t full0 = mapa_shared(smem_u32(full), 0);  // the even CTA's full[0]
    int stage = 0, used = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += n_pairs) {
      int r, mb, nb;
      batch_tile(tile, num_m, num_n, raster, r, mb, nb);
      const CUtensorMap* tmA = &maps.a[r];
      const CUtensorMap* tmB = &maps.b[r];
      const int m0 = mb * PAIR_BM + int(rank) * 128, n0 = nb * PBN + int(rank) * (PBN / 2);
      for (int kb = 0; kb < num_k; ++kb) {
        if (!mbar_wait_warp(&empty[stage], phase ^ 1)) {
          if (lane == 0) report_status(status, FL_DEV_TIMEOUT_EMPTY);
          ok = false;
          break;
        }
        if (elect_one()) {
          if (leader) mbar_arrive_expect_tx(&full[stage], 2 * C::STAGE_BYTES);
          const uint32_t fb = full0 + 8u * stage;
          const int k0 = kb * BK;
          uint8_t* a_dst = sA + stage * C::A_BYTES;
          uint8_t* b_dst = sB + stage * C::B_BYTES;
          if (!A_MN) {
            tma_load_2d_pair(a_dst, tmA, fb, k0, m0);
          } else {
            tma_load_2d_pair(a_dst, tmA, fb, m0, k0);
            tma_load_2d_pair(a_dst + 64 * BK * 2, tmA, fb, m0 + 64, k0);
          }
          if (!B_MN) {
            tma_load_2d_pair(b_dst, tmB, fb, k0, n0);
          } else {
#pragma unroll
            for (int j = 0; j < PBN / 128; ++j) tma_load_2d_pair(b_dst + j * 64 * BK * 2, tmB, fb, n0 + 64 * j, k0);
          }
        }
        __syncwarp();
        if (used < STAGES) ++used;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    // Drain: a stage loaded in phase p is released (empty phase p completes) only after
    // the MMAs that read it, and so after its copies landed.
    for (int s = 0; s < used; ++s)
      if (!mbar_wait_warp(&empty[s], s < stage ? phase : phase ^ 1))
        if (lane == 0) report_status(status, FL_DEV_TIMEOUT_DRAIN);
  } else if (warp == 1) {
    if (leader) {
      // ------------------------------------------------------------ MMA issuer (even CTA)
      constexpr uint32_t IDESC = umma_idesc_bf16(PAIR_BM, PBN, A_MN, B_MN);
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += n_pairs, ++local) {
        const int acc = local & 1;
        const uint32_t acc_par = (local >> 1) & 1;
        if (!mbar_wait_warp(&acc_empty[acc], acc_par ^ 1)) {
          if (lane == 0) report_status(status, FL_DEV_TIMEOUT_ACC_EMPTY);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * PBN;
        for (int kb = 0; kb < num_k; ++kb) {
          if (!mbar_wait_warp(&full[stage], phase)) {
            if (lane == 0) report_status(status, FL_DEV_TIMEOUT_FULL);
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            const uint64_t ad = stage_desc<A_MN>(smem_u32(sA + stage * C::A_BYTES));
            const uint64_t bd = stage_desc<B_MN>(smem_u32(sB + stage * C::B_BYTES));
#pragma unroll
            for (int kk = 0; kk < BK / UMMA_K; ++kk)
              umma_bf16_pair(d_tmem, ad + kk * kstep_desc<A_MN>(), bd + kk * kstep_desc<B_MN>(), IDESC,
                             (kb | kk) != 0 ? 1u : 0u);
            umma_commit_pair(&empty[stage], 3);
            if (kb + 1 == num_k) umma_commit_pair(&acc_full[acc], 3);
          }
          __syncwarp();
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
      // Drain: all MMAs issued by this warp (and their arrivals) complete before the pair
      // releases TMEM and shared memory.
      if (elect_one()) umma_commit_pair(drain, 1);
      __syncwarp();
      if (!mbar_wait_warp(drain, 0) && lane == 0) report_status(status, FL_DEV_TIMEOUT_DRAIN);
    }
  } else {
    // -------------------------------------------------------------- epilogue warps (both CTAs)
    const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
    auto place = [&](int tile, TilePos& t) {
      int mb, nb;
      batch_tile(tile, num_m, num_n, raster, t.r, mb, nb);
      t.row0 = mb * PAIR_BM + int(rank) * 128 + (warp & 3) * 32;
      t.rows = M - t.row0 < 32 ? M - t.row0 : 32;  // may be <= 0 for the ragged last tile
      t.n0 = nb * PBN;
    };
    auto release = [&](int acc) {
      if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8u * acc);
    };
    if constexpr (FAM == FAM_ADAMW)
      adamw_epilogue<PBN>(epi, maps, epi_smem, epi_bars, tmem_base, warp, lane, pair, n_pairs, num_tiles, acc_full, status,
                          place, release);
    else if constexpr (FAM == FAM_F32)
      f32_epilogue<PBN>(epi, maps, epi_smem, epi_bars, tmem_base, warp, lane, pair, n_pairs, num_tiles, acc_full, status,
                          place, release);
    else
      epilogue_loop<FAM, PBN>(epi, reinterpret_cast<float*>(epi_smem) + (warp - 2) * 32 * 64, tmem_base, warp, lane, pair,
                              n_pairs, num_tiles, acc_full, epi_bars, status, place, release);
  }

  tc_fence_before();
  cluster_sync();  // neither CTA leaves while the pair's MMAs or arrivals may still touch it
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
  }
}

// ------------------------------------------------------------------ host side

typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline PFN_encodeTiled get_encode_fn() {
  static PFN_encodeTiled fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_encodeTiled>(p);
  });
  return fn;
}

// 2-D bf16 tensor [outer, inner] (inner contiguous, row stride ld elements), box {64, box_outer}.
inline int make_map(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, int64_t ld, uint32_t box_outer) {
  PFN_encodeTiled enc = get_encode_fn();
  if (!enc) return fl_internal_error(FL_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {cuuint64_t(ld) * 2};
  cuuint32_t box[2] = {64, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fl_internal_error(FL_ERR_INVALID_ARG, "tensor map encode failed (%d): inner %llu outer %llu ld %lld", (int)r,
                             (unsigned long long)inner, (unsigned long long)outer, (long long)ld);
  return FL_OK;
}

// 2-D tensor of a ring epilogue: fp32 or bf16 [rows, cols], boxes of cc columns x 32 rows, swizzled
// over the box's row.
inline int make_ring_map(CUtensorMap* map, const void* base, bool bf16, uint64_t cols, uint64_t rows, int64_t ld,
                         uint32_t cc) {
  PFN_encodeTiled enc = get_encode_fn();
  if (!enc) return fl_internal_error(FL_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cuuint64_t(ld) * (bf16 ? 2 : 4)};
  cuuint32_t box[2] = {cc, 32};
  const uint32_t row = cc * (bf16 ? 2 : 4);
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                   const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   row == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : row == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    return fl_internal_error(FL_ERR_INVALID_ARG, "tensor map encode failed (%d): epilogue operand, ld %lld", (int)r, (long long)ld);
  return FL_OK;
}
// The ring epilogues' maps of every problem of a launch.
inline int make_ring_maps(GemmMaps<FAM_F32>& maps, const fl_gemm_args* a, const Problems& pr, const Epi& e) {
  for (int r = 0; r < pr.n; ++r)
    if (int rc = make_ring_map(&maps.w[r], static_cast<float*>(e.D) + e.o_d[r], false, a->N, a->M, e.ldd, F32Ring::CC)) return rc;
  return FL_OK;
}
inline int make_ring_maps(GemmMaps<FAM_ADAMW>& maps, const fl_gemm_args* a, const Problems& pr, const Epi& e) {
  for (int r = 0; r < pr.n; ++r) {
    int rc = make_ring_map(&maps.w[r], static_cast<float*>(e.D) + e.o_d[r], false, a->N, a->M, e.ldd, AdamRing::CC);
    if (!rc) rc = make_ring_map(&maps.m[r], e.adam_m + e.o_adam[r], false, a->N, a->M, e.ldd, AdamRing::CC);
    if (!rc) rc = make_ring_map(&maps.v[r], e.adam_v + e.o_adam[r], false, a->N, a->M, e.ldd, AdamRing::CC);
    if (!rc) rc = make_ring_map(&maps.h[r], e.aux_out + e.o_aux_out[r], true, a->N, a->M, e.ld_aux_out, AdamRing::CC);
    if (rc) return rc;
  }
  return FL_OK;
}

inline int num_sms() { return fl_sm_count(); }

// Row-group raster that minimises DRAM reads for tiles of bm x bn (see Raster).
inline Raster pick_raster(int M, int N, int K, int bm, int bn) {
  const int num_m = (M + bm - 1) / bm, num_n = N / bn;
  const double pa = double(bm) * K * 2, pb = double(bn) * K * 2;
  const double budget = K <= 8192 ? L2_GROUP_BUDGET_SHORT_K : L2_GROUP_BUDGET;
  int gm = (int)(budget / pa), gn = (int)(budget / pb);
  gm = gm < 1 ? 1 : (gm > num_m ? num_m : gm);
  gn = gn < 1 ? 1 : (gn > num_n ? num_n : gn);
  const double cost_m = pa * num_m + pb * num_n * ((num_m + gm - 1) / gm);
  const double cost_n = pb * num_n + pa * num_m * ((num_n + gn - 1) / gn);
  Raster r;
  r.along_n = cost_n < cost_m ? 1 : 0;
  r.gsz = r.along_n ? gn : gm;
  return r;
}

template <int BN, bool A_MN, bool B_MN, int FAM>
int launch(const fl_gemm_args* a, const Problems& pr, const Epi& epi, int* status, cudaStream_t st) {
  using C = Cfg<BN, FAM>;
  auto kern = gemm_tc_kernel<BN, A_MN, B_MN, FAM>;
  FL_CUDA_TRY(fl_func_smem((const void*)kern, C::SMEM_BYTES));
  GemmMaps<FAM> maps;
  const int batch = pr.n;
  for (int r = 0; r < batch; ++r) {
    int rc;
    // A(m,k): K-major -> [M rows, K inner]; MN-major -> [K rows, M inner]
    if (!A_MN) rc = make_map(&maps.a[r], pr.A[r], a->K, a->M, pr.lda[r], BM);
    else rc = make_map(&maps.a[r], pr.A[r], a->M, a->K, pr.lda[r], BK);
    if (rc) return rc;
    if (!B_MN) rc = make_map(&maps.b[r], pr.B[r], a->K, a->N, pr.ldb[r], BN);
    else rc = make_map(&maps.b[r], pr.B[r], a->N, a->K, pr.ldb[r], BK);
    if (rc) return rc;
  }
  if constexpr (FAM == FAM_ADAMW || FAM == FAM_F32)
    if (int rc = make_ring_maps(maps, a, pr, epi)) return rc;
  const int num_m = (a->M + BM - 1) / BM, num_n = a->N / BN;
  const int tiles = batch * num_m * num_n;
  const int grid = tiles < num_sms() ? tiles : num_sms();
  const Raster r = pick_raster(a->M, a->N, a->K, BM, BN);
  FL_CUDA_TRY(fl_launch(gemm_tc_kernel<BN, A_MN, B_MN, FAM>, dim3(grid), dim3(EpiCfg<FAM, BN>::THREADS), C::SMEM_BYTES, st, maps,
                        epi, a->M, a->N, a->K, batch, r, status));
  return FL_OK;
}

// CTA pairs the current device keeps resident at once for the pair kernel (0 if it cannot
// run there); queried once per device (each of the first 64 devices caches its answer).
template <int PBN, bool A_MN, bool B_MN, int FAM>
int pair_slots() {
  constexpr int MAX_DEV = 64;
  static std::atomic<int> cache[MAX_DEV];  // slots + 1; 0: not queried yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const bool cached = dev >= 0 && dev < MAX_DEV;
  if (cached) {
    const int c = cache[dev].load(std::memory_order_relaxed);
    if (c > 0) return c - 1;
  }
  auto kern = gemm_pair_kernel<PBN, A_MN, B_MN, FAM>;
  int slots = 0;
  if (fl_func_smem((const void*)kern, CfgPair<PBN, FAM>::SMEM_BYTES) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(2 * num_sms());
    cfg.blockDim = dim3(EpiCfg<FAM, PBN>::THREADS);
    cfg.dynamicSmemBytes = CfgPair<PBN, FAM>::SMEM_BYTES;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) slots = n;
  }
  cudaGetLastError();  // a refused query leaves the single-SM kernel in use
  if (cached) cache[dev].store(slots + 1, std::memory_order_relaxed);
  return slots;
}

template <int PBN, bool A_MN, bool B_MN, int FAM>
int launch_pair(const fl_gemm_args* a, const Problems& pr, const Epi& epi, int* status, cudaStream_t st) {
  auto kern = gemm_pair_kernel<PBN, A_MN, B_MN, FAM>;
  const int slots = pair_slots<PBN, A_MN, B_MN, FAM>();
  if (slots <= 0) return fl_internal_error(FL_ERR_CUDA, "gemm: the CTA-pair kernel cannot be resident");
  GemmMaps<FAM> maps;
  const int batch = pr.n;
  for (int r = 0; r < batch; ++r) {
    int rc;
    // each CTA loads 128 rows of A and PBN / 2 columns of B per k-block
    if (!A_MN) rc = make_map(&maps.a[r], pr.A[r], a->K, a->M, pr.lda[r], 128);
    else rc = make_map(&maps.a[r], pr.A[r], a->M, a->K, pr.lda[r], BK);
    if (rc) return rc;
    if (!B_MN) rc = make_map(&maps.b[r], pr.B[r], a->K, a->N, pr.ldb[r], PBN / 2);
    else rc = make_map(&maps.b[r], pr.B[r], a->N, a->K, pr.ldb[r], BK);
    if (rc) return rc;
  }
  if constexpr (FAM == FAM_ADAMW || FAM == FAM_F32)
    if (int rc = make_ring_maps(maps, a, pr, epi)) return rc;
  const int tiles = batch * ((a->M + PAIR_BM - 1) / PAIR_BM) * (a->N / PBN);
  const int pairs = tiles < slots ? tiles : slots;
  const Raster r = pick_raster(a->M, a->N, a->K, PAIR_BM, PBN);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see pdl_wait
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(EpiCfg<FAM, PBN>::THREADS);
  cfg.dynamicSmemBytes = CfgPair<PBN, FAM>::SMEM_BYTES;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  FL_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, maps, epi, a->M, a->N, a->K, batch, r, status));
  return FL_OK;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Every (layout, family) pair of each tile shape; the operand layouts and the single-SM and
// CTA-pair kernels are instantiated in separate translation units so that the build compiles
// them in parallel.
#define FL_GEMM_LAUNCH_ARGS const fl_gemm_args*, const Problems&, const Epi&, int*, cudaStream_t
#define FL_GEMM_PAIR_FAM(EXT, PBN, AMN, BMN, FAM)          \
  EXT template int pair_slots<PBN, AMN, BMN, FAM>();       \
  EXT template int launch_pair<PBN, AMN, BMN, FAM>(FL_GEMM_LAUNCH_ARGS);
#define FL_GEMM_SINGLE_FAM(EXT, BN, AMN, BMN, FAM) EXT template int launch<BN, AMN, BMN, FAM>(FL_GEMM_LAUNCH_ARGS);
#define FL_GEMM_FAMS(X, EXT, W, AMN, BMN) \
  X(EXT, W, AMN, BMN, FAM_PLAIN)          \
  X(EXT, W, AMN, BMN, FAM_GELU)           \
  X(EXT, W, AMN, BMN, FAM_RESID)          \
  X(EXT, W, AMN, BMN, FAM_ROPE)           \
  X(EXT, W, AMN, BMN, FAM_ADAMW)
// The narrow tiles (256 x 128 on a pair, 128 x 64) are for outputs of few tiles, which weight
// updates are not.
#define FL_GEMM_NARROW_FAMS(X, EXT, W, AMN, BMN) \
  X(EXT, W, AMN, BMN, FAM_PLAIN)                 \
  X(EXT, W, AMN, BMN, FAM_GELU)                  \
  X(EXT, W, AMN, BMN, FAM_RESID)                 \
  X(EXT, W, AMN, BMN, FAM_ROPE)
// The weight gradients' families on CTA pairs only: AdamW over long contractions, fp32 gradients.
#define FL_GEMM_INSTANTIATE_WGRAD(EXT)                  \
  FL_GEMM_PAIR_FAM(EXT, 256, true, true, FAM_ADAMW_LONG) \
  FL_GEMM_PAIR_FAM(EXT, 256, true, true, FAM_F32)
#define FL_GEMM_INSTANTIATE_PAIR(EXT, AMN, BMN)      \
  FL_GEMM_FAMS(FL_GEMM_PAIR_FAM, EXT, 256, AMN, BMN) \
  FL_GEMM_NARROW_FAMS(FL_GEMM_PAIR_FAM, EXT, 128, AMN, BMN)
#define FL_GEMM_INSTANTIATE_SINGLE(EXT, AMN, BMN)      \
  FL_GEMM_FAMS(FL_GEMM_SINGLE_FAM, EXT, 256, AMN, BMN) \
  FL_GEMM_FAMS(FL_GEMM_SINGLE_FAM, EXT, 128, AMN, BMN) \
  FL_GEMM_NARROW_FAMS(FL_GEMM_SINGLE_FAM, EXT, 64, AMN, BMN)

}  // namespace fl_gemm
