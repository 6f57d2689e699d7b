// fl_k_gemm: argument checks, epilogue set-up and dispatch to the instantiation of the
// operand layout, tile width and epilogue family (kernels: gemm_tc.cuh; instantiations:
// gemm_inst_fwd.cu, gemm_inst_dgrad.cu, gemm_inst_wgrad.cu).
#include <cstring>

#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_PAIR(extern, false, false)
FL_GEMM_INSTANTIATE_PAIR(extern, false, true)
FL_GEMM_INSTANTIATE_PAIR(extern, true, true)
FL_GEMM_INSTANTIATE_WGRAD(extern)
FL_GEMM_INSTANTIATE_SINGLE(extern, false, false)
FL_GEMM_INSTANTIATE_SINGLE(extern, false, true)
FL_GEMM_INSTANTIATE_SINGLE(extern, true, true)

// Contractions this long take the AdamW epilogue that leaves the operand ring six stages (its
// own operands in registers, FAM_ADAMW_LONG) instead of the one whose TMA ring takes two of
// them.  Measured, two 4096 x 16384 weights per launch, ring / registers: 730 / 790 us at K =
// 2048, 832 / 807 at 3072, 1038 / 878 at 4096, 1381 / 1156 at 6144, 1693 / 1450 at 8192.
constexpr int ADAMW_LONG_K = 3072;

// fp32 weight gradients on CTA pairs whose epilogue moves by TMA (FAM_F32): added ones always,
// stored ones below K = 1024.  Measured, two 4096 x 16384 gradients per launch, registers / ring:
// added 230 / 191 us at K = 77, 236 / 198 at 512, 244 / 220 at 1024, 330 / 327 at 2048; stored 102 /
// 97, 118 / 122, 181 / 186 and 309 / 306.
constexpr int F32_SHORT_K = 1024;
bool f32_ring(const fl_gemm_args* a) {
  return a->a_mn_major && !a->bias &&
         (a->epilogue == FL_EPI_ACCUM_F32 || (a->epilogue == FL_EPI_STORE_F32 && a->K < F32_SHORT_K));
}
// A short contraction's gradients are bound by their output: past what L2 holds the pair tile
// with the ring is the fastest whatever pick_shape estimates, two 4096 x 16384 (537 MB) added 225 ->
// 191 us at K = 77, 230 -> 198 at 512, stored 104 -> 97, 155 -> 122; 12288 x 4096 (201 MB) added 91 ->
// 81, 95 -> 86.  4096 x 4096 (67 MB, kept in L2) added takes 30 us on narrow tiles, 36 on these.
constexpr double F32_RING_MIN_BYTES = 128.0 * (1 << 20);
bool f32_ring_tile(const fl_gemm_args* a, int batch, int pairs) {
  return pairs > 0 && a->N % 256 == 0 && a->K < F32_SHORT_K && f32_ring(a) &&
         4.0 * batch * a->M * a->N > F32_RING_MIN_BYTES;
}

// Tile shapes: FL_TILE_* - 1, and two narrow ones that only the library picks.
enum { SHAPE_128 = 0, SHAPE_256 = 1, SHAPE_PAIR256 = 2, SHAPE_64 = 3, SHAPE_PAIR128 = 4 };

template <bool AMN, bool BMN, int FAM>
int dispatch_shape(int shape, const fl_gemm_args* a, const Problems& pr, const Epi& e, int* status, cudaStream_t st) {
  if constexpr (FAM != FAM_ADAMW) {
    if (shape == SHAPE_PAIR128) return launch_pair<128, AMN, BMN, FAM>(a, pr, e, status, st);
    if (shape == SHAPE_64) return launch<64, AMN, BMN, FAM>(a, pr, e, status, st);
  }
  switch (shape) {
    case SHAPE_PAIR256: return launch_pair<256, AMN, BMN, FAM>(a, pr, e, status, st);
    case SHAPE_256: return launch<256, AMN, BMN, FAM>(a, pr, e, status, st);
    default: return launch<128, AMN, BMN, FAM>(a, pr, e, status, st);
  }
}
template <bool AMN, bool BMN>
int dispatch_layout(int fam, int shape, const fl_gemm_args* a, const Problems& pr, const Epi& e, int* status,
                    cudaStream_t st) {
  switch (fam) {
    case FAM_GELU: return dispatch_shape<AMN, BMN, FAM_GELU>(shape, a, pr, e, status, st);
    case FAM_RESID: return dispatch_shape<AMN, BMN, FAM_RESID>(shape, a, pr, e, status, st);
    case FAM_ROPE: return dispatch_shape<AMN, BMN, FAM_ROPE>(shape, a, pr, e, status, st);
    case FAM_ADAMW: return dispatch_shape<AMN, BMN, FAM_ADAMW>(shape, a, pr, e, status, st);
    default: return dispatch_shape<AMN, BMN, FAM_PLAIN>(shape, a, pr, e, status, st);
  }
}

int dispatch_fam(int fam, int shape, bool amn, bool bmn, const fl_gemm_args* a, const Problems& pr, const Epi& e,
                 int* status, cudaStream_t st) {
  if (fam == FAM_ADAMW && shape == SHAPE_PAIR256 && amn && a->K >= ADAMW_LONG_K)
    return launch_pair<256, true, true, FAM_ADAMW_LONG>(a, pr, e, status, st);
  if (fam == FAM_PLAIN && shape == SHAPE_PAIR256 && f32_ring(a))
    return launch_pair<256, true, true, FAM_F32>(a, pr, e, status, st);
  if (!amn && !bmn) return dispatch_layout<false, false>(fam, shape, a, pr, e, status, st);
  if (!amn && bmn) return dispatch_layout<false, true>(fam, shape, a, pr, e, status, st);
  return dispatch_layout<true, true>(fam, shape, a, pr, e, status, st);
}

template <int PBN>
int pair_slots_for(int fam, bool amn, bool bmn) {
#define FL_SLOTS(AMN, BMN)                                               \
  switch (fam) {                                                         \
    case FAM_GELU: return pair_slots<PBN, AMN, BMN, FAM_GELU>();         \
    case FAM_RESID: return pair_slots<PBN, AMN, BMN, FAM_RESID>();       \
    case FAM_ROPE: return pair_slots<PBN, AMN, BMN, FAM_ROPE>();         \
    case FAM_ADAMW: return pair_slots<PBN, AMN, BMN, FAM_ADAMW>();       \
    default: return pair_slots<PBN, AMN, BMN, FAM_PLAIN>();              \
  }
  if (!amn && !bmn) { FL_SLOTS(false, false) }
  if (!amn && bmn) { FL_SLOTS(false, true) }
  FL_SLOTS(true, true)
#undef FL_SLOTS
}
}  // namespace fl_gemm

using namespace fl_gemm;

namespace {

// Checks one problem's arguments (everything but the batch fields).
int check_args(const fl_gemm_args* a) {
  if (!a || !a->A || !a->B || !a->D) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: null pointer");
  if (a->M < 0 || a->N <= 0 || a->K <= 0) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: bad sizes");
  if (a->N % 128) return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: N=%d is not a multiple of 128", a->N);
  if (a->epilogue < 0 || a->epilogue >= FL_EPI_COUNT) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: epilogue");
  if ((a->lda % 8) || (a->ldb % 8) || (a->ldd % 8) || !aligned16(a->A) || !aligned16(a->B) || !aligned16(a->D))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: leading dims must be multiples of 8 and pointers 16-byte aligned");
  if (a->a_mn_major && a->lda < a->M) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: lda < M");
  if (!a->a_mn_major && a->lda < a->K) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: lda < K");
  if (a->b_mn_major && a->ldb < a->N) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: ldb < N");
  if (!a->b_mn_major && a->ldb < a->K) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: ldb < K");
  if (a->a_mn_major && (a->M % 8)) return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: MN-major A needs M % 8 == 0");
  const int mode = a->epilogue;
  if ((mode == FL_EPI_BIAS_RESID || mode == FL_EPI_RESID || mode == FL_EPI_GELU_BWD) &&
      (!a->aux || (a->ld_aux % 8) || !aligned16(a->aux)))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: epilogue needs an aligned aux tensor");
  if ((a->aux_dtype != FL_DT_BF16 && a->aux_dtype != FL_DT_F32) || (a->d_dtype != FL_DT_BF16 && a->d_dtype != FL_DT_F32))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: aux/d dtype");
  if (a->aux_dtype == FL_DT_F32 && !(mode == FL_EPI_BIAS_RESID || mode == FL_EPI_RESID))
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: fp32 aux only for the residual epilogues");
  if (a->d_dtype == FL_DT_F32 && !(mode == FL_EPI_STORE || mode == FL_EPI_BIAS_RESID || mode == FL_EPI_RESID))
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: fp32 D only for STORE and the residual epilogues");
  if (a->ln_mean && (!a->ln_rstd || !a->ln_gamma || !a->ln_beta || !aligned16(a->ln_gamma) || !aligned16(a->ln_beta) ||
                     !(mode == FL_EPI_BIAS_RESID || mode == FL_EPI_RESID)))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: LayerNorm residual needs mean, rstd, gamma, beta");
  if ((mode == FL_EPI_BIAS_GELU || mode == FL_EPI_ADAMW) &&
      (!a->aux_out || (a->ld_aux_out % 8) || !aligned16(a->aux_out)))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: epilogue needs an aligned aux_out");
  if (mode == FL_EPI_ADAMW && (!a->adam_m || !a->adam_v || !aligned16(a->adam_m) || !aligned16(a->adam_v) ||
                               a->bias || (a->ldd % 4)))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: AdamW epilogue needs aligned moments and no bias");
  if (mode == FL_EPI_BIAS_ROPE) {
    if (!a->pos || !a->rope_tab || a->head_dim <= 0 || a->head_dim % 64 ||
        !(a->rotary_dim == 32 || a->rotary_dim == 64) || a->rotary_dim > a->head_dim)
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: RoPE epilogue arguments");
    if (a->pos2 && 2 * a->rotary_dim != a->head_dim)
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: 2D rotary needs rotary_dim = head_dim / 2");
  } else if (a->pos2) {
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: block positions only with the RoPE epilogue");
  }
  if (a->bias && !aligned16(a->bias)) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: bias alignment");
  if (fl_misaligned(a->rope_tab, 8) || fl_misaligned(a->pos, 4) || fl_misaligned(a->pos2, 4) ||
      fl_misaligned(a->ln_mean, 4) || fl_misaligned(a->ln_rstd, 4))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: rope_tab must be 8-byte and per-row arrays 4-byte aligned");
  if (a->colsum && mode != FL_EPI_GELU_BWD)
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: column sums only with the GeLU-backward epilogue");
  if (a->colsum && !aligned16(a->colsum))
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: colsum must be 16-byte aligned");
  if (a->tile < FL_TILE_AUTO || a->tile > FL_TILE_256x256_PAIR)
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: tile %d", a->tile);
  if (a->tile >= FL_TILE_128x256 && (a->N % 256))
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: 256-column tiles need N %% 256 == 0 (N=%d)", a->N);
  if (a->a_mn_major && !a->b_mn_major)
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: MN-major A with K-major B is not built");
  return FL_OK;
}

// The epilogue of problem 0 (offsets of the other problems zero).
Epi make_epi(const fl_gemm_args* a) {
  const int mode = a->epilogue;
  Epi e;
  memset(&e, 0, sizeof e);
  e.mode = mode;
  e.bias = a->bias;
  e.aux = reinterpret_cast<const __nv_bfloat16*>(a->aux);
  e.ld_aux = a->ld_aux;
  e.alpha = a->alpha;
  e.aux_out = reinterpret_cast<__nv_bfloat16*>(a->aux_out);
  e.ld_aux_out = a->ld_aux_out;
  e.D = a->D;
  e.ldd = a->ldd;
  e.pos = a->pos;
  e.pos2 = a->pos2;
  e.rope_tab = reinterpret_cast<const float2*>(a->rope_tab);
  e.rope_cols = 2 * a->n_heads * a->head_dim;
  e.head_dim = a->head_dim > 0 ? a->head_dim : 64;
  e.rotary_dim = a->rotary_dim;
  e.aux_f32 = a->aux_dtype == FL_DT_F32;
  e.d_f32 = a->d_dtype == FL_DT_F32 && mode != FL_EPI_ACCUM_F32;
  e.ln_mean = a->ln_mean;
  e.ln_rstd = a->ln_rstd;
  e.ln_gamma = a->ln_gamma;
  e.ln_beta = a->ln_beta;
  e.adam_m = a->adam_m;
  e.adam_v = a->adam_v;
  e.lr = a->lr;
  e.b1 = a->beta1;
  e.b2 = a->beta2;
  e.eps = a->eps;
  e.den_scale = a->eps < 0x1p-100f ? 0x1p40f : 1.f;  // the square root alone is 0 or at least 2^-75
  e.wd = a->weight_decay;
  e.inv_bc1 = a->inv_bc1;
  e.inv_bc2 = a->inv_bc2;
  e.colsum = a->colsum;
  return e;
}

bool d_is_f32(const fl_gemm_args* a) {
  const int mode = a->epilogue;
  return a->d_dtype == FL_DT_F32 || mode == FL_EPI_STORE_F32 || mode == FL_EPI_ACCUM_F32 || mode == FL_EPI_ADAMW;
}

// The tile shape with the least estimated time: waves of tiles, each as long as its main loop
// or its epilogue, and the fill and last epilogue.  Measured on GB300 (ns per 64-deep k-block
// of a CTA or pair with one tile at a time; us for the fixed part): 256 x 256 on a pair 295 and
// 9.7, 256 x 128 on a pair 230 and 5.4, 128 x 128 262 and 6.1, 128 x 64 180 and 5.0 (the two narrow
// tiles' fixed parts chosen by the H 256 step, which takes 119 us on 128 x 64 and 137 where the pair
// tile's 5.4 is set to 4.0; alone with operands in L2, K 256 .. 4096, they measure 5.0 and 4.6, the
// others 6.3 and 4.6, the k-blocks 263, 170, 230 and 150 ns).  So one wave of narrow tiles over all SMs beats a wide tile on a few of them: 4096 columns, K = 16384
// take 85 / 63 / 73 / 51 us (in that order) at 77 rows, 87 / 65 / 75 / 96 at 512; and wide tiles
// win once they fill the device: 170 / 224 / 271 / 319 us at 2048 rows.
int pick_shape(const fl_gemm_args* a, int batch, int fam, int pairs) {
  struct Shape {
    int id, bm, bn;
    double k_us, fixed_us, epi_us;  // per k-block; once; least per tile
  };
  static constexpr Shape shapes[] = {{SHAPE_PAIR256, 256, 256, 0.295, 9.7, 4.0},
                                     {SHAPE_PAIR128, 256, 128, 0.230, 5.4, 2.0},
                                     {SHAPE_128, 128, 128, 0.262, 6.1, 2.0},
                                     {SHAPE_64, 128, 64, 0.180, 5.0, 2.0},
                                     {SHAPE_256, 128, 256, 0.400, 9.7, 4.0}};
  const int num_k = (a->K + BK - 1) / BK;
  int best = SHAPE_128;
  double best_us = 0;
  for (const Shape& s : shapes) {
    const bool pair = s.bm == 256, narrow = s.id == SHAPE_PAIR128 || s.id == SHAPE_64;
    const int slots = pair ? pairs : num_sms();
    // 128 x 256 stands in for the pair where the device cannot hold it; weight updates have no narrow tiles
    if (slots <= 0 || a->N % s.bn || (s.id == SHAPE_256 && pairs > 0) || (narrow && fam == FAM_ADAMW)) continue;
    const long tiles = (long)batch * ((a->M + s.bm - 1) / s.bm) * (a->N / s.bn);
    const long waves = (tiles + slots - 1) / slots;
    const double main_us = num_k * s.k_us;
    const double us = waves * (main_us > s.epi_us ? main_us : s.epi_us) + s.fixed_us;
    if (best_us == 0 || us < best_us) {
      best = s.id;
      best_us = us;
    }
  }
  return best;
}

// Tile shape for the launch (see fl_k_gemm) and the dispatch.
int run(const fl_gemm_args* a, const Problems& pr, const Epi& e, int* status, cudaStream_t st) {
  const bool amn = a->a_mn_major != 0, bmn = a->b_mn_major != 0;
  const int fam = family_of(a->epilogue);
  const int batch = pr.n;
  if (a->tile == FL_TILE_256x256_PAIR && pair_slots_for<256>(fam, amn, bmn) <= 0)
    return fl_internal_error(FL_ERR_UNSUPPORTED, "gemm: this device cannot hold the CTA-pair kernel");
  if (a->tile != FL_TILE_AUTO) return dispatch_fam(fam, a->tile - 1, amn, bmn, a, pr, e, status, st);
  const int pairs = pair_slots_for<256>(fam, amn, bmn);
  const int shape = f32_ring_tile(a, batch, pairs) ? SHAPE_PAIR256 : pick_shape(a, batch, fam, pairs);
  return dispatch_fam(fam, shape, amn, bmn, a, pr, e, status, st);
}

// Element offset of p from p0 (both null, or both in the same address space; elem bytes).
int64_t elem_off(const void* p, const void* p0, int elem) {
  return (reinterpret_cast<intptr_t>(p) - reinterpret_cast<intptr_t>(p0)) / elem;
}

}  // namespace

extern "C" int fl_k_gemm(const fl_gemm_args* a, int* status, void* stream) {
  if (int rc = check_args(a)) return rc;
  if (a->M == 0) return FL_OK;
  if (a->batch < 0 || a->batch > FL_GEMM_MAX_BATCH)
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: batch %d outside 0..%d", a->batch, FL_GEMM_MAX_BATCH);
  const int batch = a->batch > 1 ? a->batch : 1;
  if (batch > 1) {
    // every problem's pointers keep the 16-byte alignment of the first problem's: strides in
    // bf16 elements multiples of 8, in fp32 elements multiples of 4 (and of 4 for the
    // per-row int32 / fp32 arrays read one element at a time)
    const bool d32 = d_is_f32(a);
    if ((a->a_bstride % 8) || (a->b_bstride % 8) || (a->d_bstride % (d32 ? 4 : 8)) ||
        (a->aux && (a->aux_bstride % (a->aux_dtype == FL_DT_F32 ? 4 : 8))) || (a->aux_out && (a->aux_out_bstride % 8)) ||
        ((a->bias || a->colsum) && (a->bias_bstride % 4)) || (a->ln_mean && (a->lnp_bstride % 4)) ||
        (a->adam_m && (a->adam_bstride % 4)))
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm: batch strides break the 16-byte alignment");
  }
  Epi e = make_epi(a);
  Problems pr;
  memset(&pr, 0, sizeof pr);
  pr.n = batch;
  for (int r = 0; r < batch; ++r) {
    pr.A[r] = static_cast<const __nv_bfloat16*>(a->A) + r * a->a_bstride;
    pr.B[r] = static_cast<const __nv_bfloat16*>(a->B) + r * a->b_bstride;
    pr.lda[r] = a->lda;
    pr.ldb[r] = a->ldb;
    e.o_d[r] = r * a->d_bstride;
    e.o_aux[r] = r * a->aux_bstride;
    e.o_aux_out[r] = r * a->aux_out_bstride;
    e.o_bias[r] = r * a->bias_bstride;
    e.o_row[r] = r * a->row_bstride;
    e.o_lnp[r] = r * a->lnp_bstride;
    e.o_adam[r] = r * a->adam_bstride;
  }
  return run(a, pr, e, status, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int fl_k_gemm_multi(const fl_gemm_args* probs, int32_t n, int* status, void* stream) {
  if (!probs || n < 1 || n > FL_GEMM_MAX_BATCH)
    return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: need 1..%d problems", FL_GEMM_MAX_BATCH);
  const fl_gemm_args* a = probs;
  for (int r = 0; r < n; ++r) {
    const fl_gemm_args* q = probs + r;
    if (int rc = check_args(q)) return rc;
    if (q->batch > 1) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: problem %d has batch %d", r, q->batch);
    // one shape, layout, epilogue and set of scalars; output leading dimensions shared
    const bool same = q->M == a->M && q->N == a->N && q->K == a->K && q->a_mn_major == a->a_mn_major &&
                      q->b_mn_major == a->b_mn_major && q->epilogue == a->epilogue && q->ldd == a->ldd &&
                      q->ld_aux == a->ld_aux && q->ld_aux_out == a->ld_aux_out && q->aux_dtype == a->aux_dtype &&
                      q->d_dtype == a->d_dtype && q->alpha == a->alpha && q->lr == a->lr && q->beta1 == a->beta1 &&
                      q->beta2 == a->beta2 && q->eps == a->eps && q->weight_decay == a->weight_decay &&
                      q->inv_bc1 == a->inv_bc1 && q->inv_bc2 == a->inv_bc2 && q->n_heads == a->n_heads &&
                      q->head_dim == a->head_dim && q->rotary_dim == a->rotary_dim && q->rope_tab == a->rope_tab &&
                      q->tile == a->tile;
    if (!same) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: problem %d differs in shape or epilogue", r);
    // each optional operand present in every problem or in none
    const bool present = (!q->aux == !a->aux) && (!q->aux_out == !a->aux_out) && (!q->bias == !a->bias) &&
                         (!q->colsum == !a->colsum) && (!q->pos == !a->pos) && (!q->pos2 == !a->pos2) &&
                         (!q->ln_mean == !a->ln_mean) && (!q->adam_m == !a->adam_m);
    if (!present) return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: problem %d lacks an operand", r);
  }
  if (a->M == 0) return FL_OK;
  Epi e = make_epi(a);
  Problems pr;
  memset(&pr, 0, sizeof pr);
  pr.n = n;
  const int d_el = d_is_f32(a) ? 4 : 2, aux_el = a->aux_dtype == FL_DT_F32 ? 4 : 2;
  for (int r = 0; r < n; ++r) {
    const fl_gemm_args* q = probs + r;
    pr.A[r] = q->A;
    pr.B[r] = q->B;
    pr.lda[r] = q->lda;
    pr.ldb[r] = q->ldb;
    // offsets from problem 0's pointers: every pointer is 16-byte aligned, so each offset
    // keeps the vector alignment the epilogue relies on
    e.o_d[r] = elem_off(q->D, a->D, d_el);
    e.o_aux[r] = a->aux ? elem_off(q->aux, a->aux, aux_el) : 0;
    e.o_aux_out[r] = a->aux_out ? elem_off(q->aux_out, a->aux_out, 2) : 0;
    e.o_bias[r] = a->bias ? elem_off(q->bias, a->bias, 4) : a->colsum ? elem_off(q->colsum, a->colsum, 4) : 0;
    if (a->bias && a->colsum && elem_off(q->colsum, a->colsum, 4) != e.o_bias[r])
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: bias and colsum offsets differ");
    e.o_row[r] = a->pos ? elem_off(q->pos, a->pos, 4) : a->ln_mean ? elem_off(q->ln_mean, a->ln_mean, 4) : 0;
    if ((a->pos2 && elem_off(q->pos2, a->pos2, 4) != e.o_row[r]) ||
        (a->ln_mean && (elem_off(q->ln_mean, a->ln_mean, 4) != e.o_row[r] ||
                        elem_off(q->ln_rstd, a->ln_rstd, 4) != e.o_row[r])))
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: per-row operand offsets differ");
    e.o_lnp[r] = a->ln_gamma ? elem_off(q->ln_gamma, a->ln_gamma, 4) : 0;
    if (a->ln_gamma && elem_off(q->ln_beta, a->ln_beta, 4) != e.o_lnp[r])
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: LayerNorm gain and shift offsets differ");
    e.o_adam[r] = a->adam_m ? elem_off(q->adam_m, a->adam_m, 4) : 0;
    if (a->adam_m && elem_off(q->adam_v, a->adam_v, 4) != e.o_adam[r])
      return fl_internal_error(FL_ERR_INVALID_ARG, "gemm multi: Adam moment offsets differ");
  }
  return run(a, pr, e, status, reinterpret_cast<cudaStream_t>(stream));
}
