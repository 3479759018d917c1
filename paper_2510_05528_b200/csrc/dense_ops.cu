// Dense contractions of the ARMOR iteration, dispatched by the configured precision:
// right-multiplication by the weighting H_w, the calibration Gram, and the core product of the
// deployment form.  SIMT = fp32 CUDA cores; TF32 / FP32X3 = tcgen05 tensor cores (1 or 3 tf32 passes);
// FP16X3 = three fp16 passes on operands scaled into the fp16 range (split_f16.cu).
#include <cuda_fp16.h>

#include "armor_internal.cuh"

// The tensor-core accumulator adds with truncation, so a long run of same-sign terms drifts by about
// (K / 8) * passes * 2^-24.  The GEMM therefore drains its accumulator every K_SEGMENT columns of the
// contraction into running sums held by its epilogue warps (ordinary round-to-nearest fp32 adds).
static const int64_t K_SEGMENT = 1024;

// Products this small run on the fp32 lanes: one launch instead of the operand split, the tensor-core product and the sum
// of its pieces, whose fixed costs (tensor memory, cluster launch, a second pass over the operand) exceed the arithmetic.
static bool dense_on_lanes(const armor_ctx* c, int64_t rows) {
  if (c->cfg.precision == ARMOR_PREC_SIMT) return true;
  return c->cfg.precision != ARMOR_PREC_TF32 && rows * c->d_in * c->d_in <= (1 << 25);
}

armor_status prepare_H(armor_ctx* c, const float* H, cudaStream_t s) {
  launch_extract_hblocks(c, H, s);
  if (c->cfg.h_mode == ARMOR_H_FULL && c->cfg.precision == ARMOR_PREC_FP32X3)
    launch_split_hilo(c, H, nullptr, c->Hlo, c->d_in * c->d_in, s);
  if (c->cfg.h_mode == ARMOR_H_FULL && c->cfg.precision == ARMOR_PREC_FP16X3)
    launch_f16_prepare_H(c, H, s);
  return ARMOR_OK;
}

armor_status rmul_H(armor_ctx* c, const float* in, const float* H, float* out, int64_t rows, const float* d1,
                    double* out1, const float* d2, double* out2, cudaStream_t s) {
  const int64_t d_in = c->d_in;
  if (c->cap_split && c->cfg.h_mode == ARMOR_H_FULL) {
    // capture in pieces: close the piece, remember this product, open the next piece (s is the capturing stream)
    if (c->cap_failed) return ARMOR_OK;
    if (c->cap_n >= ARMOR_MAX_PIECES - 1 || cudaStreamEndCapture(s, &c->cap_graph[c->cap_n]) != cudaSuccess) {
      c->cap_failed = 1;
      return ARMOR_OK;
    }
    c->cap_call[c->cap_n] = {in, H, out, rows, d1, out1, d2, out2};
    ++c->cap_n;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) c->cap_failed = 1;
    return ARMOR_OK;
  }
  if (c->cfg.h_mode == ARMOR_H_DIAG) {
    launch_colscale(c, in, c->hdiag, out, rows, d_in, s);
  } else if (dense_on_lanes(c, rows)) {
    BGemm g{};
    g.A = in; g.sAm = d_in; g.sAk = 1;
    g.B = H; g.sBk = d_in; g.sBn = 1;
    g.C = out; g.sCm = d_in; g.sCn = 1;
    g.M = (int)rows; g.N = (int)d_in; g.K = (int)d_in; g.batch = 1; g.alpha = 1.f;
    launch_bgemm(c, g, s);
  } else {
    TcGemm g{};
    g.lda = d_in; g.ldb = d_in; g.ldc = d_in;
    g.M = rows; g.N = d_in; g.K = d_in;
    g.C = out;
    if (c->cfg.precision == ARMOR_PREC_FP32X3) {
      // left operand as a high part plus the fp32 remainder.  The tensor core ignores the low 13 bits of a
      // 32-bit operand, so the operand itself serves as its high part and only the remainder is written.
      launch_split_hilo(c, in, nullptr, c->Lo, rows * d_in, s);
      g.A = in; g.Alo = c->Lo; g.B = H; g.Blo = c->Hlo; g.passes = 3;
    } else if (c->cfg.precision == ARMOR_PREC_FP16X3) {
      // in . H = rowscale . [(in d) rho] [H / (d d^T) 2^12] . d : both factors as fp16 high and low parts
      __half* ahi = reinterpret_cast<__half*>(c->Lo);
      __half* hhi = reinterpret_cast<__half*>(c->Hlo);
      launch_f16_split_rows(c, in, d_in, rows, d_in, c->hpow, f16_H_post_scale(), ahi, ahi + rows * d_in, c->rowscale, s);
      g.A = ahi; g.Alo = ahi + rows * d_in; g.B = hhi; g.Blo = hhi + d_in * d_in; g.passes = 6; g.fp16 = 1;
      g.row_scale = c->rowscale; g.col_scale = c->hpow;
    } else {
      g.A = in; g.B = H; g.passes = 1;
    }
    g.d1 = d1; g.d2 = d2;
    g.k_segment = (g.passes >= 3) ? K_SEGMENT : 0;   // one-pass tf32 rounding (2^-11) dwarfs the accumulator drift
    g.part1 = d1 ? c->partials : nullptr;
    g.part2 = d2 ? c->partials + 8 * c->npart : nullptr;
    int n_part = 0;
    armor_status st = launch_tc_gemm(c, g, &n_part, s);
    if (st != ARMOR_OK) return st;
    if (d1) reduce_partials_to(c, c->partials, n_part, out1, s);
    if (d2) reduce_partials_to(c, c->partials + 8 * c->npart, n_part, out2, s);
    return ARMOR_OK;
  }
  if (d1) dot_to_ptr(c, out, d1, rows * d_in, out1, s);
  if (d2) dot_to_ptr(c, out, d2, rows * d_in, out2, s);
  return ARMOR_OK;
}

// The product of a Gram with more room for the sums of cut tiles: `floats` of scratch at `spare`, where that holds more slabs
// (128 x 256 sums) than the context's own.  A Gram of 1,024 channels has 10 tiles for 74 pairs of CTAs and 16 segments of 1,024 tokens
// a launch, 320 slabs: uncut it kept 10 pairs busy (bf16, 30,000 tokens: 188 us).  Same sums in the same order.
static armor_status gram_product(armor_ctx* c, const TcGemm& g, float* spare, int64_t floats, cudaStream_t s) {
  float* const own = c->gemm_slabs;
  const int64_t own_count = c->gemm_slab_count, n = floats / (128 * 256);
  if (spare && n > own_count) { c->gemm_slabs = spare; c->gemm_slab_count = n; }
  const armor_status st = launch_tc_gemm(c, g, nullptr, s);
  c->gemm_slabs = own; c->gemm_slab_count = own_count;
  return st;
}

armor_status gram_accumulate(armor_ctx* c, const void* Xv, int x_dtype, int64_t n_rows, int64_t ldx, float* H,
                             cudaStream_t s) {
  const int64_t d_in = c->d_in;
  const float* X = static_cast<const float*>(Xv);
  const bool bf16 = (x_dtype == ARMOR_DTYPE_BF16);
  if (c->cfg.precision == ARMOR_PREC_SIMT) {
    if (bf16) return ARMOR_ERR_UNSUPPORTED;
    // H += X^T X, element (m, k) of the left operand is X[k][m]
    const int64_t step = 1 << 20;
    for (int64_t r0 = 0; r0 < n_rows; r0 += step) {
      const int64_t n = n_rows - r0 < step ? n_rows - r0 : step;
      BGemm g{};
      g.A = X + r0 * ldx; g.sAm = 1; g.sAk = ldx;
      g.B = X + r0 * ldx; g.sBk = ldx; g.sBn = 1;
      g.C = H; g.sCm = d_in; g.sCn = 1;
      g.D = H; g.sDm = d_in; g.sDn = 1;
      g.M = (int)d_in; g.N = (int)d_in; g.K = (int)n; g.batch = 1; g.alpha = 1.f; g.beta = 1.f;
      launch_bgemm(c, g, s);
    }
    return ARMOR_OK;
  }
  if (bf16 && ldx % 8 == 0 && reinterpret_cast<uintptr_t>(Xv) % 16 == 0 && d_in % 32 == 0) {
    // bf16 activations go to the tensor cores as they lie in memory: X is an operand of X^T X that is contiguous along
    // the channels, products of two bf16 values have 16 significant bits, so nothing is scaled, transposed or staged.  (A
    // leading dimension or base that TMA does not take leaves the staged path below.)
    // The accumulator rounds to multiples of 2^-149: about 2^-139 in a sum of 16,384 tokens, which counts only between two
    // channels whose norms multiply to less than 2^-115.  In the mode that scales its operands a channel that nowhere reaches
    // 2^-57 is therefore left out of the product (its scale is 0) and its entries are summed in fp64 before the mirroring.
    // One launch per gram_rows tokens, as in the staged path: a long call sums like a sequence of shorter ones.
    float* const in_range = c->cfg.precision == ARMOR_PREC_FP16X3 ? c->gscale : nullptr;
    if (in_range) launch_gram_range(c, Xv, ldx, n_rows, in_range, s);
    for (int64_t r0 = 0; r0 < n_rows; r0 += c->gram_rows) {
      TcGemm g{};
      g.A = static_cast<const char*>(Xv) + (size_t)(r0 * ldx) * 2; g.lda = ldx;
      g.B = g.A; g.ldb = ldx;
      g.C = H; g.ldc = d_in;
      g.M = d_in; g.N = d_in; g.K = n_rows - r0 < c->gram_rows ? n_rows - r0 : c->gram_rows;
      g.passes = 0; g.mn_major = 1;
      g.row_scale = g.col_scale = in_range;
      g.dependent = in_range && r0 == 0;
      g.accumulate = 1;
      g.symmetric_lower = 1;
      g.k_segment = K_SEGMENT;
      const armor_status st = gram_product(c, g, c->Xt_hi, d_in * c->gram_rows, s);     // (nothing is staged)
      if (st != ARMOR_OK) return st;
    }
    launch_mirror_lower(c, H, d_in, s, Xv, ldx, n_rows, in_range);
    return ARMOR_OK;
  }
  if (c->cfg.precision == ARMOR_PREC_FP16X3) {
    // every chunk is scaled per channel into the fp16 range; bf16 activations are then exact in one fp16 part
    const size_t esz = bf16 ? 2 : 4;
    // A call of several chunks stages chunk p + 1 (HBM bound) on the context's side stream while the tensor cores
    // contract chunk p on the caller's stream: two staging buffers with their scales, an event per hand-over.  The
    // contractions stay in the caller's stream in chunk order, so H is the same bit for bit.
    const int64_t n_chunks = (n_rows + c->gram_rows - 1) / c->gram_rows;
    bool overlap = n_chunks > 1 && c->side_stream && c->Xt_hi2 && c->timing_on < 2;
    if (overlap) {
      cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(s, &cst) != cudaSuccess || cst != cudaStreamCaptureStatusNone) overlap = false;
    }
    if (overlap) {
      // the side stream starts where the caller's stream is now: the inputs are ready and both buffers are free
      if (cudaEventRecord(c->ev_fork, s) != cudaSuccess || cudaStreamWaitEvent(c->side_stream, c->ev_fork, 0) != cudaSuccess)
        return ARMOR_ERR_CUDA;
    }
    int64_t p = 0;
    for (int64_t r0 = 0; r0 < n_rows; r0 += c->gram_rows, ++p) {
      const int b = overlap ? (int)(p & 1) : 0;
      __half* thi = reinterpret_cast<__half*>(b ? c->Xt_hi2 : c->Xt_hi);
      __half* tlo = thi + d_in * c->gram_rows;
      float* gscale = b ? c->gscale2 : c->gscale;
      cudaStream_t ss = overlap ? c->side_stream : s;
      const int64_t n = n_rows - r0 < c->gram_rows ? n_rows - r0 : c->gram_rows;
      // buffer b was last read by the contraction of chunk p - 2
      if (overlap && p >= 2 && cudaStreamWaitEvent(ss, c->ev_used[b], 0) != cudaSuccess) return ARMOR_ERR_CUDA;
      armor_status st = launch_f16_gram_stage(c, static_cast<const char*>(Xv) + (size_t)(r0 * ldx) * esz, x_dtype, ldx, n,
                                              d_in, thi, tlo, gscale, ss);
      if (st != ARMOR_OK) return st;
      if (overlap && (cudaEventRecord(c->ev_staged[b], ss) != cudaSuccess ||
                      cudaStreamWaitEvent(s, c->ev_staged[b], 0) != cudaSuccess))
        return ARMOR_ERR_CUDA;
      TcGemm g{};
      g.A = thi; g.Alo = tlo; g.lda = d_in;
      g.B = thi; g.Blo = tlo; g.ldb = d_in;
      g.C = H; g.ldc = d_in;
      g.M = d_in; g.N = d_in; g.K = n;
      g.passes = bf16 ? 0 : 6; g.fp16 = 1; g.mn_major = 1;
      g.row_scale = gscale; g.col_scale = gscale;
      g.accumulate = 1;
      g.symmetric_lower = 1;
      g.k_segment = K_SEGMENT;
      st = gram_product(c, g, overlap ? nullptr : c->Xt_hi2, d_in * c->gram_rows, s);   // (the second staging buffer is idle)
      if (st != ARMOR_OK) return st;
      if (overlap && cudaEventRecord(c->ev_used[b], s) != cudaSuccess) return ARMOR_ERR_CUDA;
    }
    launch_mirror_lower(c, H, d_in, s);
    return ARMOR_OK;
  }
  // bf16 values are exact in tf32: one tensor-core pass gives exact products
  const bool x3 = c->cfg.precision == ARMOR_PREC_FP32X3 && !bf16;
  const size_t esz = bf16 ? 2 : 4;
  for (int64_t r0 = 0; r0 < n_rows; r0 += c->gram_rows) {
    const int64_t n = n_rows - r0 < c->gram_rows ? n_rows - r0 : c->gram_rows;
    const int64_t kpad = (n + 31) / 32 * 32;     // staged row length (zero padded)
    launch_transpose_split(c, static_cast<const char*>(Xv) + (size_t)(r0 * ldx) * esz, x_dtype, ldx, n, d_in, c->Xt_hi,
                           x3 ? c->Xt_lo : nullptr, kpad, s);
    TcGemm g{};
    g.A = c->Xt_hi; g.Alo = c->Xt_lo; g.lda = kpad;
    g.B = c->Xt_hi; g.Blo = c->Xt_lo; g.ldb = kpad;
    g.C = H; g.ldc = d_in;
    g.M = d_in; g.N = d_in; g.K = kpad;
    g.passes = x3 ? 3 : 1;
    g.accumulate = 1;
    g.symmetric_lower = 1;
    g.k_segment = (c->cfg.precision == ARMOR_PREC_FP32X3) ? K_SEGMENT : 4 * K_SEGMENT;
    armor_status st = launch_tc_gemm(c, g, nullptr, s);
    if (st != ARMOR_OK) return st;
  }
  launch_mirror_lower(c, H, d_in, s);   // the product accumulates the lower triangle only
  return ARMOR_OK;
}

// The core product of the fp32 forward in the three-pass fp16 mode: rows of z1 (tokens) and rows of S (outputs) each scaled
// by their own power of two.  S is split once for all chunks of a call, into U; z1 into the Gram's staging buffer, whose
// gram_rows x d_in words hold the two parts of up to gram_rows tokens, with the scales in the normalisation's scratch (128
// d_in floats).
bool core_f16_ok(const armor_ctx* c) {
  return c->cfg.precision == ARMOR_PREC_FP16X3 && c->d_out % 32 == 0 && c->d_in % 8 == 0;
}
// On the sparse tensor cores (sparse_tcgen05.cu) once tiles of 64 tokens fill the pairs of CTAs; for fewer the dense product cuts the
// contraction.  Whole forward, sparse / dense: 4096 x 4096, 200 tokens 90 / 84 us, 400 97 / 103, 1,600 152 / 198; 2048 x 8192, 400 tokens 122 / 105, 800
// 136 / 146; 14336 x 4096, 100 tokens 160 / 168; 512 x 4096, 1,600 tokens 82 / 78.
bool core_f16_sparse(const armor_ctx* c, int64_t n_tokens) {
  return tc_sparse3_ok(c) && n_tokens * (c->d_out / 256) >= (int64_t)c->n_sm / 2 * 64;
}
// S's parts in U (hi, then lo).  sparse: the parts of what a 2:4 core keeps, positions in Lo; if it is not 2:4 core_dense says so, and the first
// chunk's split puts the parts of the whole of S in their place.
armor_status core_f16_split_S(armor_ctx* c, const float* S, bool sparse, cudaStream_t s) {
  __half* shi = reinterpret_cast<__half*>(c->U);
  if (sparse) {
    if (cudaMemsetAsync(c->core_dense, 0, sizeof(int32_t), s) != cudaSuccess) return ARMOR_ERR_CUDA;
    launch_split_core24(c, S, shi, shi + c->wn, c->Lo, c->rowscale2, c->core_dense, s);
  } else {
    launch_f16_split_rows(c, S, c->d_in, c->d_out, c->d_in, nullptr, 1.f, shi, shi + c->wn, c->rowscale2, s);
  }
  return ARMOR_OK;
}
armor_status core_f16_product(armor_ctx* c, const float* z1, const float* S, bool sparse, bool first, float* z2, int64_t n, cudaStream_t s) {
  const int64_t d_in = c->d_in, d_out = c->d_out;
  __half* ahi = reinterpret_cast<__half*>(c->Xt_hi);
  __half* shi = reinterpret_cast<__half*>(c->U);
  float* scales = reinterpret_cast<float*>(c->colpart);         // 64 d_in doubles
  if (sparse) {
    // One of the two products does nothing, and which is known on the device only.  For a core that is not 2:4 that costs 10 to 25 us a
    // call over the dense product alone (14336 x 4096, 2,048 tokens 649 and 656 us, 1024 x 1024, 8,192 134 and 148, 14336 x 1024, 150 82 and
    // 104), for a 2:4 core up to 1 us.  Two sparse products for the former, of the first and the other two of every four: 1,047, 154, 155.
    launch_split_tokens(c, z1, n, ahi, ahi + n * d_in, scales, first ? S : nullptr, shi, shi + c->wn, c->rowscale2, c->core_dense, s);
    const armor_status st = launch_tc_sparse3(c, shi, shi + c->wn, c->Lo, c->rowscale2, ahi, ahi + n * d_in, scales, c->core_dense, z2, n, s);
    if (st != ARMOR_OK) return st;
  } else {
    launch_f16_split_rows(c, z1, d_in, n, d_in, nullptr, 1.f, ahi, ahi + n * d_in, scales, s);
  }
  TcGemm g{};
  g.lda = d_in; g.ldb = d_in; g.ldc = d_out;
  g.M = n; g.N = d_out; g.K = d_in;
  g.C = z2;
  g.A = ahi; g.Alo = ahi + n * d_in; g.B = shi; g.Blo = shi + c->wn; g.passes = 6; g.fp16 = 1;
  g.row_scale = scales; g.col_scale = c->rowscale2;
  g.k_segment = K_SEGMENT;
  g.only_if = sparse ? c->core_dense : nullptr;
  return launch_tc_gemm(c, g, nullptr, s);
}

armor_status apply_core(armor_ctx* c, const float* z1, const float* S, const void* packed, float* z2, int64_t n,
                        bool bf16, cudaStream_t s) {
  const int64_t d_in = c->d_in, d_out = c->d_out;
  if (packed) {
    // bf16 deployment with the 2:4 core on the sparse tensor cores: kept values, then positions
    if (!bf16 || !tc_sparse_ok(c)) return ARMOR_ERR_UNSUPPORTED;
    const char* buf = static_cast<const char*>(packed);
    launch_f32_to_bf16(c, z1, nullptr, c->U, n, d_in, s);
    return launch_tc_sparse(c, buf, buf + tc_sparse_values_bytes(c), c->U, z2, false, n, s);
  }
  if (bf16 && c->cfg.precision != ARMOR_PREC_SIMT && d_out % 32 == 0 && d_in % 8 == 0) {
    // bf16 deployment: the core and the wrapped activations are rounded to bf16 and multiplied on the bf16
    // tensor-core path with fp32 accumulation
    launch_f32_to_bf16(c, z1, nullptr, c->U, n, d_in, s);
    launch_f32_to_bf16(c, S, nullptr, c->P, d_out, d_in, s);
    TcGemm g{};
    g.lda = d_in; g.ldb = d_in; g.ldc = d_out;
    g.M = n; g.N = d_out; g.K = d_in;
    g.C = z2;
    g.A = c->U; g.B = c->P; g.passes = 0;
    g.k_segment = 0;
    return launch_tc_gemm(c, g, nullptr, s);
  }
  if (c->cfg.precision == ARMOR_PREC_SIMT || (d_out % 32) || (d_in % 4)) {
    BGemm g{};
    g.A = z1; g.sAm = d_in; g.sAk = 1;
    g.B = S; g.sBk = 1; g.sBn = d_in;
    g.C = z2; g.sCm = d_out; g.sCn = 1;
    g.M = (int)n; g.N = (int)d_out; g.K = (int)d_in; g.batch = 1; g.alpha = 1.f;
    launch_bgemm(c, g, s);
    return ARMOR_OK;
  }
  TcGemm g{};
  g.lda = d_in; g.ldb = d_in; g.ldc = d_out;
  g.M = n; g.N = d_out; g.K = d_in;
  g.C = z2;
  if (c->cfg.precision == ARMOR_PREC_FP32X3) {
    launch_split_hilo(c, z1, nullptr, c->Lo, n * d_in, s);
    launch_split_hilo(c, S, nullptr, c->U, c->wn, s);
    g.A = z1; g.Alo = c->Lo; g.B = S; g.Blo = c->U; g.passes = 3;
  } else if (c->cfg.precision == ARMOR_PREC_FP16X3) {
    return ARMOR_ERR_UNSUPPORTED;          // (fp32 activations of every shape the mode takes: core_f16_product)
  } else {
    g.A = z1; g.B = S; g.passes = 1;
  }
  g.k_segment = (g.passes >= 3) ? K_SEGMENT : 0;
  return launch_tc_gemm(c, g, nullptr, s);
}
