// Operand preparation for the three-pass fp16 mode of the dense contractions (ARMOR_PREC_FP16X3).
//
// An fp32 value x is written as hi + lo with hi = fp16(x), lo = fp16(x - hi): 22 significant bits, as with two
// tf32 parts, but fp16 has 5 exponent bits only.  Every operand is therefore scaled by powers of two (exact)
// so that the entries that matter for a dot product land in the range where both parts are normal numbers:
//   * a left operand L of L.H is scaled per column by d_k = 2^floor(log2 sqrt(H_kk)) and then per row so that
//     the row's largest entry lies in [2^14, 2^15);
//   * H is replaced by H_kn / (d_k d_n) * 2^12: a positive semidefinite H has |H_kn| <= sqrt(H_kk H_nn), so these
//     entries are below 2^14 in magnitude whatever the spread of the channel scales;
//   * a chunk of activations X (Gram X^T X, Section 2 of the paper) is scaled per channel by its largest
//     magnitude inside the chunk.
// Entries far below their row's or column's maximum lose relative accuracy (absolute error 2^-25 after scaling,
// i.e. 2^-39 of the maximum) -- less than what the fp32 inputs themselves carry.  The GEMM's epilogue multiplies
// the accumulator by the inverse scales.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "armor_internal.cuh"
#include "tc_common.cuh"

namespace {

constexpr int NT = 256;
constexpr int TARGET_EXP = 15;   // frexp exponent of the scaled maximum: values in [2^14, 2^15)
constexpr int H_SHIFT = 12;      // H / (d d^T) has entries below 4; times 2^12 they stay below 2^14

// Finite values beyond the fp16 range are clamped (after the scalings above this happens only to an H that is not
// positive semidefinite); NaN and Inf pass through, so that unusable inputs stay visible in the result.
__device__ __forceinline__ float clamp_f16(float v) { return isfinite(v) ? fminf(fmaxf(v, -65504.f), 65504.f) : v; }

__device__ __forceinline__ void split2(float v, __half& hi, __half& lo) {
  v = clamp_f16(v);
  hi = __float2half_rn(v);
  lo = __float2half_rn(v - __half2float(hi));
}

// power of two that brings a maximum magnitude `mx` into [2^14, 2^15); 0 for an all-zero or non-finite line
__device__ __forceinline__ int scale_exp(float mx) {
  if (!(mx > 0.f) || isinf(mx)) return 0;
  int ex;
  frexpf(mx, &ex);
  int e = TARGET_EXP - ex;
  return e < -100 ? -100 : (e > 100 ? 100 : e);
}

__device__ __forceinline__ float block_max(float v) {
  __shared__ float sm[32];
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sm[w] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (lane < nw) ? sm[lane] : 0.f;
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  return v;   // valid in every thread
}

// hpow[k] = 2^floor(log2 sqrt(H_kk)) (1 for a dead channel)
__global__ void hpow_kernel(const float* hdiag, float* __restrict__ hpow, int64_t n) {
  grid_begin();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float h = hdiag[k];
  int e = 0;
  if (h > 0.f && !isinf(h)) {
    int q;
    frexpf(h, &q);                       // h = f 2^q, f in [0.5, 1)
    e = (q - 1) >> 1;                    // floor((q - 1) / 2)
  }
  hpow[k] = scalbnf(1.f, e);
}

// 2^shift / d for a power of two d = 2^e, |e| < 100: arithmetic on the exponent field instead of a division per entry
__device__ __forceinline__ float over_pow2(float d, int shift) {
  return __uint_as_float((uint32_t)((254 + shift) << 23) - __float_as_uint(d));
}

// Hhi + Hlo = H_kn / (d_k d_n) * 2^H_SHIFT, four columns per thread
__global__ void __launch_bounds__(NT) split_H_kernel(const float4* H, const float* hpow,
                                                     __half2* __restrict__ hi, __half2* __restrict__ lo, int64_t n,
                                                     int32_t* __restrict__ status) {
  grid_begin();
  const int64_t n4 = n / 4;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n * n4; i += (int64_t)gridDim.x * NT) {
    const int64_t k = i / n4, c4 = (i % n4) * 4;
    const float rk = over_pow2(hpow[k], H_SHIFT);
    const float4 v = H[i];
    const float4 d = *reinterpret_cast<const float4*>(hpow + c4);
    const float x0 = v.x * rk * over_pow2(d.x, 0), x1 = v.y * rk * over_pow2(d.y, 0), x2 = v.z * rk * over_pow2(d.z, 0),
                x3 = v.w * rk * over_pow2(d.w, 0);
    const int over = (fabsf(x0) > 65504.f && isfinite(x0)) + (fabsf(x1) > 65504.f && isfinite(x1)) +
                     (fabsf(x2) > 65504.f && isfinite(x2)) + (fabsf(x3) > 65504.f && isfinite(x3));
    if (over) atomicAdd(&status[ST_H_RANGE], over);
    __half h0, h1, h2, h3, l0, l1, l2, l3;
    split2(x0, h0, l0);
    split2(x1, h1, l1);
    split2(x2, h2, l2);
    split2(x3, h3, l3);
    hi[2 * i] = __halves2half2(h0, h1); hi[2 * i + 1] = __halves2half2(h2, h3);
    lo[2 * i] = __halves2half2(l0, l1); lo[2 * i + 1] = __halves2half2(l2, l3);
  }
}

// One CTA per row of `in` [rows, cols] (leading dimension ld): the row times the column scales, brought into
// range by a power of two of its own; out_scale[row] = post / that power.  KEEP float4 per thread stay in registers between
// the maximum and the split (0: the row is read again).  The scaling is a product with a power of two: exact, or rounded
// once where the result is subnormal.
// FINITE: a row with an entry that is not finite gets NaN as its scale, and with it a result of nothing but NaN.  (The dense
// product has that without help: the low part of infinity is NaN, times whatever the other operand holds.  The sparse
// one leaves out half of it.)
template <int KEEP, bool FINITE>
__device__ __forceinline__ void split_row(const float* in, int64_t ld, int64_t cols, const float* colscale, float post, int64_t row,
                                          __half2* __restrict__ hi, __half2* __restrict__ lo, float* __restrict__ out_scale) {
  const float4* src = reinterpret_cast<const float4*>(in + row * ld);
  const float4* cs4 = reinterpret_cast<const float4*>(colscale);
  const int64_t c4n = cols / 4;
  auto fetch = [&](int64_t i) {
    float4 v = src[i];
    if (colscale) { const float4 d = cs4[i]; v.x *= d.x; v.y *= d.y; v.z *= d.z; v.w *= d.w; }
    return v;
  };
  auto larger = [](float m, const float4& v) { return fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)))); };
  float4 kept[KEEP > 0 ? KEEP : 1];
  float mx = 0.f;
  if (KEEP > 0) {
#pragma unroll
    for (int u = 0; u < KEEP; ++u) {
      const int64_t i = threadIdx.x + (int64_t)u * NT;
      kept[u] = i < c4n ? fetch(i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < KEEP; ++u) mx = larger(mx, kept[u]);
  } else {
    for (int64_t i = threadIdx.x; i < c4n; i += NT) mx = larger(mx, fetch(i));
  }
  mx = block_max(mx);
  const int e = scale_exp(mx);
  const float p = scalbnf(1.f, e);
  if (!FINITE && threadIdx.x == 0) out_scale[row] = scalbnf(post, -e);
  uint2* dh = reinterpret_cast<uint2*>(hi + row * (cols / 2));
  uint2* dl = reinterpret_cast<uint2*>(lo + row * (cols / 2));
  bool odd = false;
  auto put = [&](int64_t i, const float4& v) {
    if (FINITE) odd |= !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z) && isfinite(v.w));
    __half2 h[2], l[2];
    split2(v.x * p, h[0].x, l[0].x);
    split2(v.y * p, h[0].y, l[0].y);
    split2(v.z * p, h[1].x, l[1].x);
    split2(v.w * p, h[1].y, l[1].y);
    dh[i] = *reinterpret_cast<const uint2*>(h);
    dl[i] = *reinterpret_cast<const uint2*>(l);
  };
  if (KEEP > 0) {
#pragma unroll
    for (int u = 0; u < KEEP; ++u) {
      const int64_t i = threadIdx.x + (int64_t)u * NT;
      if (i < c4n) put(i, kept[u]);
    }
  } else {
    for (int64_t i = threadIdx.x; i < c4n; i += NT) put(i, fetch(i));
  }
  if (FINITE) {
    odd = __syncthreads_or(odd) != 0;
    if (threadIdx.x == 0) out_scale[row] = odd ? __uint_as_float(0x7fc00000u) : scalbnf(post, -e);
  }
}

template <int KEEP>
__global__ void __launch_bounds__(NT) split_rows_kernel(const float* in, int64_t ld, int64_t cols, const float* colscale, float post,
                                                        __half2* __restrict__ hi, __half2* __restrict__ lo, float* __restrict__ out_scale) {
  grid_begin();
  split_row<KEEP, false>(in, ld, cols, colscale, post, blockIdx.x, hi, lo, out_scale);
}

// The activations of the fp32 forward, `tokens` rows of z.  The CTAs behind the first `tokens` split the rows of the core S as the dense
// product wants them, in turn, if *dense says that it will run: work for a core that is not 2:4, nothing otherwise.
template <int KEEP>
__global__ void __launch_bounds__(NT) split_tokens_kernel(const float* z, int64_t cols, int64_t tokens, __half2* __restrict__ hi,
                                                          __half2* __restrict__ lo, float* __restrict__ out_scale, const float* S, int64_t rows,
                                                          __half2* __restrict__ s_hi, __half2* __restrict__ s_lo, float* __restrict__ s_scale,
                                                          const int32_t* dense) {
  grid_begin();
  if ((int64_t)blockIdx.x < tokens) {
    split_row<KEEP, true>(z, cols, cols, nullptr, 1.f, blockIdx.x, hi, lo, out_scale);
    return;
  }
  if (*dense == 0) return;
  // (a warp per row instead: 4096 x 4096, 400 tokens 114 -> 132 us a forward)
  for (int64_t row = blockIdx.x - tokens; row < rows; row += gridDim.x - tokens)
    split_row<KEEP, false>(S, cols, cols, nullptr, 1.f, row, s_hi, s_lo, s_scale);
}

// A row of the 2:4 core for the sparse tensor cores: scaled by a power of two of its own as in split_rows_kernel, two of every
// four entries (those that are not zero, else whatever fills them up) as fp16 parts, their positions in the order
// that sparse_tcgen05.cu describes.  *dense becomes 1 where a group holds more than two.  One CTA per row, KEEP float4 per thread in
// registers as in split_row.  Bound by issue: 4096 x 4096, 67 MB in
// and 36 out, 28 us (31 with the positions found by branches instead of the table, 33 with two reads of a row)
// The two positions (lower in bits 0-1, higher in bits 2-3) for every pattern of entries that are not zero, four bits each
constexpr unsigned long long pick24() {
  unsigned long long table = 0;
  for (int nz = 0; nz < 16; ++nz) {
    int pos[4] = {0, 0, 0, 0}, n = 0;
    for (int k = 0; k < 4 && n < 2; ++k) if (nz >> k & 1) { pos[n] = k; ++n; }
    if (n == 0) { pos[0] = 0; pos[1] = 1; }
    if (n == 1 && pos[0] < 3) pos[1] = pos[0] + 1;
    if (n == 1 && pos[0] == 3) { pos[0] = 2; pos[1] = 3; }
    table |= (unsigned long long)(pos[0] | pos[1] << 2) << 4 * nz;
  }
  return table;
}
constexpr unsigned long long PICK24 = pick24();
template <int KEEP>
__global__ void __launch_bounds__(NT) split_core24_kernel(const float* S, int64_t cols, __half2* __restrict__ hi, __half2* __restrict__ lo,
                                                          uint16_t* __restrict__ E, float* __restrict__ scale, int32_t* dense) {
  grid_begin();
  if (__syncthreads_or(threadIdx.x == 0 && __ldcg(dense) != 0)) return;        // nobody will read it
  const int64_t row = blockIdx.x, c4n = cols / 4, k_tiles = cols / 128;
  const float4* src = reinterpret_cast<const float4*>(S + row * cols);
  float4 kept[KEEP > 0 ? KEEP : 1];
  float mx = 0.f;
  auto larger = [&](const float4& v) { mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)))); };
  if (KEEP > 0) {
#pragma unroll
    for (int u = 0; u < KEEP; ++u) {
      const int64_t i = threadIdx.x + (int64_t)u * NT;
      kept[u] = i < c4n ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < KEEP; ++u) larger(kept[u]);
  } else {
    for (int64_t i = threadIdx.x; i < c4n; i += NT) larger(src[i]);
  }
  const int e = scale_exp(block_max(mx));
  const float p = scalbnf(1.f, e);
  if (threadIdx.x == 0) scale[row] = scalbnf(1.f, -e);
  bool more = false;
  const int m0 = row & 7, hf = (row >> 3) & 1, m2 = (row >> 4) & 7;
  const int64_t mt = row >> 7;
  auto put = [&](int64_t i, const float4& x) {               // (c4n is a multiple of 32: whole warps)
    const unsigned nz = (x.x != 0.f ? 1u : 0u) | (x.y != 0.f ? 2u : 0u) | (x.z != 0.f ? 4u : 0u) | (x.w != 0.f ? 8u : 0u);
    more |= __popc(nz) > 2;
    const unsigned pos = (unsigned)(PICK24 >> (4 * nz)) & 15u, i0 = pos & 3u, i1 = pos >> 2;
    const float a = i0 == 0 ? x.x : (i0 == 1 ? x.y : x.z), b = i1 == 1 ? x.y : (i1 == 2 ? x.z : x.w);
    __half2 h, l;
    split2(a * p, h.x, l.x);
    split2(b * p, h.y, l.y);
    hi[row * (cols / 4) + i] = h;
    lo[row * (cols / 4) + i] = l;
    // four neighbouring groups are the 16 bits of one position word's half
    uint32_t nib = pos << (4 * (i & 3));
    nib |= __shfl_xor_sync(0xffffffffu, nib, 1);
    nib |= __shfl_xor_sync(0xffffffffu, nib, 2);
    if ((i & 3) == 0) {
      const int64_t kt = i >> 5;                              // 32 groups to 128 columns
      const int k2 = (int)(i >> 3) & 3, k1 = (int)(i >> 2) & 1;
      E[2 * ((mt * k_tiles + kt) * 512 + (m0 + 8 * k1 + 16 * m2) * 4 + k2) + hf] = (uint16_t)nib;
    }
  };
  if (KEEP > 0) {
#pragma unroll
    for (int u = 0; u < KEEP; ++u)
      if (threadIdx.x + (int64_t)u * NT < c4n) put(threadIdx.x + (int64_t)u * NT, kept[u]);
  } else {
    for (int64_t i = threadIdx.x; i < c4n; i += NT) put(i, src[i]);
  }
  // (one store a CTA: with one from every thread that found a group a core of nothing else took 296 us)
  if (__syncthreads_or(more) && threadIdx.x == 0) atomicOr(dense, 1);
}

__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// Four neighbouring elements of a row: one access where every row starts on a boundary of four elements (VEC)
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p) {
  return VEC ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC>
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  if (!VEC) return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// Largest magnitude of every column of a chunk X [rows, cols]: the order of the atomic maxima does not matter,
// so the result is deterministic.  Magnitudes compare like their bit patterns.  Four columns per thread, eight rows in
// flight (one element per thread and row ran at a quarter of the memory's rate: 167 us for 268 MB).
constexpr int MAX_ROWS = 64;
template <typename TIn, bool VEC>
__global__ void __launch_bounds__(NT) colabsmax_kernel(const TIn* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols,
                                                       unsigned* __restrict__ umax) {
  const int64_t col = 4 * ((int64_t)blockIdx.x * NT + threadIdx.x);
  if (col >= cols) return;
  const int64_t r0 = (int64_t)blockIdx.y * MAX_ROWS;
  const int64_t r1 = r0 + MAX_ROWS < rows ? r0 + MAX_ROWS : rows;
  float mx[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int64_t r = r0; r < r1; ++r) {
    const float4 v = load4<VEC>(X + r * ldx + col);
    const float a[4] = {fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w)};
#pragma unroll
    for (int j = 0; j < 4; ++j) mx[j] = (a[j] > mx[j] || a[j] != a[j]) ? a[j] : mx[j];           // a NaN sticks
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) atomicMax(umax + col + j, __float_as_uint(mx[j]));
}

// gscale[c] = 2^-e_c, the factor the Gram's epilogue multiplies row c and column c by
__global__ void gram_scale_kernel(const unsigned* __restrict__ umax, float* __restrict__ gscale, int64_t n) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) gscale[k] = scalbnf(1.f, -scale_exp(__uint_as_float(umax[k])));
}

// X [rows, cols] (ld ldx) -> Thi / Tlo [rows, cols] fp16: column c scaled by 2^e_c (exact, or rounded once where the result
// is subnormal) and split.  The product takes its operands contiguous along the channels, as X lies, so this is a
// streaming pass (turning the chunk around on the way ran at 0.63 of the memory's rate).  bf16 input has 8 significant
// bits: it is exact in one fp16 part, Tlo is then not written.  Four columns per thread, SPLIT_ROWS rows.
constexpr int SPLIT_ROWS = 16;
template <typename TIn, bool VEC>
__global__ void __launch_bounds__(NT) split_columns_kernel(const TIn* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols,
                                                           const unsigned* __restrict__ umax, __half* __restrict__ Thi,
                                                           __half* __restrict__ Tlo) {
  const int64_t col = 4 * ((int64_t)blockIdx.x * NT + threadIdx.x);
  if (col >= cols) return;
  const uint4 m = *reinterpret_cast<const uint4*>(umax + col);
  const float p[4] = {scalbnf(1.f, scale_exp(__uint_as_float(m.x))), scalbnf(1.f, scale_exp(__uint_as_float(m.y))),
                      scalbnf(1.f, scale_exp(__uint_as_float(m.z))), scalbnf(1.f, scale_exp(__uint_as_float(m.w)))};
  const int64_t r0 = (int64_t)blockIdx.y * SPLIT_ROWS;
  const int64_t r1 = r0 + SPLIT_ROWS < rows ? r0 + SPLIT_ROWS : rows;
#pragma unroll 4
  for (int64_t r = r0; r < r1; ++r) {
    const float4 v = load4<VEC>(X + r * ldx + col);
    __half2 h[2], l[2];
    split2(v.x * p[0], h[0].x, l[0].x);
    split2(v.y * p[1], h[0].y, l[0].y);
    split2(v.z * p[2], h[1].x, l[1].x);
    split2(v.w * p[3], h[1].y, l[1].y);
    *reinterpret_cast<uint2*>(Thi + r * cols + col) = *reinterpret_cast<const uint2*>(h);
    if (Tlo) *reinterpret_cast<uint2*>(Tlo + r * cols + col) = *reinterpret_cast<const uint2*>(l);
  }
}

// Which channels of a bf16 X are in range for a Gram without scaling: 64 channels per CTA, 128 rows at a time until each of
// them has shown a value that is large enough -- one batch as a rule, so that the kernel is over before the product beside
// it (a dependent launch) needs the answer; a channel of zeros is read to its end.  256 threads of few registers: a CTA of the
// product finds room beside one.
constexpr unsigned RANGE_BITS = (127 - 57) << 7;           // 2^-57
__global__ void __launch_bounds__(NT) gram_range_kernel(const uint16_t* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols,
                                                        float* __restrict__ in_range) {
  __shared__ unsigned big[8], nonzero[8];                  // a bit per channel
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  const int64_t col = (int64_t)blockIdx.x * 64 + 8 * tx;
  tc::grid_launch_dependents();
  if (threadIdx.x < 8) { big[threadIdx.x] = 0u; nonzero[threadIdx.x] = 0u; }
  __syncthreads();
  const bool mine = col < cols;                            // (a multiple of 8)
  bool open = mine;
  for (int64_t r0 = 0; r0 < rows; r0 += 128) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t r = r0 + ty + 32 * u;
      v[u] = open && r < rows ? __ldg(reinterpret_cast<const uint4*>(X + r * ldx + col)) : make_uint4(0u, 0u, 0u, 0u);
    }
    unsigned b = 0u, z = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const unsigned lo = w[k] & 0x7fffu, hi = (w[k] >> 16) & 0x7fffu;      // magnitudes compare like their bits
        b |= (unsigned)(lo >= RANGE_BITS) << (2 * k) | (unsigned)(hi >= RANGE_BITS) << (2 * k + 1);
        z |= (unsigned)(lo != 0u) << (2 * k) | (unsigned)(hi != 0u) << (2 * k + 1);
      }
    }
    if (b) atomicOr(&big[tx], b);
    if (z) atomicOr(&nonzero[tx], z);
    __syncthreads();
    open = mine && big[tx] != 0xffu;
    if (!__syncthreads_or(open)) break;
  }
  if (mine && ty < 8) in_range[col + ty] = ((nonzero[tx] & ~big[tx]) >> ty) & 1u ? 0.f : 1.f;
}

inline unsigned grid_for(int64_t n) {
  int64_t b = (n + NT - 1) / NT;
  return (unsigned)(b < 148 * 8 ? (b < 1 ? 1 : b) : 148 * 8);
}

}  // namespace

void launch_f16_prepare_H(armor_ctx* c, const float* H, cudaStream_t s) {
  const int64_t n = c->d_in;
  KTimer kt(c, ARMOR_KC_OPERAND_SPLIT, 8.0 * (double)n * (double)n, s);
  launch_dependent(hpow_kernel, (unsigned)((n + 255) / 256), 256, 0, s, c->hdiag, c->hpow, n);
  __half* hi = reinterpret_cast<__half*>(c->Hlo);
  launch_dependent(split_H_kernel, grid_for(n * n / 4), NT, 0, s, reinterpret_cast<const float4*>(H), c->hpow,
                                                    reinterpret_cast<__half2*>(hi), reinterpret_cast<__half2*>(hi + n * n), n, c->status);
  c->launches += 2;
}

void launch_f16_split_rows(armor_ctx* c, const float* in, int64_t ld, int64_t rows, int64_t cols, const float* colscale,
                           float post, void* hi, void* lo, float* out_scale, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_OPERAND_SPLIT, 8.0 * (double)rows * (double)cols, s);
  __half2 *h = static_cast<__half2*>(hi), *l = static_cast<__half2*>(lo);
  auto launch = [&](auto kernel) { launch_dependent(kernel, (unsigned)rows, NT, 0, s, in, ld, cols, colscale, post, h, l, out_scale); };
  // a row in registers up to 8,192 columns: one read of it instead of two (from L1 or L2)
  if (cols <= 4 * NT) launch(split_rows_kernel<1>);
  else if (cols <= 16 * NT) launch(split_rows_kernel<4>);
  else if (cols <= 32 * NT) launch(split_rows_kernel<8>);
  else launch(split_rows_kernel<0>);
  c->launches++;
}

void launch_split_tokens(armor_ctx* c, const float* z, int64_t tokens, void* hi, void* lo, float* out_scale, const float* S, void* s_hi, void* s_lo,
                         float* s_scale, const int32_t* dense, cudaStream_t s) {
  const int64_t rows = c->d_out, cols = c->d_in;
  const int64_t more = !S ? 0 : (rows < 8 * c->n_sm ? rows : 8 * c->n_sm);
  KTimer kt(c, ARMOR_KC_OPERAND_SPLIT, 8.0 * (double)tokens * (double)cols, s);
  __half2 *h = static_cast<__half2*>(hi), *l = static_cast<__half2*>(lo), *sh = static_cast<__half2*>(s_hi), *sl = static_cast<__half2*>(s_lo);
  auto launch = [&](auto kernel) {
    launch_dependent(kernel, (unsigned)(tokens + more), NT, 0, s, z, cols, tokens, h, l, out_scale, S, rows, sh, sl, s_scale, dense);
  };
  if (cols <= 4 * NT) launch(split_tokens_kernel<1>);
  else if (cols <= 16 * NT) launch(split_tokens_kernel<4>);
  else if (cols <= 32 * NT) launch(split_tokens_kernel<8>);
  else launch(split_tokens_kernel<0>);
  c->launches++;
}

void launch_split_core24(armor_ctx* c, const float* S, void* hi, void* lo, void* E, float* scale, int32_t* dense, cudaStream_t s) {
  const int64_t cols = c->d_in;
  KTimer kt(c, ARMOR_KC_OPERAND_SPLIT, 6.125 * (double)c->wn, s);
  __half2 *h = static_cast<__half2*>(hi), *l = static_cast<__half2*>(lo);
  auto launch = [&](auto kernel) { launch_dependent(kernel, (unsigned)c->d_out, NT, 0, s, S, cols, h, l, static_cast<uint16_t*>(E), scale, dense); };
  if (cols <= 4 * NT) launch(split_core24_kernel<1>);
  else if (cols <= 16 * NT) launch(split_core24_kernel<4>);
  else if (cols <= 32 * NT) launch(split_core24_kernel<8>);
  else launch(split_core24_kernel<0>);
  c->launches++;
}

float f16_H_post_scale() { return 1.f / (float)(1 << H_SHIFT); }

namespace {
template <typename TIn, bool VEC>
void stage_chunk(armor_ctx* c, const void* Xv, int64_t ldx, int64_t rows, int64_t cols, void* Thi, void* Tlo, cudaStream_t s) {
  const TIn* X = static_cast<const TIn*>(Xv);
  const unsigned gx = (unsigned)((cols / 4 + NT - 1) / NT);
  colabsmax_kernel<TIn, VEC><<<dim3(gx, (unsigned)((rows + MAX_ROWS - 1) / MAX_ROWS)), NT, 0, s>>>(X, ldx, rows, cols, c->gmax);
  split_columns_kernel<TIn, VEC><<<dim3(gx, (unsigned)((rows + SPLIT_ROWS - 1) / SPLIT_ROWS)), NT, 0, s>>>(
      X, ldx, rows, cols, c->gmax, static_cast<__half*>(Thi), static_cast<__half*>(Tlo));
}
}  // namespace

// A chunk of X [rows, cols] as fp16 parts Thi, Tlo [rows, cols] (bf16: Thi alone), cols a multiple of 32
armor_status launch_f16_gram_stage(armor_ctx* c, const void* X, int x_dtype, int64_t ldx, int64_t rows, int64_t cols,
                                   void* Thi, void* Tlo, float* gscale, cudaStream_t s) {
  if (cols % 32) return ARMOR_ERR_UNSUPPORTED;
  if (cudaMemsetAsync(c->gmax, 0, (size_t)cols * sizeof(unsigned), s) != cudaSuccess) return ARMOR_ERR_CUDA;
  // one read for the maxima, one read and one 16-bit write per part for the staged chunk
  KTimer kt(c, ARMOR_KC_GRAM_STAGING, (double)rows * (double)cols * (x_dtype == ARMOR_DTYPE_BF16 ? 6.0 : 12.0), s);
  const bool bf16 = x_dtype == ARMOR_DTYPE_BF16;
  const bool vec = ldx % 4 == 0 && reinterpret_cast<uintptr_t>(X) % (bf16 ? 8 : 16) == 0;
  if (bf16) {
    if (vec) stage_chunk<__nv_bfloat16, true>(c, X, ldx, rows, cols, Thi, nullptr, s);
    else stage_chunk<__nv_bfloat16, false>(c, X, ldx, rows, cols, Thi, nullptr, s);
  } else {
    if (vec) stage_chunk<float, true>(c, X, ldx, rows, cols, Thi, Tlo, s);
    else stage_chunk<float, false>(c, X, ldx, rows, cols, Thi, Tlo, s);
  }
  gram_scale_kernel<<<(unsigned)((cols + 255) / 256), 256, 0, s>>>(c->gmax, gscale, cols);
  c->launches += 3;
  return ARMOR_OK;
}

void launch_gram_range(armor_ctx* c, const void* X, int64_t ldx, int64_t n_rows, float* in_range, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_GRAM_STAGING, 0.0, s);
  gram_range_kernel<<<(unsigned)((c->d_in + 63) / 64), NT, 0, s>>>(static_cast<const uint16_t*>(X), ldx, n_rows, c->d_in, in_range);
  c->launches++;
}
