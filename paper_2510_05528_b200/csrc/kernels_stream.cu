// Streaming (HBM-bound) kernels over W-shaped tensors, reductions and small bookkeeping kernels.
#include <cuda_bf16.h>

#include "armor_internal.cuh"

namespace {

constexpr int NT = 256;

__device__ __forceinline__ double block_reduce_sum(double v) {
  __shared__ double sm[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sm[w] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sm[threadIdx.x] : 0.0;
  if (w == 0) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  __syncthreads();
  return v;  // valid in thread 0
}

// ---- deterministic two-stage dot product: fixed grid, fixed order --------------------------------
__global__ void __launch_bounds__(NT) dot_partial_kernel(const float4* x,
                                                         const float4* y, int64_t n4,
                                                         double* __restrict__ part) {
  grid_begin();
  double acc = 0.0;
  const int64_t stride = (int64_t)gridDim.x * NT;
  // four independent pairs of loads in flight per thread; the order of the additions is fixed by the grid
  for (int64_t i0 = (int64_t)blockIdx.x * NT + threadIdx.x; i0 < n4; i0 += 4 * stride) {
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + u * stride;
      a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < n4) { a[u] = x[i]; b[u] = y[i]; }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float s = a[u].x * b[u].x;
      s = fmaf(a[u].y, b[u].y, s);
      s = fmaf(a[u].z, b[u].z, s);
      s = fmaf(a[u].w, b[u].w, s);
      acc += (double)s;
    }
  }
  acc = block_reduce_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

__global__ void __launch_bounds__(NT) reduce_final_kernel(const double* part, int n,
                                                          double* __restrict__ out) {
  grid_begin();
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += NT) acc += part[i];
  acc = block_reduce_sum(acc);
  if (threadIdx.x == 0) *out = acc;
}

// Grid-stride loop over n elements, four a thread at a time: all four are loaded before the first is stored.  (The compiler makes
// this of a plain loop only where what is read is __restrict__, which a kernel that waits in grid_begin() may not say: left to
// it, the bf16 conversions took 59 us for 4,736 x 6,144 elements against 34, the column scales of 4,096 x 4,096 39 against 36.)
template <typename T, typename Load, typename Store>
__device__ __forceinline__ void by_fours(int64_t n, Load load, Store store) {
  const int64_t stride = (int64_t)gridDim.x * NT;
  int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x;
  for (; i + 3 * stride < n; i += 4 * stride) {
    T v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = load(i + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) store(i + u * stride, v[u]);
  }
  T v[3];
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if (i + u * stride < n) v[u] = load(i + u * stride);
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if (i + u * stride < n) store(i + u * stride, v[u]);
}

// ---- column scale: out = in * diag(h) -----------------------------------------------------------
__global__ void __launch_bounds__(NT) colscale_kernel(const float4* in, const float4* h,
                                                      float4* __restrict__ out, int64_t n4, int cols4) {
  grid_begin();
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n4; i += (int64_t)gridDim.x * NT) {
    float4 a = in[i], s = h[i % cols4];
    out[i] = make_float4(a.x * s.x, a.y * s.y, a.z * s.z, a.w * s.w);
  }
}

// (in and out may be the same array)
__global__ void __launch_bounds__(NT) scale_cols_kernel(const float* in, const float* cs, float* out, int64_t n, int64_t cols) {
  grid_begin();
  by_fours<float>(n, [&](int64_t i) { return in[i] * cs[i % cols]; }, [&](int64_t i, float v) { out[i] = v; });
}

// ---- H diagonal and diagonal blocks -------------------------------------------------------------
// (eight rows of a block per CTA: with a CTA per block the dependent loads of 16,384 elements took 33 us)
constexpr int HB_ROWS = 8;
__global__ void __launch_bounds__(NT) extract_hblocks_kernel(const float* H, float* __restrict__ hdiag,
                                                             float* __restrict__ Hjj, int64_t d_in, int db, int diag_only) {
  grid_begin();
  const int j = blockIdx.x, a0 = blockIdx.y * HB_ROWS;
#pragma unroll 4
  for (int e = threadIdx.x; e < HB_ROWS * db; e += NT) {
    const int a = a0 + e / db, b = e % db;
    if (a >= db) break;
    float v = H[(int64_t)(j * db + a) * d_in + (j * db + b)];
    if (diag_only && a != b) v = 0.f;
    Hjj[((int64_t)j * db + a) * db + b] = v;
    if (a == b) hdiag[j * db + a] = v;
  }
}

__global__ void __launch_bounds__(NT) diag_kernel(const float* H, float* __restrict__ hdiag, int64_t d_in) {
  grid_begin();
  const int64_t k = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (k < d_in) hdiag[k] = H[k * d_in + k];
}

// ---- Gamma_M = Gamma (.) M and its squared norm -------------------------------------------------
// One float4 per thread step; a mask byte covers m_group / 4 consecutive float4 (q4 = 1 or 2).
__global__ void __launch_bounds__(NT) masked_copy_kernel(const float4* gam, const uint8_t* M,
                                                         float4* __restrict__ out, int64_t n4, int q4,
                                                         double* __restrict__ part) {
  grid_begin();
  double acc = 0.0;
  const int64_t stride = (int64_t)gridDim.x * NT;
  for (int64_t g0 = (int64_t)blockIdx.x * NT + threadIdx.x; g0 < n4; g0 += 4 * stride) {
    float4 v4[4];
    unsigned m4[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t g = g0 + u * stride;
      v4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      m4[u] = 0u;
      if (g < n4) { v4[u] = gam[g]; m4[u] = (q4 == 1) ? M[g] : ((unsigned)M[g >> 1] >> (4 * (int)(g & 1))); }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t g = g0 + u * stride;
      if (g >= n4) break;
      const unsigned m = m4[u];
      float4 v = v4[u];
      v.x = (m & 1u) ? v.x : 0.f;
      v.y = (m & 2u) ? v.y : 0.f;
      v.z = (m & 4u) ? v.z : 0.f;
      v.w = (m & 8u) ? v.w : 0.f;
      out[g] = v;
      float s = v.x * v.x;
      s = fmaf(v.y, v.y, s);
      s = fmaf(v.z, v.z, s);
      s = fmaf(v.w, v.w, s);
      acc += (double)s;
    }
  }
  acc = block_reduce_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// ---- y += sign * sc[slot] * x -------------------------------------------------------------------
__global__ void __launch_bounds__(NT) axpy_slot_kernel(float4* y, const float4* x,
                                                       int64_t n4, const double* sc, int slot,
                                                       float sign) {
  grid_begin();
  const float a = sign * (float)sc[slot];
  if (a == 0.f) return;                 // a zero step (also what withheld updates look like): y stays bit for bit
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n4; i += (int64_t)gridDim.x * NT) {
    float4 u = y[i], v = x[i];
    y[i] = make_float4(fmaf(a, v.x, u.x), fmaf(a, v.y, u.y), fmaf(a, v.z, u.z), fmaf(a, v.w, u.w));
  }
}

// the same for up to three arrays that move by the same step: one launch.  The last may make an earlier step on the way
// (y += sc[slot_before] x_before first): the two moves of an array that nothing reads in between cost one read and one write of
// it less.
struct AxpyTerm { float4* y; const float4* x; float sign; int64_t n4; };
__device__ __forceinline__ float4 axpy4(float a, const float4 v, const float4 u) {
  return make_float4(fmaf(a, v.x, u.x), fmaf(a, v.y, u.y), fmaf(a, v.z, u.z), fmaf(a, v.w, u.w));
}
template <int TERMS, bool BEFORE>
__global__ void __launch_bounds__(NT) axpy_multi_slot_kernel(AxpyTerm t0, AxpyTerm t1, AxpyTerm t2, int64_t n4, const double* sc,
                                                             int slot, const float4* x_before, int slot_before) {
  grid_begin();
  const float a = (float)sc[slot], ab = BEFORE ? (float)sc[slot_before] : 0.f;
  if (a == 0.f && ab == 0.f) return;               // (a zero step: y stays bit for bit)
  const AxpyTerm t[3] = {t0, t1, t2};
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n4; i += (int64_t)gridDim.x * NT) {
    float4 u[TERMS], v[TERMS], w = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < TERMS; ++k) {
      u[k] = v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < t[k].n4) { u[k] = t[k].y[i]; v[k] = t[k].x[i]; }
    }
    if (BEFORE && i < t[TERMS - 1].n4) w = x_before[i];
#pragma unroll
    for (int k = 0; k < TERMS; ++k) {
      if (i >= t[k].n4) continue;
      const bool before = BEFORE && k == TERMS - 1 && ab != 0.f;
      if (before) u[k] = axpy4(ab, w, u[k]);
      if (a != 0.f) u[k] = axpy4(t[k].sign * a, v[k], u[k]);
      if (a != 0.f || before) t[k].y[i] = u[k];
    }
  }
}

// ---- normalisation (Section 3.2): r1 = column norms, r2 = row norms of W / r1 -------------------
constexpr int COLSUM_CHUNKS = 64;
__global__ void __launch_bounds__(NT) colsumsq_partial_kernel(const float* W, int64_t rows, int64_t cols,
                                                              double* __restrict__ part) {
  grid_begin();
  const int64_t col = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (col >= cols) return;
  const int64_t per = (rows + COLSUM_CHUNKS - 1) / COLSUM_CHUNKS;
  const int64_t r0 = blockIdx.y * per, r1 = min(rows, r0 + per);
  double acc = 0.0;
  for (int64_t r = r0; r < r1; ++r) {
    double w = W[r * cols + col];
    acc += w * w;
  }
  part[(int64_t)blockIdx.y * cols + col] = acc;
}
__global__ void __launch_bounds__(NT) colnorm_final_kernel(const double* part, int64_t cols,
                                                           float* __restrict__ r1) {
  grid_begin();
  const int64_t col = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (col >= cols) return;
  double acc = 0.0;
  for (int ch = 0; ch < COLSUM_CHUNKS; ++ch) acc += part[(int64_t)ch * cols + col];
  float r = (float)sqrt(acc);
  r1[col] = (r == 0.f) ? 1.f : r;
}
// The row norm of W / r1 to more than double the digits of fp32, without fp64 in the loop (a division in fp64 per element
// took this pass to three times its memory time): 1 / r1 as a pair of floats, product and square with their rounding errors,
// the sum as an unevaluated pair per thread, fp64 across threads.
__global__ void __launch_bounds__(NT) rownorm_scale_kernel(const float* W, const float* r1,
                                                           float* __restrict__ r2, float* __restrict__ Wbar,
                                                           int64_t cols) {
  grid_begin();
  const int64_t row = blockIdx.x;
  const float* w = W + row * cols;
  float hi = 0.f, lo = 0.f;
#pragma unroll 2
  for (int64_t c = threadIdx.x; c < cols; c += NT) {
    const float d = r1[c], x = w[c];
    const float ih = 1.f / d, il = fmaf(-d, ih, 1.f) * ih;             // 1 / d = ih + il
    const float vh = x * ih, vl = fmaf(x, ih, -vh) + x * il;           // x / d
    const float qh = vh * vh, ql = fmaf(vh, vh, -qh) + 2.f * vh * vl;  // its square
    const float s = hi + qh, bb = s - hi;
    lo += (hi - (s - bb)) + (qh - bb) + ql;
    hi = (d > 1e-30f && d < 1e30f) ? s : __int_as_float(0x7fc00000);   // (else the pair of 1 / d loses digits)
  }
  __shared__ float r2s;
  double acc = (double)hi + (double)lo;
  if (!isfinite(acc) || acc < 1e-30) {
    // out of the range in which the pairs carry their digits: every term in fp64
    acc = 0.0;
    for (int64_t c = threadIdx.x; c < cols; c += NT) {
      const double v = (double)w[c] / (double)r1[c];
      acc += v * v;
    }
  }
  acc = block_reduce_sum(acc);
  if (threadIdx.x == 0) {
    float r = (float)sqrt(acc);
    r = (r == 0.f) ? 1.f : r;
    r2[row] = r;
    r2s = r;
  }
  __syncthreads();
  const float rr = r2s;
#pragma unroll 4
  for (int64_t c = threadIdx.x; c < cols; c += NT) Wbar[row * cols + c] = (w[c] / r1[c]) / rr;
}

// ---- initialisation (Eq. init): top-n_keep of each group of MG by W^2 * H_jj ---------------------
// Position p is kept iff fewer than n_keep positions beat it; q beats p if its score is larger, or equal
// with q < p (ties keep the lower column).
// The order is the one of the scores in fp64.  Scores in fp32 (two roundings, 2^-23 relative) give the same order unless two
// of a group lie within 5e-7 of each other, are all below the range where fp32 keeps its digits, or are not finite: only
// such a group is scored again in fp64, whose instructions otherwise took this pass to three times its memory time.
template <int MG>
__global__ void __launch_bounds__(NT) init_core_kernel(const float* W, const float* hdiag,
                                                       float* __restrict__ S, uint8_t* __restrict__ M,
                                                       int64_t ngroups, int groups_per_row, int n_keep) {
  grid_begin();
  for (int64_t g = (int64_t)blockIdx.x * NT + threadIdx.x; g < ngroups; g += (int64_t)gridDim.x * NT) {
    const int64_t c0 = (g % groups_per_row) * MG;
    float wv[MG], hv[MG], sc[MG];
#pragma unroll
    for (int h = 0; h < MG / 4; ++h) {
      const float4 w = *reinterpret_cast<const float4*>(W + g * MG + 4 * h);
      const float4 d = *reinterpret_cast<const float4*>(hdiag + c0 + 4 * h);
      wv[4 * h] = w.x; wv[4 * h + 1] = w.y; wv[4 * h + 2] = w.z; wv[4 * h + 3] = w.w;
      hv[4 * h] = d.x; hv[4 * h + 1] = d.y; hv[4 * h + 2] = d.z; hv[4 * h + 3] = d.w;
    }
#pragma unroll
    for (int p = 0; p < MG; ++p) sc[p] = wv[p] * (wv[p] * hv[p]);
    bool clear = true;
#pragma unroll
    for (int p = 0; p < MG; ++p)
#pragma unroll
      for (int q = p + 1; q < MG; ++q) {
        const float big = fmaxf(fabsf(sc[p]), fabsf(sc[q]));
        clear &= big > 1e-30f && fabsf(sc[p] - sc[q]) > 5e-7f * big;     // (false for NaN and for two infinities)
      }
    unsigned m = 0;
    if (clear) {
#pragma unroll
      for (int p = 0; p < MG; ++p) {
        int beaten = 0;
#pragma unroll
        for (int q = 0; q < MG; ++q) beaten += (q != p) && sc[q] > sc[p];
        if (beaten < n_keep) m |= 1u << p;
      }
    } else {
      double sd[MG];
#pragma unroll
      for (int p = 0; p < MG; ++p) sd[p] = (double)wv[p] * (double)wv[p] * (double)hv[p];
#pragma unroll
      for (int p = 0; p < MG; ++p) {
        int beaten = 0;
#pragma unroll
        for (int q = 0; q < MG; ++q) beaten += (q != p) && (sd[q] > sd[p] || (sd[q] == sd[p] && q < p));
        if (beaten < n_keep) m |= 1u << p;
      }
    }
    M[g] = (uint8_t)m;
#pragma unroll
    for (int h = 0; h < MG / 4; ++h)
      *reinterpret_cast<float4*>(S + g * MG + 4 * h) =
          make_float4((m >> (4 * h) & 1u) ? wv[4 * h] : 0.f, (m >> (4 * h + 1) & 1u) ? wv[4 * h + 1] : 0.f,
                      (m >> (4 * h + 2) & 1u) ? wv[4 * h + 2] : 0.f, (m >> (4 * h + 3) & 1u) ? wv[4 * h + 3] : 0.f);
  }
}

__global__ void identity_blocks_kernel(float* __restrict__ A, int db) {
  grid_begin();
  const int64_t off = (int64_t)blockIdx.x * db * db;
  for (int e = threadIdx.x; e < db * db; e += blockDim.x) A[off + e] = (e / db == e % db) ? 1.f : 0.f;
}

__global__ void copy_kernel(const float4* in, float4* __restrict__ out, int64_t n4) {
  grid_begin();
  by_fours<float4>(n4, [&](int64_t i) { return in[i]; }, [&](int64_t i, const float4& v) { out[i] = v; });
}

// ---- scalars and per-iteration bookkeeping ------------------------------------------------------
__device__ __forceinline__ void start_record(armor_iter_stats* st, double loss) {
  st->loss_start = loss;
  st->chol_failed = 0;
  st->groups_changed = 0;
  st->mask_accepted = 0;
  st->delta_L_mask = 0.0;
  st->tau_B = 0.f;
  st->tau_S = 0.f;
  st->reserved = 0;
}

// advance: the iteration counter moves on first (every iteration of a call but its first).
// carry_loss: the running loss of the previous iteration becomes this iteration's starting loss, and the
// iteration's record is opened here (no loss evaluation follows)
static_assert(SC_COUNT == 32, "one scalar per lane");
__global__ void zero_scalars_kernel(double* sc, int32_t* failflag, int nflag, int carry_loss, armor_iter_stats* st_base,
                                    int64_t* it_dev, int advance) {
  grid_begin();
  const double carried = sc[SC_LOSS];
  __syncthreads();
  for (int i = threadIdx.x; i < SC_COUNT; i += blockDim.x)
    sc[i] = (carry_loss && (i == SC_L0 || i == SC_LOSS)) ? carried : 0.0;
  for (int i = threadIdx.x; i < nflag; i += blockDim.x) failflag[i] = 0;
  if (threadIdx.x == 0) {
    const int64_t it = *it_dev + advance;
    if (advance) *it_dev = it;
    if (carry_loss && st_base) start_record(st_base + it, carried);
  }
}

// Fixed-order sums by the CTA of the bookkeeping kernel (STAGE_NT threads): thread t adds entries t, t + STAGE_NT, ...
// (eight loads in flight).  The line searches hand over thousands of partial sums (four or eight per tile).
constexpr int STAGE_NT = 1024;
__device__ __forceinline__ double stage_thread_sum(const double* p, int n) {
  double v = 0.0;
  int i = threadIdx.x;
  for (; i + 7 * STAGE_NT < n; i += 8 * STAGE_NT) {
    double t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = p[i + STAGE_NT * u];
#pragma unroll
    for (int u = 0; u < 8; ++u) v += t[u];
  }
#pragma unroll 4
  for (; i < n; i += STAGE_NT) v += p[i];
  return v;
}

// One thread's part of a stage: step lengths, accept flag, running loss, the iteration's record.
__device__ __forceinline__ void stage_scalars(double* sc, armor_iter_stats* st, int stage, double psum, int nf, int32_t* status,
                                              bool poisoned) {
  if (stage == 0) {
    sc[SC_LOSS] = sc[SC_L0];
    if (st) start_record(st, sc[SC_L0]);
  } else if (stage == 1) {
    sc[SC_DEC_A] = psum;
    sc[SC_LOSS] -= psum;
    if (st) { st->loss_A = sc[SC_LOSS]; st->chol_failed += nf; }
    if (nf) atomicAdd(&status[ST_CHOL_FAILS], nf);
  } else if (stage == 2 || stage == 10) {
    if (stage == 10) {       // the A-step's share first, its decrease in sc[SC_DEC_A]
      sc[SC_LOSS] -= sc[SC_DEC_A];
      if (st) st->loss_A = sc[SC_LOSS];
    }
    const double gd = psum;
    sc[SC_GD_B] = gd;
    const double q = sc[SC_Q_B];
    const double tau = (q > 0.0 && !poisoned) ? gd / q : 0.0;
    sc[SC_TAU_B] = tau;
    sc[SC_LOSS] -= 2.0 * tau * gd - tau * tau * q;
    if (st) { st->loss_B = sc[SC_LOSS]; st->tau_B = (float)tau; st->chol_failed += nf; }
    if (nf) atomicAdd(&status[ST_CHOL_FAILS], nf);
  } else if (stage == 3 || stage == 6) {
    const double nrm = sc[SC_NRM_S], q = sc[SC_Q_S];
    double tau = (q > 0.0) ? nrm / q : 0.0;
    if (stage == 6) {  // the paper's step 1 / beta_W' (Eq. lrWprime): the move is Gamma_M / (|A^T A|_F |B H_w B^T|_F)
      const double bh = sqrt(sc[SC_BETA_A]) * sqrt(sc[SC_BETA_K]);
      tau = (bh > 0.0) ? 1.0 / bh : 0.0;
    }
    if (poisoned) tau = 0.0;
    sc[SC_TAU_S] = tau;
    sc[SC_LOSS] -= 2.0 * tau * nrm - tau * tau * q;
    if (st) { st->loss_S = sc[SC_LOSS]; st->tau_S = (float)tau; }
  } else if (stage == 4) {
    sc[SC_EHV_M] = psum;   // <Gamma, dS> = <E H_w, V>, one term per block
    const double dl = -2.0 * sc[SC_EHV_M] + sc[SC_Q_M];
    const bool acc = (dl <= 0.0) && !poisoned;
    sc[SC_DL_M] = dl;
    sc[SC_ACCEPT] = acc ? 1.0 : 0.0;
    if (acc) sc[SC_LOSS] += dl;
    if (st) { st->delta_L_mask += dl; st->mask_accepted += acc ? 1 : 0; st->loss_mask = sc[SC_LOSS]; }   // summed over the sweeps
  } else if (stage == 7) {   // A gradient step with the step of Eq. lrA: tau = 1 / (beta_A / 2)
    const double hb = sc[SC_HB_A], nrm = sc[SC_TMP0], q = sc[SC_TMP1];
    const double tau = (hb > 0.0 && !poisoned) ? 1.0 / hb : 0.0;
    sc[SC_TAU_A] = tau;
    sc[SC_DEC_A] = 2.0 * tau * nrm - tau * tau * q;   // exact decrease of the quadratic in A along Gamma
    sc[SC_LOSS] -= sc[SC_DEC_A];
    if (st) st->loss_A = sc[SC_LOSS];
  } else if (stage == 8) {   // B gradient step with the step of Eq. lrB
    const double hb = sc[SC_HB_B], gd = sc[SC_GD_B], q = sc[SC_Q_B];
    const double tau = (hb > 0.0 && !poisoned) ? 1.0 / hb : 0.0;
    sc[SC_TAU_B] = tau;
    sc[SC_LOSS] -= 2.0 * tau * gd - tau * tau * q;
    if (st) { st->loss_B = sc[SC_LOSS]; st->tau_B = (float)tau; }
  } else if (stage == 9) {   // joint Adam step: the loss was evaluated afresh from the new state
    sc[SC_LOSS] = sc[SC_L0];
    if (st) st->loss_A = st->loss_B = st->loss_S = sc[SC_LOSS];
  } else if (stage == 5) {  // sparse-core update switched off: nothing was evaluated, nothing accepted
    sc[SC_ACCEPT] = 0.0;
    sc[SC_DL_M] = 0.0;
    if (st) st->loss_mask = sc[SC_LOSS];
  }
}

// stage 0: start, 1: after A, 2: after B, 10: after A and B, 3 / 6: after S, 4: mask accept, 5: mask phase off.  One CTA of STAGE_NT threads.
// Up to two arrays of partial sums (p1, p2) are first added, in a fixed order, into the scalars slot1 / slot2: the
// reductions of the dot products that precede the stage need no launch of their own.
// All sums of a call go through one shuffle tree and one barrier; the scalars and the record thread 0 will need are on their
// way meanwhile (the kernel is nothing but latency: as a chain of separate sums it took 4 to 6 us, four times an iteration).
// Left to the last CTA of the kernel that writes the partial sums it costs more than this launch: fences, a counter and cold code, dot
// product and stage of a 256 x 256 layer 8.1 us together against 1.9 and 2.7.
// flag_a, flag_b: the flags of the A-step's and of the B-step's solves that this stage counts.
__global__ void __launch_bounds__(STAGE_NT)
stage_kernel(double* sc_g, armor_iter_stats* st_base, const int64_t* it_dev, int stage, const int32_t* flag_a, int n_flag_a,
             const int32_t* flag_b, int n_flag_b, const double* partA, int nA, int32_t* status, const double* p1, int n1, int slot1,
             const double* p2, int n2, int slot2) {
  grid_begin();
  __shared__ double sc[SC_COUNT];
  __shared__ double sums[3][STAGE_NT / 32];
  __shared__ int flags[STAGE_NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double mine = threadIdx.x < SC_COUNT ? sc_g[threadIdx.x] : 0.0;
  armor_iter_stats* st = nullptr;
  bool poisoned = false;                  // unusable inputs: every step length is zero, nothing is accepted
  if (threadIdx.x == 0) {
    if (st_base) st = st_base + *it_dev;
    poisoned = status[ST_POISON] != 0;
  }
  double v[3] = {0.0, 0.0, 0.0};
  int nf = 0;
  if (p1) v[0] = stage_thread_sum(p1, n1);
  if (p2) v[1] = stage_thread_sum(p2, n2);
  if (partA) v[2] = stage_thread_sum(partA, nA);
  for (int i = threadIdx.x; i < n_flag_a; i += STAGE_NT) nf += flag_a[i] ? 1 : 0;
  for (int i = threadIdx.x; i < n_flag_b; i += STAGE_NT) nf += flag_b[i] ? 1 : 0;
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    nf += __shfl_xor_sync(0xffffffffu, nf, o);
  }
  if (threadIdx.x < SC_COUNT) sc[threadIdx.x] = mine;
  if (lane == 0) { sums[0][warp] = v[0]; sums[1][warp] = v[1]; sums[2][warp] = v[2]; flags[warp] = nf; }
  __syncthreads();
  if (warp != 0) return;
  v[0] = sums[0][lane]; v[1] = sums[1][lane]; v[2] = sums[2][lane]; nf = flags[lane];
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    nf += __shfl_xor_sync(0xffffffffu, nf, o);
  }
  if (lane == 0) {
    if (p1) sc[slot1] = v[0];
    if (p2) sc[slot2] = v[1];
    stage_scalars(sc, st, stage, v[2], nf, status, poisoned);
  }
  __syncwarp();
  sc_g[lane] = sc[lane];                  // SC_COUNT == 32
}

// ---- input screening -----------------------------------------------------------------------------
__device__ __forceinline__ int bad4(const float4 v) {
  return (isfinite(v.x) ? 0 : 1) + (isfinite(v.y) ? 0 : 1) + (isfinite(v.z) ? 0 : 1) + (isfinite(v.w) ? 0 : 1);
}
__global__ void __launch_bounds__(NT) screen_count_kernel(const float4* W, int64_t wn4,
                                                          const float4* H, int64_t hn4,
                                                          const float* Hs, int64_t d_in,
                                                          int32_t* __restrict__ scr) {
  grid_begin();
  int bw = 0, bh = 0, neg = 0, zero = 0;
  const int64_t stride = (int64_t)gridDim.x * NT, i0 = (int64_t)blockIdx.x * NT + threadIdx.x;
  for (int64_t i = i0; i < wn4; i += stride) bw += bad4(W[i]);
  for (int64_t i = i0; i < hn4; i += stride) bh += bad4(H[i]);
  for (int64_t i = i0; i < d_in; i += stride) {
    const float d = Hs[i * d_in + i];
    neg += (d < 0.f) ? 1 : 0;
    zero += (d == 0.f) ? 1 : 0;
  }
  for (int o = 16; o > 0; o >>= 1) {
    bw += __shfl_xor_sync(0xffffffffu, bw, o); bh += __shfl_xor_sync(0xffffffffu, bh, o);
    neg += __shfl_xor_sync(0xffffffffu, neg, o); zero += __shfl_xor_sync(0xffffffffu, zero, o);
  }
  if ((threadIdx.x & 31) == 0) {        // integer sums: the order does not matter
    if (bw) atomicAdd(&scr[0], bw);
    if (bh) atomicAdd(&scr[1], bh);
    if (neg) atomicAdd(&scr[2], neg);
    if (zero) atomicAdd(&scr[3], zero);
  }
}
__global__ void screen_final_kernel(const int32_t* scr, int32_t* status) {
  grid_begin();
  status[ST_NONFINITE_W] += scr[0];
  status[ST_NONFINITE_H] += scr[1];
  status[ST_NEG_DIAG_H] += scr[2];
  status[ST_DEAD_CHANNELS] = scr[3];
  const bool bad = scr[0] || scr[1] || scr[2];
  status[ST_POISON] = bad ? 1 : 0;
  if (bad) status[ST_LAST_ERR] = ARMOR_ERR_INVALID_ARG;
}

// ---- operand split for the three-pass tensor-core mode ------------------------------------------
__global__ void __launch_bounds__(NT) split_hilo_kernel(const float4* in, float4* __restrict__ hi,
                                                        float4* __restrict__ lo, int64_t n4) {
  grid_begin();
  by_fours<float4>(n4, [&](int64_t i) { return in[i]; }, [&](int64_t i, const float4& v) {
    float4 h;
    h.x = __uint_as_float(__float_as_uint(v.x) & 0xffffe000u);
    h.y = __uint_as_float(__float_as_uint(v.y) & 0xffffe000u);
    h.z = __uint_as_float(__float_as_uint(v.z) & 0xffffe000u);
    h.w = __uint_as_float(__float_as_uint(v.w) & 0xffffe000u);
    if (hi) hi[i] = h;
    lo[i] = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
  });
}

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// X [rows, cols] (ld ldx) -> Thi/Tlo [cols, rows] (ld ldt): transposed and split.  bf16 input is exact in
// tf32, so its low part is zero and Tlo is not needed.
template <typename TIn>
__global__ void transpose_split_kernel(const TIn* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols,
                                       float* __restrict__ Thi, float* __restrict__ Tlo, int64_t ldt) {
  __shared__ float tile[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32, r0 = (int64_t)blockIdx.y * 32;
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    int64_t r = r0 + j, cidx = c0 + threadIdx.x;
    tile[j][threadIdx.x] = (r < rows && cidx < cols) ? to_f32(X[r * ldx + cidx]) : 0.f;
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    int64_t cidx = c0 + j, r = r0 + threadIdx.x;
    if (cidx < cols && r < ldt) {
      float v = tile[threadIdx.x][j];
      float h = __uint_as_float(__float_as_uint(v) & 0xffffe000u);
      Thi[cidx * ldt + r] = h;
      if (Tlo) Tlo[cidx * ldt + r] = v - h;
    }
  }
}

// bf16 <-> fp32 with an optional per-column scale (the denormalisation of the deployment form)
__global__ void __launch_bounds__(NT) bf16_to_f32_kernel(const __nv_bfloat16* in,
                                                         const float* cs, float* __restrict__ out,
                                                         int64_t n, int64_t cols) {
  grid_begin();
  by_fours<float>(n, [&](int64_t i) { return cs ? __bfloat162float(in[i]) * cs[i % cols] : __bfloat162float(in[i]); },
                  [&](int64_t i, float v) { out[i] = v; });
}
__global__ void __launch_bounds__(NT) f32_to_bf16_kernel(const float* in, const float* cs,
                                                         __nv_bfloat16* __restrict__ out, int64_t n, int64_t cols) {
  grid_begin();
  by_fours<float>(n, [&](int64_t i) { return cs ? in[i] * cs[i % cols] : in[i]; },
                  [&](int64_t i, float v) { out[i] = __float2bfloat16_rn(v); });
}

// H[r][c] = H[c][r] for c > r: the upper triangle from the lower one, 64 x 64 tiles through shared memory, 16 bytes an access
// (VEC: rows start on 16-byte boundaries and n is a multiple of 4); a CTA per tile on or below the diagonal.
// LEFT_OUT: H is the Gram of a bf16 X [n_rows][ldx] whose product left out the channels with in_range 0: their entries are added
// first, a warp per entry, in fp64 (a channel of values below 2^-57 throughout: time does not count).  Eight CTAs per SM in
// either form: with five, the 409 MB of 10,112 channels took 12 us more.
constexpr int MIR = 64;
template <bool VEC, bool LEFT_OUT>
__global__ void __launch_bounds__(NT, 8) mirror_lower_kernel(float* H, int64_t n, const __nv_bfloat16* __restrict__ X, int64_t ldx,
                                                          int64_t n_rows, const float* __restrict__ in_range) {
  // blockIdx.x counts the tiles (i, j), j <= i, of the lower triangle row by row
  int i = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((int64_t)(i + 1) * (i + 2) / 2 <= (int64_t)blockIdx.x) ++i;
  while ((int64_t)i * (i + 1) / 2 > (int64_t)blockIdx.x) --i;
  const int j = (int)((int64_t)blockIdx.x - (int64_t)i * (i + 1) / 2);
  __shared__ float tile[MIR][MIR + 1];
  const int64_t r0 = (int64_t)i * MIR, c0 = (int64_t)j * MIR;            // source tile
  const int q = threadIdx.x & 15, w = threadIdx.x >> 4;
  float4 v[4];
  auto fetch = [&]() {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t r = r0 + w + 16 * k, c = c0 + 4 * q;
      v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r >= n) continue;
      if (VEC) { if (c < n) v[k] = *reinterpret_cast<const float4*>(H + r * n + c); }
      else {
        float* f = &v[k].x;
        for (int t = 0; t < 4; ++t) if (c + t < n) f[t] = H[r * n + c + t];
      }
    }
  };
  fetch();
  if (LEFT_OUT) {
    const int64_t k = (threadIdx.x < MIR ? r0 : c0 - MIR) + threadIdx.x;
    if (__syncthreads_or(threadIdx.x < 2 * MIR && k < n && in_range[k] == 0.f)) {
      const int lane = threadIdx.x & 31;
      for (int e = threadIdx.x >> 5; e < MIR * MIR; e += NT / 32) {
        const int64_t r = r0 + e / MIR, c = c0 + e % MIR;
        if (r >= n || c > r || (in_range[r] != 0.f && in_range[c] != 0.f)) continue;
        double acc = 0.0;
        for (int64_t t = lane; t < n_rows; t += 32)
          acc += (double)__bfloat162float(X[t * ldx + r]) * (double)__bfloat162float(X[t * ldx + c]);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) H[r * n + c] = (float)((double)H[r * n + c] + acc);
      }
      __syncthreads();
      fetch();
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float* t = &tile[w + 16 * k][4 * q];
    t[0] = v[k].x; t[1] = v[k].y; t[2] = v[k].z; t[3] = v[k].w;
  }
  __syncthreads();
  // row c0 + w + 16 k of the upper triangle, columns r0 + 4 q ..
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t r = c0 + w + 16 * k, c = r0 + 4 * q;
    if (r >= n) continue;
    const float f[4] = {tile[4 * q][w + 16 * k], tile[4 * q + 1][w + 16 * k], tile[4 * q + 2][w + 16 * k], tile[4 * q + 3][w + 16 * k]};
    if (VEC && i != j) {
      if (c < n) *reinterpret_cast<float4*>(H + r * n + c) = make_float4(f[0], f[1], f[2], f[3]);
    } else {
      for (int t = 0; t < 4; ++t)
        if (c + t < n && c + t > r) H[r * n + c + t] = f[t];
    }
  }
}

// part[b] = weight * || X_b ||_F for block b of db x db floats (the terms of beta_A and beta_B, Eq. lrA / lrB)
__global__ void __launch_bounds__(NT) block_fro_kernel(const float4* X, int n4_per_block,
                                                       const float* hdiag, int db, int nbi,
                                                       double* __restrict__ part) {
  grid_begin();
  const float4* xb = X + (int64_t)blockIdx.x * n4_per_block;
  double acc = 0.0;
  for (int i = threadIdx.x; i < n4_per_block; i += NT) {
    const float4 v = xb[i];
    float s = v.x * v.x;
    s = fmaf(v.y, v.y, s);
    s = fmaf(v.z, v.z, s);
    s = fmaf(v.w, v.w, s);
    acc += (double)s;
  }
  acc = block_reduce_sum(acc);
  double wsum = 0.0;
  if (hdiag) {
    const float* h = hdiag + (int64_t)(blockIdx.x % nbi) * db;
    for (int k = threadIdx.x; k < db; k += NT) wsum += (double)h[k] * (double)h[k];
    wsum = block_reduce_sum(wsum);
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sqrt(acc) * (hdiag ? sqrt(wsum) : 1.0);
}

// ---- Adam (Kingma & Ba, Algorithm 1, with bias correction) ----------------------------------------------
__global__ void __launch_bounds__(NT) adam_kernel(float4* theta, const float4* gamma,
                                                  float4* m, float4* v, int64_t n4,
                                                  const uint8_t* M, int q4, float lr, float b1, float b2,
                                                  float eps, int64_t step_base, const int64_t* it_dev,
                                                  const int32_t* status) {
  grid_begin();
  if (status[ST_POISON] != 0) return;   // unusable inputs: parameters and moments stay as they are
  // bias corrections 1 / (1 - beta^step), step = step_base + the iteration counter: once per block
  __shared__ float s_bc[2];
  if (threadIdx.x == 0) {
    const double step = (double)(step_base + *it_dev);
    s_bc[0] = (float)(1.0 / (1.0 - pow((double)b1, step)));
    s_bc[1] = (float)(1.0 / (1.0 - pow((double)b2, step)));
  }
  __syncthreads();
  const float inv_bc1 = s_bc[0], inv_bc2 = s_bc[1];
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < n4; i += (int64_t)gridDim.x * NT) {
    const float4 ga = gamma[i];
    float4 mm = m[i], vv = v[i], th = theta[i];
    unsigned keep = 0xFu;
    if (M) keep = (q4 == 1) ? M[i] : ((unsigned)M[i >> 1] >> (4 * (int)(i & 1)));
    const float g[4] = {-2.f * ga.x, -2.f * ga.y, -2.f * ga.z, -2.f * ga.w};
    float mo[4] = {mm.x, mm.y, mm.z, mm.w}, vo[4] = {vv.x, vv.y, vv.z, vv.w}, t[4] = {th.x, th.y, th.z, th.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float gk = ((keep >> k) & 1u) ? g[k] : 0.f;      // the core's gradient is masked
      mo[k] = fmaf(b1, mo[k], (1.f - b1) * gk);
      vo[k] = fmaf(b2, vo[k], (1.f - b2) * gk * gk);
      const float upd = lr * (mo[k] * inv_bc1) / (sqrtf(vo[k] * inv_bc2) + eps);
      t[k] = ((keep >> k) & 1u) ? t[k] - upd : 0.f;
    }
    m[i] = make_float4(mo[0], mo[1], mo[2], mo[3]);
    v[i] = make_float4(vo[0], vo[1], vo[2], vo[3]);
    theta[i] = make_float4(t[0], t[1], t[2], t[3]);
  }
}

inline int grid_for(int64_t n) {
  int64_t b = (n + NT - 1) / NT;
  return (int)(b < 1 ? 1 : (b > 148 * 16 ? 148 * 16 : b));
}

}  // namespace

void dot_to_ptr(armor_ctx* c, const float* x, const float* y, int64_t n, double* out, cudaStream_t s) {
  KTimer kt(c, n >= (1 << 22) ? ARMOR_KC_DOT : ARMOR_KC_SMALL, 8.0 * (double)n, s);
  launch_dependent(dot_partial_kernel, ARMOR_DOT_BLOCKS, NT, 0, s, (const float4*)x, (const float4*)y, n / 4, c->partials);
  launch_dependent(reduce_final_kernel, 1, NT, 0, s, c->partials, ARMOR_DOT_BLOCKS, out);
  c->launches += 2;
}

// partial sums of <x, y> only (ARMOR_DOT_BLOCKS entries at `part`); the consumer adds them up
void dot_partials(armor_ctx* c, const float* x, const float* y, int64_t n, double* part, cudaStream_t s) {
  KTimer kt(c, n >= (1 << 22) ? ARMOR_KC_DOT : ARMOR_KC_SMALL, 8.0 * (double)n, s);
  launch_dependent(dot_partial_kernel, ARMOR_DOT_BLOCKS, NT, 0, s, (const float4*)x, (const float4*)y, n / 4, part);
  c->launches++;
}

void reduce_partials_to(armor_ctx* c, const double* part, int n, double* out, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(reduce_final_kernel, 1, NT, 0, s, part, n, out);
  c->launches++;
}

void launch_colscale(armor_ctx* c, const float* in, const float* h, float* out, int64_t rows, int64_t cols,
                     cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_AXPY, 8.0 * (double)rows * (double)cols, s);
  launch_dependent(colscale_kernel, grid_for(rows * cols / 4), NT, 0, s, (const float4*)in, (const float4*)h, (float4*)out,
                                                          rows * cols / 4, (int)(cols / 4));
  c->launches++;
}

void launch_scale_cols(armor_ctx* c, const float* in, const float* colscale, float* out, int64_t rows, int64_t cols, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_FORWARD, 8.0 * (double)rows * (double)cols, s);
  launch_dependent(scale_cols_kernel, grid_for(rows * cols), NT, 0, s, in, colscale, out, rows * cols, cols);
  c->launches++;
}

void launch_extract_hblocks(armor_ctx* c, const float* H, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(extract_hblocks_kernel, dim3(c->nbi, (c->db + HB_ROWS - 1) / HB_ROWS), NT, 0, s, H, c->hdiag, c->Hjj, c->d_in, c->db,
                   c->cfg.h_mode == ARMOR_H_DIAG);
  c->launches++;
}

void launch_masked_copy(armor_ctx* c, const float* Gam, const uint8_t* M, float* out, double* part, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_MASKED_COPY, (8.0 + 1.0 / c->cfg.m_group) * (double)c->wn, s);
  launch_dependent(masked_copy_kernel, ARMOR_DOT_BLOCKS, NT, 0, s, (const float4*)Gam, M, (float4*)out, c->wn / 4,
                                                    c->cfg.m_group / 4, part);
  c->launches++;
}

void launch_axpy_slot(armor_ctx* c, float* y, const float* x, int64_t n, int slot, float sign, cudaStream_t s) {
  KTimer kt(c, n >= (1 << 22) ? ARMOR_KC_AXPY : ARMOR_KC_SMALL, 12.0 * (double)n, s);
  launch_dependent(axpy_slot_kernel, grid_for(n / 4), NT, 0, s, (float4*)y, (const float4*)x, n / 4, c->sc, slot, sign);
  c->launches++;
}

// y_k += sign_k * sc[slot] * x_k for up to three pairs of lengths n_k (a pair with y == nullptr is skipped); with x2_before the
// third, which then exists beside at least one other, takes y2 += sc[slot_before] * x2_before first
void launch_axpy_multi(armor_ctx* c, float* y0, const float* x0, float s0, int64_t n0, float* y1, const float* x1, float s1,
                       int64_t n1, float* y2, const float* x2, float s2, int64_t n2, int slot, cudaStream_t s,
                       const float* x2_before, int slot_before) {
  AxpyTerm t[3];
  int k = 0;
  if (y0) t[k++] = {(float4*)y0, (const float4*)x0, s0, n0 / 4};
  if (y1) t[k++] = {(float4*)y1, (const float4*)x1, s1, n1 / 4};
  if (y2) t[k++] = {(float4*)y2, (const float4*)x2, s2, n2 / 4};
  if (k == 0) return;
  int64_t n4 = 0;
  double elems = 0.0;
  for (int j = 0; j < k; ++j) { n4 = t[j].n4 > n4 ? t[j].n4 : n4; elems += 4.0 * (double)t[j].n4; }
  for (int j = k; j < 3; ++j) t[j] = t[0];
  KTimer kt(c, n4 >= (1 << 20) ? ARMOR_KC_AXPY : ARMOR_KC_SMALL, 12.0 * elems + (x2_before ? 4.0 * (double)n2 : 0.0), s);
  const float4* xb = reinterpret_cast<const float4*>(x2_before);
  if (xb && k == 3) launch_dependent(axpy_multi_slot_kernel<3, true>, grid_for(n4), NT, 0, s, t[0], t[1], t[2], n4, c->sc, slot, xb, slot_before);
  else if (xb) launch_dependent(axpy_multi_slot_kernel<2, true>, grid_for(n4), NT, 0, s, t[0], t[1], t[2], n4, c->sc, slot, xb, slot_before);
  else if (k == 3) launch_dependent(axpy_multi_slot_kernel<3, false>, grid_for(n4), NT, 0, s, t[0], t[1], t[2], n4, c->sc, slot, xb, slot_before);
  else if (k == 2) launch_dependent(axpy_multi_slot_kernel<2, false>, grid_for(n4), NT, 0, s, t[0], t[1], t[2], n4, c->sc, slot, xb, slot_before);
  else launch_dependent(axpy_multi_slot_kernel<1, false>, grid_for(n4), NT, 0, s, t[0], t[1], t[2], n4, c->sc, slot, xb, slot_before);
  c->launches++;
}

void launch_init(armor_ctx* c, const float* W, const float* H, float* Wbar, float* r1, float* r2, float* A, float* B,
                 float* S, uint8_t* M, cudaStream_t s) {
  const int64_t rows = c->d_out, cols = c->d_in;
  // W read (twice more with the normalisation), Wbar, S and the mask bytes written
  KTimer kt(c, ARMOR_KC_INIT, (double)c->wn * (c->cfg.normalize ? 20.0 : 12.0 + (Wbar != W ? 4.0 : 0.0)) +
                                  (double)c->wn / c->cfg.m_group, s);
  if (c->cfg.normalize) {
    double* part = c->colpart;
    dim3 g1((unsigned)((cols + NT - 1) / NT), COLSUM_CHUNKS);
    launch_dependent(colsumsq_partial_kernel, g1, NT, 0, s, W, rows, cols, part);
    launch_dependent(colnorm_final_kernel, (unsigned)((cols + NT - 1) / NT), NT, 0, s, part, cols, r1);
    launch_dependent(rownorm_scale_kernel, (unsigned)rows, NT, 0, s, W, r1, r2, Wbar, cols);
    c->launches += 3;
  } else if (Wbar != W) {
    launch_dependent(copy_kernel, grid_for(c->wn / 4), NT, 0, s, (const float4*)W, (float4*)Wbar, c->wn / 4);
    c->launches++;
  }
  const int mg = c->cfg.m_group;
  launch_dependent(diag_kernel, (unsigned)((cols + NT - 1) / NT), NT, 0, s, H, c->hdiag, cols);
  if (mg == 8)
    launch_dependent(init_core_kernel<8>, grid_for(c->wn / 8), NT, 0, s, Wbar, c->hdiag, S, M, c->wn / 8, (int)(cols / 8),
                                                          c->cfg.n_keep);
  else
    launch_dependent(init_core_kernel<4>, grid_for(c->wn / 4), NT, 0, s, Wbar, c->hdiag, S, M, c->wn / 4, (int)(cols / 4),
                                                          c->cfg.n_keep);
  launch_dependent(identity_blocks_kernel, c->nbo, NT, 0, s, A, c->db);
  launch_dependent(identity_blocks_kernel, c->nbi, NT, 0, s, B, c->db);
  c->launches += 4;
}

armor_status launch_screen_inputs(armor_ctx* c, const float* W, const float* H, cudaStream_t s) {
  if (cudaMemsetAsync(c->screen, 0, 4 * sizeof(int32_t), s) != cudaSuccess) return ARMOR_ERR_CUDA;
  const int64_t wn4 = c->wn / 4, hn4 = c->d_in * c->d_in / 4;
  KTimer kt(c, ARMOR_KC_INIT, 4.0 * ((double)c->wn + (double)c->d_in * (double)c->d_in), s);
  launch_dependent(screen_count_kernel, grid_for(wn4 > hn4 ? wn4 : hn4), NT, 0, s, reinterpret_cast<const float4*>(W), wn4,
                                                                     reinterpret_cast<const float4*>(H), hn4, H, c->d_in,
                                                                     c->screen);
  launch_dependent(screen_final_kernel, 1, 1, 0, s, c->screen, c->status);
  c->launches += 2;
  return ARMOR_OK;
}

void launch_zero_scalars(armor_ctx* c, bool advance, bool carry_loss, armor_iter_stats* st, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(zero_scalars_kernel, 1, NT, 0, s, c->sc, c->failflag, 2 * (c->nbo > c->nbi ? c->nbo : c->nbi), carry_loss ? 1 : 0, st,
                   c->it_dev, advance ? 1 : 0);
  c->launches++;
}

void launch_stage(armor_ctx* c, armor_iter_stats* st, int stage, const double* part, int npart, cudaStream_t s, const double* p1, int n1,
                  int slot1, const double* p2, int n2, int slot2) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  const int32_t* flag_b = c->failflag + (c->nbo > c->nbi ? c->nbo : c->nbi);
  launch_dependent(stage_kernel, 1, STAGE_NT, 0, s, c->sc, st, c->it_dev, stage, c->failflag, stage == 1 || stage == 10 ? c->nbo : 0, flag_b,
                   stage == 2 || stage == 10 ? c->nbi : 0, part, npart, c->status, p1, n1, slot1, p2, n2, slot2);
  c->launches++;
}

void launch_split_hilo(armor_ctx* c, const float* in, float* hi, float* lo, int64_t n, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_OPERAND_SPLIT, 8.0 * (double)n, s);
  launch_dependent(split_hilo_kernel, grid_for(n / 4), NT, 0, s, (const float4*)in, (float4*)hi, (float4*)lo, n / 4);
  c->launches++;
}

void launch_transpose_split(armor_ctx* c, const void* X, int x_dtype, int64_t ldx, int64_t rows, int64_t cols,
                            float* Thi, float* Tlo, int64_t ldt, cudaStream_t s) {
  dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((ldt + 31) / 32));
  KTimer kt(c, ARMOR_KC_GRAM_STAGING, (double)rows * (double)cols * (x_dtype == ARMOR_DTYPE_BF16 ? 6.0 : (Tlo ? 12.0 : 8.0)), s);
  if (x_dtype == ARMOR_DTYPE_BF16)
    transpose_split_kernel<<<grid, dim3(32, 8), 0, s>>>(static_cast<const __nv_bfloat16*>(X), ldx, rows, cols, Thi,
                                                       (float*)nullptr, ldt);
  else
    transpose_split_kernel<<<grid, dim3(32, 8), 0, s>>>(static_cast<const float*>(X), ldx, rows, cols, Thi, Tlo, ldt);
  c->launches++;
}

void launch_mirror_lower(armor_ctx* c, float* H, int64_t n, cudaStream_t s, const void* X_bf16, int64_t ldx, int64_t n_rows,
                         const float* in_range) {
  const int64_t t = (n + MIR - 1) / MIR;
  const unsigned tiles = (unsigned)(t * (t + 1) / 2);
  const __nv_bfloat16* X = static_cast<const __nv_bfloat16*>(X_bf16);
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  const bool vec = n % 4 == 0 && reinterpret_cast<uintptr_t>(H) % 16 == 0;
  if (in_range) {
    if (vec) mirror_lower_kernel<true, true><<<tiles, NT, 0, s>>>(H, n, X, ldx, n_rows, in_range);
    else mirror_lower_kernel<false, true><<<tiles, NT, 0, s>>>(H, n, X, ldx, n_rows, in_range);
  } else {
    if (vec) mirror_lower_kernel<true, false><<<tiles, NT, 0, s>>>(H, n, nullptr, 0, 0, nullptr);
    else mirror_lower_kernel<false, false><<<tiles, NT, 0, s>>>(H, n, nullptr, 0, 0, nullptr);
  }
  c->launches++;
}

void launch_block_fro_sum(armor_ctx* c, const float* X, int nblk, const float* hdiag, double* out, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(block_fro_kernel, nblk, NT, 0, s, (const float4*)X, c->db * c->db / 4, hdiag, c->db, c->nbi, c->quadpart);
  launch_dependent(reduce_final_kernel, 1, NT, 0, s, c->quadpart, nblk, out);
  c->launches += 2;
}

void launch_adam(armor_ctx* c, float* theta, const float* gamma, float* m, float* v, int64_t n, const uint8_t* M,
                 int64_t step_base, cudaStream_t s) {
  const float lr = c->cfg.adam_lr > 0.f ? c->cfg.adam_lr : 1e-4f;
  const float b1 = c->cfg.adam_beta1 > 0.f ? c->cfg.adam_beta1 : 0.9f;
  const float b2 = c->cfg.adam_beta2 > 0.f ? c->cfg.adam_beta2 : 0.999f;
  const float eps = c->cfg.adam_eps > 0.f ? c->cfg.adam_eps : 1e-8f;
  KTimer kt(c, n >= (1 << 22) ? ARMOR_KC_AXPY : ARMOR_KC_SMALL, 28.0 * (double)n, s);
  launch_dependent(adam_kernel, grid_for(n / 4), NT, 0, s, (float4*)theta, (const float4*)gamma, (float4*)m, (float4*)v, n / 4, M,
                                            c->cfg.m_group / 4, lr, b1, b2, eps, step_base, c->it_dev, c->status);
  c->launches++;
}

void launch_bf16_to_f32(armor_ctx* c, const void* in, const float* colscale, float* out, int64_t rows, int64_t cols,
                        cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_FORWARD, 6.0 * (double)rows * (double)cols, s);
  launch_dependent(bf16_to_f32_kernel, grid_for(rows * cols), NT, 0, s, static_cast<const __nv_bfloat16*>(in), colscale, out,
                                                         rows * cols, cols);
  c->launches++;
}

void launch_f32_to_bf16(armor_ctx* c, const float* in, const float* colscale, void* out, int64_t rows, int64_t cols,
                        cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_FORWARD, 6.0 * (double)rows * (double)cols, s);
  launch_dependent(f32_to_bf16_kernel, grid_for(rows * cols), NT, 0, s, in, colscale, static_cast<__nv_bfloat16*>(out), rows * cols,
                                                         cols);
  c->launches++;
}
