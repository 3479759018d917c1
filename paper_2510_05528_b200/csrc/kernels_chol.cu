// Per-block SPD solves for the wrapper updates.  The block systems are the zeros of the paper's
// gradients with respect to A and B (Appendix D.1 and D.2) made proximal by a relative ridge:
//   mode 0 (A update): X = Gamma (G + lam I)^-1;  A += X;  dA = X;  part = <Gamma, X> + lam |X|^2
//   mode 1 (left)    : out = (G + lam I)^-1 rhs
//   mode 2 (right+gd): out = rhs (G + lam I)^-1;  part = <dotw, out>
// A failed factorisation leaves A unchanged / writes zeros and raises failflag[block].
//
// One CTA factorises one d_block x d_block matrix in shared memory and solves for a slice of the right-hand sides beside it;
// the slices of a block repeat the factorisation.  What bounds this is the chain of pivots (130 to 190 cycles each in the
// factorisation, 70 in a solve), what shared memory returns to the small products (a 16-byte broadcast costs four cycles), and
// fetching instructions: a launch meets its code cold, about 100 cycles a line of eight, so the loops stay rolled.  fp64
// conversions cost as much as dozens of fp32 instructions and are kept out of the sums:
//   storage: panels of 32 columns, rows of 32 floats, the 16-byte units of a row swizzled so that eight lanes reading the
//            same unit of consecutive rows, or of every fourth row, or all units of one row, meet no bank conflict; G
//            arrives by cp.async, and everything below reads four columns per access.
//   factor : blocked left-looking Cholesky.  A panel receives the contributions of the earlier panels as one small product
//            (fp32 over 32 terms, panels added as unevaluated pairs of floats, one rounding), then eliminate_panel.
//   solve  : left-looking with the same two-level sums, see solve_block.
// Measured and left: pivots eight at a time with every thread factorising the 8 x 8 block (elimination 2 x slower), rows
// or right-hand sides moving down one register per pivot in a rolled loop (3 x and 1.4 x); two CTAs per SM with fewer right-hand
// sides each (40 blocks: 59 us a launch against 52).
// A launch, d_block 128: 32 blocks over 4 CTAs each 46.5 us (62.2 with the panel's elimination unrolled and a row a thread in the last
// panels' updates), 40 blocks over 2 to 4 CTAs 50.6 (65.1), 112 and 32 blocks 59.4 on average (74.4); d_block 32, 8 blocks 16 k cycles
// (22 k); d_block 256 (chol_ctas_per_block), 40 and 56 blocks 240 us (312 with a CTA per slice), 112 blocks of a 28672 x 8192 layer 630 (956).
#include "armor_internal.cuh"

namespace {

constexpr int NT = 256;
constexpr int NB = 32;       // panel width

struct PanelMap {
  int db;
  // offset (floats) of panel kb: rows NB*kb .. db-1, NB floats each
  __device__ __forceinline__ int off(int kb) const { return NB * (kb * db - NB * kb * (kb - 1) / 2); }
};
// 16-byte unit u (columns 4u .. 4u + 3) of row r of a panel
__device__ __forceinline__ int unit(int r, int u) { return r * NB + 4 * (u ^ (((r >> 2) ^ (r << 1)) & 7)); }
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__host__ __device__ inline size_t panel_floats(int db) {
  const int np = db / NB;
  return (size_t)NB * ((size_t)np * db - (size_t)NB * np * (np - 1) / 2);
}

// running sum of fp32 values as an unevaluated pair: every rounding error of an addition is kept (Knuth's two-sum)
struct Pair { float hi, lo; };
__device__ __forceinline__ void pair_add(Pair& a, float v) {
  const float s = a.hi + v, bb = s - a.hi;
  a.lo += (a.hi - (s - bb)) + (v - bb);
  a.hi = s;
}
// v - a, rounded once
__device__ __forceinline__ float pair_sub_from(float v, const Pair& a) {
  const float s = v - a.hi, bb = s - v;
  return s + (((v - (s - bb)) - (a.hi + bb)) - a.lo);
}

// The panel's 32 columns, eliminated right-looking, eight at a time.  Warp 0 holds the eight columns of the diagonal block in
// registers (lane = row) and takes the pivots; behind a barrier warp w > 0 does the same to the 32 rows below it that it owns
// (group w - 1 of `below`), with the factors and reciprocals that warp 0 has left, and every warp brings the panel's later
// columns of its rows up to date.  An element meets the pivots in ascending order, one fused multiply-add each.  Rolled over
// the four groups of eight and over the columns behind them, because what bounded this was fetching instructions: with all 32
// columns in registers and 32 pivots unrolled (30 KB of code) a launch's first panel took 31 k cycles and the others 5.5 k.
__device__ __forceinline__ void later_columns(float* P, int row, int c0, const float (&l)[8]) {
#pragma unroll 1
  for (int u = c0 / 4 + 2; u < NB / 4; ++u) {
    float4* dst = reinterpret_cast<float4*>(P + unit(row, u));
    const float4 v = *dst;
    float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 a = ld4(P + unit(4 * u + q, c0 / 4)), b = ld4(P + unit(4 * u + q, c0 / 4 + 1));
      const float m[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int k = 0; k < 8; ++k) w[q] = fmaf(-l[k], m[k], w[q]);
    }
    *dst = make_float4(w[0], w[1], w[2], w[3]);
  }
}
__device__ __noinline__ void eliminate_panel(float* P, float* invd, int below, int* s_fail) {
  __shared__ float s_inv[NB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = NB * warp + lane;
  bool bad = false;
  float dg = 1.f;
#pragma unroll 1
  for (int c0 = 0; c0 < NB; c0 += 8) {
    float l[8];
    if (warp <= below) {
      const float4 a = ld4(P + unit(row, c0 / 4)), b = ld4(P + unit(row, c0 / 4 + 1));
      l[0] = a.x; l[1] = a.y; l[2] = a.z; l[3] = a.w; l[4] = b.x; l[5] = b.y; l[6] = b.z; l[7] = b.w;
    }
    if (warp == 0) {
      float akk = __shfl_sync(0xffffffffu, l[0], c0);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        bad |= !(akk > 0.f) | !isfinite(akk);
        // 1 / sqrt(a): hardware estimate refined by one Newton step
        float inv = rsqrtf(akk);
        inv = inv * fmaf(-0.5f * akk * inv, inv, 1.5f);
        const float ld = l[k] * inv;
        l[k] = ld;
        if (lane == c0 + k) { dg = ld; s_inv[lane] = inv; }
        // the next pivot needs lane k + 1's own multiplier only: it goes ahead of the rest of the column
        if (k < 7) akk = __shfl_sync(0xffffffffu, fmaf(-ld, ld, l[k + 1]), c0 + k + 1);
#pragma unroll
        for (int j = k + 1; j < 8; ++j) l[j] = fmaf(-ld, __shfl_sync(0xffffffffu, ld, c0 + j), l[j]);
      }
      *reinterpret_cast<float4*>(P + unit(row, c0 / 4)) = make_float4(l[0], l[1], l[2], l[3]);
      *reinterpret_cast<float4*>(P + unit(row, c0 / 4 + 1)) = make_float4(l[4], l[5], l[6], l[7]);
    }
    __syncthreads();
    if (warp > 0 && warp <= below) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        l[k] *= s_inv[c0 + k];
#pragma unroll
        for (int j = k + 1; j < 8; ++j) l[j] = fmaf(-l[k], P[unit(c0 + j, (c0 + k) / 4) + (k & 3)], l[j]);
      }
      *reinterpret_cast<float4*>(P + unit(row, c0 / 4)) = make_float4(l[0], l[1], l[2], l[3]);
      *reinterpret_cast<float4*>(P + unit(row, c0 / 4 + 1)) = make_float4(l[4], l[5], l[6], l[7]);
    }
    if (warp <= below) later_columns(P, row, c0, l);
    __syncwarp();
  }
  if (warp == 0) {
    if (bad) { if (lane == 0) *s_fail = 1; }
    else invd[lane] = 1.f / dg;
  }
  __syncthreads();
}

// panel kb (at P, first row c0) -= sum_{p < c0} L(i, p) L(k, p): 4 x 4 elements per thread, rows TR*tr.., columns 4*tc..  (Also
// where that leaves most warps without a tile: with one row a thread the panels of 64 and 32 rows of a block of 128 took 6.3 and
// 4.7 k cycles, what shared memory needs to return five 16-byte accesses per 16 multiply-adds.)
__device__ __forceinline__ void update_panel(float* Lp, const PanelMap& pm, int kb) {
  constexpr int TR = 4;
  const int db = pm.db, c0 = NB * kb;
  float* P = Lp + pm.off(kb);
  const int ntiles = ((db - c0) / TR) * (NB / 4);
  for (int tix = threadIdx.x; tix < ntiles; tix += NT) {
    const int tr = tix / (NB / 4), tc = tix % (NB / 4);
    Pair acc[TR][4];
#pragma unroll
    for (int a = 0; a < TR; ++a)
#pragma unroll
      for (int bb = 0; bb < 4; ++bb) acc[a][bb] = {0.f, 0.f};
    for (int pb = 0; pb < kb; ++pb) {
      const float* Q = Lp + pm.off(pb);
      const int ri = c0 - NB * pb + TR * tr, rk = c0 - NB * pb + 4 * tc;      // rows of panel pb
      float a32[TR][4];
#pragma unroll
      for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) a32[a][bb] = 0.f;
#pragma unroll 2
      for (int u = 0; u < NB / 4; ++u) {
        float4 li[TR], lk[4];
#pragma unroll
        for (int a = 0; a < TR; ++a) li[a] = ld4(Q + unit(ri + a, u));
#pragma unroll
        for (int a = 0; a < 4; ++a) lk[a] = ld4(Q + unit(rk + a, u));
#pragma unroll
        for (int a = 0; a < TR; ++a)
#pragma unroll
          for (int bb = 0; bb < 4; ++bb) {
            a32[a][bb] = fmaf(li[a].x, lk[bb].x, a32[a][bb]);
            a32[a][bb] = fmaf(li[a].y, lk[bb].y, a32[a][bb]);
            a32[a][bb] = fmaf(li[a].z, lk[bb].z, a32[a][bb]);
            a32[a][bb] = fmaf(li[a].w, lk[bb].w, a32[a][bb]);
          }
      }
#pragma unroll
      for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) pair_add(acc[a][bb], a32[a][bb]);
    }
#pragma unroll
    for (int a = 0; a < TR; ++a) {
      float4* dst = reinterpret_cast<float4*>(P + unit(TR * tr + a, tc));
      const float4 v = *dst;
      *dst = make_float4(pair_sub_from(v.x, acc[a][0]), pair_sub_from(v.y, acc[a][1]), pair_sub_from(v.z, acc[a][2]),
                         pair_sub_from(v.w, acc[a][3]));
    }
  }
}

// Block kb's 32 unknowns of every right-hand side: x (in X, one column per right-hand side) becomes L^-1 x, or with T L^-T x.
// First the solved blocks' share (forward: blocks before kb with the rows of L; T: blocks after kb with its columns; in block
// order either way): lane = right-hand side (G of them, 32 apart), warp = four rows.  Then the block itself.  G 1: lane = unknown,
// a warp takes four right-hand sides side by side and hands every solution round by a shuffle, without a barrier in the
// chain of 32.  More right-hand sides: lanes and warps as before, four unknowns at a time with a barrier behind them (32 and
// more shuffles an unknown cost more: 12 and 20 k cycles a CTA of 64 and 128 right-hand sides against 10.6 and 17.7, while 32 take
// 16.9 against 18.5).  Called by the whole CTA.
template <bool T, int G>
__device__ __forceinline__ void solve_block(const float* Lp, const PanelMap& pm, const float* invd, float* X, int ldx, int kb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r0 = 4 * warp;
  const int p_begin = T ? kb + 1 : 0, p_end = T ? pm.db / NB : kb;
  float* own = X + (NB * kb + r0) * ldx + lane;
  float y[G][4];
  {
    Pair acc[G][4];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[g][m] = {0.f, 0.f};
#pragma unroll 1
    for (int pb = p_begin; pb < p_end; ++pb) {
      const float* Q = Lp + pm.off(T ? kb : pb);
      const float* xp = X + NB * pb * ldx + lane;
      float a32[G][4];
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int m = 0; m < 4; ++m) a32[g][m] = 0.f;
#pragma unroll (G == 1 ? 4 : 2)
      for (int u = 0; u < NB / 4; ++u) {
        float l[4][4];                                        // [row][unknown 4 u + j]
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float4 v = ld4(T ? Q + unit(NB * (pb - kb) + 4 * u + t, warp) : Q + unit(NB * (kb - pb) + r0 + t, u));
          if (T) { l[0][t] = v.x; l[1][t] = v.y; l[2][t] = v.z; l[3][t] = v.w; }
          else { l[t][0] = v.x; l[t][1] = v.y; l[t][2] = v.z; l[t][3] = v.w; }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float x = xp[(4 * u + j) * ldx + 32 * g];
#pragma unroll
            for (int m = 0; m < 4; ++m) a32[g][m] = fmaf(l[m][j], x, a32[g][m]);
          }
      }
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int m = 0; m < 4; ++m) pair_add(acc[g][m], a32[g][m]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int m = 0; m < 4; ++m) y[g][m] = pair_sub_from(own[m * ldx + 32 * g], acc[g][m]);
  }
  const float* D = Lp + pm.off(kb);
  if constexpr (G == 1) {
    if (p_begin < p_end) {
#pragma unroll
      for (int m = 0; m < 4; ++m) own[m * ldx] = y[0][m];
      __syncthreads();
    }
    float* x0 = X + (NB * kb + lane) * ldx + 4 * warp;
    const float iv = invd[NB * kb + lane];
    float z[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = x0[i];
#pragma unroll 1
    for (int s = 0; s < NB / 4; ++s) {
      const int u = T ? NB / 4 - 1 - s : s;
      float l[4];                                               // what unknown 4 u + j contributes to this lane's
      if (T) {
#pragma unroll
        for (int j = 0; j < 4; ++j) l[j] = D[unit(4 * u + j, lane >> 2) + (lane & 3)];
      } else {
        const float4 v = ld4(D + unit(lane, u));
        l[0] = v.x; l[1] = v.y; l[2] = v.z; l[3] = v.w;
      }
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const int j = T ? 3 - jj : jj, k = 4 * u + j;
        const bool open = T ? lane < k : lane > k;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = __shfl_sync(0xffffffffu, z[i] * iv, k);
          if (open) z[i] = fmaf(-l[j], x, z[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) x0[i] = z[i] * iv;
    __syncthreads();
    return;
  }
#pragma unroll 1
  for (int s = 0; s < NB / 4; ++s) {
    const int u = T ? NB / 4 - 1 - s : s;                     // the warp whose four rows are solved now
    const bool open = T ? warp <= u : warp >= u;
    float l[4][4];                                            // [row of this warp][unknown 4 u + j]
    if (open) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float4 v = ld4(T ? D + unit(4 * u + t, warp) : D + unit(r0 + t, u));
        if (T) { l[0][t] = v.x; l[1][t] = v.y; l[2][t] = v.z; l[3][t] = v.w; }
        else { l[t][0] = v.x; l[t][1] = v.y; l[t][2] = v.z; l[t][3] = v.w; }
      }
    }
    if (warp == u) {
      const float4 iv4 = ld4(invd + NB * kb + r0);
      const float iv[4] = {iv4.x, iv4.y, iv4.z, iv4.w};
#pragma unroll
      for (int g = 0; g < G; ++g) {
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = T ? 3 - jj : jj;
          y[g][j] *= iv[j];
#pragma unroll
          for (int m = 0; m < 4; ++m)
            if (T ? m < j : m > j) y[g][m] = fmaf(-l[m][j], y[g][j], y[g][m]);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) own[m * ldx + 32 * g] = y[g][m];
      }
    }
    __syncthreads();
    if (open && warp != u) {
      const float* xu = X + (NB * kb + 4 * u) * ldx + lane;
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = T ? 3 - jj : jj;
          const float x = xu[j * ldx + 32 * g];
#pragma unroll
          for (int m = 0; m < 4; ++m) y[g][m] = fmaf(-l[m][j], x, y[g][m]);
        }
    }
  }
}

constexpr int MAX_DB = 256;

// G: a CTA takes 32 G right-hand sides at a time; SLICES: several times (a loop round a single slice costs 5 % of a launch)
template <int G, bool SLICES>
__global__ void __launch_bounds__(NT, 1)
chol_blocked_kernel(int mode, const float* Gmat, const float* rhs, float* __restrict__ out,
                    const float* dotw, float* A, float ridge, int db, double* __restrict__ part,
                    int32_t* __restrict__ failflag, int32_t* status) {
  grid_begin();
  constexpr int W = 32 * G, LDX = W + 1;                // (odd: neither a row of X nor 8 x 4 floats along a column conflict)
  extern __shared__ __align__(16) float smem[];
  const PanelMap pm{db};
  const int np = db / NB;
  float* Lp = smem;
  float* X = smem + panel_floats(db);                   // [unknown][right-hand side]
  __shared__ __align__(16) float invd[MAX_DB];          // reciprocals of the factor's diagonal
  __shared__ double red[NT / 32];
  __shared__ int s_fail;
  __shared__ double s_lam;
  const int b = blockIdx.x, tid = threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t off = (int64_t)b * db * db;
  const bool right = (mode != 1);
  const int slices = (db + W - 1) / W;                  // of the block's right-hand sides; this CTA takes every gridDim.y-th
  const int q4 = db / 4;                                // 16-byte units per row

  // ---- load: the units of G on and below the diagonal, then the right-hand sides
  for (int e = tid; e < db * q4; e += NT) {
    const int r = e / q4, u = e % q4, kb = u / (NB / 4);
    if (4 * u > r) continue;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Lp + pm.off(kb) + unit(r - NB * kb, u - kb * (NB / 4)));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Gmat + off + 4 * (int64_t)e) : "memory");
  }
  // A right solve's right-hand side is a row of rhs (eight lanes along it, four rows per warp access), a left solve's a
  // column (lanes along the row of rhs).  Right-hand sides past the end are zeros.
  auto load_rhs = [&](int v0) {
    if (right) {
#pragma unroll 4
      for (int e = tid; e < W * q4; e += NT) {
        const int c8 = e & 7, v = (e >> 3) % W, i = 4 * (c8 + 8 * ((e >> 3) / W));
        const float4 x = v0 + v < db ? ld4(rhs + off + (int64_t)(v0 + v) * db + i) : make_float4(0.f, 0.f, 0.f, 0.f);
        X[i * LDX + v] = x.x; X[(i + 1) * LDX + v] = x.y; X[(i + 2) * LDX + v] = x.z; X[(i + 3) * LDX + v] = x.w;
      }
    } else {
#pragma unroll 8
      for (int e = tid; e < W * db; e += NT) {
        const int v = e % W, i = e / W;
        X[i * LDX + v] = v0 + v < db ? rhs[off + (int64_t)i * db + v0 + v] : 0.f;
      }
    }
  };
  load_rhs((int)blockIdx.y * W);
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (tid == 0) s_fail = 0;
  __syncthreads();
  if (tid < 32) {
    double tr = 0.0;
    for (int kb = 0; kb < np; ++kb) tr += (double)Lp[pm.off(kb) + unit(tid, tid >> 2) + (tid & 3)];
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (tid == 0) s_lam = (double)ridge * tr / (double)db;
  }
  __syncthreads();
  const double lam = s_lam;
  for (int i = tid; i < db; i += NT) {
    float* d = Lp + pm.off(i / NB) + unit(i % NB, (i % NB) >> 2) + (i & 3);
    *d = (float)((double)*d + lam);
  }
  __syncthreads();

  // ---- blocked Cholesky
  for (int kb = 0; kb < np; ++kb) {
    if (kb > 0) {
      update_panel(Lp, pm, kb);
      __syncthreads();
    }
    eliminate_panel(Lp + pm.off(kb), invd + NB * kb, np - 1 - kb, &s_fail);
    if (s_fail) break;
  }
  const bool fail = (s_fail != 0);
  const bool hold = (mode == 0) && status[ST_POISON] != 0;   // unusable inputs: the A-step is withheld (X = 0)

  int q = blockIdx.y;
  do {
  const int v0 = q * W;                                 // first right-hand side of the slice
  if (SLICES && q != (int)blockIdx.y) {                 // (the first one has come with the factor)
    __syncthreads();
    load_rhs(v0);
    __syncthreads();
  }
  if (!fail) {
    // ---- forward substitution  L y = r, then backward substitution  L^T x = y
    for (int kb = 0; kb < np; ++kb) solve_block<false, G>(Lp, pm, invd, X, LDX, kb);
    for (int kb = np - 1; kb >= 0; --kb) solve_block<true, G>(Lp, pm, invd, X, LDX, kb);
    __syncthreads();
  }

  // ---- write back.  Right solves: right-hand side vid is row vid of the result; left solves: column vid.
  double acc = 0.0;
  if (right) {
    // (four at a time, all loads ahead of the first store: A is read and written)
    constexpr int U = 4;
    for (int e0 = tid; e0 < W * q4; e0 += U * NT) {
      float4 aold[U], gin[U];
      int64_t idx[U];
      int cell[U];                                      // first of its four unknowns in X, -1: nothing there
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * NT, c8 = e & 7, v = (e >> 3) % W, i = 4 * (c8 + 8 * ((e >> 3) / W));
        cell[u] = e < W * q4 && v0 + v < db ? i * LDX + v : -1;
        idx[u] = off + (int64_t)(v0 + v) * db + i;
        aold[u] = gin[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cell[u] < 0) continue;
        if (mode == 0) aold[u] = ld4(A + idx[u]);
        gin[u] = ld4((mode == 0 ? rhs : dotw) + idx[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (cell[u] < 0) continue;
        const float* xs = X + cell[u];
        const float4 g = gin[u], a = aold[u];
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!fail && !hold) x = make_float4(xs[0], xs[LDX], xs[2 * LDX], xs[3 * LDX]);
        *reinterpret_cast<float4*>(out + idx[u]) = x;
        if (mode == 0) {
          *reinterpret_cast<float4*>(A + idx[u]) = make_float4(a.x + x.x, a.y + x.y, a.z + x.z, a.w + x.w);
          acc += (double)g.x * (double)x.x + lam * (double)x.x * (double)x.x;
          acc += (double)g.y * (double)x.y + lam * (double)x.y * (double)x.y;
          acc += (double)g.z * (double)x.z + lam * (double)x.z * (double)x.z;
          acc += (double)g.w * (double)x.w + lam * (double)x.w * (double)x.w;
        } else {
          acc += (double)g.x * (double)x.x + (double)g.y * (double)x.y + (double)g.z * (double)x.z + (double)g.w * (double)x.w;
        }
      }
    }
  } else {
#pragma unroll 4
    for (int e = tid; e < W * db; e += NT) {
      const int v = e % W, i = e / W;
      if (v0 + v < db) out[off + (int64_t)i * db + v0 + v] = fail ? 0.f : X[i * LDX + v];
    }
  }
  if (mode != 1) {
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int wp = 0; wp < NT / 32; ++wp) t += red[wp];
      part[(int64_t)b * slices + q] = t;
    }
  }
  q += gridDim.y;
  } while (SLICES && q < slices);
  if (tid == 0 && blockIdx.y == 0 && fail) {
    failflag[b] = 1;
    atomicCAS(&status[ST_FIRST_FAIL], 0, b + 1);
  }
}

// Unblocked variant for block sizes that are not a multiple of 32: thread i owns row i.
__global__ void chol_kernel(int mode, const float* Gmat, const float* rhs,
                            float* __restrict__ out, const float* dotw, float* A,
                            float ridge, int db, double* __restrict__ part,
                            int32_t* __restrict__ failflag, int32_t* status) {
  grid_begin();
  extern __shared__ float smem[];
  const int ld = db + 1;
  float* L = smem;
  float* Rs = smem + (size_t)db * ld;
  __shared__ double red[8];
  __shared__ float s_diag;
  __shared__ int s_fail;
  __shared__ double s_lam;
  const int b = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const int64_t off = (int64_t)b * db * db;
  const bool right = (mode != 1);
  for (int e = tid; e < db * db; e += nt) {
    const int r = e / db, cidx = e % db;
    L[r * ld + cidx] = Gmat[off + e];
    const float v = rhs[off + e];
    if (right) Rs[cidx * ld + r] = v; else Rs[r * ld + cidx] = v;
  }
  if (tid == 0) s_fail = 0;
  __syncthreads();
  if (tid == 0) {
    double tr = 0.0;
    for (int i = 0; i < db; ++i) tr += (double)L[i * ld + i];
    s_lam = (double)ridge * tr / (double)db;
  }
  __syncthreads();
  const double lam = s_lam;
  if (tid < db) L[tid * ld + tid] = (float)((double)L[tid * ld + tid] + lam);
  __syncthreads();

  const int i = tid;
  for (int k = 0; k < db; ++k) {
    double s = 0.0;
    if (i >= k && i < db) {
      s = (double)L[i * ld + k];
      for (int p = 0; p < k; ++p) s -= (double)L[i * ld + p] * (double)L[k * ld + p];
      if (i == k) {
        if (!(s > 0.0) || !isfinite(s)) s_fail = 1; else s_diag = (float)sqrt(s);
      }
    }
    __syncthreads();
    if (s_fail) break;
    if (i >= k && i < db) L[i * ld + k] = (i == k) ? s_diag : (float)(s / (double)s_diag);
    __syncthreads();
  }
  const bool fail = (s_fail != 0);
  const bool hold = (mode == 0) && status[ST_POISON] != 0;   // unusable inputs: the A-step is withheld (X = 0)

  double acc = 0.0;
  if (!fail) {
    const int cidx = tid;
    if (cidx < db) {
      for (int r = 0; r < db; ++r) {
        double s = (double)Rs[r * ld + cidx];
        for (int p = 0; p < r; ++p) s -= (double)L[r * ld + p] * (double)Rs[p * ld + cidx];
        Rs[r * ld + cidx] = (float)(s / (double)L[r * ld + r]);
      }
      for (int r = db - 1; r >= 0; --r) {
        double s = (double)Rs[r * ld + cidx];
        for (int p = r + 1; p < db; ++p) s -= (double)L[p * ld + r] * (double)Rs[p * ld + cidx];
        Rs[r * ld + cidx] = (float)(s / (double)L[r * ld + r]);
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < db * db; e += nt) {
    const int r = e / db, cidx = e % db;
    float x = 0.f;
    if (!fail && !hold) x = right ? Rs[cidx * ld + r] : Rs[r * ld + cidx];
    if (mode == 0) {
      const float a = A[off + e] + x;
      A[off + e] = a;
      out[off + e] = x;
      acc += (double)rhs[off + e] * (double)x + lam * (double)x * (double)x;
    } else {
      out[off + e] = x;
      if (mode == 2) acc += (double)dotw[off + e] * (double)x;
    }
  }
  if (mode != 1) {
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < (nt + 31) / 32; ++w) t += red[w];
      part[b] = t;
    }
  }
  if (tid == 0 && fail) {
    failflag[b] = 1;
    atomicCAS(&status[ST_FIRST_FAIL], 0, b + 1);
  }
}

}  // namespace

namespace {

// right-hand sides per CTA in units of 32: as few as still give one wave of CTAs (d_block > 128: what fits beside the factor)
int chol_groups(int db, int nb) {
  if (db > 128) return 2;
  for (int g = 1; g < 4; g *= 2)
    if ((int64_t)nb * ((db + 32 * g - 1) / (32 * g)) <= 148 || 32 * g >= db) return g;
  return 4;
}

// CTAs per block, each of which factorises it and then solves for its share of the block's slices of right-hand sides.  A
// block of up to 128 has a CTA for each slice.  One of 256 fills an SM's shared memory, so that 56 or 112 blocks in four slices came in
// two and four waves that each repeated the factorisation: the number of CTAs with the shortest chain of waves, a factorisation
// counted as FACTOR_SLICES slices.
constexpr double FACTOR_SLICES = 0.8;
int chol_ctas_per_block(int db, int nb, int n_sm, int slices) {
  if (db <= 128) return slices;
  int best = slices;
  double least = 0.0;
  for (int y = slices; y >= 1; --y) {
    const int waves = (nb * y + n_sm - 1) / n_sm;
    const double t = waves * (FACTOR_SLICES + (slices + y - 1) / y);
    if (y == slices || t < least) { least = t; best = y; }
  }
  return best;
}

// the A-step's flags, the B-step's
int32_t* chol_flags(armor_ctx* c, int mode) { return c->failflag + (mode == 0 ? 0 : (c->nbo > c->nbi ? c->nbo : c->nbi)); }

template <int G, bool SLICES = false>
armor_status launch_blocked(armor_ctx* c, int mode, const float* Gm, const float* rhs, float* out, const float* dotw, float* A,
                            int nb, double* part, cudaStream_t s) {
  const int db = c->db, slices = (db + 32 * G - 1) / (32 * G);
  const size_t smem = (panel_floats(db) + (size_t)db * (32 * G + 1)) * sizeof(float);
  const int widest = G == 2 ? MAX_DB : 128;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, chol_blocked_kernel<G, SLICES>,
                          (panel_floats(widest) + (size_t)widest * (32 * G + 1)) * sizeof(float)) != ARMOR_OK)
    return ARMOR_ERR_CUDA;
  launch_dependent(chol_blocked_kernel<G, SLICES>, dim3(nb, chol_ctas_per_block(db, nb, c->n_sm, slices)), NT, smem, s, mode, Gm, rhs, out, dotw, A,
                   c->cfg.ridge, db, part, chol_flags(c, mode), c->status);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

}  // namespace

// The right-hand sides of one block come in this many slices (at most four), with a partial sum each.
int chol_parts_per_block(int db, int nb) {
  if (db % NB) return 1;
  const int w = 32 * chol_groups(db, nb);
  return (db + w - 1) / w;
}

armor_status launch_chol(armor_ctx* c, int mode, const float* Gmat, const float* rhs, float* out, const float* dotw,
                         float* A, int nb, double* part, cudaStream_t s) {
  const int db = c->db;
  KTimer kt(c, ARMOR_KC_CHOLESKY, (double)nb * (7.0 / 3.0) * (double)db * (double)db * (double)db, s);   // flops
  if (db % NB == 0) {
    const int g = chol_groups(db, nb);
    if (g == 1) return launch_blocked<1>(c, mode, Gmat, rhs, out, dotw, A, nb, part, s);
    if (db > 128) return launch_blocked<2, true>(c, mode, Gmat, rhs, out, dotw, A, nb, part, s);
    if (g == 2) return launch_blocked<2>(c, mode, Gmat, rhs, out, dotw, A, nb, part, s);
    return launch_blocked<4>(c, mode, Gmat, rhs, out, dotw, A, nb, part, s);
  }
  const size_t smem = 2 * (size_t)db * (db + 1) * sizeof(float);
  static PerDeviceOnce attr_set;
  if (ensure_dynamic_smem(attr_set, c->device, chol_kernel, 2 * 128 * 129 * 4) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int nt = ((db + 31) / 32) * 32;
  launch_dependent(chol_kernel, nb, nt < 64 ? 64 : nt, smem, s, mode, Gmat, rhs, out, dotw, A, c->cfg.ridge, db, part,
                                                 chol_flags(c, mode), c->status);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

namespace {

__global__ void identity_rhs_kernel(float* X, int db) {
  grid_begin();
  float* Xb = X + (int64_t)blockIdx.x * db * db;
  for (int e = threadIdx.x; e < db * db; e += blockDim.x) Xb[e] = (e / db == e % db) ? 1.f : 0.f;
}

__global__ void save_flags_kernel(const int32_t* failflag, int32_t* __restrict__ saved, int n) {
  grid_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) saved[i] = failflag[i];
}

// DELTA_PARTS CTAs per block: Delta_j = 0 and failflag[j] = 1 where the inverse does not exist; partial sums of
// <dotw_j, Delta_j>
__global__ void __launch_bounds__(NT) delta_finish_kernel(float* Delta, const float* dotw,
                                                          const int32_t* hinv_fail,
                                                          int32_t* __restrict__ failflag, double* __restrict__ part,
                                                          int db) {
  grid_begin();
  const int j = blockIdx.x / DELTA_PARTS, q = blockIdx.x % DELTA_PARTS;
  const int64_t off = (int64_t)j * db * db;
  const int n4 = db * db / 4, e1 = n4 * (q + 1) / DELTA_PARTS;
  const bool bad = hinv_fail[j] != 0;
  double acc = 0.0;
  const int e0 = n4 * q / DELTA_PARTS + threadIdx.x;
  float4* d = reinterpret_cast<float4*>(Delta + off);
  if (bad) {
    for (int e = e0; e < e1; e += NT) d[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
#pragma unroll 4
    for (int e = e0; e < e1; e += NT) {
      const float4 w = *(reinterpret_cast<const float4*>(dotw + off) + e), v = d[e];
      acc += (double)w.x * (double)v.x + (double)w.y * (double)v.y + (double)w.z * (double)v.z + (double)w.w * (double)v.w;
    }
  }
  __shared__ double red[NT / 32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < NT / 32; ++w) t += red[w];
    part[blockIdx.x] = t;
    if (bad) failflag[j] = 1;
  }
}

}  // namespace

armor_status launch_hjj_inverse(armor_ctx* c, cudaStream_t s) {
  const int nbi = c->nbi;
  if (cudaMemsetAsync(chol_flags(c, 1), 0, (size_t)nbi * sizeof(int32_t), s) != cudaSuccess) return ARMOR_ERR_CUDA;
  {
    KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
    launch_dependent(identity_rhs_kernel, nbi, NT, 0, s, c->Ktmp, c->db);
    c->launches++;
  }
  armor_status st = launch_chol(c, 1, c->Hjj, c->Ktmp, c->Hinv, nullptr, nullptr, nbi, nullptr, s);
  if (st != ARMOR_OK) return st;
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(save_flags_kernel, (nbi + 255) / 256, 256, 0, s, chol_flags(c, 1), c->hinv_fail, nbi);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

void launch_delta_finish(armor_ctx* c, float* Delta, const float* dotw, double* part, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_SMALL, 0.0, s);
  launch_dependent(delta_finish_kernel, DELTA_PARTS * c->nbi, NT, 0, s, Delta, dotw, c->hinv_fail, chol_flags(c, 1), part, c->db);
  c->launches++;
}

