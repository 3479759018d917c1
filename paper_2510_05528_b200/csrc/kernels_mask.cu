// Greedy sparse-core update (Algorithm 3 and Appendix B.1 of the paper): every 2:4 group of every
// (i, j) block is scored by the L1 norm of the core gradient, one group per block is drawn with
// probability proportional to its score, and that group is re-solved in closed form over all six
// masks (Eq. mask_loss_opt / mask_loss_opt_sol).
#include "armor_internal.cuh"

namespace {

constexpr int NT = 256;

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// -ln(u) for u = (k + 1/2) / 2^24, k the top 24 bits of the hash.  Both branches feed the logarithm an
// argument that is exact in fp32, so the result is good to a few ulp even for u next to 1, where the
// winners of the exponential race live.
__device__ __forceinline__ float neg_log_uniform(uint32_t k24) {
  if (k24 < (1u << 23)) return -logf((float)(2u * k24 + 1u) * 2.98023223876953125e-8f);        // * 2^-25
  return -log1pf(-(float)(2u * ((1u << 24) - k24) - 1u) * 2.98023223876953125e-8f);
}

// 2x2 PSD solve with the pseudo-inverse rule: w = K^+ z, red = z^T K^+ z.
__device__ __forceinline__ void pinv2(double k11, double k12, double k22, double z1, double z2, double& w1,
                                      double& w2, double& red) {
  const double det = k11 * k22 - k12 * k12;
  if (det <= 1e-12 * k11 * k22) {
    const double tr = k11 + k22;
    if (tr <= 0.0) { w1 = w2 = 0.0; red = 0.0; return; }
    const double inv = 1.0 / (tr * tr);
    w1 = (k11 * z1 + k12 * z2) * inv;
    w2 = (k12 * z1 + k22 * z2) * inv;
  } else {
    w1 = (k22 * z1 - k12 * z2) / det;
    w2 = (k11 * z2 - k12 * z1) / det;
  }
  red = z1 * w1 + z2 * w2;
}

// n x n SPD solve (n <= NKM) by unpivoted Cholesky; false if a pivot is not positive (that mask is skipped).
template <int NKM>
__device__ __forceinline__ bool chol_small(int n, const double (&Kin)[NKM][NKM], const double (&z)[NKM],
                                           double (&w)[NKM],
                                           double& red) {
  double L[NKM][NKM];
#pragma unroll
  for (int i = 0; i < NKM; ++i) {
#pragma unroll
    for (int j = 0; j < NKM; ++j) {
      if (i >= n || j > i) continue;
      double sacc = Kin[i][j];
#pragma unroll
      for (int p = 0; p < NKM; ++p)
        if (p < j) sacc -= L[i][p] * L[j][p];
      if (i == j) {
        if (!(sacc > 0.0) || !isfinite(sacc)) return false;
        L[i][i] = sqrt(sacc);
      } else {
        L[i][j] = sacc / L[j][j];
      }
    }
  }
  double y[NKM];
#pragma unroll
  for (int i = 0; i < NKM; ++i) {
    if (i >= n) continue;
    double sacc = z[i];
#pragma unroll
    for (int p = 0; p < NKM; ++p)
      if (p < i) sacc -= L[i][p] * y[p];
    y[i] = sacc / L[i][i];
  }
#pragma unroll
  for (int i = NKM - 1; i >= 0; --i) {
    if (i >= n) continue;
    double sacc = y[i];
#pragma unroll
    for (int p = 0; p < NKM; ++p)
      if (p > i && p < n) sacc -= L[p][i] * w[p];
    w[i] = sacc / L[i][i];
  }
  red = 0.0;
#pragma unroll
  for (int i = 0; i < NKM; ++i)
    if (i < n) red += z[i] * w[i];
  return true;
}

// The group updates of one iteration change the core by dS (one group per (i, j) block) and the
// reconstruction by V = A dS B.  Block (i, j) of dS has a single non-zero row r, so
//   tr(V H_w V^T) = sum_i sum_{j, j'} (a_ij . a_ij') * (z_ij H_w[j, j'] z_ij'^T)
// with a_ij = A_i[:, r_ij] and z_ij = delta_ij^T B_j[rows of the group, :]: row-blocks decouple because A is
// block diagonal.  a and z are gathered by the CTA that has solved the group (write_vectors; a launch of its own for several draws per
// block), a batched product forms y_ij = z_ij H_w[j-th block row, :], and mask_quad_kernel sums the pairs in a fixed order.
// blk: row block bi, virtual column block v = draw * nbi + column block; by threads t0, t0 + step, .. of a CTA.
struct VectorArgs { const float* A; const float* B; float* Zsel; float* Acol; int nbo_pad; };
__device__ __forceinline__ void write_vectors(const VectorArgs& w, const SelRec& rec, int bi, int v, int nbi, int nbv, int db, int mg, int t0, int step) {
  const int rl = rec.row - bi * db, lc = (rec.cgrp % (db / mg)) * mg;
  const float* Ai = w.A + (int64_t)bi * db * db + rl;
  const float* Bj = w.B + (int64_t)(v % nbi) * db * db + (int64_t)lc * db;
#pragma unroll 4
  for (int k = t0; k < db; k += step) {
    float a = 0.f, z = 0.f;
    if (rec.valid) {
      a = Ai[(int64_t)k * db];
      for (int p = 0; p < mg; ++p) z = fmaf(rec.new_val[p] - rec.old_val[p], Bj[(int64_t)p * db + k], z);
    }
    w.Acol[((int64_t)bi * nbv + v) * db + k] = a;
    w.Zsel[((int64_t)v * w.nbo_pad + bi) * db + k] = z;
  }
}

__global__ void __launch_bounds__(NT) mask_vectors_kernel(VectorArgs w, const SelRec* sel, int db, int nbi, int mg, int nbv) {
  grid_begin();
  const int blk = blockIdx.x;
  const SelRec rec = sel[blk];
  write_vectors(w, rec, blk / nbv, blk % nbv, nbi, nbv, db, mg, threadIdx.x, NT);
}

// One CTA per (i, j) block of the core, N:M groups with M = MG (4 or 8) and N = n_keep (<= NKM: 4 for 2:4 and 4:8, 6 for 5:8 and 6:8).
// Pass 1: every group of the block is scored, keyed and the arg-min found by warp shuffles.
// Pass 2: thread b < 2^MG evaluates the mask with bit pattern b (if it keeps exactly n_keep positions);
// the best one is found in this order: larger reduction first; among equal reductions the
// incumbent, then the lexicographically first index tuple.
// PHASE 0: both passes in one launch (several draws per block).  A single draw runs as two launches, so that the
// streaming pass keeps few registers and the per-block solves, which are chains of dependent loads, all run
// side by side: PHASE 1 is pass 1 alone (the block's winner goes to best_key / best_g), PHASE 2 is pass 2
// alone (one warp per block for groups of four, 256 threads for groups of eight) and gathers the block's vectors for the guard.
template <int MG, int NKM, bool MULTI, int PHASE>
__global__ void __launch_bounds__(NT) mask_select_kernel(const float* Gam, const float* S,
                                                         const uint8_t* M, const float* alpha,
                                                         const float* Kfull, SelRec* __restrict__ sel,
                                                         double* __restrict__ part, int64_t d_in, int db, int nbi,
                                                         int n_keep, int select_mode, uint64_t seed, uint64_t t_base,
                                                         uint64_t t_mul, const int64_t* it_dev,
                                                         uint64_t n_groups_total, int kg_arg,
                                                         float* tab_key, unsigned long long* tab_g, VectorArgs vec) {
  grid_begin();
  const uint64_t t = t_base + t_mul * (uint64_t)(*it_dev);   // selection counter of this run of Algorithm 3
  const int kg = MULTI ? kg_arg : 1;                       // one draw: the loop and the key cache compile away
  const int bi = blockIdx.x / nbi, bj = blockIdx.x % nbi;
  extern __shared__ float s_keys[];         // kg > 1: the keys of the block's groups, kept for the later draws
  const int gpb = db / MG;                // groups per block row
  const int64_t ng_row = d_in / MG;       // groups per matrix row
  const int n_in_block = db * gpb;
  // kg draws: the kg smallest keys of the block, one after the other; the record of draw kk of block (i, j) is
  // entry (i, kk * nbi + j) of a [nbo][kg * nbi] table (kk * nbi + j acts as a column block of its own downstream)
  for (int kk = 0; kk < kg; ++kk) {
  const int blk = bi * (kg * nbi) + kk * nbi + bj;
  float best_key = INFINITY;
  uint64_t best_g = ~0ull;
  if (PHASE == 2) {
    best_key = tab_key[blk];
    best_g = tab_g[blk];
  } else {
  if (MULTI && kk > 0) {
    // later draws: keys from the first pass, drawn ones at +inf
    for (int idx = threadIdx.x; idx < n_in_block; idx += NT) {
      const int rl = idx / gpb, cl = idx % gpb;
      const float key = s_keys[idx];
      const uint64_t g = (uint64_t)((int64_t)bi * db + rl) * (uint64_t)ng_row + (uint64_t)((int64_t)bj * gpb + cl);
      if (key < best_key || (key == best_key && g < best_g)) { best_key = key; best_g = g; }
    }
  } else {
    // A thread keeps one group column of the block and walks down its rows, NT / gpb rows apart (threads beyond
    // the last whole row of groups idle), so the group index, the hash counter and the addresses advance by
    // additions.  Four groups per thread and step: the loads are issued together, then scores and hashes.
    // With a single draw most logarithms are skipped: -ln(u) >= 1 - u, so a group whose (1 - u) / score
    // exceeds the best key its warp has seen cannot win (the bound is tight exactly where winners live, u next
    // to 1; the warp-wide bound, refreshed after every step, makes whole warps skip the logarithm, which a
    // per-thread bound would not: among 32 lanes one almost always passes its own).
    constexpr int U = 4;
    const int rstep = NT / gpb;                                  // rows of the block covered per step (gpb <= 64)
    const int cl = (int)threadIdx.x % gpb, rl0 = (int)threadIdx.x / gpb;
    {
      const bool lane_on = rl0 < rstep;
      float wbound = INFINITY;                                   // warp-uniform: the smallest key any lane holds
      int best_rl = -1;                                          // row in the block of the thread's best group: it meets its
                                                                 // groups in ascending order, so a tie stays with the first
      const int n_steps = (db + U * rstep - 1) / (U * rstep);    // the same for every lane: the shuffles below need all 32
      const int64_t row0 = (int64_t)bi * db + (lane_on ? rl0 : 0);
      const int64_t cg = (int64_t)bj * gpb + cl;
      const float* gp = Gam + row0 * d_in + cg * MG;
      const float* ap = alpha + row0;
      uint64_t ctr = t * n_groups_total + (uint64_t)row0 * (uint64_t)ng_row + (uint64_t)cg;
      const uint64_t gstep = (uint64_t)rstep * (uint64_t)ng_row;
      const int64_t pstep = (int64_t)rstep * d_in;
      for (int step = 0, rl = rl0; step < n_steps; ++step, rl += U * rstep) {
        float4 g4[U][MG / 4];
        float al[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          al[u] = 0.f;
#pragma unroll
          for (int h = 0; h < MG / 4; ++h) g4[u][h] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (lane_on && rl + u * rstep < db) {
            al[u] = ap[u * rstep];
#pragma unroll
            for (int h = 0; h < MG / 4; ++h) g4[u][h] = *reinterpret_cast<const float4*>(gp + u * pstep + 4 * h);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (lane_on && rl + u * rstep < db) {
            float score = 0.f, sq = 0.f;
#pragma unroll
            for (int h = 0; h < MG / 4; ++h) {
              score += fabsf(g4[u][h].x);
              score += fabsf(g4[u][h].y);
              score += fabsf(g4[u][h].z);
              score += fabsf(g4[u][h].w);
              if (select_mode == ARMOR_SELECT_L2_RANDOM) {
                sq = fmaf(g4[u][h].x, g4[u][h].x, sq);
                sq = fmaf(g4[u][h].y, g4[u][h].y, sq);
                sq = fmaf(g4[u][h].z, g4[u][h].z, sq);
                sq = fmaf(g4[u][h].w, g4[u][h].w, sq);
              }
            }
            // the ablation's weights (Appendix E.1): L2 norm of the group's gradient, or equal weights
            if (select_mode == ARMOR_SELECT_L2_RANDOM) score = sqrtf(sq);
            else if (select_mode == ARMOR_SELECT_UNIFORM_RANDOM) score = 1.f;
            if (!(al[u] > 0.f)) score = 0.f;
            float key = INFINITY;
            if (score > 0.f) {
              if (select_mode != ARMOR_SELECT_L1_GREEDY) {
                const uint64_t bits = splitmix64(seed ^ splitmix64(ctr + (uint64_t)u * gstep));
                const uint32_t k24 = (uint32_t)(bits >> 40);
                // 1 - u = (2^24 - k24 - 1/2) 2^-24, exact in fp32; the factor 1 - 1e-5 covers the few ulp by
                // which the computed key can fall below (1 - u) / score
                const float one_minus_u = (float)(2u * ((1u << 24) - k24) - 1u) * 2.98023223876953125e-8f;
                if (MULTI || !(one_minus_u * 0.99999f >= wbound * score))
                  key = neg_log_uniform(k24) / score;
              } else {
                key = -score;
              }
              if (key < best_key) { best_key = key; best_rl = rl + u * rstep; }
            }
            if (MULTI) s_keys[(rl + u * rstep) * gpb + cl] = key;
          }
        }
        gp += U * pstep;
        ap += U * rstep;
        ctr += U * gstep;
        if (!MULTI) {
          asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(wbound) : "f"(best_key));
        }
      }
      if (best_rl >= 0) best_g = (uint64_t)((int64_t)bi * db + best_rl) * (uint64_t)ng_row + (uint64_t)cg;
    }
  }
  // arg-min over the CTA; ties go to the lower group index
  for (int o = 16; o > 0; o >>= 1) {
    const float ok = __shfl_down_sync(0xffffffffu, best_key, o);
    const uint64_t og = __shfl_down_sync(0xffffffffu, best_g, o);
    if (ok < best_key || (ok == best_key && og < best_g)) { best_key = ok; best_g = og; }
  }
  __shared__ float skey[NT / 32];
  __shared__ uint64_t sg[NT / 32];
  __shared__ float s_key;
  __shared__ uint64_t s_g;
  if ((threadIdx.x & 31) == 0) { skey[threadIdx.x >> 5] = best_key; sg[threadIdx.x >> 5] = best_g; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NT / 32; ++w)
      if (skey[w] < best_key || (skey[w] == best_key && sg[w] < best_g)) { best_key = skey[w]; best_g = sg[w]; }
    s_key = best_key;
    s_g = best_g;
  }
  __syncthreads();
  best_key = s_key;
  best_g = s_g;
  if (PHASE == 1) {
    if (threadIdx.x == 0) { tab_key[blk] = best_key; tab_g[blk] = best_g; }
    return;
  }
  }
  if (!(best_key < INFINITY)) {                               // nothing left to draw in this block (uniform)
    if (threadIdx.x == 0) {
      SelRec rec;
      rec.valid = 0; rec.row = 0; rec.cgrp = 0; rec.new_mask = 0; rec.old_mask = 0;
      for (int p = 0; p < 8; ++p) { rec.new_val[p] = 0.f; rec.old_val[p] = 0.f; }
      for (int k2 = kk; k2 < kg; ++k2) {
        sel[bi * (kg * nbi) + k2 * nbi + bj] = rec;
        part[bi * (kg * nbi) + k2 * nbi + bj] = 0.0;
      }
    }
    if (PHASE == 2) {
      SelRec none{};
      write_vectors(vec, none, bi, bj, nbi, nbi, db, MG, threadIdx.x, blockDim.x);
    }
    return;
  }
  if (MULTI && threadIdx.x == 0) {                          // out of the race for the later draws
    const int rl0 = (int)(best_g / (uint64_t)ng_row) - bi * db, cl0 = (int)(best_g % (uint64_t)ng_row) - bj * gpb;
    s_keys[rl0 * gpb + cl0] = INFINITY;
  }

  // ---- the selected group: z = Gamma_g + alpha K_c s_g, one candidate mask per thread
  const int64_t row = (int64_t)(best_g / (uint64_t)ng_row);
  const int64_t cg = (int64_t)(best_g % (uint64_t)ng_row);
  const int lc = (int)(cg % gpb) * MG;   // first row of the group inside B_j
  const float* Kj = Kfull + (int64_t)bj * db * db;
  const double a_r = (double)alpha[row];
  const unsigned om = M[row * ng_row + cg];
  double z[MG], sg_old[MG];
#pragma unroll
  for (int p = 0; p < MG; ++p) sg_old[p] = (double)S[row * d_in + cg * MG + p];
#pragma unroll
  for (int p = 0; p < MG; ++p) {
    double kz = 0.0;
#pragma unroll
    for (int q = 0; q < MG; ++q) kz += (double)Kj[(int64_t)(lc + p) * db + (lc + q)] * sg_old[q];
    z[p] = (double)Gam[row * d_in + cg * MG + p] + a_r * kz;
  }
  const unsigned cand = threadIdx.x;
  bool ok = cand < (1u << MG) && __popc(cand) == n_keep;
  double red = 0.0, wv[NKM];
  int pos[NKM];
#pragma unroll
  for (int i = 0; i < NKM; ++i) { wv[i] = 0.0; pos[i] = 0; }
  if (ok) {
    int cnt = 0;
#pragma unroll
    for (int p = 0; p < MG; ++p)
      if ((cand >> p) & 1u) { if (cnt < NKM) pos[cnt] = p; ++cnt; }
    if (n_keep == 2) {
      pinv2((double)Kj[(int64_t)(lc + pos[0]) * db + lc + pos[0]], (double)Kj[(int64_t)(lc + pos[0]) * db + lc + pos[1]],
            (double)Kj[(int64_t)(lc + pos[1]) * db + lc + pos[1]], z[pos[0]], z[pos[1]], wv[0], wv[1], red);
    } else {
      double Ks[NKM][NKM], zs[NKM];
#pragma unroll
      for (int i = 0; i < NKM; ++i) {
        zs[i] = 0.0;
#pragma unroll
        for (int j = 0; j < NKM; ++j) Ks[i][j] = 0.0;
      }
#pragma unroll
      for (int i = 0; i < NKM; ++i) {
        if (i >= n_keep) continue;
#pragma unroll
        for (int p = 0; p < MG; ++p)
          if (p == pos[i]) zs[i] = z[p];
#pragma unroll
        for (int j = 0; j < NKM; ++j)
          if (j < n_keep) Ks[i][j] = (double)Kj[(int64_t)(lc + pos[i]) * db + lc + pos[j]];
      }
      ok = chol_small<NKM>(n_keep, Ks, zs, wv, red);
    }
    red /= a_r;
  }
  // order: larger reduction; then the incumbent; then the lexicographically first tuple (= larger
  // bit-reversed pattern)
  const unsigned rev = __brev(cand) >> (32 - MG);
  double b_red = ok ? red : -INFINITY;
  unsigned b_tie = ok ? (((cand == om) ? (1u << MG) : 0u) | rev) : 0u;
  unsigned b_cand = ok ? cand : 0xffffffffu;
  for (int o = 16; o > 0; o >>= 1) {
    const double o_red = __shfl_down_sync(0xffffffffu, b_red, o);
    const unsigned o_tie = __shfl_down_sync(0xffffffffu, b_tie, o);
    const unsigned o_cand = __shfl_down_sync(0xffffffffu, b_cand, o);
    const bool take = (o_cand != 0xffffffffu) &&
                      (b_cand == 0xffffffffu || o_red > b_red || (o_red == b_red && o_tie > b_tie));
    if (take) { b_red = o_red; b_tie = o_tie; b_cand = o_cand; }
  }
  __shared__ double sred[NT / 32];
  __shared__ unsigned stie[NT / 32], scand[NT / 32];
  __shared__ unsigned s_win;
  __shared__ SelRec s_rec;
  if ((threadIdx.x & 31) == 0) { sred[threadIdx.x >> 5] = b_red; stie[threadIdx.x >> 5] = b_tie; scand[threadIdx.x >> 5] = b_cand; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      const bool take = (scand[w] != 0xffffffffu) &&
                        (b_cand == 0xffffffffu || sred[w] > b_red || (sred[w] == b_red && stie[w] > b_tie));
      if (take) { b_red = sred[w]; b_tie = stie[w]; b_cand = scand[w]; }
    }
    s_win = b_cand;
    if (b_cand == 0xffffffffu) {   // every mask failed its factorisation: nothing happens in this block
      SelRec rec;
      rec.valid = 0; rec.row = 0; rec.cgrp = 0; rec.new_mask = 0; rec.old_mask = 0;
      for (int p = 0; p < 8; ++p) { rec.new_val[p] = 0.f; rec.old_val[p] = 0.f; }
      sel[blk] = rec;
      part[blk] = 0.0;
      if (PHASE == 2) s_rec = rec;
    }
  }
  __syncthreads();
  if (s_win != 0xffffffffu && cand == s_win) {
  // the winning thread writes the record
  SelRec rec;
  rec.valid = 1;
  rec.row = (int32_t)row;
  rec.cgrp = (int32_t)cg;
  rec.old_mask = (int32_t)om;
  rec.new_mask = (int32_t)cand;
  for (int p = 0; p < 8; ++p) { rec.new_val[p] = 0.f; rec.old_val[p] = 0.f; }
#pragma unroll
  for (int p = 0; p < MG; ++p) rec.old_val[p] = (float)sg_old[p];
#pragma unroll
  for (int i = 0; i < NKM; ++i)
    if (i < n_keep) rec.new_val[pos[i]] = (float)(wv[i] / a_r);
  // <Gamma, dS> restricted to this group: this block's share of <E H_w, V>
  double ehv = 0.0;
#pragma unroll
  for (int p = 0; p < MG; ++p)
    ehv += (double)Gam[row * d_in + cg * MG + p] * ((double)rec.new_val[p] - (double)rec.old_val[p]);
  part[blk] = ehv;
  sel[blk] = rec;
  if (PHASE == 2) s_rec = rec;
  }
  __syncthreads();                                          // the shared scratch is reused by the next draw
  if (PHASE == 2) write_vectors(vec, s_rec, bi, bj, nbi, nbi, db, MG, threadIdx.x, blockDim.x);
  }
}

// One CTA per block (i, j), one warp per pair (j, j') at a time.  Y == nullptr: diagonal weighting, only the
// j == j' pair contributes and y = z (.) hdiag.
__global__ void __launch_bounds__(NT) mask_quad_kernel(const float* Zsel, const float* Acol,
                                                       const float* Y, const float* hdiag,
                                                       double* __restrict__ part, int64_t d_in, int db, int nbo_pad,
                                                       int nbi, int nbv) {
  grid_begin();
  const int bi = blockIdx.x / nbv, j = blockIdx.x % nbv;      // j, j2: virtual column blocks (draw * nbi + column block)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = NT / 32;
  double acc = 0.0;
  const float* a1 = Acol + ((int64_t)bi * nbv + j) * db;
  const float* z1 = Zsel + ((int64_t)j * nbo_pad + bi) * db;
  for (int j2 = warp; j2 < nbv; j2 += nw) {
    if (!Y && (j2 % nbi) != (j % nbi)) continue;              // diagonal weighting: other column blocks do not interact
    const float* a2 = Acol + ((int64_t)bi * nbv + j2) * db;
    const float* z2 = Zsel + ((int64_t)j2 * nbo_pad + bi) * db;
    float w = 0.f, m = 0.f;
    if (Y) {
      const float* y = Y + ((int64_t)j * nbo_pad + bi) * d_in + (int64_t)(j2 % nbi) * db;
      for (int k = lane; k < db; k += 32) { w = fmaf(a1[k], a2[k], w); m = fmaf(y[k], z2[k], m); }
    } else {
      const float* h = hdiag + (int64_t)(j % nbi) * db;
      for (int k = lane; k < db; k += 32) { w = fmaf(a1[k], a2[k], w); m = fmaf(z1[k] * h[k], z2[k], m); }
    }
    for (int o = 16; o > 0; o >>= 1) {
      w += __shfl_xor_sync(0xffffffffu, w, o);
      m += __shfl_xor_sync(0xffffffffu, m, o);
    }
    acc += (double)w * (double)m;
  }
  __shared__ double red[NT / 32];
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w2 = 0; w2 < nw; ++w2) t += red[w2];
    part[blockIdx.x] = t;
  }
}

// The accepted group of a block goes into the core and its mask; returns whether the mask changed.
struct CommitArgs { float* S; uint8_t* M; armor_iter_stats* st_base; const int64_t* it_dev; int mg; };
__device__ __forceinline__ bool commit_group(const CommitArgs& w, const SelRec& rec, int64_t d_in) {
  if (!rec.valid) return false;
  float* sp = w.S + (int64_t)rec.row * d_in + (int64_t)rec.cgrp * w.mg;
  for (int h = 0; h < w.mg / 4; ++h)
    *reinterpret_cast<float4*>(sp + 4 * h) =
        make_float4(rec.new_val[4 * h], rec.new_val[4 * h + 1], rec.new_val[4 * h + 2], rec.new_val[4 * h + 3]);
  w.M[(int64_t)rec.row * (d_in / w.mg) + rec.cgrp] = (uint8_t)rec.new_mask;
  return rec.new_mask != rec.old_mask;
}
__device__ __forceinline__ void count_changed(const CommitArgs& w, bool changed) {          // whole warps
  const int n = __popc(__ballot_sync(0xffffffffu, changed));
  if (w.st_base && n && (threadIdx.x & 31) == 0) atomicAdd(&w.st_base[*w.it_dev].groups_changed, n);   // summed over the sweeps of the iteration
}

// Where nothing is carried: a thread per block (one CTA walking 3,584 blocks took 21 us).
constexpr int COMMIT_NT = 64;
__global__ void __launch_bounds__(COMMIT_NT) mask_commit_kernel(const SelRec* sel, int nblocks, int64_t d_in, const double* sc, CommitArgs w) {
  grid_begin();
  if (sc[SC_ACCEPT] == 0.0) return;
  const int b = blockIdx.x * COMMIT_NT + threadIdx.x;
  count_changed(w, b < nblocks && commit_group(w, sel[b], d_in));
}

// The accepted group updates change T H_w = S B H_w by the rows (delta^T B_j[group rows, :]) H_w[j-th block
// row, :] = y_ij, added to row r_ij.  Groups of one row-block may share a row; its additions happen in the order of the column
// blocks (deterministic sums), all of them by the CTA that holds the first.  The grid is (row-block, chunk of 1024 columns,
// CARRY_PICKS column blocks at a time): one CTA walking all column blocks in batches took 20 us for 50 MB, a chain of batches
// with few CTAs in flight.  Which pick is a row's first and which its last is found once per CTA in a table of the block's
// rows (d_block <= 256; one CTA of a row-block also commits its groups), so that neither shared memory nor, with at most CARRY_CTAS along the picks, the work grows faster
// than their number (thousands with small blocks and several draws).
constexpr int CARRY_PICKS = 4;
constexpr int CARRY_CTAS = 64;
constexpr int CARRY_TAB = 2048;                            // picks whose rows are kept in shared memory
__device__ __forceinline__ int carry_row(const SelRec& rec, int row0) { return rec.valid ? rec.row - row0 : -1; }
__global__ void __launch_bounds__(NT) mask_carry_kernel(const SelRec* sel, const float* Y,
                                                        float* P, const double* sc,
                                                        int64_t d_in, int db, int nbo_pad, int nbv, CommitArgs w) {
  grid_begin();
  __shared__ int row_of[CARRY_TAB];                        // row inside the block, -1: no group
  __shared__ int first[256], last[256];                    // picks of a row
  if (sc[SC_ACCEPT] == 0.0) return;
  const int bi = blockIdx.x, row0 = bi * db;
  const SelRec* mine_sel = sel + (int64_t)bi * nbv;
  if (blockIdx.y == 0 && blockIdx.z == 0)                   // the block row's groups go into the core
    for (int j0 = 0; j0 < nbv; j0 += NT) {
      const int j = j0 + threadIdx.x;
      count_changed(w, j < nbv && commit_group(w, mine_sel[j], d_in));
    }
  for (int r = threadIdx.x; r < db; r += NT) { first[r] = nbv; last[r] = -1; }
  __syncthreads();
  for (int j = threadIdx.x; j < nbv; j += NT) {
    const int r = carry_row(mine_sel[j], row0);
    if (j < CARRY_TAB) row_of[j] = r;
    if (r >= 0) { atomicMin(&first[r], j); atomicMax(&last[r], j); }
  }
  __syncthreads();
  const int64_t c4 = (int64_t)blockIdx.y * 1024 + 4 * threadIdx.x;
  if (c4 >= d_in) return;
  auto row_at = [&](int j) { return j < CARRY_TAB ? row_of[j] : carry_row(mine_sel[j], row0); };
  for (int j0 = blockIdx.z * CARRY_PICKS; j0 < nbv; j0 += gridDim.z * CARRY_PICKS) {
    float4 v[CARRY_PICKS], y[CARRY_PICKS];
    int row[CARRY_PICKS];                                  // -1: nothing to do for this pick
#pragma unroll
    for (int u = 0; u < CARRY_PICKS; ++u) {
      const int j = j0 + u;
      row[u] = j < nbv ? row_at(j) : -1;
      if (row[u] >= 0 && first[row[u]] != j) row[u] = -1;
      if (row[u] < 0) continue;
      v[u] = *reinterpret_cast<const float4*>(P + (int64_t)(row0 + row[u]) * d_in + c4);
      y[u] = *reinterpret_cast<const float4*>(Y + ((int64_t)j * nbo_pad + bi) * d_in + c4);
    }
#pragma unroll
    for (int u = 0; u < CARRY_PICKS; ++u) {
      if (row[u] < 0) continue;
      float4 x = v[u];
      x.x += y[u].x; x.y += y[u].y; x.z += y[u].z; x.w += y[u].w;
      const int end = last[row[u]];
      for (int j = j0 + u + 1; j <= end; ++j) {
        if (row_at(j) != row[u]) continue;
        const float4 w = *reinterpret_cast<const float4*>(Y + ((int64_t)j * nbo_pad + bi) * d_in + c4);
        x.x += w.x; x.y += w.y; x.z += w.z; x.w += w.w;
      }
      *reinterpret_cast<float4*>(P + (int64_t)(row0 + row[u]) * d_in + c4) = x;
    }
  }
}

}  // namespace

// alpha (alpha[r] = || A[:, r] ||^2, column r of the block that owns row r of the core) and the m x m diagonal blocks of K_j = (B_j H_jj) B_j^T, the only entries
// of K_j the group solves read (Appendix B.1: B' D B'^T for the m rows of one group), in one launch.
// Y = B_j H_jj comes from a block product.  CTAs [0, n_kc): one warp per group, lane l takes columns l, l + 32, ..;
// the remaining CTAs compute alpha.
template <int MG>
__global__ void __launch_bounds__(NT) mask_prep_kernel(const float* A, const float* B,
                                                       const float* Y, float* __restrict__ Kfull,
                                                       float* __restrict__ alpha, int db, int nbi, int n_kc) {
  grid_begin();
  if ((int)blockIdx.x < n_kc) {
    const int gpb = db / MG;
    const int wg = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);       // (column block, group)
    const int lane = threadIdx.x & 31;
    if (wg >= nbi * gpb) return;
    const int j = wg / gpb, lc = (wg % gpb) * MG;
    const float* Yj = Y + (int64_t)j * db * db;
    const float* Bj = B + (int64_t)j * db * db;
    float acc[MG][MG];
#pragma unroll
    for (int p = 0; p < MG; ++p)
#pragma unroll
      for (int q = 0; q < MG; ++q) acc[p][q] = 0.f;
    for (int k = lane; k < db; k += 32) {
      float y[MG], b[MG];
#pragma unroll
      for (int p = 0; p < MG; ++p) { y[p] = Yj[(int64_t)(lc + p) * db + k]; b[p] = Bj[(int64_t)(lc + p) * db + k]; }
#pragma unroll
      for (int p = 0; p < MG; ++p)
#pragma unroll
        for (int q = 0; q < MG; ++q) acc[p][q] = fmaf(y[p], b[q], acc[p][q]);
    }
#pragma unroll
    for (int p = 0; p < MG; ++p)
#pragma unroll
      for (int q = 0; q < MG; ++q) {
        float v = acc[p][q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) Kfull[(int64_t)j * db * db + (int64_t)(lc + p) * db + (lc + q)] = v;
      }
    return;
  }
  // alpha[r] = || A_i[:, r] ||^2: 256 threads = 32 columns x 8 row slices
  const int ab = blockIdx.x - n_kc;
  const int per = (db + 31) / 32;
  const int i = ab / per;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int r = (ab % per) * 32 + tx;
  const float* Ai = A + (int64_t)i * db * db;
  double acc = 0.0;
  if (r < db)
    for (int o = ty; o < db; o += 8) {
      const double v = Ai[(int64_t)o * db + r];
      acc += v * v;
    }
  __shared__ double part[8][33];
  part[ty][tx] = acc;
  __syncthreads();
  if (ty == 0 && r < db) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += part[k][tx];
    alpha[i * db + r] = (float)t;
  }
}

void launch_mask_prep(armor_ctx* c, const float* A, const float* B, const float* Y, cudaStream_t s) {
  const int db = c->db, mg = c->cfg.m_group;
  const int n_kc = (c->nbi * (db / mg) + NT / 32 - 1) / (NT / 32);
  const int n_al = c->nbo * ((db + 31) / 32);
  KTimer kt(c, ARMOR_KC_MASK_GUARD, 0.0, s);
  if (mg == 8) launch_dependent(mask_prep_kernel<8>, n_kc + n_al, NT, 0, s, A, B, Y, c->Kfull, c->alpha, db, c->nbi, n_kc);
  else launch_dependent(mask_prep_kernel<4>, n_kc + n_al, NT, 0, s, A, B, Y, c->Kfull, c->alpha, db, c->nbi, n_kc);
  c->launches++;
}

void launch_mask_select(armor_ctx* c, const float* A, const float* B, const float* Gam, const float* S, const uint8_t* M, uint64_t t_base,
                        uint64_t t_mul, LaunchStream at) {
  const int mg = c->cfg.m_group;
  const uint64_t n_groups = (uint64_t)(c->d_out * (c->d_in / mg));
  const VectorArgs vec{A, B, c->Zsel, c->Acol, c->nbo_pad};
#define ARMOR_SELECT_ARGS Gam, S, M, c->alpha, c->Kfull, c->sel, c->partblk, c->d_in, c->db, c->nbi, c->cfg.n_keep, \
                          c->cfg.select_mode, c->cfg.seed, t_base, t_mul, c->it_dev, n_groups, c->kg, c->tab_key, c->tab_g, vec
  // kg > 1: the block's keys stay in shared memory between the draws (up to 64 KiB: d_block 256, groups of four)
  const size_t smem = c->kg > 1 ? (size_t)c->db * (c->db / mg) * sizeof(float) : 0;
#define ARMOR_SELECT_LAUNCH(MGV, NKV, MULTIV)                                                                           \
  do {                                                                                                                  \
    if (MULTIV) {                                                                                                       \
      if (smem > 48 * 1024)                                                                                             \
        cudaFuncSetAttribute(mask_select_kernel<MGV, NKV, MULTIV, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                             (int)smem);                                                                                \
      launch_dependent(mask_select_kernel<MGV, NKV, MULTIV, 0>, c->nbo * c->nbi, NT, smem, at, ARMOR_SELECT_ARGS);      \
    } else {                                                                                                            \
      launch_dependent(mask_select_kernel<MGV, NKV, false, 1>, c->nbo * c->nbi, NT, 0, at, ARMOR_SELECT_ARGS);          \
      launch_dependent(mask_select_kernel<MGV, NKV, false, 2>, c->nbo * c->nbi, MGV == 4 ? 32 : NT, 0, at.s,            \
                       ARMOR_SELECT_ARGS);                                                                              \
      c->launches++;                                                                                                    \
    }                                                                                                                   \
  } while (0)
  const bool multi = c->kg > 1;
  KTimer kt(c, ARMOR_KC_MASK_SELECT, 4.0 * (double)c->wn, at.s);   // one read of the core gradient
  if (mg == 8 && c->cfg.n_keep > 4) { if (multi) ARMOR_SELECT_LAUNCH(8, 6, true); else ARMOR_SELECT_LAUNCH(8, 6, false); }
  else if (mg == 8) { if (multi) ARMOR_SELECT_LAUNCH(8, 4, true); else ARMOR_SELECT_LAUNCH(8, 4, false); }
  else { if (multi) ARMOR_SELECT_LAUNCH(4, 4, true); else ARMOR_SELECT_LAUNCH(4, 4, false); }
#undef ARMOR_SELECT_LAUNCH
#undef ARMOR_SELECT_ARGS
  c->launches++;
}

void launch_mask_quadratic(armor_ctx* c, const float* A, const float* B, const float* H, armor_iter_stats* st, cudaStream_t s) {
  const int db = c->db, nbo = c->nbo, nbi = c->nbi, nbo_pad = c->nbo_pad, kg = c->kg, nbv = nbi * kg;
  if (kg > 1) {
    KTimer kt(c, ARMOR_KC_MASK_GUARD, 0.0, s);
    launch_dependent(mask_vectors_kernel, nbo * nbv, NT, 0, s, VectorArgs{A, B, c->Zsel, c->Acol, nbo_pad}, c->sel, db, nbi, c->cfg.m_group, nbv);
    c->launches++;
  }
  const float* Y = nullptr;
  if (c->cfg.h_mode == ARMOR_H_FULL) {
    // y_v = z_v H[j-th block row, :], batched over the column blocks j, one launch per draw:  [nbo, db] x [db, d_in]
    for (int kk = 0; kk < kg; ++kk) {
      const float* Zk = c->Zsel + (int64_t)kk * nbi * nbo_pad * db;
      float* Yk = c->Ysel + (int64_t)kk * nbi * nbo_pad * c->d_in;
      if (!(c->tc_blocks && tc_gram_ok(c) && tc_done(c, tc_select_rows_times_H(c, Zk, H, Yk, nbo_pad, s)))) {
        BGemm g{};
        g.A = Zk; g.sAb = (int64_t)nbo_pad * db; g.sAm = db; g.sAk = 1;
        g.B = H; g.sBb = (int64_t)db * c->d_in; g.sBk = c->d_in; g.sBn = 1;
        g.C = Yk; g.sCb = (int64_t)nbo_pad * c->d_in; g.sCm = c->d_in; g.sCn = 1;
        g.M = nbo; g.N = (int)c->d_in; g.K = db; g.batch = nbi; g.alpha = 1.f;
        launch_bgemm(c, g, s);
      }
    }
    Y = c->Ysel;
  }
  double* part = c->quadpart;
  {
    KTimer kt(c, ARMOR_KC_MASK_GUARD, 0.0, s);
    launch_dependent(mask_quad_kernel, nbo * nbv, NT, 0, s, c->Zsel, c->Acol, Y, c->hdiag, part, c->d_in, db, nbo_pad, nbi, nbv);
  }
  c->launches++;
  launch_stage(c, st, 4, c->partblk, nbo * nbv, s, part, nbo * nbv, SC_Q_M);     // the sum of the terms and the decision
}

void launch_mask_commit(armor_ctx* c, float* S, uint8_t* M, float* P, armor_iter_stats* st, cudaStream_t s) {
  KTimer kt(c, ARMOR_KC_MASK_GUARD, 0.0, s);
  const int nbv = c->nbi * c->kg, n = c->nbo * nbv;
  const CommitArgs w{S, M, st, c->it_dev, c->cfg.m_group};
  if (P) {
    int groups = (nbv + CARRY_PICKS - 1) / CARRY_PICKS;
    if (groups > CARRY_CTAS) groups = CARRY_CTAS;
    launch_dependent(mask_carry_kernel, dim3(c->nbo, (unsigned)((c->d_in + 1023) / 1024), (unsigned)groups), NT, 0, s, c->sel, c->Ysel, P, c->sc,
                     c->d_in, c->db, c->nbo_pad, nbv, w);
  } else {
    launch_dependent(mask_commit_kernel, (n + COMMIT_NT - 1) / COMMIT_NT, COMMIT_NT, 0, s, c->sel, n, c->d_in, c->sc, w);
  }
  c->launches++;
}
