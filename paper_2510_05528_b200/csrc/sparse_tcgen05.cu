// The core product of the deployment form (Section 3.1: y = A (S (B x)), S the 2:4 sparse core) on the sparse
// tensor cores of sm_100a:  Z2[t][m] = sum_k S[m][k] * Z1[t][k]  with S given as its kept values (two of every
// four along k, bf16) plus the 2-bit positions of the kept values, Z1 bf16, fp32 accumulation and output.
//
// S is the A operand of tcgen05.mma.sp (kind::f16): each instruction multiplies a 128 x 32 slice of S, held in
// shared memory as 128 x 16 kept values, by a 32 x 128 slice of Z1^T; the positions come from tensor memory.
//
// Layout of the positions (what the instruction reads, M = 128, 16-bit operands): one 32-bit tensor-memory column
// per instruction; lane l = m0 + 8 k1 + 16 m2 (m0 < 8, k1 < 2, m2 < 8) holds, in its low half, the 16 bits of row
// m0 + 16 m2 for the k-half k1 (16 consecutive k: four groups, four bits each, the lower kept position in bits
// 0-1 and the higher one in bits 2-3 of the group's nibble) and, in its high half, the same for row m0 + 16 m2 + 8.
// Consecutive instructions along k use consecutive columns; the instruction is given the even column of the pair
// and the column's parity as the selector field of its descriptor.  compress_24_kernel writes the positions in
// exactly this order, 128 lanes x 4 columns (16 bytes per lane) per 128 x 128 block of S: 2 KiB that travel with
// the stage's operands by TMA and go from shared to tensor memory with one tcgen05.cp (128 lanes x 128 bits)
// issued by the MMA thread in front of the stage's four instructions -- the copy runs in the tensor-core pipe,
// in order with the MMAs.  (Writing the positions with tcgen05.st from other warps was measured first: every
// store waited about 1600 cycles behind the running MMAs and the kernel ran at a quarter of its rate.)
//
// Kernel: persistent, one CTA per SM, 192 threads: warp 0 TMA producer, warp 1 MMA issuer, warps 2-5 epilogue
// (transposing store: lanes are rows m of S, columns are tokens).  128 x 128 output tiles, 128 k per stage
// (16 KiB of kept values + 32 KiB of Z1 + 2 KiB of positions), four stages, two accumulator buffers.  Every wait
// is bounded.
#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BM = 128, BN = 128, BKL = 128;        // BKL: logical k per stage (64 kept values = 128 bytes per row)
constexpr int NTHREADS = 192;
constexpr int STAGES = 4;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t META_COL0 = 256;                 // accumulators: columns 0-127 and 128-255
constexpr int A_BYTES = BM * 64 * 2;                // 16 KiB
constexpr int BH_BYTES = BN * 64 * 2;               // 16 KiB: one half (64 k) of the Z1 stage
constexpr int E_BYTES = 128 * 16;                   // positions of one stage
constexpr int STAGE_BYTES = A_BYTES + 2 * BH_BYTES + E_BYTES; // 50 KiB

struct SParams {
  float* Z; int64_t ldz;        // [N tokens][ldz], written transposed
  __nv_bfloat16* Zb;            // non-null: the output is written as bf16 here instead
  int64_t M, N, K;              // rows of S, tokens, logical k
  int m_tiles, n_tiles, k_tiles, tile_n;
  int32_t* status;
};

__device__ __forceinline__ uint64_t smem_desc_k(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;                           // 128-byte swizzle
  return d;
}

// bf16 operands, fp32 accumulation, both K-major, sparse A; sel = parity of the position column
__device__ __forceinline__ uint32_t instr_desc_sp(uint32_t sel) {
  uint32_t d = sel & 3u;          // position selector
  d |= 1u << 2;                   // A is 2:4 sparse
  d |= 1u << 4;                   // D format: F32
  d |= 1u << 7;                   // A format: BF16
  d |= 1u << 10;                  // B format: BF16
  d |= (uint32_t)(BN >> 3) << 17;
  d |= (uint32_t)(BM >> 4) << 24;
  return d;
}

__device__ __forceinline__ void umma_bf16_sp(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t tmem_e,
                                             uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.sp.cta_group::1.kind::f16 [%0], %1, %2, [%3], %4, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(tmem_e), "r"(idesc), "r"(acc)
      : "memory");
}

// Tile order: groups of GROUP_M row tiles of S; inside a group the row tile runs fastest, then the token tile.
// The CTAs running at one time then share a few row tiles of S (read from DRAM once) and a band of token tiles
// (Z1 stays in L2), instead of sweeping all of S for every token tile.
constexpr int GROUP_M = 8;
__device__ __forceinline__ void tile_to_mn(int tile, int m_tiles, int n_tiles, int& mt, int& nt) {
  const int per_group = GROUP_M * n_tiles;
  const int g = tile / per_group, r = tile - g * per_group;
  const int gm = min(GROUP_M, m_tiles - g * GROUP_M);
  mt = g * GROUP_M + r % gm;
  nt = r / gm;
}

// 128 rows of 16 bytes, packed (8-row groups 128 bytes apart), no swizzle: the positions of one stage
__device__ __forceinline__ uint64_t smem_desc_e(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(128 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// shared -> tensor memory, 128 lanes x 128 bits (four columns), in the tensor-core pipe
__device__ __forceinline__ void tmem_cp_e(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::1.128x128b [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void tmem_cp_e_pair(uint32_t taddr, uint64_t sdesc) {
  asm volatile("tcgen05.cp.cta_group::2.128x128b [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}

// Epilogue store of 32 tokens of one row of S per lane (the output is [token][row], so a warp's 32 rows are
// contiguous for every token).  bf16: neighbouring lanes swap one value per pair of tokens so that every lane
// stores two adjacent rows (4 bytes) of one token -- as many store instructions per element as in fp32.
__device__ __forceinline__ void store_chunk(const SParams& p, const uint32_t (&r)[32], int64_t row, int64_t tok0, int lane) {
  if (p.Zb == nullptr) {
    if (row < p.M) {
#pragma unroll
      for (int cidx = 0; cidx < 32; ++cidx)
        if (tok0 + cidx < p.N) p.Z[(tok0 + cidx) * p.ldz + row] = __uint_as_float(r[cidx]);
    }
    return;
  }
  const bool odd = lane & 1;
  const int64_t row2 = row - (odd ? 1 : 0);                  // the even row of the lane pair (p.M is even)
#pragma unroll
  for (int cidx = 0; cidx < 32; cidx += 2) {
    const uint32_t give = odd ? r[cidx] : r[cidx + 1];
    const uint32_t got = __shfl_xor_sync(0xffffffffu, give, 1);
    const float lo = __uint_as_float(odd ? got : r[cidx]), hi = __uint_as_float(odd ? r[cidx + 1] : got);
    const int64_t tok = tok0 + cidx + (odd ? 1 : 0);
    if (row2 < p.M && tok < p.N) {
      const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
      *reinterpret_cast<__nv_bfloat162*>(p.Zb + tok * p.ldz + row2) = v;
    }
  }
}

__global__ void __launch_bounds__(NTHREADS, 1)
tc_sparse_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                 const __grid_constant__ CUtensorMap mapE, const SParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 4];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * STAGES]), tempty0 = smem_u32(&bars[2 * STAGES + 2]);
  const int n_tiles_total = p.m_tiles * p.n_tiles;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) { mbar_init(tfull0 + 8 * s, 1); mbar_init(tempty0 + 8 * s, 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < n_tiles_total && ok; tile += gridDim.x) {
        int mt, nt;
        tile_to_mn(tile, p.m_tiles, p.n_tiles, mt, nt);
        for (int kt = 0; kt < p.k_tiles; ++kt) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
          const uint32_t fb = full0 + 8 * stage;
          mbar_expect_tx(fb, STAGE_BYTES);
          const uint32_t dst = smem_u32(smem + (size_t)stage * STAGE_BYTES);
          tma_load_2d(dst, &mapA, kt * 64, mt * BM, fb);                      // 64 kept values = 128 logical k
          tma_load_2d(dst + A_BYTES, &mapB, kt * BKL, nt * BN, fb);
          tma_load_2d(dst + A_BYTES + BH_BYTES, &mapB, kt * BKL + 64, nt * BN, fb);
          tma_load_2d(dst + A_BYTES + 2 * BH_BYTES, &mapE, 0, (mt * p.k_tiles + kt) * 128, fb);
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) {
        for (int back = 1; back <= STAGES && back <= issued; ++back) {
          int s = stage - back; uint32_t ph = phase;
          if (s < 0) { s += STAGES; ph ^= 1; }
          const long long t0 = clock64();
          while (!mbar_try(full0 + 8 * s, ph) && clock64() - t0 < 20000000ll) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < n_tiles_total && ok; tile += gridDim.x, ++local) {
        const int as = local & 1;
        const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
        if (!mbar_wait(tempty0 + 8 * as, aphase ^ 1, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tacc = tmem_base + (uint32_t)(as * BN);
        for (int kt = 0; kt < p.k_tiles; ++kt) {
          if (!mbar_wait(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + (size_t)stage * STAGE_BYTES);
          const uint32_t sb = sa + A_BYTES;
          tmem_cp_e(tmem_base + META_COL0 + (uint32_t)(4 * stage), smem_desc_e(sb + 2 * BH_BYTES));
#pragma unroll
          for (int j = 0; j < 4; ++j) {                                        // 32 logical k per instruction
            const uint64_t da = smem_desc_k(sa + j * 32);                      // 16 kept values = 32 bytes
            const uint64_t dbm = smem_desc_k(sb + (j >> 1) * BH_BYTES + (j & 1) * 64);
            const uint32_t ecol = tmem_base + META_COL0 + (uint32_t)(4 * stage + j);
            umma_bf16_sp(tacc, da, dbm, ecol & ~1u, instr_desc_sp(ecol & 1u), (uint32_t)((kt > 0) | (j != 0)));
          }
          umma_commit(empty0 + 8 * stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
        if (ok) umma_commit(tfull0 + 8 * as);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    const int q = warp & 3;
    int local = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < n_tiles_total && ok; tile += gridDim.x, ++local) {
      int mt, nt;
        tile_to_mn(tile, p.m_tiles, p.n_tiles, mt, nt);
      const int as = local & 1;
      const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
      if (!mbar_wait(tfull0 + 8 * as, aphase, abortp, p.status)) { ok = false; break; }
      tc_fence_after();
      const int64_t row = (int64_t)mt * BM + q * 32 + lane;                    // row of S = column of Z
#pragma unroll 1
      for (int ch = 0; ch < BN / 32; ++ch) {
        uint32_t r[32];
        tmem_ld32(tmem_base + (uint32_t)(as * BN + ch * 32) + ((uint32_t)(q * 32) << 16), r);
        const int64_t tok0 = (int64_t)nt * BN + ch * 32;
        store_chunk(p, r, row, tok0, lane);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * as);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------------------
// The same product on pairs of CTAs (cta_group::2): a cluster of two CTAs works on a 256 x 256 output tile.
// Each CTA holds 128 rows of S (kept values in shared memory, positions in its own tensor memory) and half of
// the tile's tokens (128 rows of Z1); one instruction issued by the even CTA multiplies 256 x 32 of S by
// 32 x 256 of Z1^T, every SM reading only half of Z1's tile from its shared memory.  Per SM and 128 k this
// loads 16 KiB + 32 KiB for 128 x 256 outputs, half of what the one-CTA kernel above loads.
//   full[s]   (even CTA): armed by the even CTA's producer for the bytes of both CTAs; both CTAs' TMA loads
//             complete on it (cta_group::2 loads may signal the pair's other CTA)
//   empty[s], tfull (both CTAs): tcgen05.commit multicast to the pair
//   tempty    (even CTA): 8 arrivals, one per epilogue warp of either CTA
// The positions of both CTAs go from their shared to their tensor memory with one tcgen05.cp of the pair.
// One accumulator buffer of 256 columns (the positions need tensor-memory columns too), or two row tiles' of up to 224 that share
// the stage's tokens: an SM then loads 64 KiB for 256 x 224 outputs and 128 k instead of 50 KiB for 128 x 256, and what L2 delivers
// (52 bytes a clock and SM) bounds the kernel at the burst clock.  28672 x 8192, 4,096 tokens 898 -> 822 us, 2.34 PFLOP/s of dense-equivalent
// products.  (Positions copied one stage ahead of their MMAs: 985 us, the stage is held longer; eight epilogue warps with one row tile:
// 4096 x 4096, 4,096 tokens 94 -> 98.)

__device__ __forceinline__ void umma_bf16_sp_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t tmem_e,
                                                  uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "tcgen05.mma.sp.cta_group::2.kind::f16 [%0], %1, %2, [%3], %4, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(tmem_e), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ uint32_t instr_desc_sp_pair(int n) {
  uint32_t d = 0;
  d |= 1u << 2;
  d |= 1u << 4;
  d |= 1u << 7;
  d |= 1u << 10;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(256 >> 4) << 24;
  return d;
}
// MT: row tiles of 256 that share a stage's tokens
template <int MT>
struct PairN {
  static constexpr int MAX_N = MT == 1 ? 256 : 224;                       // accumulators and positions fit tensor memory
  static constexpr int STAGES = MT == 1 ? 4 : 3;
  static constexpr int BH = MAX_N / 2 * 64 * 2;                           // one half (64 k) of the Z1 stage
  static constexpr int E = MT * A_BYTES + 2 * BH;
  static constexpr int STAGE = E + MT * E_BYTES;
  static constexpr uint32_t META = MT * MAX_N;                            // 4 MT columns a stage
  static constexpr int EPI = MT == 1 ? 4 : 8;                             // epilogue warps
  static constexpr int THREADS = 64 + 32 * EPI;
  static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024;
};

template <int MT>
__global__ void __launch_bounds__(PairN<MT>::THREADS, 1)
tc_sparse_pair_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                      const __grid_constant__ CUtensorMap mapE, const SParams p) {
  using T = PairN<MT>;
  constexpr int STAGES = T::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 2];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[STAGES]);
  const uint32_t tfull = smem_u32(&bars[2 * STAGES]), tempty = smem_u32(&bars[2 * STAGES + 1]);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int m_groups = p.m_tiles / (2 * MT);
  const int n_tiles_total = m_groups * p.n_tiles;           // p.n_tiles counts tiles of p.tile_n tokens here
  const int half_n = p.tile_n / 2;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 2 * T::EPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                       // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  grid_begin();                                             // (tensor memory is this CTA's before the next kernel's CTAs start)
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      bool ok = true;
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs) {
        int mt, nt;
        tile_to_mn(tile, m_groups, p.n_tiles, mt, nt);
        const int row0 = mt * (256 * MT) + (int)rank * 128, tok0 = nt * p.tile_n + (int)rank * half_n;
        for (int kt = 0; kt < p.k_tiles; ++kt) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
          if (rank == 0) mbar_expect_tx(full0 + 8 * stage, 2 * (MT * (A_BYTES + E_BYTES) + 2 * half_n * 128));
          const uint32_t fb = map_to_cta(full0 + 8 * stage, 0);
          const uint32_t dst = smem_u32(smem + (size_t)stage * T::STAGE);
#pragma unroll
          for (int m = 0; m < MT; ++m) tma_load_2d_pair(dst + m * A_BYTES, &mapA, kt * 64, row0 + 256 * m, fb);
          tma_load_2d_pair(dst + MT * A_BYTES, &mapB, kt * BKL, tok0, fb);
          tma_load_2d_pair(dst + MT * A_BYTES + T::BH, &mapB, kt * BKL + 64, tok0, fb);
#pragma unroll
          for (int m = 0; m < MT; ++m)
            tma_load_2d_pair(dst + T::E + m * E_BYTES, &mapE, 0, ((2 * (MT * mt + m) + (int)rank) * p.k_tiles + kt) * 128, fb);
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      // tail: the MMAs that read the stages issued last have finished (their commits reach both CTAs), so
      // nothing is in flight towards this CTA's shared memory when it leaves
      for (int back = 1; back <= STAGES && back <= issued; ++back) {
        int s = stage - back; uint32_t ph = phase;
        if (s < 0) { s += STAGES; ph ^= 1; }
        const long long t0 = clock64();
        while (!mbar_try(empty0 + 8 * s, ph) && clock64() - t0 < (ok ? WAIT_CYCLES : 20000000ll)) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA only)
    if (lane == 0 && rank == 0) {
      const uint64_t da0 = smem_desc_k(smem_u32(smem)), db0 = smem_desc_k(smem_u32(smem) + MT * A_BYTES), de0 = smem_desc_e(smem_u32(smem) + T::E);
      const uint32_t idesc = instr_desc_sp_pair(p.tile_n);
      int stage = 0; uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs, ++local) {
        if (!mbar_wait_cluster(tempty, ((uint32_t)local & 1u) ^ 1u, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
        for (int kt = 0; kt < p.k_tiles; ++kt) {
          if (!mbar_wait_cluster(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint64_t off = (uint64_t)(uint32_t)(stage * (T::STAGE >> 4));
          const uint32_t meta = tmem_base + T::META + (uint32_t)(4 * MT * stage);
#pragma unroll
          for (int m = 0; m < MT; ++m) tmem_cp_e_pair(meta + 4 * m, de0 + off + (uint64_t)(m * (E_BYTES >> 4)));
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              umma_bf16_sp_pair(tmem_base + m * T::MAX_N, da0 + off + (uint64_t)(m * (A_BYTES >> 4) + 2 * j),
                                db0 + off + (uint64_t)((j >> 1) * (T::BH >> 4) + 4 * (j & 1)), meta + 4 * m + (j & 2), idesc | (uint32_t)(j & 1),
                                (uint32_t)((kt > 0) | (j != 0)));
          umma_commit_pair(empty0 + 8 * stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
        if (ok) umma_commit_pair(tfull);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps (both CTAs)
    const int q = warp & 3, m = (warp - 2) >> 2;                 // lane quarter, row tile
    const uint32_t tempty_lead = map_to_cta(tempty, 0);
    int local = 0;
    bool ok = true;
    for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs, ++local) {
      int mt, nt;
        tile_to_mn(tile, m_groups, p.n_tiles, mt, nt);
      if (!mbar_wait(tfull, (uint32_t)local & 1u, abortp, p.status)) { ok = false; break; }
      tc_fence_after();
      // (trip count and row in constants where they are: with p.tile_n / 32 a tile of 256 took 3 us longer)
      const int64_t row = (int64_t)(MT * mt + (MT == 1 ? 0 : m)) * 256 + rank * 128 + q * 32 + lane;
#pragma unroll 1
      for (int ch = 0; ch < T::MAX_N / 32; ++ch) {
        if (MT > 1 && ch * 32 >= p.tile_n) break;
        uint32_t r[32];
        tmem_ld32(tmem_base + (uint32_t)(m * T::MAX_N + ch * 32) + ((uint32_t)(q * 32) << 16), r);
        store_chunk(p, r, row, (int64_t)nt * (MT == 1 ? T::MAX_N : p.tile_n) + ch * 32, lane);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty_lead);
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                       // neither CTA leaves while its partner may still signal it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------------------
// The same product for few tokens (a tile of BNS, or some of 128), where reading S is the whole cost and the tiles
// above leave most of the chip idle (one 256 x 256 tile per pair: 32 of 148 SMs at 4096 x 4096, 21 us).  The contraction
// is cut into pieces so that (row tiles) x (pieces) fills two CTAs per SM; a CTA keeps up to 72 KiB of S in flight, sums
// its piece in tensor memory and writes it as fp32, and the kernel that multiplies with A adds the pieces in a fixed
// order (fwd_small_kernel).  S does not depend on the kernel before: its first stages are requested before the wait for
// that kernel's z1 (programmatic dependent launch).
template <int BNS>
struct SmallN {
  static constexpr int BH = BNS * 64 * 2;                       // one half (64 k) of the Z1 stage
  static constexpr int STAGE = A_BYTES + 2 * BH + E_BYTES;
  static constexpr int STAGES = BNS <= 32 ? 4 : (BNS == 64 ? 3 : 2);   // two CTAs share an SM's shared memory
  static constexpr uint32_t COLS = BNS <= 32 ? 64 : (BNS == 64 ? 128 : 256);   // accumulator, then 4 columns per stage
  static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024;
};

template <int BNS>
__global__ void __launch_bounds__(NTHREADS, 2)
tc_sparse_small_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                       const __grid_constant__ CUtensorMap mapE, const SParams p, int k_per_piece) {
  using T = SmallN<BNS>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * T::STAGES + 1];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[T::STAGES]), tfull = smem_u32(&bars[2 * T::STAGES]);
  const int mt = blockIdx.x;
  const int k0 = blockIdx.y * k_per_piece, k1 = min(p.k_tiles, k0 + k_per_piece);
  const int tok0 = BNS == 128 ? blockIdx.z * BNS : 0;                 // (only a tile of 128 has others beside it)

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < T::STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    mbar_init(tfull, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(T::COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_launch_dependents();
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    if (lane == 0) {
      auto load_s = [&](int kt, int stage) {
        const uint32_t dst = smem_u32(smem + (size_t)stage * T::STAGE), fb = full0 + 8 * stage;
        mbar_expect_tx(fb, T::STAGE);
        tma_load_2d(dst, &mapA, kt * 64, mt * BM, fb);
        tma_load_2d(dst + A_BYTES + 2 * T::BH, &mapE, 0, (mt * p.k_tiles + kt) * 128, fb);
      };
      auto load_z = [&](int kt, int stage) {
        const uint32_t dst = smem_u32(smem + (size_t)stage * T::STAGE) + A_BYTES, fb = full0 + 8 * stage;
        tma_load_2d(dst, &mapB, kt * BKL, tok0, fb);
        tma_load_2d(dst + T::BH, &mapB, kt * BKL + 64, tok0, fb);
      };
      const int pre = min(T::STAGES, k1 - k0);
      for (int i = 0; i < pre; ++i) load_s(k0 + i, i);
      grid_dependency_wait();
      for (int i = 0; i < pre; ++i) load_z(k0 + i, i);
      int stage = pre % T::STAGES; uint32_t phase = pre == T::STAGES ? 1 : 0;
      long long issued = pre;
      bool ok = true;
      for (int kt = k0 + pre; kt < k1; ++kt) {
        if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
        load_s(kt, stage);
        load_z(kt, stage);
        ++issued;
        if (++stage == T::STAGES) { stage = 0; phase ^= 1; }
      }
      if (!ok) {
        for (int back = 1; back <= T::STAGES && back <= issued; ++back) {
          int s = stage - back; uint32_t ph = phase;
          if (s < 0) { s += T::STAGES; ph ^= 1; }
          const long long t0 = clock64();
          while (!mbar_try(full0 + 8 * s, ph) && clock64() - t0 < 20000000ll) {}
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = (instr_desc_sp(0) & ~(0x3Fu << 17)) | ((uint32_t)(BNS >> 3) << 17);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int kt = k0; kt < k1; ++kt) {
        if (!mbar_wait(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + (size_t)stage * T::STAGE);
        const uint32_t sb = sa + A_BYTES;
        const uint32_t meta = tmem_base + BNS + (uint32_t)(4 * stage);
        tmem_cp_e(meta, smem_desc_e(sb + 2 * T::BH));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t da = smem_desc_k(sa + j * 32);
          const uint64_t dbm = smem_desc_k(sb + (j >> 1) * T::BH + (j & 1) * 64);
          umma_bf16_sp(tmem_base, da, dbm, meta + (uint32_t)(j & ~1), idesc | (uint32_t)(j & 1), (uint32_t)((kt > k0) | (j != 0)));
        }
        umma_commit(empty0 + 8 * stage);
        if (++stage == T::STAGES) { stage = 0; phase ^= 1; }
      }
      if (ok) umma_commit(tfull);
    }
  } else {
    const int q = warp & 3;
    if (mbar_wait(tfull, 0, abortp, p.status)) {
      tc_fence_after();
      const int64_t row = (int64_t)mt * BM + q * 32 + lane;
      float* Z = p.Z + ((int64_t)blockIdx.y * p.N + tok0) * p.ldz + row;          // this piece's sums, [tokens][d_out]
#pragma unroll 1
      for (int ch = 0; ch < BNS / 16; ++ch) {
        uint32_t r[16];
        tmem_ld16(tmem_base + (uint32_t)(ch * 16) + ((uint32_t)(q * 32) << 16), r);
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (tok0 + ch * 16 + i < p.N) Z[(int64_t)(ch * 16 + i) * p.ldz] = __uint_as_float(r[i]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(T::COLS) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------------------
// The fp32-grade product with the 2:4 core (the core product of the fp32 forward): both operands as fp16 high and low parts
// of rows scaled by powers of two (split_f16.cu), three sparse MMAs lo*hi + hi*lo + hi*hi per 32 of k where the dense product issues
// six.  Same pairs of CTAs as above; differences:
//   * 128 k of a stage are 32 KiB of kept values, up to 56 KiB of z1 and 2 KiB of positions, so there are two stages;
//   * tiles of 256 rows of S by tile_n <= 224 tokens, so that two accumulators and the positions fit tensor memory: the sums of
//     a segment of the contraction leave for the epilogue warps' registers while the next segment runs.  The host picks the tile_n that
//     fills the last wave best;
//   * a core that is not 2:4 is left to the dense product, which is launched behind this one: *dense says so.
// Segments of 1,024 columns as in the dense product, which are half as many truncating additions here (whole forward 4.0e-6 off fp64
// sums where the dense core was 5.8e-6; segments of 2,048 6.1e-6, at the same speed).
// What bounds it: the sparse tensor cores under the power cap, and at the burst clock what L2 delivers (90 KiB per SM and stage).
// 4096 x 4096, 8,195 tokens: 325 us where the dense product takes 525 (846 TFLOP/s of fp32-grade products, dense-equivalent).
constexpr int S3_MAX_N = 224, S3_STAGES = 2, S3_THREADS = 320, S3_SEG = 8;      // segment: stages of 128 columns
constexpr uint32_t S3_META = 2 * S3_MAX_N;
constexpr int S3_B = 2 * A_BYTES, S3_E = S3_B + 4 * BH_BYTES, S3_STAGE = S3_E + E_BYTES;

struct S3Params {
  float* Z; int64_t ldz;                            // [tokens][d_out]
  int64_t N;                                        // tokens
  int m_pairs, n_tiles, k_tiles, tile_n;            // tiles of 256 rows of S, tiles of tile_n tokens, k tiles of 128
  const float* row_scale;                           // per row of S, per token
  const float* tok_scale;
  const int32_t* dense;                             // not 0: the dense product runs instead
  int32_t* status;
};

__global__ void __launch_bounds__(S3_THREADS, 1)
tc_sparse3_pair_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapAlo,
                       const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBlo,
                       const __grid_constant__ CUtensorMap mapE, const S3Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * S3_STAGES + 4];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[S3_STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * S3_STAGES]), tempty0 = smem_u32(&bars[2 * S3_STAGES + 2]);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int half_n = p.tile_n / 2;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < S3_STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(tfull0 + 8 * s, 1); mbar_init(tempty0 + 8 * s, 16); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                       // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  grid_begin();                                             // (tensor memory is this CTA's before the next kernel's CTAs start)
  const int n_tiles_total = *p.dense != 0 ? 0 : p.m_pairs * p.n_tiles;
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      bool ok = true;
      const int stage_bytes = 2 * A_BYTES + 4 * half_n * 128 + E_BYTES;
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs) {
        int mt, nt;
        tile_to_mn(tile, p.m_pairs, p.n_tiles, mt, nt);
        const int row0 = mt * 256 + (int)rank * 128, tok0 = nt * p.tile_n + (int)rank * half_n;
        for (int kt = 0; kt < p.k_tiles; ++kt) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
          if (rank == 0) mbar_expect_tx(full0 + 8 * stage, 2 * stage_bytes);
          const uint32_t fb = map_to_cta(full0 + 8 * stage, 0);
          const uint32_t dst = smem_u32(smem + (size_t)stage * S3_STAGE);
          tma_load_2d_pair(dst, &mapA, kt * 64, row0, fb);
          tma_load_2d_pair(dst + A_BYTES, &mapAlo, kt * 64, row0, fb);
          tma_load_2d_pair(dst + S3_B, &mapB, kt * BKL, tok0, fb);
          tma_load_2d_pair(dst + S3_B + BH_BYTES, &mapB, kt * BKL + 64, tok0, fb);
          tma_load_2d_pair(dst + S3_B + 2 * BH_BYTES, &mapBlo, kt * BKL, tok0, fb);
          tma_load_2d_pair(dst + S3_B + 3 * BH_BYTES, &mapBlo, kt * BKL + 64, tok0, fb);
          tma_load_2d_pair(dst + S3_E, &mapE, 0, ((2 * mt + (int)rank) * p.k_tiles + kt) * 128, fb);
          ++issued;
          if (++stage == S3_STAGES) { stage = 0; phase ^= 1; }
        }
      }
      // tail: the MMAs that read the stages issued last have finished (their commits reach both CTAs), so
      // nothing is in flight towards this CTA's shared memory when it leaves
      for (int back = 1; back <= S3_STAGES && back <= issued; ++back) {
        int s = stage - back; uint32_t ph = phase;
        if (s < 0) { s += S3_STAGES; ph ^= 1; }
        const long long t0 = clock64();
        while (!mbar_try(empty0 + 8 * s, ph) && clock64() - t0 < (ok ? WAIT_CYCLES : 20000000ll)) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA only)
    if (lane == 0 && rank == 0) {
      // fp16 operands, fp32 sums, M = 256, N = tile_n, sparse A
      const uint32_t idesc = (1u << 2) | (1u << 4) | ((uint32_t)(p.tile_n >> 3) << 17) | (uint32_t)(256 >> 4) << 24;
      const uint64_t d0 = smem_desc_k(smem_u32(smem)), e0 = smem_desc_e(smem_u32(smem) + S3_E);
      int stage = 0; uint32_t phase = 0;
      int local = 0;                                        // (tile, segment) items so far: selects the accumulator
      bool ok = true;
      for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs) {
        for (int f0 = 0; f0 < p.k_tiles && ok; f0 += S3_SEG, ++local) {
          const int as = local & 1;
          if (!mbar_wait_cluster(tempty0 + 8 * as, ((uint32_t)(local >> 1) & 1u) ^ 1u, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tacc = tmem_base + (uint32_t)(as * S3_MAX_N);
          const int f1 = min(p.k_tiles, f0 + S3_SEG);
          for (int f = f0; f < f1; ++f) {
            if (!mbar_wait_cluster(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint64_t so = (uint64_t)(uint32_t)(stage * (S3_STAGE >> 4));
            const uint32_t meta = tmem_base + S3_META + (uint32_t)(4 * stage);
            tmem_cp_e_pair(meta, e0 + so);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint64_t da = d0 + so + j * (32 >> 4), dal = da + (A_BYTES >> 4);
              const uint64_t dbm = d0 + so + ((S3_B + (j >> 1) * BH_BYTES + (j & 1) * 64) >> 4), dbl = dbm + ((2 * BH_BYTES) >> 4);
              const uint32_t id = idesc | (uint32_t)(j & 1), ecol = meta + (uint32_t)(j & ~1);
              umma_bf16_sp_pair(tacc, dal, dbm, ecol, id, (uint32_t)((f > f0) | (j != 0)));
              umma_bf16_sp_pair(tacc, da, dbl, ecol, id, 1u);
              umma_bf16_sp_pair(tacc, da, dbm, ecol, id, 1u);
            }
            umma_commit_pair(empty0 + 8 * stage);
            if (++stage == S3_STAGES) { stage = 0; phase ^= 1; }
          }
          if (ok) umma_commit_pair(tfull0 + 8 * as);
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps (both CTAs)
    // warp w: rows 32 (w % 4) .. of S, one of the two halves of the tile's tokens, one running sum per token and lane
    const int q = warp & 3, half = (warp - 2) >> 2;
    int local = 0;
    bool ok = true;
    for (int tile = pair; tile < n_tiles_total && ok; tile += n_pairs) {
      int mt, nt;
      tile_to_mn(tile, p.m_pairs, p.n_tiles, mt, nt);
      float acc[128];
#pragma unroll
      for (int i = 0; i < 128; ++i) acc[i] = 0.f;
      for (int f0 = 0; f0 < p.k_tiles && ok; f0 += S3_SEG, ++local) {
        const int as = local & 1;
        if (!mbar_wait(tfull0 + 8 * as, (uint32_t)(local >> 1) & 1u, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          if (ch * 32 >= half_n) continue;                  // uniform; columns past the half are not stored
          uint32_t r[32];
          tmem_ld32(tmem_base + (uint32_t)(as * S3_MAX_N + half * half_n + ch * 32) + ((uint32_t)(q * 32) << 16), r);
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[ch * 32 + i] += __uint_as_float(r[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_cta(tempty0 + 8 * as, 0));
      }
      if (!ok) break;
      const int64_t row = (int64_t)mt * 256 + rank * 128 + q * 32 + lane;
      const int64_t tok0 = (int64_t)nt * p.tile_n + half * half_n;
      const int left = (int)(p.N - tok0 < half_n ? p.N - tok0 : half_n);
      const float rs = p.row_scale[row];
      float* out = p.Z + tok0 * p.ldz + row;
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        if (ch * 32 >= left) continue;
        const float ts = ch * 32 + lane < left ? p.tok_scale[tok0 + ch * 32 + lane] : 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const float t = __shfl_sync(0xffffffffu, ts, i);
          if (ch * 32 + i < left) out[(int64_t)(ch * 32 + i) * p.ldz] = acc[ch * 32 + i] * t * rs;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                       // neither CTA leaves while its partner may still signal it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// One thread per 32-bit word of positions: 2 rows x 16 k.  Writes the word and the eight pairs of kept values.
// A group whose mask byte keeps fewer than two positions is padded with unkept positions (their values are
// written as zeros); more than two kept positions cannot be represented: the first two are taken and the
// status word counts the group.
__global__ void __launch_bounds__(256)
compress_24_kernel(const float* __restrict__ S, const uint8_t* __restrict__ Mk, __nv_bfloat16* __restrict__ Sc,
                   uint32_t* __restrict__ E, int64_t d_out, int64_t d_in, int32_t* status) {
  const int64_t k_tiles = d_in / 128;
  const int64_t n_words = d_out * (d_in / 32);          // (d_out / 128) * k_tiles * 128 * 4
  const int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (w >= n_words) return;
  const int k2 = (int)(w & 3), l = (int)((w >> 2) & 127);
  const int64_t blk = w >> 9;
  const int64_t kt = blk % k_tiles, mt = blk / k_tiles;
  const int m0 = l & 7, k1 = (l >> 3) & 1, m2 = l >> 4;
  const int64_t kbase = kt * 128 + k2 * 32 + k1 * 16;
  uint32_t word = 0;
  int bad = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t row = mt * 128 + m0 + 16 * m2 + 8 * h;
#pragma unroll
    for (int qd = 0; qd < 4; ++qd) {
      const int64_t g = kbase / 4 + qd;
      const unsigned m = Mk[row * (d_in / 4) + g] & 15u;
      const float4 v = *reinterpret_cast<const float4*>(S + row * d_in + 4 * g);
      const float vals[4] = {v.x, v.y, v.z, v.w};
      int i0 = -1, i1 = -1, cnt = 0;
#pragma unroll
      for (int pidx = 0; pidx < 4; ++pidx)
        if ((m >> pidx) & 1u) { if (cnt == 0) i0 = pidx; else if (cnt == 1) i1 = pidx; ++cnt; }
      if (cnt > 2) bad = 1;
      if (cnt < 2) {                                   // pad with unkept positions, keeping i0 < i1
        if (cnt == 0) { i0 = 0; i1 = 1; }
        else if (i0 < 3) i1 = i0 + 1;
        else { i1 = 3; i0 = 2; }
      }
      const float a = ((m >> i0) & 1u) ? vals[i0] : 0.f, b = ((m >> i1) & 1u) ? vals[i1] : 0.f;
      __nv_bfloat162 pr;
      pr.x = __float2bfloat16(a);
      pr.y = __float2bfloat16(b);
      *reinterpret_cast<__nv_bfloat162*>(Sc + row * (d_in / 2) + 2 * g) = pr;
      word |= (uint32_t)(i0 | (i1 << 2)) << (16 * h + 4 * qd);
    }
  }
  E[w] = word;
  if (bad) atomicAdd(&status[ST_SPARSE_BAD_GROUPS], 1);
}

bool make_map_16(CUtensorMap* map, const void* base, int64_t rows, int64_t K, int64_t ld, int box_rows, CUtensorMapDataType type) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, type, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
bool make_map_bf16(CUtensorMap* map, const void* base, int64_t rows, int64_t K, int64_t ld, int box_rows = 128) {
  return make_map_16(map, base, rows, K, ld, box_rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
}

bool make_map_e(CUtensorMap* map, const void* base, int64_t rows);

template <int BNS>
armor_status launch_small(armor_ctx* c, const void* Sc, const void* E, const void* z1, SParams p, int pieces, int per,
                          cudaStream_t s) {
  CUtensorMap mA, mB, mE;
  if (!make_map_bf16(&mA, Sc, c->d_out, c->d_in / 2, c->d_in / 2)) return ARMOR_ERR_CUDA;
  if (!make_map_bf16(&mB, z1, p.N, c->d_in, c->d_in, BNS)) return ARMOR_ERR_CUDA;
  if (!make_map_e(&mE, E, (c->d_out / 128) * (c->d_in / 128) * 128)) return ARMOR_ERR_CUDA;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_sparse_small_kernel<BNS>, SmallN<BNS>::SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  KTimer kt(c, ARMOR_KC_GEMM, 2.0 * (double)p.M * (double)p.N * (double)p.K, s);   // dense-equivalent flops
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)p.m_tiles, (unsigned)pieces, (unsigned)p.n_tiles); cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = SmallN<BNS>::SMEM; cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, tc_sparse_small_kernel<BNS>, mA, mB, mE, p, per) != cudaSuccess) return ARMOR_ERR_CUDA;
  c->launches++;
  return ARMOR_OK;
}

// positions: [rows of 16 bytes], box = 128 rows, no swizzle
bool make_map_e(CUtensorMap* map, const void* base, int64_t rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {4, (cuuint64_t)rows};
  cuuint64_t strides[1] = {16};
  cuuint32_t box[2] = {4, 128};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

bool tc_sparse_ok(const armor_ctx* c) {
  return c->cfg.n_keep == 2 && c->cfg.m_group == 4 && c->d_out % 128 == 0 && c->d_in % 128 == 0 &&
         c->cfg.precision != ARMOR_PREC_SIMT;
}

size_t tc_sparse_values_bytes(const armor_ctx* c) { return (size_t)c->d_out * (size_t)c->d_in; }   // bf16, half the entries

void launch_compress_24(armor_ctx* c, const float* S, const uint8_t* M, void* Sc, void* E, cudaStream_t s) {
  const int64_t n_words = c->d_out * (c->d_in / 32);
  KTimer kt(c, ARMOR_KC_FORWARD, (double)c->wn * 5.125, s);
  compress_24_kernel<<<(unsigned)((n_words + 255) / 256), 256, 0, s>>>(S, M, static_cast<__nv_bfloat16*>(Sc),
                                                                        static_cast<uint32_t*>(E), c->d_out, c->d_in,
                                                                        c->status);
  c->launches++;
}

// The product on pairs of CTAs, MT row tiles of 256 to a stage's tokens, tiles of tile_n tokens
template <int MT>
static armor_status launch_pairs(armor_ctx* c, const CUtensorMap& mA, const void* z1, const CUtensorMap& mE, SParams p, int tile_n, cudaStream_t s) {
  CUtensorMap mB;
  if (!make_map_bf16(&mB, z1, p.N, p.K, p.K, tile_n / 2)) return ARMOR_ERR_CUDA;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_sparse_pair_kernel<MT>, PairN<MT>::SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  p.tile_n = tile_n;
  p.n_tiles = (int)((p.N + tile_n - 1) / tile_n);
  const int tiles = p.m_tiles / (2 * MT) * p.n_tiles, pairs = tiles < c->n_sm / 2 ? tiles : c->n_sm / 2;
  // (a dependent launch: 4096 x 4096, 400 tokens 26.8 -> 24.9 us a forward)
  launch_dependent(tc_sparse_pair_kernel<MT>, 2 * pairs, PairN<MT>::THREADS, PairN<MT>::SMEM, LaunchStream(s, false, 2), mA, mB, mE, p);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

// Z2[n][d_out] = Z1[n][d_in] * S^T with S given compressed (Sc, E); Z1 bf16; Z2 fp32, or bf16 if out_bf16.
armor_status launch_tc_sparse(armor_ctx* c, const void* Sc, const void* E, const void* z1_bf16, void* z2, bool out_bf16,
                              int64_t n, cudaStream_t s) {
  if (!tc_sparse_ok(c) || n <= 0) return ARMOR_ERR_UNSUPPORTED;
  CUtensorMap mA, mE;
  if (!make_map_bf16(&mA, Sc, c->d_out, c->d_in / 2, c->d_in / 2)) return ARMOR_ERR_CUDA;
  if (!make_map_e(&mE, E, (c->d_out / 128) * (c->d_in / 128) * 128)) return ARMOR_ERR_CUDA;
  SParams p{};
  p.Z = out_bf16 ? nullptr : static_cast<float*>(z2); p.Zb = out_bf16 ? static_cast<__nv_bfloat16*>(z2) : nullptr;
  p.ldz = c->d_out; p.M = c->d_out; p.N = n; p.K = c->d_in;
  p.m_tiles = (int)(c->d_out / BM); p.n_tiles = (int)((n + BN - 1) / BN); p.k_tiles = (int)(c->d_in / BKL);
  p.status = c->status;
  const int n_sm = c->n_sm;
  KTimer kt(c, ARMOR_KC_GEMM, 2.0 * (double)p.M * (double)p.N * (double)p.K, s);   // dense-equivalent flops
  if (c->d_out % 256 == 0 && n_sm >= 2) {
    // Two row tiles at a time, or one: rounds of the pairs times what a tile takes, its tokens plus, with two, 200 tokens' worth (a tile
    // of 512 x 224 takes 1.62 times one of 256 x 256, of 512 x 192 1.48 times), 240 with the output in fp32: 14336 x 2048, 1,459 tokens, 3
    // rounds of two or 5 of one, 149 us and 144 a forward with fp32 wrappers.  Whole forwards, one and two: 28672 x 8192, 4,096 tokens
    // (25 rounds and 15) 1,192 and 1,123 us; 8192 x 8192, 640 (2 and 1) 76.5 and 63.2, 2,000 (4 and 2) 156 and 139; 4096 x 4096, 4,096
    // (4 and 3) 93 and 107: one.
    int width = 256;
    if (c->d_out % 512 == 0) {
      const int pairs = n_sm / 2;
      int64_t least = (p.m_tiles / 2 * ((n + 255) / 256) + pairs - 1) / pairs * 262;
      for (int w = PairN<2>::MAX_N; w >= 128; w -= 32) {
        const int64_t cost = (p.m_tiles / 4 * ((n + w - 1) / w) + pairs - 1) / pairs * (w + (out_bf16 ? 200 : 240));
        if (cost < least) { least = cost; width = w; }
      }
    }
    if (width < 256) return launch_pairs<2>(c, mA, z1_bf16, mE, p, width, s);
    return launch_pairs<1>(c, mA, z1_bf16, mE, p, 256, s);
  } else {
    CUtensorMap mB;
    if (!make_map_bf16(&mB, z1_bf16, n, c->d_in, c->d_in)) return ARMOR_ERR_CUDA;
    constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024;
    static PerDeviceOnce attr;
    if (ensure_dynamic_smem(attr, c->device, tc_sparse_kernel, SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
    const int tiles = p.m_tiles * p.n_tiles;
    const int grid = tiles < n_sm ? tiles : n_sm;
    tc_sparse_kernel<<<grid, NTHREADS, SMEM, s>>>(mA, mB, mE, p);
  }
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

// Zp[piece][n][d_out] = the pieces of Z1[n][d_in] * S^T (bf16 operands, fp32 sums), beyond 64 tokens in tiles of 128; their number
// goes to *pieces.  pieces * n <= 5 d_in, so Zp fits five W-shaped fp32 buffers.
armor_status launch_tc_sparse_small(armor_ctx* c, const void* Sc, const void* E, const void* z1_bf16, float* Zp, int64_t n,
                                    int* pieces, cudaStream_t s) {
  if (!tc_sparse_ok(c) || n <= 0 || n > 5 * c->d_in) return ARMOR_ERR_UNSUPPORTED;
  SParams p{};
  p.Z = Zp; p.ldz = c->d_out; p.M = c->d_out; p.N = n; p.K = c->d_in;
  p.m_tiles = (int)(c->d_out / BM); p.n_tiles = (int)((n + 127) / 128); p.k_tiles = (int)(c->d_in / BKL);
  p.status = c->status;
  // Pieces of a row (and token) tile.  Two CTAs an SM keep most of S in flight, which a large core needs (14336 x 4096, 37 tokens: 224 CTAs
  // 15.2 us a forward, 112 18.2; 8192 x 8192 256 19.4, 128 25).  A small one is bound by latency, 0.3 us a k tile and 0.1 us a
  // piece to be written and added: one CTA an SM, one SM in twelve with two, while that leaves a CTA about eight k tiles (4096 x
  // 4096, 256 -> 160 CTAs: 1 token 8.98 -> 8.2 us, 64 10.9 -> 9.3; 2048 x 2048, 256 -> 128: 7.7 -> 6.5 and 10.4 -> 7.8; beyond 64
  // tokens, two stages a CTA: five k tiles), and no fewer k tiles than make those two costs alike (512 x 8192, 64 -> 13 pieces:
  // 14.3 -> 8.2 us).  From 40 row tiles on fewer pieces are worth their longer chains only where the pieces are large, from 25 tokens
  // on (6144 x 2048, two CTAs an SM and one: 1 token 7.7 and 8.0 us, 17 9.1 and 9.7, 64 9.7 and 8.8; 5120 x 2560, 8 tokens 7.8 and 8.2,
  // 64 10.3 and 9.4; 7168 x 2048 in blocks of 256 33 10.6 and 10.9, 64 11.7 and 10.7).  Below 40 the one size seen to lose is 4096 x 2048, 1
  // token: 7.2 and 7.4.  The twelfth is for 32 row tiles (five
  // pieces; four of them, 128 CTAs, 8.7 us for 1 token at 4096 x 4096); 20 row tiles do without (2560 x 5120, 1 token 8.5, with seven pieces
  // for eight 8.2).
  int want = 2 * c->n_sm / (p.m_tiles * p.n_tiles);
  const int one_an_sm = (c->n_sm + c->n_sm / 12) / (p.m_tiles * p.n_tiles);
  const bool small = one_an_sm >= 2 && (n > 24 || p.m_tiles < 40) && (int64_t)p.m_tiles * p.n_tiles * p.k_tiles <= (int64_t)(n <= 64 ? 8 : 5) * c->n_sm;
  if (small) want = one_an_sm;
  if (want < 1) want = 1;
  if (want > p.k_tiles) want = p.k_tiles;
  if (want > 5 * p.K / n) want = (int)(5 * p.K / n);                 // what Zp holds
  int per = (p.k_tiles + want - 1) / want;
  while (3 * per * per < p.k_tiles) ++per;
  *pieces = (p.k_tiles + per - 1) / per;
  if (n <= 16) return launch_small<16>(c, Sc, E, z1_bf16, p, *pieces, per, s);
  // (a small core's tile of 32 tokens takes longer than one of 64, 4096 x 4096, 24 tokens 9.4 and 8.9 us; not for its stages nor its
  // place in tensor memory, and the reverse for a large one, 14336 x 4096 13.8 and 14.3)
  if (n <= 32 && !small) return launch_small<32>(c, Sc, E, z1_bf16, p, *pieces, per, s);
  if (n <= 64) return launch_small<64>(c, Sc, E, z1_bf16, p, *pieces, per, s);
  return launch_small<128>(c, Sc, E, z1_bf16, p, *pieces, per, s);
}

// Z2[n][d_out] = Z1[n][d_in] * S^T, fp32-grade: the parts of what S keeps (hi, lo, [d_out][d_in / 2] each) with their positions, z1's
// parts and the rows' scales; nothing if *dense.
bool tc_sparse3_ok(const armor_ctx* c) {
  return tc_sparse_ok(c) && c->cfg.precision == ARMOR_PREC_FP16X3 && c->d_out % 256 == 0 && c->n_sm >= 2;
}
armor_status launch_tc_sparse3(armor_ctx* c, const void* hi, const void* lo, const void* E, const float* row_scale, const void* zhi,
                               const void* zlo, const float* tok_scale, const int32_t* dense, float* z2, int64_t n, cudaStream_t s) {
  if (!tc_sparse3_ok(c) || n <= 0) return ARMOR_ERR_UNSUPPORTED;
  const int pairs = c->n_sm / 2;
  S3Params p{};
  p.Z = z2; p.ldz = c->d_out; p.N = n;
  p.m_pairs = (int)(c->d_out / 256); p.k_tiles = (int)(c->d_in / BKL);
  p.row_scale = row_scale; p.tok_scale = tok_scale; p.dense = dense; p.status = c->status;
  // the width of a tile that costs least: waves of tiles times what a tile takes, its MMAs (proportional to the width) plus what
  // comes with every tile whatever its width (S's share of the loads, the first stage, the last segment's way out: about 48 tokens' worth)
  int64_t least = 0;
  for (int w = S3_MAX_N; w >= 64; w -= 32) {
    const int64_t tiles = p.m_pairs * ((n + w - 1) / w), cost = (tiles + pairs - 1) / pairs * (w + 48);
    if (w == S3_MAX_N || cost < least) { least = cost; p.tile_n = w; }
  }
  p.n_tiles = (int)((n + p.tile_n - 1) / p.tile_n);
  CUtensorMap mA, mAlo, mB, mBlo, mE;
  const CUtensorMapDataType f16 = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  if (!make_map_16(&mA, hi, c->d_out, c->d_in / 2, c->d_in / 2, 128, f16)) return ARMOR_ERR_CUDA;
  if (!make_map_16(&mAlo, lo, c->d_out, c->d_in / 2, c->d_in / 2, 128, f16)) return ARMOR_ERR_CUDA;
  if (!make_map_16(&mB, zhi, n, c->d_in, c->d_in, p.tile_n / 2, f16)) return ARMOR_ERR_CUDA;
  if (!make_map_16(&mBlo, zlo, n, c->d_in, c->d_in, p.tile_n / 2, f16)) return ARMOR_ERR_CUDA;
  if (!make_map_e(&mE, E, (c->d_out / 128) * (c->d_in / 128) * 128)) return ARMOR_ERR_CUDA;
  constexpr size_t SMEM = (size_t)S3_STAGES * S3_STAGE + 1024;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_sparse3_pair_kernel, SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int tiles = p.m_pairs * p.n_tiles;
  KTimer kt(c, ARMOR_KC_GEMM, 2.0 * (double)c->d_out * (double)n * (double)c->d_in, s);   // dense-equivalent flops
  launch_dependent(tc_sparse3_pair_kernel, 2 * (tiles < pairs ? tiles : pairs), S3_THREADS, SMEM, LaunchStream(s, false, 2), mA, mAlo, mB, mBlo, mE, p);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}
