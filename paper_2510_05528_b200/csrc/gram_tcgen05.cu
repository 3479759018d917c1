// Per-block Grams of the wrapper updates on the tensor cores: G_i = P_i T_i^T over the row-blocks (contraction over d_in) and
// C_j = U_j^T Y_j over the column-blocks (contraction over d_out), 128 x 128 tiles of the block, long contractions.
//
//   MODE 0: one product           C = A.B
//   MODE 1: two products, one N side   C = A.B, C2 = A2.B          (A-step: P and E H against T)
//   MODE 2: an operand with itself     C = A.A, C2 = A.B           (B-step: U with itself and with E H; d_block 128)
//
// Three tf32 MMAs per k-step (low.high, high.low, high.high; the raw fp32 word is the high part, x - trunc_tf32(x) the low one)
// in the order of the streaming kernel of block_tcgen05.cu, so the same bits.
//
// What bounds it: the M-side and N-side operands of a 128 x 128 x 8 instruction are 8 KiB, the whole bandwidth of shared memory
// at the instruction's 65 cycles, and beside them the chunks come in, are read for their low parts and these are written: a
// chunk of 32 along k of the pair with a shared N side takes 2.6 k cycles of shared memory against 1.6 k of MMAs and 2.1 k of
// HBM.  So the M side goes to TENSOR MEMORY: the warps that form its low part put both parts there (lane = row, a column per
// k) and its raw chunk is free at once.  That leaves 1.6 k cycles of shared memory.  M and N sides come through rings of their
// own, so that as many chunks as fit are under way: 96 KiB of 224 (the streaming kernel had one stage of 48 in flight).
// With the streaming kernel / here, slabs added: 4096 x 4096 both pairs 59.7 / 47.4 us on average, one product 36.4 / 28.1;
// 14336 x 4096 183 / 151; 1024 x 5120, A-step 31.1 / 21.0.
//
// Persistent kernel; warps: 0 TMA producer, 1 MMA issuer, then groups of four: M side to tensor memory, MODE 1 the second M side
// likewise, low part of each N side, and the epilogue (tcgen05.ld, staging box, TMA store).  Tensor memory: accumulators 0..127,
// 128..255; two stages of M-side parts (32 columns high, 32 low for each operand) from 256.
// Every wait is bounded; a wait that runs out raises a status word and the CTA leaves through the common exit.
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int TILE = 128, BK = 32;
constexpr int OP_BYTES = TILE * BK * 4;           // 16 KiB: one operand chunk
constexpr uint32_t TMEM_COLS = 512, T_A = 256;
constexpr int EPI_BYTES = 2 * 32 * 32 * 4;        // per epilogue warp: two swizzled 32 x 32 boxes, used in turn
constexpr int AST = 2;                            // stages of M-side parts in tensor memory

template <int MODE> struct Geo {
  static constexpr int MS = MODE == 0 ? 1 : MODE == 1 ? 2 : 0;      // operands per stage of the M ring (MODE 2: read off the N ring)
  static constexpr int NS = MODE == 2 ? 2 : 1;                      // operands per stage of the N ring (MODE 2: A, B)
  static constexpr int STM = MODE == 0 ? 5 : MODE == 1 ? 3 : 1;
  static constexpr int STN = MODE == 0 ? 5 : 4;
  static constexpr int LST = 2;                                     // stages of low parts, NS chunks each
  static constexpr int TA = MODE == 1 ? 2 : 1;                      // M-side operands in tensor memory
  static constexpr int GROUPS = TA + NS + 1;                        // groups of four warps
  static constexpr int NT = 64 + 128 * GROUPS;
  static constexpr size_t N_OFF = (size_t)MS * STM * OP_BYTES, L_OFF = N_OFF + (size_t)NS * STN * OP_BYTES,
                          E_OFF = L_OFF + (size_t)NS * LST * OP_BYTES;
  static constexpr size_t SMEM = E_OFF + 4 * EPI_BYTES + 1024;
};

struct GParams {
  int mn_major;                     // 1: operands contiguous along M / N (contraction over rows), 0: along K
  int db;                           // rows (columns) of a block
  int m_tiles, n_tiles, batch, n_split, k_chunks;    // k_chunks: chunks of 32 along K per work item
  int64_t c_rows, c_cols;
  int64_t r_s;                      // rows of C between two slabs of the contraction
  int32_t* status;
};

__device__ __forceinline__ void item_decode(const GParams& p, int item, int& tn, int& tm, int& b, int& ks) {
  tn = item % p.n_tiles;
  tm = (item / p.n_tiles) % p.m_tiles;
  b = (item / (p.n_tiles * p.m_tiles)) % p.batch;
  ks = item / (p.n_tiles * p.m_tiles * p.batch);
}

// chunk kc of tile t of block b: K-major one box of 128 rows x 32 columns, MN-major four boxes of 32 x 32
__device__ __forceinline__ void load_chunk(uint32_t dst, const CUtensorMap* map, const GParams& p, int b, int t, int kc, uint32_t bar) {
  const int mn = p.db * b + TILE * t, k = BK * kc;
  if (p.mn_major) {
    tma_load_mn(dst, map, 1, mn, k, bar);
  } else {
    tma_load_2d(dst, map, k, mn, bar);
  }
}

__device__ __forceinline__ uint64_t chunk_desc(uint32_t base, int mn_major) {
  return mn_major ? smem_desc_mn_sw128_32b(base, 4096, 512) : smem_desc_sw128(base, 16, 1024);
}

__device__ __forceinline__ float low_part(float x) { return x - __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// position in a ring
struct Ring {
  int s; uint32_t ph;
  __device__ __forceinline__ void next(int n) { if (++s == n) { s = 0; ph ^= 1; } }
};

template <int MODE>
__global__ void __launch_bounds__(Geo<MODE>::NT, 1)
tc_gram_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapA2,
               const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapC,
               const __grid_constant__ CUtensorMap mapC2, const GParams p) {
  using G = Geo<MODE>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // full / empty of the two rings, ready / free of the low parts and of the M-side parts in tensor memory, accumulators
  __shared__ __align__(8) uint64_t bars[2 * G::STM + 2 * G::STN + 2 * G::LST + 2 * AST + 2];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const uint32_t fullM = smem_u32(&bars[0]), emptyM = fullM + 8 * G::STM;
  const uint32_t fullN = emptyM + 8 * G::STM, emptyN = fullN + 8 * G::STN;
  const uint32_t lready = emptyN + 8 * G::STN, lfree = lready + 8 * G::LST;
  const uint32_t aready = lfree + 8 * G::LST, afree = aready + 8 * AST;
  const uint32_t tfull = afree + 8 * AST, tempty = tfull + 8;
  const int n_items = p.batch * p.m_tiles * p.n_tiles * p.n_split;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < G::STM; ++s) { mbar_init(fullM + 8 * s, 1); mbar_init(emptyM + 8 * s, 4 * G::TA); }
    for (int s = 0; s < G::STN; ++s) { mbar_init(fullN + 8 * s, 1); mbar_init(emptyN + 8 * s, 1); }
    for (int s = 0; s < G::LST; ++s) { mbar_init(lready + 8 * s, 4 * G::NS); mbar_init(lfree + 8 * s, 1); }
    for (int s = 0; s < AST; ++s) { mbar_init(aready + 8 * s, 4 * G::TA); mbar_init(afree + 8 * s, 1); }
    mbar_init(tfull, 1);
    mbar_init(tempty, 4);
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
  grid_begin();                                     // (tensor memory is this CTA's before the next kernel's CTAs start)
  const uint32_t tmem_base = uniform(tmem_base_holder);
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      Ring m{0, 0}, n{0, 0};
      long long issued = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
        int tn, tm, b, ks;
        item_decode(p, item, tn, tm, b, ks);
        for (int kc = 0; kc < p.k_chunks; ++kc) {
          const int k = ks * p.k_chunks + kc;
          if (G::MS > 0) {
            if (!mbar_wait(emptyM + 8 * m.s, m.ph ^ 1, abortp, p.status)) { ok = false; break; }
            const uint32_t fb = fullM + 8 * m.s, dst = smem_u32(smem) + (uint32_t)(m.s * G::MS * OP_BYTES);
            mbar_expect_tx(fb, G::MS * OP_BYTES);
            load_chunk(dst, &mapA, p, b, tm, k, fb);
            if (MODE == 1) load_chunk(dst + OP_BYTES, &mapA2, p, b, tm, k, fb);
            m.next(G::STM);
          }
          // (the M-side load counts as issued only with its N side: after a failed wait both rings are drained below)
          if (!mbar_wait(emptyN + 8 * n.s, n.ph ^ 1, abortp, p.status)) { ok = false; break; }
          const uint32_t fb = fullN + 8 * n.s, dst = smem_u32(smem) + (uint32_t)(G::N_OFF + n.s * G::NS * OP_BYTES);
          mbar_expect_tx(fb, G::NS * OP_BYTES);
          if (MODE == 2) {
            load_chunk(dst, &mapA, p, b, tm, k, fb);
            load_chunk(dst + OP_BYTES, &mapB, p, b, tn, k, fb);
          } else {
            load_chunk(dst, &mapB, p, b, tn, k, fb);
          }
          ++issued;
          n.next(G::STN);
        }
      }
      if (!ok) {
        // leave no bulk copy in flight: wait (bounded) for the stages armed most recently
        auto drain = [&](uint32_t full, Ring r, int stages, long long armed) {
          for (int back = 0; back < stages && back < armed; ++back) {
            if (--r.s < 0) { r.s += stages; r.ph ^= 1; }
            const long long t0 = clock64();
            while (!mbar_try(full + 8 * r.s, r.ph) && clock64() - t0 < 20000000ll) {}
          }
        };
        drain(fullN, n, G::STN, issued);
        if (G::MS > 0) drain(fullM, m, G::STM, issued + 1);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    {
      const uint32_t leader = elect_lane();
      const uint32_t idesc = instr_desc_tf32_mn(TILE, TILE, 0, p.mn_major);    // (M side from tensor memory)
      // descriptors of stage 0: only their address field moves
      const uint64_t dn0 = chunk_desc(smem_u32(smem) + (uint32_t)G::N_OFF, p.mn_major);
      const uint64_t dl0 = chunk_desc(smem_u32(smem) + (uint32_t)G::L_OFF, p.mn_major);
      const uint64_t kinc = p.mn_major ? (1024u >> 4) : (32u >> 4);            // one k-step of 8 in the address field
      Ring n{0, 0}, l{0, 0}, a{0, 0};
      uint32_t local = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x, ++local) {
        if (!mbar_wait_warp(tempty, (local & 1u) ^ 1u, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
        for (int kc = 0; kc < p.k_chunks; ++kc) {
          if (!mbar_wait_warp(lready + 8 * l.s, l.ph, abortp, p.status)) { ok = false; break; }
          if (!mbar_wait_warp(aready + 8 * a.s, a.ph, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint64_t dn = dn0 + (uint64_t)(uint32_t)(n.s * G::NS * (OP_BYTES >> 4));
          const uint64_t dl = dl0 + (uint64_t)(uint32_t)(l.s * G::NS * (OP_BYTES >> 4));
          const uint32_t ta = tmem_base + T_A + (uint32_t)(a.s * G::TA * 64);
          const uint32_t first = (uint32_t)(kc > 0);
#pragma unroll
          for (int which = 0; which < (MODE == 0 ? 1 : 2); ++which) {
            const uint32_t hi = ta + (MODE == 1 ? 64u * which : 0u), lo = hi + 32u;
            const uint64_t d = dn + (MODE == 2 ? which * (OP_BYTES >> 4) : 0), dlo = dl + (MODE == 2 ? which * (OP_BYTES >> 4) : 0);
            const uint32_t acc = tmem_base + (uint32_t)(which * TILE);
#pragma unroll
            for (int k = 0; k < BK / 8; ++k) {
              if (k == 0) umma_tf32_ta_w(leader, acc, lo, d, idesc, first); else umma_tf32_ta_w(leader, acc, lo + 8 * k, d + k * kinc, idesc, 1u);
              umma_tf32_ta_w(leader, acc, hi + 8 * k, dlo + k * kinc, idesc, 1u);
              umma_tf32_ta_w(leader, acc, hi + 8 * k, d + k * kinc, idesc, 1u);
            }
          }
          umma_commit_w(leader, emptyN + 8 * n.s);
          umma_commit_w(leader, lfree + 8 * l.s);
          umma_commit_w(leader, afree + 8 * a.s);
          n.next(G::STN); l.next(G::LST); a.next(AST);
        }
        if (ok) umma_commit_w(leader, tfull);
      }
    }
  } else if (warp < 2 + 4 * G::TA) {
    // ------------------------------------------------------------ M side: raw chunk -> both parts in tensor memory
    const int g = (warp - 2) >> 2;                  // operand
    const int q = warp & 3;                         // TMEM lane quarter this warp may write
    const uint32_t lane_sel = (uint32_t)(q * 32) << 16;
    constexpr int ST = MODE == 2 ? G::STN : G::STM, SLOTS = MODE == 2 ? G::NS : G::MS;
    const uint32_t full = MODE == 2 ? fullN : fullM;
    const uint8_t* ring = smem + (MODE == 2 ? G::N_OFF : 0) + (size_t)g * OP_BYTES;
    Ring r{0, 0}, a{0, 0};
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x)
      for (int kc = 0; kc < p.k_chunks; ++kc) {
        if (!__all_sync(0xffffffffu, mbar_wait(full + 8 * r.s, r.ph, abortp, p.status))) { ok = false; break; }
        const uint8_t* src = ring + (size_t)r.s * SLOTS * OP_BYTES;
        uint32_t v[32];
        if (p.mn_major) {
          // element [k][m]: box q, row k, word `lane`; 32-byte atom c of a row sits at c ^ (row % 4)
          const uint8_t* box = src + q * 4096 + (lane & 7) * 4;
#pragma unroll
          for (int k = 0; k < 32; ++k) v[k] = *reinterpret_cast<const uint32_t*>(box + k * 128 + (((lane >> 3) ^ (k & 3)) << 5));
        } else {
          // row m = 32 q + lane, 16-byte chunk c sits at c ^ (row % 8)
          const uint8_t* rowp = src + (q * 32 + lane) * 128;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 w = *reinterpret_cast<const uint4*>(rowp + ((i ^ (lane & 7)) << 4));
            v[4 * i] = w.x; v[4 * i + 1] = w.y; v[4 * i + 2] = w.z; v[4 * i + 3] = w.w;
          }
        }
        if (MODE != 2) {
          __syncwarp();
          if (lane == 0) mbar_arrive(emptyM + 8 * r.s);
        }
        if (!__all_sync(0xffffffffu, mbar_wait(afree + 8 * a.s, a.ph ^ 1, abortp, p.status))) { ok = false; break; }
        tc_fence_after();
        const uint32_t dst = tmem_base + T_A + (uint32_t)(a.s * G::TA * 64 + g * 64) + lane_sel;
        tmem_st32(dst, v);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(low_part(__uint_as_float(v[i])));
        tmem_st32(dst + 32u, v);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(aready + 8 * a.s);
        r.next(ST); a.next(AST);
      }
  } else if (warp < 2 + 4 * (G::TA + G::NS)) {
    // ------------------------------------------------------------ N sides: low parts
    const int g = (warp - 2 - 4 * G::TA) >> 2;
    const int t = (threadIdx.x - 64) & 127;
    Ring n{0, 0}, l{0, 0};
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x)
      for (int kc = 0; kc < p.k_chunks; ++kc) {
        if (!mbar_wait(fullN + 8 * n.s, n.ph, abortp, p.status)) { ok = false; break; }
        const float4* hi = reinterpret_cast<const float4*>(smem + G::N_OFF + (size_t)(n.s * G::NS + g) * OP_BYTES);
        float4 v[OP_BYTES / 16 / 128];
#pragma unroll
        for (int e = 0; e < OP_BYTES / 16 / 128; ++e) v[e] = hi[t + e * 128];
        if (!mbar_wait(lfree + 8 * l.s, l.ph ^ 1, abortp, p.status)) { ok = false; break; }
        float4* lo = reinterpret_cast<float4*>(smem + G::L_OFF + (size_t)(l.s * G::NS + g) * OP_BYTES);
#pragma unroll
        for (int e = 0; e < OP_BYTES / 16 / 128; ++e)
          lo[t + e * 128] = make_float4(low_part(v[e].x), low_part(v[e].y), low_part(v[e].z), low_part(v[e].w));
        // make the generic-proxy writes visible to the tensor-core (async proxy) reads
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(lready + 8 * l.s);
        n.next(G::STN); l.next(G::LST);
      }
  } else {
    // ------------------------------------------------------------ epilogue: both accumulators as they are
    const int q = warp & 3;
    uint8_t* buf = smem + G::E_OFF + (size_t)q * EPI_BYTES;
    const uint32_t buf_u32 = smem_u32(buf);
    uint32_t local = 0;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++local) {
      int tn, tm, b, ks;
      item_decode(p, item, tn, tm, b, ks);
      const int row = (int)((int64_t)p.db * b + p.r_s * ks) + TILE * tm + 32 * q;
      if (!__all_sync(0xffffffffu, mbar_wait(tfull, local & 1u, abortp, p.status))) break;
      tc_fence_after();
#pragma unroll 1
      for (int box = 0; box < (MODE == 0 ? 4 : 8); ++box) {
        uint32_t r[32];
        tmem_ld32(tmem_base + (uint32_t)(32 * box) + ((uint32_t)(q * 32) << 16), r);
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the store before last has read this box
        __syncwarp();
        uint8_t* rowp = buf + (box & 1) * 4096 + lane * 128;
#pragma unroll
        for (int cq = 0; cq < 8; ++cq)
          *reinterpret_cast<uint4*>(rowp + ((cq ^ (lane & 7)) << 4)) = make_uint4(r[4 * cq], r[4 * cq + 1], r[4 * cq + 2], r[4 * cq + 3]);
        if (box == (MODE == 0 ? 3 : 7)) tc_fence_before();
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          if (box == (MODE == 0 ? 3 : 7)) mbar_arrive(tempty);
          tma_store_2d(box < 4 ? &mapC : &mapC2, TILE * tn + 32 * (box & 3), row, buf_u32 + (box & 1) * 4096);
          tma_store_commit();
        }
      }
    }
    if (lane == 0) tma_store_wait_read();           // shared memory stays valid until the stores have read it
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

template <int MODE>
armor_status launch(armor_ctx* c, const float* A, const float* A2, const float* B, float* C, float* C2, const GParams& p, cudaStream_t s) {
  using G = Geo<MODE>;
  CUtensorMap mA, mA2, mB, mC, mC2;
  int wide = 0;                                     // (d_in is a multiple of 128: always 1)
  auto op_map = [&](CUtensorMap* m, const float* at) {
    return p.mn_major ? make_map_mn(m, at, c->d_in, c->d_out, c->d_in, &wide) : make_map_2d(m, at, c->d_in, c->d_out, c->d_in, 32, TILE);
  };
  if (!op_map(&mA, A) || !op_map(&mB, B) || !make_map_2d(&mC, C, p.c_cols, p.c_rows, p.c_cols, 32, 32)) return ARMOR_ERR_CUDA;
  mA2 = mA;
  mC2 = mC;
  if (MODE == 1 && !op_map(&mA2, A2)) return ARMOR_ERR_CUDA;
  if (MODE != 0 && !make_map_2d(&mC2, C2, p.c_cols, p.c_rows, p.c_cols, 32, 32)) return ARMOR_ERR_CUDA;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_gram_kernel<MODE>, G::SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int64_t n_items = (int64_t)p.batch * p.m_tiles * p.n_tiles * p.n_split;
  const int grid = (int)(n_items < c->n_sm ? n_items : c->n_sm);
  KTimer kt(c, ARMOR_KC_BLOCK_GRAM, (MODE == 1 ? 12.0 : 8.0) * (double)c->wn, s);    // W-shaped operands read once each
  launch_dependent(tc_gram_kernel<MODE>, grid, G::NT, G::SMEM, s, mA, mA2, mB, mC, mC2, p);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

}  // namespace

// A and B are W-shaped; C (and C2) [n_split][blocks][db][db].  by_rows: G_i = A_i B_i^T over the row-blocks, else
// C_j = A_j^T B_j over the column-blocks.  A2: second M side (C2 = A2.B); self: C = A.A, C2 = A.B (d_block 128).
armor_status tc_gram_launch(armor_ctx* c, const float* A, const float* A2, const float* B, bool by_rows, bool self, float* C, float* C2,
                            int n_split, cudaStream_t s) {
  GParams p{};
  p.mn_major = by_rows ? 0 : 1;
  p.db = c->db;
  p.batch = by_rows ? c->nbo : c->nbi;
  p.m_tiles = p.n_tiles = c->db / TILE;
  p.n_split = n_split;
  p.k_chunks = (int)((by_rows ? c->d_in : c->d_out) / BK / n_split);
  p.r_s = (int64_t)p.batch * c->db;
  p.c_rows = p.r_s * n_split; p.c_cols = c->db;
  p.status = c->status;
  if (self) return launch<2>(c, A, nullptr, B, C, C2, p, s);
  return A2 ? launch<1>(c, A, A2, B, C, C2, p, s) : launch<0>(c, A, nullptr, B, C, nullptr, p, s);
}
