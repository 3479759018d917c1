// Products with the block-diagonal wrappers (Section 3.1 of the paper) and per-block Grams for d_block = 256, on pairs of
// CTAs (cluster of two, cta_group::2): a pair works on 256 x 256 output tiles, the size of a wrapper block.
//
// The streaming kernel of block_tcgen05.cu cuts such a block into 128 x 128 tiles; each of them fetches and splits both its
// operands for itself and reads 8 KiB of shared memory per 65-cycle instruction, 1.7 MB through the SM's shared memory for
// 64 KB of output: at 28672 x 8192 a pass took 889 us where HBM needs 290 and the tensor pipe 330.  Here an instruction makes
// 128 x 256 outputs of an SM from the same 8 KiB (each SM holds 128 rows of the M side and half of the N side), and what is
// fetched and split per output halves: 0.9 MB per 64 KB.  At 14336 x 8192: left 333 us, with an addend 371, right 319, against
// 348 and 338 on the streaming kernel; products and Grams of three iterations at 28672 x 8192 48.0 -> 42.6 ms.
//
// Operands, split into high and low parts, order of the MMAs (lo*hi, hi*lo, hi*hi per 8 of k) and therefore the bits are
// those of block_tcgen05.cu.  Persistent kernel, 448 threads per CTA:
//   warp 0     : TMA producer: the CTA's 128 rows of either operand, chunks of 32 along k
//   warp 1     : MMA issuer (even CTA): tcgen05.mma.cta_group::2 kind::tf32, 256 x 256 x 8
//   warps 2-5  : low parts of the CTA's chunks; they report to the even CTA
//   warps 6-13 : epilogue of the CTA's 128 rows (a warp: 32 rows x 128 columns, one 32 x 32 box at a time: addend by TMA,
//                alpha / beta, TMA store)
// One product: two accumulators of 256 columns in turn.  Dual mode (A.X2 stored, <A.X1, A.X2> summed): one each for the two
// products of a tile.  Every wait is bounded; a wait that runs out raises a status word and the CTA leaves through the
// common exit that frees its tensor memory.
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BLK = 256, HALF = 128, BK = 32;
constexpr int NTHREADS = 448;
constexpr int STAGES = 3;
constexpr int OP_BYTES = HALF * BK * 4;           // 16 KiB: a CTA's share of an operand chunk
constexpr int STAGE_BYTES = 4 * OP_BYTES;         // M side raw, M side low part, N side raw, N side low part
constexpr uint32_t TMEM_COLS = 512;
constexpr int EPI_BYTES = 32 * 32 * 4;            // per epilogue warp: one swizzled 32 x 32 box
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + 8 * EPI_BYTES + 1024;

struct OpCoord {
  int mn_major;                     // 0: K-major, 1: MN-major
  int x_b, x_t, x_k;                // TMA x (inner) coordinate = x_b * batch + x_t * (tile of 128) + x_k * chunk
  int y_b, y_t, y_k;
  int wide;                         // MN-major: see tma_load_mn
};

struct PParams {
  OpCoord a, b;
  const float* D;                   // addend or nullptr
  int64_t c_rows, c_cols;           // extent of C (stores are guarded)
  int64_t r_b, c_b;                 // tile origin: row = r_b * batch + 256 * tm, column = c_b * batch + 256 * tn
  int m_tiles, n_tiles, batch, k_chunks;            // tiles of 256; k_chunks: chunks of 32 per work item
  int batch_fastest;                // 1: consecutive work items are consecutive batches (neighbouring column blocks)
  float alpha, beta;
  int32_t* status;
  int dual;                         // two N-side operands (mapB, mapB2); C = alpha * A.B2, dot_part = <A.B1, A.B2>
  double* dot_part;                 // dual: 16 partial sums per tile (one per epilogue warp of the pair)
  int two;                          // two products with the same N side: C = A.B and, for the odd work items, C2 = A2.B (A2
                                    // through mapB2, C2 through mapD); neighbouring pairs read the same chunks of B
};

__device__ __forceinline__ void load_operand(uint32_t dst, const CUtensorMap* map, const OpCoord& o, int b, int t, int kc,
                                             uint32_t bar) {
  const int x = o.x_b * b + o.x_t * t + o.x_k * kc;
  const int y = o.y_b * b + o.y_t * t + o.y_k * kc;
  if (o.mn_major) {
    tma_load_mn(dst, map, o.wide, x, y, bar);
  } else {
    tma_load_2d(dst, map, x, y, bar);
  }
}

__device__ __forceinline__ void item_decode(const PParams& p, int item, int& tn, int& tm, int& b, int& which) {
  which = p.two ? item & 1 : 0;
  if (p.two) item >>= 1;
  if (p.batch_fastest) {
    b = item % p.batch;
    const int rest = item / p.batch;
    tn = rest % p.n_tiles;
    tm = rest / p.n_tiles;
  } else {
    tn = item % p.n_tiles;
    tm = (item / p.n_tiles) % p.m_tiles;
    b = item / (p.n_tiles * p.m_tiles);
  }
}

__device__ __forceinline__ uint64_t operand_desc(uint32_t base, int mn_major) {
  return mn_major ? smem_desc_mn_sw128_32b(base, 4096, 512) : smem_desc_sw128(base, 16, 1024);
}

__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
               : "memory");
}
__device__ __forceinline__ void umma_pair_acc(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"
               "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc)
               : "memory");
}

__global__ void __launch_bounds__(NTHREADS, 1)
tc_blockpair_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                    const __grid_constant__ CUtensorMap mapB2, const __grid_constant__ CUtensorMap mapC,
                    const __grid_constant__ CUtensorMap mapD, const PParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[3 * STAGES + 12];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  // full (own loads), empty (commits reach both CTAs); split and tempty are used in the even CTA (both CTAs' warps report
  // there), tfull in both
  const uint32_t full0 = smem_u32(&bars[0]), split0 = smem_u32(&bars[STAGES]), empty0 = smem_u32(&bars[2 * STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[3 * STAGES]), tempty0 = smem_u32(&bars[3 * STAGES + 2]);
  const uint32_t dfull0 = smem_u32(&bars[3 * STAGES + 4]);
  const int n_items = p.batch * p.m_tiles * p.n_tiles * (p.two ? 2 : 1);
  const int n_sub = p.dual ? 2 : 1;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(split0 + 8 * s, 8);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) { mbar_init(tfull0 + 8 * s, 1); mbar_init(tempty0 + 8 * s, 16); }
    for (int s = 0; s < 8; ++s) mbar_init(dfull0 + 8 * s, 1);
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
  cluster_sync_all();                               // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  grid_begin();                                     // (tensor memory is this CTA's before the next kernel's CTAs start)
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      bool ok = true;
      for (int item = pair; item < n_items && ok; item += n_pairs) {
        int tn, tm, b, which;
        item_decode(p, item, tn, tm, b, which);
        for (int sub = 0; sub < n_sub && ok; ++sub)
          for (int kc = 0; kc < p.k_chunks; ++kc) {
            if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
            const uint32_t fb = full0 + 8 * stage;
            mbar_expect_tx(fb, 2 * OP_BYTES);
            const uint32_t dst = smem_u32(smem + (size_t)stage * STAGE_BYTES);
            load_operand(dst, which ? &mapB2 : &mapA, p.a, b, 2 * tm + rank, kc, fb);
            load_operand(dst + 2 * OP_BYTES, sub ? &mapB2 : &mapB, p.b, b, 2 * tn + rank, kc, fb);
            ++issued;
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
      }
      // tail: the MMAs that read the stages issued last have finished (their commits reach both CTAs), so nothing is in
      // flight towards this CTA's shared memory when it leaves
      for (int back = 1; back <= STAGES && back <= issued; ++back) {
        int s = stage - back; uint32_t ph = phase;
        if (s < 0) { s += STAGES; ph ^= 1; }
        const long long t0 = clock64();
        while (!mbar_try(empty0 + 8 * s, ph) && clock64() - t0 < (ok ? WAIT_CYCLES : 20000000ll)) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA)
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = instr_desc_tf32_mn(BLK, BLK, p.a.mn_major, p.b.mn_major);
      const uint64_t da0 = operand_desc(smem_u32(smem), p.a.mn_major);
      const uint64_t db0 = operand_desc(smem_u32(smem) + 2 * OP_BYTES, p.b.mn_major);
      const uint64_t kinc_a = p.a.mn_major ? (1024u >> 4) : (32u >> 4);   // one k-step of 8 in the address field
      const uint64_t kinc_b = p.b.mn_major ? (1024u >> 4) : (32u >> 4);
      int stage = 0; uint32_t phase = 0;
      uint32_t local = 0;                           // (tile, product) passes so far: accumulators take turns
      bool ok = true;
      for (int item = pair; item < n_items && ok; item += n_pairs)
        for (int sub = 0; sub < n_sub && ok; ++sub, ++local) {
          const uint32_t as = local & 1u, aphase = (local >> 1) & 1u;
          if (!mbar_wait_cluster(tempty0 + 8 * as, aphase ^ 1u, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tacc = tmem_base + as * (uint32_t)BLK;
          for (int kc = 0; kc < p.k_chunks; ++kc) {
            if (!mbar_wait_cluster(split0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint64_t so = (uint64_t)(uint32_t)(stage * (STAGE_BYTES >> 4));
            const uint64_t da = da0 + so, dal = da + (OP_BYTES >> 4);
            const uint64_t dbm = db0 + so, dbl = dbm + (OP_BYTES >> 4);
            const uint32_t first = (uint32_t)(kc > 0);
            umma_pair(tacc, dal, dbm, idesc, first);
            umma_pair_acc(tacc, da, dbl, idesc);
            umma_pair_acc(tacc, da, dbm, idesc);
#pragma unroll
            for (int k = 1; k < BK / 8; ++k) {
              umma_pair_acc(tacc, dal + k * kinc_a, dbm + k * kinc_b, idesc);
              umma_pair_acc(tacc, da + k * kinc_a, dbl + k * kinc_b, idesc);
              umma_pair_acc(tacc, da + k * kinc_a, dbm + k * kinc_b, idesc);
            }
            umma_commit_pair(empty0 + 8 * stage);   // frees the stage in both CTAs once these MMAs have read it
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
          if (ok) umma_commit_pair(tfull0 + 8 * as);
        }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------ low parts (both CTAs)
    const int t = threadIdx.x - 64;   // 0..127
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    for (int item = pair; item < n_items && ok; item += n_pairs) {
      for (int kc = 0; kc < n_sub * p.k_chunks; ++kc) {
        if (!mbar_wait(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
        float4* base = reinterpret_cast<float4*>(smem + (size_t)stage * STAGE_BYTES);
#pragma unroll
        for (int op = 0; op < 2; ++op) {
          float4* hi = base + op * (2 * OP_BYTES / 16);
          float4* lo = hi + OP_BYTES / 16;
#pragma unroll
          for (int e = 0; e < OP_BYTES / 16 / 128; ++e) {
            const int idx = t + e * 128;
            const float4 v = hi[idx];
            float4 h;
            h.x = __uint_as_float(__float_as_uint(v.x) & 0xffffe000u);
            h.y = __uint_as_float(__float_as_uint(v.y) & 0xffffe000u);
            h.z = __uint_as_float(__float_as_uint(v.z) & 0xffffe000u);
            h.w = __uint_as_float(__float_as_uint(v.w) & 0xffffe000u);
            lo[idx] = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
          }
        }
        // make the generic-proxy writes visible to the tensor-core (async proxy) reads of the pair
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_cta(split0 + 8 * stage, 0));
        if (++stage == STAGES) { stage = 0; phase ^= 1; }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps (both CTAs)
    const int q = warp & 3;                         // TMEM lane quarter this warp may read
    const int e = warp - 6, half = e >> 2;          // which 128 columns of the tile
    uint8_t* buf = smem + (size_t)STAGES * STAGE_BYTES + (size_t)e * EPI_BYTES;
    const uint32_t buf_u32 = smem_u32(buf);
    const uint32_t dbar = dfull0 + 8 * e;
    uint8_t* rowp = buf + lane * 128;               // lane = row of the box; 16-byte unit u sits at u ^ (row % 8)
    uint32_t local = 0, d_loads = 0;
    bool ok = true;
    for (int item = pair; item < n_items && ok; item += n_pairs, ++local) {
      int tn, tm, b, which;
      item_decode(p, item, tn, tm, b, which);
      const uint32_t as = p.dual ? 0u : (local & 1u), aphase = (p.dual ? local : local >> 1) & 1u;
      const int64_t row = p.r_b * b + (int64_t)tm * BLK + rank * HALF + q * 32;
      const int64_t col = p.c_b * b + (int64_t)tn * BLK + half * HALF;
      double dot = 0.0;
      bool got = false;
#pragma unroll 1
      for (int ch = 0; ch < 4; ++ch) {
        const bool in = row < p.c_rows && col + 32 * ch < p.c_cols;      // warp-uniform; TMA clips a box that reaches over
        if (lane == 0) {
          tma_store_wait_read();                    // the previous store has read the staging box
          if (p.D && in) {
            mbar_expect_tx(dbar, 4096u);
            tma_load_2d(buf_u32, &mapD, (int)(col + 32 * ch), (int)row, dbar);
          }
        }
        __syncwarp();
        if (!got) {
          if (!__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * as, aphase, abortp, p.status))) { ok = false; break; }
          if (p.dual && !__all_sync(0xffffffffu, mbar_wait(tfull0 + 8, aphase, abortp, p.status))) { ok = false; break; }
          tc_fence_after();
          got = true;
        }
        uint32_t r[32];
        const uint32_t tcol = (uint32_t)(half * HALF + 32 * ch) + ((uint32_t)(q * 32) << 16);
        if (p.dual) {
          uint32_t r1[32];
          tmem_ld32(tmem_base + tcol, r1);
          tmem_ld32(tmem_base + (uint32_t)BLK + tcol, r);
          float part = 0.f;
#pragma unroll
          for (int i = 0; i < 32; ++i) part = fmaf(__uint_as_float(r1[i]), __uint_as_float(r[i]), part);
          dot += (double)part;
        } else {
          tmem_ld32(tmem_base + as * (uint32_t)BLK + tcol, r);
        }
        if (p.D && in) {
          if (!__all_sync(0xffffffffu, mbar_wait(dbar, d_loads & 1u, abortp, p.status))) { ok = false; break; }
          ++d_loads;
        }
        if (in) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            float4* cell = reinterpret_cast<float4*>(rowp + ((u ^ (lane & 7)) << 4));
            float4 v = make_float4(p.alpha * __uint_as_float(r[4 * u]), p.alpha * __uint_as_float(r[4 * u + 1]),
                                   p.alpha * __uint_as_float(r[4 * u + 2]), p.alpha * __uint_as_float(r[4 * u + 3]));
            if (p.D) {
              const float4 d = *cell;
              v.x = fmaf(p.beta, d.x, v.x); v.y = fmaf(p.beta, d.y, v.y);
              v.z = fmaf(p.beta, d.z, v.z); v.w = fmaf(p.beta, d.w, v.w);
            }
            *cell = v;
          }
        }
        if (ch == 3) tc_fence_before();             // all reads of the accumulator are done
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          if (ch == 3) {
            mbar_arrive_cluster(map_to_cta(tempty0 + 8 * as, 0));
            if (p.dual) mbar_arrive_cluster(map_to_cta(tempty0 + 8, 0));
          }
          if (in) tma_store_2d(which ? &mapD : &mapC, (int)(col + 32 * ch), (int)row, buf_u32);
          tma_store_commit();
        }
      }
      if (p.dual) {
        // lanes in a fixed order
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if (ok && lane == 0) p.dot_part[(size_t)item * 16 + rank * 8 + e] = dot;
      }
    }
    if (lane == 0) tma_store_wait_read();           // shared memory stays valid until the stores have read it
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // neither CTA leaves while its partner may still signal it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

struct HostOp {
  const float* base; int64_t inner, outer, ld;   // global 2-D view [outer][inner]
  OpCoord c;
};

inline bool map_operand(CUtensorMap* m, const HostOp& o, const float* base, OpCoord& c) {
  return o.c.mn_major ? make_map_mn(m, base, o.inner, o.outer, o.ld, &c.wide) : make_map_2d(m, base, o.inner, o.outer, o.ld, 32, HALF);
}

// ldc: leading dimension of C and D.  B2: the second N-side operand (dual); A2, C2: the second M-side operand and output (two)
armor_status launch(armor_ctx* c, const HostOp& A, const HostOp& B, PParams p, float* C, int64_t ldc, int kclass, double kbytes,
                    cudaStream_t s, const float* B2 = nullptr, const float* A2 = nullptr, float* C2 = nullptr) {
  CUtensorMap mA, mB, mB2, mC, mD;
  if (!make_map_2d(&mC, C, p.c_cols, p.c_rows, ldc, 32, 32)) return ARMOR_ERR_CUDA;
  p.two = A2 ? 1 : 0;
  if (A2 && (B2 || p.D || !C2)) return ARMOR_ERR_INVALID_ARG;
  if (A2) {
    if (!make_map_2d(&mD, C2, p.c_cols, p.c_rows, ldc, 32, 32)) return ARMOR_ERR_CUDA;
  } else if (p.D) {
    if (!make_map_2d(&mD, p.D, p.c_cols, p.c_rows, ldc, 32, 32)) return ARMOR_ERR_CUDA;
  } else {
    mD = mC;
  }
  p.a = A.c; p.b = B.c;
  if (!map_operand(&mA, A, A.base, p.a) || !map_operand(&mB, B, B.base, p.b)) return ARMOR_ERR_CUDA;
  if (B2) {
    if (!map_operand(&mB2, B, B2, p.b)) return ARMOR_ERR_CUDA;
  } else if (A2) {
    if (!map_operand(&mB2, A, A2, p.a)) return ARMOR_ERR_CUDA;
  } else {
    mB2 = mB;
  }
  p.status = c->status;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_blockpair_kernel, SMEM_BYTES) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int n_items = p.batch * p.m_tiles * p.n_tiles * (p.two ? 2 : 1);
  const int pairs = n_items < c->n_sm / 2 ? n_items : c->n_sm / 2;
  KTimer kt(c, kclass, kbytes, s);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * pairs); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = SMEM_BYTES; cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, tc_blockpair_kernel, mA, mB, mB2, mC, mD, p) != cudaSuccess) return ARMOR_ERR_CUDA;
  c->launches++;
  return ARMOR_OK;
}

inline bool ptr_ok(const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; }

}  // namespace

// Two waves of tiles at least: with fewer, 128 x 128 tiles on single CTAs spread better (3840 x 6400, 148 tokens: 64 us against
// 76 for a forward).  Products that round their operands to one pass are bound by neither fetching nor splitting (23808 x
// 3072, 2,292 tokens: 397 us against 428).
bool tc_blockpair_ok(const armor_ctx* c, int64_t tiles) {
  return c->db == BLK && !c->block_one_pass && c->n_sm >= 2 && tiles >= c->n_sm;
}

// out[:, j-th block] = alpha * in[:, j-th block] * Q_j (+ beta * add[:, j-th block]),  Q_j = Bblk[j] or its transpose
armor_status tc_blockpair_right(armor_ctx* c, const float* in, const float* Bblk, bool transB, float* out, int64_t rows,
                                int64_t cols, float alpha, const float* add, float beta, cudaStream_t s) {
  if (!ptr_ok(in) || !ptr_ok(Bblk) || !ptr_ok(out) || (add && !ptr_ok(add))) return ARMOR_ERR_UNSUPPORTED;
  const int nb = (int)(cols / BLK);
  HostOp A{in, cols, rows, cols, {0, BLK, 0, BK, 0, HALF, 0}};
  HostOp B{Bblk, BLK, (int64_t)nb * BLK, BLK, {}};
  if (transB) B.c = {0, 0, 0, BK, BLK, HALF, 0};        // [n][k] = B_j[n][k]: K-major
  else        B.c = {1, 0, HALF, 0, BLK, 0, BK};        // [n][k] = B_j[k][n]: N-major
  PParams p{};
  p.D = add; p.c_rows = rows; p.c_cols = cols;
  p.c_b = BLK;
  p.m_tiles = (int)((rows + BLK - 1) / BLK); p.n_tiles = 1; p.batch = nb; p.k_chunks = BLK / BK;
  p.batch_fastest = 1;
  p.alpha = alpha; p.beta = add ? beta : 0.f;
  return launch(c, A, B, p, out, cols, ARMOR_KC_BLOCK_PRODUCT, (add ? 12.0 : 8.0) * (double)rows * (double)cols, s);
}

// out[i-th block, :] = alpha * P_i * in[i-th block, :] (+ beta * add[i-th block, :]),  P_i = Ablk[i] or its transpose.
// in2: out takes the product with in2, and *n_part partial sums of <P_i in, P_i in2> go to part
armor_status tc_blockpair_left(armor_ctx* c, const float* Ablk, bool transA, const float* in, float* out, int64_t rows,
                               int64_t cols, float alpha, const float* add, float beta, cudaStream_t s, const float* in2,
                               double* part, int* n_part) {
  if (!ptr_ok(in) || !ptr_ok(Ablk) || !ptr_ok(out) || (add && !ptr_ok(add)) || (in2 && !ptr_ok(in2))) return ARMOR_ERR_UNSUPPORTED;
  const int nb = (int)(rows / BLK);
  HostOp A{Ablk, BLK, (int64_t)nb * BLK, BLK, {}};
  if (transA) A.c = {1, 0, HALF, 0, BLK, 0, BK};        // [m][k] = A_i[k][m]: M-major
  else        A.c = {0, 0, 0, BK, BLK, HALF, 0};        // [m][k] = A_i[m][k]: K-major
  HostOp B{in, cols, rows, cols, {1, 0, HALF, 0, BLK, 0, BK}};   // [n][k] = in[256 i + k][n]: N-major
  PParams p{};
  p.D = add; p.c_rows = rows; p.c_cols = cols;
  p.r_b = BLK;
  p.m_tiles = 1; p.n_tiles = (int)((cols + BLK - 1) / BLK); p.batch = nb; p.k_chunks = BLK / BK;
  p.alpha = alpha; p.beta = add ? beta : 0.f;
  if (in2) {
    p.dual = 1; p.dot_part = part;
    *n_part = 16 * p.batch * p.n_tiles;
  }
  return launch(c, A, B, p, out, cols, ARMOR_KC_BLOCK_PRODUCT, (add || in2 ? 12.0 : 8.0) * (double)rows * (double)cols, s, in2);
}

// by_rows: G_i = P_i T_i^T over the row blocks (contraction over d_in); else G_j = P_j^T T_j over the column blocks
// (contraction over d_out).  P2: G2 likewise with P2 in the place of P, in the same launch.
armor_status tc_blockpair_gram(armor_ctx* c, const float* P, const float* T, bool by_rows, float* G, cudaStream_t s,
                               const float* P2, float* G2) {
  if (!ptr_ok(P) || !ptr_ok(T) || !ptr_ok(G) || (P2 && (!ptr_ok(P2) || !ptr_ok(G2)))) return ARMOR_ERR_UNSUPPORTED;
  const int nb = by_rows ? c->nbo : c->nbi;
  OpCoord o;
  if (by_rows) o = {0, 0, 0, BK, BLK, HALF, 0};         // [m][k] = P[256 i + m][k]: K-major
  else         o = {1, BLK, HALF, 0, 0, 0, BK};         // [m][k] = P[k][256 j + m]: M-major
  HostOp A{P, c->d_in, c->d_out, c->d_in, o}, B{T, c->d_in, c->d_out, c->d_in, o};
  PParams p{};
  p.c_rows = (int64_t)nb * BLK; p.c_cols = BLK;
  p.r_b = BLK;
  p.m_tiles = 1; p.n_tiles = 1; p.batch = nb; p.k_chunks = (int)((by_rows ? c->d_in : c->d_out) / BK);
  p.alpha = 1.f;
  return launch(c, A, B, p, G, BLK, ARMOR_KC_BLOCK_GRAM, (P2 ? 12.0 : 8.0) * (double)c->wn, s, nullptr, P2, G2);
}
