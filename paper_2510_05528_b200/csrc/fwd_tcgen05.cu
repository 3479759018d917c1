// The two thin products of the deployment form (Section 3.1: y = A (S (B x)) with block-diagonal A and B applied
// as batched d_block x d_block products) in bf16:  out[t][n] = sum_k X[t][j*db + k] * Q[n][k]  for the block j that
// holds column n, with Q the wrapper's blocks stacked as [d][db] (row n of the stack = row n - j*db of block j).
// Both operands are K-major as they lie in memory, so the kernel is a batched GEMM over the blocks: 128 x 128
// output tiles, the contraction runs over the db columns of X that belong to the tile's block (two or four
// k-tiles of 64), bf16 operands by TMA (128-byte swizzle), tcgen05.mma kind::f16 with fp32 accumulation in tensor
// memory, bf16 output.  Per output element the product moves 2 bytes in and 2 bytes out and does 2*db flops: it
// is a streaming kernel, bound by HBM.
//
// Also here: the packing of the wrappers for this kernel (bf16, the normalisation's scales folded in, Section 3.2
// last paragraph) and the layer forward built from this kernel and the sparse core product.
//
// Kernel: persistent, 320 threads: warp 0 TMA producer, warp 1 MMA issuer, warps 2-9 epilogue (accumulator -> bf16 -> swizzled
// staging box of 32 rows x 64 columns -> TMA store).  A CTA works through consecutive row tiles of ONE block, which stays in shared memory
// (32 or 128 KiB), and takes all its columns in one instruction: X is read once.  (Tiles of 128 columns that fetched their block and
// their X every time moved four bytes through L2 for each byte written: 28672 columns x 4,096 tokens 104 us, 8192 33 us, 0.66 of the copy
// bandwidth; now 85 and 27.)  Two accumulators.  Every wait is bounded.
#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BM = 128, BKE = 64;                   // BKE bf16 = 128 bytes = one swizzle row
constexpr int NTHREADS = 320;
constexpr int X_BYTES = BM * BKE * 2;               // 16 KiB: a stage
constexpr int BOX_BYTES = 32 * 64 * 2;              // an epilogue warp's staging box
template <int DB, int N> struct Geo {               // N: output columns of a tile, a block's or half of them
  static constexpr int KT = DB / BKE;               // k tiles of a block
  static constexpr int Q_BYTES = N * DB * 2;
  static constexpr int STAGES = N == 256 ? 4 : 8;
  static constexpr uint32_t COLS = 2 * N;           // two accumulators
  static constexpr size_t SMEM = (size_t)Q_BYTES + (size_t)STAGES * X_BYTES + 8 * BOX_BYTES + 1024;
};

struct FParams {
  int64_t rows;                      // tokens
  int m_tiles, n_groups;             // groups of N columns
  int32_t* status;
};

__device__ __forceinline__ uint64_t smem_desc_k(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ uint32_t instr_desc_bf16(int n) {
  uint32_t d = 0;
  d |= 1u << 4;                   // D format: F32
  d |= 1u << 7;                   // A format: BF16
  d |= 1u << 10;                  // B format: BF16
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(BM >> 4) << 24;
  return d;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <int DB, int N>
__global__ void __launch_bounds__(NTHREADS, 1)
fwd_block_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapC,
                 const FParams p) {
  using G = Geo<DB, N>;
  constexpr int STAGES = G::STAGES, KT = G::KT;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 6];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * STAGES]), tempty0 = tfull0 + 16, qfull = tfull0 + 32, qfree = tfull0 + 40;
  // the CTA's row tiles: contiguous over all groups, balanced to one tile
  const int64_t n_items = (int64_t)p.n_groups * p.m_tiles;
  const int i0 = (int)(n_items * blockIdx.x / gridDim.x), i1 = (int)(n_items * (blockIdx.x + 1) / gridDim.x);

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(tfull0 + 8 * s, 1); mbar_init(tempty0 + 8 * s, 8); }
    mbar_init(qfull, 1);
    mbar_init(qfree, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(G::COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_begin();                                     // (tensor memory is this CTA's before the next kernel's CTAs start)
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;
  uint8_t* const stage0 = smem + G::Q_BYTES;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      int cur = -1;
      uint32_t q_loads = 0;
      bool ok = true;
      for (int item = i0; item < i1 && ok; ++item) {
        const int b = item / p.m_tiles, mt = item - b * p.m_tiles;
        if (b != cur) {
          // the MMAs of the block before have read it
          if (q_loads > 0 && !mbar_wait(qfree, (q_loads - 1) & 1u, abortp, p.status)) { ok = false; break; }
          mbar_expect_tx(qfull, G::Q_BYTES);
          for (int kt = 0; kt < KT; ++kt) tma_load_2d(smem_u32(smem) + kt * N * 128, &mapQ, kt * BKE, b * N, qfull);
          ++q_loads;
          cur = b;
        }
        for (int kt = 0; kt < KT; ++kt) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
          const uint32_t fb = full0 + 8 * stage;
          mbar_expect_tx(fb, X_BYTES);
          tma_load_2d(smem_u32(stage0 + (size_t)stage * X_BYTES), &mapX, b / (DB / N) * DB + kt * BKE, mt * BM, fb);
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) {
        // leave no bulk copy in flight: wait (bounded) for the block and the stages armed most recently
        const long long tq = clock64();
        while (q_loads > 0 && !mbar_try(qfull, (q_loads - 1) & 1u) && clock64() - tq < 20000000ll) {}
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
      const uint32_t idesc = instr_desc_bf16(N);
      const uint64_t dq0 = smem_desc_k(smem_u32(smem)), dx0 = smem_desc_k(smem_u32(stage0));
      int stage = 0; uint32_t phase = 0;
      int local = 0, cur = -1;
      uint32_t q_waits = 0;
      bool ok = true;
      for (int item = i0; item < i1 && ok; ++item, ++local) {
        const int b = item / p.m_tiles;
        if (b != cur) {
          if (!mbar_wait(qfull, q_waits & 1u, abortp, p.status)) { ok = false; break; }
          ++q_waits;
          cur = b;
        }
        const int as = local & 1;
        const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
        if (!mbar_wait(tempty0 + 8 * as, aphase ^ 1, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tacc = tmem_base + (uint32_t)(as * N);
        for (int kt = 0; kt < KT; ++kt) {
          if (!mbar_wait(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint64_t dx = dx0 + (uint64_t)(uint32_t)(stage * (X_BYTES >> 4)), dq = dq0 + (uint64_t)(uint32_t)(kt * (N * 128 >> 4));
#pragma unroll
          for (int k = 0; k < BKE / 16; ++k) umma_bf16(tacc, dx + 2 * k, dq + 2 * k, idesc, (uint32_t)((kt > 0) | (k != 0)));
          umma_commit(empty0 + 8 * stage);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        umma_commit(tfull0 + 8 * as);
        if (item + 1 < i1 && (item + 1) / p.m_tiles != b) umma_commit(qfree);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    const int q = warp & 3;                 // tensor-memory lane quarter this warp may read
    const int half = (warp - 2) >> 2;       // which half of the tile's columns
    uint8_t* const box = stage0 + (size_t)STAGES * X_BYTES + (size_t)(warp - 2) * BOX_BYTES;
    const uint32_t box_u32 = smem_u32(box);
    int local = 0;
    bool ok = true;
    for (int item = i0; item < i1 && ok; ++item, ++local) {
      const int b = item / p.m_tiles, mt = item - b * p.m_tiles;
      const int as = local & 1;
      const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
      if (!mbar_wait(tfull0 + 8 * as, aphase, abortp, p.status)) { ok = false; break; }
      tc_fence_after();
      const int64_t row0 = (int64_t)mt * BM + q * 32;
#pragma unroll 1
      for (int ch = 0; ch < N / 128; ++ch) {
        // 64 columns of the lane's row as bf16: 16-byte unit c of the box's row sits at unit c ^ (row % 8)
        const int col = half * (N / 2) + ch * 64;
        uint32_t r0[32], r1[32];
        tmem_ld32(tmem_base + (uint32_t)(as * N + col) + ((uint32_t)(q * 32) << 16), r0);
        tmem_ld32(tmem_base + (uint32_t)(as * N + col + 32) + ((uint32_t)(q * 32) << 16), r1);
        if (ch == N / 128 - 1) {                   // all reads of the accumulator are done
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty0 + 8 * as);
        }
        if (lane == 0) tma_store_wait_read();       // the previous store has read the box
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t w0[4], w1[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            w0[k] = pack_bf16(__uint_as_float(r0[8 * u + 2 * k]), __uint_as_float(r0[8 * u + 2 * k + 1]));
            w1[k] = pack_bf16(__uint_as_float(r1[8 * u + 2 * k]), __uint_as_float(r1[8 * u + 2 * k + 1]));
          }
          *reinterpret_cast<uint4*>(box + lane * 128 + ((u ^ (lane & 7)) << 4)) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
          *reinterpret_cast<uint4*>(box + lane * 128 + (((u + 4) ^ (lane & 7)) << 4)) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0 && row0 < p.rows) {           // (rows past the end are clipped)
          tma_store_2d(&mapC, b * N + col, (int)row0, box_u32);
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
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(G::COLS) : "memory");
  }
}

// The same product for few tokens: one CTA per 16 tokens x 128 columns, eight warps of 16 columns.  At this size only
// latency counts, and the persistent kernel above pays for tensor memory, barriers and 128-row tiles that are mostly
// padding (4.6 us a launch at one token); here a warp requests its wrapper rows before it waits for the kernel before
// (programmatic dependent launch), the tokens go through shared memory once, and mma.sync m16n8k16 (tokens on the M side)
// does the rest.  The order of k inside an instruction is free as long as both operands agree, so a lane takes eight
// consecutive k (16 bytes) of its rows as the operands of two instructions; the columns of the two n-tiles are dealt out so
// that a lane ends with four neighbouring ones.
// SUM: the tokens come as `pieces` arrays of fp32 partial sums [rows][d], added in order and rounded to bf16 once.
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

template <int DB, bool SUM>
__global__ void __launch_bounds__(256)
fwd_small_kernel(const void* X, int pieces, const __nv_bfloat16* Q, __nv_bfloat16* __restrict__ out,
                 int rows, int64_t d) {
  constexpr int LD = DB * 2 + 64;                     // bytes per staged token: eight lanes of a phase hit eight banks
  __shared__ __align__(16) uint8_t tok[16 * LD];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t n0 = (int64_t)blockIdx.x * 128 + warp * 16;
  const int64_t kbase = (int64_t)blockIdx.x * 128 / DB * DB;   // first column of X of the block these columns belong to
  const int r0 = blockIdx.y * 16;
  // The first product of a pass waits before anything else and lets the core product in only then: that one fetches the packed core
  // before its own wait, and what wrote the core may be the kernel before this one.  The last product's weights are there.
  if (!SUM) grid_dependency_wait();
  grid_launch_dependents();
  uint4 w[2][DB / 32];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int ch = 0; ch < DB / 32; ++ch)
      w[nt][ch] = *reinterpret_cast<const uint4*>(Q + (n0 + 4 * (g >> 1) + 2 * nt + (g & 1)) * DB + ch * 32 + 8 * t);
  if (SUM) grid_dependency_wait();
#pragma unroll
  for (int e = threadIdx.x; e < 16 * DB / 8; e += 256) {
    const int r = e / (DB / 8), c8 = e % (DB / 8);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r0 + r < rows) {
      const int64_t o = (int64_t)(r0 + r) * d + kbase + 8 * c8;
      if (SUM) {
        const float* z = static_cast<const float*>(X) + o;
        float4 a = *reinterpret_cast<const float4*>(z), b = *reinterpret_cast<const float4*>(z + 4);
#pragma unroll 4
        for (int k = 1; k < pieces; ++k) {
          z += (int64_t)rows * d;
          const float4 a2 = *reinterpret_cast<const float4*>(z), b2 = *reinterpret_cast<const float4*>(z + 4);
          a.x += a2.x; a.y += a2.y; a.z += a2.z; a.w += a2.w;
          b.x += b2.x; b.y += b2.y; b.z += b2.z; b.w += b2.w;
        }
        v = make_uint4(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w), pack_bf16(b.x, b.y), pack_bf16(b.z, b.w));
      } else {
        v = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(X) + o);
      }
    }
    *reinterpret_cast<uint4*>(tok + r * LD + 16 * c8) = v;
  }
  __syncthreads();
  float acc[2][4] = {};
#pragma unroll
  for (int ch = 0; ch < DB / 32; ++ch) {
    const uint4 a0 = *reinterpret_cast<const uint4*>(tok + g * LD + ch * 64 + t * 16);
    const uint4 a1 = *reinterpret_cast<const uint4*>(tok + (g + 8) * LD + ch * 64 + t * 16);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      mma_bf16(acc[nt], a0.x, a1.x, a0.y, a1.y, w[nt][ch].x, w[nt][ch].y);
      mma_bf16(acc[nt], a0.z, a1.z, a0.w, a1.w, w[nt][ch].z, w[nt][ch].w);
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (r0 + g + 8 * h < rows)
      *reinterpret_cast<uint2*>(out + (int64_t)(r0 + g + 8 * h) * d + n0 + 4 * t) =
          make_uint2(pack_bf16(acc[0][2 * h], acc[0][2 * h + 1]), pack_bf16(acc[1][2 * h], acc[1][2 * h + 1]));
}

// Q[i][m][k] = rowscale[i*db + m] * colscale[i*db + k] * P[i][m][k], rounded to bf16 (either scale may be null)
__global__ void __launch_bounds__(256)
pack_blocks_kernel(const float* __restrict__ P, const float* __restrict__ rowscale, const float* __restrict__ colscale,
                   __nv_bfloat16* __restrict__ Q, int64_t n, int db) {
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (int64_t)gridDim.x * 256) {
    const int64_t i = e / ((int64_t)db * db);
    const int m = (int)((e / db) % db), k = (int)(e % db);
    float v = P[e];
    if (rowscale) v *= rowscale[i * db + m];
    if (colscale) v *= colscale[i * db + k];
    Q[e] = __float2bfloat16(v);
  }
}

bool make_map_bf16(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BKE, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int DB, int N>
armor_status launch_block(armor_ctx* c, const void* X, const void* Q, void* out, int64_t rows, int64_t d, cudaStream_t s) {
  CUtensorMap mX, mQ, mC;
  if (!make_map_bf16(&mX, X, rows, d, d, BM) || !make_map_bf16(&mQ, Q, d, DB, DB, N) || !make_map_bf16(&mC, out, rows, d, d, 32)) return ARMOR_ERR_CUDA;
  FParams p{};
  p.rows = rows; p.m_tiles = (int)((rows + BM - 1) / BM); p.n_groups = (int)(d / N);
  p.status = c->status;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, fwd_block_kernel<DB, N>, Geo<DB, N>::SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int64_t tiles = (int64_t)p.m_tiles * p.n_groups;
  KTimer kt(c, ARMOR_KC_FORWARD, 4.0 * (double)rows * (double)d, s);
  launch_dependent(fwd_block_kernel<DB, N>, (unsigned)(tiles < c->n_sm ? tiles : c->n_sm), NTHREADS, Geo<DB, N>::SMEM, s, mX, mQ, mC, p);
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

}  // namespace

bool fwd_block_ok(const armor_ctx* c) { return c->db % 128 == 0 && c->d_in % 128 == 0 && c->d_out % 128 == 0; }

void launch_pack_blocks(armor_ctx* c, const float* P, const float* rowscale, const float* colscale, void* Q, int nb,
                        cudaStream_t s) {
  const int64_t n = (int64_t)nb * c->db * c->db;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 148 * 16) blocks = 148 * 16;
  KTimer kt(c, ARMOR_KC_FORWARD, 0.0, s);
  pack_blocks_kernel<<<(unsigned)blocks, 256, 0, s>>>(P, rowscale, colscale, static_cast<__nv_bfloat16*>(Q), n, c->db);
  c->launches++;
}

// out[rows][d] (bf16) = X[rows][d] (bf16) times the block-diagonal matrix whose stacked blocks are Q[d][db] (bf16):
// out[t][n] = sum_k X[t][j*db + k] Q[n][k], j = n / db
armor_status launch_fwd_block(armor_ctx* c, const void* X, const void* Q, void* out, int64_t rows, int64_t d,
                              cudaStream_t s) {
  if (!fwd_block_ok(c) || rows <= 0 || d % c->db) return ARMOR_ERR_UNSUPPORTED;
  if (c->db == 128) return launch_block<128, 128>(c, X, Q, out, rows, d, s);
  // a block of 256 in halves while an SM has no more than one: 4096 columns x 400 tokens 28.1 us a forward in halves, 30.4 whole;
  // x 640 31.8 and 30.9; x 1,000 34.3 and 31.9
  return 2 * ((rows + BM - 1) / BM) * (d / 256) <= c->n_sm ? launch_block<256, 128>(c, X, Q, out, rows, d, s)
                                                          : launch_block<256, 256>(c, X, Q, out, rows, d, s);
}

// The same for few rows.  pieces == 0: X is bf16 [rows][d]; otherwise X holds that many fp32 arrays
// [rows][d] whose sum, rounded to bf16, is the operand.  Either way a dependent launch.
armor_status launch_fwd_small(armor_ctx* c, const void* X, int pieces, const void* Q, void* out, int64_t rows, int64_t d,
                              cudaStream_t s) {
  if (!fwd_block_ok(c) || rows <= 0 || d % 128) return ARMOR_ERR_UNSUPPORTED;
  KTimer kt(c, ARMOR_KC_FORWARD, 4.0 * (double)rows * (double)d, s);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(d / 128), (unsigned)((rows + 15) / 16)); cfg.blockDim = dim3(256); cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  const __nv_bfloat16* q = static_cast<const __nv_bfloat16*>(Q);
  __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out);
  const int n = (int)rows;
  cudaError_t e;
  if (c->db == 128) e = pieces > 0 ? cudaLaunchKernelEx(&cfg, fwd_small_kernel<128, true>, X, pieces, q, o, n, d)
                                   : cudaLaunchKernelEx(&cfg, fwd_small_kernel<128, false>, X, 0, q, o, n, d);
  else e = pieces > 0 ? cudaLaunchKernelEx(&cfg, fwd_small_kernel<256, true>, X, pieces, q, o, n, d)
                      : cudaLaunchKernelEx(&cfg, fwd_small_kernel<256, false>, X, 0, q, o, n, d);
  c->launches++;
  return e == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}
