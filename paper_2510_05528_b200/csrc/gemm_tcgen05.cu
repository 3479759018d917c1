// Tensor-core GEMM for sm_100a:  C[M][N] (+)= sum_k A[m][k] * B[n][k]   (fp32 storage, both operands K-major)
//
// Used for the dense contractions of the ARMOR iteration: the calibration Gram X^T X (Section 2 of the
// paper; both operands are the transposed, staged chunk of X) and the right-multiplications by the
// symmetric Gram, E.H, T.H and V.H (H[n][k] = H[k][n], so H itself is the K-major B operand).
//
// Design: persistent kernel on pairs of CTAs (cluster of two, cta_group::2), a 256 x 256 tile of C per pair:
//   warp 0   : TMA producer  (cp.async.bulk.tensor.2d, 128-byte swizzle; each CTA loads its 128 rows of A and its
//                             128 rows of B and signals the even CTA's barrier)
//   warp 1   : MMA issuer    (one thread of the even CTA issues tcgen05.mma.cta_group::2, 256 x 256 x 16 (x 8 for
//                             tf32); every SM holds its own 128 rows of the accumulator in tensor memory, two
//                             accumulator buffers of 256 columns)
//   warps 2-9: epilogue      (tcgen05.ld 32 lanes x 32 columns; the K segments of a tile are summed in registers,
//                             then one fused C-update / dot products; a symmetric product writes its lower
//                             triangle only, the caller mirrors it once at the end)
// Why pairs: per 64 columns of K one SM fetches 32 KB (64 KB with split operands) for its 128 x 256 outputs, where a
// CTA of its own fetches 48 KB (96 KB).  With one MMA per product the single CTA was bound by what L2 delivers
// (8.7 TB/s into shared memory at 720 TFLOP/s), not by the tensor pipe.
// passes == 3: every operand is given as a tf32-exact high part and an fp32 low part; the three products
// hi*hi, lo*hi, hi*lo are accumulated into the same fp32 accumulator (error-compensated tf32, fp32-grade).
// passes == 6: the same three products on fp16 high and low parts (kind::f16, twice the tf32 issue rate, half
// the operand bytes).  Two fp16 parts carry 22 significant bits like two tf32 parts, but only 5 exponent bits,
// so the caller scales rows of the operands by powers of two into the fp16 range beforehand and the epilogue
// multiplies the accumulator by the inverse scales (a per-row and a per-column vector): every scaling is
// exact, the result is fp32-grade.
// Few rows (FEW, the bf16 core product of up to 512 tokens): the operands change sides.  256 columns of C are the M side of an
// instruction and the rows of a tile, only as many as there are, its N side, so that neither the MMAs nor the fetched bytes
// are spent on rows that do not exist (a 256 x 256 tile of one row took 43 us of MMAs for 21 us of reading at 8192 x 8192).
// Every wait is bounded: a wait that runs out raises a status word and the CTA leaves through the common
// exit that frees its tensor memory.
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BMP = 256, BM = 128, BN = 256, BK = 32;   // pair tile rows, rows per CTA, columns; BK fp32 = 128 bytes
constexpr int BNH = BN / 2;                         // rows of B each CTA of the pair holds
constexpr int NTHREADS = 320;                       // TMA warp, MMA warp, eight epilogue warps
constexpr int EPI_COLS = 128;                       // accumulator columns per epilogue warp
constexpr int EPI_BYTES = 32 * 32 * 4;              // an epilogue warp's 32 x 32 staging tile
constexpr uint32_t TMEM_COLS = 512;                 // two accumulator buffers of BN columns
constexpr int A_BYTES = BM * BK * 4;                // 16 KiB
constexpr int B_BYTES = BNH * BK * 4;               // 16 KiB
constexpr int MN_BOX = 64 * 64 * 2;                 // 64 k x 64 rows of a 16-bit operand that is contiguous along M / N

// stages of the shared-memory ring: 3 x 64 KiB with split operands, 6 x 32 KiB otherwise
template <int PASSES>
struct Ring {
  static constexpr int BYTES = (PASSES == 3 || PASSES == 6 ? 2 : 1) * (A_BYTES + B_BYTES);
  static constexpr int STAGES = PASSES == 3 || PASSES == 6 ? 3 : 6;
};

constexpr int PARTS = 16;                           // partial dot products per tile: one per epilogue warp of the pair

struct Params {
  float* C; int64_t ldc;
  int64_t M, N, K;
  int m_tiles, n_tiles, n_tiles_total;
  int accumulate, symmetric_lower;
  int c_vec;             // rows of C start on 16-byte boundaries
  int kt_seg;            // k-tiles accumulated in tensor memory before the epilogue folds them into C
  const float* d1; const float* d2;
  double* part1; double* part2;
  const float* row_scale; const float* col_scale;   // optional powers of two the accumulator is multiplied by
  int dependent;         // launched beside the kernel that writes the scales: the epilogue waits for it
  int f16;               // 16-bit operands are fp16 (1) or bf16 (0)
  const int32_t* only_if;
  int32_t* status;
  // Tail split: tiles [split_first, n_tiles_total) are cut into split_parts pieces of split_kt k-tiles (the last one
  // may be shorter), each piece a work item of its own that writes a 256 x 256 slab of partial sums; a second kernel
  // adds the slabs.  This fills the last, partly empty wave of tiles.
  int split_first, split_parts, split_kt, n_items;
  int tile_m;            // rows of C per tile: 256; FEW: the rows dealt evenly to one or two tiles, a multiple of 32
  float* slabs;
};

// K-major operand tile, rows of 128 bytes, 128-byte swizzle: 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_k_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address
  d |= (uint64_t)1 << 16;                           // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset
  d |= (uint64_t)1 << 46;                           // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                           // 128-byte swizzle
  return d;
}

// The other form of a 16-bit operand: contiguous along M / N (a row-major X is such an operand of X^T X).  A k-row
// holds 64 elements (128 bytes), groups of 8 k-rows are 1024 bytes apart, the next 64 elements one box further.
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t addr) { return smem_desc_sw128(addr, MN_BOX, 1024); }

// tcgen05.mma of the pair; ACC: the accumulate flag is a constant, which costs no instruction
template <bool F16>
__device__ __forceinline__ void umma_acc(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc) {
  if (F16)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc) : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc) : "memory");
}
template <bool F16>
__device__ __forceinline__ void umma_first(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  if (F16)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}

// fp32 accumulate, M = 256 (the pair), N = 256; operand format 0: fp16, 1: bf16 (both kind::f16), 2: tf32
// (kind::tf32); mn: both operands are contiguous along M / N instead of K.
__device__ __forceinline__ uint32_t instr_desc(uint32_t fmt, uint32_t mn, uint32_t n = BN) {
  uint32_t d = 0;
  d |= 1u << 4;                   // D format: F32
  d |= fmt << 7;                  // A format
  d |= fmt << 10;                 // B format
  d |= mn << 15;
  d |= mn << 16;
  d |= (n >> 3) << 17;            // N
  d |= (uint32_t)(BMP >> 4) << 24; // M
  return d;
}

// tile index -> (m tile, n tile).  Groups of GROUP_M m tiles; inside a group m runs fastest, then n: the 74 tiles
// in flight are about 8 x 9, which minimises what a wave reads -- with m running over all m tiles every wave read up
// to 74 A panels, and on the large shapes (operands far beyond L2) the product became DRAM-bound.
constexpr int GROUP_M = 8;
__device__ __forceinline__ void tile_coords(const Params& p, int tile, int& mt, int& nt) {
  if (!p.symmetric_lower) {
    const int per_group = GROUP_M * p.n_tiles;
    const int g = tile / per_group, r = tile - g * per_group;
    const int gm = min(GROUP_M, p.m_tiles - g * GROUP_M);
    mt = g * GROUP_M + r % gm;
    nt = r / gm;
    return;
  }
  // only tiles that hold an element with column <= row: m tile >= n tile.  Same grouping: bands of GROUP_M
  // m tiles, inside a band the n tile is the outer index and m runs fastest
  int rem = tile;
  for (int m0 = 0; m0 < p.m_tiles; m0 += GROUP_M) {
    const int m1 = min(m0 + GROUP_M, p.m_tiles);
    for (nt = 0; nt < m1 && nt < p.n_tiles; ++nt) {
      const int lo = max(m0, nt);
      const int cnt = m1 - lo;
      if (rem < cnt) { mt = lo + rem; return; }
      rem -= cnt;
    }
  }
  mt = 0; nt = 0;   // not reached: tile < number of tiles
}

// work item -> tile, and its range of k-tiles
__device__ __forceinline__ void item_decode(const Params& p, int item, int kt_total, int& tile, int& part, int& kt_begin,
                                            int& kt_end) {
  if (item < p.split_first) {
    tile = item; part = -1; kt_begin = 0; kt_end = kt_total;
  } else {
    const int idx = item - p.split_first;
    tile = p.split_first + idx / p.split_parts;
    part = idx % p.split_parts;
    kt_begin = part * p.split_kt; kt_end = min(kt_total, kt_begin + p.split_kt);
  }
}

// four floats of C: one access where every row of C starts on a 16-byte boundary (vec)
__device__ __forceinline__ float4 load4(const float* q, int vec) {
  return vec ? *reinterpret_cast<const float4*>(q) : make_float4(q[0], q[1], q[2], q[3]);
}
__device__ __forceinline__ void store4(float* q, const float4& v, int vec) {
  if (vec) { *reinterpret_cast<float4*>(q) = v; return; }
  q[0] = v.x; q[1] = v.y; q[2] = v.z; q[3] = v.w;
}

// One epilogue warp's 32 rows x 128 columns of finished sums (lane = row) go out through a 32 x 32 staging tile in
// shared memory (16-byte units, swizzled by the row: no bank conflicts either way), so that every access to C writes or
// reads four rows of 128 contiguous bytes.  Optional: power-of-two scales, C += (read-modify-write), chunks of 32 x 32
// above the diagonal left out, partial dot products with d1 / d2 (DOTS; without, the code for them is not there: fp64 conversions
// of nothing cost a Gram of few tokens 3 %).
template <bool DOTS>
__device__ __forceinline__ void write_out(const float (&acc)[EPI_COLS], float4* stg, int lane, float* C, int64_t ldc, int vec,
                                          int64_t row_base, int64_t col_base, int64_t M, int64_t N, bool accum, bool sym,
                                          const float* rs, const float* cs, const float* d1, const float* d2, int64_t ldd,
                                          double& dot1, double& dot2) {
  if (row_base >= M) return;                                  // warp-uniform
  const int rr = lane >> 3, cc = lane & 7;
  const float rscale = (rs && row_base + lane < M) ? rs[row_base + lane] : 1.f;
#pragma unroll
  for (int ch = 0; ch < EPI_COLS / 32; ++ch) {
    const int64_t col0 = col_base + ch * 32;
    if (col0 >= N) continue;                                   // warp-uniform (N is a multiple of 32)
    if (sym && col0 > row_base + 31) continue;                 // chunk lies above the diagonal
#pragma unroll
    for (int j = 0; j < 8; ++j)
      stg[lane * 8 + (j ^ (lane & 7))] = make_float4(acc[ch * 32 + 4 * j] * rscale, acc[ch * 32 + 4 * j + 1] * rscale,
                                                     acc[ch * 32 + 4 * j + 2] * rscale, acc[ch * 32 + 4 * j + 3] * rscale);
    __syncwarp();
    const int64_t col = col0 + 4 * cc;
    const float4 sc4 = cs ? *reinterpret_cast<const float4*>(cs + col) : make_float4(1.f, 1.f, 1.f, 1.f);
    float f1[2] = {0.f, 0.f}, f2[2] = {0.f, 0.f};              // 16 terms each in fp32, then fp64
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 o[4];
      if (accum) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int64_t grow = row_base + 16 * h + 4 * i + rr;
          o[i] = grow < M ? load4(C + grow * ldc + col, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 16 * h + 4 * i + rr;
        const int64_t grow = row_base + r;
        if (grow >= M) continue;
        float4 x = stg[r * 8 + (cc ^ (r & 7))];
        x.x *= sc4.x; x.y *= sc4.y; x.z *= sc4.z; x.w *= sc4.w;
        if (accum) { x.x += o[i].x; x.y += o[i].y; x.z += o[i].z; x.w += o[i].w; }
        if (DOTS && d1) {
          const float4 w = *reinterpret_cast<const float4*>(d1 + grow * ldd + col);
          f1[h] += x.x * w.x + x.y * w.y + x.z * w.z + x.w * w.w;
        }
        if (DOTS && d2) {
          const float4 w = *reinterpret_cast<const float4*>(d2 + grow * ldd + col);
          f2[h] += x.x * w.x + x.y * w.y + x.z * w.z + x.w * w.w;
        }
        store4(C + grow * ldc + col, x, vec);
      }
    }
    if (DOTS) {
      dot1 += (double)f1[0] + (double)f1[1];
      dot2 += (double)f2[0] + (double)f2[1];
    }
    __syncwarp();
  }
}

// MN: both operands are 16-bit arrays contiguous along M / N (PASSES 0 and 6).  FEW: PASSES 0, K-major, C = A B^T and nothing else.
// DOTS: with dot products.
template <int PASSES, bool MN, bool FEW, bool DOTS>
__global__ void __launch_bounds__(NTHREADS, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapAlo,
               const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapBlo, const Params p) {
  constexpr bool SPLIT = (PASSES == 3 || PASSES == 6);   // operands come as high and low parts
  constexpr bool H16 = (PASSES == 0 || PASSES == 6);     // 16-bit operands (kind::f16)
  constexpr int STAGE_BYTES = Ring<PASSES>::BYTES;
  constexpr int STAGES = Ring<PASSES>::STAGES;
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 4];
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * STAGES]), tempty0 = smem_u32(&bars[2 * STAGES + 2]);
  constexpr int BKE = H16 ? 64 : 32;                // elements of K per 128-byte row: 16-bit or fp32
  const int kt_total = (int)((p.K + BKE - 1) / BKE);
  if (!MN && p.only_if) {
    grid_dependency_wait();
    if (*p.only_if == 0) return;                    // (before anything is allocated, both CTAs of the pair alike)
  }

  // full, empty of the stages; tfull, tempty of the accumulator buffers.  full and tempty are used in the even CTA
  // only (both CTAs' loads and epilogue warps signal it there), empty and tfull in both (commits reach the pair).
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
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
  cluster_sync_all();                                  // both CTAs' barriers exist before anyone signals them
  tc_fence_after();
  // (tensor memory is this CTA's before the next kernel's CTAs start; a Gram's product waits where its scales are read)
  if (!MN) grid_begin();
  const uint32_t tmem_base = tmem_base_holder;
  volatile int* abortp = &abort_flag;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0; long long issued = 0;
      bool ok = true;
      for (int item = pair; item < p.n_items && ok; item += n_pairs) {
        int tile, part, kt_begin, kt_end, mt, nt;
        item_decode(p, item, kt_total, tile, part, kt_begin, kt_end);
        tile_coords(p, tile, mt, nt);
        const int arow = mt * BMP + (int)rank * BM, brow = nt * BN + (int)rank * BNH;
        for (int kt = kt_begin; kt < kt_end; ++kt) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abortp, p.status)) { ok = false; break; }
          if (rank == 0) mbar_expect_tx(full0 + 8 * stage, FEW ? 2 * (A_BYTES + (p.tile_m / 2) * 128) : 2 * STAGE_BYTES);
          const uint32_t fb = map_to_cta(full0 + 8 * stage, 0);
          uint32_t dst = smem_u32(smem + (size_t)stage * STAGE_BYTES);
          if (FEW) {
            tma_load_2d_pair(dst, &mapB, kt * BKE, brow, fb);
            tma_load_2d_pair(dst + A_BYTES, &mapA, kt * BKE, mt * p.tile_m + (int)rank * (p.tile_m / 2), fb);
          } else if (MN) {
            // x = row of the operand (a channel), y = k (a token); rows and k beyond the operand are zero-filled
#pragma unroll
            for (int part = 0; part < (SPLIT ? 2 : 1); ++part) {
              const CUtensorMap* ma = part ? &mapAlo : &mapA;
              const CUtensorMap* mb = part ? &mapBlo : &mapB;
              const uint32_t da = dst + part * A_BYTES, db = dst + (SPLIT ? 2 : 1) * A_BYTES + part * B_BYTES;
              tma_load_2d_pair(da, ma, arow, kt * BKE, fb);
              tma_load_2d_pair(da + MN_BOX, ma, arow + 64, kt * BKE, fb);
              tma_load_2d_pair(db, mb, brow, kt * BKE, fb);
              tma_load_2d_pair(db + MN_BOX, mb, brow + 64, kt * BKE, fb);
            }
          } else {
            tma_load_2d_pair(dst, &mapA, kt * BKE, arow, fb);
            dst += A_BYTES;
            if (SPLIT) { tma_load_2d_pair(dst, &mapAlo, kt * BKE, arow, fb); dst += A_BYTES; }
            tma_load_2d_pair(dst, &mapB, kt * BKE, brow, fb);
            dst += B_BYTES;
            if (SPLIT) tma_load_2d_pair(dst, &mapBlo, kt * BKE, brow, fb);
          }
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      // tail: the MMAs that read the stages issued last have finished (their commits reach both CTAs), so nothing is
      // in flight towards this CTA's shared memory when it leaves
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
      const uint32_t idesc = instr_desc(H16 ? (p.f16 ? 0u : 1u) : 2u, MN ? 1u : 0u, FEW ? (uint32_t)p.tile_m : BN);
      const uint64_t d0 = MN ? smem_desc_mn_sw128(smem_u32(smem)) : smem_desc_k_sw128(smem_u32(smem));
      int stage = 0; uint32_t phase = 0;
      int local = 0;   // (tile, K segment) items handled so far: selects the accumulator buffer
      bool ok = true;
      for (int item = pair; item < p.n_items && ok; item += n_pairs) {
        int tile, part, kt_begin, kt_end;
        item_decode(p, item, kt_total, tile, part, kt_begin, kt_end);
        for (int kt0 = kt_begin; kt0 < kt_end && ok; kt0 += p.kt_seg, ++local) {
          const int as = local & 1;
          const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
          if (!mbar_wait_cluster(tempty0 + 8 * as, aphase ^ 1, abortp, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tacc = tmem_base + (uint32_t)(as * BN);
          const int kt1 = min(kt_end, kt0 + p.kt_seg);
          for (int kt = kt0; kt < kt1; ++kt) {
            if (!mbar_wait_cluster(full0 + 8 * stage, phase, abortp, p.status)) { ok = false; break; }
            tc_fence_after();
            // One thread issues every MMA: the descriptors of stage 0 are formed once and only their address field
            // moves, and every MMA but a tile's first carries a constant accumulate flag, so that the instructions
            // around a tcgen05.mma stay well below the time it takes to execute.
            const uint64_t da = d0 + (uint64_t)(uint32_t)(stage * (STAGE_BYTES >> 4));
            const uint64_t dal = da + (A_BYTES >> 4);
            const uint64_t dbm = da + (((SPLIT ? 2 : 1) * A_BYTES) >> 4);
            const uint64_t dbl = dbm + (B_BYTES >> 4);
            const uint32_t acc = (uint32_t)(kt > kt0);
            if (SPLIT) {
              umma_first<H16>(tacc, dal, dbm, idesc, acc);
              umma_acc<H16>(tacc, da, dbl, idesc);
              umma_acc<H16>(tacc, da, dbm, idesc);
            } else {
              umma_first<H16>(tacc, da, dbm, idesc, acc);
            }
#pragma unroll
            for (int k = 1; k < BK / 8; ++k) {
              // 8 fp32 (16 halves) of K: 32 bytes along the row, or 16 k-rows of 128 bytes
              const uint64_t ko = (uint64_t)(MN ? k * (2048 >> 4) : k * (32 >> 4));
              if (SPLIT) {
                umma_acc<H16>(tacc, dal + ko, dbm + ko, idesc);
                umma_acc<H16>(tacc, da + ko, dbl + ko, idesc);
              }
              umma_acc<H16>(tacc, da + ko, dbm + ko, idesc);
            }
            umma_commit_pair(empty0 + 8 * stage);   // frees the stage in both CTAs once these MMAs have read it
            if (++stage == STAGES) { stage = 0; phase ^= 1; }
          }
          if (ok) umma_commit_pair(tfull0 + 8 * as);
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps (both CTAs)
    // Eight warps: warp w reads TMEM lanes 32 (w % 4) .. and one half (128 columns) of the accumulator, one
    // row per lane.  The K segments of a tile are summed in registers (ordinary round-to-nearest adds), so the
    // accumulator buffer is handed back right after it has been read and C is touched once per tile.
    const int q = warp & 3;
    const int half = (warp - 2) >> 2;
    float4* stg = reinterpret_cast<float4*>(smem + (size_t)STAGES * STAGE_BYTES + (size_t)(warp - 2) * EPI_BYTES);
    int local = 0;
    bool ok = true;
    if (p.dependent) grid_dependency_wait();
    for (int item = pair; item < p.n_items && ok; item += n_pairs) {
      int tile, part, kt_begin, kt_end, mt, nt;
      item_decode(p, item, kt_total, tile, part, kt_begin, kt_end);
      tile_coords(p, tile, mt, nt);
      float acc[EPI_COLS];
#pragma unroll
      for (int i = 0; i < EPI_COLS; ++i) acc[i] = 0.f;
      for (int kt0 = kt_begin; kt0 < kt_end && ok; kt0 += p.kt_seg, ++local) {
        const int as = local & 1;
        const uint32_t aphase = (uint32_t)(local >> 1) & 1u;
        if (!mbar_wait(tfull0 + 8 * as, aphase, abortp, p.status)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int ch = 0; ch < EPI_COLS / 32; ++ch) {
          if (FEW && half * EPI_COLS + ch * 32 >= p.tile_m) continue;    // warp-uniform
          uint32_t r[32];
          tmem_ld32(tmem_base + (uint32_t)(as * BN + half * EPI_COLS + ch * 32) + ((uint32_t)(q * 32) << 16), r);
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[ch * 32 + i] += __uint_as_float(r[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_cta(tempty0 + 8 * as, 0));
      }
      if (!ok) break;
      if (FEW) {
        // lane = column of C, accumulator column = row: 128 bytes of a row per store; a piece into its slab, [row][column]
        const int64_t col = (int64_t)nt * BN + rank * BM + q * 32 + lane, row0 = (int64_t)mt * p.tile_m;
        float* out = part < 0 ? p.C + row0 * p.ldc + col
                              : p.slabs + ((int64_t)(tile - p.split_first) * p.split_parts + part) * (BMP * BN) + rank * BM + q * 32 + lane;
        const int64_t ld = part < 0 ? p.ldc : BN;
        const int64_t left = p.M - row0;
        const int rows = (int)(left < p.tile_m ? left : p.tile_m) - half * EPI_COLS;
        out += (int64_t)half * EPI_COLS * ld;
        if (col < p.N) {                                                 // warp-uniform (N is a multiple of 32)
#pragma unroll
          for (int i = 0; i < EPI_COLS; ++i)
            if (i < rows) out[i * ld] = acc[i];
        }
        continue;
      }
      // A whole tile goes to C; the partial sums of a piece go, plainly, to this item's slab: one copy of the code for both (with
      // two the registers of a lane's sums spill twice as often; 1,024 x 4,480, 16 iterations 11.77 -> 11.67 ms), two in the Gram,
      // which is faster so (1,024 channels, 30,000 tokens 194 -> 189 us).
      const int64_t row0 = (int64_t)mt * BMP + rank * BM;
      float* const slab = p.slabs + (((int64_t)(tile - p.split_first) * p.split_parts + part) * 2 + rank) * (BM * BN);
      const int64_t rows = p.M - row0 < BM ? p.M - row0 : BM;              // (rows past the end are not read back)
      double dot1 = 0.0, dot2 = 0.0;
      if (MN && part >= 0) {
        write_out<false>(acc, stg, lane, slab, BN, 1, q * 32, half * EPI_COLS, rows, BN, false, false, nullptr, nullptr, nullptr, nullptr, 0,
                         dot1, dot2);
        continue;
      }
      const bool whole = MN || part < 0;
      float* const out = whole ? p.C : slab;
      write_out<DOTS>(acc, stg, lane, out, whole ? p.ldc : BN, whole ? p.c_vec : 1, (whole ? row0 : 0) + q * 32,
                      (whole ? (int64_t)nt * BN : 0) + half * EPI_COLS, whole ? p.M : rows, whole ? p.N : BN, whole && p.accumulate != 0,
                      whole && p.symmetric_lower != 0, whole ? p.row_scale : nullptr, whole ? p.col_scale : nullptr, whole ? p.d1 : nullptr,
                      whole ? p.d2 : nullptr, p.ldc, dot1, dot2);
      if (!whole) continue;
      if (DOTS) {
        for (int o = 16; o > 0; o >>= 1) {
          dot1 += __shfl_down_sync(0xffffffffu, dot1, o);
          dot2 += __shfl_down_sync(0xffffffffu, dot2, o);
        }
        if (lane == 0) {
          if (p.part1) p.part1[(int64_t)tile * PARTS + rank * 8 + half * 4 + q] = dot1;
          if (p.part2) p.part2[(int64_t)tile * PARTS + rank * 8 + half * 4 + q] = dot2;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                  // neither CTA leaves while its partner may still signal it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// Adds the slabs of every split tile into C (+ what C held, if the product accumulates) and forms the tile's
// share of the fused dot products.  Sixteen CTAs per split tile, 16 rows each, one float4 per thread (the kernel is nothing
// but latency), four pieces in flight; fixed order.
constexpr int FIX_NT = BMP / PARTS * BN / 4;
__global__ void __launch_bounds__(FIX_NT) tc_gemm_fixup_kernel(const Params p) {
  constexpr int FR = BMP / PARTS;                         // rows per CTA
  grid_begin();
  if (p.only_if && *p.only_if == 0) return;
  const int slots = gridDim.x / (p.n_tiles_total - p.split_first);       // PARTS, or those that hold rows
  const int tile = p.split_first + blockIdx.x / slots, slot = blockIdx.x % slots;
  int mt, nt;
  tile_coords(p, tile, mt, nt);
  const float* slab0 = p.slabs + (int64_t)(blockIdx.x / slots) * p.split_parts * (BMP * BN) + (int64_t)slot * FR * BN;
  double d1 = 0.0, d2 = 0.0;
  const int r = threadIdx.x / (BN / 4), c4 = (threadIdx.x % (BN / 4)) * 4;
  const int64_t grow = (int64_t)mt * p.tile_m + slot * FR + r, gcol = (int64_t)nt * BN + c4;
  if (slot * FR + r < p.tile_m && grow < p.M && gcol < p.N && !(p.symmetric_lower && gcol > grow)) {
    const float* sp = slab0 + (int64_t)r * BN + c4;
    float4 v = *reinterpret_cast<const float4*>(sp);
#pragma unroll 4
    for (int k = 1; k < p.split_parts; ++k) {
      const float4 w = *reinterpret_cast<const float4*>(sp + (int64_t)k * (BMP * BN));
      v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    if (p.row_scale) {
      // one scale after the other, as write_out applies them: their product may leave fp32's range where the result does not
      const float rs = p.row_scale[grow];
      const float4 cs = *reinterpret_cast<const float4*>(p.col_scale + gcol);
      v.x = v.x * rs * cs.x; v.y = v.y * rs * cs.y; v.z = v.z * rs * cs.z; v.w = v.w * rs * cs.w;
    }
    float* cp = p.C + grow * p.ldc + gcol;
    if (p.accumulate) {
      const float4 o = load4(cp, p.c_vec);
      v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
    }
    store4(cp, v, p.c_vec);
    if (p.d1) {
      const float4 w = *reinterpret_cast<const float4*>(p.d1 + grow * p.ldc + gcol);
      d1 += (double)(v.x * w.x + v.y * w.y) + (double)(v.z * w.z + v.w * w.w);
    }
    if (p.d2) {
      const float4 w = *reinterpret_cast<const float4*>(p.d2 + grow * p.ldc + gcol);
      d2 += (double)(v.x * w.x + v.y * w.y) + (double)(v.z * w.z + v.w * w.w);
    }
  }
  if (!p.part1 && !p.part2) return;
  __shared__ double red1[FIX_NT / 32], red2[FIX_NT / 32];
  for (int o = 16; o > 0; o >>= 1) {
    d1 += __shfl_down_sync(0xffffffffu, d1, o);
    d2 += __shfl_down_sync(0xffffffffu, d2, o);
  }
  if ((threadIdx.x & 31) == 0) { red1[threadIdx.x >> 5] = d1; red2[threadIdx.x >> 5] = d2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t1 = 0.0, t2 = 0.0;
    for (int w = 0; w < FIX_NT / 32; ++w) { t1 += red1[w]; t2 += red2[w]; }
    // the slots of the tile's epilogue warps, filled by this kernel's CTAs instead
    if (p.part1) p.part1[(int64_t)tile * PARTS + slot] = t1;
    if (p.part2) p.part2[(int64_t)tile * PARTS + slot] = t2;
  }
}

// ------------------------------------------------------------------ host side
// [rows][K] fp32, leading dimension ld: box = BK x box_rows, 128-byte swizzle, zero fill out of bounds.
// bits16: 0 fp32 elements, 1 bf16, 2 fp16
// mn: the array is [K][rows] of 16-bit elements (contiguous along the rows of the operand): box = 64 rows x 64 k
bool make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t K, int64_t ld, int box_rows, int bits16, bool mn) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)(mn ? rows : K), (cuuint64_t)(mn ? K : rows)};
  cuuint64_t strides[1] = {(cuuint64_t)ld * (bits16 ? 2 : 4)};
  cuuint32_t box[2] = {(cuuint32_t)(bits16 ? 64 : BK), (cuuint32_t)(mn ? 64 : box_rows)};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapDataType dt = bits16 == 0 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : bits16 == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  CUresult r = enc(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int PASSES, bool MN, bool FEW = false, bool DOTS = false>
armor_status launch_impl(armor_ctx* c, const TcGemm& g, Params p, cudaStream_t s) {
  CUtensorMap mA, mAlo, mB, mBlo;
  constexpr bool SPLIT = (PASSES == 3 || PASSES == 6);
  constexpr bool H16 = (PASSES == 0 || PASSES == 6);
  const int bits16 = H16 ? (g.fp16 ? 2 : 1) : 0;
  if (!make_map(&mA, g.A, g.M, g.K, g.lda, FEW ? p.tile_m / 2 : BM, bits16, MN)) return ARMOR_ERR_CUDA;
  if (!make_map(&mB, g.B, g.N, g.K, g.ldb, BNH, bits16, MN)) return ARMOR_ERR_CUDA;
  if (SPLIT) {
    if (!make_map(&mAlo, g.Alo, g.M, g.K, g.lda, BM, bits16, MN)) return ARMOR_ERR_CUDA;
    if (!make_map(&mBlo, g.Blo, g.N, g.K, g.ldb, BNH, bits16, MN)) return ARMOR_ERR_CUDA;
  } else {
    mAlo = mA;
    mBlo = mB;
  }
  constexpr size_t SMEM = (size_t)Ring<PASSES>::STAGES * Ring<PASSES>::BYTES + 1024 + 8 * EPI_BYTES;
  static PerDeviceOnce attr;
  if (ensure_dynamic_smem(attr, c->device, tc_gemm_kernel<PASSES, MN, FEW, DOTS>, SMEM) != ARMOR_OK) return ARMOR_ERR_CUDA;
  const int n_pairs = c->n_sm / 2;
  if (n_pairs < 1) return ARMOR_ERR_UNSUPPORTED;
  // Tail split: the tiles of the last, partly filled wave are cut along K so that their pieces fill the wave.  Where the
  // contraction is summed in segments, the pieces are the segments themselves (the slabs are then added in the order in which
  // an uncut tile adds its segments: the same bits), except that the tiles of a general product are cut in two to four equal
  // pieces where these are whole segments or lie within one: fewer slabs.  One-pass products without segments: any pieces.
  p.split_first = p.n_tiles_total; p.split_parts = 1; p.split_kt = 0; p.n_items = p.n_tiles_total; p.slabs = c->gemm_slabs;
  const int kt_total = (int)((p.K + (H16 ? 64 : BK) - 1) / (H16 ? 64 : BK));
  const int rem = p.n_tiles_total % n_pairs;
  if (c->gemm_slabs && rem > 0) {
    // A piece writes 256 KB of sums and the second kernel reads them: about 6 us, 8 k-tiles with three MMAs per
    // product (0.8 us each) or 24 with one, which the shorter wave has to give back
    const int worth = SPLIT ? 8 : 24;
    const int fill = n_pairs / rem;                                // pieces per tile that still fit the wave
    int per = kt_total;
    if (!SPLIT && p.kt_seg >= kt_total) {
      // (more pieces are more slabs to add: at most four, eight of the bf16 product: 1,024 x 5,120, 600 tokens 80 -> 78 us)
      const int most = PASSES == 0 && !MN ? 8 : 4;
      if (fill > 1) per = (kt_total + (fill < most ? fill : most) - 1) / (fill < most ? fill : most);
    } else {
      for (int parts = fill < 4 ? fill : 4; parts > 1 && !p.symmetric_lower && per == kt_total; --parts)
        if (kt_total % parts == 0 && kt_total / parts >= 8 && ((kt_total / parts) % p.kt_seg == 0 || kt_total / parts <= p.kt_seg))
          per = kt_total / parts;
      if (per == kt_total && fill > 1 && p.kt_seg < kt_total) per = p.kt_seg;
    }
    const int parts = (kt_total + per - 1) / per;
    // (a slab holds 128 x 256 sums, a piece writes two.)  More than the context's own slabs come with a Gram of few channels, whose
    // pieces may take several rounds of the pairs: 0.8 or 0.25 us a k-tile saved against 0.1 us a piece for its 256 KB and 6 us.
    const int64_t slabs = (int64_t)rem * parts * 2;
    const int rounds = (rem * parts + n_pairs - 1) / n_pairs;
    const bool pays = slabs <= ARMOR_GEMM_SLABS || (kt_total - rounds * per) * (SPLIT ? 32 : 10) > 4 * rem * parts + 240;
    if (parts > 1 && kt_total - per >= worth && slabs <= c->gemm_slab_count && pays) {
      p.split_kt = per;
      p.split_parts = parts;
      p.split_first = p.n_tiles_total - rem;
      p.n_items = p.split_first + rem * parts;
    }
  }
  const int pairs = p.n_items < n_pairs ? p.n_items : n_pairs;
  {
    KTimer kt(c, ARMOR_KC_GEMM, p.only_if ? 0.0 : p.symmetric_lower ? (double)p.M * (double)(p.N + BM) * (double)p.K
                                                  : 2.0 * (double)p.M * (double)p.N * (double)p.K, s);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2 * pairs); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = SMEM; cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = !MN || p.dependent ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, tc_gemm_kernel<PASSES, MN, FEW, DOTS>, mA, mAlo, mB, mBlo, p) != cudaSuccess) return ARMOR_ERR_CUDA;
    if (p.split_parts > 1) {
      // 16 rows per CTA; the slots of rows that do not exist are launched only where each has a partial sum to write
      const int64_t rows = p.M < p.tile_m ? p.M : p.tile_m;
      const int slots = (p.part1 || p.part2) ? PARTS : (int)((rows + BMP / PARTS - 1) / (BMP / PARTS));
      cudaLaunchConfig_t fc{};
      fc.gridDim = dim3(slots * (p.n_tiles_total - p.split_first)); fc.blockDim = dim3(FIX_NT); fc.stream = s;
      fc.attrs = &at[1]; fc.numAttrs = MN ? 0 : 1;
      if (cudaLaunchKernelEx(&fc, tc_gemm_fixup_kernel, p) != cudaSuccess) return ARMOR_ERR_CUDA;
      c->launches++;
    }
  }
  c->launches++;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

}  // namespace

bool tc_gemm_shape_ok(int64_t M, int64_t N, int64_t K) {
  return M > 0 && N > 0 && K > 0 && (N % 32 == 0) && (K % 4 == 0);
}

armor_status launch_tc_gemm(armor_ctx* c, const TcGemm& g, int* n_part, cudaStream_t s) {
  if (!tc_gemm_shape_ok(g.M, g.N, g.mn_major ? 4 : g.K)) return ARMOR_ERR_UNSUPPORTED;   // (k beyond K reads as zero)
  const bool h16 = (g.passes == 0 || g.passes == 6);
  if ((g.lda % (h16 ? 8 : 4)) || (g.ldb % (h16 ? 8 : 4)) || (g.ldc % 4)) return ARMOR_ERR_UNSUPPORTED;
  if ((g.row_scale == nullptr) != (g.col_scale == nullptr)) return ARMOR_ERR_INVALID_ARG;
  if (g.symmetric_lower && g.M != g.N) return ARMOR_ERR_INVALID_ARG;
  Params p{};
  p.C = g.C; p.ldc = g.ldc; p.M = g.M; p.N = g.N; p.K = g.K;
  p.m_tiles = (int)((g.M + BMP - 1) / BMP);
  p.n_tiles = (int)((g.N + BN - 1) / BN);
  p.n_tiles_total = g.symmetric_lower ? p.m_tiles * (p.m_tiles + 1) / 2 : p.m_tiles * p.n_tiles;
  p.accumulate = g.accumulate; p.symmetric_lower = g.symmetric_lower;
  p.d1 = g.d1; p.d2 = g.d2; p.part1 = g.part1; p.part2 = g.part2;
  p.row_scale = g.row_scale; p.col_scale = g.col_scale; p.dependent = g.dependent; p.f16 = g.fp16;
  p.only_if = g.only_if;
  p.status = c->status;
  p.c_vec = (reinterpret_cast<uintptr_t>(g.C) % 16 == 0) ? 1 : 0;   // (ldc is a multiple of 4)
  const int bke = h16 ? 64 : BK;
  p.kt_seg = g.k_segment > 0 ? (int)((g.k_segment + bke - 1) / bke) : (int)((g.K + bke - 1) / bke);
  if (p.kt_seg < 1) p.kt_seg = 1;
  p.tile_m = BMP;
  if (n_part) *n_part = PARTS * p.n_tiles_total;
  const bool dots = g.part1 || g.part2;
  if (g.mn_major) {
    // a map's rows start at multiples of 64 elements; the base and the leading dimension must be multiples of 16 bytes
    if (!h16 || dots || reinterpret_cast<uintptr_t>(g.A) % 16 || reinterpret_cast<uintptr_t>(g.B) % 16) return ARMOR_ERR_UNSUPPORTED;
    return g.passes == 6 ? launch_impl<6, true>(c, g, p, s) : launch_impl<0, true>(c, g, p, s);
  }
  if (dots) {
    if (g.passes == 3) return launch_impl<3, false, false, true>(c, g, p, s);
    if (g.passes == 6) return launch_impl<6, false, false, true>(c, g, p, s);
    if (g.passes == 1) return launch_impl<1, false, false, true>(c, g, p, s);
    return ARMOR_ERR_UNSUPPORTED;
  }
  if (g.passes == 3) return launch_impl<3, false>(c, g, p, s);
  if (g.passes == 6) return launch_impl<6, false>(c, g, p, s);
  if (g.passes == 0) {
    // Few rows: dealt evenly to one or two tiles.  (The core product of a forward with them, whole pass at 8192 x 8192: 1 token
    // 156 -> 142 us, 300 186 -> 176, 512 198 -> 191; from three tiles on the two forms are alike.)
    const int even = (int)((g.M + p.m_tiles - 1) / p.m_tiles + 31) / 32 * 32;
    if (p.m_tiles <= 2 && !g.row_scale && !g.accumulate && !g.symmetric_lower) {
      p.tile_m = even;
      return launch_impl<0, false, true>(c, g, p, s);
    }
    return launch_impl<0, false>(c, g, p, s);
  }
  return launch_impl<1, false>(c, g, p, s);
}
