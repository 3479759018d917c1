// Internal declarations shared by the translation units of libarmor.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "armor.h"

// ---------------------------------------------------------------- scalars
// Device-resident double scalars (one set per context).  Kernels read step
// lengths and accept flags from here so that no sub-step needs the host.
enum {
  SC_L0 = 0,     // <E H_w, E> at the start of the iteration
  SC_DEC_A,      // exact decrease of the A-step
  SC_GD_B,       // <Gamma^B, Delta>
  SC_Q_B,        // tr(V H_w V^T) of the B direction
  SC_NRM_S,      // ||Gamma (.) M||_F^2
  SC_Q_S,        // tr(V H_w V^T) of the S direction
  SC_EHV_M,      // <E H_w, V> of the group updates
  SC_Q_M,        // tr(V H_w V^T) of the group updates
  SC_TAU_B,
  SC_TAU_S,
  SC_ACCEPT,     // 1.0 if the group updates are kept
  SC_DL_M,       // exact loss change of the group updates
  SC_LOSS,       // running loss inside an iteration
  SC_BETA_A,     // ||A^T A||_F^2 (BETA step)
  SC_BETA_K,     // ||B H_w B^T||_F^2 (BETA step)
  SC_TMP0,
  SC_TMP1,
  SC_TAU_A,      // step of the A gradient step (ab_step GD)
  SC_HB_A,       // beta_A / 2 of Eq. lrA
  SC_HB_B,       // beta_B / 2 of Eq. lrB
  SC_COUNT = 32
};

// status words in the device status buffer
enum {
  ST_CHOL_FAILS = 0, ST_FIRST_FAIL = 1, ST_WAIT_TIMEOUTS = 2, ST_LAST_ERR = 3, ST_SPARSE_BAD_GROUPS = 4,
  ST_NONFINITE_W = 5,    // NaN / Inf entries seen in W by the input screening (cumulative)
  ST_NONFINITE_H = 6,    // NaN / Inf entries seen in H
  ST_NEG_DIAG_H = 7,     // negative diagonal entries of H (H cannot be a Gram matrix)
  ST_DEAD_CHANNELS = 8,  // zero diagonal entries of H in the last screened call (legal: the channel carries no weight)
  ST_POISON = 9,         // 1 while the last screened call had unusable inputs: its updates were all withheld
  ST_H_RANGE = 10,       // entries of the scaled H beyond the fp16 range (FP16X3; H not positive semidefinite): clamped
  ST_COUNT = 16
};

static const int ARMOR_MAX_PIECES = 16;   // graph pieces of one iteration when it is captured around its dense products

// One selected group per (i, j) block of the sparse core (Algorithm 3).
struct SelRec {
  int32_t valid;      // 0: nothing selected in this block
  int32_t row;        // global row r
  int32_t cgrp;       // group index inside the row (columns m*cgrp ..)
  int32_t new_mask;   // bit p <=> position p kept
  int32_t old_mask;
  float new_val[8];
  float old_val[8];
};

static const int ARMOR_GEMM_SLABS = 160;  // slabs of partial sums of cut tiles in the workspace
static const int ARMOR_DOT_BLOCKS = 592;  // 4 x 148 partial sums per reduction

struct armor_ctx {
  armor_config cfg;
  int64_t d_out, d_in, wn;  // wn = d_out * d_in
  int db, nbo, nbi;
  char* ws;
  size_t ws_bytes;
  // W-shaped fp32 scratch
  float *T, *E, *EH, *P, *U, *V, *VH, *Gam, *Tmp, *WH;
  // low parts of the left operands / of H for the three-pass tensor-core mode
  float *Lo, *Hlo;
  // [nb, db, db] scratch
  float *G, *GamA, *dA, *C, *GamB, *Delta, *Hjj, *Kfull, *Ktmp;
  float* Hinv;           // (H_jj + mu I)^-1 per column block, formed once per armor_bcd_step call
  int32_t* hinv_fail;    // [nbi] 1 where that block was not positive definite
  float *alpha, *hdiag;
  float *mA, *vA, *mB, *vB, *mS, *vS;   // Adam moment estimates (ab_step ADAM)
  float *Hq1, *Hq2;      // [d_in, d_in] scratch of the paper's step size (s_step BETA, full weighting)
  float* gemm_slabs;     // 128 x 256 slabs of partial sums of the dense product's split tail tiles
  int64_t gemm_slab_count;
  float* gpart;          // partial products of split contractions
  int64_t gpart_floats;
  // sparse-core update: per selected group z = delta^T B_j[rows of the group, :] and a = A_i[:, r]
  float *Zsel, *Acol, *Ysel;  // [nbi][nbo_pad][db], [nbo][nbi][db], [nbi][nbo_pad][d_in]
  int nbo_pad;                // nbo rounded up to a multiple of 32
  // three-pass fp16 mode: column scales derived from diag(H), per-row output scales of the two operands,
  // per-channel maxima and output scales of a Gram chunk
  float *hpow, *rowscale, *rowscale2, *gscale;
  float* gscale2;       // output scales of the chunk staged in Xt_hi2
  unsigned* gmax;
  // Gram staging (split chunk of X; transposed in the tf32 modes)
  float *Xt_hi, *Xt_lo;
  float* Xt_hi2;        // second staging buffer (FP16X3): chunk p + 1 is staged on side_stream while chunk p is contracted
  cudaStream_t side_stream;
  cudaEvent_t ev_fork, ev_staged[2], ev_used[2];
  cudaEvent_t ev_prep, ev_prepared;   // the group solves' systems are formed on side_stream beside the core's update
  int64_t gram_rows;  // rows of X staged per pass
  double* sc;         // [SC_COUNT]
  double* partials;   // [2][8 * npart] partial sums of the fused / streaming reductions
  int64_t npart;
  double* partblk;    // [max(4 * nbo, 4 * nbi, nbo * nbi)] per-block partial sums
  double* quadpart;   // [nbo * nbi] per-block terms of the group updates' quadratic form
  double* colpart;    // [64][d_in] column partial sums of the normalisation
  double* partA;      // [4 * nbo] the A-step's decreases, kept until the B-step's bookkeeping
  int32_t* failflag;  // [2][max(nbo, nbi)] failed solves of the A-step, of the B-step
  SelRec* sel;        // [nbo * nbi]
  float* tab_key;     // [nbo * nbi] winning race key of every block (single draw)
  unsigned long long* tab_g;   // its global group index
  int32_t* status;    // [ST_COUNT]
  int32_t* screen;    // [4] per-call counters of the input screening
  int32_t* core_dense;   // fp32 forward: 1 if the core is not 2:4, so that the dense product runs instead of the sparse one
  int64_t* it_dev;    // iteration index inside the running armor_bcd_step call (advanced by the first kernel of an iteration)
  int use_graphs;     // 1: repeated iterations of a call are replayed from a CUDA graph
  cudaStream_t cap_stream;   // the context's own stream, used only to capture that graph
  // Capture in pieces (while the dense products are being timed with events, which a graph cannot replay): every
  // dense product with H closes the piece being captured, is remembered with its arguments and opens the next
  // piece; the replay alternates graph pieces and directly launched products.
  int cap_split;             // 1 while such a capture runs
  int cap_n;                 // pieces closed so far (= products remembered)
  int cap_failed;            // too many pieces or a failed capture call: the iteration is enqueued directly instead
  cudaGraph_t cap_graph[ARMOR_MAX_PIECES];
  struct RmulCall { const float* in; const float* H; float* out; int64_t rows; const float* d1; double* out1;
                    const float* d2; double* out2; } cap_call[ARMOR_MAX_PIECES];
  int64_t launches;
  int device;           // the device that was current at armor_create; every call must be issued with it current
  int n_sm;             // its number of SMs
  int tc_blocks;        // 1, 2, 3: block products and per-block Grams on the tensor cores where the shape allows.
                        // 1: the streaming kernel for every product; 2: with d_block = 128 the kernel that keeps the
                        // wrapper block in tensor memory (products and dual products); 3 (default): that kernel for
                        // dual products and other three-pass
                        // products of many tiles, else the streaming kernel, the two-sided kernel where both wrappers apply;
                        // 0: always the fp32 CUDA-core kernels (exact products with 0 and 1)
  int gram_pairs;       // 1: the two per-block Grams of a step in one launch (shared operand read once)
  armor_status host_err;   // first launch failure inside the running call that no fallback covers
  int kg;               // groups drawn per block in one sparse-core update (mask_groups, at least 1)
  int block_one_pass;   // 1: products with the wrappers take one tf32 pass (the bf16 forward, whose operands are
                        // rounded to 8 bits anyway); 0: three passes, fp32-grade
  // identity of the H whose low part is cached in Hlo
  const float* h_cached;
  // optional event timing of the launches: 0 off, 1 the dense tensor-core products only, 2 every kernel class
  int timing_on;
  int timing_n;              // launches recorded
  cudaEvent_t* ev_beg;       // [ARMOR_MAX_TIMED]
  cudaEvent_t* ev_end;
  int32_t* ev_cls;           // kernel class of the recorded launch (ARMOR_KC_*)
  double* ev_work;           // its algorithmic work: flops (dense products, Cholesky) or bytes (everything else)
  int ev_created;
};
static const int ARMOR_MAX_TIMED = 8192;

// ---------------------------------------------------------------- programmatic dependent launches
// The kernels of an iteration are short (a layer of 256 x 256: 36 launches, most of them of 2 to 4 us, solves 9, contractions of 256 7 to 9), so the gap between the end of one and
// the start of the next counts.  They open with grid_begin(): launched with the attribute below, a kernel's CTAs are put on the
// SMs once every CTA of the kernel before it has come past its own grid_begin(), and wait there until that kernel has ended and
// its writes are visible; everything earlier in the stream has ended by then as well.  (Letting the next kernel in before
// the wait made chains of waiting kernels: 3,280 us for 20 iterations of a 256 x 256 layer, 2,996 without any of this, 2,747
// this way.)  Three rules follow.  grid_begin() stands before the first access to global memory and before any return.  A
// kernel that takes tensor memory takes it first: the CTAs that grid_begin() lets in may wait for theirs while this one runs.
// And what a kernel reads is not declared __restrict__, const or not, nor read through __ldg (but for data written two or more
// kernels before: it is there when a kernel starts): a load of data that nothing else is known to write may be moved above the wait.
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Kernels of more threads than this start behind their predecessor as ever: CTAs of a streaming kernel that wait in their
// hundreds beside the products slow those down (a 4096 x 4096 layer's diagonal Adam iterations with a limit of 592 CTAs of 256
// threads 6,561 us, 6,775 without a limit, 6,626 with no dependent launches; limits of 1, 148 and 1,100 CTAs: 256 x 256 layer 2,886,
// 2,767 and 2,746 us).
constexpr int64_t DEPENDENT_THREADS = 592 * 256;
// A stream to launch on; waits: for another stream's event as well, so that what is launched starts behind everything it waits for.
struct LaunchStream {
  cudaStream_t s; bool waits; int cluster;            // cluster: CTAs of one along x
  LaunchStream(cudaStream_t s_, bool waits_ = false, int cluster_ = 1) : s(s_), waits(waits_), cluster(cluster_) {}
};
template <typename... Params, typename... Args>
inline void launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, LaunchStream s, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s.s;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (!s.waits && (int64_t)grid.x * grid.y * grid.z * block.x * block.y <= DEPENDENT_THREADS) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (s.cluster > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = (unsigned)s.cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = at; cfg.numAttrs = n;
  cudaLaunchKernelEx(&cfg, kernel, Params(args)...);   // (an error is found by the call's cudaGetLastError)
}

// Brackets the launches made during its lifetime with a pair of events on the launching stream when timing is on.
struct KTimer {
  armor_ctx* c; cudaStream_t s; int slot;
  KTimer(armor_ctx* c_, int cls, double work, cudaStream_t s_) : c(c_), s(s_), slot(-1) {
    if (!c->timing_on || (c->timing_on == 1 && cls != ARMOR_KC_GEMM) || c->timing_n >= c->ev_created) return;
    slot = c->timing_n++;
    c->ev_cls[slot] = cls;
    c->ev_work[slot] = work;
    cudaEventRecord(c->ev_beg[slot], s);
  }
  ~KTimer() { if (slot >= 0) cudaEventRecord(c->ev_end[slot], s); }
  KTimer(const KTimer&) = delete;
  KTimer& operator=(const KTimer&) = delete;
};

#define ARMOR_CUDA_OK(expr)                                  \
  do {                                                       \
    cudaError_t _e = (expr);                                 \
    if (_e != cudaSuccess) return ARMOR_ERR_CUDA;            \
  } while (0)

// ---------------------------------------------------------------- launchers
// Generic strided batched fp32 GEMM on CUDA cores:
//   C_b[m][n] = alpha * sum_k A_b[m][k] B_b[k][n] + beta * D_b[m][n]
// element (m,k) of A_b lives at A + b*sAb + m*sAm + k*sAk (likewise B, C, D).
struct BGemm {
  const float* A; int64_t sAb, sAm, sAk;
  const float* B; int64_t sBb, sBk, sBn;
  float* C; int64_t sCb, sCm, sCn;
  const float* D; int64_t sDb, sDm, sDn;
  int M, N, K, batch;
  float alpha, beta;
  // two-level batch: batch index b = bo * batch_inner + bi, operand offset bo * s?b2 + bi * s?b
  // (batch_inner == 0: one level)
  int batch_inner;
  int64_t sAb2, sBb2, sCb2, sDb2;
  // split of the contraction into ksplit equal chunks whose partial products are summed in a fixed order
  // (needs c->gpart; only without D)
  int ksplit;
  int waits;             // see LaunchStream
};
void launch_bgemm(armor_ctx* c, const BGemm& g, cudaStream_t s);
// number of chunks a long contraction is cut into so that batch * tiles * chunks fills the GPU about twice
inline int pick_ksplit(int64_t batch, int64_t tiles, int64_t K) {
  int64_t ks = (296 + batch * tiles - 1) / (batch * tiles);
  if (ks > K / 256) ks = K / 256;
  while (ks > 1 && K % (16 * ks)) --ks;
  return ks < 1 ? 1 : (int)ks;
}

// block-diagonal products on row-major [rows, cols] matrices
//  right: out[:, jblk] = alpha * in[:, jblk] * Bblk[j] (+ beta * add[:, jblk]); transB uses Bblk[j]^T
//  left : out[iblk, :] = alpha * Ablk[i] * in[iblk, :] (+ beta * add[iblk, :]); transA uses Ablk[i]^T
void bd_right(armor_ctx* c, const float* in, const float* Bblk, bool transB, float* out, int64_t rows,
              int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);
void bd_left(armor_ctx* c, const float* Ablk, bool transA, const float* in, float* out, int64_t rows,
             int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);
// out = in Bdiag and outH = out H_w for the layer's shape [d_out, d_in] (one launch with the diagonal weighting where the
// tensor-core kernel takes d_block)
armor_status bd_right_H(armor_ctx* c, const float* in, const float* Bblk, const float* H, float* out, float* outH, cudaStream_t s);
// out = alpha * Lop X Rop with both wrappers (Lop_i = Lblk[i] or its transpose, Rop_j likewise): one fused launch on
// the tensor cores where the shape allows (d_block 128; the intermediate stays in tensor memory), else the two
// one-sided products through tmp
void bd_two_sided(armor_ctx* c, const float* Lblk, bool transL, const float* X, const float* Rblk, bool transR, float* tmp,
                  float* out, int64_t rows, int64_t cols, float alpha, cudaStream_t s);
// out = Ablk in2 and partial sums of <Ablk in1, Ablk in2> at part, *n_part of them (the consumer adds them up): one
// fused launch on the tensor cores (Ablk in1 never reaches memory), else two products (the first into tmp) and a dot
void bd_left_dual(armor_ctx* c, const float* Ablk, const float* in1, const float* in2, float* tmp, float* out,
                  int64_t rows, int64_t cols, double* part, int* n_part, cudaStream_t s);

// R = in Bdiag (into R), out = Ablk (R H_w) and partial sums of <Ablk R, Ablk (R H_w)>: the products behind a line search's step.  RH takes
// R H_w where a later move needs it (full weighting) or the kernels want it in memory; with the diagonal weighting and d_block 128 it
// stays in shared memory.  tmp: scratch
armor_status bd_direction(armor_ctx* c, const float* in, const float* Bblk, const float* Ablk, const float* H, float* R, float* RH, float* tmp,
                          float* out, double* part, int* n_part, cudaStream_t s);

// the same two products on the tensor cores (block_tcgen05.cu); d_block must be a multiple of 128
bool tc_block_ok(const armor_ctx* c, int64_t rows, int64_t cols);
armor_status tc_bd_right(armor_ctx* c, const float* in, const float* Bblk, bool transB, float* out, int64_t rows,
                         int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);
armor_status tc_bd_right_scaled(armor_ctx* c, const float* in, const float* Bblk, float* out, const float* colw, float* out2, int64_t rows, int64_t cols,
                                cudaStream_t s);
armor_status tc_bd_left(armor_ctx* c, const float* Ablk, bool transA, const float* in, float* out, int64_t rows,
                        int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);

// out = P in2 per block row, with the partial sums of <P in1, P in2> (four per 128 x 128 tile) at part
armor_status tc_bd_left_dual(armor_ctx* c, const float* Ablk, bool transA, const float* in1, const float* in2, float* out,
                             int64_t rows, int64_t cols, double* part, int* n_part, cudaStream_t s);

// both wrappers in one launch (block2_tcgen05.cu); d_block = 128
bool tc_block2_ok(const armor_ctx* c, int64_t rows, int64_t cols);
// moves -sc[slot] v that an array still has to make, in this order (v: arrays of the library's own, of the array's shape)
struct Moves {
  int n; const float* v[2]; int slot[2];
  void add(const float* x, int at) { v[n] = x; slot[n] = at; ++n; }
};
armor_status tc_two_sided(armor_ctx* c, const float* Lblk, bool transL, const float* X, const float* Rblk, bool transR,
                          float* out, int64_t rows, int64_t cols, float alpha, cudaStream_t s, const uint8_t* mask = nullptr,
                          double* norm_part = nullptr, int* n_norm = nullptr, const Moves& moves = Moves{});

// EH = E diag(colw) with E = add - Ablk in, partial sums of <E, EH> at part: one launch, E stays in the SMs
armor_status tc_bd_left_residual(armor_ctx* c, const float* Ablk, const float* in, const float* add, const float* colw,
                                 float* EH, int64_t rows, int64_t cols, double* part, int* n_part, cudaStream_t s);

// the same with the wrapper block held in tensor memory (blockres_tcgen05.cu); d_block = 128
bool tc_blockres_ok(const armor_ctx* c);
armor_status tc_blockres_right(armor_ctx* c, const float* in, const float* Bblk, bool transB, float* out, int64_t rows,
                               int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);
armor_status tc_blockres_left(armor_ctx* c, const float* Ablk, bool transA, const float* in, float* out, int64_t rows,
                              int64_t cols, float alpha, const float* add, float beta, cudaStream_t s, const float* colw = nullptr,
                              double* part = nullptr);

armor_status tc_blockres_thin(armor_ctx* c, const float* Z, const float* X, float* out, int n, int pad, int blocks, int64_t cols, cudaStream_t s);
armor_status tc_blockres_left_dual(armor_ctx* c, const float* Ablk, const float* in1, const float* in2, float* out,
                                   int64_t rows, int64_t cols, double* part, int* n_part, cudaStream_t s, const float* colw = nullptr);

// products and per-block Grams of 256 x 256 blocks on pairs of CTAs (blockpair_tcgen05.cu)
bool tc_blockpair_ok(const armor_ctx* c, int64_t tiles);   // tiles of 256 x 256
armor_status tc_blockpair_right(armor_ctx* c, const float* in, const float* Bblk, bool transB, float* out, int64_t rows,
                                int64_t cols, float alpha, const float* add, float beta, cudaStream_t s);
armor_status tc_blockpair_left(armor_ctx* c, const float* Ablk, bool transA, const float* in, float* out, int64_t rows,
                               int64_t cols, float alpha, const float* add, float beta, cudaStream_t s,
                               const float* in2 = nullptr, double* part = nullptr, int* n_part = nullptr);
armor_status tc_blockpair_gram(armor_ctx* c, const float* P, const float* T, bool by_rows, float* G, cudaStream_t s,
                               const float* P2 = nullptr, float* G2 = nullptr);

// per-block Grams over a long contraction on the tensor cores
bool tc_gram_ok(const armor_ctx* c);
armor_status tc_rowblock_gram(armor_ctx* c, const float* P, const float* T, float* G, cudaStream_t s);
armor_status tc_colblock_gram(armor_ctx* c, const float* U, const float* Y, float* Cm, cudaStream_t s);
// two Grams with a shared operand in one launch (the shared chunks are read once)
armor_status tc_gram_launch(armor_ctx* c, const float* A, const float* A2, const float* B, bool by_rows, bool self, float* C, float* C2,
                            int n_split, cudaStream_t s);
armor_status tc_rowblock_gram_pair(armor_ctx* c, const float* P, const float* P2, const float* T, float* G, float* G2,
                                   cudaStream_t s);
armor_status tc_colblock_gram_self_pair(armor_ctx* c, const float* U, const float* Y, float* Cm, float* Cm2, cudaStream_t s);
armor_status tc_select_rows_times_H(armor_ctx* c, const float* Z, const float* H, float* Y, int nbo_pad, cudaStream_t s);
// A tensor-core launch that is refused for its shape or alignment (UNSUPPORTED) is replaced by the CUDA-core
// kernel; any other failure is an error of the call: it is recorded and the entry point returns it.
inline bool tc_done(armor_ctx* c, armor_status st) {
  if (st == ARMOR_OK) return true;
  if (st == ARMOR_ERR_UNSUPPORTED) return false;
  if (c->host_err == ARMOR_OK) c->host_err = st;
  return true;
}
// what an entry point returns: the recorded launch failure, else the state of the runtime
inline armor_status finish_call(armor_ctx* c) {
  const armor_status st = c->host_err;
  c->host_err = ARMOR_OK;
  if (st != ARMOR_OK) return st;
  return cudaGetLastError() == cudaSuccess ? ARMOR_OK : ARMOR_ERR_CUDA;
}

// Function attributes (the dynamic shared-memory limit) hold per device: one bit per device ordinal and call
// site remembers where the attribute has been set.
struct PerDeviceOnce {
  std::atomic<unsigned long long> mask{0};
  bool done(int dev) const { return dev >= 0 && dev < 64 && ((mask.load(std::memory_order_relaxed) >> dev) & 1ull); }
  void set(int dev) { if (dev >= 0 && dev < 64) mask.fetch_or(1ull << dev, std::memory_order_relaxed); }
};
template <typename K>
inline armor_status ensure_dynamic_smem(PerDeviceOnce& once, int device, K kernel, size_t bytes) {
  if (once.done(device)) return ARMOR_OK;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
    return ARMOR_ERR_CUDA;
  once.set(device);
  return ARMOR_OK;
}

// out = in * H_w (FULL: dense GEMM by cfg.precision; DIAG: column scale) with up to two
// fused dot products <out, d1> -> sc[slot1], <out, d2> -> sc[slot2] (slot < 0: none).
armor_status rmul_H(armor_ctx* c, const float* in, const float* H, float* out, int64_t rows,
                    const float* d1, double* out1, const float* d2, double* out2, cudaStream_t s);
// per-call preparation of everything derived from H (diagonal, diagonal blocks, split copy)
armor_status prepare_H(armor_ctx* c, const float* H, cudaStream_t s);
armor_status gram_accumulate(armor_ctx* c, const void* X, int x_dtype, int64_t n_rows, int64_t ldx, float* H,
                             cudaStream_t s);
// z2 [n, d_out] = z1 [n, d_in] * S^T
armor_status apply_core(armor_ctx* c, const float* z1, const float* S, const void* packed, float* z2, int64_t n,
                        bool bf16, cudaStream_t s);

// the same in the three-pass fp16 mode with S split beforehand (once per call), up to gram_rows tokens at a time
// (sparse: on the sparse tensor cores unless S is not 2:4; core_f16_sparse says where that is faster, for calls of so many
// tokens; first: the call's first chunk)
bool core_f16_ok(const armor_ctx* c);
bool core_f16_sparse(const armor_ctx* c, int64_t n_tokens);
armor_status core_f16_split_S(armor_ctx* c, const float* S, bool sparse, cudaStream_t s);
armor_status core_f16_product(armor_ctx* c, const float* z1, const float* S, bool sparse, bool first, float* z2, int64_t n, cudaStream_t s);

// operand preparation of the three-pass fp16 mode (split_f16.cu)
void launch_f16_prepare_H(armor_ctx* c, const float* H, cudaStream_t s);   // hpow, scaled H as fp16 hi | lo in Hlo
void launch_f16_split_rows(armor_ctx* c, const float* in, int64_t ld, int64_t rows, int64_t cols, const float* colscale,
                           float post, void* hi, void* lo, float* out_scale, cudaStream_t s);
// the 2:4 core [d_out, d_in] as fp16 parts of its kept entries with their positions, see split_core24_kernel; *dense 1 if it is not 2:4
void launch_split_core24(armor_ctx* c, const float* S, void* hi, void* lo, void* E, float* scale, int32_t* dense, cudaStream_t s);
// z1 as launch_f16_split_rows has it, tokens that are not finite with NaN as their scale; with S, and if *dense, S as well
void launch_split_tokens(armor_ctx* c, const float* z, int64_t tokens, void* hi, void* lo, float* out_scale, const float* S, void* s_hi, void* s_lo,
                         float* s_scale, const int32_t* dense, cudaStream_t s);
float f16_H_post_scale();
armor_status launch_f16_gram_stage(armor_ctx* c, const void* X, int x_dtype, int64_t ldx, int64_t rows, int64_t cols,
                                   void* Thi, void* Tlo, float* gscale, cudaStream_t s);

// deterministic reductions (two stages, fixed order)
void dot_to_ptr(armor_ctx* c, const float* x, const float* y, int64_t n, double* out, cudaStream_t s);
void dot_partials(armor_ctx* c, const float* x, const float* y, int64_t n, double* part, cudaStream_t s);
void reduce_partials_to(armor_ctx* c, const double* part, int n, double* out, cudaStream_t s);

// streaming kernels (kernels_stream.cu)
void launch_colscale(armor_ctx* c, const float* in, const float* h, float* out, int64_t rows, int64_t cols,
                     cudaStream_t s);
void launch_extract_hblocks(armor_ctx* c, const float* H, cudaStream_t s);   // hdiag, Hjj (per h_mode)
void launch_masked_copy(armor_ctx* c, const float* Gam, const uint8_t* M, float* out, double* part,
                        cudaStream_t s);              // out = Gam (.) M; ARMOR_DOT_BLOCKS partial sums of ||out||^2
// y += sign * sc[slot] * x; for up to three arrays at once, the last may move by sc[slot_before] * x2_before first
void launch_axpy_slot(armor_ctx* c, float* y, const float* x, int64_t n, int slot, float sign,
                      cudaStream_t s);
void launch_axpy_multi(armor_ctx* c, float* y0, const float* x0, float s0, int64_t n0, float* y1, const float* x1, float s1,
                       int64_t n1, float* y2, const float* x2, float s2, int64_t n2, int slot, cudaStream_t s,
                       const float* x2_before = nullptr, int slot_before = 0);
void launch_init(armor_ctx* c, const float* W, const float* H, float* Wbar, float* r1, float* r2,
                 float* A, float* B, float* S, uint8_t* M, cudaStream_t s);
// st: base of the iteration records (the kernels add c->it_dev), or null
// advance: ++*c->it_dev first
void launch_zero_scalars(armor_ctx* c, bool advance, bool carry_loss, armor_iter_stats* st, cudaStream_t s);
// Input screening at the top of a call: counts non-finite entries of W and H and negative / zero diagonal
// entries of H into the status words and sets or clears ST_POISON for the call.
armor_status launch_screen_inputs(armor_ctx* c, const float* W, const float* H, cudaStream_t s);
// One Adam step (Kingma & Ba, Algorithm 1) on n parameters with gradient g = -2 * gamma; step counts from 1.
// M != nullptr: theta is the N:M core, one mask byte per m_group entries, masked-out entries stay zero.
void launch_adam(armor_ctx* c, float* theta, const float* gamma, float* m, float* v, int64_t n, const uint8_t* M,
                 int64_t step_base, cudaStream_t s);   // step = step_base + *c->it_dev
// part[b] = weight_b * || X_b ||_F for the nblk blocks of db x db floats in X; weight_b = 1, or the Euclidean
// norm of hdiag over the (b % nbi)-th block of columns; out = sum of the parts (fixed order)
void launch_block_fro_sum(armor_ctx* c, const float* X, int nblk, const float* hdiag, double* out, cudaStream_t s);
// per-iteration bookkeeping on the device: stage 0 start, 1 after A, 2 after B, 10 after both, 3 after S, 4 mask accept
// (p1, n1, slot1), (p2, n2, slot2): partial sums the stage first adds up into sc[slot] (a preceding dot product)
void launch_stage(armor_ctx* c, armor_iter_stats* st, int stage, const double* part, int npart, cudaStream_t s, const double* p1 = nullptr,
                  int n1 = 0, int slot1 = 0, const double* p2 = nullptr, int n2 = 0, int slot2 = 0);
void launch_scale_cols(armor_ctx* c, const float* in, const float* colscale, float* out, int64_t rows, int64_t cols, cudaStream_t s);
void launch_split_hilo(armor_ctx* c, const float* in, float* hi, float* lo, int64_t n, cudaStream_t s);
void launch_transpose_split(armor_ctx* c, const void* X, int x_dtype, int64_t ldx, int64_t rows, int64_t cols,
                            float* Thi, float* Tlo, int64_t ldt, cudaStream_t s);
void launch_mirror_lower(armor_ctx* c, float* H, int64_t n, cudaStream_t s, const void* X_bf16 = nullptr, int64_t ldx = 0,
                         int64_t n_rows = 0, const float* in_range = nullptr);
// in_range[k] = 0 for a channel of X (bf16, [n_rows][ldx], rows on 16-byte boundaries) that is not all zeros and nowhere reaches
// 2^-57 in magnitude, else 1
void launch_gram_range(armor_ctx* c, const void* X_bf16, int64_t ldx, int64_t n_rows, float* in_range, cudaStream_t s);
void launch_bf16_to_f32(armor_ctx* c, const void* in, const float* colscale, float* out, int64_t rows, int64_t cols,
                        cudaStream_t s);
void launch_f32_to_bf16(armor_ctx* c, const float* in, const float* colscale, void* out, int64_t rows, int64_t cols,
                        cudaStream_t s);

// block solves (kernels_chol.cu)
// mode 0: X = rhs (G + lam I)^-1, A += X, out = X, part[b] = exact decrease of block b
// mode 1: out = (G + lam I)^-1 rhs
// mode 2: out = rhs (G + lam I)^-1, part[b] = <dotw, out>
// partial sums written per block by launch_chol (modes 0 and 2)
int chol_parts_per_block(int db, int nb);
// (H_jj + mu I)^-1 for every column block into c->Hinv (H_jj does not change inside a call), failures into c->hinv_fail
armor_status launch_hjj_inverse(armor_ctx* c, cudaStream_t s);
// after Delta = Y Hinv: zeroes the blocks whose H_jj was not positive definite (raising their failflag, as a failed
// solve would) and writes DELTA_PARTS partial sums of <dotw_j, Delta_j> per block
static const int DELTA_PARTS = 4;
void launch_delta_finish(armor_ctx* c, float* Delta, const float* dotw, double* part, cudaStream_t s);
armor_status launch_chol(armor_ctx* c, int mode, const float* Gmat, const float* rhs, float* out, const float* dotw,
                         float* A, int nb, double* part, cudaStream_t s);

// sparse-core update (kernels_mask.cu)
// alpha and the m x m diagonal blocks of K_j = Y_j B_j^T (Y = B_j H_jj, [nbi, db, db]) in one launch
void launch_mask_prep(armor_ctx* c, const float* A, const float* B, const float* Y, cudaStream_t s);
// selection counter t = t_base + t_mul * (*c->it_dev); with one draw per block also the vectors of launch_mask_quadratic
void launch_mask_select(armor_ctx* c, const float* A, const float* B, const float* Gam, const float* S, const uint8_t* M, uint64_t t_base,
                        uint64_t t_mul, LaunchStream s);
// exact loss change of the iteration's group updates without a dense product: the per-block terms of tr(V H_w V^T), V = A dS B,
// from the selection records, their sum and the decision (stage 4)
void launch_mask_quadratic(armor_ctx* c, const float* A, const float* B, const float* H, armor_iter_stats* st, cudaStream_t s);
// the accepted group updates: S and M, and with P (full weighting) P += dS B H_w, for which the guard has formed the rows
void launch_mask_commit(armor_ctx* c, float* S, uint8_t* M, float* P, armor_iter_stats* st, cudaStream_t s);

// tensor-core GEMM (gemm_tcgen05.cu):  C[M][N] (+)= sum_k A[m][k] * B[n][k]  (both K-major, fp32 storage).
// passes == 3 uses the split operands (A, Alo, B, Blo).  Partial dot products of the output tile with up
// to two W-shaped tensors go to dot partial buffers.
struct TcGemm {
  const void* A; const void* Alo; int64_t lda;   // fp32 arrays (passes 1, 3) or 16-bit arrays (passes 0, 6)
  const void* B; const void* Blo; int64_t ldb;
  float* C; int64_t ldc;
  int64_t M, N, K;
  int passes;            // 1 or 3 tf32 passes on fp32 operands; 0: A and B are 16-bit arrays (one kind::f16 pass);
                         // 6: 16-bit high and low parts, three kind::f16 passes
  int fp16;              // passes 0 / 6: the 16-bit type is fp16 (1) or bf16 (0)
  int mn_major;          // passes 0 / 6: A and B (and their low parts) are [K][M] and [K][N] arrays (lda, ldb: distance of two k)
  const float* row_scale; const float* col_scale;   // both or neither: C = acc * row_scale[m] * col_scale[n]
  int dependent;         // programmatic dependent launch behind the kernel that writes the scales (only they are waited for)
  int64_t k_segment;     // K extent accumulated in tensor memory before it is folded into C (0: all of K)
  int accumulate;        // C += (read-modify-write) instead of C =
  int symmetric_lower;   // only the lower triangle (tiles with n0 <= m0, elements with column <= row) is computed (M == N)
  const float* d1; const float* d2;  // optional dot operands (ld = ldc)
  double* part1; double* part2;      // partial sums, launch_tc_gemm says how many
  const int32_t* only_if;            // not null: nothing happens where it points to 0 (K-major operands)
};
armor_status launch_tc_gemm(armor_ctx* c, const TcGemm& g, int* n_part, cudaStream_t s);
bool tc_gemm_shape_ok(int64_t M, int64_t N, int64_t K);
// the 2:4 core on the sparse tensor cores (sparse_tcgen05.cu)
bool tc_sparse_ok(const armor_ctx* c);
size_t tc_sparse_values_bytes(const armor_ctx* c);
void launch_compress_24(armor_ctx* c, const float* S, const uint8_t* M, void* Sc, void* E, cudaStream_t s);
armor_status launch_tc_sparse(armor_ctx* c, const void* Sc, const void* E, const void* z1_bf16, void* z2, bool out_bf16,
                              int64_t n, cudaStream_t s);
bool tc_sparse3_ok(const armor_ctx* c);
armor_status launch_tc_sparse3(armor_ctx* c, const void* hi, const void* lo, const void* E, const float* row_scale, const void* zhi,
                               const void* zlo, const float* tok_scale, const int32_t* dense, float* z2, int64_t n, cudaStream_t s);
// the wrapper products of the bf16 forward (fwd_tcgen05.cu)
bool fwd_block_ok(const armor_ctx* c);
void launch_pack_blocks(armor_ctx* c, const float* P, const float* rowscale, const float* colscale, void* Q, int nb,
                        cudaStream_t s);
armor_status launch_fwd_block(armor_ctx* c, const void* X, const void* Q, void* out, int64_t rows, int64_t d,
                              cudaStream_t s);
// Few tokens (decoding): up to this many, and beyond while the layer is small (fwd_is_small), the three products of the bf16 forward
// run as latency-bound kernels whose contraction over d_in is split over the chip; the tiles of the persistent kernels fill it themselves.
static const int64_t ARMOR_SMALL_TOKENS = 128;
armor_status launch_fwd_small(armor_ctx* c, const void* X, int pieces, const void* Q, void* out, int64_t rows, int64_t d,
                              cudaStream_t s);
armor_status launch_tc_sparse_small(armor_ctx* c, const void* Sc, const void* E, const void* z1_bf16, float* Zp, int64_t n,
                                    int* pieces, cudaStream_t s);
