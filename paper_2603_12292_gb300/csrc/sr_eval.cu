// sr_eval.cu -- population evaluation: the postfix interpreter with fused
// MSE / 1 - r^2 reductions (sr_eval, sr_eval_batched) and the raw program
// outputs (sr_predict).
//
// Paper: all genomes of a generation go to the GPU together, each runs a
// batch of fitness cases and one aggregate per genome comes back (Sec.
// 2.1.2); genomes are RPN programs (Sec. 2.1.4); correlation fitness is r of
// Eq. 1, scored here as 1 - r^2 (Sec. 2.1.5).
//
// Design on the device
//   1. Decode pre-pass, a warp per program (sr_decode.cuh): validation, then the
//      expression tree is rescheduled Sethi-Ullman style -- at every binary node
//      the child that needs more stack is evaluated first (a reversed opcode
//      keeps a - b and a / b exact when the right child goes first).  The stack
//      depth of any program is then at most floor(log2(leaves)) + 1 (9 for 512
//      tokens), so floor(log2((Lmax + 1) / 2)) slots always suffice; most programs
//      need far fewer, so the main passes give each warp only what fits 4 or 5
//      CTAs per SM and the rare deeper programs run in a third pass.
//      A terminal evaluated second is fused into its binary operator
//      ("top = top op x_j"), and every operand is resolved here (constant
//      value, X row offset, stack-slot byte offset): the interpreter does no
//      per-token address or index arithmetic.  Values are bit-identical to
//      plain left-to-right evaluation (same operation on the same operands).
//   2. Evaluation, persistent grid: a work item is (case chunk, program),
//      handed out chunk-major by one atomic counter to single warps, so
//      warps running together share X columns in L1/L2 and uneven program
//      lengths balance out.  The warp copies the program's code into shared
//      memory and interprets it with lanes over cases, 8 cases per lane, 256
//      cases per step (sr_vm.cuh); the op stream is warp-uniform (no
//      divergence).  Top of stack in registers, the slots below in shared
//      memory [slot][half][lane] (conflict-free float4).
//   3. Per lane, FP32 Kahan-compensated sums over the item's cases, out of line
//      and in local memory, so that they cost the interpreter no registers
//      (4,096 x 100,000 at 5 CTAs per SM, one population: 5,824 -> 5,434 us); FP64 warp
//      reduction; one FP64 partial per (program, chunk); a finalize kernel
//      merges the chunks of each program (a group of lanes each, fixed order).
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <vector>

#include "sr_common.cuh"
#include "sr_decode.cuh"
#include "sr_interp.cuh"
#include "sr_vm.cuh"

namespace sr {
namespace {

constexpr int WARPS = 8;        // warps per CTA (measured best of 4, 8, 16 warps per CTA)
constexpr int PSTRIDE = 8;      // doubles per partial record
// Calls of at least this many cases and programs read the unary transforms
// of the variables from a table (sr_set_transforms' automatic mode); below
// that the table's launch and copy cost more than the few programs sharing
// each row save.
constexpr int XFORM_MIN_N = 16384, XFORM_MIN_P = 64;
// The compositions u(v(x_j)) join the table while it stays within this size
// (a call), and while a batch's tables with them stay within the second.
constexpr long long XFORM2_MAX_BYTES = 2ll << 30, XFORM2_BATCH_BYTES = 16ll << 30;
// A work item's slice of the table (its rows over the item's cases) is kept
// within this size when the library picks the cases per item, so that the
// items running at one time share a part of the table that stays in L2:
// on 262,144 programs x 10^6 cases, one item per program read the 520 MB
// table from DRAM, 3,961 GPop/s; 64k cases per item 4,236.
constexpr long long XFORM_SLICE_BYTES = 32ll << 20;
constexpr int TARGET_ITEMS_PER_WARP = 16;  // balances the launch tail; measured best of 8 to 28 at 4,096 x 100k
// Occupancy variants of the evaluation kernel: MINB CTAs of WARPS warps per
// SM.  Shared memory per CTA that leaves room for MINB of them (228 KB per
// SM, 1 KB of it reserved per CTA); the registers are bounded to match
// (5 CTAs: 48 registers).  Measured on 4,096 programs x 100,000 cases
// (Lmax 128): 5 CTAs with 4 stack slots 2,579 -> 2,649 GPop/s, Table 1
// operators 1,432 -> 1,592; at Lmax 256 the 48-register bound costs more than
// it gives (2,810 -> 2,625), so there it stays at 4 CTAs.
// (228 KB / MINB - 1 KB, rounded down to 512 bytes: 3 -> 76,800, 4 -> 57,344,
// 5 -> 45,568)
__host__ __device__ constexpr int smem_target(int minb) { return (233472 / minb - 1024) / 512 * 512; }

enum Mode { MODE_PREDICT = 0, MODE_MSE = 1, MODE_CORR = 2, MODE_BOTH = 3, MODE_R4 = 4, MODE_P2P = 5 };

struct EvalParams {
  const uint8_t *programs;
  const int32_t *lengths;
  const float *consts;
  int P, Lmax, K;
  const float *X;
  const float *y;
  const float *yc;         // centred target (1 - r^2 only), padded with zeros
  int nvars, N;
  long long ldx;
  int chunk, nchunks;
  long long total_items;
  double *partials;        // [P * nchunks][PSTRIDE]
  int32_t *flags;          // [P]
  uint2 *code;             // [P][Lmax] decoded instructions
  int32_t *ncode;          // [P]
  // [0] work counter, [1] work counter of the EXT pass, [2] the decoder's note that
  // it has programs, [3], [4] the same of the deep pass, [5], [6] the notes as the
  // later passes read them (hand_over)
  unsigned long long *queue;
  float *yhat;             // predict: [P][ldy]
  long long ldy;
  int warp_bytes;          // shared memory per warp
  int slots;               // stack slots per warp
  int words;               // words of code per warp, in the main passes
  int pass;                // Pass: the programs this launch takes
  int score_M;             // Beagle scores: the maximum score per case
  const int32_t *abort;    // sr_set_abort_flag (or NULL)
  unsigned *err;           // the context's latched error word
  int xform = 0;           // >= 1: X is the variable table of this depth (DecodeArgs::xform)
  const float *Xsrc = nullptr;  // rows to copy into X (the caller's X, not laid out for 256-bit loads), or NULL
  long long ldsrc = 0;
  double *ysum = nullptr;    // [nchunks][2] chunk sums and counts of y, where the target is centred, or NULL
  int finite_only = 0;       // 1: over the finite targets (Eq. 2)
  uint8_t *xneed = nullptr;  // the transforms some program reads
};

// shared memory of a warp: stack slots | decoded code, in words of 8 bytes (at most
// one per token, and the end marker)
constexpr int code_bytes(int words) { return (words * 8 + 15) / 16 * 16; }
constexpr int warp_smem_bytes(int slots, int words) { return slots * SLOT_BYTES + code_bytes(words); }
constexpr int ctas_per_sm(int slots, int words) { return 233472 / (WARPS * warp_smem_bytes(slots, words) + 1024); }

// Stack slots of the main evaluation passes: as many as fit smem_target(minb)
// beside `code` bytes of code, at most slots_for(Lmax) and at least
// min(slots_for(Lmax), 4).  Programs of up to 256 tokens, random or evolved,
// rarely need more than 4 (Sethi-Ullman order) while slots_for(256) = 7 would
// leave room for only 3 CTAs per SM; the few that need more than the main
// passes give (NCODE_DEEP) run in a third pass with slots_for(Lmax) slots.
constexpr int fit_slots(int Lmax, int minb, int code) {
  const int full = slots_for(Lmax), lo = full < 4 ? full : 4;
  const int s = (smem_target(minb) / WARPS - code) / SLOT_BYTES;
  return s < lo ? lo : (s > full ? full : s);
}
// The words of code of the main passes: Lmax + 1, or one less where that saves a
// CTA per SM (200 and 384 tokens).  Programs that keep an instruction for each of
// Lmax tokens (none that fuses an operand or folds constants) then run in the third
// pass too.  2,048 programs x 60,000 cases of <= 200 tokens, 4 CTAs -> 5: 2,524 -> 2,361 us;
// x 40,000 of <= 384, 3 -> 4: 3,614 -> 3,214.  Where it saves only a slot it gives
// nothing (256 tokens 3,203 -> 3,197) or costs L1 cache (72 tokens 687 -> 696).
constexpr int shallow_words(int Lmax, int minb) {
  const int s = fit_slots(Lmax, minb, code_bytes(Lmax)), t = fit_slots(Lmax, minb, code_bytes(Lmax + 1));
  const int cs = ctas_per_sm(s, Lmax), ct = ctas_per_sm(t, Lmax + 1);
  return (cs < minb ? cs : minb) > (ct < minb ? ct : minb) ? Lmax : Lmax + 1;
}
constexpr int shallow_slots(int Lmax, int minb) { return fit_slots(Lmax, minb, code_bytes(shallow_words(Lmax, minb))); }
// shared memory of a CTA in the main passes, and in the third (0: none)
constexpr int shallow_smem(int Lmax, int minb) {
  return WARPS * warp_smem_bytes(shallow_slots(Lmax, minb), shallow_words(Lmax, minb));
}
constexpr int deep_smem(int Lmax, int minb) {
  return slots_for(Lmax) > shallow_slots(Lmax, minb) || shallow_words(Lmax, minb) <= Lmax
             ? WARPS * warp_smem_bytes(slots_for(Lmax), Lmax + 1)
             : 0;
}


// 5 CTAs per SM where they fit with at least min(slots_for(Lmax), 4) slots
// (Lmax <= 200), else 4.
constexpr int minb_for(int Lmax) { return shallow_smem(Lmax, 5) <= smem_target(5) ? 5 : 4; }
static_assert(minb_for(200) == 5 && minb_for(201) == 4, "5 CTAs per SM up to 200 tokens");
static_assert(shallow_smem(384, 4) <= smem_target(4), "384 tokens: 4 CTAs per SM");
// The evaluation's CTAs per SM: the tuned choice where it fits, else the
// automatic one
inline int eval_minb(int Lmax, int tuned) {
  if (tuned == 5) return minb_for(Lmax);
  if (tuned == 4) return 4;
  return minb_for(Lmax);
}

// The CTAs per SM that the cases per work item are chosen by: those of a warp
// with its stack slots and 8 bytes of code per token (no end marker).  The
// FP32 sums of a program follow its case chunks, so this rule is part of the
// results and stays as it is whatever the kernels take.
inline int chunk_ctas(int Lmax, int minb) {
  const int code = ((Lmax * 8 + 15) / 16) * 16;
  const int smem = WARPS * (fit_slots(Lmax, minb, code) * SLOT_BYTES + code);
  const int fit = 233472 / (smem + 1024);
  return fit < minb ? fit : minb;
}
inline int chunk_minb(int Lmax, int tuned) {  // eval_minb by the same rule
  const int code = ((Lmax * 8 + 15) / 16) * 16;
  const bool five = WARPS * (fit_slots(Lmax, 5, code) * SLOT_BYTES + code) <= smem_target(5);
  return tuned == 4 || !five ? 4 : 5;
}

// ---------------------------------------------------------------- operators
__device__ __forceinline__ float4 ldx4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// ---------------------------------------------------------------- target prep (1 - r^2)
// Two passes over y: the sum of every chunk, then the centred target with its
// sums.  They run as blocks of the decode launch and of the table's launch: a
// block per chunk leaves most of the GPU idle (11 + 18 us for 23 chunks of 4,352
// cases, 22 + 32 for 10 of 13,312), and both are done before those launches are.
constexpr int PREP_THREADS = 512;

__device__ double block_sum(double v, double *red) {
  v = warp_sum(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  __syncthreads();
  return s;  // valid in thread 0
}

// FP64 sum and count of one chunk of y: every value, or (finite_only) the
// finite ones.  ysum [nchunks][2].
__device__ void ysum_chunk(const float *y, int N, int chunk, int c, bool finite_only,
                           double *ysum, double *red) {
  const int beg = c * chunk, end = min(N, beg + chunk);
  double a = 0.0, n = 0.0;
  for (int i = beg + threadIdx.x; i < end; i += blockDim.x) {
    const float v = y[i];
    if (!finite_only || isfinite(v)) {
      a += (double)v;
      n += 1.0;
    }
  }
  a = block_sum(a, red);
  n = block_sum(n, red);
  if (threadIdx.x == 0) {
    ysum[2 * c] = a;
    ysum[2 * c + 1] = n;
  }
}

// ybar = (sum of the chunk sums) / (their count), chunks in order; then
// yc = fl32(y - ybar) on one chunk (NaN at invalid targets when
// nan_invalid) with the chunk's FP64 sum and sum of squares of yc
__device__ void ycenter_chunk(const float *y, int N, int chunk, int nchunks, int c,
                              const double *ysum, bool nan_invalid, float *yc, double *ychunk,
                              double *red) {
  __shared__ double ybar_s;
  if (threadIdx.x == 0) {
    double t = 0.0, n = 0.0;
    for (int k = 0; k < nchunks; ++k) {
      t += ysum[2 * k];
      n += ysum[2 * k + 1];
    }
    ybar_s = n > 0.0 ? t / n : 0.0;
  }
  __syncthreads();
  const double ybar = ybar_s;
  const int beg = c * chunk, end = min(N, beg + chunk);
  double a = 0.0, b = 0.0;
  for (int i = beg + threadIdx.x; i < end; i += blockDim.x) {
    const float yi = y[i];
    if (nan_invalid && !isfinite(yi)) {
      yc[i] = __int_as_float(0x7fc00000);
      continue;
    }
    const float v = (float)((double)yi - ybar);
    yc[i] = v;
    a += (double)v;
    b += (double)v * (double)v;
  }
  if (c == nchunks - 1) {
    const int padded = (N + STEP - 1) / STEP * STEP;
    for (int i = N + threadIdx.x; i < padded; i += blockDim.x) yc[i] = 0.0f;
  }
  a = block_sum(a, red);
  b = block_sum(b, red);
  if (threadIdx.x == 0) {
    ychunk[2 * c] = a;
    ychunk[2 * c + 1] = b;
  }
}


// ---------------------------------------------------------------- decode pre-pass
// slots, words: those of the main passes; programs that need more get NCODE_DEEP
__device__ __forceinline__ DecodeArgs decode_args(const EvalParams &p, int slots, int words) {
  DecodeArgs a;
  a.programs = p.programs;
  a.lengths = p.lengths;
  a.consts = p.consts;
  a.Lmax = p.Lmax;
  a.K = p.K;
  a.nvars = p.nvars;
  a.ldx = p.ldx;
  a.slot_bytes = SLOT_BYTES;
  a.code = p.code;
  a.ncode = p.ncode;
  a.flags = p.flags;
  a.max_slots = slots_for(p.Lmax);
  a.cap_slots = slots;
  a.cap_words = words;
  a.ext_note = p.queue + 2;
  a.deep_note = p.queue + 4;
  a.xform = p.xform;
  a.xneed = p.xneed;
  return a;
}

// Copies X's rows (nvars x N, row stride ldsrc) into rows of ldx floats that
// start on 32-byte boundaries, so that the interpreter reads a lane's 8 cases
// with one load.  Blocks of STAGE_CASES cases of one row.
constexpr int STAGE_CASES = 2048;
__host__ __device__ inline int stage_blocks(int nvars, int N) { return nvars * ((N + STAGE_CASES - 1) / STAGE_CASES); }
__device__ void stage_rows(const EvalParams &p, int block) {
  const int per_row = (p.N + STAGE_CASES - 1) / STAGE_CASES;
  const int j = block / per_row, end = min(p.N, (block % per_row + 1) * STAGE_CASES);
  const float *src = p.Xsrc + (size_t)j * p.ldsrc;
  float *dst = const_cast<float *>(p.X) + (size_t)j * p.ldx;
  for (int i = (block % per_row) * STAGE_CASES + threadIdx.x * 4; i < end; i += blockDim.x * 4)
    *reinterpret_cast<float4 *>(dst + i) = ldx4(src + i);  // i + 3 < both strides: multiples of 4, >= N
}

// The first blocks sum the chunks of y where the target is centred, the next
// decode (one warp per program, scratch in shared memory), the last copy X where
// it is not laid out for 256-bit loads.
__global__ void __launch_bounds__(DECODE_WARPS * 32) decode_kernel(EvalParams p) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[DECODE_WARPS];
  launch_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) p.queue[0] = p.queue[1] = p.queue[3] = 0;
  const int yblocks = p.ysum ? p.nchunks : 0, dblocks = (p.P + DECODE_WARPS - 1) / DECODE_WARPS;
  const int block = (int)blockIdx.x - yblocks;
  if (block < 0) {
    ysum_chunk(p.y, p.N, p.chunk, blockIdx.x, p.finite_only != 0, p.ysum, red);
    return;
  }
  if (block >= dblocks) {
    stage_rows(p, block - dblocks);
    return;
  }
  const int warp = threadIdx.x >> 5, prog = block * DECODE_WARPS + warp;
  if (prog < p.P)
    decode_eval_warp(decode_args(p, p.slots, p.words), prog, dsm + (size_t)warp * decode_scratch_bytes(p.Lmax));
}

// The variable table of an evaluation with transforms (DecodeArgs::xform):
// row j < nvars is x_j, row xform_row(nvars, u, j) is u(x_j) and row
// xform_row2(nvars, u, v, j) is u(v(x_j)), for the rows some program reads
// (xneed, marked by the decoder), by the interpreter's own FP32 functions
// (fold_op's), so a program reads the bits its own per-case evaluation would
// give.  Blocks: (XF_THREADS * 4 cases, variable and part): part 0 the variable
// and the operators beyond the base ones, part 1 + v the base operator v and its
// compositions, which read v(x_j) from registers.  What bounds it: issue slots.
// A block per row, each value through a call of fold_op, computed v(x_j) seven
// times: 118 us for 490 rows of 100,003 cases, now 40.
constexpr int XF_THREADS = 256, XF_PARTS = 1 + XFORM_BASE;
static __device__ __noinline__ float4 unary4(int tok, float4 x) {
#define SR_EACH(f) make_float4(f(x.x), f(x.y), f(x.z), f(x.w))
  switch (tok) {
    case TOK_SIN: return SR_EACH(f_sin);
    case TOK_COS: return SR_EACH(f_cos);
    case TOK_EXP: return SR_EACH(op_exp);
    case TOK_LOG: return SR_EACH(op_log);
    case TOK_SQRT: return SR_EACH(f_sqrt);
    case TOK_SQ: return make_float4(__fmul_rn(x.x, x.x), __fmul_rn(x.y, x.y), __fmul_rn(x.z, x.z), __fmul_rn(x.w, x.w));
    default:
      return make_float4(fold_op(tok, x.x, 0.f), fold_op(tok, x.y, 0.f), fold_op(tok, x.z, 0.f), fold_op(tok, x.w, 0.f));
  }
#undef SR_EACH
}
__device__ void xform_block(const float *X, long long ldx, int nvars, int N, int ldxt, int depth,
                            const uint8_t *xneed, float *xt, int block, int j, int part) {
  const int c = (block * XF_THREADS + threadIdx.x) * 4;
  if (c >= N) return;  // c + 3 < ldx and < ldxt: both are multiples of 4 and >= N
  const float4 x = ldx4(X + (size_t)j * ldx + c);
  auto put = [&](int row, float4 v) { *reinterpret_cast<float4 *>(xt + (size_t)row * ldxt + c) = v; };
  auto needed = [&](int row) { return xneed[row - nvars] != 0; };
  if (part == 0) {
    put(j, x);
    for (int u = TOK_SQ + 1; u <= TOK_TANH; ++u)
      if (needed(xform_row(nvars, u, j))) put(xform_row(nvars, u, j), unary4(u, x));
    return;
  }
  const int v = TOK_SIN + part - 1;
  bool any = needed(xform_row(nvars, v, j));
  if (depth > 1)
    for (int u = TOK_SIN; u <= TOK_SQ; ++u) any = any || needed(xform_row2(nvars, u, v, j));
  if (!any) return;
  const float4 y = unary4(v, x);
  if (needed(xform_row(nvars, v, j))) put(xform_row(nvars, v, j), y);
  if (depth > 1)
    for (int u = TOK_SIN; u <= TOK_SQ; ++u)
      if (needed(xform_row2(nvars, u, v, j))) put(xform_row2(nvars, u, v, j), unary4(u, y));
}
struct CenterParams {
  const float *y;
  int N, chunk, nchunks, nan_invalid;
  const double *ysum;
  float *yc;
  double *ychunk;
};
__global__ void __launch_bounds__(PREP_THREADS) ycenter_kernel(CenterParams y) {
  __shared__ double red[PREP_THREADS / 32];
  launch_wait();
  ycenter_chunk(y.y, y.N, y.chunk, y.nchunks, blockIdx.x, y.ysum, y.nan_invalid != 0, y.yc, y.ychunk, red);
}
// The first yblocks blocks centre the target, one chunk each.
__global__ void __launch_bounds__(XF_THREADS)
    xform_kernel(const float *X, long long ldx, int nvars, int N, int ldxt, int depth, const uint8_t *xneed, float *xt,
                 int yblocks, CenterParams y) {
  __shared__ double red[XF_THREADS / 32];
  launch_wait();
  const int block = (int)blockIdx.x - yblocks, per_part = (N + XF_THREADS * 4 - 1) / (XF_THREADS * 4);
  if (block < 0) {
    ycenter_chunk(y.y, y.N, y.chunk, y.nchunks, blockIdx.x, y.ysum, y.nan_invalid != 0, y.yc, y.ychunk, red);
    return;
  }
  const int part = block / per_part;
  xform_block(X, ldx, nvars, N, ldxt, depth, xneed, xt, block % per_part, part / XF_PARTS, part % XF_PARTS);
}
static_assert(DECODE_WARPS * 8192 <= 48 * 1024, "the decode launch needs no shared memory opt-in");
inline int xform_blocks(int nvars, int N) { return nvars * XF_PARTS * ((N + XF_THREADS * 4 - 1) / (XF_THREADS * 4)); }

// ---------------------------------------------------------------- reductions
struct Kahan {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float yv = x - c;
    const float t = s + yv;
    c = (t - s) - yv;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

__device__ __forceinline__ float sel(bool ok, float v) { return ok ? v : 0.0f; }

__device__ __forceinline__ float4 load_y4(const float *y, int c0, int N) {
  if (c0 + 3 < N) return ldx4(y + c0);
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c0 < N) r.x = y[c0];
  if (c0 + 1 < N) r.y = y[c0 + 1];
  if (c0 + 2 < N) r.z = y[c0 + 2];
  return r;
}

// Eq. 3 on one case, FP32, every operation rounded on its own (no
// contraction), the result rounded half to even.
__device__ __forceinline__ int p2p_case(float yh, float y, int M, float Mf, float pen) {
  const bool vh = isfinite(yh), vy = isfinite(y);
  if (!(vh && vy)) return (vh || vy) ? -M : M;
  const float a = fabsf(yh), b = fabsf(y);
  const float mx = fmaxf(a, b), mn = fminf(a, b);
  if (mx == 0.0f) return M;
  float v = __fmul_rn(Mf, __fdiv_rn(mn, mx));
  if ((yh < 0.0f && y > 0.0f) || (yh > 0.0f && y < 0.0f)) v = __fsub_rn(v, pen);
  return (int)rintf(v);
}

// Eq. 2 sums over one lane's 8 cases (nvalid of them inside the chunk):
// pairs with both values finite give the moments of the shifted output d
// and the centred target e; one invalid value counts in n1, both in n2.
// Four values at a time, so that these sums and the interpreter's operators stay
// in the instruction cache together (the only copy is inside `accumulate`): 4,096 x
// 100,000 with the base operators 6,120 -> 5,605 us, a population under way 5,357 ->
// 4,970, all operators 2,048 x 50,001 2,115 -> 2,064 (the eight at once and inline:
// 5,940, 5,207, 2,066).
struct R4Part { float s1, s2, s3, s4, s5; int n1, n2; };
__device__ __forceinline__ R4Part r4_part(V8 T, float4 ya, float4 yb, int nvalid, float shift) {
  float tv[CPL];
  unpack8(T, tv);
  float t0 = tv[0], t1 = tv[1], t2 = tv[2], t3 = tv[3], y0 = ya.x, y1 = ya.y, y2 = ya.z, y3 = ya.w;
  R4Part r{0.f, 0.f, 0.f, 0.f, 0.f, 0, 0};
#pragma unroll 1
  for (int h = 0; h < CPL; h += 4) {
    const float t[4] = {t0, t1, t2, t3}, y[4] = {y0, y1, y2, y3};
    float d[4], e[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool ok = h + i < nvalid;
      const bool vh = isfinite(t[i]), vy = isfinite(y[i]);
      const bool pair = ok && vh && vy;
      r.n1 += (ok && vh != vy) ? 1 : 0;
      r.n2 += (ok && !vh && !vy) ? 1 : 0;
      d[i] = pair ? t[i] - shift : 0.0f;
      e[i] = pair ? y[i] : 0.0f;
    }
    r.s1 += (d[0] + d[1]) + (d[2] + d[3]);
    r.s2 += (d[0] * d[0] + d[1] * d[1]) + (d[2] * d[2] + d[3] * d[3]);
    r.s3 += (d[0] * e[0] + d[1] * e[1]) + (d[2] * e[2] + d[3] * e[3]);
    r.s4 += (e[0] + e[1]) + (e[2] + e[3]);
    r.s5 += (e[0] * e[0] + e[1] * e[1]) + (e[2] * e[2] + e[3] * e[3]);
    t0 = tv[4]; t1 = tv[5]; t2 = tv[6]; t3 = tv[7];
    y0 = yb.x; y1 = yb.y; y2 = yb.z; y3 = yb.w;
  }
  return r;
}

// ---------------------------------------------------------------- one work item
struct WarpSmem {
  char *stk;        // shared stack slots of this warp, [DSM][2][32] float4
  uint2 *code;      // this warp's copy of the program's code
};

__device__ __forceinline__ WarpSmem warp_smem(unsigned char *smem, int warp, int warp_bytes, int slots) {
  unsigned char *wbase = smem + (size_t)warp * warp_bytes;
  WarpSmem w;
  w.stk = reinterpret_cast<char *>(wbase);
  w.code = reinterpret_cast<uint2 *>(wbase + slots * SLOT_BYTES);
  return w;
}

// A lane's running sums over an item's cases.
struct Acc {
  Kahan se, s1, s2, s3, s4, s5;
  float shift;
  int c1, c2;
  long long score;
};

// Adds one step's 8 outputs per lane (cases c0 .. c0 + 7, those below cend
// valid; cl / cl4 the readable positions of the two halves of the target) to
// the sums of the mode.  MODE_BOTH takes those selected by `want` (bit 0:
// squared error, bit 1: correlation moments).  y: the target (MSE, Eq. 3) with
// N values; yc: the centred target (1 - r^2, Eq. 2).
template <int MODE>
__device__ __noinline__ void accumulate(Acc *acc, V8 T, int c0, int cl, int cl4, int cend, int first,
                                  const float *y, const float *yc, int N, int want, int M) {
  const bool do_mse = MODE == MODE_MSE || (MODE == MODE_BOTH && (want & 1));
  const bool do_corr = MODE == MODE_CORR || (MODE == MODE_BOTH && (want & 2));
  float tv[CPL];
  unpack8(T, tv);
  bool ok[CPL];
#pragma unroll
  for (int i = 0; i < CPL; ++i) ok[i] = c0 + i < cend;
  if (do_mse) {
    const float4 ya = load_y4(y, cl, N), yb = load_y4(y, cl4, N);
    const float yv[CPL] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
    float e[CPL];
#pragma unroll
    for (int i = 0; i < CPL; ++i) e[i] = sel(ok[i], tv[i] - yv[i]);
    acc->se.add(((e[0] * e[0] + e[1] * e[1]) + (e[2] * e[2] + e[3] * e[3])) +
                ((e[4] * e[4] + e[5] * e[5]) + (e[6] * e[6] + e[7] * e[7])));
  }
  if (do_corr) {
    if (first) acc->shift = __shfl_sync(FULL, tv[0], 0);
    const float shift = acc->shift;
    const float4 ya = ldx4(yc + cl), yb = ldx4(yc + cl4);
    const float yv[CPL] = {ya.x, ya.y, ya.z, ya.w, yb.x, yb.y, yb.z, yb.w};
    float d[CPL];
#pragma unroll
    for (int i = 0; i < CPL; ++i) d[i] = sel(ok[i], tv[i] - shift);
    acc->s1.add(((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])));
    acc->s2.add(((d[0] * d[0] + d[1] * d[1]) + (d[2] * d[2] + d[3] * d[3])) +
                ((d[4] * d[4] + d[5] * d[5]) + (d[6] * d[6] + d[7] * d[7])));
    acc->s3.add(((d[0] * yv[0] + d[1] * yv[1]) + (d[2] * yv[2] + d[3] * yv[3])) +
                ((d[4] * yv[4] + d[5] * yv[5]) + (d[6] * yv[6] + d[7] * yv[7])));
  }
  if (MODE == MODE_R4) {
    // pairs: both finite -> moments; one invalid -> c1; both -> c2.  yc
    // holds y - ybar for finite y and NaN for invalid targets.
    if (first) {
      const unsigned fin = __ballot_sync(FULL, isfinite(tv[0]));
      acc->shift = fin ? __shfl_sync(FULL, tv[0], __ffs(fin) - 1) : 0.0f;
    }
    const float4 ya = ldx4(yc + cl), yb = ldx4(yc + cl4);
    const R4Part q = r4_part(T, ya, yb, cend - c0, acc->shift);
    acc->s1.add(q.s1);
    acc->s2.add(q.s2);
    acc->s3.add(q.s3);
    acc->s4.add(q.s4);
    acc->s5.add(q.s5);
    acc->c1 += q.n1;
    acc->c2 += q.n2;
  }
  if (MODE == MODE_P2P) {
    const float Mf = (float)M, pen = __fdiv_rn(Mf, 11.0f);
    const float4 ya = load_y4(y, cl, N), yb = load_y4(y, cl4, N);
    // one copy of the per-case body: the values rotate through it
    float t0 = tv[0], t1 = tv[1], t2 = tv[2], t3 = tv[3], t4 = tv[4], t5 = tv[5], t6 = tv[6], t7 = tv[7];
    float y0 = ya.x, y1 = ya.y, y2 = ya.z, y3 = ya.w, y4 = yb.x, y5 = yb.y, y6 = yb.z, y7 = yb.w;
    int c1 = 0, c2 = 0;
    long long score = 0;
#pragma unroll 1
    for (int i = 0; i < CPL; ++i) {
      if (c0 + i < cend) {
        const bool vh = isfinite(t0), vy = isfinite(y0);
        c1 += vh != vy ? 1 : 0;
        c2 += (!vh && !vy) ? 1 : 0;
        score += p2p_case(t0, y0, M, Mf, pen);
      }
      t0 = t1; t1 = t2; t2 = t3; t3 = t4; t4 = t5; t5 = t6; t6 = t7;
      y0 = y1; y1 = y2; y2 = y3; y3 = y4; y4 = y5; y5 = y6; y6 = y7;
    }
    acc->c1 += c1;
    acc->c2 += c2;
    acc->score += score;
  }
}

// Evaluates program `prog` of problem p on case chunk `c` with the calling
// warp.  MODE_BOTH accumulates the sums selected by `want` (bit 0: squared
// error, bit 1: correlation moments); the other modes ignore `want`.
template <int MODE, bool EXT, bool WIDE, bool LEAN>
__device__ __forceinline__ void eval_item(const EvalParams &p, int c, int prog, const WarpSmem &w,
                                          int lane, int want) {
  const bool do_mse = MODE == MODE_MSE || (MODE == MODE_BOTH && (want & 1));
  const bool do_corr = MODE == MODE_CORR || (MODE == MODE_BOTH && (want & 2));
  const int cbeg = c * p.chunk;
  const int cend = min(p.N, cbeg + p.chunk);
  if (p.flags[prog]) {
    if (MODE == MODE_PREDICT) {
      float *row = p.yhat + (size_t)prog * p.ldy;
      for (int i = cbeg + lane; i < cend; i += 32) row[i] = __int_as_float(0x7fc00000);
    }
    return;
  }
  const int n = ncode_count(p.ncode[prog]);
  __syncwarp();  // the previous item is done reading the code
  const uint2 *src = p.code + (size_t)prog * p.Lmax;
  for (int i = lane; i < n; i += 32) w.code[i] = src[i];
  if (lane == 0) w.code[n] = make_uint2(OP_END, 0u);
  __syncwarp();

  char *stk = w.stk + lane * 16;
  const int last_group = (cend - 1) & ~(CPL - 1);

  Acc acc;
  acc.se = acc.s1 = acc.s2 = acc.s3 = acc.s4 = acc.s5 = Kahan();
  acc.shift = 0.f;
  acc.c1 = acc.c2 = 0;
  acc.score = 0;
  for (int base = cbeg; base < cend; base += STEP) {
    const int c0 = base + CPL * lane;
    const int cl = c0 < cend ? c0 : last_group;           // first 4 cases, always readable
    const int cl4 = cl + 4 < cend ? cl + 4 : cl;          // second 4, or a re-read when none valid
    const V8 T = interpret<EXT, WIDE, LEAN>(w.code, stk, p.X + cl, p.X + cl4);
    if (MODE == MODE_PREDICT) {
      float tv[CPL];
      unpack8(T, tv);
      float *row = p.yhat + (size_t)prog * p.ldy;
#pragma unroll
      for (int i = 0; i < CPL; ++i)
        if (c0 + i < cend) row[c0 + i] = tv[i];
    } else {
      accumulate<MODE>(&acc, T, c0, cl, cl4, cend, base == cbeg, p.y, p.yc, p.N, want, p.score_M);
    }
  }
  if (MODE != MODE_PREDICT) {
    double *rec = p.partials + ((size_t)prog * p.nchunks + c) * PSTRIDE;
    if (do_mse) {
      const double v = warp_sum(acc.se.value());
      if (lane == 0) rec[0] = v;
    }
    if (do_corr) {
      const double a = warp_sum(acc.s1.value());
      const double b = warp_sum(acc.s2.value());
      const double d = warp_sum(acc.s3.value());
      if (lane == 0) {
        rec[1] = (double)acc.shift;
        rec[2] = a;
        rec[3] = b;
        rec[4] = d;
      }
    }
    if (MODE == MODE_R4) {
      // [shift, sum d, sum d^2, sum d e, sum e, sum e^2, c1, c2]
      const double v1 = warp_sum(acc.s1.value()), v2 = warp_sum(acc.s2.value()), v3 = warp_sum(acc.s3.value());
      const double v4 = warp_sum(acc.s4.value()), v5 = warp_sum(acc.s5.value());
      const double n1 = warp_sum((double)acc.c1), n2 = warp_sum((double)acc.c2);
      if (lane == 0) {
        rec[0] = (double)acc.shift;
        rec[1] = v1;
        rec[2] = v2;
        rec[3] = v3;
        rec[4] = v4;
        rec[5] = v5;
        rec[6] = n1;
        rec[7] = n2;
      }
    }
    if (MODE == MODE_P2P) {
      // [sum of the integer scores (exact), c1, c2]
      const double v = warp_sum((double)acc.score);
      const double n1 = warp_sum((double)acc.c1), n2 = warp_sum((double)acc.c2);
      if (lane == 0) {
        rec[0] = v;
        rec[6] = n1;
        rec[7] = n2;
      }
    }
  }
}

// ---------------------------------------------------------------- single problem
// Up to three passes over the work items: the programs of the base operators
// (and the invalid ones), those that use 1/x, tan, asin, acos, atan or tanh
// (which returns at once when there are none), and those that need
// more than the main passes' shallow_slots(Lmax, MINB) stack slots or shallow_words
// (NCODE_DEEP; made only where a program can).  Keeping the extended operators out
// of the first kernel keeps its loop inside the instruction cache.  Where the
// rows of X could not be laid out for 256-bit loads, the same passes read them in
// halves.  (One pass of the EXT kernel for base and extended programs then took,
// 1,500 programs of <= 64 tokens x 500,004 cases, 7,535 us instead of 6,105; 1,024 of
// <= 128 x 400,004, both kinds, 7,810 instead of 6,260.)
enum Pass { PASS_BASE = 0, PASS_EXT = 1, PASS_DEEP = 2 };

__device__ __forceinline__ bool takes(int pass, int ncode) {
  if (pass == PASS_DEEP) return ncode_deep(ncode);
  if (ncode_deep(ncode)) return false;
  return ncode_ext(ncode) == (pass == PASS_EXT);
}
// The first pass hands the decoder's notes over to the passes
// after it and clears them for the next call.  A replay of a captured call then
// makes a pass only when its own programs need it (a note that stayed had every
// replay after it walk the items of an empty pass).
__device__ __forceinline__ void hand_over(unsigned long long *queue) {
  queue[5] = queue[2];
  queue[6] = queue[4];
  queue[2] = queue[4] = 0;
}
// the pass's work counter; NULL when it has no programs
__device__ __forceinline__ unsigned long long *pass_queue(unsigned long long *queue, int pass) {
  if (pass == PASS_EXT) return queue[5] ? queue + 1 : nullptr;
  if (pass == PASS_DEEP) return queue[6] ? queue + 3 : nullptr;
  if (blockIdx.x == 0 && threadIdx.x == 0) hand_over(queue);
  return queue;
}

template <int MODE, bool EXT, bool WIDE, int MINB>
__global__ void __launch_bounds__(WARPS * 32, MINB) eval_kernel(EvalParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_wait();
  const int pass = EXT ? p.pass : PASS_BASE;
  unsigned long long *q = pass_queue(p.queue, pass);
  if (!q) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WarpSmem w = warp_smem(smem, warp, p.warp_bytes, p.slots);
  for (;;) {
    const long long item = next_item(q, p.total_items, p.abort, p.err, lane);
    if (item >= p.total_items) break;
    const int c = (int)(item / (unsigned long long)p.P);
    const int prog = (int)(item % (unsigned long long)p.P);
    if (!takes(pass, p.ncode[prog])) continue;
    eval_item<MODE, EXT, WIDE, MODE == MODE_P2P>(p, c, prog, w, lane, 3);
  }
}

// ---------------------------------------------------------------- many problems, one launch
constexpr int MAX_BATCH = 64;

struct BatchProblem {
  const uint8_t *programs;
  const int32_t *lengths;
  const float *consts;
  const float *X;
  const float *y;
  float *yc;           // centred target (1 - r^2), padded
  double *partials;    // [P * nchunks][PSTRIDE]
  int32_t *flags;      // [P]
  uint2 *code;         // [P][Lmax]
  int32_t *ncode;      // [P]
  double *fitness;     // [P] or [2][P]
  double *ychunk;      // [nchunks][2]
  double *ysum;        // [nchunks][2]: FP64 sum and count of y per chunk
  long long ldx;
  long long item_begin;  // first work item of this problem in the launch
  int prog_begin;        // first program of this problem in the decode launch
  int P, Lmax, K, nvars, N, chunk, nchunks;
  int mode;              // MODE_MSE, MODE_CORR or MODE_BOTH
  int corr_chunk_begin;  // first block of this problem in the batched centring launch (-1: none)
  int xform;             // >= 1: X / ldx are the problem's variable table of this depth (EvalParams::xform)
  uint8_t *xneed;
  const float *Xsrc;     // as EvalParams::Xsrc
  long long ldsrc;
  int stage_begin;       // first staging block of this problem in the decode launch
};

struct BatchParams {
  BatchProblem prob[MAX_BATCH];
  int nprob;
  int corr_list[MAX_BATCH];  // problems that need the centred target, in order
  int ncorr;
  int total_progs;
  long long total_items;
  unsigned long long *queue;  // as EvalParams::queue
  int warp_bytes;
  int slots, words;           // as EvalParams
  int maxL;                   // the largest Lmax of the batch
  int pass;                   // as EvalParams::pass
  // blocks of the decode launch: those that sum chunks of y, that decode, that copy X
  int ysum_blocks, decode_blocks, stage_blocks;
  const int32_t *abort;       // as EvalParams::abort
  unsigned *err;
};

static_assert(sizeof(BatchParams) <= 32764, "the problem table must fit the kernel parameters");

__device__ __forceinline__ EvalParams view(const BatchProblem &q) {
  EvalParams p;
  p.programs = q.programs;
  p.lengths = q.lengths;
  p.consts = q.consts;
  p.P = q.P;
  p.Lmax = q.Lmax;
  p.K = q.K;
  p.X = q.X;
  p.y = q.y;
  p.yc = q.yc;
  p.nvars = q.nvars;
  p.N = q.N;
  p.ldx = q.ldx;
  p.chunk = q.chunk;
  p.nchunks = q.nchunks;
  p.partials = q.partials;
  p.flags = q.flags;
  p.code = q.code;
  p.ncode = q.ncode;
  p.xform = q.xform;
  p.xneed = q.xneed;
  p.Xsrc = q.Xsrc;
  p.ldsrc = q.ldsrc;
  return p;
}

// the problem whose target chunk a block of the target's launches takes
__device__ __forceinline__ int corr_problem_of_block(const BatchParams &b) {
  int r = 0;
  while (r + 1 < b.ncorr && b.prob[b.corr_list[r + 1]].corr_chunk_begin <= (int)blockIdx.x) ++r;
  return b.corr_list[r];
}

// a warp per program of every problem in the batch (shared regions sized
// for the batch's largest Lmax, b.maxL)
__global__ void __launch_bounds__(DECODE_WARPS * 32) decode_batched_kernel(const __grid_constant__ BatchParams b) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[DECODE_WARPS];
  launch_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) b.queue[0] = b.queue[1] = b.queue[3] = 0;
  const int block = (int)blockIdx.x - b.ysum_blocks;
  if (block < 0) {
    const BatchProblem &q = b.prob[corr_problem_of_block(b)];
    ysum_chunk(q.y, q.N, q.chunk, (int)blockIdx.x - q.corr_chunk_begin, false, q.ysum, red);
    return;
  }
  if (block >= b.decode_blocks) {
    const int r = block - b.decode_blocks;
    int i = 0;
    while (i + 1 < b.nprob && b.prob[i + 1].stage_begin <= r) ++i;
    const EvalParams p = view(b.prob[i]);
    if (p.Xsrc) stage_rows(p, r - b.prob[i].stage_begin);
    return;
  }
  const int warp = threadIdx.x >> 5;
  const int g = block * DECODE_WARPS + warp;
  if (g >= b.total_progs) return;
  int lo = 0, hi = b.nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (b.prob[mid].prog_begin <= g) lo = mid;
    else hi = mid - 1;
  }
  EvalParams p = view(b.prob[lo]);
  p.queue = b.queue;
  decode_eval_warp(decode_args(p, b.slots, b.words), g - b.prob[lo].prog_begin,
                   dsm + (size_t)warp * decode_scratch_bytes(b.maxL));
}

// Work items of every problem come from one atomic counter: problem q owns
// items [item_begin_q, item_begin_q + P_q * nchunks_q), chunk-major inside.
// Passes as for eval_kernel.
// At most 64 registers, so that 4 CTAs fit an SM (75 unbounded, 3 CTAs):
// 2,608 -> 2,949 GPop/s on the 64-problem batch.
// LEAN where items are short: then the code around the interpreter (the item,
// its problem, the sums) runs as often as its operators and the instruction
// cache has to hold both.  us with and without, 64 problems of 512 or 1,024
// programs of <= 64 tokens: 3 steps an item 439 / 562, 6 steps 2,039 / 2,211, 20
// steps 6,059 / 5,831; 16 problems of <= 128 tokens, 60,000 cases 25,794 / 25,015.
constexpr int LEAN_MAX_STEPS = 10;
template <bool EXT, bool WIDE, int MINB, bool LEAN>
__global__ void __launch_bounds__(WARPS * 32, MINB) eval_batched_kernel(const __grid_constant__ BatchParams b) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_wait();
  const int pass = EXT ? b.pass : PASS_BASE;
  unsigned long long *qc = pass_queue(b.queue, pass);
  if (!qc) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WarpSmem w = warp_smem(smem, warp, b.warp_bytes, b.slots);
  for (;;) {
    const long long item = next_item(qc, b.total_items, b.abort, b.err, lane);
    if (item >= b.total_items) break;
    int lo = 0, hi = b.nprob - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b.prob[mid].item_begin <= (long long)item) lo = mid;
      else hi = mid - 1;
    }
    const BatchProblem &q = b.prob[lo];
    const EvalParams p = view(q);
    const long long local = (long long)item - q.item_begin;
    const int c = (int)(local / q.P);
    const int prog = (int)(local % q.P);
    if (!takes(pass, q.ncode[prog])) continue;
    const int want = q.mode == MODE_MSE ? 1 : (q.mode == MODE_CORR ? 2 : 3);
    eval_item<MODE_BOTH, EXT, WIDE, LEAN>(p, c, prog, w, lane, want);
  }
}

// ---------------------------------------------------------------- finalize
// The merges below run with a group of lanes per program, a power of two by the
// number of chunks (about four chunks a lane): lane l of the group takes chunks
// l, l + lanes, ...; every sum over chunks is a per-lane sum followed by a fixed
// xor-butterfly over the group, so the result is deterministic and the same on
// every lane.  What bounds it: the FP64 pipe (two lanes an SM), which a warp per
// program kept busy with idle lanes.  Before -> now (us): 64 small problems,
// 22,000 programs of 1 to 40 chunks, 106 -> 21; 8,192 programs of 10 chunks 54 -> 14;
// 4,096 of 23 33 -> 16; 1,500 of 56 27 -> 23.
__host__ __device__ inline int merge_lanes(int nchunks) {
  int g = 1;
  while (g < 32 && g * 4 < nchunks) g *= 2;
  return g;
}
struct Group {
  int lane, lanes;
  unsigned mask;
  __device__ __forceinline__ double sum(double v) const {
    for (int o = lanes >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
  }
};
__device__ __forceinline__ Group group_of(int lanes) {
  const int l = threadIdx.x & 31;
  return Group{l & (lanes - 1), lanes, (lanes == 32 ? FULL : (1u << lanes) - 1u) << (l & ~(lanes - 1))};
}

// 1 - r^2 of one program from its chunk records.
// chunk c: n_c cases, shift s_c, S1 = sum d, S2 = sum d^2, S3 = sum d yc with
// d = yhat - s_c.  Chunk mean m_c = s_c + S1/n_c, chunk M2 = S2 - S1^2/n_c;
// merged (Chan et al.): Shh = sum M2_c + n_c (m_c - m)^2.
// sum yhat*yc = sum (S3_c + s_c Yc_c); Shy = that - m * Y1; Syy = Y2 - Y1^2/N.
__device__ double corr_fitness(const double *rec, const double *ychunk, int Nc, int chunk,
                               int nchunks, const Group &g) {
  const double N = (double)Nc;
  double y1 = 0.0, y2 = 0.0, tot = 0.0;
  for (int c = g.lane; c < nchunks; c += g.lanes) {
    y1 += ychunk[2 * c];
    y2 += ychunk[2 * c + 1];
    const double nc = (double)min(chunk, Nc - c * chunk);
    tot += nc * rec[c * PSTRIDE + 1] + rec[c * PSTRIDE + 2];
  }
  y1 = g.sum(y1);
  y2 = g.sum(y2);
  const double m = g.sum(tot) / N;
  // every chunk but the last has `chunk` cases: one reciprocal instead of two divisions a chunk
  const double inv_full = 1.0 / (double)chunk, inv_last = 1.0 / (double)(Nc - (nchunks - 1) * chunk);
  double shh = 0.0, cross = 0.0;
  for (int c = g.lane; c < nchunks; c += g.lanes) {
    const double nc = (double)min(chunk, Nc - c * chunk), inv = c == nchunks - 1 ? inv_last : inv_full;
    const double s = rec[c * PSTRIDE + 1], a = rec[c * PSTRIDE + 2];
    const double b = rec[c * PSTRIDE + 3], d = rec[c * PSTRIDE + 4];
    const double mc = s + a * inv;
    shh += (b - a * a * inv) + nc * (mc - m) * (mc - m);
    cross += d + s * ychunk[2 * c];
  }
  shh = g.sum(shh);
  const double shy = g.sum(cross) - m * y1;
  const double syy = y2 - y1 * y1 / N;
  double fit = 1.0;
  if (isfinite(shh) && isfinite(shy) && isfinite(syy) && shh > 0.0 && syy > 0.0 && Nc >= 2) {
    const double r2 = (shy * shy) / (syy * shh);
    fit = 1.0 - r2;
    fit = fit < 0.0 ? 0.0 : (fit > 1.0 ? 1.0 : fit);
  }
  return fit;
}

// Eq. 2 of one program from its chunk records [shift s, S1 = sum d,
// S2 = sum d^2, X = sum d e, E1 = sum e, E2 = sum e^2, c1, c2] over the
// valid pairs (d = yhat - s, e = y - ybar).  Valid pairs of chunk c:
// n_c = cases - c1 - c2.  Shh merges the chunks by Chan et al.; e shares one
// centre, so See = E2 - E1^2 / n; Seh = sum (X_c + s_c E1_c) - m E1.
__device__ double r4_score(const double *rec, int Nc, int chunk, int nchunks, double M, double *c1o,
                           double *c2o, const Group &g) {
  double c1 = 0.0, c2 = 0.0, n = 0.0, tot = 0.0, e1 = 0.0, e2 = 0.0;
  for (int c = g.lane; c < nchunks; c += g.lanes) {
    const double *r = rec + c * PSTRIDE;
    const double nv = (double)min(chunk, Nc - c * chunk) - r[6] - r[7];
    c1 += r[6];
    c2 += r[7];
    n += nv;
    tot += r[1] + nv * r[0];
    e1 += r[4];
    e2 += r[5];
  }
  c1 = g.sum(c1);
  c2 = g.sum(c2);
  n = g.sum(n);
  tot = g.sum(tot);
  e1 = g.sum(e1);
  e2 = g.sum(e2);
  double r2 = 0.0;
  if (n >= 2.0) {
    const double m = tot / n;
    double shh = 0.0, seh = 0.0;
    for (int c = g.lane; c < nchunks; c += g.lanes) {
      const double *r = rec + c * PSTRIDE;
      const double nv = (double)min(chunk, Nc - c * chunk) - r[6] - r[7];
      if (nv <= 0.0) continue;
      const double mc = r[0] + r[1] / nv;
      shh += (r[2] - r[1] * r[1] / nv) + nv * (mc - m) * (mc - m);
      seh += r[3] + r[0] * r[4];
    }
    shh = g.sum(shh);
    seh = g.sum(seh) - m * e1;
    const double see = e2 - e1 * e1 / n;
    if (isfinite(shh) && isfinite(seh) && isfinite(see) && shh > 0.0 && see > 0.0) {
      r2 = (seh * seh) / (shh * see);
      r2 = r2 < 0.0 ? 0.0 : (r2 > 1.0 ? 1.0 : r2);
    }
  }
  *c1o = c1;
  *c2o = c2;
  return M * (r2 * r2) * n - M * (c1 - c2);
}

// fitness of program p from its partial records (mode picks the outputs);
// called by all lanes of a group, lane 0 writes
__device__ void finalize_one(int mode, const double *partials, const int32_t *flags,
                             const double *ychunk, int P, int N, int chunk, int nchunks,
                             double *fitness, int p, const Group &g, int M = 0, int32_t *counts = nullptr) {
  const double INF = __longlong_as_double(0x7ff0000000000000ll);
  if (mode == MODE_R4 || mode == MODE_P2P) {
    double c1 = 0.0, c2 = 0.0, sc = -INF;
    if (!flags[p]) {
      const double *rec = partials + (size_t)p * nchunks * PSTRIDE;
      if (mode == MODE_R4) {
        sc = r4_score(rec, N, chunk, nchunks, (double)M, &c1, &c2, g);
      } else {
        sc = 0.0;
        for (int c = g.lane; c < nchunks; c += g.lanes) {
          sc += rec[c * PSTRIDE];
          c1 += rec[c * PSTRIDE + 6];
          c2 += rec[c * PSTRIDE + 7];
        }
        sc = g.sum(sc);  // integers below 2^53: exact in any order
        c1 = g.sum(c1);
        c2 = g.sum(c2);
      }
    }
    if (g.lane == 0) {
      fitness[p] = sc;
      if (counts) {
        counts[2 * p] = (int32_t)c1;
        counts[2 * p + 1] = (int32_t)c2;
      }
    }
    return;
  }
  double *mse_out = fitness;
  double *corr_out = mode == MODE_BOTH ? fitness + P : fitness;
  if (flags[p]) {
    if (g.lane == 0 && mode != MODE_CORR) mse_out[p] = INF;
    if (g.lane == 0 && mode != MODE_MSE) corr_out[p] = INF;
    return;
  }
  const double *rec = partials + (size_t)p * nchunks * PSTRIDE;
  if (mode != MODE_CORR) {
    double se = 0.0;
    for (int c = g.lane; c < nchunks; c += g.lanes) se += rec[c * PSTRIDE];
    se = g.sum(se);
    if (g.lane == 0) mse_out[p] = isfinite(se) ? se / (double)N : INF;
  }
  if (mode != MODE_MSE) {
    const double f = corr_fitness(rec, ychunk, N, chunk, nchunks, g);
    if (g.lane == 0) corr_out[p] = f;
  }
}

struct FinalParams {
  const double *partials;
  const int32_t *flags;
  const double *ychunk;
  int P, N, chunk, nchunks, mode;
  double *fitness;  // [P] or [2][P]
  int M;            // Beagle scores
  int32_t *counts;  // Beagle scores: [P][2] (c1, c2) or NULL
};

constexpr int FINAL_THREADS = 128;

__global__ void __launch_bounds__(FINAL_THREADS) finalize_kernel(FinalParams f) {
  launch_wait();
  const int lanes = merge_lanes(f.nchunks), p = (blockIdx.x * FINAL_THREADS + threadIdx.x) / lanes;
  if (p >= f.P) return;
  finalize_one(f.mode, f.partials, f.flags, f.ychunk, f.P, f.N, f.chunk, f.nchunks, f.fitness, p, group_of(lanes), f.M,
               f.counts);
}

// ---------------------------------------------------------------- batched prep / finalize
// one block per (problem, chunk) of the problems that need the centred
// target (its chunk sums come from the decode launch)

__global__ void __launch_bounds__(PREP_THREADS) ycenter_batched_kernel(const __grid_constant__ BatchParams b) {
  __shared__ double red[PREP_THREADS / 32];
  launch_wait();
  const BatchProblem &q = b.prob[corr_problem_of_block(b)];
  ycenter_chunk(q.y, q.N, q.chunk, q.nchunks, (int)blockIdx.x - q.corr_chunk_begin, q.ysum, false, q.yc,
                q.ychunk, red);
}

// blocks (problem, FINAL_THREADS / merge_lanes programs of it)
__global__ void __launch_bounds__(FINAL_THREADS) finalize_batched_kernel(const __grid_constant__ BatchParams b) {
  launch_wait();
  const BatchProblem &q = b.prob[blockIdx.x];
  const int lanes = merge_lanes(q.nchunks), per = FINAL_THREADS / lanes;
  const Group g = group_of(lanes);
  for (int p = blockIdx.y * per + threadIdx.x / lanes; p < q.P; p += gridDim.y * per)
    finalize_one(q.mode, q.partials, q.flags, q.ychunk, q.P, q.N, q.chunk, q.nchunks, q.fitness, p, g);
}

// ---------------------------------------------------------------- host side
typedef void (*EvalKernel)(EvalParams);

// The instantiations: base and EXT with 4 or 5 CTAs per SM, and those that read
// rows in halves (4 CTAs the EXT one).
template <int MODE>
EvalKernel eval_kernel_m(bool ext, bool wide, int minb) {
  if (!wide && ext) return eval_kernel<MODE, true, false, 4>;
  if (!wide) return minb == 5 ? eval_kernel<MODE, false, false, 5> : eval_kernel<MODE, false, false, 4>;
  if (minb == 5) return ext ? eval_kernel<MODE, true, true, 5> : eval_kernel<MODE, false, true, 5>;
  return ext ? eval_kernel<MODE, true, true, 4> : eval_kernel<MODE, false, true, 4>;
}
EvalKernel eval_kernel_for(int mode, bool ext, bool wide, int minb) {
  switch (mode) {
    case MODE_PREDICT: return eval_kernel_m<MODE_PREDICT>(ext, wide, minb);
    case MODE_MSE: return eval_kernel_m<MODE_MSE>(ext, wide, minb);
    case MODE_CORR: return eval_kernel_m<MODE_CORR>(ext, wide, minb);
    case MODE_R4: return eval_kernel_m<MODE_R4>(ext, wide, minb);
    case MODE_P2P: return eval_kernel_m<MODE_P2P>(ext, wide, minb);
    default: return eval_kernel_m<MODE_BOTH>(ext, wide, minb);
  }
}

// CTAs of `kernel` with `smem` bytes each on the whole GPU
sr_status persistent_grid(sr_ctx *ctx, const void *kernel, int smem, int *grid) {
  sr_status st = allow_dynamic_smem(ctx, kernel);
  if (st != SR_OK) return st;
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, WARPS * 32, smem);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  if (nb < 1) return fail(ctx, SR_EINVAL, "Lmax too large for shared memory");
  *grid = nb * ctx->num_sms;
  return SR_OK;
}

sr_status launch_pass(sr_ctx *ctx, int mode, bool ext, bool wide, int minb, int smem, const EvalParams &ep) {
  const EvalKernel k = eval_kernel_for(mode, ext, wide, minb);
  int grid = 0;
  sr_status st = persistent_grid(ctx, reinterpret_cast<const void *>(k), smem, &grid);
  if (st != SR_OK) return st;
  SR_CHECK_CUDA(ctx, launch(k, grid, WARPS * 32, smem, ctx->stream, ep));
  ctx->launches += 1;
  return SR_OK;
}

struct Plan {
  int minb;       // CTAs per SM of the main passes (eval_kernel's MINB)
  int slots, words;  // stack slots and words of code per warp of the main passes
  int smem, chunk, nchunks;
  int smem_deep;  // shared memory of the deep pass (0: none)
  long long items;
  bool wide;      // the rows of X are laid out for 256-bit loads (its own, or the table's)
  bool stage;     // X is copied to the table's first rows (no transforms)
  int xform;      // the variable table's depth (0: none; rows of ldxt floats)
  int ldxt;
  size_t off_queue, off_flags, off_ncode, off_code, off_part, off_yc,
      off_ych, off_ysum, off_xt, off_xneed, bytes;
};

// Whether a call (or a batch's problem) of P programs and N cases over nvars variables
// reads the variable table (0: no; 1: u(x_j); 2: also the compositions, where the
// table stays within XFORM2_MAX_BYTES), and that table's row stride.
inline int use_xform(const sr_ctx *ctx, int P, int nvars, int N, int *ldxt) {
  *ldxt = (int)align_up((size_t)N, CPL);  // whole groups of 8 cases (sr_vm.cuh, WIDE)
  const bool automatic = ctx->xform == 1 && N >= XFORM_MIN_N && P >= XFORM_MIN_P;
  if (!(ctx->xform == 2 || automatic)) return 0;
  const long long cells2 = (long long)xform_rows(nvars, 2) * align_up((size_t)N, 4);
  if (cells2 < 0xFFFFFFFFll && cells2 * 4 <= XFORM2_MAX_BYTES) return 2;
  return (long long)xform_rows(nvars, 1) * *ldxt < 0xFFFFFFFFll ? 1 : 0;
}

// whether rows of X at this address and stride can be read by 256-bit loads
// (8 cases from any multiple of 8 on)
inline bool rows_are_wide(const float *X, long long ldx) { return ((uintptr_t)X & 31) == 0 && ldx % CPL == 0; }

// How a call lays out its rows: the variable table, a copy of X where X itself
// is not laid out for wide loads, or X as it is.
enum Layout { LAY_TABLE, LAY_COPY, LAY_PLAIN };

void make_plan(sr_ctx *ctx, int P, int Lmax, int N, Plan *pl, int nvars, bool x_wide, Layout lay) {
  pl->minb = eval_minb(Lmax, ctx->eval_ctas);
  pl->slots = shallow_slots(Lmax, pl->minb);
  pl->words = shallow_words(Lmax, pl->minb);
  pl->smem = shallow_smem(Lmax, pl->minb);
  pl->smem_deep = deep_smem(Lmax, pl->minb);
  const long long warps =
      (long long)chunk_ctas(Lmax, chunk_minb(Lmax, ctx->eval_ctas)) * ctx->num_sms * WARPS;
  const long long want = warps * TARGET_ITEMS_PER_WARP;
  int nch = (int)((want + P - 1) / (P > 0 ? P : 1));
  // chunks of at least one warp step: a small problem (few programs, few
  // cases) then still spreads over many warps, its items one step each
  const int max_chunks = (N + STEP - 1) / STEP;
  nch = nch < 1 ? 1 : (nch > max_chunks ? max_chunks : nch);
  int chunk = (N + nch - 1) / nch;
  pl->xform = use_xform(ctx, P, nvars, N, &pl->ldxt);
  if (lay != LAY_TABLE) pl->xform = 0;
  pl->stage = !pl->xform && !x_wide && lay != LAY_PLAIN;
  pl->wide = pl->xform || pl->stage || x_wide;
  if (ctx->tile_cases > 0) {
    chunk = ctx->tile_cases;  // autotuned cases per work item
  } else if (pl->xform) {
    const long long cap = XFORM_SLICE_BYTES / (4ll * xform_rows(nvars, pl->xform));
    if (chunk > cap) chunk = (int)(cap > STEP ? cap : STEP);
  }
  chunk = (chunk + STEP - 1) / STEP * STEP;
  pl->chunk = chunk;
  pl->nchunks = (N + chunk - 1) / chunk;
  pl->items = (long long)P * pl->nchunks;
  const size_t tokens = (size_t)P * Lmax;
  Carver cv;
  pl->off_queue = cv.take(256);
  pl->off_flags = cv.take((size_t)P * 4);
  pl->off_ncode = cv.take((size_t)P * 4);
  pl->off_code = cv.take(tokens * 8);
  pl->off_part = cv.take((size_t)pl->items * PSTRIDE * 8);
  pl->off_yc = cv.take(align_up((size_t)N, STEP) * 4);
  pl->off_ych = cv.take((size_t)pl->nchunks * 16);
  pl->off_ysum = cv.take((size_t)pl->nchunks * 16);
  // the variable table: X's rows, then u(x_j) for the 12 unary operators
  // (those some program reads are filled per call); where the call is large
  // enough for it to pay and its row offsets fit the 32-bit operand
  pl->off_xt = pl->off_xneed = 0;
  if (pl->xform) {
    const size_t rows = (size_t)xform_rows(nvars, pl->xform);
    pl->off_xt = cv.take(rows * pl->ldxt * 4);
    pl->off_xneed = cv.take(rows - nvars);
  } else if (pl->stage) {
    pl->off_xt = cv.take((size_t)nvars * pl->ldxt * 4);
  }
  pl->bytes = cv.off;
}

sr_status check_common(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths,
                       const float *consts, int P, int Lmax, int K, const float *X, int nvars,
                       int N, int ldx) {
  if (!ctx) return SR_EINVAL;
  if (P < 0) return fail(ctx, SR_EINVAL, "P < 0");
  if (Lmax < 1 || Lmax > SR_MAX_LMAX) return fail(ctx, SR_EINVAL, "Lmax %d outside [1, %d]", Lmax, SR_MAX_LMAX);
  if (K < 0 || K > SR_MAX_CONSTS) return fail(ctx, SR_EINVAL, "K %d outside [0, %d]", K, SR_MAX_CONSTS);
  if (nvars < 1 || nvars > SR_MAX_VARS) return fail(ctx, SR_EINVAL, "nvars %d outside [1, %d]", nvars, SR_MAX_VARS);
  if (N < 1) return fail(ctx, SR_EINVAL, "N must be >= 1");
  if (ldx < N || ldx % 4) return fail(ctx, SR_EINVAL, "ldx %d must be >= N and a multiple of 4", ldx);
  if ((long long)ldx * nvars > 0xFFFFFFFFll)
    return fail(ctx, SR_EINVAL, "X too large: nvars * ldx must stay below 2^32 elements");
  if (P > 0 && (!programs || !lengths || (K > 0 && !consts) || !X))
    return fail(ctx, SR_EINVAL, "NULL input pointer");
  if (((uintptr_t)X) & 15) return fail(ctx, SR_EINVAL, "X must be 16-byte aligned");
  return SR_OK;
}

int mode_of(sr_fitness_kind k) {
  return k == SR_MSE ? MODE_MSE : (k == SR_CORR ? MODE_CORR : MODE_BOTH);
}

sr_status launch_eval(sr_ctx *ctx, int mode, const uint8_t *programs, const int32_t *lengths,
                      const float *consts, int P, int Lmax, int K, const float *X, const float *y,
                      int nvars, int N, int ldx, double *fitness, int32_t *prog_flags, float *yhat,
                      int ldy, int M = 0, int32_t *counts = nullptr) {
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  Plan pl;
  const bool x_wide = rows_are_wide(X, ldx);
  // with less room (as inside stream capture): without the variable table,
  // then without a copy of X
  sr_status st = SR_ENOMEM;
  for (Layout lay : {LAY_TABLE, LAY_COPY, LAY_PLAIN}) {
    make_plan(ctx, P, Lmax, N, &pl, nvars, x_wide, lay);
    st = ensure_workspace(ctx, pl.bytes);
    if (st != SR_ENOMEM) break;
  }
  if (st != SR_OK) return st;
  char *ws = ctx->ws;
  cudaStream_t s = ctx->stream;

  EvalParams ep;
  ep.programs = programs;
  ep.lengths = lengths;
  ep.consts = consts;
  ep.P = P;
  ep.Lmax = Lmax;
  ep.K = K;
  ep.X = X;
  ep.y = y;
  ep.yc = reinterpret_cast<const float *>(ws + pl.off_yc);
  ep.nvars = nvars;
  ep.N = N;
  ep.ldx = ldx;
  ep.chunk = pl.chunk;
  ep.nchunks = pl.nchunks;
  ep.total_items = pl.items;
  ep.partials = reinterpret_cast<double *>(ws + pl.off_part);
  ep.flags = prog_flags ? prog_flags : reinterpret_cast<int32_t *>(ws + pl.off_flags);
  ep.code = reinterpret_cast<uint2 *>(ws + pl.off_code);
  ep.ncode = reinterpret_cast<int32_t *>(ws + pl.off_ncode);
  ep.queue = reinterpret_cast<unsigned long long *>(ws + pl.off_queue);
  ep.yhat = yhat;
  ep.ldy = ldy;
  ep.slots = pl.slots;
  ep.words = pl.words;
  ep.warp_bytes = pl.smem / WARPS;
  ep.pass = PASS_BASE;
  ep.abort = ctx->abort_flag;
  ep.err = ctx->dev_words;
  ep.score_M = M;
  ep.xform = pl.xform;
  ep.xneed = pl.xform ? reinterpret_cast<uint8_t *>(ws + pl.off_xneed) : nullptr;
  if (pl.xform || pl.stage) {  // the kernels read the table's rows; the decoder writes its row offsets
    ep.X = reinterpret_cast<const float *>(ws + pl.off_xt);
    ep.ldx = pl.ldxt;
  }
  if (pl.stage) {
    ep.Xsrc = X;
    ep.ldsrc = ldx;
  }

  if (pl.xform) SR_CHECK_CUDA(ctx, cudaMemsetAsync(ep.xneed, 0, (size_t)(xform_rows(nvars, pl.xform) - nvars), s));
  const int stage = pl.stage ? stage_blocks(nvars, N) : 0;
  const bool centred = mode == MODE_CORR || mode == MODE_BOTH || mode == MODE_R4;
  double *ych = reinterpret_cast<double *>(ws + pl.off_ych);
  ep.finite_only = mode == MODE_R4;
  if (centred) ep.ysum = reinterpret_cast<double *>(ws + pl.off_ysum);
  const CenterParams cp{y, N, pl.chunk, pl.nchunks, ep.finite_only, ep.ysum, const_cast<float *>(ep.yc), ych};
  const int yblocks = centred ? pl.nchunks : 0;
  SR_CHECK_CUDA(ctx, launch(decode_kernel, yblocks + (P + DECODE_WARPS - 1) / DECODE_WARPS + stage, DECODE_WARPS * 32,
                            DECODE_WARPS * decode_scratch_bytes(Lmax), s, ep));
  ctx->launches += 1;
  if (pl.xform) {
    SR_CHECK_CUDA(ctx, launch(xform_kernel, yblocks + xform_blocks(nvars, N), XF_THREADS, 0, s, X, ldx, nvars, N, pl.ldxt,
                              pl.xform, ep.xneed, reinterpret_cast<float *>(ws + pl.off_xt), yblocks, cp));
    ctx->launches += 1;
  } else if (centred) {
    SR_CHECK_CUDA(ctx, launch(ycenter_kernel, pl.nchunks, PREP_THREADS, 0, s, cp));
    ctx->launches += 1;
  }
  st = launch_pass(ctx, mode, false, pl.wide, pl.minb, pl.smem, ep);
  ep.pass = PASS_EXT;
  if (st == SR_OK) st = launch_pass(ctx, mode, true, pl.wide, pl.minb, pl.smem, ep);
  if (st == SR_OK && pl.smem_deep) {
    ep.pass = PASS_DEEP;
    ep.slots = slots_for(Lmax);
    ep.warp_bytes = pl.smem_deep / WARPS;
    st = launch_pass(ctx, mode, true, pl.wide, 4, pl.smem_deep, ep);
  }
  if (st != SR_OK) return st;
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  if (mode != MODE_PREDICT) {
    FinalParams fp{ep.partials, ep.flags, ych, P, N, pl.chunk, pl.nchunks, mode, fitness, M, counts};
    const int per = FINAL_THREADS / merge_lanes(pl.nchunks);
    SR_CHECK_CUDA(ctx, launch(finalize_kernel, (P + per - 1) / per, FINAL_THREADS, 0, s, fp));
    SR_CHECK_CUDA(ctx, cudaGetLastError());
    ctx->launches += 1;
  }
  return SR_OK;
}

// ---------------------------------------------------------------- batched host side
typedef void (*BatchKernel)(const BatchParams);
template <int MINB>
BatchKernel batch_kernel_m(bool ext, bool lean) {
  if (ext) return eval_batched_kernel<true, true, MINB, false>;
  return lean ? eval_batched_kernel<false, true, MINB, true> : eval_batched_kernel<false, true, MINB, false>;
}
BatchKernel batch_kernel_for(bool ext, bool wide, int minb, bool lean) {
  if (!wide) return ext ? eval_batched_kernel<true, false, 4, false> : eval_batched_kernel<false, false, 4, false>;
  return minb == 3 ? batch_kernel_m<3>(ext, lean) : (minb == 5 ? batch_kernel_m<5>(ext, lean) : batch_kernel_m<4>(ext, lean));
}
sr_status launch_batch_pass(sr_ctx *ctx, bool ext, bool wide, int minb, int smem, const BatchParams &b, bool lean = false) {
  const BatchKernel k = batch_kernel_for(ext, wide, minb, lean);
  int grid = 0;
  sr_status st = persistent_grid(ctx, reinterpret_cast<const void *>(k), smem, &grid);
  if (st != SR_OK) return st;
  SR_CHECK_CUDA(ctx, launch(k, grid, WARPS * 32, smem, ctx->stream, b));
  ctx->launches += 1;
  return SR_OK;
}

sr_status launch_batched(sr_ctx *ctx, const sr_problem *pr, int nprob) {
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  int maxL = 1;
  double work = 0.0;
  for (int i = 0; i < nprob; ++i) {
    const sr_problem &q = pr[i];
    sr_status st = check_common(ctx, q.programs, q.lengths, q.consts, q.P, q.Lmax, q.K, q.X, q.nvars,
                                q.N, q.ldx);
    if (st != SR_OK) return fail(ctx, st, "problem %d: %s", i, ctx->msg);
    if (q.kind != SR_MSE && q.kind != SR_CORR && q.kind != SR_MSE_CORR)
      return fail(ctx, SR_EINVAL, "problem %d: unknown fitness kind", i);
    if (q.P > 0 && (!q.y || !q.fitness || (((uintptr_t)q.y) & 15)))
      return fail(ctx, SR_EINVAL, "problem %d: y NULL or not 16-byte aligned, or fitness NULL", i);
    if (q.cases_per_tile < 0) return fail(ctx, SR_EINVAL, "problem %d: cases_per_tile < 0", i);
    maxL = q.Lmax > maxL ? q.Lmax : maxL;
    work += (double)q.P * (double)q.N;
  }
  // CTAs per SM of the main passes: 4 unless tuned (3 gives more stack slots
  // and registers, 5 more warps); it must leave room for min(slots_for, 4)
  // stack slots
  int bminb = ctx->batched_ctas ? ctx->batched_ctas : 4;
  if (bminb == 5 && shallow_smem(maxL, 5) > smem_target(5)) bminb = 4;
  const int smem = shallow_smem(maxL, bminb), smem_deep = deep_smem(maxL, bminb);
  // the cases per item by chunk_ctas' rule, whatever the kernels take
  const int code = ((maxL * 8 + 15) / 16) * 16;
  const int cminb = ctx->batched_ctas == 5 && WARPS * (fit_slots(maxL, 5, code) * SLOT_BYTES + code) > smem_target(5)
                        ? 4
                        : (ctx->batched_ctas ? ctx->batched_ctas : 4);
  const long long warps = (long long)chunk_ctas(maxL, cminb) * ctx->num_sms * WARPS;
  Layout lay = LAY_TABLE;
  const double want = (double)warps * TARGET_ITEMS_PER_WARP;

  // chunking per problem: items in proportion to its share of the work
  std::vector<int> chunk(nprob), nch(nprob), order;
  for (int i = 0; i < nprob; ++i) {
    const sr_problem &q = pr[i];
    if (q.P == 0) continue;
    int c;
    if (q.cases_per_tile > 0) {
      c = q.cases_per_tile;
    } else {
      const double share = want * ((double)q.P * (double)q.N) / (work > 0 ? work : 1.0);
      int n = (int)ceil(share / q.P);
      const int max_chunks = (q.N + STEP - 1) / STEP;
      n = n < 1 ? 1 : (n > max_chunks ? max_chunks : n);
      c = (q.N + n - 1) / n;
      int ldxt = 0;
      const int xf = use_xform(ctx, q.P, q.nvars, q.N, &ldxt);
      if (xf) {  // as in make_plan: the item's slice of the problem's table
        const long long cap = XFORM_SLICE_BYTES / (4ll * xform_rows(q.nvars, xf));
        if (c > cap) c = (int)(cap > STEP ? cap : STEP);
      }
    }
    c = (c + STEP - 1) / STEP * STEP;
    chunk[i] = c;
    nch[i] = (q.N + c - 1) / c;
    order.push_back(i);
  }
  // longest items first (cases per item x longest program), so the tail of
  // the launch is made of short items
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return (double)chunk[a] * pr[a].Lmax > (double)chunk[b] * pr[b].Lmax;
  });

  // workspace: the largest group decides (all groups reuse it in turn)
  auto group_bytes = [&](size_t g0, size_t g1, BatchParams *bpar) -> size_t {
    Carver cv;
    long long depth2 = 0;  // bytes of the group's tables with compositions
    const size_t off_q = cv.take(256);
    long long items = 0;
    int corr_chunks = 0, ncorr = 0, progs = 0, stages = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int i = order[g];
      const sr_problem &q = pr[i];
      const int mode = mode_of(q.kind);
      const size_t tokens = (size_t)q.P * q.Lmax;
      const size_t off_f = q.prog_flags ? 0 : cv.take((size_t)q.P * 4);
      const size_t off_nc = cv.take((size_t)q.P * 4);
      const size_t off_code = cv.take(tokens * 8);
      const size_t off_p = cv.take((size_t)q.P * nch[i] * PSTRIDE * 8);
      size_t off_yc = 0, off_ych = 0, off_st = 0, off_xt = 0, off_xn = 0;
      const bool corr = mode != MODE_MSE;
      if (corr) {
        off_yc = cv.take(align_up((size_t)q.N, STEP) * 4);
        off_ych = cv.take((size_t)nch[i] * 16);
        off_st = cv.take((size_t)nch[i] * 16);
      }
      int ldxt = 0;
      int xf = lay == LAY_TABLE ? use_xform(ctx, q.P, q.nvars, q.N, &ldxt) : 0;
      ldxt = (q.N + CPL - 1) / CPL * CPL;
      const bool stage = !xf && lay != LAY_PLAIN && !rows_are_wide(q.X, q.ldx);
      if (xf == 2) {
        const long long b2 = (long long)xform_rows(q.nvars, 2) * ldxt * 4;
        if (depth2 + b2 > XFORM2_BATCH_BYTES) xf = 1;
        else depth2 += b2;
      }
      if (xf) {
        const size_t rows = (size_t)xform_rows(q.nvars, xf);
        off_xt = cv.take(rows * ldxt * 4);
        off_xn = cv.take(rows - q.nvars);
      } else if (stage) {
        off_xt = cv.take((size_t)q.nvars * ldxt * 4);
      }
      if (bpar) {
        BatchProblem &b = bpar->prob[g - g0];
        char *ws = ctx->ws;
        b.programs = q.programs;
        b.lengths = q.lengths;
        b.consts = q.consts;
        b.X = q.X;
        b.y = q.y;
        b.yc = corr ? reinterpret_cast<float *>(ws + off_yc) : nullptr;
        b.partials = reinterpret_cast<double *>(ws + off_p);
        b.flags = q.prog_flags ? q.prog_flags : reinterpret_cast<int32_t *>(ws + off_f);
        b.code = reinterpret_cast<uint2 *>(ws + off_code);
        b.ncode = reinterpret_cast<int32_t *>(ws + off_nc);
        b.fitness = q.fitness;
        b.ychunk = corr ? reinterpret_cast<double *>(ws + off_ych) : nullptr;
        b.ysum = corr ? reinterpret_cast<double *>(ws + off_st) : nullptr;
        b.ldx = q.ldx;
        b.item_begin = items;
        b.prog_begin = progs;
        b.P = q.P;
        b.Lmax = q.Lmax;
        b.K = q.K;
        b.nvars = q.nvars;
        b.N = q.N;
        b.chunk = chunk[i];
        b.nchunks = nch[i];
        b.mode = mode;
        b.corr_chunk_begin = corr ? corr_chunks : -1;
        b.xform = xf;
        b.xneed = xf ? reinterpret_cast<uint8_t *>(ws + off_xn) : nullptr;
        b.Xsrc = stage ? q.X : nullptr;
        b.ldsrc = q.ldx;
        b.stage_begin = stages;
        if (xf || stage) {
          b.X = reinterpret_cast<const float *>(ws + off_xt);
          b.ldx = ldxt;
        }
        if (corr) bpar->corr_list[ncorr] = (int)(g - g0);
      }
      items += (long long)q.P * nch[i];
      progs += q.P;
      if (stage) stages += stage_blocks(q.nvars, q.N);
      if (corr) {
        corr_chunks += nch[i];
        ++ncorr;
      }
    }
    if (bpar) {
      bpar->nprob = (int)(g1 - g0);
      bpar->ncorr = ncorr;
      bpar->total_progs = progs;
      bpar->total_items = items;
      bpar->queue = reinterpret_cast<unsigned long long *>(ctx->ws + off_q);
      bpar->slots = shallow_slots(maxL, bminb);
      bpar->words = shallow_words(maxL, bminb);
      bpar->maxL = maxL;
      bpar->warp_bytes = smem / WARPS;
      bpar->pass = PASS_BASE;
      bpar->decode_blocks = (progs + DECODE_WARPS - 1) / DECODE_WARPS;
      bpar->stage_blocks = stages;
      bpar->ysum_blocks = corr_chunks;
      bpar->abort = ctx->abort_flag;
      bpar->err = ctx->dev_words;
    }
    return cv.off;
  };
  if (order.empty()) return SR_OK;
  // with less room: without the variable tables, then without copies of X
  sr_status st = SR_ENOMEM;
  for (Layout l : {LAY_TABLE, LAY_COPY, LAY_PLAIN}) {
    lay = l;
    size_t need = 0;
    for (size_t g0 = 0; g0 < order.size(); g0 += MAX_BATCH)
      need = std::max(need, group_bytes(g0, std::min(order.size(), g0 + MAX_BATCH), nullptr));
    st = ensure_workspace(ctx, need);
    if (st != SR_ENOMEM) break;
  }
  if (st != SR_OK) return st;
  bool wide = true;
  for (int i : order) wide = wide && (lay != LAY_PLAIN || rows_are_wide(pr[i].X, pr[i].ldx));

  cudaStream_t s = ctx->stream;
  for (size_t g0 = 0; g0 < order.size(); g0 += MAX_BATCH) {
    const size_t g1 = std::min(order.size(), g0 + MAX_BATCH);
    BatchParams b;
    group_bytes(g0, g1, &b);
    for (int r = 0; r < b.nprob; ++r)
      if (b.prob[r].xform)
        SR_CHECK_CUDA(ctx, cudaMemsetAsync(b.prob[r].xneed, 0,
                                           (size_t)(xform_rows(b.prob[r].nvars, b.prob[r].xform) - b.prob[r].nvars), s));
    SR_CHECK_CUDA(ctx, launch(decode_batched_kernel, b.ysum_blocks + b.decode_blocks + b.stage_blocks, DECODE_WARPS * 32,
                              DECODE_WARPS * decode_scratch_bytes(maxL), s, b));
    ctx->launches += 1;
    for (size_t g = g0; g < g1; ++g) {  // the variable tables, from the problems' own X
      const BatchProblem &q = b.prob[g - g0];
      if (!q.xform) continue;
      const sr_problem &o = pr[order[g]];
      SR_CHECK_CUDA(ctx, launch(xform_kernel, xform_blocks(q.nvars, q.N), XF_THREADS, 0, s, o.X, o.ldx, q.nvars, q.N, (int)q.ldx,
                                q.xform, q.xneed, const_cast<float *>(q.X), 0, CenterParams{}));
      ctx->launches += 1;
    }
    if (b.ncorr > 0) {
      SR_CHECK_CUDA(ctx, launch(ycenter_batched_kernel, b.ysum_blocks, PREP_THREADS, 0, s, b));
      ctx->launches += 1;
    }
    double steps = 0.0;
    for (int r = 0; r < b.nprob; ++r) steps += (double)b.prob[r].P * ((b.prob[r].N + STEP - 1) / STEP);
    st = launch_batch_pass(ctx, false, wide, bminb, smem, b, steps <= (double)LEAN_MAX_STEPS * (double)b.total_items);
    b.pass = PASS_EXT;
    if (st == SR_OK) st = launch_batch_pass(ctx, true, wide, bminb, smem, b);
    if (st == SR_OK && smem_deep) {
      BatchParams bd = b;
      bd.pass = PASS_DEEP;
      bd.slots = slots_for(maxL);
      bd.warp_bytes = smem_deep / WARPS;
      st = launch_batch_pass(ctx, true, wide, 4, smem_deep, bd);
    }
    if (st != SR_OK) return st;
    int yblocks = 1;
    for (int r = 0; r < b.nprob; ++r) {
      const int per = FINAL_THREADS / merge_lanes(b.prob[r].nchunks);
      yblocks = std::max(yblocks, std::min((b.prob[r].P + per - 1) / per, 65535));
    }
    SR_CHECK_CUDA(ctx, launch(finalize_batched_kernel, dim3(b.nprob, yblocks), FINAL_THREADS, 0, s, b));
    SR_CHECK_CUDA(ctx, cudaGetLastError());
    ctx->launches += 1;
  }
  return SR_OK;
}

}  // namespace
}  // namespace sr

extern "C" {

sr_status sr_eval(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths, const float *consts,
                  int P, int Lmax, int K, const float *X, const float *y, int nvars, int N, int ldx,
                  sr_fitness_kind kind, double *fitness, int32_t *prog_flags) {
  using namespace sr;
  sr_status st = check_common(ctx, programs, lengths, consts, P, Lmax, K, X, nvars, N, ldx);
  if (st != SR_OK) return st;
  if (kind != SR_MSE && kind != SR_CORR && kind != SR_MSE_CORR)
    return fail(ctx, SR_EINVAL, "unknown fitness kind %d", (int)kind);
  if (P == 0) return SR_OK;
  if (!y || !fitness) return fail(ctx, SR_EINVAL, "NULL y or fitness");
  if (((uintptr_t)y) & 15) return fail(ctx, SR_EINVAL, "y must be 16-byte aligned");
  return launch_eval(ctx, mode_of(kind), programs, lengths, consts, P, Lmax, K, X, y, nvars, N, ldx,
                     fitness, prog_flags, nullptr, 0);
}

sr_status sr_eval_score(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths,
                        const float *consts, int P, int Lmax, int K, const float *X, const float *y,
                        int nvars, int N, int ldx, sr_score_kind kind, int M, double *score,
                        int32_t *pair_counts, int32_t *prog_flags) {
  using namespace sr;
  sr_status st = check_common(ctx, programs, lengths, consts, P, Lmax, K, X, nvars, N, ldx);
  if (st != SR_OK) return st;
  if (kind != SR_SCORE_R4 && kind != SR_SCORE_P2P)
    return fail(ctx, SR_EINVAL, "unknown score kind %d", (int)kind);
  if (M < 1 || M > (1 << 24)) return fail(ctx, SR_EINVAL, "M %d outside [1, 2^24]", M);
  if ((double)M * (double)N > 9007199254740992.0)
    return fail(ctx, SR_EINVAL, "M * N above 2^53: the score sum would not be exact");
  if (P == 0) return SR_OK;
  if (!y || !score) return fail(ctx, SR_EINVAL, "NULL y or score");
  if (((uintptr_t)y) & 15) return fail(ctx, SR_EINVAL, "y must be 16-byte aligned");
  return launch_eval(ctx, kind == SR_SCORE_R4 ? MODE_R4 : MODE_P2P, programs, lengths, consts, P, Lmax, K,
                     X, y, nvars, N, ldx, score, prog_flags, nullptr, 0, M, pair_counts);
}

sr_status sr_predict(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths,
                     const float *consts, int P, int Lmax, int K, const float *X, int nvars, int N,
                     int ldx, float *yhat, int ldy, int32_t *prog_flags) {
  using namespace sr;
  sr_status st = check_common(ctx, programs, lengths, consts, P, Lmax, K, X, nvars, N, ldx);
  if (st != SR_OK) return st;
  if (P == 0) return SR_OK;
  if (!yhat || ldy < N) return fail(ctx, SR_EINVAL, "yhat NULL or ldy < N");
  return launch_eval(ctx, MODE_PREDICT, programs, lengths, consts, P, Lmax, K, X, nullptr, nvars,
                     N, ldx, nullptr, prog_flags, yhat, ldy);
}

sr_status sr_eval_batched(sr_ctx *ctx, const sr_problem *problems, int nprob) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  if (nprob < 0 || (nprob > 0 && !problems)) return fail(ctx, SR_EINVAL, "bad problem list");
  if (nprob == 0) return SR_OK;
  return launch_batched(ctx, problems, nprob);
}

sr_status sr_set_tile(sr_ctx *ctx, int cases_per_tile) {
  if (!ctx || cases_per_tile < 0) return SR_EINVAL;
  ctx->tile_cases = cases_per_tile;
  return SR_OK;
}

sr_status sr_set_occupancy(sr_ctx *ctx, int eval_ctas_per_sm, int batched_ctas_per_sm) {
  if (!ctx) return SR_EINVAL;
  if (eval_ctas_per_sm != 0 && eval_ctas_per_sm != 4 && eval_ctas_per_sm != 5)
    return sr::fail(ctx, SR_EINVAL, "eval_ctas_per_sm %d: 0, 4 or 5", eval_ctas_per_sm);
  if (batched_ctas_per_sm != 0 && (batched_ctas_per_sm < 3 || batched_ctas_per_sm > 5))
    return sr::fail(ctx, SR_EINVAL, "batched_ctas_per_sm %d: 0, 3, 4 or 5", batched_ctas_per_sm);
  ctx->eval_ctas = eval_ctas_per_sm;
  ctx->batched_ctas = batched_ctas_per_sm;
  return SR_OK;
}

sr_status sr_set_transforms(sr_ctx *ctx, int mode) {
  if (!ctx) return SR_EINVAL;
  if (mode < 0 || mode > 2) return sr::fail(ctx, SR_EINVAL, "transform mode %d: 0, 1 or 2", mode);
  ctx->xform = mode;
  return SR_OK;
}

sr_status sr_reserve(sr_ctx *ctx, int P, int Lmax, int N) {
  using namespace sr;
  if (!ctx || P < 0 || Lmax < 1 || Lmax > SR_MAX_LMAX || N < 1) return SR_EINVAL;
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  size_t need = 0;
  for (int nv = 1; nv <= SR_MAX_VARS; ++nv) {  // the table's size depends on the variable count
    Plan pl;
    make_plan(ctx, P, Lmax, N, &pl, nv, false, LAY_TABLE);
    need = pl.bytes > need ? pl.bytes : need;
  }
  return ensure_workspace(ctx, need);
}

}  // extern "C"

// ---------------------------------------------------------------- allocation-free evaluation
// sr_eval_noalloc: the same kernels as sr_eval, with every byte of scratch
// taken from one file-scope device array instead of a context workspace.
#include <mutex>

namespace sr {
namespace {

constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)16 << 20;  // 16 MiB, held per device until exit
constexpr int NOALLOC_MAX_DEVICES = 64;

__device__ __align__(256) char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

std::mutex g_noalloc_mutex;
void *g_noalloc_addr[NOALLOC_MAX_DEVICES];  // device address of the array, per device

// Looks up the device address of the scratch array on the current device
// (once per device; the host-side symbol is not a device address).
sr_status noalloc_scratch(int dev, void **out) {
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return SR_EINVAL;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_addr[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return SR_ECUDA;
    }
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return SR_OK;
}

}  // namespace
}  // namespace sr

extern "C" sr_status sr_eval_noalloc(void *cuda_stream, const uint8_t *programs,
                                     const int32_t *lengths, const float *consts, int P, int Lmax,
                                     int K, const float *X, const float *y, int nvars, int N,
                                     int ldx, sr_fitness_kind kind, double *fitness,
                                     int32_t *prog_flags) {
  using namespace sr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SR_ECUDA;
  }
  // a context on the stack: nothing is allocated for it, and its workspace
  // is the static array, so the workspace never needs to grow
  sr_ctx local;
  local.device = dev;
  local.xform = 0;  // no variable table: the scratch stays within the terms sr.h lists
  local.stream = (cudaStream_t)cuda_stream;
  if (cudaDeviceGetAttribute(&local.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return SR_ECUDA;
  }
  sr_status st = check_common(&local, programs, lengths, consts, P, Lmax, K, X, nvars, N, ldx);
  if (st != SR_OK) return st;
  if (kind != SR_MSE && kind != SR_CORR && kind != SR_MSE_CORR) return SR_EINVAL;
  if (P == 0) return SR_OK;
  if (!y || !fitness || (((uintptr_t)y) & 15)) return SR_EINVAL;
  const int mode = mode_of(kind);
  // fit the plan into the array: fewer SMs' worth of persistent CTAs means
  // fewer work items and partial records
  Plan pl;
  for (;;) {
    make_plan(&local, P, Lmax, N, &pl, nvars, false, LAY_PLAIN);  // (a copy of X only where it fits as well)
    if (pl.bytes <= NOALLOC_SCRATCH_BYTES) break;
    if (local.num_sms == 1) return SR_ENOMEM;  // does not fit even on one SM
    local.num_sms = local.num_sms / 2 > 0 ? local.num_sms / 2 : 1;
  }
  void *scratch = nullptr;
  st = noalloc_scratch(dev, &scratch);
  if (st != SR_OK) return st;
  local.ws = static_cast<char *>(scratch);
  local.ws_bytes = NOALLOC_SCRATCH_BYTES;
  local.ws_fixed = true;
  return launch_eval(&local, mode, programs, lengths, consts, P, Lmax, K, X, y, nvars, N, ldx,
                     fitness, prog_flags, nullptr, 0);
}
