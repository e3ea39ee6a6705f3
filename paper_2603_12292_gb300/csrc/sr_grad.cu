// sr_grad.cu -- reverse-mode derivative of the interpreter (dMSE/dconst) and
// the Adam update of the constants.
//
// A program is decoded into a forward and a reverse program (sr_gradvm.cuh:
// Sethi-Ullman order, constant subtrees evaluated once).  Work item = (case
// chunk, program), one warp, 4 cases per lane (one 16-byte access per value),
// 128 cases per step.  Per step:
//   forward  -- the top of stack in registers, the slots below in shared memory.
//               What the reverse program wants and cannot have as an immediate or
//               a row goes on a LIFO tape: for a unary operator its local
//               derivative, computed next to the value (cos x with sin x from one
//               sincos, exp x, 1/x, ...), for a product the factors, for a quotient
//               the denominator and the result.  The tape lives in this warp's
//               global scratch (it stays in L2).
//   reverse  -- the adjoint in registers; where both operands of an operator read
//               constants, one operand's adjoint waits in a stack slot (the values
//               there are dead by then); constants add their adjoint into their
//               gradient sum.
// Nothing is kept between an evaluation and this call: the forward pass is
// recomputed.  Sums: per lane FP32 compensated (Kahan) over the item's
// cases, FP64 across lanes (shuffles) and chunks (finalize).
#include <math.h>

#include <algorithm>
#include <vector>

#include "sr_common.cuh"
#include "sr_gradvm.cuh"

namespace sr {
namespace {

constexpr int GWARPS = 8;    // warps per CTA
// CTAs per SM (64 registers a thread; 5 with 48 and 1.4 code words a token: 4,620 ->
// 5,387 us on 2,048 x 65,536, 4 with 1.4 words 4,882: programs go to the big pass)
constexpr int GMINB = 4;
constexpr int GSTRIDE = 32;  // doubles per partial record: [0] sum e^2, [1 + k] sum e dyhat/dc_k
constexpr int GTARGET_ITEMS_PER_WARP = 24;

struct GradParams {
  const uint8_t *programs;
  const int32_t *lengths;
  const float *consts;
  int P, Lmax, K;
  const float *X;
  const float *y;
  int nvars, N;
  long long ldx;
  int chunk, nchunks;
  long long total_items;
  double *partials;   // [P * nchunks][GSTRIDE]
  int32_t *flags;     // [P]
  uint2 *code;        // [P][grad_code_words(Lmax)] forward, then reverse program
  int32_t *nfwd, *nrev;  // [P] their words
  // [0] work counter, [1] work counter of the big pass, [2] the decoder's note that
  // some program's code is longer than the first pass's share (the big pass takes
  // those, with room for any), [5] the note as that pass reads it (grad_pass);
  // the decode launch zeroes the counters
  unsigned long long *queue;
  int cap;            // code words that a program of the first pass has at most
  int room;           // code words per warp of this launch
  int big;            // 1: the big pass
  char *gtape;        // per warp: Lmax entries of GSLOT bytes
  const int32_t *abort;  // sr_set_abort_flag (or NULL)
  unsigned *err;         // the context's latched error word
};

// shared memory of one warp: stack slots [slots_for(Lmax)] | gradient sums
// and compensations [2][K][32] | code
__host__ __device__ inline int grad_warp_bytes(int Lmax, int K, int words) {
  return slots_for(Lmax) * GSLOT + 2 * K * 128 + (words * 8 + 15) / 16 * 16;
}
// The code words a warp has room for in the first pass: all that any program can
// have where they fit beside GMINB CTAs, and then there is no big pass; else 2 a
// token and a few, or the fewer that one more CTA leaves as long as they are 1.9 a
// token (most programs of random or evolved populations have less).  With 2 a token
// and a few whatever the sizes (us): 2,048 programs of <= 24 tokens x 1,637 cases,
// K = 8, a few of them big, 158 -> 94 (their items come after all others); 512 x
// 20,000, K = 8, <= 128 tokens 776 -> 733 (3 CTAs -> 4), <= 256 tokens 1,867 -> 1,557
// (2 -> 3); three Adam steps on 23 problems of <= 16 tokens 311 -> 298 (one launch
// less a step); the larger share of shared memory costs 1 % on some of 64 tokens.
constexpr int words_beside(int ctas, int fixed) { return ((233472 / ctas - 1024) / GWARPS / 16 * 16 - fixed) / 8; }
constexpr int cap_words(int Lmax, int full, int fixed) {
  if (words_beside(GMINB, fixed) >= full) return full;
  for (int ctas = GMINB;; --ctas) {
    const int room = words_beside(ctas, fixed), some = 2 * Lmax + 8;
    if (10 * room >= 19 * Lmax) return room < some ? room : some;
  }
}
inline int grad_cap_words(int Lmax, int K) {
  return std::min(grad_code_words(Lmax), cap_words(Lmax, grad_code_words(Lmax), grad_warp_bytes(Lmax, K, 0)));
}
static_assert(cap_words(128, 9 * 128 / 2 + 4, 6 * GSLOT + 2 * 8 * 128) == 256, "128 tokens, 8 constants: 4 CTAs");
static_assert(cap_words(70, 9 * 70 / 2 + 4, 5 * GSLOT + 2 * 8 * 128) == 319, "70 tokens, 8 constants: no big pass");
// (one CTA leaves the longest programs more than enough: the search ends)
static_assert(10 * words_beside(1, DSM * GSLOT + 2 * SR_MAX_CONSTS * 128) >= 19 * SR_MAX_LMAX, "cap_words");

__device__ __forceinline__ GradDecode grad_decode_args(const GradParams &p, unsigned long long *queue, int cap) {
  return GradDecode{p.programs, p.lengths, p.consts, p.Lmax, p.K, p.nvars, p.ldx, p.code, p.nfwd, p.nrev, p.flags,
                    cap, queue + 2};
}

// a warp per program
__global__ void __launch_bounds__(DECODE_WARPS * 32) grad_decode_kernel(GradParams p) {
  extern __shared__ __align__(16) unsigned char dsm[];
  launch_wait();
  if (blockIdx.x == 0 && threadIdx.x < 2) p.queue[threadIdx.x] = 0;
  const int warp = threadIdx.x >> 5, prog = blockIdx.x * DECODE_WARPS + warp;
  if (prog < p.P)
    decode_grad_warp(grad_decode_args(p, p.queue, p.cap), prog, dsm + (size_t)warp * grad_scratch_bytes(p.Lmax),
                     slots_for(p.Lmax));
}

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

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// A warp's shared regions, laid out for the largest Lmax (Lw) and K (Kw) of a
// launch, and its tape.
struct GradWarp {
  uint32_t slot;  // shared address of this lane's entry of stack slot 0
  float *sums;    // this lane's gradient sums, [Kw][32], then their compensations
  uint2 *code;
  char *tape;     // this lane's entry of tape entry 0
};
__device__ __forceinline__ GradWarp grad_warp(unsigned char *smem, int Lw, int Kw, int room, char *gtape) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char *wb = smem + (size_t)warp * grad_warp_bytes(Lw, Kw, room);
  GradWarp w;
  w.slot = (uint32_t)__cvta_generic_to_shared(wb + lane * (GCPL * 4));
  w.sums = reinterpret_cast<float *>(wb + slots_for(Lw) * GSLOT) + lane;
  w.code = reinterpret_cast<uint2 *>(wb + slots_for(Lw) * GSLOT + 2 * Kw * 128);
  w.tape = gtape + (size_t)(blockIdx.x * GWARPS + warp) * Lw * GSLOT + lane * (GCPL * 4);
  return w;
}

// One work item: program `prog` on case chunk `c` with the calling warp.
// comp: floats from a sum to its compensation (32 Kw).
__device__ __forceinline__ void grad_item(const GradParams &p, int c, int prog, const GradWarp &w, int comp, int lane) {
  const int nf = p.nfwd[prog], words = nf + p.nrev[prog];
  __syncwarp();
  const uint2 *src = p.code + (size_t)prog * grad_code_words(p.Lmax);
  for (int i = lane; i < words; i += 32) w.code[i] = src[i];
  for (int k = 0; k < p.K; ++k) w.sums[k * 32] = w.sums[k * 32 + comp] = 0.f;
  __syncwarp();

  const uint32_t fwd = (uint32_t)__cvta_generic_to_shared(w.code), rev = fwd + 8 * nf;
  const int cbeg = c * p.chunk, cend = min(p.N, cbeg + p.chunk);
  const int last_group = (cend - 1) & ~(GCPL - 1);
  Kahan se;
  for (int base = cbeg; base < cend; base += GSTEP) {
    const int c0 = base + GCPL * lane;
    unsigned okm = 0;  // bit i: case c0 + i is inside the chunk
#pragma unroll
    for (int i = 0; i < GCPL; ++i) okm |= (c0 + i < cend ? 1u : 0u) << i;
    const float *xr = p.X + (okm ? c0 : last_group);
    char *tape = w.tape;
    const V4 T = run_forward(fwd, w.slot, xr, tape);
    // loss and seed: e = yhat - y on valid cases, 0 elsewhere
    float t[GCPL], e[GCPL];
    unpack4(T, t);
    float e2 = 0.0f;
#pragma unroll
    for (int i = 0; i < GCPL; ++i) {
      const bool ok = (okm >> i) & 1u;
      e[i] = ok ? t[i] - p.y[c0 + i] : 0.0f;
      e2 += e[i] * e[i];
    }
    se.add(e2);
    run_reverse(rev, w.slot, xr, tape, pack4(e), w.sums, comp, okm);
  }
  double *rec = p.partials + ((size_t)prog * p.nchunks + c) * GSTRIDE;
  const double sv = warp_sum(se.value());
  if (lane == 0) rec[0] = sv;
  for (int k = 0; k < p.K; ++k) {
    const double g = warp_sum((double)w.sums[k * 32] - (double)w.sums[k * 32 + comp]);
    if (lane == 0) rec[1 + k] = g;
  }
}

// whether a launch takes the program (big: the big pass)
__device__ __forceinline__ bool grad_takes(const GradParams &p, int prog, int cap, int big) {
  const int nf = p.nfwd[prog];
  return nf > 0 && ((nf + p.nrev[prog] > cap) == (big != 0));
}

// Whether a pass has programs.  The first hands the decoder's note over to the big
// pass and clears it for the next call, so that a replay of a captured call walks
// the big pass's items only when its own programs need it.
__device__ __forceinline__ bool grad_pass(unsigned long long *queue, int big) {
  if (big) return queue[5] != 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    queue[5] = queue[2];
    queue[2] = 0;
  }
  return true;
}

// Two passes over the work items: the second (big) for the programs whose code
// does not fit the first's share, which returns at once when there are none.
__global__ void __launch_bounds__(GWARPS * 32, GMINB) grad_kernel(GradParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_wait_only();
  if (!grad_pass(p.queue, p.big)) return;
  const int lane = threadIdx.x & 31;
  const GradWarp w = grad_warp(smem, p.Lmax, p.K, p.room, p.gtape);
  for (;;) {
    const long long item = next_item(p.queue + p.big, p.total_items, p.abort, p.err, lane);
    if (item >= p.total_items) break;
    const int c = (int)(item / (unsigned long long)p.P);
    const int prog = (int)(item % (unsigned long long)p.P);
    if (grad_takes(p, prog, p.cap, p.big)) grad_item(p, c, prog, w, 32 * p.K, lane);
  }
}

// ---------------------------------------------------------------- many problems, one launch
constexpr int MAX_GBATCH = 64;

struct GradBatch {
  GradParams prob[MAX_GBATCH];    // per problem (queue / tape / abort fields unused)
  long long item_begin[MAX_GBATCH];  // first work item of each problem
  int prog_begin[MAX_GBATCH];     // first program of each problem in the decode launch
  double *mse[MAX_GBATCH];
  double *dconst[MAX_GBATCH];
  int nprob, total_progs;
  long long total_items;
  unsigned long long *queue;
  char *gtape;
  const int32_t *abort;
  unsigned *err;
  int cap, room, big;             // as GradParams
  int Lw, Kw;                     // shared layout: the largest Lmax and K
};

__device__ __forceinline__ int batch_problem(const long long *begin, int nprob, long long x) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (begin[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// a warp per program of every problem
__global__ void __launch_bounds__(DECODE_WARPS * 32) grad_decode_batched_kernel(const __grid_constant__ GradBatch b) {
  extern __shared__ __align__(16) unsigned char dsm[];
  launch_wait();
  if (blockIdx.x == 0 && threadIdx.x < 2) b.queue[threadIdx.x] = 0;
  const int warp = threadIdx.x >> 5;
  const int g = blockIdx.x * DECODE_WARPS + warp;
  if (g >= b.total_progs) return;
  int q = 0;
  while (q + 1 < b.nprob && b.prog_begin[q + 1] <= g) ++q;
  decode_grad_warp(grad_decode_args(b.prob[q], b.queue, b.cap), g - b.prog_begin[q],
                   dsm + (size_t)warp * grad_scratch_bytes(b.Lw), slots_for(b.prob[q].Lmax));
}

// Work items of every problem from one atomic counter, longest items first
// (problems ordered by cases per item x Lmax); problem q owns items
// [item_begin_q, item_begin_q + P_q nchunks_q), chunk-major inside.
__global__ void __launch_bounds__(GWARPS * 32, GMINB) grad_batched_kernel(const __grid_constant__ GradBatch b) {
  extern __shared__ __align__(16) unsigned char smem[];
  launch_wait_only();
  if (!grad_pass(b.queue, b.big)) return;
  const int lane = threadIdx.x & 31;
  const GradWarp w = grad_warp(smem, b.Lw, b.Kw, b.room, b.gtape);
  for (;;) {
    const long long item = next_item(b.queue + b.big, b.total_items, b.abort, b.err, lane);
    if (item >= b.total_items) break;
    const int q = batch_problem(b.item_begin, b.nprob, item);
    const GradParams &p = b.prob[q];
    const long long local = item - b.item_begin[q];
    const int prog = (int)(local % p.P);
    if (grad_takes(p, prog, b.cap, b.big)) grad_item(p, (int)(local / p.P), prog, w, 32 * b.Kw, lane);
  }
}

struct GradFinal {
  const double *partials;
  const int32_t *flags;
  int P, N, K, nchunks;
  double *mse, *dconst;
};

// The 1 + K sums of a program on as many lanes of a group of 16 (K = 16: 32),
// each over the chunks in order (the order of the results since the first
// adjoint), the chunks' records read ahead of the adds.  A thread per program
// read them one after the other: 83 us for 2,048 programs of 64 chunks, now
// 13.
constexpr int GFINAL_THREADS = 128;
__host__ __device__ inline int grad_final_group(int K) { return K < 16 ? 16 : 32; }
__device__ void finalize_grad_one(const GradFinal &f, int p, int k) {
  if (k > f.K) return;
  double v = 0.0;
  const bool bad = f.flags[p] != 0;
  if (!bad) {
    const double *rec = f.partials + (size_t)p * f.nchunks * GSTRIDE + k;
    int c = 0;
    for (; c + 8 <= f.nchunks; c += 8) {
      double r[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) r[i] = rec[(c + i) * GSTRIDE];
#pragma unroll
      for (int i = 0; i < 8; ++i) v += r[i];
    }
    for (; c < f.nchunks; ++c) v += rec[c * GSTRIDE];
  }
  if (k == 0) f.mse[p] = !bad && isfinite(v) ? v / (double)f.N : __longlong_as_double(0x7ff0000000000000ll);
  else f.dconst[(size_t)p * f.K + k - 1] = bad ? 0.0 : 2.0 * v / (double)f.N;
}

__global__ void __launch_bounds__(GFINAL_THREADS) grad_finalize_kernel(GradFinal f) {
  launch_wait();
  const int g = grad_final_group(f.K), p = (blockIdx.x * GFINAL_THREADS + threadIdx.x) / g;
  if (p < f.P) finalize_grad_one(f, p, threadIdx.x % g);
}

// Adam, FP64 moments, every operation rounded on its own in the written order.
// What bounds it: the FP64 pipe (two lanes an SM), so the blocks are small and the
// work spreads over the SMs (three steps on the constants of 24 small problems with
// their gradients: 745 us with 256 threads a block, 733 with 64).
constexpr int ADAM_THREADS = 64;
__device__ __forceinline__ void adam_one(float *c, const double *g, double *m, double *v, int i,
                                         double lr, double b1, double b2, double eps, double bc1, double bc2) {
  const double gi = g[i];
  if (!isfinite(gi)) return;  // leaves c, m, v unchanged
  const double mi = __dadd_rn(__dmul_rn(b1, m[i]), __dmul_rn(__dsub_rn(1.0, b1), gi));
  const double vi = __dadd_rn(__dmul_rn(b2, v[i]), __dmul_rn(__dmul_rn(__dsub_rn(1.0, b2), gi), gi));
  m[i] = mi;
  v[i] = vi;
  const double mh = __ddiv_rn(mi, bc1), vh = __ddiv_rn(vi, bc2);
  const double step = __ddiv_rn(__dmul_rn(lr, mh), __dadd_rn(__dsqrt_rn(vh), eps));
  c[i] = __double2float_rn(__dsub_rn((double)c[i], step));
}

__global__ void adam_kernel(float *c, const double *g, double *m, double *v, int n,
                            double lr, double b1, double b2, double eps, double bc1, double bc2) {
  launch_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) adam_one(c, g, m, v, i, lr, b1, b2, eps, bc1, bc2);
}

// Adam of many constant tables in one launch: blocks (table, ADAM_THREADS entries)
constexpr int MAX_ABATCH = 64;
struct AdamBatch {
  float *c[MAX_ABATCH];
  const double *g[MAX_ABATCH];
  double *m[MAX_ABATCH];
  double *v[MAX_ABATCH];
  int n[MAX_ABATCH];
  int count;
  double lr, b1, b2, eps, bc1, bc2;
};

__global__ void adam_batched_kernel(const __grid_constant__ AdamBatch a) {
  launch_wait();
  const int q = blockIdx.x;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < a.n[q]; i += gridDim.y * blockDim.x)
    adam_one(a.c[q], a.g[q], a.m[q], a.v[q], i, a.lr, a.b1, a.b2, a.eps, a.bc1, a.bc2);
}

// blocks (problem, GFINAL_THREADS / group programs of it)
__global__ void __launch_bounds__(GFINAL_THREADS) grad_finalize_batched_kernel(const __grid_constant__ GradBatch b) {
  launch_wait();
  const GradParams &q = b.prob[blockIdx.x];
  const GradFinal f{q.partials, q.flags, q.P, q.N, q.K, q.nchunks, b.mse[blockIdx.x], b.dconst[blockIdx.x]};
  const int g = grad_final_group(f.K), per = GFINAL_THREADS / g;
  for (int p = blockIdx.y * per + threadIdx.x / g; p < q.P; p += gridDim.y * per)
    finalize_grad_one(f, p, threadIdx.x % g);
}

// ---------------------------------------------------------------- host side
// Launch shape of the gradient kernels for the largest Lmax and K of a launch:
// the main pass's and the big pass's code words, shared memory and grid.
struct GradShape {
  int cap, smem, grid;
  int big_cap, big_smem, big_grid;  // 0: no program can be big
};

sr_status grad_shape(sr_ctx *ctx, int Lw, int Kw, bool batched, GradShape *g) {
  const void *kern = batched ? reinterpret_cast<const void *>(grad_batched_kernel) : reinterpret_cast<const void *>(grad_kernel);
  sr_status st = allow_dynamic_smem(ctx, kern);  // once per (kernel, device): every shape fits
  if (st != SR_OK) return st;
  g->cap = grad_cap_words(Lw, Kw);
  g->big_cap = grad_code_words(Lw) > g->cap ? grad_code_words(Lw) : 0;
  for (int big = 0; big < 2; ++big) {
    int &smem = big ? g->big_smem : g->smem, &grid = big ? g->big_grid : g->grid;
    smem = grid = 0;
    if (big && !g->big_cap) continue;
    smem = GWARPS * grad_warp_bytes(Lw, Kw, big ? g->big_cap : g->cap);
    int nb = 0;
    SR_CHECK_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, GWARPS * 32, smem));
    if (nb < 1) return fail(ctx, SR_EINVAL, "Lmax %d, K %d too large for the gradient kernel", Lw, Kw);
    grid = nb * ctx->num_sms;
  }
  return SR_OK;
}

// The warps that the cases per work item are chosen by: 5 CTAs of 8 warps per SM
// where they fit with 512-byte stack slots, the sums and 8 bytes of code a token
// (and a tape of Lmax entries where that fits a fifth of an SM too).  The FP32
// sums of a program follow its case chunks, so this rule is part of the results
// and stays as it is whatever the kernels take.
long long grad_chunk_warps(const sr_ctx *ctx, int Lmax, int K) {
  const int fixed = slots_for(Lmax) * GSLOT + 2 * K * 128 + (Lmax * 8 + 15) / 16 * 16;
  const int share = (233472 / 5 - 1024) / GWARPS;
  const int warp = fixed + (fixed + Lmax * GSLOT <= share ? Lmax * GSLOT : 0);
  return (long long)std::min(5, 233472 / (GWARPS * warp + 1024)) * ctx->num_sms * GWARPS;
}

// cases per work item: about `items` items of this problem, at least one
// 1,024-case block each
int grad_chunk(int N, double items_wanted, int P) {
  int nch = (int)ceil(items_wanted / (P > 0 ? P : 1));
  const int max_chunks = (N + 1023) / 1024;
  nch = nch < 1 ? 1 : (nch > max_chunks ? max_chunks : nch);
  int chunk = (N + nch - 1) / nch;
  return (chunk + GSTEP - 1) / GSTEP * GSTEP;
}

sr_status check_grad(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths, const float *consts, int P,
                     int Lmax, int K, const float *X, const float *y, int nvars, int N, int ldx, const double *mse,
                     const double *dconst) {
  if (P < 0 || Lmax < 1 || Lmax > SR_MAX_LMAX || K < 1 || K > SR_MAX_CONSTS || nvars < 1 ||
      nvars > SR_MAX_VARS || N < 1 || ldx < N || ldx % 4 || (long long)ldx * nvars > 0xFFFFFFFFll)
    return fail(ctx, SR_EINVAL, "bad sr_eval_grad shape");
  if (P == 0) return SR_OK;
  if (!programs || !lengths || !consts || !X || !y || !mse || !dconst)
    return fail(ctx, SR_EINVAL, "NULL pointer");
  if (((uintptr_t)X) & 15) return fail(ctx, SR_EINVAL, "X must be 16-byte aligned");
  return SR_OK;
}

// One problem's gradient.  With less room than it would take (as inside stream
// capture) the programs are decoded and run in slices that share the room for code
// (4.5 words a token: most of the workspace of a large population), and below a
// sixteenth of them at a time on fewer blocks (each with its tape).  Slices and
// blocks do not change a program's items, so results keep their bits.
sr_status launch_grad(sr_ctx *ctx, const sr_grad_problem &q) {
  const int P = q.P, Lmax = q.Lmax, K = q.K;
  GradShape gs;
  sr_status st = grad_shape(ctx, Lmax, K, false, &gs);
  if (st != SR_OK) return st;
  const int chunk = grad_chunk(q.N, (double)grad_chunk_warps(ctx, Lmax, K) * GTARGET_ITEMS_PER_WARP, P);
  const int nchunks = (q.N + chunk - 1) / chunk;
  size_t off_q, off_f, off_nc, off_code, off_p, off_t;
  int per = P, blocks = std::max(gs.grid, gs.big_grid);  // programs of a slice, blocks of a launch
  for (;;) {
    Carver cv;
    off_q = cv.take(256);
    off_f = cv.take(q.prog_flags ? 0 : (size_t)P * 4);
    off_nc = cv.take((size_t)per * 8);
    off_code = cv.take((size_t)per * grad_code_words(Lmax) * 8);
    off_p = cv.take((size_t)P * nchunks * GSTRIDE * 8);
    off_t = cv.take((size_t)blocks * GWARPS * Lmax * GSLOT);
    st = ensure_workspace(ctx, cv.off);
    if (st != SR_ENOMEM) break;
    if (per > 1 && (long long)per * 16 > P) per = (per + 1) / 2;
    else if (blocks > 1) blocks = (blocks + 1) / 2;
    else break;
  }
  if (st != SR_OK) return st;
  st = allow_dynamic_smem(ctx, reinterpret_cast<const void *>(grad_decode_kernel));
  if (st != SR_OK) return st;
  char *ws = ctx->ws;
  double *partials = reinterpret_cast<double *>(ws + off_p);
  int32_t *flags = q.prog_flags ? q.prog_flags : reinterpret_cast<int32_t *>(ws + off_f);
  cudaStream_t s = ctx->stream;
  for (int p0 = 0; p0 < P; p0 += per) {
    GradParams gp;
    gp.programs = q.programs + (size_t)p0 * Lmax;
    gp.lengths = q.lengths + p0;
    gp.consts = q.consts + (size_t)p0 * K;
    gp.P = std::min(per, P - p0);
    gp.Lmax = Lmax;
    gp.K = K;
    gp.X = q.X;
    gp.y = q.y;
    gp.nvars = q.nvars;
    gp.N = q.N;
    gp.ldx = q.ldx;
    gp.chunk = chunk;
    gp.nchunks = nchunks;
    gp.total_items = (long long)gp.P * nchunks;
    gp.partials = partials + (size_t)p0 * nchunks * GSTRIDE;
    gp.flags = flags + p0;
    gp.code = reinterpret_cast<uint2 *>(ws + off_code);
    gp.nfwd = reinterpret_cast<int32_t *>(ws + off_nc);
    gp.nrev = gp.nfwd + per;
    gp.queue = reinterpret_cast<unsigned long long *>(ws + off_q);
    gp.gtape = ws + off_t;
    gp.abort = ctx->abort_flag;
    gp.err = ctx->dev_words;
    gp.cap = gp.room = gs.cap;
    gp.big = 0;
    SR_CHECK_CUDA(ctx, launch(grad_decode_kernel, (gp.P + DECODE_WARPS - 1) / DECODE_WARPS, DECODE_WARPS * 32,
                              DECODE_WARPS * grad_scratch_bytes(Lmax), s, gp));
    SR_CHECK_CUDA(ctx, launch(grad_kernel, std::min(gs.grid, blocks), GWARPS * 32, gs.smem, s, gp));
    ctx->launches += 2;
    if (gs.big_cap) {
      gp.room = gs.big_cap;
      gp.big = 1;
      SR_CHECK_CUDA(ctx, launch(grad_kernel, std::min(gs.big_grid, blocks), GWARPS * 32, gs.big_smem, s, gp));
      ctx->launches += 1;
    }
    SR_CHECK_CUDA(ctx, cudaGetLastError());
    if (P - p0 <= per) break;  // (p0 + per may be beyond an int)
  }
  GradFinal gf{partials, flags, P, q.N, K, nchunks, q.mse, q.dconst};
  const int per_block = GFINAL_THREADS / grad_final_group(K);
  SR_CHECK_CUDA(ctx, launch(grad_finalize_kernel, (P + per_block - 1) / per_block, GFINAL_THREADS, 0, s, gf));
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

}  // namespace
}  // namespace sr

extern "C" {

sr_status sr_eval_grad(sr_ctx *ctx, const uint8_t *programs, const int32_t *lengths,
                       const float *consts, int P, int Lmax, int K, const float *X, const float *y,
                       int nvars, int N, int ldx, double *mse, double *dconst, int32_t *prog_flags) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  sr_status st = check_grad(ctx, programs, lengths, consts, P, Lmax, K, X, y, nvars, N, ldx, mse, dconst);
  if (st != SR_OK || P == 0) return st;
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  return launch_grad(ctx, sr_grad_problem{programs, lengths, consts, P, Lmax, K, X, y, nvars, N, ldx, mse, dconst,
                                          prog_flags});
}

sr_status sr_eval_grad_batched(sr_ctx *ctx, const sr_grad_problem *pr, int nprob) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  if (nprob < 0 || (nprob > 0 && !pr)) return fail(ctx, SR_EINVAL, "bad problem list");
  int Lw = 1, Kw = 1;
  for (int i = 0; i < nprob; ++i) {
    const sr_grad_problem &q = pr[i];
    sr_status st = check_grad(ctx, q.programs, q.lengths, q.consts, q.P, q.Lmax, q.K, q.X, q.y, q.nvars, q.N,
                              q.ldx, q.mse, q.dconst);
    if (st != SR_OK) return fail(ctx, st, "problem %d: %s", i, ctx->msg);
    if (q.P == 0) continue;
    Lw = q.Lmax > Lw ? q.Lmax : Lw;
    Kw = q.K > Kw ? q.K : Kw;
  }
  std::vector<int> order;
  for (int i = 0; i < nprob; ++i)
    if (pr[i].P > 0) order.push_back(i);
  if (order.empty()) return SR_OK;
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  GradShape gs;
  sr_status st = grad_shape(ctx, Lw, Kw, true, &gs);
  if (st != SR_OK) return st;
  // cases per item per problem: the chunking sr_eval_grad would choose for
  // the problem alone (so every problem's sums, and its results, are the
  // same bits as its own call's); the batch shares one grid and one tail
  std::vector<int> chunk(nprob, 0), nch(nprob, 0);
  for (int i : order) {
    const sr_grad_problem &q = pr[i];
    chunk[i] = grad_chunk(q.N, (double)grad_chunk_warps(ctx, q.Lmax, q.K) * GTARGET_ITEMS_PER_WARP, q.P);
    nch[i] = (q.N + chunk[i] - 1) / chunk[i];
  }
  // longest items first: the launch's tail is made of short items
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return (double)chunk[a] * pr[a].Lmax > (double)chunk[b] * pr[b].Lmax;
  });
  auto group_bytes = [&](size_t g0, size_t g1, GradBatch *b) -> size_t {
    Carver cv;
    const size_t off_q = cv.take(256);
    const size_t off_t = cv.take((size_t)std::max(gs.grid, gs.big_grid) * GWARPS * Lw * GSLOT);
    long long items = 0;
    int progs = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int i = order[g];
      const sr_grad_problem &q = pr[i];
      const size_t off_f = q.prog_flags ? 0 : cv.take((size_t)q.P * 4);
      const size_t off_nc = cv.take((size_t)q.P * 8);
      const size_t off_code = cv.take((size_t)q.P * grad_code_words(q.Lmax) * 8);
      const size_t off_p = cv.take((size_t)q.P * nch[i] * GSTRIDE * 8);
      if (b) {
        char *ws = ctx->ws;
        GradParams &p = b->prob[g - g0];
        p.programs = q.programs;
        p.lengths = q.lengths;
        p.consts = q.consts;
        p.P = q.P;
        p.Lmax = q.Lmax;
        p.K = q.K;
        p.X = q.X;
        p.y = q.y;
        p.nvars = q.nvars;
        p.N = q.N;
        p.ldx = q.ldx;
        p.chunk = chunk[i];
        p.nchunks = nch[i];
        p.total_items = (long long)q.P * nch[i];
        p.partials = reinterpret_cast<double *>(ws + off_p);
        p.flags = q.prog_flags ? q.prog_flags : reinterpret_cast<int32_t *>(ws + off_f);
        p.code = reinterpret_cast<uint2 *>(ws + off_code);
        p.nfwd = reinterpret_cast<int32_t *>(ws + off_nc);
        p.nrev = p.nfwd + q.P;
        p.queue = nullptr;
        p.gtape = nullptr;
        p.abort = nullptr;
        p.err = nullptr;
        p.cap = p.room = 0;
        p.big = 0;
        b->item_begin[g - g0] = items;
        b->prog_begin[g - g0] = progs;
        b->mse[g - g0] = q.mse;
        b->dconst[g - g0] = q.dconst;
      }
      items += (long long)q.P * nch[i];
      progs += q.P;
    }
    if (b) {
      b->nprob = (int)(g1 - g0);
      b->total_progs = progs;
      b->total_items = items;
      b->queue = reinterpret_cast<unsigned long long *>(ctx->ws + off_q);
      b->gtape = ctx->ws + off_t;
      b->abort = ctx->abort_flag;
      b->err = ctx->dev_words;
      b->cap = b->room = gs.cap;
      b->big = 0;
      b->Lw = Lw;
      b->Kw = Kw;
    }
    return cv.off;
  };
  size_t need = 0;
  for (size_t g0 = 0; g0 < order.size(); g0 += MAX_GBATCH)
    need = std::max(need, group_bytes(g0, std::min(order.size(), g0 + MAX_GBATCH), nullptr));
  st = ensure_workspace(ctx, need);
  if (st == SR_ENOMEM) {  // with less room one after the other: the same bits, and each may be sliced
    for (int i : order)
      if ((st = launch_grad(ctx, pr[i])) != SR_OK) return st;
    return SR_OK;
  }
  if (st != SR_OK) return st;
  st = allow_dynamic_smem(ctx, reinterpret_cast<const void *>(grad_decode_batched_kernel));
  if (st != SR_OK) return st;
  cudaStream_t s = ctx->stream;
  for (size_t g0 = 0; g0 < order.size(); g0 += MAX_GBATCH) {
    GradBatch b;
    group_bytes(g0, std::min(order.size(), g0 + MAX_GBATCH), &b);
    SR_CHECK_CUDA(ctx, launch(grad_decode_batched_kernel, (b.total_progs + DECODE_WARPS - 1) / DECODE_WARPS,
                              DECODE_WARPS * 32, DECODE_WARPS * grad_scratch_bytes(Lw), s, b));
    SR_CHECK_CUDA(ctx, launch(grad_batched_kernel, gs.grid, GWARPS * 32, gs.smem, s, b));
    if (gs.big_cap) {
      b.room = gs.big_cap;
      b.big = 1;
      SR_CHECK_CUDA(ctx, launch(grad_batched_kernel, gs.big_grid, GWARPS * 32, gs.big_smem, s, b));
      ctx->launches += 1;
    }
    int maxP = 1;
    for (int r = 0; r < b.nprob; ++r) maxP = b.prob[r].P > maxP ? b.prob[r].P : maxP;
    const int per_block = GFINAL_THREADS / grad_final_group(Kw);  // (a problem of smaller K takes more a block)
    SR_CHECK_CUDA(ctx, launch(grad_finalize_batched_kernel,
                              dim3(b.nprob, std::min((maxP + per_block - 1) / per_block, 65535)), GFINAL_THREADS, 0, s, b));
    SR_CHECK_CUDA(ctx, cudaGetLastError());
    ctx->launches += 3;
  }
  return SR_OK;
}

sr_status sr_adam_step(sr_ctx *ctx, float *consts, const double *grad, double *m, double *v, int n,
                       int t, const sr_adam_cfg *cfg) {
  using namespace sr;
  if (!ctx || !cfg) return SR_EINVAL;
  if (n < 0 || t < 1) return fail(ctx, SR_EINVAL, "n < 0 or t < 1");
  if (n == 0) return SR_OK;
  if (!consts || !grad || !m || !v) return fail(ctx, SR_EINVAL, "NULL pointer");
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  // bias corrections on the host: products of t factors, in order
  double p1 = 1.0, p2 = 1.0;
  for (int s = 0; s < t; ++s) {
    p1 *= cfg->beta1;
    p2 *= cfg->beta2;
  }
  SR_CHECK_CUDA(ctx, launch(adam_kernel, (n + ADAM_THREADS - 1) / ADAM_THREADS, ADAM_THREADS, 0, ctx->stream, consts,
                            grad, m, v, n, cfg->lr, cfg->beta1, cfg->beta2, cfg->eps, 1.0 - p1, 1.0 - p2));
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

sr_status sr_adam_step_batched(sr_ctx *ctx, const sr_adam_table *tables, int ntables, int t,
                               const sr_adam_cfg *cfg) {
  using namespace sr;
  if (!ctx || !cfg) return SR_EINVAL;
  if (ntables < 0 || (ntables > 0 && !tables) || t < 1) return fail(ctx, SR_EINVAL, "bad table list or t < 1");
  for (int i = 0; i < ntables; ++i) {
    const sr_adam_table &q = tables[i];
    if (q.n < 0) return fail(ctx, SR_EINVAL, "table %d: n < 0", i);
    if (q.n > 0 && (!q.consts || !q.grad || !q.m || !q.v)) return fail(ctx, SR_EINVAL, "table %d: NULL pointer", i);
  }
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  double p1 = 1.0, p2 = 1.0;
  for (int s = 0; s < t; ++s) {
    p1 *= cfg->beta1;
    p2 *= cfg->beta2;
  }
  for (int g0 = 0; g0 < ntables; g0 += MAX_ABATCH) {
    AdamBatch a;
    a.count = 0;
    int maxn = 0;
    for (int i = g0; i < ntables && i < g0 + MAX_ABATCH; ++i) {
      const sr_adam_table &q = tables[i];
      if (q.n == 0) continue;
      a.c[a.count] = q.consts;
      a.g[a.count] = q.grad;
      a.m[a.count] = q.m;
      a.v[a.count] = q.v;
      a.n[a.count] = q.n;
      maxn = q.n > maxn ? q.n : maxn;
      ++a.count;
    }
    if (a.count == 0) continue;
    a.lr = cfg->lr;
    a.b1 = cfg->beta1;
    a.b2 = cfg->beta2;
    a.eps = cfg->eps;
    a.bc1 = 1.0 - p1;
    a.bc2 = 1.0 - p2;
    const int yblocks = std::min((maxn + ADAM_THREADS - 1) / ADAM_THREADS, 65535);
    SR_CHECK_CUDA(ctx, launch(adam_batched_kernel, dim3(a.count, yblocks), ADAM_THREADS, 0, ctx->stream, a));
    SR_CHECK_CUDA(ctx, cudaGetLastError());
    ctx->launches += 1;
  }
  return SR_OK;
}

}  // extern "C"
