// sr_interp.cuh -- the scheduled instruction stream shared by the evaluation
// kernels (sr_eval.cu) and the adjoint kernel (sr_grad.cu).
//
// A program (RPN, paper Sec. 2.1.4) is decoded once per call by a pre-pass, a
// warp per program (sr_decode.cuh): validation, then the expression tree is
// rescheduled Sethi-Ullman style -- at every binary node the child that needs
// more stack is evaluated first, with a reversed opcode keeping a - b and
// a / b exact when the right child goes first.  The number of live values is
// then at most floor(log2(leaves)) + 1: 9 for 512 tokens, so 8 stack slots
// below the top always suffice.  A terminal evaluated second is fused into
// its binary operator ("top = top op x_j").  Values are bit-identical to
// plain left-to-right evaluation: every operator sees the same operands.
#pragma once

#include "sr_common.cuh"

namespace sr {

// stack slots below the top register (see above)
constexpr int DSM = 8;
static_assert(SR_MAX_LMAX <= 512, "8 slots cover programs of up to 512 tokens");

// The slots programs of up to Lmax tokens can need: floor(log2(leaves)) with
// leaves <= (Lmax + 1) / 2.  Kernels size their shared stack by it (6 slots
// for Lmax = 128 instead of 8 -- more warps per SM).
__host__ __device__ constexpr int slots_for(int Lmax) {
  int leaves = (Lmax + 1) / 2, s = 0;
  while ((2 << s) <= leaves) ++s;
  return s < 1 ? 1 : (s > DSM ? DSM : s);
}

// ---------------------------------------------------------------- operators (FP32)
// The protected quotient.  The quotient itself comes from PTX div.full.f32:
// full range, at most 2 ulp off (subnormal results included) -- within the
// 2-ulp allowance the oracle's enclosure gives every operation.  Computed
// whatever b is and selected, so the vector loops stay branch-free.
// Measured on the paper-shaped population: +12 % over the IEEE quotient; a redo of
// the subnormal results by the IEEE quotient cost back 11 %.
__device__ __forceinline__ float op_div(float a, float b) {
  float q;
  asm("div.full.f32 %0, %1, %2;" : "=f"(q) : "f"(a), "f"(b));
  // |b| < 1e-3f in FP32 is exactly "|b| <= 1e-3" for FP32 values of b
  return fabsf(b) < 1e-3f ? 1.0f : q;
}
__device__ __forceinline__ float op_log(float x) {
  return fabsf(x) < 1e-3f ? 0.0f : logf(fabsf(x));
}
__device__ __forceinline__ float op_exp(float x) {
  x = x > 80.0f ? 80.0f : (x < -80.0f ? -80.0f : x);  // NaN passes through
  return expf(x);
}
__device__ __forceinline__ float f_sqrt(float x) { return sqrtf(fabsf(x)); }

// sinf / cosf carry a long path for large arguments; keep one out-of-line
// copy of it and let the inlined copies assume a moderate argument (NaN and
// +-inf also take the out-of-line call)
static __device__ __noinline__ float sin_wide(float x) { return sinf(x); }
static __device__ __noinline__ float cos_wide(float x) { return cosf(x); }
__device__ __forceinline__ float f_sin(float x) {
  if (!(fabsf(x) <= 4.0e4f)) return sin_wide(x);
  __builtin_assume(fabsf(x) <= 4.0e4f);
  return sinf(x);
}
__device__ __forceinline__ float f_cos(float x) {
  if (!(fabsf(x) <= 4.0e4f)) return cos_wide(x);
  __builtin_assume(fabsf(x) <= 4.0e4f);
  return cosf(x);
}
static __device__ __noinline__ float tan_wide(float x) { return tanf(x); }
__device__ __forceinline__ float f_tan(float x) {
  if (!(fabsf(x) <= 4.0e4f)) return tan_wide(x);
  __builtin_assume(fabsf(x) <= 4.0e4f);
  return tanf(x);
}
// The rest of Table 1: 1/x protected like division; tan, asin, acos, atan,
// tanh as the FP32 library computes them (asin / acos outside [-1, 1] give
// NaN: a non-real result, which the NaN-aware scores of Eq. 2 / Eq. 3 take
// as an invalid output and MSE / 1 - r^2 as the worst fitness).
__device__ __forceinline__ float op_inv(float x) { return op_div(1.0f, x); }
__device__ __forceinline__ float f_asin(float x) { return asinf(x); }
__device__ __forceinline__ float f_acos(float x) { return acosf(x); }
__device__ __forceinline__ float f_atan(float x) { return atanf(x); }
__device__ __forceinline__ float f_tanh(float x) { return tanhf(x); }


// Instruction (uint2):
//   x bits 0..7   opcode
//   x bits 8..23  byte offset of the stack slot it pushes to / pops from
//   y             operand: FP32 bits of c_k, or the row offset j * ldx of x_j
enum Op : uint32_t {
  OP_LDV = 0,   // top = x_j                        (stack empty)
  OP_LDC,       // top = c_k
  OP_PUSHV,     // stack[slot] = top; top = x_j
  OP_PUSHC,     // stack[slot] = top; top = c_k
  OP_ADD,       // top = stack[slot] op top         (left operand evaluated first)
  OP_SUB,
  OP_MUL,
  OP_DIV,
  OP_RSUB,      // top = top - stack[slot]          (right operand evaluated first)
  OP_RDIV,      // top = top / stack[slot]
  OP_SIN,       // top = f(top)
  OP_COS,
  OP_EXP,
  OP_LOG,
  OP_SQRT,
  OP_SQ,
  OP_INV,       // 1 / top (protected as /)
  OP_TAN,
  OP_ASIN,
  OP_ACOS,
  OP_ATAN,
  OP_TANH,
  OP_VADD,      // top = top op x_j   (terminal right operand, evaluated second)
  OP_VSUB,
  OP_VMUL,
  OP_VDIV,
  OP_VRSUB,     // top = x_j - top    (terminal left operand, evaluated second)
  OP_VRDIV,     // top = x_j / top
  OP_CADD,      // top = top op c_k
  OP_CSUB,
  OP_CMUL,
  OP_CDIV,
  OP_CRSUB,     // top = c_k - top
  OP_CRDIV,     // top = c_k / top
  OP_END,       // the program is done (appended by the evaluation kernels)
};

// ncode[p] holds the instruction count in its low 16 bits; NCODE_EXT is set
// when the program uses one of 1/x, tan, asin, acos, atan, tanh, so that
// the kernels can run those programs in a separate copy of their loop and
// keep the loop of the base operators free of the extra call site.
constexpr int NCODE_EXT = 1 << 30;
// NCODE_DEEP is set when the program needs more stack slots than the
// decoder's cap_slots (or more words than its cap_words): the evaluation kernels
// give most programs a few slots (more warps fit on an SM) and run the rare deeper
// ones in a separate pass.
constexpr int NCODE_DEEP = 1 << 29;
__device__ __forceinline__ int ncode_count(int v) { return v & 0xffff; }
__device__ __forceinline__ bool ncode_ext(int v) { return (v & NCODE_EXT) != 0; }
__device__ __forceinline__ bool ncode_deep(int v) { return (v & NCODE_DEEP) != 0; }

struct DecodeArgs {
  const uint8_t *programs;  // [P][Lmax]
  const int32_t *lengths;
  const float *consts;      // [P][K]
  int Lmax, K, nvars;
  long long ldx;
  int slot_bytes;           // bytes between consecutive stack slots of a warp
  uint2 *code;              // [P][Lmax] out
  int32_t *ncode;           // [P] out
  int32_t *flags;           // [P] out
  int max_slots;            // stack slots the kernel provides (<= DSM)
  int cap_slots;            // programs that need more than this get NCODE_DEEP (<= max_slots),
  int cap_words;            // and so do those with more words than this, their end marker counted
  unsigned long long *ext_note, *deep_note;  // set to 1 when some program has NCODE_EXT / NCODE_DEEP
  // >= 1: a unary operator applied to a variable, u(x_j),
  // reads row xform_row(nvars, u, j) of the variable table instead (the
  // table's first nvars rows are X); with 2, also a base unary operator
  // applied to a base u(x_j), u(v(x_j)), reads row xform_row2(nvars, u, v, j).
  // The decoder marks in xneed[row - nvars] each row some program reads, and
  // a kernel fills those rows before the evaluation.  ldx is then the
  // table's row stride.
  int xform = 0;
  uint8_t *xneed = nullptr;
};

// The variable table of an evaluation with transforms: X's nvars rows, then
// u(x_j) for the twelve unary operators, then (depth 2) u(v(x_j)) for the
// 36 pairs of the six base ones (sin cos exp log sqrt sq).
constexpr int XFORM_BASE = TOK_SQ - TOK_SIN + 1;
__host__ __device__ inline int xform_row(int nvars, int u, int j) { return nvars + (u - TOK_SIN) * nvars + j; }
__host__ __device__ inline int xform_row2(int nvars, int u, int v, int j) {
  return nvars * (1 + UNARY_ALL) + ((u - TOK_SIN) * XFORM_BASE + (v - TOK_SIN)) * nvars + j;
}
__host__ __device__ inline int xform_rows(int nvars, int depth) {
  return nvars * (1 + UNARY_ALL + (depth > 1 ? XFORM_BASE * XFORM_BASE : 0));
}

// The FP32 value of an operator node whose operands are constants, by the
// same functions the interpreter applies to every case, so that a folded
// subtree gives the bits its per-case evaluation gives.  Each operation is
// one function call: nothing is contracted across operations.
static __device__ __noinline__ float fold_op(int v, float a, float b) {
  switch (v) {
    case TOK_ADD: return __fadd_rn(a, b);
    case TOK_SUB: return __fsub_rn(a, b);
    case TOK_MUL: return __fmul_rn(a, b);
    case TOK_DIV: return op_div(a, b);
    case TOK_SIN: return f_sin(a);
    case TOK_COS: return f_cos(a);
    case TOK_EXP: return op_exp(a);
    case TOK_LOG: return op_log(a);
    case TOK_SQRT: return f_sqrt(a);
    case TOK_SQ: return __fmul_rn(a, a);
    case TOK_INV: return op_inv(a);
    case TOK_TAN: return f_tan(a);
    case TOK_ASIN: return f_asin(a);
    case TOK_ACOS: return f_acos(a);
    case TOK_ATAN: return f_atan(a);
    default: return f_tanh(a);
  }
}

constexpr int DECODE_WARPS = 4;  // warps (programs) per block of the decode kernels

}  // namespace sr
