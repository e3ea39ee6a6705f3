// sr_vm.cuh -- the case-parallel interpreter of the evaluation kernels: one
// warp runs one decoded program on 256 cases, 8 per lane.
//
// What bounds it: issue slots.  A node is a few instructions of arithmetic and
// as many again of dispatch, so the loop is built to issue few:
//   - the 8 cases of a lane are four FP32 pairs, and + - * and the square run on
//     the packed instructions (add / sub / mul .f32x2, each half rounded as the
//     scalar instruction rounds it);
//   - the loads, stack moves and packed operators run in one PTX loop that
//     branches through a table on the opcode instead of a C++ switch;
//   - a row of X is read with one 256-bit load per lane;
//   - sin, cos, exp, log, sqrt and the quotient leave that loop, run inline
//     instead of as calls, and enter it again.  Their range tests are made once
//     for the lane's 8 values.
// Instructions executed (the profiler's counter) per node and 256 cases, before ->
// then: x_j op 33 -> 14, square 27 -> 11, (push, x_i op x_j, op) 98 -> 42, quotient
// 137 -> 69, sin 253 -> 202, log 264 -> 248, exp 120 ->
// 105, sqrt 119 -> 113 (5 CTAs per SM).
// Evaluation of 8,192 programs of <= 256 tokens x 131,072 cases: 33.0 -> 24.9 ms.
// Every value keeps its bits: each operator sees the operands it saw before and
// rounds once.
#pragma once

#include "sr_interp.cuh"

namespace sr {
namespace {

constexpr int CPL = 8;                    // cases per lane
constexpr int STEP = 32 * CPL;            // cases per warp step
constexpr int SLOT_BYTES = 32 * CPL * 4;  // one stack slot of a warp: [2][32 lanes] float4

typedef unsigned long long pair_t;  // two FP32 values, the lower case in the lower half
struct V8 {
  pair_t p[4];
};

__device__ __forceinline__ pair_t pack(float lo, float hi) {
  pair_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ V8 splat8(float c) {
  const pair_t v = pack(c, c);
  return V8{{v, v, v, v}};
}
__device__ __forceinline__ void unpack8(const V8 &v, float (&t)[CPL]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) asm("mov.b64 {%0, %1}, %2;" : "=f"(t[2 * i]), "=f"(t[2 * i + 1]) : "l"(v.p[i]));
}
__device__ __forceinline__ V8 pack8(const float (&t)[CPL]) {
  return V8{{pack(t[0], t[1]), pack(t[2], t[3]), pack(t[4], t[5]), pack(t[6], t[7])}};
}

// ---------------------------------------------------------------- library operators on 8 values
// f on every value, W of them in flight: W < 8 keeps one copy of the body and
// rotates the values through it (an indexed array would live in local memory).
// Wide copies hide latency, but the bodies of all operators have to stay in the
// instruction cache together.
template <int W, typename F>
__device__ __forceinline__ V8 map8(const V8 &v, F f) {
  float t[CPL];
  unpack8(v, t);
  if constexpr (W == CPL) {
#pragma unroll
    for (int i = 0; i < CPL; ++i) t[i] = f(t[i]);
  } else {
#pragma unroll 1
    for (int i = 0; i < CPL; i += W) {
      float r[W];
#pragma unroll
      for (int j = 0; j < W; ++j) r[j] = f(t[j]);
#pragma unroll
      for (int j = 0; j < CPL - W; ++j) t[j] = t[j + W];
#pragma unroll
      for (int j = 0; j < W; ++j) t[CPL - W + j] = r[j];
    }
  }
  return pack8(t);
}
template <int W, typename F>
__device__ __forceinline__ V8 zip8(const V8 &a, const V8 &b, F f) {
  float t[CPL], u[CPL];
  unpack8(a, t);
  unpack8(b, u);
  if constexpr (W == CPL) {
#pragma unroll
    for (int i = 0; i < CPL; ++i) t[i] = f(t[i], u[i]);
  } else {
#pragma unroll 1
    for (int i = 0; i < CPL; i += W) {
      float r[W];
#pragma unroll
      for (int j = 0; j < W; ++j) r[j] = f(t[j], u[j]);
#pragma unroll
      for (int j = 0; j < CPL - W; ++j) t[j] = t[j + W], u[j] = u[j + W];
#pragma unroll
      for (int j = 0; j < W; ++j) t[CPL - W + j] = r[j];
    }
  }
  return pack8(t);
}

// sin and cos: the library's path for moderate arguments (|x| <= 4e4) runs inline and is
// told that its argument is one; what is told holds for every value it gets.
// In the base copy a warp votes on its arguments first, one test for eight values; one
// with an argument beyond, or NaN, calls the whole function on each value, out of line.
// In the EXT copy, where NaN is common (asin and acos outside [-1, 1]), each value
// that is not moderate is replaced by 0 there, passed through instead of the result and
// recognised afterwards by its magnitude (a result is at most 1).  That / the vote, us:
// 1,500 programs x 100,003 cases 2,051 / 1,968, 8,192 x 131,072 25,400 / 24,805, 64 small
// problems 479 / 467; Eq. 2 with 16 operators 2,045 / 2,110 by the vote in the EXT copy too.
constexpr float NEAR = 4.0e4f;
template <bool COS>
struct SinCosNear {  // |x| <= NEAR
  __device__ __forceinline__ float operator()(float x) const {
    __builtin_assume(fabsf(x) <= NEAR);
    return COS ? cosf(x) : sinf(x);
  }
};
template <bool COS>
struct SinCosOrArg {  // of a moderate x, else x
  __device__ __forceinline__ float operator()(float x) const {
    const bool near = fabsf(x) <= NEAR;
    const float r = SinCosNear<COS>()(near ? x : 0.0f);
    return near ? r : x;
  }
};
template <bool COS>
struct SinCosWide { __device__ __forceinline__ float operator()(float x) const { return COS ? cos_wide(x) : sin_wide(x); } };
template <bool COS>
struct SinCosFar { __device__ __forceinline__ float operator()(float x) const { return fabsf(x) > 2.0f ? SinCosWide<COS>()(x) : x; } };
template <bool COS>
__device__ __noinline__ V8 sincos8_wide(V8 v) { return map8<1>(v, SinCosWide<COS>()); }
template <bool COS>
__device__ __noinline__ V8 sincos8_far(V8 v) { return map8<1>(v, SinCosFar<COS>()); }
// some |value| of the warp is beyond `limit`, or NaN
__device__ __forceinline__ bool any_beyond(const V8 &v, float limit) {
  float t[CPL];
  unpack8(v, t);
  bool ok = true;
#pragma unroll
  for (int i = 0; i < CPL; ++i) ok = ok & (fabsf(t[i]) <= limit);
  return __any_sync(FULL, !ok);
}
// some |value| of the warp is beyond any sine (a NaN argument has given NaN)
__device__ __forceinline__ bool any_far(const V8 &v) {
  float t[CPL];
  unpack8(v, t);
  const float m = fmaxf(fmaxf(fmaxf(fabsf(t[0]), fabsf(t[1])), fmaxf(fabsf(t[2]), fabsf(t[3]))),
                        fmaxf(fmaxf(fabsf(t[4]), fabsf(t[5])), fmaxf(fabsf(t[6]), fabsf(t[7]))));
  return __any_sync(FULL, m > 2.0f);
}
template <bool COS, bool EXT, int W>
__device__ __forceinline__ V8 sincos8(V8 v) {
  if (EXT) {
    v = map8<W>(v, SinCosOrArg<COS>());
    if (any_far(v)) v = sincos8_far<COS>(v);
  } else if (any_beyond(v, NEAR)) {
    v = sincos8_wide<COS>(v);
  } else {
    v = map8<W>(v, SinCosNear<COS>());
  }
  return v;
}
// op_exp with its clamp in two instructions (NaN passes through both)
struct Exp {
  __device__ __forceinline__ float operator()(float x) const {
    asm("min.NaN.f32 %0, %0, 0f42A00000;\n\tmax.NaN.f32 %0, %0, 0fC2A00000;" : "+f"(x));  // 80, -80
    return expf(x);
  }
};
struct Log { __device__ __forceinline__ float operator()(float x) const { return op_log(x); } };
struct Sqrt { __device__ __forceinline__ float operator()(float x) const { return f_sqrt(x); } };
struct Inv { __device__ __forceinline__ float operator()(float x) const { return op_inv(x); } };
struct Tan { __device__ __forceinline__ float operator()(float x) const { return f_tan(x); } };
struct Asin { __device__ __forceinline__ float operator()(float x) const { return f_asin(x); } };
struct Acos { __device__ __forceinline__ float operator()(float x) const { return f_acos(x); } };
struct Atan { __device__ __forceinline__ float operator()(float x) const { return f_atan(x); } };
struct Tanh { __device__ __forceinline__ float operator()(float x) const { return f_tanh(x); } };
struct Div { __device__ __forceinline__ float operator()(float a, float b) const { return op_div(a, b); } };
// The quotient where no |b| of the warp is beyond DIV_NEAR, just below 2^126: a times
// the approximate reciprocal of b, the form in which the PTX manual defines
// div.approx.f32, a * (1/b), at most 2 ulp off for |b| in [2^-126, 2^126].  The
// reciprocal is the instruction rcp.approx.ftz.f32: |b| < 1e-3 is protected, so
// neither b nor 1/b is subnormal and nothing is flushed, and a and the product keep
// their subnormals.  Its bits are op_div's, by test over every binade of b (all
// mantissas of each with four a tried once).  1,500 programs x 100,003 cases: 2,048 us;
// with div.approx.f32 itself, which covers subnormal b as well, 2,273.
constexpr float DIV_NEAR = 8.5e37f;
struct DivNear {
  __device__ __forceinline__ float operator()(float a, float b) const {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
    return fabsf(b) < 1e-3f ? 1.0f : __fmul_rn(a, r);
  }
};
__device__ __noinline__ V8 div8_wide(V8 a, V8 b) { return zip8<1>(a, b, Div()); }

// 1/x, tan, asin, acos, atan, tanh (EXT programs)
__device__ __noinline__ V8 ext8(uint32_t op, V8 v) {
  switch (op) {
    case OP_INV: return map8<2>(v, Inv());
    case OP_TAN: return map8<2>(v, Tan());
    case OP_ASIN: return map8<2>(v, Asin());
    case OP_ACOS: return map8<2>(v, Acos());
    case OP_ATAN: return map8<2>(v, Atan());
    default: return map8<2>(v, Tanh());
  }
}

// ---------------------------------------------------------------- the core loop
// Operands: %0-%3 T (top of stack), %4-%7 X (the other operand of an operator
// that leaves the loop), %8 address of the next instruction, %9 opcode left
// with, %10 this lane's entry of stack slot 0, %11 this lane's cases of row 0,
// %12 their second half where rows are read by two 128-bit loads.
// clang-format off
#define SR_FETCH \
  "ld.shared.v2.b32 {wx, wy}, [%8];\n\tadd.u32 %8, %8, 8;\n\tand.b32 %9, wx, 255;\n\t" \
  "brx.idx.uni %9, TABLE;\n\t"
#define SR_LDX_WIDE \
  "mad.wide.u32 a, wy, 4, %11;\n\tld.global.v4.b64 {%4, %5, %6, %7}, [a];\n\t"
#define SR_LDT_WIDE \
  "mad.wide.u32 a, wy, 4, %11;\n\tld.global.v4.b64 {%0, %1, %2, %3}, [a];\n\t"
#define SR_LDX_HALVES \
  "mad.wide.u32 a, wy, 4, %11;\n\tld.global.v2.b64 {%4, %5}, [a];\n\t" \
  "mad.wide.u32 a, wy, 4, %12;\n\tld.global.v2.b64 {%6, %7}, [a];\n\t"
#define SR_LDT_HALVES \
  "mad.wide.u32 a, wy, 4, %11;\n\tld.global.v2.b64 {%0, %1}, [a];\n\t" \
  "mad.wide.u32 a, wy, 4, %12;\n\tld.global.v2.b64 {%2, %3}, [a];\n\t"
#define SR_SLOT "shr.u32 s, wx, 8;\n\tadd.u32 s, s, %10;\n\t"
#define SR_LDS SR_SLOT "ld.shared.v2.b64 {%4, %5}, [s];\n\tld.shared.v2.b64 {%6, %7}, [s + 512];\n\t"
#define SR_STS SR_SLOT "st.shared.v2.b64 [s], {%0, %1};\n\tst.shared.v2.b64 [s + 512], {%2, %3};\n\t"
#define SR_SPLAT(d0, d1, d2, d3) \
  "mov.b64 " d0 ", {wy, wy};\n\tmov.b64 " d1 ", " d0 ";\n\tmov.b64 " d2 ", " d0 ";\n\tmov.b64 " d3 ", " d0 ";\n\t"
#define SR_TX(op, NEXT_OP) /* T = T op X */ \
  op ".rn.f32x2 %0, %0, %4;\n\t" op ".rn.f32x2 %1, %1, %5;\n\t" \
  op ".rn.f32x2 %2, %2, %6;\n\t" op ".rn.f32x2 %3, %3, %7;\n\t" NEXT_OP
#define SR_XT(op, NEXT_OP) /* T = X op T */ \
  op ".rn.f32x2 %0, %4, %0;\n\t" op ".rn.f32x2 %1, %5, %1;\n\t" \
  op ".rn.f32x2 %2, %6, %2;\n\t" op ".rn.f32x2 %3, %7, %3;\n\t" NEXT_OP
#define SR_TC(op, NEXT_OP) /* T = T op constant */ "mov.b64 c, {wy, wy};\n\t" \
  op ".rn.f32x2 %0, %0, c;\n\t" op ".rn.f32x2 %1, %1, c;\n\t" \
  op ".rn.f32x2 %2, %2, c;\n\t" op ".rn.f32x2 %3, %3, c;\n\t" NEXT_OP
#define SR_CT(op, NEXT_OP) /* T = constant op T */ "mov.b64 c, {wy, wy};\n\t" \
  op ".rn.f32x2 %0, c, %0;\n\t" op ".rn.f32x2 %1, c, %1;\n\t" \
  op ".rn.f32x2 %2, c, %2;\n\t" op ".rn.f32x2 %3, c, %3;\n\t" NEXT_OP
// The quotients leave with their operand in X, as OP_VDIV (T / X) or OP_VRDIV (X / T).
#define SR_JUMP "bra NEXT;\n\t"
#define SR_CORE(LDX, LDT, NEXT_OP) \
  "{\n\t.reg .b32 wx, wy, s;\n\t.reg .b64 a, c;\n\t" \
  "TABLE: .branchtargets LDV, LDC, PUSHV, PUSHC, ADD, SUB, MUL, DIV, RSUB, RDIV, " \
  "EXIT, EXIT, EXIT, EXIT, EXIT, SQ, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, " \
  "VADD, VSUB, VMUL, VDIV, VRSUB, EXITV, CADD, CSUB, CMUL, CDIV, CRSUB, CRDIV, EXIT;\n\t" \
  "NEXT:\n\t" SR_FETCH \
  "PUSHV:\n\t" SR_STS \
  "LDV:\n\t" LDT NEXT_OP \
  "PUSHC:\n\t" SR_STS \
  "LDC:\n\t" SR_SPLAT("%0", "%1", "%2", "%3") NEXT_OP \
  "ADD:\n\t" SR_LDS SR_XT("add", NEXT_OP) \
  "SUB:\n\t" SR_LDS SR_XT("sub", NEXT_OP) \
  "MUL:\n\t" SR_LDS SR_XT("mul", NEXT_OP) \
  "RSUB:\n\t" SR_LDS SR_TX("sub", NEXT_OP) \
  "SQ:\n\t" \
  "mul.rn.f32x2 %0, %0, %0;\n\tmul.rn.f32x2 %1, %1, %1;\n\t" \
  "mul.rn.f32x2 %2, %2, %2;\n\tmul.rn.f32x2 %3, %3, %3;\n\t" NEXT_OP \
  "VADD:\n\t" LDX SR_TX("add", NEXT_OP) \
  "VSUB:\n\t" LDX SR_TX("sub", NEXT_OP) \
  "VMUL:\n\t" LDX SR_TX("mul", NEXT_OP) \
  "VRSUB:\n\t" LDX SR_XT("sub", NEXT_OP) \
  "CADD:\n\t" SR_TC("add", NEXT_OP) \
  "CSUB:\n\t" SR_TC("sub", NEXT_OP) \
  "CMUL:\n\t" SR_TC("mul", NEXT_OP) \
  "CRSUB:\n\t" SR_CT("sub", NEXT_OP) \
  "DIV:\n\t" SR_LDS "mov.u32 %9, 27;\n\tbra EXIT;\n\t" \
  "RDIV:\n\t" SR_LDS "mov.u32 %9, 25;\n\tbra EXIT;\n\t" \
  "CDIV:\n\t" SR_SPLAT("%4", "%5", "%6", "%7") "mov.u32 %9, 25;\n\tbra EXIT;\n\t" \
  "CRDIV:\n\t" SR_SPLAT("%4", "%5", "%6", "%7") "mov.u32 %9, 27;\n\tbra EXIT;\n\t" \
  "VDIV:\n\t" LDX "bra EXIT;\n\t" \
  "EXITV:\n\t" LDX \
  "EXIT:\n\t}\n\t"
#define SR_CORE_OUT(T, X, ip, op) \
  "+l"(T.p[0]), "+l"(T.p[1]), "+l"(T.p[2]), "+l"(T.p[3]), "=&l"(X.p[0]), "=&l"(X.p[1]), "=&l"(X.p[2]), "=&l"(X.p[3]), \
      "+r"(ip), "=&r"(op)
// clang-format on
static_assert(OP_LDV == 0 && OP_PUSHC == 3 && OP_ADD == 4 && OP_RDIV == 9 && OP_SIN == 10 && OP_SQ == 15 &&
                  OP_TANH == 21 && OP_VADD == 22 && OP_VDIV == 25 && OP_VRDIV == 27 && OP_CADD == 28 &&
                  OP_CRDIV == 33 && OP_END == 34,
              "the order of the core loop's table");

// How a copy of the interpreter is laid out.  All operators of one copy and the
// kernel around it have to stay in the instruction cache together, so a copy
// with more in it keeps its bodies narrower (values in flight; map8) or fetches
// the next instruction in one place instead of after every operator.
// Measured (us), each row of figures on one population: base copy, threaded and 8
// wide against one fetch: 4,096 x 100,000 5,290 / 5,423, 8,192 x 131,072 25,308 /
// 26,600; log 4 wide 5,356 / 25,539.  Eq. 3 kernel, 4,096 x 40,000: threaded 8 wide 2,773, sin, cos
// and log 4 wide 2,562, one fetch 8 wide 2,580.  EXT copy (twelve library
// operators), 2,048 x 50,001: 2 wide with one fetch 2,102, threaded 2,287,
// 4 wide 2,265, 8 wide 2,706.
template <bool EXT, bool LEAN>
struct Shape {
  static constexpr bool THREADED = !EXT;
  static constexpr int TRIG = EXT ? 2 : (LEAN ? 4 : CPL);  // sin, cos, log
  static constexpr int POW = EXT ? 2 : CPL;                // exp, sqrt
  static constexpr int DIV = EXT ? 4 : CPL;
};

// Runs the decoded program for this lane's 8 cases.  xa / xb point at the
// lane's first and second case group in row 0 of X; `stk` at this lane's entry
// of stack slot 0 in shared memory.  The code ends with OP_END, its words hold
// the opcode in the low byte and the slot offset above it (with no flags), and
// the opcode is at most OP_END (the branch table has no default).
// EXT: the copy that also runs 1/x, tan, asin, acos, atan, tanh.
// WIDE: rows start on 32-byte boundaries and hold whole groups of 8 cases (one
// 256-bit load a row); else two 128-bit loads.
// LEAN: the code around it is large, or runs nearly as often (Shape).
template <bool EXT, bool WIDE, bool LEAN>
__device__ __forceinline__ V8 interpret(const uint2 *code, const char *stk, const float *xa,
                                        const float *xb) {
  using S = Shape<EXT, LEAN>;
  V8 T = splat8(0.f), X;
  uint32_t ip = (uint32_t)__cvta_generic_to_shared(code), op;
  const uint32_t st = (uint32_t)__cvta_generic_to_shared(stk);
  for (;;) {
    if (WIDE && S::THREADED)
      asm volatile(SR_CORE(SR_LDX_WIDE, SR_LDT_WIDE, SR_FETCH) : SR_CORE_OUT(T, X, ip, op) : "r"(st), "l"(xa) : "memory");
    else if (WIDE)
      asm volatile(SR_CORE(SR_LDX_WIDE, SR_LDT_WIDE, SR_JUMP) : SR_CORE_OUT(T, X, ip, op) : "r"(st), "l"(xa) : "memory");
    else if (S::THREADED)
      asm volatile(SR_CORE(SR_LDX_HALVES, SR_LDT_HALVES, SR_FETCH)
                   : SR_CORE_OUT(T, X, ip, op) : "r"(st), "l"(xa), "l"(xb) : "memory");
    else
      asm volatile(SR_CORE(SR_LDX_HALVES, SR_LDT_HALVES, SR_JUMP)
                   : SR_CORE_OUT(T, X, ip, op) : "r"(st), "l"(xa), "l"(xb) : "memory");
    switch (op) {
      case OP_VDIV:
        if (any_beyond(X, DIV_NEAR)) T = div8_wide(T, X);
        else T = zip8<S::DIV>(T, X, DivNear());
        break;
      case OP_VRDIV:
        if (any_beyond(T, DIV_NEAR)) T = div8_wide(X, T);
        else T = zip8<S::DIV>(X, T, DivNear());
        break;
      case OP_SIN: T = sincos8<false, EXT, S::TRIG>(T); break;
      case OP_COS: T = sincos8<true, EXT, S::TRIG>(T); break;
      case OP_EXP: T = map8<S::POW>(T, Exp()); break;
      case OP_LOG: T = map8<S::TRIG>(T, Log()); break;
      case OP_SQRT: T = map8<S::POW>(T, Sqrt()); break;
      case OP_INV:
      case OP_TAN:
      case OP_ASIN:
      case OP_ACOS:
      case OP_ATAN:
      case OP_TANH:
        if (EXT) T = ext8(op, T);
        break;
      default: return T;
    }
  }
}

}  // namespace
}  // namespace sr
