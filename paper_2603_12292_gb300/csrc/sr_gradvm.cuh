// sr_gradvm.cuh -- the instructions of the adjoint kernel: a forward and a
// reverse program per program, decoded together by one warp, and the two loops
// that run them on 128 cases, 4 per lane.
//
// What bounds it: issue slots, then the tape.  A node of the first adjoint cost
// 114 warp instructions a step (the profiler's counter): a switch over the opcodes
// each way, a tape entry written and read for most operators, and constants --
// half of the leaves -- evaluated on every case.  Now
//   - a subtree that reads only constants is evaluated once, by the decoder,
//     with its partial derivatives: the forward program loads its value, the
//     reverse program multiplies by immediates;
//   - the reverse program is written out by the decoder: nothing for a subtree
//     without constants, no tests of what is wanted, the saves and restores of
//     adjoints only where both operands have constants;
//   - operands that are immediates or rows are not taped (13 entries a program of
//     <= 96 tokens instead of 23);
//   - both loops branch through tables in PTX and run on FP32 pairs (sr_vm.cuh).
// Every value, partial and sum is rounded as before, in the same order.
// 2,048 programs of <= 96 tokens x 65,536 cases, K = 8 (us): 7,365 -> 4,440; warp
// instructions 5.97e9 -> 3.33e9, DRAM 11.1 -> 0.9 GB (the tape stays in L2); 24
// small problems, one gradient 245 -> 185.
#pragma once

#include "sr_decode.cuh"
#include "sr_vm.cuh"

namespace sr {
namespace {

constexpr int GCPL = 4;           // cases per lane (one 16-byte access per value)
constexpr int GSTEP = 32 * GCPL;  // cases per warp step
constexpr int GSLOT = GSTEP * 4;  // bytes of one stack slot / tape entry of a warp

// Instruction words as in sr_interp.cuh: opcode, slot offset from bit 8, constant
// index from bit 24; y an FP32 immediate or a row offset.
enum FwdOp : uint32_t {
  FW_LDV = 0, FW_LDC, FW_PUSHV, FW_PUSHC,  // top = row / constant (PUSH: the old top into its slot)
  FW_ADD, FW_SUB, FW_RSUB, FW_MUL,         // top = slot op top (RSUB: top - slot)
  FW_VADD, FW_VSUB, FW_VRSUB, FW_VMUL,     // top = top op row (VRSUB: row - top)
  FW_CADD, FW_CSUB, FW_CRSUB, FW_CMUL,     // top = top op constant
  FW_TAPE, FW_TAPES,                       // the top / a slot's value onto the tape
  FW_SQ, FW_SQT,                           // top^2 (T: its partial onto the tape)
  FW_DIV, FW_RDIV, FW_VDIV, FW_VRDIV, FW_CDIV, FW_CRDIV,  // quotients, as OP_DIV ... (leave the loop)
  FW_UNARY,                                // + (token - TOK_SIN): the other unary operators (leave the loop)
  FW_UNARYT = FW_UNARY + UNARY_ALL,        // the same, partial onto the tape
  FW_END = FW_UNARYT + UNARY_ALL,
};
// A: the adjoint of the value whose turn it is; X: the last result popped by RV_DIVT2
enum RevOp : uint32_t {
  RV_POP = 0,       // A = slot
  RV_SLOT,          // slot = A
  RV_SLOTN,         // slot = -A
  RV_SLOTMULT,      // slot = A * tape
  RV_SLOTMULI,      // slot = A * immediate
  RV_SLOTNEGMULX,   // slot = -(A * X)
  RV_SLOTNEGMULT,   // slot = -(A * tape)
  RV_NEG,           // A = -A
  RV_MULT,          // A = A * tape
  RV_MULI,          // A = A * immediate
  RV_MULV,          // A = A * row
  RV_NEGMULX,       // A = -(A * X)
  RV_NEGMULT,       // A = -(A * tape)
  RV_DIVT,          // A = A / tape (0 where the quotient took its fallback); leaves the loop, as those below
  RV_DIVT2,         // X = tape, A = A / tape
  RV_DIVI,          // A = A / immediate
  RV_DIVV,          // A = A / row
  RV_GACC,          // constant k's sum += A
  RV_GACCN,         // ... -A
  RV_GACCMULT,      // ... A * tape
  RV_GACCMULI,      // ... A * immediate
  RV_GACCMULV,      // ... A * row
  RV_GACCNEGMULT,   // ... -(A * tape)
  RV_END,
};
// words of both programs of up to L tokens: at most 2 L + 2 and 2.5 L + 2
__host__ __device__ inline int grad_code_words(int Lmax) { return 9 * Lmax / 2 + 4; }

// ---------------------------------------------------------------- operators and their partials
// Derivative conventions at the kinks: a protected fallback, a clamped exp and
// sqrt|x| at 0 have derivative 0.
static __device__ __noinline__ float2 sincos_wide(float x) {
  float s, c;
  sincosf(x, &s, &c);
  return make_float2(s, c);
}
__device__ __forceinline__ float2 sincos_near(float x) {  // |x| <= NEAR
  __builtin_assume(fabsf(x) <= NEAR);
  float s, c;
  sincosf(x, &s, &c);
  return make_float2(s, c);
}
__device__ __forceinline__ float d_exp(float x, float v) { return (x > 80.0f || x < -80.0f) ? 0.0f : v; }
__device__ __forceinline__ float d_log(float x) { return fabsf(x) < 1e-3f ? 0.0f : 1.0f / x; }
__device__ __forceinline__ float d_sqrt(float x, float v) { return x == 0.0f ? 0.0f : copysignf(0.5f / v, x); }
// 1/x (derivative -1/x^2, 0 where the fallback was taken), tan (1 + tan^2),
// asin (1/sqrt(1 - x^2)), acos (-1/sqrt(1 - x^2)), atan (1/(1 + x^2)), tanh (sech^2)
__device__ __forceinline__ float d_inv(float x, float v) { return fabsf(x) < 1e-3f ? 0.0f : -(v * v); }
// 1 - x^2 as (1 - x)(1 + x): no cancellation near |x| = 1
__device__ __forceinline__ float d_asin(float x) { return 1.0f / sqrtf((1.0f - x) * (1.0f + x)); }
// sech^2 x = 4e / (1 + e)^2 with e = exp(-2|x|): 1 - tanh^2 would cancel
// to 0 long before the derivative underflows
__device__ __forceinline__ float d_tanh(float x) {
  const float e = expf(-2.0f * fabsf(x));
  const float q = 1.0f + e;
  return 4.0f * e / (q * q);
}
// value and partial of 1/x ... tanh
static __device__ __noinline__ float2 ext_partial(int tok, float x) {
  switch (tok) {
    case TOK_INV: {
      const float a = op_inv(x);
      return make_float2(a, d_inv(x, a));
    }
    case TOK_TAN: {
      const float a = f_tan(x);
      return make_float2(a, 1.0f + a * a);
    }
    case TOK_ASIN: return make_float2(f_asin(x), d_asin(x));
    case TOK_ACOS: return make_float2(f_acos(x), -d_asin(x));
    case TOK_ATAN: return make_float2(f_atan(x), 1.0f / (1.0f + x * x));
    default: return make_float2(f_tanh(x), d_tanh(x));
  }
}
// value and partial of a unary operator (the decoder's constant subtrees)
static __device__ __noinline__ float2 unary_partial(int tok, float x) {
  switch (tok) {
    case TOK_SIN: {
      const float2 sc = fabsf(x) <= NEAR ? sincos_near(x) : sincos_wide(x);
      return sc;
    }
    case TOK_COS: {
      const float2 sc = fabsf(x) <= NEAR ? sincos_near(x) : sincos_wide(x);
      return make_float2(sc.y, -sc.x);
    }
    case TOK_EXP: {
      const float v = op_exp(x);
      return make_float2(v, d_exp(x, v));
    }
    case TOK_LOG: return make_float2(op_log(x), d_log(x));
    case TOK_SQRT: {
      const float v = f_sqrt(x);
      return make_float2(v, d_sqrt(x, v));
    }
    case TOK_SQ: return make_float2(__fmul_rn(x, x), __fadd_rn(x, x));
    default: return ext_partial(tok, x);
  }
}

// ---------------------------------------------------------------- decoding
struct GradDecode {
  const uint8_t *programs;  // [P][Lmax]
  const int32_t *lengths;
  const float *consts;      // [P][K]
  int Lmax, K, nvars;
  long long ldx;
  uint2 *code;              // [P][grad_code_words(Lmax)]: forward, then reverse
  int32_t *nfwd, *nrev;     // [P] words of each (with its end marker); nfwd 0: invalid
  int32_t *flags;           // [P]
  int cap_words;            // *big_note is set to 1 when some program has more words than this
  unsigned long long *big_note;
};

// info[] of a token, beside the need: what its subtree reads
constexpr uint8_t GI_CONST = 0x80;  // only constants: a leaf of the forward program (value in val)
constexpr uint8_t GI_ROW = 0x40;    // a variable (its index in val)
constexpr uint8_t GI_HASC = 0x20;   // some constant: an adjoint flows into it

// one token's scratch beside DecodeScratch's (cnt, base, live: forward)
__host__ __device__ inline int grad_scratch_bytes(int Lmax) {
  const int n = (Lmax + 3) & ~3;
  return decode_scratch_bytes(Lmax) + 4 * n + 2 * 2 * n + ((n + 15) & ~15) + 16;
}

// where an operand's value is when the reverse program wants it
enum Src { S_TAPE, S_IMM, S_ROW };
__device__ __forceinline__ Src source(uint8_t info) { return info & GI_CONST ? S_IMM : (info & GI_ROW ? S_ROW : S_TAPE); }

// A binary node as both programs see it: first / second: operands in the order of
// evaluation; rev: the right operand is the first.
struct BinNode {
  int first, second;
  uint8_t fi, si;       // their info
  bool rev, leaf;       // leaf: the second is fused (a row or a constant)
  bool cleaf;           // ... the second is a constant token of the program
  bool nf, ns;          // adjoints wanted
};
__device__ __forceinline__ BinNode bin_node(const DecodeScratch &s, int t, int a) {
  BinNode n;
  const uint8_t ia = s.info[a], ib = s.info[t - 1];
  n.rev = (ib & INFO_NEED) > (ia & INFO_NEED);
  n.first = n.rev ? t - 1 : a;
  n.second = n.rev ? a : t - 1;
  n.fi = n.rev ? ib : ia;
  n.si = n.rev ? ia : ib;
  n.leaf = (n.si & (GI_CONST | GI_ROW)) != 0;
  n.cleaf = tok_class(s.tok[n.second]) == CLS_CONST;
  n.nf = n.fi & GI_HASC;
  n.ns = n.si & GI_HASC;
  return n;
}
// what a (not constant) binary node puts on the tape: bit 0 the operand that is
// in the slot (or, fused, the top) before the operator, bit 1 the top before a
// stack operator, bit 2 the result
__device__ __forceinline__ int bin_tape(const BinNode &n, int v) {
  const bool ft = source(n.fi) == S_TAPE, st = source(n.si) == S_TAPE;
  if (v == TOK_MUL) return (n.ns && ft ? 1 : 0) | (n.nf && st ? 2 : 0);
  if (v == TOK_DIV) {
    const bool any = n.nf || n.ns;
    const bool dt = n.rev ? ft : st;              // the denominator is taped
    const bool nd = n.rev ? n.nf : n.ns;          // its adjoint is wanted
    return (any && dt ? (n.rev ? 1 : 2) : 0) | (nd ? 4 : 0);
  }
  return 0;
}

// The reverse instructions of a binary node, its own before its operands': calls
// put(op, immediate, row) for each, row 1 / 2: of the first / second operand.
// vf / vs / vt: the values of first, second and the node where they are constant;
// konst: the node itself is.  The first operand's adjoint goes to a slot where
// both are wanted; a constant token second has its sum here.
template <typename Put>
__device__ __forceinline__ void bin_reverse(const BinNode &n, int v, bool konst, float vf, float vs, float vt, Put put) {
  const Src sf = source(n.fi), ss = source(n.si);
  const Src sden = n.rev ? sf : ss;               // a quotient's denominator
  const bool nden = n.rev ? n.nf : n.ns;          // whether its adjoint is wanted
  const float vden = n.rev ? vf : vs;
  auto divide = [&] {                             // A = A / denominator; its adjoint will want the result in X
    if (sden == S_TAPE) put(nden ? RV_DIVT2 : RV_DIVT, 0.f, 0);
    else if (sden == S_IMM) put(RV_DIVI, vden, 0);
    else put(RV_DIVV, 0.f, n.rev ? 1 : 2);
  };
  auto times_first = [&] {
    if (sf == S_TAPE) put(RV_MULT, 0.f, 0);
    else if (sf == S_IMM) put(RV_MULI, vf, 0);
    else put(RV_MULV, 0.f, 1);
  };
  if (n.cleaf) {
    if (v == TOK_ADD) {
      put(RV_GACC, 0.f, 0);
    } else if (v == TOK_SUB) {
      put(n.rev ? RV_GACC : RV_GACCN, 0.f, 0);
      if (n.rev && n.nf) put(RV_NEG, 0.f, 0);
    } else if (v == TOK_MUL) {
      if (sf == S_TAPE) put(RV_GACCMULT, 0.f, 0);
      else if (sf == S_IMM) put(RV_GACCMULI, vf, 0);
      else put(RV_GACCMULV, 0.f, 1);
      if (n.nf) put(RV_MULI, vs, 0);
    } else if (!n.rev) {  // first / constant
      divide();
      if (konst) put(RV_GACCMULI, -vt, 0);
      else put(RV_GACCNEGMULT, 0.f, 0);
    } else {              // constant / first
      divide();
      put(RV_GACC, 0.f, 0);
      if (n.nf && konst) put(RV_MULI, -vt, 0);
      else if (n.nf) put(RV_NEGMULX, 0.f, 0);
    }
    return;
  }
  const bool both = n.nf && n.ns;
  if (v == TOK_ADD) {
    if (both) put(RV_SLOT, 0.f, 0);
  } else if (v == TOK_SUB) {
    if (both) put(n.rev ? RV_SLOTN : RV_SLOT, 0.f, 0);
    if (n.ns != n.rev) put(RV_NEG, 0.f, 0);  // into the second as right operand, or the first as right operand
  } else if (v == TOK_MUL) {
    if (both) {
      if (ss == S_TAPE) put(RV_SLOTMULT, 0.f, 0);
      else put(RV_SLOTMULI, vs, 0);
      times_first();
    } else if (n.ns) {
      times_first();
    } else {
      if (ss == S_TAPE) put(RV_MULT, 0.f, 0);
      else put(RV_MULV, 0.f, 2);
    }
  } else {
    divide();
    if (both && !n.rev) put(RV_SLOT, 0.f, 0);
    if (nden) {  // -(q T): T in X after a taped denominator, else next on the tape, or constant
      const bool save = both && n.rev;
      if (konst) put(save ? RV_SLOTMULI : RV_MULI, -vt, 0);
      else if (sden == S_TAPE) put(save ? RV_SLOTNEGMULX : RV_NEGMULX, 0.f, 0);
      else put(save ? RV_SLOTNEGMULT : RV_NEGMULT, 0.f, 0);
    }
  }
}

// Decodes program `prog` into its forward and reverse programs with the calling
// warp (scratch: grad_scratch_bytes).
__device__ inline void decode_grad_warp(const GradDecode &p, int prog, unsigned char *smem, int max_slots) {
  const int lane = threadIdx.x & 31;
  const DecodeScratch s = decode_scratch(smem, p.Lmax);
  const int n4 = (p.Lmax + 3) & ~3;
  float *part = reinterpret_cast<float *>(smem + decode_scratch_bytes(p.Lmax));  // partials of constant unary nodes
  uint16_t *rcnt = reinterpret_cast<uint16_t *>(part + n4), *rbase = rcnt + n4;  // reverse program, as cnt / base
  uint8_t *save = reinterpret_cast<uint8_t *>(rbase + n4);                       // saved adjoints below, as live
  const int L = p.lengths[prog];
  int flags = SR_PF_BAD_LENGTH;
  if (L >= 1 && L <= p.Lmax) {
    const uint8_t *src = p.programs + (size_t)prog * p.Lmax;
    for (int t = lane; t < L; t += 32) s.tok[t] = src[t];
    if (lane < p.K) s.consts[lane] = p.consts[(size_t)prog * p.K + lane];
    __syncwarp();
    flags = validate_warp(s, L, p.nvars, p.K, lane);
  }
  if (flags) {
    if (lane == 0) {
      p.flags[prog] = flags;
      p.nfwd[prog] = 0;
    }
    return;
  }
  // up the tree
  for (int t0 = 0; t0 < L; t0 += 32) {
    const int t = t0 + lane;
    const int v = t < L ? s.tok[t] : 0, cls = tok_class(v);
    bool todo = t < L;
    if (todo) {
      s.info[t] = 0;
      if (cls == CLS_VAR || cls == CLS_CONST) {
        s.info[t] = 1 | (cls == CLS_VAR ? GI_ROW : GI_CONST | GI_HASC);
        s.val[t] = cls == CLS_VAR ? v - TOK_VAR0 : __float_as_int(s.consts[v - TOK_CONST0]);
        s.cnt[t] = 1;
        rcnt[t] = cls == CLS_CONST;
        todo = false;
      }
    }
    const int a = todo && cls == CLS_BINARY ? s.left[t] : t - 1;
    __syncwarp();
    while (__any_sync(FULL, todo)) {
      const bool go = todo && s.info[t - 1] && s.info[a];
      __syncwarp();
      if (go) {
        todo = false;
        const uint8_t ia = s.info[a], ib = s.info[t - 1];
        const bool konst = ia & ib & GI_CONST;
        uint8_t info = ((ia | ib) & GI_HASC) | (konst ? GI_CONST : 0);
        int cnt, rc = 0;
        if (cls == CLS_UNARY) {
          info |= ib & INFO_NEED;
          if (konst) {
            const float2 vd = unary_partial(v, __int_as_float(s.val[t - 1]));
            s.val[t] = __float_as_int(vd.x);
            part[t] = vd.y;
          }
          cnt = s.cnt[t - 1] + 1;
          if (info & GI_HASC) rc = rcnt[t - 1] + 1;
        } else {
          const int na = ia & INFO_NEED, nb = ib & INFO_NEED;
          info |= (uint8_t)(na == nb ? na + 1 : (na > nb ? na : nb));
          if (konst) s.val[t] = __float_as_int(fold_op(v, __int_as_float(s.val[a]), __int_as_float(s.val[t - 1])));
          const BinNode n = bin_node(s, t, a);
          cnt = s.cnt[n.first] + (n.leaf ? 0 : s.cnt[n.second]) + 1 + __popc(bin_tape(n, v));
          if (info & GI_HASC) {
            bin_reverse(n, v, konst, 0.f, 0.f, 0.f, [&](uint32_t, float, int) { ++rc; });
            if (n.nf) rc += rcnt[n.first];
            if (n.ns && !n.cleaf) rc += rcnt[n.second] + (n.nf ? 1 : 0);
          }
        }
        s.cnt[t] = (uint16_t)(konst ? 1 : cnt);
        rcnt[t] = (uint16_t)rc;
        s.info[t] = info;
      }
      __syncwarp();
    }
  }
  // down the tree; live / save: 0xff not reached (yet), 0xfe no part in that program
  constexpr int NOT_YET = 0xff, NONE = 0xfe;
  for (int t = lane; t < L; t += 32) s.live[t] = NOT_YET;
  __syncwarp();
  const int nf = s.cnt[L - 1] + 1, nr = rcnt[L - 1] + 1;
  uint2 *fwd = p.code + (size_t)prog * grad_code_words(p.Lmax), *rv = fwd + nf;
  if (lane == 0) {
    s.base[L - 1] = rbase[L - 1] = 0;
    save[L - 1] = s.info[L - 1] & GI_HASC ? 0 : NONE;
    s.live[L - 1] = 0;
    fwd[nf - 1] = make_uint2(FW_END, 0u);
    rv[nr - 1] = make_uint2(RV_END, 0u);
  }
  __syncwarp();
  auto row_of = [&](int node) { return (uint32_t)((long long)s.val[node] * p.ldx); };
  bool deep = false;
  for (int t0 = (L - 1) & ~31; t0 >= 0; t0 -= 32) {
    const int t = t0 + lane;
    bool todo = t < L;
    const int v = todo ? s.tok[t] : 0, cls = tok_class(v);
    const uint8_t info = todo ? s.info[t] : 0;
    const int a = todo && cls == CLS_BINARY ? s.left[t] : t - 1;
    for (;;) {
      const int d = todo ? s.live[t] : NOT_YET;
      const bool go = d != NOT_YET;
      if (!__any_sync(FULL, go)) break;  // the rest of the block is inside fused leaves
      __syncwarp();
      if (go) {
        todo = false;
        const int sv = save[t], pos = s.base[t], rpos = rbase[t];
        const bool leaf = info & (GI_CONST | GI_ROW);
        if (d != NONE && leaf) {
          const bool row = info & GI_ROW;
          if (d > max_slots) deep = true;  // cannot happen for programs of <= Lmax tokens
          else
            fwd[pos] = make_uint2(d == 0 ? (row ? FW_LDV : FW_LDC)
                                         : ((row ? FW_PUSHV : FW_PUSHC) | ((uint32_t)((d - 1) * GSLOT) << 8)),
                                  row ? row_of(t) : (uint32_t)s.val[t]);
        }
        if (cls == CLS_CONST) {
          if (sv != NONE) rv[rpos] = make_uint2(RV_GACC | ((uint32_t)(v - TOK_CONST0) << 24), 0u);
        } else if (cls == CLS_UNARY) {
          const bool konst = info & GI_CONST, hasc = info & GI_HASC;
          if (!konst)
            fwd[pos + s.cnt[t] - 1] =
                make_uint2(v == TOK_SQ ? (hasc ? FW_SQT : FW_SQ) : (hasc ? FW_UNARYT : FW_UNARY) + (v - TOK_SIN), 0u);
          if (hasc) rv[rpos] = konst ? make_uint2(RV_MULI, __float_as_uint(part[t])) : make_uint2(RV_MULT, 0u);
          s.base[t - 1] = (uint16_t)pos;
          rbase[t - 1] = (uint16_t)(rpos + 1);
          save[t - 1] = (uint8_t)(hasc ? sv : NONE);
          s.live[t - 1] = (uint8_t)(konst ? NONE : d);
        } else if (cls == CLS_BINARY) {
          const bool konst = info & GI_CONST;
          const BinNode n = bin_node(s, t, a);
          if (!konst) {
            int q = pos + s.cnt[n.first] + (n.leaf ? 0 : s.cnt[n.second]);
            const int tape = bin_tape(n, v);
            const uint32_t off = (uint32_t)(d * GSLOT) << 8;
            if (tape & 1) fwd[q++] = n.leaf ? make_uint2(FW_TAPE, 0u) : make_uint2(FW_TAPES | off, 0u);
            if (tape & 2) fwd[q++] = make_uint2(FW_TAPE, 0u);
            uint32_t op;
            if (n.leaf) {
              const bool row = n.si & GI_ROW;
              if (v == TOK_DIV) op = row ? (n.rev ? FW_VRDIV : FW_VDIV) : (n.rev ? FW_CRDIV : FW_CDIV);
              else op = (row ? FW_VADD : FW_CADD) + (v == TOK_SUB ? (n.rev ? 2 : 1) : (v == TOK_MUL ? 3 : 0));
              fwd[q++] = make_uint2(op, row ? row_of(n.second) : (uint32_t)s.val[n.second]);
            } else {
              if (v == TOK_DIV) op = n.rev ? FW_RDIV : FW_DIV;
              else op = FW_ADD + (v == TOK_SUB ? (n.rev ? 2 : 1) : (v == TOK_MUL ? 3 : 0));
              fwd[q++] = make_uint2(op | off, 0u);
            }
            if (tape & 4) fwd[q++] = make_uint2(FW_TAPE, 0u);
          }
          int q = rpos;
          const bool hasc = info & GI_HASC;
          if (hasc) {
            const uint32_t k = n.cleaf ? (uint32_t)(s.tok[n.second] - TOK_CONST0) : 0u;
            const uint32_t x = ((uint32_t)(sv * GSLOT) << 8) | (k << 24);
            bin_reverse(n, v, konst, __int_as_float(s.val[n.first]), __int_as_float(s.val[n.second]),
                        __int_as_float(s.val[t]), [&](uint32_t op, float imm, int row) {
                          rv[q++] = make_uint2(op | x, row ? row_of(row == 1 ? n.first : n.second) : __float_as_uint(imm));
                        });
          }
          const bool both = n.nf && n.ns && !n.cleaf;
          const int qs = q;  // the second operand's reverse part, then (both) the first's adjoint back, then its part
          if (n.ns && !n.cleaf) q += rcnt[n.second];
          if (both) rv[q++] = make_uint2(RV_POP | ((uint32_t)(sv * GSLOT) << 8), 0u);
          if (!n.cleaf && !(n.si & GI_ROW)) {  // (a fused constant subtree still has a reverse part)
            s.base[n.second] = (uint16_t)(pos + s.cnt[n.first]);
            rbase[n.second] = (uint16_t)qs;
            save[n.second] = (uint8_t)(n.ns ? (both ? sv + 1 : sv) : NONE);
            s.live[n.second] = (uint8_t)(konst || n.leaf ? NONE : d + 1);
          }
          s.base[n.first] = (uint16_t)pos;
          rbase[n.first] = (uint16_t)q;
          save[n.first] = (uint8_t)(n.nf ? sv : NONE);
          s.live[n.first] = (uint8_t)(konst ? NONE : d);
        }
      }
      __syncwarp();
    }
  }
  deep = __any_sync(FULL, deep);
  if (lane == 0) {
    p.flags[prog] = deep ? SR_PF_TOO_DEEP : 0;
    p.nfwd[prog] = deep ? 0 : nf;
    p.nrev[prog] = nr;
    if (!deep && nf + nr > p.cap_words) *p.big_note = 1;
  }
}

// ---------------------------------------------------------------- the two loops
struct V4 {  // this lane's 4 cases of a value
  pair_t p[2];
};
__device__ __forceinline__ void unpack4(const V4 &v, float (&t)[GCPL]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) asm("mov.b64 {%0, %1}, %2;" : "=f"(t[2 * i]), "=f"(t[2 * i + 1]) : "l"(v.p[i]));
}
__device__ __forceinline__ V4 pack4(const float (&t)[GCPL]) { return V4{{pack(t[0], t[1]), pack(t[2], t[3])}}; }

// Operands of both: %0-%1 T / A, %2-%3 X (the operand an instruction leaves the
// loop with), %4 address of the next instruction, %5 its first word (the opcode of
// the forward loop), %6 tape, then %7 slot 0 and %8 row 0 of this lane; the
// reverse loop has %7-%8 its X register (RV_DIVT2) and %9, %10 those.
// clang-format off
#define GR_ROW(d0, d1, xa) "mad.wide.u32 a, wy, 4, " xa ";\n\tld.global.v2.b64 {" d0 ", " d1 "}, [a];\n\t"
#define GR_SLOT(st) "bfe.u32 s, wx, 8, 16;\n\tadd.u32 s, s, " st ";\n\t"
#define GR_SPLAT(d0, d1) "mov.b64 " d0 ", {wy, wy};\n\tmov.b64 " d1 ", " d0 ";\n\t"
#define GR_PUSH(s0, s1) "st.global.v2.b64 [%6], {" s0 ", " s1 "};\n\tadd.u64 %6, %6, 512;\n\t"
#define GR_POP(d0, d1) "add.u64 %6, %6, -512;\n\tld.global.v2.b64 {" d0 ", " d1 "}, [%6];\n\t"
#define GR_OP2(op, d0, d1, a0, a1, b0, b1) \
  op ".rn.f32x2 " d0 ", " a0 ", " b0 ";\n\t" op ".rn.f32x2 " d1 ", " a1 ", " b1 ";\n\t"
#define GR_NEG(d0, d1, s0, s1) "xor.b64 " d0 ", " s0 ", 0x8000000080000000;\n\txor.b64 " d1 ", " s1 ", 0x8000000080000000;\n\t"
#define GR_FETCH_F "ld.shared.v2.b32 {wx, wy}, [%4];\n\tadd.u32 %4, %4, 8;\n\tand.b32 %5, wx, 255;\n\tbrx.idx.uni %5, TABLE;\n\t"
#define GR_TX(op) GR_OP2(op, "%0", "%1", "%0", "%1", "%2", "%3") GR_FETCH_F
#define GR_XT(op) GR_OP2(op, "%0", "%1", "%2", "%3", "%0", "%1") GR_FETCH_F
#define GR_LDX GR_ROW("%2", "%3", "%8")
#define GR_LDSX GR_SLOT("%7") "ld.shared.v2.b64 {%2, %3}, [s];\n\t"
#define GR_STS GR_SLOT("%7") "st.shared.v2.b64 [s], {%0, %1};\n\t"
#define GR_FWD \
  "{\n\t.reg .b32 wx, wy, s;\n\t.reg .b64 a;\n\t" \
  "TABLE: .branchtargets LDV, LDC, PUSHV, PUSHC, ADD, SUB, RSUB, MUL, VADD, VSUB, VRSUB, VMUL, " \
  "CADD, CSUB, CRSUB, CMUL, TAPE, TAPES, SQ, SQT, DIV, DIV, VDIV, VDIV, CDIV, CDIV, " \
  "EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, " \
  "EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT, EXIT;\n\t" \
  GR_FETCH_F \
  "PUSHV:\n\t" GR_STS \
  "LDV:\n\t" GR_ROW("%0", "%1", "%8") GR_FETCH_F \
  "PUSHC:\n\t" GR_STS \
  "LDC:\n\t" GR_SPLAT("%0", "%1") GR_FETCH_F \
  "ADD:\n\t" GR_LDSX GR_XT("add") \
  "SUB:\n\t" GR_LDSX GR_XT("sub") \
  "RSUB:\n\t" GR_LDSX GR_TX("sub") \
  "MUL:\n\t" GR_LDSX GR_XT("mul") \
  "VADD:\n\t" GR_LDX GR_TX("add") \
  "VSUB:\n\t" GR_LDX GR_TX("sub") \
  "VRSUB:\n\t" GR_LDX GR_XT("sub") \
  "VMUL:\n\t" GR_LDX GR_TX("mul") \
  "CADD:\n\t" GR_SPLAT("%2", "%3") GR_TX("add") \
  "CSUB:\n\t" GR_SPLAT("%2", "%3") GR_TX("sub") \
  "CRSUB:\n\t" GR_SPLAT("%2", "%3") GR_XT("sub") \
  "CMUL:\n\t" GR_SPLAT("%2", "%3") GR_TX("mul") \
  "TAPE:\n\t" GR_PUSH("%0", "%1") GR_FETCH_F \
  "TAPES:\n\t" GR_LDSX GR_PUSH("%2", "%3") GR_FETCH_F \
  "SQT:\n\t" GR_OP2("add", "%2", "%3", "%0", "%1", "%0", "%1") GR_PUSH("%2", "%3") \
  "SQ:\n\t" GR_OP2("mul", "%0", "%1", "%0", "%1", "%0", "%1") GR_FETCH_F \
  "DIV:\n\t" GR_LDSX "bra EXIT;\n\t" \
  "CDIV:\n\t" GR_SPLAT("%2", "%3") "bra EXIT;\n\t" \
  "VDIV:\n\t" GR_LDX \
  "EXIT:\n\t}\n\t"

#define GR_FETCH_R "ld.shared.v2.b32 {wx, wy}, [%4];\n\tadd.u32 %4, %4, 8;\n\tand.b32 s, wx, 255;\n\tbrx.idx.uni s, TABLE;\n\t"
#define GR_SLOTR GR_SLOT("%9")
#define GR_PUT(s0, s1) GR_SLOTR "st.shared.v2.b64 [s], {" s0 ", " s1 "};\n\t" GR_FETCH_R
#define GR_MULX(d0, d1) GR_OP2("mul", d0, d1, "%0", "%1", "%2", "%3")
#define GR_REV \
  "{\n\t.reg .b32 wx, wy, s;\n\t.reg .b64 a;\n\t" \
  "TABLE: .branchtargets POP, SLOT, SLOTN, SLOTMULT, SLOTMULI, SLOTNEGMULX, SLOTNEGMULT, NEG, MULT, MULI, MULV, " \
  "NEGMULX, NEGMULT, DIVT, DIVT2, DIVI, DIVV, GACC, GACCN, GACCMULT, GACCMULI, GACCMULV, GACCNEGMULT, EXIT;\n\t" \
  GR_FETCH_R \
  "POP:\n\t" GR_SLOTR "ld.shared.v2.b64 {%0, %1}, [s];\n\t" GR_FETCH_R \
  "SLOT:\n\t" GR_PUT("%0", "%1") \
  "SLOTN:\n\t" GR_NEG("%2", "%3", "%0", "%1") GR_PUT("%2", "%3") \
  "SLOTMULT:\n\t" GR_POP("%2", "%3") GR_MULX("%2", "%3") GR_PUT("%2", "%3") \
  "SLOTMULI:\n\t" GR_SPLAT("%2", "%3") GR_MULX("%2", "%3") GR_PUT("%2", "%3") \
  "SLOTNEGMULT:\n\t" GR_POP("%7", "%8") \
  "SLOTNEGMULX:\n\t" GR_OP2("mul", "%2", "%3", "%0", "%1", "%7", "%8") GR_NEG("%2", "%3", "%2", "%3") GR_PUT("%2", "%3") \
  "NEG:\n\t" GR_NEG("%0", "%1", "%0", "%1") GR_FETCH_R \
  "MULT:\n\t" GR_POP("%2", "%3") GR_MULX("%0", "%1") GR_FETCH_R \
  "MULI:\n\t" GR_SPLAT("%2", "%3") GR_MULX("%0", "%1") GR_FETCH_R \
  "MULV:\n\t" GR_ROW("%2", "%3", "%10") GR_MULX("%0", "%1") GR_FETCH_R \
  "NEGMULT:\n\t" GR_POP("%7", "%8") \
  "NEGMULX:\n\t" GR_OP2("mul", "%0", "%1", "%0", "%1", "%7", "%8") GR_NEG("%0", "%1", "%0", "%1") GR_FETCH_R \
  "DIVT2:\n\t" GR_POP("%7", "%8") \
  "DIVT:\n\t" GR_POP("%2", "%3") "bra EXIT;\n\t" \
  "DIVI:\n\t" GR_SPLAT("%2", "%3") "bra EXIT;\n\t" \
  "DIVV:\n\t" GR_ROW("%2", "%3", "%10") "bra EXIT;\n\t" \
  "GACC:\n\tmov.b64 %2, %0;\n\tmov.b64 %3, %1;\n\tbra EXIT;\n\t" \
  "GACCN:\n\t" GR_NEG("%2", "%3", "%0", "%1") "bra EXIT;\n\t" \
  "GACCMULT:\n\t" GR_POP("%2", "%3") GR_MULX("%2", "%3") "bra EXIT;\n\t" \
  "GACCMULI:\n\t" GR_SPLAT("%2", "%3") GR_MULX("%2", "%3") "bra EXIT;\n\t" \
  "GACCMULV:\n\t" GR_ROW("%2", "%3", "%10") GR_MULX("%2", "%3") "bra EXIT;\n\t" \
  "GACCNEGMULT:\n\t" GR_POP("%2", "%3") GR_MULX("%2", "%3") GR_NEG("%2", "%3", "%2", "%3") \
  "EXIT:\n\tmov.b32 %5, wx;\n\t}\n\t"
// clang-format on
static_assert(FW_TAPE == 16 && FW_SQT == 19 && FW_DIV == 20 && FW_CRDIV == 25 && FW_UNARY == 26 && FW_UNARYT == 38 &&
                  FW_END == 50 && RV_NEGMULT == 12 && RV_DIVT == 13 && RV_GACC == 17 && RV_GACCMULV == 21 && RV_END == 23 &&
                  GSLOT == 512,
              "the order of the loops' tables, and the tape's stride");

struct SinCos4 {
  V4 s, c;
};
// Some argument of the warp is not moderate, or NaN: the whole function on each value.
// (With such values replaced by 0 and recognised afterwards 2,048 x 65,536 took 4,500 us
// instead of 4,440, with 16 operators 8,838 instead of 8,390.)
__device__ __noinline__ SinCos4 sincos4_wide(V4 x) {
  float a[GCPL], b[GCPL];
  unpack4(x, a);
#pragma unroll 1
  for (int i = 0; i < GCPL; ++i) {
    const float2 r = sincos_wide(a[0]);
#pragma unroll
    for (int j = 0; j < GCPL - 1; ++j) a[j] = a[j + 1], b[j] = b[j + 1];
    a[GCPL - 1] = r.x;
    b[GCPL - 1] = r.y;
  }
  return SinCos4{pack4(a), pack4(b)};
}
__device__ __forceinline__ SinCos4 sincos4(const V4 &x) {
  float a[GCPL], b[GCPL];
  unpack4(x, a);
  bool ok = true;
#pragma unroll
  for (int i = 0; i < GCPL; ++i) ok = ok & (fabsf(a[i]) <= NEAR);
  if (__any_sync(FULL, !ok)) return sincos4_wide(x);
#pragma unroll
  for (int i = 0; i < GCPL; ++i) {
    const float2 r = sincos_near(a[i]);
    a[i] = r.x;
    b[i] = r.y;
  }
  return SinCos4{pack4(a), pack4(b)};
}
__device__ __noinline__ V4 div4_wide(V4 a, V4 b) {
  float x[GCPL], y[GCPL];
  unpack4(a, x);
  unpack4(b, y);
#pragma unroll
  for (int i = 0; i < GCPL; ++i) x[i] = op_div(x[i], y[i]);
  return pack4(x);
}
__device__ __forceinline__ V4 div4(const V4 &a, const V4 &b) {  // the protected quotient (DivNear, sr_vm.cuh)
  float x[GCPL], y[GCPL];
  unpack4(a, x);
  unpack4(b, y);
  bool ok = true;
#pragma unroll
  for (int i = 0; i < GCPL; ++i) ok = ok & (fabsf(y[i]) <= DIV_NEAR);
  if (__any_sync(FULL, !ok)) return div4_wide(a, b);
#pragma unroll
  for (int i = 0; i < GCPL; ++i) x[i] = DivNear()(x[i], y[i]);
  return pack4(x);
}
// 1/x ... tanh: value and partial
struct ValPart4 {
  V4 v, d;
};
__device__ __noinline__ ValPart4 ext4(int tok, V4 x) {
  float t[GCPL], d[GCPL];
  unpack4(x, t);
#pragma unroll 1
  for (int i = 0; i < GCPL; ++i) {
    const float2 r = ext_partial(tok, t[0]);
#pragma unroll
    for (int j = 0; j < GCPL - 1; ++j) t[j] = t[j + 1], d[j] = d[j + 1];
    t[GCPL - 1] = r.x;
    d[GCPL - 1] = r.y;
  }
  return ValPart4{pack4(t), pack4(d)};
}

// The forward program at shared address ip on this lane's 4 cases (xr: their place
// in row 0); tape: this lane's next entry.  Returns the output.
__device__ __forceinline__ V4 run_forward(uint32_t ip, uint32_t st, const float *xr, char *&tape) {
  V4 T{{0ull, 0ull}}, X;
  uint32_t op;
  for (;;) {
    asm volatile(GR_FWD
                 : "+l"(T.p[0]), "+l"(T.p[1]), "=&l"(X.p[0]), "=&l"(X.p[1]), "+r"(ip), "=&r"(op), "+l"(tape)
                 : "r"(st), "l"(xr)
                 : "memory");
    if (op >= FW_END) return T;
    if (op < FW_UNARY) {  // a quotient: X / T or T / X
      const bool xt = op == FW_DIV || op == FW_VRDIV || op == FW_CRDIV;
      T = xt ? div4(X, T) : div4(T, X);
      continue;
    }
    const bool taped = op >= FW_UNARYT;
    const int tok = TOK_SIN + (int)(op - (taped ? FW_UNARYT : FW_UNARY));
    float x[GCPL], d[GCPL];
    if (tok <= TOK_COS) {
      SinCos4 r = sincos4(T);
      if (tok == TOK_SIN) {
        T = r.s;
        X = r.c;
      } else {
        T = r.c;
        X = V4{{r.s.p[0] ^ 0x8000000080000000ull, r.s.p[1] ^ 0x8000000080000000ull}};
      }
    } else if (tok == TOK_EXP) {
      unpack4(T, x);
#pragma unroll
      for (int i = 0; i < GCPL; ++i) {
        const float v = Exp()(x[i]);
        d[i] = d_exp(x[i], v);
        x[i] = v;
      }
      T = pack4(x);
      X = pack4(d);
    } else if (tok == TOK_LOG) {
      unpack4(T, x);
#pragma unroll
      for (int i = 0; i < GCPL; ++i) {
        d[i] = d_log(x[i]);
        x[i] = op_log(x[i]);
      }
      T = pack4(x);
      X = pack4(d);
    } else if (tok == TOK_SQRT) {
      unpack4(T, x);
#pragma unroll
      for (int i = 0; i < GCPL; ++i) {
        const float v = f_sqrt(x[i]);
        d[i] = d_sqrt(x[i], v);
        x[i] = v;
      }
      T = pack4(x);
      X = pack4(d);
    } else {
      const ValPart4 r = ext4(tok, T);
      T = r.v;
      X = r.d;
    }
    if (taped) {
      *reinterpret_cast<ulonglong2 *>(tape) = make_ulonglong2(X.p[0], X.p[1]);
      tape += GSLOT;
    }
  }
}

// adjoint through a protected quotient: a / d, 0 where the fallback was taken
__device__ __forceinline__ float qdiv(float a, float d) { return fabsf(d) < 1e-3f ? 0.0f : a / d; }

// The reverse program at shared address ip, from the output's adjoint A.  sums:
// this lane's entry of the constants' compensated sums, [K][32], and, comp
// floats on, their compensations.  okm: bit i, case i is inside the chunk.
__device__ __forceinline__ void run_reverse(uint32_t ip, uint32_t st, const float *xr, char *tape, V4 A, float *sums,
                                            int comp, unsigned okm) {
  V4 X, Y{{0ull, 0ull}};
  uint32_t w;
  for (;;) {
    asm volatile(GR_REV
                 : "+l"(A.p[0]), "+l"(A.p[1]), "=&l"(X.p[0]), "=&l"(X.p[1]), "+r"(ip), "=&r"(w), "+l"(tape),
                   "+l"(Y.p[0]), "+l"(Y.p[1])
                 : "r"(st), "l"(xr)
                 : "memory");
    const uint32_t op = w & 0xffu;
    if (op == RV_END) return;
    float x[GCPL];
    unpack4(X, x);
    if (op < RV_GACC) {
      float a[GCPL];
      unpack4(A, a);
#pragma unroll
      for (int i = 0; i < GCPL; ++i) a[i] = qdiv(a[i], x[i]);
      A = pack4(a);
    } else {
      float v = 0.0f;
#pragma unroll
      for (int i = 0; i < GCPL; ++i) v += ((okm >> i) & 1u) ? x[i] : 0.0f;
      float *s = sums + (w >> 24) * 32, *c = s + comp;
      const float sv = *s, cv = *c;
      const float yv = v - cv;
      const float t = sv + yv;
      *c = (t - sv) - yv;
      *s = t;
    }
  }
}

}  // namespace
}  // namespace sr
