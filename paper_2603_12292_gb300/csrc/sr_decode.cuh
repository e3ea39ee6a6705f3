// sr_decode.cuh -- validation and scheduled decoding of a program for the
// evaluation kernels, by one warp.
//
// What bounds it: latency.  A program is a chain of dependent steps, and a call
// has at most a few warps' worth of programs per scheduler.  Lane 0 walking the
// tokens took ~1,000 cycles a token (60 us for 128 tokens, 19 us for 32, of
// calls of 40 to 300 us).  Here a lane has a token:
//   - depths are prefix sums of the stack effects (two ballots give 32);
//   - a binary operator's left operand ends at the last token before it of equal
//     depth (depth moves by at most one a token), found from the masks of equal
//     depth within 32 tokens and the last position of each depth before them;
//   - attributes (stack need, folded value, table row, instruction count) go up
//     the tree and positions go down it in rounds: 32 tokens at a time, the
//     operands of a token lie before it, so a block of 32 takes as many rounds
//     as its longest chain.
// Every instruction, flag and folded value is what the serial walk gave.
// Decode launch (us, before -> now): 256 programs of <= 32 tokens 19 -> 11, 512
// of <= 128 60 -> 27, 4,096 of <= 128 80 -> 35, 8,192 of <= 256 300 -> 129; a
// captured generation of 256 x 1,000 40 -> 33, outputs of 512 x 30,011 261 -> 230.
#pragma once

#include "sr_interp.cuh"

namespace sr {

// info[] of a token: the stack need in the low bits (0: not known yet)
constexpr uint8_t INFO_CONST = 0x80;  // a leaf: a constant, or a folded subtree (value in val)
constexpr uint8_t INFO_ROW = 0x40;    // a leaf: a row of X or of the variable table (row in val)
constexpr uint8_t INFO_NEED = 0x1f;

// Shared scratch of one warp for programs of up to Lmax tokens.
struct DecodeScratch {
  int32_t *val;    // [Lmax] FP32 bits of a constant leaf, row of a row leaf
  int16_t *left;   // [Lmax] root of a binary operator's left operand
  uint16_t *cnt;   // [Lmax] instructions of the subtree
  uint16_t *base;  // [Lmax] position of its first instruction
  int16_t *last;   // [Lmax + 2] last position of each depth
  uint8_t *tok, *info, *live;  // [Lmax] token, attributes, values below the subtree's on the stack
  float *consts;   // [SR_MAX_CONSTS]
};
__host__ __device__ inline int decode_scratch_bytes(int Lmax) {
  const int n = (Lmax + 3) & ~3;
  return (4 * n + SR_MAX_CONSTS * 4 + 2 * (4 * n + 4) + 3 * n + 15) & ~15;
}
__device__ __forceinline__ DecodeScratch decode_scratch(unsigned char *p, int Lmax) {
  const int n = (Lmax + 3) & ~3;
  DecodeScratch s;
  s.val = reinterpret_cast<int32_t *>(p);
  s.consts = reinterpret_cast<float *>(s.val + n);
  s.left = reinterpret_cast<int16_t *>(s.consts + SR_MAX_CONSTS);
  s.cnt = reinterpret_cast<uint16_t *>(s.left + n);
  s.base = s.cnt + n;
  s.last = reinterpret_cast<int16_t *>(s.base + n);
  s.tok = reinterpret_cast<uint8_t *>(s.last + n + 4);
  s.info = s.tok + n;
  s.live = s.info + n;
  return s;
}

// The SR_PF_* flags of the program in s.tok (L tokens), and s.left.  Flag
// rules: bad byte; variable / constant index out of range; depth (running sum
// of +1 terminal, 0 unary or bad byte, -1 binary) below 1 after some token;
// final depth not 1.
__device__ __forceinline__ int validate_warp(const DecodeScratch &s, int L, int nvars, int K, int lane) {
  const unsigned upto = 0xffffffffu >> (31 - lane);
  int flags = 0, depth = 0;
  for (int d = lane; d <= L; d += 32) s.last[d] = -1;
  __syncwarp();
  for (int t0 = 0; t0 < L; t0 += 32) {
    const int t = t0 + lane;
    const bool in = t < L;
    const int v = in ? s.tok[t] : TOK_VAR0, cls = tok_class(v);
    if (cls == CLS_BAD) flags |= SR_PF_BAD_TOKEN;
    if (cls == CLS_VAR && in && v - TOK_VAR0 >= nvars) flags |= SR_PF_BAD_VAR;
    if (cls == CLS_CONST && v - TOK_CONST0 >= K) flags |= SR_PF_BAD_CONST;
    const int e = in ? cls_effect(cls) : 0;
    const unsigned up = __ballot_sync(FULL, e > 0), down = __ballot_sync(FULL, e < 0);
    const int d = depth + __popc(up & upto) - __popc(down & upto);  // depth after token t
    if (in && d < 1) flags |= SR_PF_UNDERFLOW;
    depth += __popc(up) - __popc(down);
    flags = __reduce_or_sync(FULL, flags);
    if (flags & SR_PF_UNDERFLOW) break;  // depths are no stack heights any more; the other tokens' bytes still count
    // left operand of a binary operator: the last token before t - 1 of its depth
    const unsigned same = __match_any_sync(FULL, in ? d : -1);
    const unsigned before = same & (upto >> 1);
    if (cls == CLS_BINARY && in) s.left[t] = (int16_t)(before ? t0 + 31 - __clz(before) : s.last[d]);
    __syncwarp();
    if (in && (same & ~upto) == 0) s.last[d] = (int16_t)t;  // the block's last of this depth
    __syncwarp();
  }
  if (flags & SR_PF_UNDERFLOW) {  // the whole program's bytes and final depth, as every token is looked at
    depth = 0;
    for (int t0 = 0; t0 < L; t0 += 32) {
      const int t = t0 + lane;
      const bool in = t < L;
      const int v = in ? s.tok[t] : TOK_VAR0, cls = tok_class(v);
      if (cls == CLS_BAD) flags |= SR_PF_BAD_TOKEN;
      if (cls == CLS_VAR && in && v - TOK_VAR0 >= nvars) flags |= SR_PF_BAD_VAR;
      if (cls == CLS_CONST && v - TOK_CONST0 >= K) flags |= SR_PF_BAD_CONST;
      const int e = in ? cls_effect(cls) : 0;
      depth += __popc(__ballot_sync(FULL, e > 0)) - __popc(__ballot_sync(FULL, e < 0));
    }
    flags = __reduce_or_sync(FULL, flags);
  }
  return depth == 1 ? flags : flags | SR_PF_BAD_FINAL;
}

// Decodes program `prog` with the calling warp for the evaluation kernels
// (constant-only subtrees folded, transforms by p.xform) in scratch `smem`.
__device__ inline void decode_eval_warp(const DecodeArgs &p, int prog, unsigned char *smem) {
  const int lane = threadIdx.x & 31;
  const DecodeScratch s = decode_scratch(smem, p.Lmax);
  const int L = p.lengths[prog];
  if (L < 1 || L > p.Lmax) {
    if (lane == 0) {
      p.flags[prog] = SR_PF_BAD_LENGTH;
      p.ncode[prog] = 0;
    }
    return;
  }
  const uint8_t *src = p.programs + (size_t)prog * p.Lmax;
  for (int t = lane; t < L; t += 32) s.tok[t] = src[t];
  if (lane < p.K) s.consts[lane] = p.consts[(size_t)prog * p.K + lane];
  __syncwarp();
  int flags = validate_warp(s, L, p.nvars, p.K, lane);
  if (flags) {
    if (lane == 0) {
      p.flags[prog] = flags;
      p.ncode[prog] = 0;
    }
    return;
  }
  // up the tree: needs (terminal 1; unary as its child; binary the larger of
  // its operands', +1 on a tie), folded values, rows, instruction counts
  bool ext = false;
  for (int t0 = 0; t0 < L; t0 += 32) {
    const int t = t0 + lane;
    const int v = t < L ? s.tok[t] : 0, cls = tok_class(v);
    bool todo = t < L;
    if (todo) {
      s.info[t] = 0;
      if (cls == CLS_VAR || cls == CLS_CONST) {
        s.info[t] = 1 | (cls == CLS_VAR ? INFO_ROW : INFO_CONST);
        s.val[t] = cls == CLS_VAR ? v - TOK_VAR0 : __float_as_int(s.consts[v - TOK_CONST0]);
        s.cnt[t] = 1;
        todo = false;
      }
    }
    const int a = todo && cls == CLS_BINARY ? s.left[t] : t - 1;
    __syncwarp();
    while (__any_sync(FULL, todo)) {
      uint8_t ib = 0, ia = 0;
      if (todo) {
        ib = s.info[t - 1];
        ia = s.info[a];
      }
      __syncwarp();
      if (todo && ia && ib) {
        todo = false;
        uint8_t info = 0;
        int cnt = 1;
        if (ia & ib & INFO_CONST) {  // only constants below
          info = 1 | INFO_CONST;
          s.val[t] = __float_as_int(fold_op(v, __int_as_float(s.val[a]), __int_as_float(s.val[t - 1])));
        } else if (cls == CLS_UNARY) {
          const int row = ib & INFO_ROW ? s.val[t - 1] : -1;
          int to = -1;
          if (p.xform && row >= 0 && row < p.nvars) to = xform_row(p.nvars, v, row);
          else if (p.xform > 1 && row >= 0 && v <= TOK_SQ && row < xform_row(p.nvars, TOK_SQ + 1, 0))
            to = xform_row2(p.nvars, v, TOK_SIN + (row - p.nvars) / p.nvars, (row - p.nvars) % p.nvars);
          if (to >= 0) {
            info = 1 | INFO_ROW;
            s.val[t] = to;
            p.xneed[to - p.nvars] = 1;
          } else {
            info = ib & INFO_NEED;
            cnt = s.cnt[t - 1] + 1;
            ext = ext || v > TOK_SQ;
          }
        } else {
          const int na = ia & INFO_NEED, nb = ib & INFO_NEED;
          info = (uint8_t)(na == nb ? na + 1 : (na > nb ? na : nb));
          const uint8_t second = nb > na ? ia : ib;  // the operand evaluated second; a leaf is fused
          const int cb = s.cnt[t - 1], ca = s.cnt[a];
          cnt = 1 + (second & (INFO_CONST | INFO_ROW) ? (nb > na ? cb : ca) : ca + cb);
        }
        s.info[t] = info;
        s.cnt[t] = (uint16_t)cnt;
      }
      __syncwarp();
    }
  }
  // down the tree: positions and live values, and the instruction of every
  // token that keeps one.  live: -1 where the token is inside a leaf
  for (int t = lane; t < L; t += 32) s.live[t] = 0xff;
  __syncwarp();
  if (lane == 0) {
    s.base[L - 1] = 0;
    s.live[L - 1] = 0;
  }
  __syncwarp();
  uint2 *code = p.code + (size_t)prog * p.Lmax;
  auto operand = [&](uint32_t x, int node) {
    const int v = s.val[node];
    return make_uint2(x, s.info[node] & INFO_CONST ? (uint32_t)v : (uint32_t)((long long)v * p.ldx));
  };
  int used = 0;
  bool deep = false;
  for (int t0 = (L - 1) & ~31; t0 >= 0; t0 -= 32) {
    const int t = t0 + lane;
    bool todo = t < L;
    const int v = todo ? s.tok[t] : 0, cls = tok_class(v);
    const uint8_t info = todo ? s.info[t] : 0;
    const int a = todo && cls == CLS_BINARY ? s.left[t] : t - 1;
    for (;;) {
      const int d = todo ? s.live[t] : 0xff;
      const bool go = d != 0xff;
      if (!__any_sync(FULL, go)) break;  // the rest of the block lies inside leaves
      if (go) {
        todo = false;
        const int pos = s.base[t], cnt = s.cnt[t];
        if (info & (INFO_CONST | INFO_ROW)) {
          const bool row = info & INFO_ROW;
          if (d > p.max_slots) {
            deep = true;  // cannot happen for programs of <= Lmax tokens; never write past the slots
          } else {
            uint32_t op = row ? OP_LDV : OP_LDC;
            if (d > 0) op = (uint32_t)(row ? OP_PUSHV : OP_PUSHC) | ((uint32_t)((d - 1) * p.slot_bytes) << 8);
            code[pos] = operand(op, t);
          }
          used = max(used, d);  // slots 0 .. d - 1 are in use
        } else if (cls == CLS_UNARY) {
          code[pos + cnt - 1] = make_uint2((uint32_t)(OP_SIN + (v - TOK_SIN)), 0u);
          s.base[t - 1] = (uint16_t)pos;
          s.live[t - 1] = (uint8_t)d;
        } else {
          const int b = t - 1;
          const bool rev = (s.info[b] & INFO_NEED) > (s.info[a] & INFO_NEED);
          const int first = rev ? b : a, second = rev ? a : b;
          s.base[first] = (uint16_t)pos;
          s.live[first] = (uint8_t)d;
          uint2 w;
          if (s.info[second] & (INFO_CONST | INFO_ROW)) {
            const bool row = s.info[second] & INFO_ROW;
            uint32_t op;
            if (rev && v == TOK_SUB) op = row ? OP_VRSUB : OP_CRSUB;
            else if (rev && v == TOK_DIV) op = row ? OP_VRDIV : OP_CRDIV;
            else op = (uint32_t)((row ? OP_VADD : OP_CADD) + v);  // + and * commute exactly
            w = operand(op, second);
          } else {
            s.base[second] = (uint16_t)(pos + s.cnt[first]);
            s.live[second] = (uint8_t)(d + 1);
            uint32_t op;
            if (rev && v == TOK_SUB) op = OP_RSUB;
            else if (rev && v == TOK_DIV) op = OP_RDIV;
            else op = (uint32_t)(OP_ADD + v);
            w = make_uint2(op | ((uint32_t)(d * p.slot_bytes) << 8), 0u);
          }
          code[pos + cnt - 1] = w;
        }
      }
      __syncwarp();
    }
  }
  used = __reduce_max_sync(FULL, used);
  ext = __any_sync(FULL, ext);
  deep = __any_sync(FULL, deep);
  if (lane == 0) {
    p.flags[prog] = deep ? SR_PF_TOO_DEEP : 0;
    const bool past_cap = used > p.cap_slots || s.cnt[L - 1] >= p.cap_words;
    p.ncode[prog] = deep ? 0 : s.cnt[L - 1] | (ext ? NCODE_EXT : 0) | (past_cap ? NCODE_DEEP : 0);
    if (!deep && ext) *p.ext_note = 1;
    if (!deep && past_cap) *p.deep_note = 1;
  }
}

}  // namespace sr
