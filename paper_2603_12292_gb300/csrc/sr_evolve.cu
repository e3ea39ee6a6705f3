// sr_evolve.cu -- selection and variation on the device: Philox4x32-10,
// k-way tournament, subtree crossover, point / subtree / constant mutation
// and random valid programs.  The paper runs selection, births and mutation
// on the CPU and only evaluation on the GPU (Sec. 2.1.2); here the whole
// generation stays resident.  Every child is a pure function of (seed,
// generation, inputs), so a CPU implementation of the same rules (the
// specification in sr.h) reproduces it bit for bit.
#include <math.h>

#include "sr_common.cuh"

namespace sr {
namespace {

// ---------------------------------------------------------------- Philox4x32-10
// Salmon, Moraes, Dror, Shaw, "Parallel Random Numbers: As Easy as 1, 2, 3"
// (SC'11): ten rounds of two 32x32 multiplies with a Weyl-sequence key.
struct Word4 {
  uint32_t v[4];
};

__device__ __forceinline__ Word4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t m0 = 0xD2511F53u * c0, h0 = __umulhi(0xD2511F53u, c0);
    const uint32_t m1 = 0xCD9E8D57u * c2, h1 = __umulhi(0xCD9E8D57u, c2);
    const uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
    c0 = n0;
    c1 = m1;
    c2 = n2;
    c3 = m0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  Word4 w;
  w.v[0] = c0;
  w.v[1] = c1;
  w.v[2] = c2;
  w.v[3] = c3;
  return w;
}

struct Rng {
  uint32_t k0, k1, gen;
  const uint64_t *gen_dev;  // when set, the generation is *gen_dev + gen (read on the device)
  __device__ __forceinline__ Word4 draw(uint32_t d, uint32_t indiv, uint32_t purpose) const {
    return philox(d, indiv, purpose, gen, k0, k1);
  }
  __device__ __forceinline__ Rng resolved() const {
    Rng r = *this;
    if (gen_dev) r.gen = (uint32_t)(*gen_dev + (uint64_t)gen);
    r.gen_dev = nullptr;
    return r;
  }
};

inline Rng make_rng(uint64_t seed, uint64_t gen, const uint64_t *gen_dev = nullptr) {
  Rng r;
  r.k0 = (uint32_t)seed;
  r.k1 = (uint32_t)(seed >> 32);
  r.gen = (uint32_t)gen;
  r.gen_dev = gen_dev;
  return r;
}

// [0, n) by multiply-high (Lemire 2019); [0, 1) from the top 24 bits
__device__ __forceinline__ uint32_t below(uint32_t w, uint32_t n) { return __umulhi(w, n); }
__device__ __forceinline__ float unit24(uint32_t w) {
  return __fmul_rn((float)(w >> 8), 5.9604644775390625e-8f);  // 2^-24, exact
}

constexpr uint32_t PU_TOURN_A = 1, PU_TOURN_B = 2, PU_DECIDE = 3, PU_CROSS = 4, PU_POINT = 5,
                   PU_SUBTREE = 6, PU_SUBGEN = 7, PU_CONSTMUT = 8, PU_INIT = 9, PU_INITC = 10,
                   PU_MICRO_SAMPLE = 11, PU_MICRO_A = 12, PU_MICRO_B = 13;

__device__ __forceinline__ int effect(int v) { return cls_effect(tok_class(v)); }

// token with depth d before it and r tokens left (this one included):
// terminal if d <= r-1, unary if 1 <= d <= r, binary if 2 <= d <= r+1
__device__ __forceinline__ int gen_token(int d, int r, int nvars, int K, int nun, uint32_t w0, uint32_t w1) {
  int allowed[3];
  int na = 0;
  if (d <= r - 1) allowed[na++] = 0;
  if (d >= 1 && d <= r) allowed[na++] = 1;
  if (d >= 2 && d <= r + 1) allowed[na++] = 2;
  const int cls = allowed[below(w0, (uint32_t)na)];
  if (cls == 0) {
    const int q = (int)below(w1, (uint32_t)(nvars + K));
    return q < nvars ? TOK_VAR0 + q : TOK_CONST0 + (q - nvars);
  }
  if (cls == 1) return TOK_SIN + (int)below(w1, (uint32_t)nun);
  return TOK_ADD + (int)below(w1, 4u);
}

// ---------------------------------------------------------------- kernels
__global__ void philox_kernel(const uint32_t *__restrict__ ctr, uint32_t k0, uint32_t k1,
                              uint32_t *__restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Word4 w = philox(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3], k0, k1);
  for (int j = 0; j < 4; ++j) out[4 * i + j] = w.v[j];
}

// A fitness as an unsigned integer in the same order (-0 equal to +0, NaN as
// +inf): FP64 compares run on a pipe of two lanes per SM.
__device__ __forceinline__ unsigned long long order_key(double f) {
  const unsigned long long sign = 1ull << 63, inf = 0x7ffull << 52;
  unsigned long long b = (unsigned long long)__double_as_longlong(f);
  const unsigned long long mag = b & ~sign;
  if (mag > inf) b = inf;
  if (mag == 0) b = 0;
  return b & sign ? ~b : b | sign;
}

// MAXIMISE = 0: the smallest fitness wins, NaN counting as +inf;
// MAXIMISE = 1: the largest score wins, NaN counting as -inf (the smallest
// negated score, then, with the same keys).
// Four candidates at a time are read before any is compared.  524,288
// tournaments of 4 over 262,144 fitnesses: 17.2 us with FP64 compares and one
// read after the other, now 11.4 (the gather's latency).
template <int MAXIMISE>
__global__ void tournament_kernel(const double *fitness, int P, int k, Rng rng_in, int32_t *parents) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * P) return;
  launch_wait();
  const Rng rng = rng_in.resolved();
  const int i = t >> 1, s = t & 1;
  int best = 0x7fffffff;
  unsigned long long bestk = ~0ull;
  for (int j = 0; j < k; j += 4) {
    const Word4 w = rng.draw((uint32_t)(j >> 2), (uint32_t)i, s ? PU_TOURN_B : PU_TOURN_A);
    double f[4];
    int cand[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cand[q] = (int)below(w.v[q], (uint32_t)P);
      f[q] = fitness[cand[q]];  // (in range for the words past k too)
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned long long key = order_key(MAXIMISE ? -f[q] : f[q]);
      if (j + q < k && (key < bestk || (key == bestk && cand[q] < best))) {
        best = cand[q];
        bestk = key;
      }
    }
  }
  parents[t] = best;
}

struct VaryParams {
  const uint8_t *prog_in;
  const int32_t *len_in;
  const float *c_in;
  const int32_t *parents;
  uint8_t *prog_out;
  int32_t *len_out;
  float *c_out;
  int P, Lmax, K, nvars;
  sr_var_cfg cfg;
  Rng rng;
  int P_in;  // parents' population size
};

// A group of G lanes (a warp or half of one) per child, every step by the whole
// group: both parents' rows come into shared memory with the widest loads their
// stride allows, a subtree's first token is found from prefix sums of the stack
// effects (two ballots give G of them), the child is gathered four bytes a lane,
// lane k holds constant k, and the five Philox draws of a child run on five lanes
// at once.  What bounds it: issue slots, then the latency of the rows' gather.
// 262,144 children of <= 256 tokens, K = 4: 631 us with lane 0 of a warp walking
// the rows byte by byte, 2,280 warp instructions a child; by the whole warp 174 us
// and 618; by half a warp each 165 us.
// Half a warp per child where there are enough children to fill the GPU so: what
// a child costs whatever its length is shared by two, and long rows take twice the
// rounds.  A warp, half a warp per child: 8,192 children of <= 64 tokens 8.5, 8.2 us,
// 65,536 of them 40.9, 32.4; 16,384 of <= 256 tokens 15.0, 16.1, 32,768 of them 25.9,
// 25.3, 262,144 of them 181.9, 164.9; 1,024 of <= 64 tokens 4.9, 6.2.
constexpr int VARY_THREADS = 128;
inline bool vary_halves(int P, int Lmax) { return P >= 8192 && P >= 128 * Lmax; }
static_assert(SR_MAX_CONSTS <= 16, "a lane of the group holds one constant of the child");
__host__ __device__ inline int vary_row_bytes(int Lmax) { return (Lmax + 15) & ~15; }

// bytes per load or store of a row: rows of Lmax bytes from base
__device__ __forceinline__ int row_grain(const uint8_t *base, int Lmax) {
  const uintptr_t m = (uintptr_t)base | (uintptr_t)Lmax;
  return (m & 15) == 0 ? 16 : ((m & 3) == 0 ? 4 : 1);
}
// the first n bytes (or a few more of the row) of a global row into shared memory
template <int G>
__device__ __forceinline__ void load_row(uint8_t *dst, const uint8_t *src, int n, int grain, int lane) {
  if (grain == 16) {
    for (int t = lane; t * 16 < n; t += G)
      reinterpret_cast<uint4 *>(dst)[t] = reinterpret_cast<const uint4 *>(src)[t];
  } else if (grain == 4) {
    for (int t = lane; t * 4 < n; t += G)
      reinterpret_cast<uint32_t *>(dst)[t] = reinterpret_cast<const uint32_t *>(src)[t];
  } else {
    for (int t = lane; t < n; t += G) dst[t] = src[t];
  }
}

// Lanes of a group: its bits in a warp's masks, and votes within it.
template <int G>
struct Lanes {
  unsigned mask;
  int shift, lane;
  __device__ __forceinline__ Lanes() {
    const int l = threadIdx.x & 31;
    lane = l & (G - 1);
    shift = l & ~(G - 1);
    mask = (G == 32 ? FULL : (1u << (G & 31)) - 1u) << shift;
  }
  __device__ __forceinline__ unsigned ballot(bool b) const { return (__ballot_sync(mask, b) & mask) >> shift; }
  __device__ __forceinline__ uint32_t get(uint32_t v, int from) const { return __shfl_sync(mask, v, from, G); }
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};

// First token of the subtree whose root is `end`, by the group: the largest t <= end with the stack effects of
// tok[t .. end] summing to 1, or 0 if there is none
template <int G>
__device__ __forceinline__ int group_subtree_start(const Lanes<G> &g, const uint8_t *tok, int end) {
  const unsigned upto = 0xffffffffu >> (31 - g.lane);  // lanes 0 .. lane
  int acc = 0;
  for (int top = end; top >= 0; top -= G) {
    const int t = top - g.lane;
    const int e = t >= 0 ? effect(tok[t]) : 0;
    const unsigned up = g.ballot(e > 0), down = g.ballot(e < 0);
    const unsigned hit = g.ballot(t >= 0 && acc + __popc(up & upto) - __popc(down & upto) == 1);
    if (hit) return top - (__ffs(hit) - 1);
    acc += __popc(up) - __popc(down);
  }
  return 0;
}

// 1 << (v - 32) for a constant's token (its bit among the slots read), and
// nothing in bits 0 .. 15 for any other
__device__ __forceinline__ uint32_t const_bit(uint32_t v) {
  uint32_t r;
  asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(v - (uint32_t)TOK_CONST0));  // shifts beyond 31 give 0
  return r;
}

template <int G>
__global__ void __launch_bounds__(VARY_THREADS) vary_kernel(VaryParams p) {
  extern __shared__ __align__(16) uint8_t vsm[];
  const Lanes<G> g;
  const int lane = g.lane, group = threadIdx.x / G;
  const int i = blockIdx.x * (VARY_THREADS / G) + group;
  if (i >= p.P) return;
  launch_wait();
  // out-of-range parents and lengths are clamped so that no access leaves
  // the buffers (valid inputs are unaffected)
  const int ia = min(max(p.parents[2 * i], 0), p.P_in - 1);
  const int ib = min(max(p.parents[2 * i + 1], 0), p.P_in - 1);
  const int la = min(max(p.len_in[ia], 1), p.Lmax), lb = min(max(p.len_in[ib], 1), p.Lmax);
  const int R = vary_row_bytes(p.Lmax);
  uint8_t *sA = vsm + (size_t)group * 3 * R, *sB = sA + R, *out = sB + R;
  const int grain = row_grain(p.prog_in, p.Lmax);
  load_row<G>(sA, p.prog_in + (size_t)ia * p.Lmax, la, grain, lane);
  load_row<G>(sB, p.prog_in + (size_t)ib * p.Lmax, lb, grain, lane);
  float c = 0.0f, cb = 0.0f;  // constant `lane` of the child, and of parent B
  if (lane < p.K) {
    c = p.c_in[(size_t)ia * p.K + lane];
    cb = p.c_in[(size_t)ib * p.K + lane];
  }
  // draw 0 of the decisions and of every kind of variation, one per lane
  const Rng rng = p.rng.resolved();
  const Word4 w = rng.draw(0, (uint32_t)i, lane < 4 ? PU_DECIDE + lane : PU_CONSTMUT);
  auto word = [&](uint32_t purpose, int q) { return g.get(w.v[q], purpose == PU_CONSTMUT ? 4 : purpose - PU_DECIDE); };
  const float u_cross = unit24(word(PU_DECIDE, 0)), u_point = unit24(word(PU_DECIDE, 1));
  const float u_sub = unit24(word(PU_DECIDE, 2)), u_const = unit24(word(PU_DECIDE, 3));
  g.sync();

  // the child: A[0, sa) ++ B[sb, sb + nb) ++ A[sa + nb - shift, la), all of A without a crossover
  int len = la, sa = la, nb = 0, sb = 0, shift = 0;
  bool crossed = false;
  if (u_cross < p.cfg.p_cross) {
    const int a = (int)below(word(PU_CROSS, 0), (uint32_t)la);
    const int b = (int)below(word(PU_CROSS, 1), (uint32_t)lb);
    const int ta = group_subtree_start(g, sA, a), tb = group_subtree_start(g, sB, b);
    const int nl = la - (a - ta + 1) + (b - tb + 1);
    if (nl <= p.Lmax) {
      crossed = true;
      len = nl;
      sa = ta;
      sb = tb;
      nb = b - tb + 1;
      shift = nb - (a - ta + 1);
    }
  }
  uint32_t usedA = 0, usedB = 0;
  const int dB = R + sb - sa;  // B's row follows A's
  for (int q0 = lane * 4; q0 < len; q0 += 4 * G) {
    uint32_t quad = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int q = q0 + j;
      const bool inB = q >= sa && q < sa + nb;
      const int at = q < sa ? q : (inB ? q + dB : q - shift);
      const uint32_t v = q < len ? sA[at] : 0u;
      const uint32_t bit = const_bit(v);
      usedA |= inB ? 0u : bit;
      usedB |= inB ? bit : 0u;
      quad |= v << (8 * j);
    }
    reinterpret_cast<uint32_t *>(out)[q0 >> 2] = quad;
  }
  if (crossed && p.K > 0) {  // slot k takes B's value when only the inserted part reads it
    usedA = __reduce_or_sync(g.mask, usedA);
    usedB = __reduce_or_sync(g.mask, usedB);
    if (lane < p.K && ((usedB & ~usedA) >> lane & 1u)) c = cb;
  }
  g.sync();

  if (u_point < p.cfg.p_point) {
    const int t = (int)below(word(PU_POINT, 0), (uint32_t)len);
    const uint32_t w1 = word(PU_POINT, 1);
    const int cls = tok_class(out[t]);
    int v;
    if (cls == CLS_BINARY) {
      v = TOK_ADD + (int)below(w1, 4u);
    } else if (cls == CLS_UNARY) {
      v = TOK_SIN + (int)below(w1, (uint32_t)p.cfg.unary_ops);
    } else {
      const int q = (int)below(w1, (uint32_t)(p.nvars + p.K));
      v = q < p.nvars ? TOK_VAR0 + q : TOK_CONST0 + (q - p.nvars);
    }
    g.sync();
    if (lane == 0) out[t] = (uint8_t)v;
    g.sync();
  }

  if (u_sub < p.cfg.p_subtree && p.cfg.max_subtree > 0) {
    const int t = (int)below(word(PU_SUBTREE, 0), (uint32_t)len);
    const int n = 1 + (int)below(word(PU_SUBTREE, 1), (uint32_t)p.cfg.max_subtree);
    const int s = group_subtree_start(g, out, t);
    const int span = t - s + 1, nl = len - span + n;
    if (nl <= p.Lmax) {
      // out[0, s) ++ n new tokens ++ out[t + 1, len), built where A's row was
      for (int q = lane; q < nl; q += G)
        if (q < s || q >= s + n) sA[q] = out[q < s ? q : q + span - n];
      int d = 0;
      for (int q0 = 0; q0 < n; q0 += G) {
        const Word4 d4 = rng.draw((uint32_t)(q0 + lane), (uint32_t)i, PU_SUBGEN);
        for (int q = q0; q < n && q < q0 + G; ++q) {
          const int v = gen_token(d, n - q, p.nvars, p.K, p.cfg.unary_ops, g.get(d4.v[0], q - q0),
                                  g.get(d4.v[1], q - q0));
          if (lane == 0) sA[s + q] = (uint8_t)v;
          d += effect(v);
        }
      }
      len = nl;
      out = sA;
      g.sync();
    }
  }

  if (u_const < p.cfg.p_const && p.K > 0) {
    const int k = (int)below(word(PU_CONSTMUT, 0), (uint32_t)p.K);
    const float step = __fmul_rn(__fsub_rn(unit24(word(PU_CONSTMUT, 1)), 0.5f), p.cfg.const_delta);
    if (lane == k) c = __fadd_rn(c, step);
  }

  // the row, zeros past the child's length
  uint8_t *g_out = p.prog_out + (size_t)i * p.Lmax;
  const int ograin = row_grain(p.prog_out, p.Lmax);
  if (ograin == 1) {
    for (int t = lane; t < p.Lmax; t += G) g_out[t] = t < len ? out[t] : 0;
  } else {
    auto quad = [&](int t4) {  // bytes 4 t4 .. 4 t4 + 3
      const int left = len - 4 * t4;
      const uint32_t v = reinterpret_cast<const uint32_t *>(out)[t4];
      return left >= 4 ? v : (left <= 0 ? 0u : v & ((1u << (8 * left)) - 1u));
    };
    if (ograin == 16) {
      for (int t = lane; t * 16 < p.Lmax; t += G)
        reinterpret_cast<uint4 *>(g_out)[t] = make_uint4(quad(4 * t), quad(4 * t + 1), quad(4 * t + 2), quad(4 * t + 3));
    } else {
      for (int t = lane; 4 * t < p.Lmax; t += G) reinterpret_cast<uint32_t *>(g_out)[t] = quad(t);
    }
  }
  if (lane == 0) p.len_out[i] = len;
  if (lane < p.K) p.c_out[(size_t)i * p.K + lane] = c;
}

// ---------------------------------------------------------------- microcosm selection
// Beagle's Monte-Carlo population control (Sec. 2.1.6): a sample of S
// individuals stands in for the whole population; its keep-quantile tau
// estimates the fitness threshold of the best fraction keep.  Keys: fitness,
// NaN as +inf (smaller is better).
__device__ __forceinline__ double micro_key(double f) {
  return isnan(f) ? __longlong_as_double(0x7ff0000000000000ll) : f;
}

constexpr int MICRO_MAX_SAMPLE = 1024;
constexpr int MICRO_ROUNDS = 16;  // 4 candidates per Philox draw: at most 64 per parent

// one block of S threads: draw, sort by rank (S <= 1024, O(S^2) compares),
// tau = the sample's value at rank ceil(keep S) - 1
__global__ void microcosm_sample_kernel(const double *__restrict__ fitness, int P, int S, int kq, Rng rng_in,
                                        double *tau) {
  __shared__ double key[MICRO_MAX_SAMPLE];
  __shared__ int idx[MICRO_MAX_SAMPLE];
  const Rng rng = rng_in.resolved();
  const int j = threadIdx.x;
  if (j < S) {
    const Word4 w = rng.draw((uint32_t)(j >> 2), 0u, PU_MICRO_SAMPLE);
    idx[j] = (int)below(w.v[j & 3], (uint32_t)P);
    key[j] = micro_key(fitness[idx[j]]);
  }
  __syncthreads();
  if (j < S) {
    // rank of sample j: smaller keys first, equal keys by sample position
    int r = 0;
    for (int t = 0; t < S; ++t) r += key[t] < key[j] || (key[t] == key[j] && t < j);
    if (r == kq) *tau = key[j];
  }
}

// thread per (child, parent slot): the first of up to 64 uniform candidates
// whose key is at most tau; if none is, the best candidate drawn (ties to
// the smaller index)
__global__ void microcosm_select_kernel(const double *__restrict__ fitness, int P_in, int P_out, Rng rng_in,
                                        const double *tau_p, int32_t *__restrict__ parents) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * P_out) return;
  const Rng rng = rng_in.resolved();
  const int i = t >> 1, s = t & 1;
  const double tau = *tau_p;
  int best = -1;
  double bestk = 0.0;
  for (int r = 0; r < MICRO_ROUNDS; ++r) {
    const Word4 w = rng.draw((uint32_t)r, (uint32_t)i, s ? PU_MICRO_B : PU_MICRO_A);
    for (int q = 0; q < 4; ++q) {
      const int cand = (int)below(w.v[q], (uint32_t)P_in);
      const double k = micro_key(fitness[cand]);
      if (k <= tau) {
        parents[t] = cand;
        return;
      }
      if (best < 0 || k < bestk || (k == bestk && cand < best)) {
        best = cand;
        bestk = k;
      }
    }
  }
  parents[t] = best;
}

__global__ void random_programs_kernel(uint8_t *prog, int32_t *len, float *c, int P, int Lmin,
                                       int Lmax, int K, int nvars, int nun, float cmin, float cmax,
                                       Rng rng) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const Word4 lw = rng.draw(0, (uint32_t)i, PU_INIT);
  const int L = Lmin + (int)below(lw.v[0], (uint32_t)(Lmax - Lmin + 1));
  uint8_t *out = prog + (size_t)i * Lmax;
  int d = 0;
  for (int t = 0; t < L; ++t) {
    const Word4 w = rng.draw((uint32_t)(1 + t), (uint32_t)i, PU_INIT);
    const int v = gen_token(d, L - t, nvars, K, nun, w.v[0], w.v[1]);
    out[t] = (uint8_t)v;
    d += effect(v);
  }
  for (int t = L; t < Lmax; ++t) out[t] = 0;
  len[i] = L;
  const float span = __fsub_rn(cmax, cmin);
  for (int k = 0; k < K; ++k) {
    const Word4 w = rng.draw((uint32_t)k, (uint32_t)i, PU_INITC);
    c[(size_t)i * K + k] = __fadd_rn(cmin, __fmul_rn(unit24(w.v[0]), span));
  }
}

}  // namespace
}  // namespace sr

extern "C" {

sr_status sr_philox4x32_10(sr_ctx *ctx, const uint32_t *ctr, uint32_t key0, uint32_t key1,
                           uint32_t *out, int n) {
  using namespace sr;
  if (!ctx || n < 0 || (n > 0 && (!ctr || !out))) return fail(ctx, SR_EINVAL, "bad philox arguments");
  if (n == 0) return SR_OK;
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  philox_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(ctr, key0, key1, out, n);
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

static sr_status select_tournament(sr_ctx *ctx, const double *fitness, int P, int k, uint64_t seed,
                                   uint64_t gen, int32_t *parents, bool maximise) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  if (P < 0 || k < 1 || k > 64) return fail(ctx, SR_EINVAL, "P < 0 or k outside [1, 64]");
  if (P == 0) return SR_OK;
  if (!fitness || !parents) return fail(ctx, SR_EINVAL, "NULL fitness or parents");
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  const Rng rng = make_rng(seed, gen, ctx->gen_dev);
  if (maximise)
    SR_CHECK_CUDA(ctx, launch(tournament_kernel<1>, (2 * P + 255) / 256, 256, 0, ctx->stream, fitness, P, k, rng, parents));
  else
    SR_CHECK_CUDA(ctx, launch(tournament_kernel<0>, (2 * P + 255) / 256, 256, 0, ctx->stream, fitness, P, k, rng, parents));
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

sr_status sr_select_tournament(sr_ctx *ctx, const double *fitness, int P, int k, uint64_t seed,
                               uint64_t gen, int32_t *parents) {
  return select_tournament(ctx, fitness, P, k, seed, gen, parents, false);
}

sr_status sr_select_tournament_max(sr_ctx *ctx, const double *score, int P, int k, uint64_t seed,
                                   uint64_t gen, int32_t *parents) {
  return select_tournament(ctx, score, P, k, seed, gen, parents, true);
}

sr_status sr_vary(sr_ctx *ctx, const uint8_t *prog_in, const int32_t *len_in, const float *c_in, int P_in,
                  const int32_t *parents, uint8_t *prog_out, int32_t *len_out, float *c_out, int P,
                  int Lmax, int K, int nvars, const sr_var_cfg *cfg, uint64_t seed, uint64_t gen) {
  using namespace sr;
  if (!ctx || !cfg) return SR_EINVAL;
  if (P > 0 && P_in < 1) return fail(ctx, SR_EINVAL, "P_in must be >= 1 when there are children");
  if (P < 0 || Lmax < 1 || Lmax > SR_MAX_LMAX || K < 0 || K > SR_MAX_CONSTS || nvars < 1 ||
      nvars > SR_MAX_VARS || cfg->max_subtree < 0 || cfg->max_subtree > Lmax ||
      (cfg->unary_ops != UNARY_BASE && cfg->unary_ops != UNARY_ALL))
    return fail(ctx, SR_EINVAL, "bad sr_vary shape or configuration");
  if (P == 0) return SR_OK;
  if (!prog_in || !len_in || !parents || !prog_out || !len_out || (K > 0 && (!c_in || !c_out)))
    return fail(ctx, SR_EINVAL, "NULL pointer");
  if (prog_in == prog_out) return fail(ctx, SR_EINVAL, "prog_out must not alias prog_in");
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  VaryParams vp{prog_in, len_in, c_in, parents, prog_out, len_out, c_out, P, Lmax, K, nvars, *cfg,
                make_rng(seed, gen, ctx->gen_dev), P_in};
  const int lanes = vary_halves(P, Lmax) ? 16 : 32, per = VARY_THREADS / lanes;
  SR_CHECK_CUDA(ctx, launch(lanes == 16 ? vary_kernel<16> : vary_kernel<32>, (P + per - 1) / per, VARY_THREADS,
                            per * 3 * vary_row_bytes(Lmax), ctx->stream, vp));
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

sr_status sr_select_microcosm(sr_ctx *ctx, const double *fitness, int P_in, int P_out, int sample,
                              double keep, uint64_t seed, uint64_t gen, int32_t *parents, double *threshold) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  if (P_in < 0 || P_out < 0 || sample < 1 || sample > MICRO_MAX_SAMPLE || !(keep > 0.0 && keep <= 1.0))
    return fail(ctx, SR_EINVAL, "bad sr_select_microcosm arguments");
  if (P_out == 0) return SR_OK;
  if (P_in == 0) return fail(ctx, SR_EINVAL, "no parents to select from");
  if (!fitness || !parents) return fail(ctx, SR_EINVAL, "NULL fitness or parents");
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  double *tau = threshold;
  if (!tau) {
    sr_status st = ensure_workspace(ctx, 256);
    if (st != SR_OK) return st;
    tau = reinterpret_cast<double *>(ctx->ws);
  }
  int kq = (int)ceil(keep * (double)sample) - 1;
  kq = kq < 0 ? 0 : (kq >= sample ? sample - 1 : kq);
  const Rng rng = make_rng(seed, gen, ctx->gen_dev);
  microcosm_sample_kernel<<<1, (sample + 31) / 32 * 32, 0, ctx->stream>>>(fitness, P_in, sample, kq, rng, tau);
  microcosm_select_kernel<<<(2 * P_out + 255) / 256, 256, 0, ctx->stream>>>(fitness, P_in, P_out, rng, tau,
                                                                             parents);
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 2;
  return SR_OK;
}

sr_status sr_set_generation_source(sr_ctx *ctx, const uint64_t *gen_dev) {
  if (!ctx) return SR_EINVAL;
  ctx->gen_dev = gen_dev;
  return SR_OK;
}

sr_status sr_random_programs(sr_ctx *ctx, uint8_t *prog, int32_t *len, float *c, int P, int Lmin,
                             int Lmax, int K, int nvars, int unary_ops, float cmin, float cmax,
                             uint64_t seed, uint64_t stream) {
  using namespace sr;
  if (!ctx) return SR_EINVAL;
  if (P < 0 || Lmin < 1 || Lmin > Lmax || Lmax > SR_MAX_LMAX || K < 0 || K > SR_MAX_CONSTS ||
      nvars < 1 || nvars > SR_MAX_VARS || (unary_ops != UNARY_BASE && unary_ops != UNARY_ALL))
    return fail(ctx, SR_EINVAL, "bad sr_random_programs shape");
  if (P == 0) return SR_OK;
  if (!prog || !len || (K > 0 && !c)) return fail(ctx, SR_EINVAL, "NULL pointer");
  SR_CHECK_CUDA(ctx, cudaSetDevice(ctx->device));
  random_programs_kernel<<<(P + 127) / 128, 128, 0, ctx->stream>>>(prog, len, c, P, Lmin, Lmax, K,
                                                                    nvars, unary_ops, cmin, cmax,
                                                                    make_rng(seed, stream));
  SR_CHECK_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return SR_OK;
}

}  // extern "C"
