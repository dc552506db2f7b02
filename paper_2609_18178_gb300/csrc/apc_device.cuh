// Device arithmetic of the committed step: the AdamW element update in its
// fixed binary32 order and the splitmix64 digest term.
//
// Every result is that of separate round-to-nearest operations (__fmul_rn,
// __fadd_rn, __fsub_rn, __fsqrt_rn, __fdiv_rn), which the compiler never fuses
// into FMA; the library is also built with -fmad=false and without
// flush-to-zero.  adamw_group forms the same square roots and quotients from
// approximations with exact remainders.  The update is decoupled-weight-decay AdamW
// (the optimizer whose committed W, M, V the paper preserves, arxiv
// 2609.18178 Section III-A, Eq. 2) and the digest realises its bitwise rank
// state checks (Sections IV-F, IV-G).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include <type_traits>

#include "apc_internal.h"

namespace apc {

// The step's eight binary32 scalars, read where they are used.  In the
// kernels they point into the launch's __grid_constant__ parameter block, so
// every use is a constant-bank operand and holds no register.
struct Scalars {
  const float *h;        // b1, 1-b1, b2, 1-b2, eps, 1-lr*wd, lr/(1-b1^t), 1/sqrt(1-b2^t)
  const uint64_t *pair;  // both lanes of the packed operations' constants (kPair*)
  float limit;           // adamw_group's bound on |m'| + den, negative if its form does not apply
  uint32_t one;          // 1, from the launch parameters (see digest_term)
};

// One element: p, m, v updated in place, returns the bf16 bits of p'.
__device__ __forceinline__ uint32_t adamw_element(float &p, float &m, float &v, uint32_t g16, const Scalars &s) {
  const float g = __uint_as_float(g16 << 16);
  const float t1 = __fmul_rn(s.h[0], m);
  const float t2 = __fmul_rn(s.h[1], g);
  const float mn = __fadd_rn(t1, t2);
  const float gg = __fmul_rn(g, g);
  const float t3 = __fmul_rn(s.h[2], v);
  const float t4 = __fmul_rn(s.h[3], gg);
  const float vn = __fadd_rn(t3, t4);
  const float sq = __fsqrt_rn(vn);
  const float t5 = __fmul_rn(sq, s.h[7]);
  const float den = __fadd_rn(t5, s.h[4]);
  const float u = __fdiv_rn(mn, den);
  const float t6 = __fmul_rn(p, s.h[5]);
  const float t7 = __fmul_rn(s.h[6], u);
  const float pn = __fsub_rn(t6, t7);
  p = pn;
  m = mn;
  v = vn;
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(pn));
}

// Two binary32 values in one 64-bit register pair, lane 0 in the low half,
// for the packed two-lane multiply (mul.rn.f32x2): each lane is an IEEE
// binary32 multiply rounded to nearest even, subnormals kept, so it gives
// each lane the bits of the scalar multiply.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  return ((uint64_t)__float_as_uint(b) << 32) | __float_as_uint(a);
}
__device__ __forceinline__ float lane0(uint64_t x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float lane1(uint64_t x) { return __uint_as_float((uint32_t)(x >> 32)); }
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// adamw_element for N elements (2 or 4) at once, p, m, v in place: the same
// binary32 results, without the branches of the general square root and
// divide, which split the schedule at every element (and take their long side
// whenever some lane's m' is zero).  Multiplies and fused multiply-adds are
// packed over pairs of elements, two lanes an instruction.  The adds and the
// subtract stay scalar __fadd_rn / __fsub_rn: a packed product feeding a packed
// add was found contracted into a fused multiply-add by the assembler (a 1-ulp
// change in a quarter of the elements), while the scalar round-to-nearest adds
// are never fused.
//
// The commit kernel with it: 1.81 G elements of bf16 state 5,738 us (5,930 with
// the general operations), 152 M of fp32 state 655 (661), 60 M in misaligned
// entries 321 (377 where 1% of the moments are zero, 322 where none is).
//
// The square root and the quotient are formed in Markstein's way (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor",
// IBM J. Res. Dev. 34, 1990): an approximation, and a last step that adds its
// exact fused remainder times an approximate reciprocal.
//   root      x = v' * 2^64 + 2^-126 (the addend only counts for v' = 0),
//             y ~ 1/sqrt(x), g = x*y, sqrt(x) = g + (x - g*g) * (y/2)
//   quotient  a = m' * 2^64, y = 1/den rounded (one Newton step),
//             q = a*y, a/den = q + (a - q*den) * y
// with the signs arranged so that no operand needs a negation and a zero m'
// keeps its sign.  On this GPU both are the rounded results without exception:
// compared with the general ones for all 1.77e9 values of x in [2^-86, 2^125),
// for the reciprocal of all values in [2^-70, 2^31), and for the quotient of
// all 2^46 pairs of significands; other exponents only scale those, since
// nothing in the ranges below overflows or becomes subnormal.  (The tests repeat
// the root and the reciprocal for every significand, with 5e7 pairs for the
// quotient.)  The factors 2^64 keep it so down to subnormal v' and m'; the
// power-of-two scaled constants 1/sqrt(1-b2^t) * 2^-32 and lr/(1-b1^t) * 2^-64
// take them out again.
//
// The form holds if |m'| + den <= limit (up to 2^30, and negative where eps,
// 1/sqrt(1-b2^t) or lr/(1-b1^t) are out of range: commit_scalars) and if the
// quotient is not subnormal before its scaling back: |a/den| >= 2^-62, or the
// decayed parameter is at least 2^-62, against which such a quotient vanishes.
// One test over the group decides, by its sum of |m'| + den and its least
// |(1-lr*wd) * p| + |a/den|.  Masked and padded elements (p, m' and g zero) fail
// its second half although their quotient, a zero, is right: a second look,
// which only such groups take, lets them stay.  152 M elements of fp32 state
// with two of every four masked take 668 us (891 without the second look, 802
// with the general operations alone), all of them zero 667 (1,026, 929), none
// 648; of bf16 state 510 (704, 638), 510 (808, 741) and 493.  In a group that is
// left (infinities, NaNs, negative or huge moments, p and a nonzero m' both
// tiny) all elements take the general operations.
template <int N>
__device__ __forceinline__ void adamw_group(float (&p)[N], float (&m)[N], float (&v)[N], const uint32_t (&g16)[N],
                                            const Scalars &s) {
  float t6[N], t7[N], high = 0.0f, low = 0.0f;
#pragma unroll
  for (int j = 0; j < N; j += 2) {
    const uint64_t g = pack2(__uint_as_float(g16[j] << 16), __uint_as_float(g16[j + 1] << 16));
    const uint64_t t1 = mul2(s.pair[kPairB1], pack2(m[j], m[j + 1]));
    const uint64_t t2 = mul2(s.pair[kPair1B1], g);
    const uint64_t t3 = mul2(s.pair[kPairB2], pack2(v[j], v[j + 1]));
    const uint64_t t4 = mul2(s.pair[kPair1B2], mul2(g, g));
    m[j] = __fadd_rn(lane0(t1), lane0(t2));
    m[j + 1] = __fadd_rn(lane1(t1), lane1(t2));
    v[j] = __fadd_rn(lane0(t3), lane0(t4));
    v[j + 1] = __fadd_rn(lane1(t3), lane1(t4));
    const uint64_t nx = fma2(pack2(v[j], v[j + 1]), s.pair[kPairNeg64], s.pair[kPairNegTiny]);  // -x
    const uint64_t y = pack2(rsqrt_approx(-lane0(nx)), rsqrt_approx(-lane1(nx)));
    const uint64_t ng = mul2(nx, y);                                                       // -g
    const uint64_t nr = fma2(fma2(ng, ng, nx), mul2(y, s.pair[kPairHalf]), ng);            // -sqrt(x)
    const uint64_t t5 = mul2(nr, s.pair[kPairRsb2]);
    const float den0 = __fadd_rn(lane0(t5), s.h[4]), den1 = __fadd_rn(lane1(t5), s.h[4]);
    const uint64_t d = pack2(den0, den1), n0 = pack2(rcp_approx(-den0), rcp_approx(-den1));
    const uint64_t n = fma2(fma2(d, n0, s.pair[kPairOne]), n0, n0);                        // -1/den
    const uint64_t na = mul2(pack2(m[j], m[j + 1]), s.pair[kPairNeg64]);                   // -a
    const uint64_t q = mul2(na, n);
    const uint64_t u = fma2(fma2(d, q, na), n, q);                                         // a/den
    const uint64_t a6 = mul2(pack2(p[j], p[j + 1]), s.pair[kPairDecay]), a7 = mul2(u, s.pair[kPairStep]);
    t6[j] = lane0(a6);
    t6[j + 1] = lane1(a6);
    t7[j] = lane0(a7);
    t7[j + 1] = lane1(a7);
    const float c = fminf(fabsf(t6[j]) + fabsf(lane0(u)), fabsf(t6[j + 1]) + fabsf(lane1(u)));
    low = j ? fminf(low, c) : c;
    high += (fabsf(m[j]) + den0) + (fabsf(m[j + 1]) + den1);
  }
  if (!(high <= s.limit && low >= 0x1p-61f)) {
    bool right = high <= s.limit;
#pragma unroll
    for (int j = 0; j < N; ++j) right = right && (m[j] == 0.0f || fabsf(t6[j]) >= 0x1p-61f);
    if (!right) {
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const float den = __fadd_rn(__fmul_rn(__fsqrt_rn(v[j]), s.h[7]), s.h[4]);
        t7[j] = __fmul_rn(s.h[6], __fdiv_rn(m[j], den));
      }
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) p[j] = __fsub_rn(t6[j], t7[j]);
}

// The two 64-bit multiplies of the splitmix64 finaliser, z * C mod 2^64 for
// a constant C = (chi : clo), in one of two instruction forms.  Which one is
// faster depends on the kernel around it (both give the same bits):
//  * MulWide: three multiply-adds, lo*clo widened, then lo*chi and hi*clo
//    added into the high word.  Fewest instructions; the commit kernel,
//    which is bound by instruction issue, runs 2.7% faster with it.
//  * MulCompiler: the compiler's own 64-bit multiply, one instruction more and
//    a shorter chain.  The verification pass's fp32 terms take MulWide first
//    and this one second: 453 M elements of fp32 state in 1,411 us, against
//    1,425 with this one twice, 1,419 with MulWide twice, 1,414 the other way
//    round.
struct MulWide {
  template <uint32_t CLO, uint32_t CHI>
  __device__ __forceinline__ static uint64_t mul(uint64_t z) {
    uint64_t r;
    asm("{\n\t.reg .u32 l, h, rl, rh;\n\t"
        "mov.b64 {l, h}, %1;\n\t"
        "mul.wide.u32 %0, l, %2;\n\t"
        "mov.b64 {rl, rh}, %0;\n\t"
        "mad.lo.u32 rh, l, %3, rh;\n\t"
        "mad.lo.u32 rh, h, %2, rh;\n\t"
        "mov.b64 %0, {rl, rh};\n\t}"
        : "=l"(r)
        : "l"(z), "n"(CLO), "n"(CHI));
    return r;
  }
};

struct MulCompiler {
  template <uint32_t CLO, uint32_t CHI>
  __device__ __forceinline__ static uint64_t mul(uint64_t z) {
    return z * (((uint64_t)CHI << 32) | CLO);
  }
};

// splitmix64 of the digest key (((G + K) mod 2^32) << 32) | bits: the first
// output of Vigna's SplitMix64 seeded with the key (golden-ratio increment,
// then the 30/27/31 xor-shift multiply finaliser).  K is a compile-time
// element offset from G.
//
// Instruction mix: the kernels are short of integer-ALU issue, so the 64-bit
// increment puts its high half on the FMA pipe as an extended-precision
// multiply-add: lo = bits + 0x7F4A7C15 sets the carry, then
// hi = one * (0x9E3779B9 + K) + G + carry, with `one` a launch parameter
// equal to 1 (so the assembler cannot turn it back into an ALU add) and the
// offset K folded into the immediate: (G + K) + 0x9E3779B9 and
// G + (0x9E3779B9 + K) are equal mod 2^32, and no add of K is issued.
//
// The first xor-shift needs hi >> 30, the top two bits of the incremented
// high word.  Callers that know them for a whole run of terms pass them as
// `hi_top` (see digest_term's four-argument form); otherwise they are
// computed here.
template <uint32_t K, class Mul1, class Mul2>
__device__ __forceinline__ uint64_t digest_term_core(uint32_t gidx, uint32_t bits, uint32_t one, bool have_top,
                                                     uint32_t hi_top) {
  uint32_t lo, hi;
  asm("add.cc.u32 %0, %2, 0x7F4A7C15;\n\t"
      "madc.lo.u32 %1, %4, %5, %3;"
      : "=r"(lo), "=r"(hi)
      : "r"(bits), "r"(gidx), "r"(one), "n"(0x9E3779B9u + K));
  const uint32_t l1 = lo ^ __funnelshift_r(lo, hi, 30);
  const uint32_t h1 = hi ^ (have_top ? hi_top : hi >> 30);
  uint64_t z = ((uint64_t)h1 << 32) | l1;
  z = Mul1::template mul<0x1CE4E5B9u, 0xBF58476Du>(z);
  z = Mul2::template mul<0x133111EBu, 0x94D049BBu>(z ^ (z >> 27));
  return z ^ (z >> 31);
}

template <uint32_t K = 0, class Mul1 = MulWide, class Mul2 = MulWide>
__device__ __forceinline__ uint64_t digest_term(uint32_t gidx, uint32_t bits, uint32_t one) {
  return digest_term_core<K, Mul1, Mul2>(gidx, bits, one, false, 0);
}

// The same term with hi >> 30 supplied: hi_top must equal the top two bits
// of gidx + 0x9E3779B9 + K + carry.  For terms whose keys G + K lie in
// [G0, G0 + R), every incremented high word lies in [B, B + R] with
// B = G0 + 0x9E3779B9 (the carry adds at most 1); when B and B + R have the
// same top two bits (top_bits_shared), those bits are B >> 30 for all of them.
template <uint32_t K = 0, class Mul1 = MulWide, class Mul2 = MulWide>
__device__ __forceinline__ uint64_t digest_term(uint32_t gidx, uint32_t bits, uint32_t one, uint32_t hi_top) {
  return digest_term_core<K, Mul1, Mul2>(gidx, bits, one, true, hi_top);
}

// splitmix64 terms of 16-bit words (bits < 2^16).  Their low key half plus
// 0x7F4A7C15 never carries and always has top bits 01, so after the
// increment lo = bits + 0x7F4A7C15, hi = gidx + 0x9E3779B9 + K, and the
// first xor-shift's low word is lo ^ ((hi << 2) | 1) = lo ^ (4 * hi + 1); `top`
// is hi >> 30, shared by the caller (digest_term's hi_top rule).
//
// Term of half HALF (0 low, 1 high) of two packed words.  The half is
// taken and the increment added by one two-way dot product (dp2a with a unit
// vector) in place of a mask or shift and an add.  The key's part is left to
// the compiler, which places it on either pipe and shares it between the three
// words of a bf16-state element (1.81 G elements in 5,693 us; 5,733 with
// explicit multiply-adds for it).  The keyed form below saves more
// instructions but spills at the bf16 layout's 72 registers and was no faster.
template <uint32_t K, int HALF>
__device__ __forceinline__ uint64_t digest_term_half(uint32_t gidx, uint32_t pair, uint32_t top) {
  const uint32_t lo = __dp2a_lo(pair, HALF ? 0x0100u : 0x0001u, 0x7F4A7C15u);
  const uint32_t hi = gidx + (0x9E3779B9u + K), m4 = 4 * hi + 1;
  const uint32_t l1 = lo ^ m4, h1 = hi ^ top;
  uint64_t z = ((uint64_t)h1 << 32) | l1;
  z = MulWide::template mul<0x1CE4E5B9u, 0xBF58476Du>(z);
  z = MulWide::template mul<0x133111EBu, 0x94D049BBu>(z ^ (z >> 27));
  return z ^ (z >> 31);
}

// The same term in a keyed form, for runs of 16-bit words whose key offsets
// differ by multiples of four: the key's two contributions to a term are
//   m4 = 4 * hi + 1   and   t = (hi ^ top) * 0x1CE4E5B9,
// the high half's part of the first multiply.  As top < 4 flips only the two
// low bits of hi, (hi + 4q) ^ top = (hi ^ top) + 4q, so one Key16 per residue
// mod 4 serves a whole run: offset OFF (a multiple of 4) adds 4 * OFF to m4
// and OFF * 0x1CE4E5B9 to t, one plain add each, in place of hi, m4, the xor
// with top and a multiply-add per term.
struct Key16 {
  uint32_t m4, t;
};

// Key16 of the index gidx.
__device__ __forceinline__ Key16 key16(uint32_t gidx, uint32_t one, uint32_t top) {
  uint32_t hi, m4;
  asm("mad.lo.u32 %0, %2, %4, %3;\n\t"
      "mad.lo.u32 %1, %0, 4, %2;"
      : "=r"(hi), "=r"(m4)
      : "r"(one), "r"(gidx), "n"(0x9E3779B9u));
  return Key16{m4, (hi ^ top) * 0x1CE4E5B9u};
}

// Term of half HALF (0 low, 1 high) of the packed words `pair`.  The half is
// taken and the increment added by one two-way dot product (dp2a with a unit
// vector), in place of a mask or shift and an add (4,234 to 4,065 us over
// 1.81 G elements of bf16 state).  The second multiply is the compiler's
// for the high halves and three multiply-adds for the low ones: with both
// integer pipes 77% busy that mix lets them interleave best (3,650 us; 3,669
// with multiply-adds for both, 3,681 with the compiler's for both, 3,741 with
// the two exchanged).
template <uint32_t OFF, int HALF>
__device__ __forceinline__ uint64_t digest_term_u16(const Key16 &k, uint32_t pair) {
  static_assert(OFF % 4 == 0, "a Key16 serves offsets of its own residue mod 4");
  const uint32_t lo = __dp2a_lo(pair, HALF ? 0x0100u : 0x0001u, 0x7F4A7C15u);
  const uint32_t l1 = lo ^ (k.m4 + 4u * OFF);
  uint64_t z;
  asm("{\n\t.reg .u32 rl, rh, u;\n\t"
      "mad.lo.u32 u, %1, %3, %4;\n\t"
      "mul.wide.u32 %0, %1, %2;\n\t"
      "mov.b64 {rl, rh}, %0;\n\t"
      "add.u32 rh, rh, u;\n\t"
      "mov.b64 %0, {rl, rh};\n\t}"
      : "=l"(z)
      : "r"(l1), "n"(0x1CE4E5B9u), "n"(0xBF58476Du), "r"(k.t + OFF * 0x1CE4E5B9u));
  z = std::conditional<HALF == 1, MulCompiler, MulWide>::type::template mul<0x133111EBu, 0x94D049BBu>(z ^ (z >> 27));
  return z ^ (z >> 31);
}

__device__ __forceinline__ bool top_bits_shared(uint32_t B, uint32_t R) { return ((B ^ (B + R)) >> 30) == 0; }

// acc += z (mod 2^64), with the high half's carry-add on the FMA pipe.  Used
// for single terms; pairs of terms are summed as acc += a + b, which the
// compiler folds into one three-input add per 32-bit half.
__device__ __forceinline__ void acc_add(uint64_t &acc, uint64_t z, uint32_t one) {
  uint32_t alo = (uint32_t)acc, ahi = (uint32_t)(acc >> 32);
  asm("add.cc.u32 %0, %0, %2;\n\t"
      "madc.lo.u32 %1, %3, %4, %1;"
      : "+r"(alo), "+r"(ahi)
      : "r"((uint32_t)z), "r"((uint32_t)(z >> 32)), "r"(one));
  acc = ((uint64_t)ahi << 32) | alo;
}

// The launches of one call form a chain (launch_plan): let the next one start,
// and wait until the ones before have completed and their writes are visible.
__device__ __forceinline__ void chain_start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Sum of a warp's values, in every lane.
__device__ __forceinline__ uint64_t warp_sum(uint64_t x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// Add a warp's running sums to its slot of the CTA's and clear them (slot -1: none yet).
__device__ __forceinline__ void flush(uint64_t &acc, int slot, unsigned long long *s_acc) {
  const uint64_t x = warp_sum(acc);
  if ((threadIdx.x & 31) == 0 && slot >= 0 && x) atomicAdd(&s_acc[slot], (unsigned long long)x);
  acc = 0;
}

// The entry of a launch plan whose tiles hold `tile`, at or after entry `lo`
// (the last one that begins at or before it: an entry without tiles begins
// where the next one does).
template <class Plan>
__device__ __forceinline__ uint32_t entry_of(const Plan &plan, uint32_t lo, uint64_t tile) {
  uint32_t hi = plan.count;  // e[lo].tile_begin <= tile, e[hi] beyond
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (plan.e[mid].tile_begin <= tile) lo = mid;
    else hi = mid;
  }
  return lo;
}

}  // namespace apc
