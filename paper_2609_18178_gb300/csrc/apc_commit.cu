// The fused committed-step kernel: AdamW over a chunk table of ragged
// tensors and the state digests, in one pass over HBM.  Two state layouts
// share the pipeline:
//  * F32State  -- fp32 master p and moments m, v, bf16 gradient g, and a bf16
//    working copy w of p'; four digests (p', m', v', w); 28 bytes per element
//    (p, m, v read and written, g read, w written).
//  * BF16State -- p, m, v kept in bf16 (the paper's setting, arxiv 2609.18178
//    Section IV-A "Workloads"): loaded exactly into binary32, updated in the
//    same fixed order, rounded once to bf16 (nearest even) at the store;
//    three digests (p', m', v'); 14 bytes per element.
// With ZERO (APC_COMMIT_ZERO_GRAD) each gradient tile is also overwritten
// with +0 once its copy has landed: 2 more bytes per element.
//
// Warp-specialized pipeline (one persistent CTA per SM by default):
//  * The producer warp walks the CTA's share of the launch's tiles (tile_walk;
//    a tile is up to L::kTile elements of one entry's 16-byte aligned body:
//    4,864 for fp32 state, 10,368 for bf16 state; less in small launches, where
//    the host chooses plan.tile for balance) and, for each, waits until a ring
//    stage is free and issues four bulk asynchronous copies -- p, m, v and g --
//    that complete on the stage's "full" mbarrier.  Loads never occupy consumer registers, and up
//    to L::kStages tiles per CTA are in flight.
//  * With each stage the producer also writes a 48-byte descriptor (the
//    tile's first-element addresses in p, m, v, w, g, its element count and
//    first digest index) into shared memory before arming the stage, so the
//    consumers never search the chunk table themselves.
//  * The consumer warps (19 for fp32 state, 27 for bf16 state) wait for a
//    stage, read its descriptor and their elements from shared memory
//    (thread t of C takes the groups 4kC+4t..4kC+4t+3 for k < L::kGroups, 2
//    for fp32 state and 3 for bf16 state, so both the shared-memory reads and
//    the global stores are contiguous across the warp), release the
//    stage to the producer, then apply AdamW, store the results with
//    streaming stores, and fold the digest terms into 64-bit registers.
//  * Entries whose buffers are not mutually 16-byte aligned run through the same
//    ring.  The usual case is a packed flat shard of odd-sized tensors, p, m and
//    v alike, beside gradients and copies with boundaries of their own: there
//    p, m and v keep their vectors, the producer copies the 16-byte blocks that
//    hold the tile's gradient, and the consumers read its words, and store the
//    copy's, at their own offsets.  Where p, m and v are at odds too, all four
//    are copied in blocks and every word is read and stored by itself,
//    lane-consecutive.  60 M elements in 291 odd entries take 275 us, 320
//    with every word by itself, 606 with element loads straight from global
//    memory (247 at the copy rate).  Tables without such an entry run an
//    instantiation without this code (MIS = false).
//  * What lies outside the tiles (fewer than 8 elements at each end of an aligned
//    entry, at most 15 of another, whole entries under 32 elements of the latter)
//    is done straight from global memory by the producer warp once it has issued
//    its copies, so that it costs the consumers nothing.
//  * At exit the CTA sums each digest (warp shuffles, shared memory) and adds
//    it into the caller's output with one 64-bit atomic; addition mod 2^64 is
//    order-free, so digests do not depend on grid size or table split.
//
// Every mbarrier wait is bounded (apc_tma.cuh).  A wait that gives up sets
// the translation unit's device status word, makes the CTA stop issuing and
// consuming, drains the copies already issued (bounded again) and returns.
#include <cuda_runtime.h>

#include <atomic>

#include "../../include/apc.h"
#include "apc_device.cuh"
#include "apc_internal.h"
#include "apc_launch.cuh"
#include "apc_tma.cuh"

namespace apc {
namespace {

__device__ unsigned int g_commit_status;

struct Acc {
  uint64_t p, m, v, w;
};

__device__ __forceinline__ uint64_t umin64(uint64_t a, uint64_t b) { return a < b ? a : b; }

__device__ __forceinline__ void fail_wait(int *abort_flag) {
  atomicOr(&g_commit_status, (unsigned)APC_ETIMEOUT);
  *(volatile int *)abort_flag = 1;
}

__device__ __forceinline__ uint32_t bf16_rne_bits(float x) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}

__device__ __forceinline__ float bf16_value(uint32_t h) { return __uint_as_float(h << 16); }

// Two binary32 values rounded to bf16 (nearest even) by one paired
// conversion, `lo` in the low half: each half equals bf16_rne_bits of its
// input for every non-NaN value.  The digest takes each half straight from
// the pair (hterm).
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}

// A consumer thread's output addresses in the current tile: element
// start + 4t of the entry (t the consumer index).  Group k of the thread then
// sits at a compile-time element offset k * 4 * L::kConsumers, which the
// stores carry as an immediate.
struct Dst {
  void *p, *m, *v;
  uint16_t *w, *g;
};

// What the consumers need of a stage's tile, written into shared memory by
// the producer before it arms the stage's "full" barrier (whose completion
// makes it visible to them): the addresses of the tile's first element in
// p, m, v, w and g, its element count and its first digest index.  The
// consumers then spend no instructions locating the tile in the chunk table.
// Where the entry's buffers are not mutually aligned, cnt also holds, from bit 16
// on, four bits each: the byte offsets of the tile's first element in the
// staged blocks of p, m, v and g; and kMisTile, or kHalfTile if only the
// gradient and the copy are at odds with p, m and v.
struct __align__(16) StageDesc {
  uint8_t *p, *m, *v;
  uint16_t *w, *g;
  uint32_t cnt, G;
};
constexpr uint32_t kMisTile = 1u << 15, kHalfTile = 1u << 14, kCntMask = kHalfTile - 1;
static_assert(kCommitTile <= kCntMask && kCommitTileBF16 <= kCntMask, "a tile's count and its flags share a word");

// Four 16-bit words at any 2-byte address.
__device__ __forceinline__ uint2 words4(const uint16_t *q) {
  return make_uint2((uint32_t)q[0] | (uint32_t)q[1] << 16, (uint32_t)q[2] | (uint32_t)q[3] << 16);
}
__device__ __forceinline__ void store_words4(uint16_t *q, uint2 x) {
  __stcs(q, (uint16_t)x.x);
  __stcs(q + 1, (uint16_t)(x.x >> 16));
  __stcs(q + 2, (uint16_t)x.y);
  __stcs(q + 3, (uint16_t)(x.y >> 16));
}
static_assert(sizeof(StageDesc) == 48, "three 16-byte shared-memory loads");

// A commit digest term.  With SHARED the caller has established that the
// whole group's terms share the top two bits of their incremented key high
// word (top_bits_shared) and passes them as `top`.
template <uint32_t K, bool SHARED>
__device__ __forceinline__ uint64_t cterm(uint32_t G, uint32_t bits, uint32_t one, uint32_t top) {
  if constexpr (SHARED) return digest_term<K>(G, bits, one, top);
  else return digest_term<K>(G, bits, one);
}

// The term of half HALF (0 low, 1 high) of a packed pair of 16-bit words (w,
// and the bf16 layout's p', m', v'): with the shared top bits, the 16-bit form
// that takes the half by a dot product.
template <uint32_t K, int HALF, bool SHARED>
__device__ __forceinline__ uint64_t hterm(uint32_t G, uint32_t pair, uint32_t one, uint32_t top) {
  if constexpr (SHARED) return digest_term_half<K, HALF>(G, pair, top);
  else return digest_term<K>(G, HALF ? pair >> 16 : pair & 0xFFFFu, one);
}

// ------------------------------------------------------------ fp32 state

struct F32State {
  static constexpr uint32_t kES = 4;        // bytes per state element
  static constexpr int kDigests = 4;
  static constexpr int kConsumerWarps = kCommitConsumerWarps;
  static constexpr int kStages = kCommitStages;
  static constexpr int kConsumers = 32 * kConsumerWarps;
  static constexpr int kThreads = kConsumers + 32;  // + the producer warp
  static constexpr int kBoundThreads = kThreads > APC_COMMIT_BOUND_THREADS ? kThreads : APC_COMMIT_BOUND_THREADS;
  static constexpr int kGroups = kCommitGroups;
  static constexpr uint64_t kTile = kCommitTile;
  static constexpr int kMisUnroll = 2;      // pairs of a misaligned tile at a time
  struct Regs {
    float4 p, m, v;
    uint2 g;
  };

  // PAD: bytes between the stage's regions (16 where misaligned tiles may come);
  // half: the gradient begins `goff` bytes into its region.
  template <uint32_t PAD>
  __device__ static void load(const uint8_t *st, uint32_t e, bool half, uint32_t goff, Regs &r) {
    r.p = *reinterpret_cast<const float4 *>(st + 4 * e);
    r.m = *reinterpret_cast<const float4 *>(st + 4 * (kTile + e) + PAD);
    r.v = *reinterpret_cast<const float4 *>(st + 4 * (2 * kTile + e) + 2 * PAD);
    const uint8_t *g = st + 12 * kTile + 2 * e + 3 * PAD;
    r.g = PAD && half ? words4(reinterpret_cast<const uint16_t *>(g + goff)) : *reinterpret_cast<const uint2 *>(g);
  }

  // Where a misaligned tile's elements sit in its stage.
  struct Mis {
    const float *p, *m, *v;
    const uint16_t *g;
    __device__ Mis(const uint8_t *st, uint32_t cnt) {
      p = reinterpret_cast<const float *>(st + (cnt >> 16 & 15));
      m = reinterpret_cast<const float *>(st + 4 * kTile + 16 + (cnt >> 20 & 15));
      v = reinterpret_cast<const float *>(st + 8 * kTile + 32 + (cnt >> 24 & 15));
      g = reinterpret_cast<const uint16_t *>(st + 12 * kTile + 48 + (cnt >> 28));
    }
  };

  // Elements e and e + kConsumers of a misaligned tile.
  template <bool ZERO>
  __device__ static void mis_pair(const StageDesc &sd, const Mis &x, uint32_t e, const Scalars &s, Acc &a) {
    const uint32_t f = e + kConsumers;
    float p[2] = {x.p[e], x.p[f]}, m[2] = {x.m[e], x.m[f]}, v[2] = {x.v[e], x.v[f]};
    const uint32_t gw[2] = {x.g[e], x.g[f]};
    adamw_group<2>(p, m, v, gw, s);
    const uint32_t w = pack_bf16x2(p[0], p[1]);
    mis_store<ZERO>(sd, e, p[0], m[0], v[0], w & 0xFFFFu);
    mis_store<ZERO>(sd, f, p[1], m[1], v[1], w >> 16);
    const uint32_t G = sd.G + e;
    a.p += digest_term<0>(G, __float_as_uint(p[0]), s.one) + digest_term<kConsumers>(G, __float_as_uint(p[1]), s.one);
    a.m += digest_term<0>(G, __float_as_uint(m[0]), s.one) + digest_term<kConsumers>(G, __float_as_uint(m[1]), s.one);
    a.v += digest_term<0>(G, __float_as_uint(v[0]), s.one) + digest_term<kConsumers>(G, __float_as_uint(v[1]), s.one);
    a.w += digest_term<0>(G, w & 0xFFFFu, s.one) + digest_term<kConsumers>(G, w >> 16, s.one);
  }

  // Element e of a misaligned tile.
  template <bool ZERO>
  __device__ static void mis_one(const StageDesc &sd, const Mis &x, uint32_t e, const Scalars &s, Acc &a) {
    float p = x.p[e], m = x.m[e], v = x.v[e];
    const uint32_t w = adamw_element(p, m, v, x.g[e], s), G = sd.G + e;
    mis_store<ZERO>(sd, e, p, m, v, w);
    acc_add(a.p, digest_term(G, __float_as_uint(p), s.one), s.one);
    acc_add(a.m, digest_term(G, __float_as_uint(m), s.one), s.one);
    acc_add(a.v, digest_term(G, __float_as_uint(v), s.one), s.one);
    acc_add(a.w, digest_term(G, w, s.one), s.one);
  }

  template <bool ZERO>
  __device__ __forceinline__ static void mis_store(const StageDesc &sd, uint32_t e, float p, float m, float v, uint32_t w) {
    __stcs(reinterpret_cast<float *>(sd.p) + e, p);
    __stcs(reinterpret_cast<float *>(sd.m) + e, m);
    __stcs(reinterpret_cast<float *>(sd.v) + e, v);
    __stcs(sd.w + e, (uint16_t)w);
    if (ZERO) __stcs(sd.g + e, (uint16_t)0);
  }

  // Four consecutive elements at the compile-time element offset OFF from
  // the thread's output addresses, whose first element has digest index G.
  template <uint32_t OFF, bool ZERO, bool MIS>
  __device__ static void compute_store(const Dst &d, uint32_t G, const Regs &r, bool half, const Scalars &s, Acc &a) {
    constexpr uint32_t off = OFF;
    float p[4] = {r.p.x, r.p.y, r.p.z, r.p.w};
    float m[4] = {r.m.x, r.m.y, r.m.z, r.m.w};
    float v[4] = {r.v.x, r.v.y, r.v.z, r.v.w};
    const uint32_t gw[4] = {r.g.x & 0xFFFFu, r.g.x >> 16, r.g.y & 0xFFFFu, r.g.y >> 16};
    if constexpr (ZERO) {
      // bound by its 30 bytes per element: the grouped form, with fewer
      // instructions, measured slower here (453 M elements in 2,150 us
      // against 2,043)
#pragma unroll
      for (int j = 0; j < 4; ++j) (void)adamw_element(p[j], m[j], v[j], gw[j], s);
    } else {
      adamw_group<4>(p, m, v, gw, s);
    }
    __stcs(reinterpret_cast<float4 *>(static_cast<float *>(d.p) + off), make_float4(p[0], p[1], p[2], p[3]));
    __stcs(reinterpret_cast<float4 *>(static_cast<float *>(d.m) + off), make_float4(m[0], m[1], m[2], m[3]));
    __stcs(reinterpret_cast<float4 *>(static_cast<float *>(d.v) + off), make_float4(v[0], v[1], v[2], v[3]));
    const uint32_t w01 = pack_bf16x2(p[0], p[1]), w23 = pack_bf16x2(p[2], p[3]);
    if (MIS && half) store_words4(d.w + off, make_uint2(w01, w23));
    else __stcs(reinterpret_cast<uint2 *>(d.w + off), make_uint2(w01, w23));
    // the group's keys are G + OFF .. G + OFF + 3
    const uint32_t B = G + (0x9E3779B9u + OFF);
    const uint32_t pb[4] = {__float_as_uint(p[0]), __float_as_uint(p[1]), __float_as_uint(p[2]), __float_as_uint(p[3])};
    const uint32_t mb[4] = {__float_as_uint(m[0]), __float_as_uint(m[1]), __float_as_uint(m[2]), __float_as_uint(m[3])};
    const uint32_t vb[4] = {__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3])};
    if (top_bits_shared(B, 4)) {
      fold<OFF, true>(G, pb, mb, vb, w01, w23, s.one, B >> 30, a);
    } else {
      fold<OFF, false>(G, pb, mb, vb, w01, w23, s.one, 0, a);
    }
  }

  template <uint32_t OFF, bool SHARED>
  __device__ static void fold(uint32_t G, const uint32_t (&p)[4], const uint32_t (&m)[4], const uint32_t (&v)[4],
                              uint32_t w01, uint32_t w23, uint32_t one, uint32_t top, Acc &a) {
    a.p += cterm<OFF, SHARED>(G, p[0], one, top) + cterm<OFF + 1, SHARED>(G, p[1], one, top);
    a.p += cterm<OFF + 2, SHARED>(G, p[2], one, top) + cterm<OFF + 3, SHARED>(G, p[3], one, top);
    a.m += cterm<OFF, SHARED>(G, m[0], one, top) + cterm<OFF + 1, SHARED>(G, m[1], one, top);
    a.m += cterm<OFF + 2, SHARED>(G, m[2], one, top) + cterm<OFF + 3, SHARED>(G, m[3], one, top);
    a.v += cterm<OFF, SHARED>(G, v[0], one, top) + cterm<OFF + 1, SHARED>(G, v[1], one, top);
    a.v += cterm<OFF + 2, SHARED>(G, v[2], one, top) + cterm<OFF + 3, SHARED>(G, v[3], one, top);
    a.w += hterm<OFF, 0, SHARED>(G, w01, one, top) + hterm<OFF + 1, 1, SHARED>(G, w01, one, top);
    a.w += hterm<OFF + 2, 0, SHARED>(G, w23, one, top) + hterm<OFF + 3, 1, SHARED>(G, w23, one, top);
  }

  __device__ static void one(const CommitEntry &E, uint64_t i, const Scalars &s, Acc &a) {
    float *P = static_cast<float *>(E.p), *M = static_cast<float *>(E.m), *V = static_cast<float *>(E.v);
    float p = P[i], m = M[i], v = V[i];
    const uint32_t w = adamw_element(p, m, v, (uint32_t)E.g[i], s);
    P[i] = p;
    M[i] = m;
    V[i] = v;
    E.w[i] = (uint16_t)w;
    const uint32_t G = E.key_base + (uint32_t)i;
    acc_add(a.p, digest_term(G, __float_as_uint(p), s.one), s.one);
    acc_add(a.m, digest_term(G, __float_as_uint(m), s.one), s.one);
    acc_add(a.v, digest_term(G, __float_as_uint(v), s.one), s.one);
    acc_add(a.w, digest_term(G, w, s.one), s.one);
  }
};

// ------------------------------------------------------------ bf16 state

struct BF16State {
  static constexpr uint32_t kES = 2;
  static constexpr int kDigests = 3;
  static constexpr int kConsumerWarps = kCommitConsumerWarpsBF16;
  static constexpr int kStages = kCommitStagesBF16;
  static constexpr int kConsumers = 32 * kConsumerWarps;
  static constexpr int kThreads = kConsumers + 32;
  static constexpr int kBoundThreads = kThreads;
  static constexpr int kGroups = kCommitGroupsBF16;
  static constexpr uint64_t kTile = kCommitTileBF16;
  static constexpr int kMisUnroll = 1;      // two spill at 72 registers
  struct Regs {
    uint2 p, m, v, g;
  };

  template <uint32_t PAD>
  __device__ static void load(const uint8_t *st, uint32_t e, bool half, uint32_t goff, Regs &r) {
    r.p = *reinterpret_cast<const uint2 *>(st + 2 * e);
    r.m = *reinterpret_cast<const uint2 *>(st + 2 * (kTile + e) + PAD);
    r.v = *reinterpret_cast<const uint2 *>(st + 2 * (2 * kTile + e) + 2 * PAD);
    const uint8_t *g = st + 6 * kTile + 2 * e + 3 * PAD;
    r.g = PAD && half ? words4(reinterpret_cast<const uint16_t *>(g + goff)) : *reinterpret_cast<const uint2 *>(g);
  }

  struct Mis {
    const uint16_t *p, *m, *v, *g;
    __device__ Mis(const uint8_t *st, uint32_t cnt) {
      p = reinterpret_cast<const uint16_t *>(st + (cnt >> 16 & 15));
      m = reinterpret_cast<const uint16_t *>(st + 2 * kTile + 16 + (cnt >> 20 & 15));
      v = reinterpret_cast<const uint16_t *>(st + 4 * kTile + 32 + (cnt >> 24 & 15));
      g = reinterpret_cast<const uint16_t *>(st + 6 * kTile + 48 + (cnt >> 28));
    }
  };

  template <bool ZERO>
  __device__ static void mis_pair(const StageDesc &sd, const Mis &x, uint32_t e, const Scalars &s, Acc &a) {
    const uint32_t f = e + kConsumers;
    float pf[2] = {bf16_value(x.p[e]), bf16_value(x.p[f])}, mf[2] = {bf16_value(x.m[e]), bf16_value(x.m[f])};
    float vf[2] = {bf16_value(x.v[e]), bf16_value(x.v[f])};
    const uint32_t gw[2] = {x.g[e], x.g[f]};
    adamw_group<2>(pf, mf, vf, gw, s);
    const uint32_t p = pack_bf16x2(pf[0], pf[1]), m = pack_bf16x2(mf[0], mf[1]), v = pack_bf16x2(vf[0], vf[1]);
    mis_store<ZERO>(sd, e, p & 0xFFFFu, m & 0xFFFFu, v & 0xFFFFu);
    mis_store<ZERO>(sd, f, p >> 16, m >> 16, v >> 16);
    const uint32_t G = sd.G + e;
    a.p += digest_term<0>(G, p & 0xFFFFu, s.one) + digest_term<kConsumers>(G, p >> 16, s.one);
    a.m += digest_term<0>(G, m & 0xFFFFu, s.one) + digest_term<kConsumers>(G, m >> 16, s.one);
    a.v += digest_term<0>(G, v & 0xFFFFu, s.one) + digest_term<kConsumers>(G, v >> 16, s.one);
  }

  template <bool ZERO>
  __device__ static void mis_one(const StageDesc &sd, const Mis &x, uint32_t e, const Scalars &s, Acc &a) {
    float p = bf16_value(x.p[e]), m = bf16_value(x.m[e]), v = bf16_value(x.v[e]);
    const uint32_t po = adamw_element(p, m, v, x.g[e], s), mo = bf16_rne_bits(m), vo = bf16_rne_bits(v);
    mis_store<ZERO>(sd, e, po, mo, vo);
    const uint32_t G = sd.G + e;
    acc_add(a.p, digest_term(G, po, s.one), s.one);
    acc_add(a.m, digest_term(G, mo, s.one), s.one);
    acc_add(a.v, digest_term(G, vo, s.one), s.one);
  }

  template <bool ZERO>
  __device__ __forceinline__ static void mis_store(const StageDesc &sd, uint32_t e, uint32_t p, uint32_t m, uint32_t v) {
    __stcs(reinterpret_cast<uint16_t *>(sd.p) + e, (uint16_t)p);
    __stcs(reinterpret_cast<uint16_t *>(sd.m) + e, (uint16_t)m);
    __stcs(reinterpret_cast<uint16_t *>(sd.v) + e, (uint16_t)v);
    if (ZERO) __stcs(sd.g + e, (uint16_t)0);
  }

  template <uint32_t OFF, bool ZERO, bool MIS>
  __device__ static void compute_store(const Dst &d, uint32_t G, const Regs &r, bool half, const Scalars &s, Acc &a) {
    constexpr uint32_t off = OFF;
    const uint32_t pw[4] = {r.p.x & 0xFFFFu, r.p.x >> 16, r.p.y & 0xFFFFu, r.p.y >> 16};
    const uint32_t mw[4] = {r.m.x & 0xFFFFu, r.m.x >> 16, r.m.y & 0xFFFFu, r.m.y >> 16};
    const uint32_t vw[4] = {r.v.x & 0xFFFFu, r.v.x >> 16, r.v.y & 0xFFFFu, r.v.y >> 16};
    const uint32_t gw[4] = {r.g.x & 0xFFFFu, r.g.x >> 16, r.g.y & 0xFFFFu, r.g.y >> 16};
    float pf[4], mf[4], vf[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      pf[j] = bf16_value(pw[j]);
      mf[j] = bf16_value(mw[j]);
      vf[j] = bf16_value(vw[j]);
    }
    adamw_group<4>(pf, mf, vf, gw, s);
    const uint32_t p01 = pack_bf16x2(pf[0], pf[1]), p23 = pack_bf16x2(pf[2], pf[3]);
    const uint32_t m01 = pack_bf16x2(mf[0], mf[1]), m23 = pack_bf16x2(mf[2], mf[3]);
    const uint32_t v01 = pack_bf16x2(vf[0], vf[1]), v23 = pack_bf16x2(vf[2], vf[3]);
    __stcs(reinterpret_cast<uint2 *>(static_cast<uint16_t *>(d.p) + off), make_uint2(p01, p23));
    __stcs(reinterpret_cast<uint2 *>(static_cast<uint16_t *>(d.m) + off), make_uint2(m01, m23));
    __stcs(reinterpret_cast<uint2 *>(static_cast<uint16_t *>(d.v) + off), make_uint2(v01, v23));
    const uint32_t B = G + (0x9E3779B9u + OFF);  // the group's keys are G + OFF .. G + OFF + 3
    if (top_bits_shared(B, 4)) {
      fold2<OFF, true>(G, p01, m01, v01, s.one, B >> 30, a);
      fold2<OFF + 2, true>(G, p23, m23, v23, s.one, B >> 30, a);
    } else {
      fold2<OFF, false>(G, p01, m01, v01, s.one, 0, a);
      fold2<OFF + 2, false>(G, p23, m23, v23, s.one, 0, a);
    }
  }

  template <uint32_t K, bool SHARED>
  __device__ __forceinline__ static void fold2(uint32_t G, uint32_t p, uint32_t m, uint32_t v, uint32_t one, uint32_t top, Acc &a) {
    a.p += hterm<K, 0, SHARED>(G, p, one, top) + hterm<K + 1, 1, SHARED>(G, p, one, top);
    a.m += hterm<K, 0, SHARED>(G, m, one, top) + hterm<K + 1, 1, SHARED>(G, m, one, top);
    a.v += hterm<K, 0, SHARED>(G, v, one, top) + hterm<K + 1, 1, SHARED>(G, v, one, top);
  }

  __device__ static void one(const CommitEntry &E, uint64_t i, const Scalars &s, Acc &a) {
    uint16_t *P = static_cast<uint16_t *>(E.p), *M = static_cast<uint16_t *>(E.m), *V = static_cast<uint16_t *>(E.v);
    float p = bf16_value(P[i]), m = bf16_value(M[i]), v = bf16_value(V[i]);
    const uint32_t po = adamw_element(p, m, v, (uint32_t)E.g[i], s);
    const uint32_t mo = bf16_rne_bits(m), vo = bf16_rne_bits(v);
    P[i] = (uint16_t)po;
    M[i] = (uint16_t)mo;
    V[i] = (uint16_t)vo;
    const uint32_t G = E.key_base + (uint32_t)i;
    acc_add(a.p, digest_term(G, po, s.one), s.one);
    acc_add(a.m, digest_term(G, mo, s.one), s.one);
    acc_add(a.v, digest_term(G, vo, s.one), s.one);
  }
};

// Group K of a consumer thread's tile: its elements sit at the compile-time
// offset K * 4 * L::kConsumers from the thread's output addresses, which
// the stores carry as immediates and the digest terms fold into their
// increment.
template <class L, bool ZERO, bool MIS, int K>
__device__ __forceinline__ void store_groups(const Dst &d, uint32_t G1, const typename L::Regs *r, const bool *ok, bool half,
                                             const Scalars &s, Acc &a) {
  constexpr uint32_t off = (uint32_t)(K * L::kConsumers) * 4;
  if (ok[K]) {
    if (ZERO) {
      if (MIS && half) store_words4(d.g + off, make_uint2(0u, 0u));
      else __stcs(reinterpret_cast<uint2 *>(d.g + off), make_uint2(0u, 0u));
    }
    L::template compute_store<off, ZERO, MIS>(d, G1, r[K], half, s, a);
  }
  if constexpr (K + 1 < L::kGroups) store_groups<L, ZERO, MIS, K + 1>(d, G1, r, ok, half, s, a);
}

// The stage's four regions; with MIS each has 16 bytes more, for the blocks
// that a misaligned tile begins and ends in.
template <class L, bool MIS>
__host__ __device__ constexpr uint32_t stage_bytes() {
  return (uint32_t)L::kTile * (3 * L::kES + 2) + (MIS ? 64 : 0);
}

template <class L, bool MIS>
__host__ __device__ constexpr uint32_t smem_bytes() {
  return (uint32_t)L::kStages * stage_bytes<L, MIS>();
}
static_assert(smem_bytes<F32State, true>() <= 226 * 1024 && smem_bytes<BF16State, true>() <= 226 * 1024,
              "shared memory per CTA");

// Copy the 16-byte blocks that hold `bytes` bytes from `src` on into the
// region at `dst`; the offset of the first byte in it is src % 16.
__device__ __forceinline__ void copy_blocks(uint8_t *dst, const uint8_t *src, uint32_t bytes, uint64_t *bar,
                                            uint64_t policy) {
  const uint32_t off = (uint32_t)((uintptr_t)src & 15);
  bulk_g2s(dst, src - off, (off + bytes + 15) & ~15u, bar, policy);
}

// The entry of a later tile of a walk that is at entry `cur`.
template <int MAXE>
__device__ __forceinline__ uint32_t next_entry(const CommitPlan<MAXE> &plan, uint32_t cur, uint64_t tile) {
  return cur + 1 < plan.count && tile >= plan.e[cur + 1].tile_begin ? entry_of(plan, cur + 1, tile) : cur;
}

// This CTA's tiles: tile = t0, t0 + ts, ... while tile < t1 (the same walk
// for the producer and the consumers).  With SWEEP the CTAs sweep the table
// together, CTA b taking tiles b, b + grid, ...; otherwise each takes one
// contiguous run (the runs differ by at most one tile).  Measured, in us, swept
// and in runs: fp32 state 152 M elements 649 and 656, 453 M 1,894 and 1,910,
// 16 M 78.7 and 80.5, 60 M misaligned 275 and 279, 7.25 G 30,330 and 30,355 on
// one GPU, 30,645 and 30,543 on another; with
// zeroed gradients 453 M of fp32 state 2,052 and 2,049, of bf16 state 1,440 and
// 1,461; bf16 state without them, the one bound by issue and not by memory,
// 1.81 G 5,695 and 5,682.
struct TileWalk {
  uint64_t t0, t1, ts;
};
template <bool SWEEP>
__device__ __forceinline__ TileWalk tile_walk(uint64_t total) {
  const uint64_t b = blockIdx.x;
  if (SWEEP) return {b, total, gridDim.x};
  const uint64_t per = total / gridDim.x, rem = total % gridDim.x;
  const uint64_t t0 = b * per + (b < rem ? b : rem);
  return {t0, t0 + per + (b < rem ? 1 : 0), 1};
}

template <class L, int MAXE, bool ZERO, bool MIS>
__global__ void __launch_bounds__(L::kBoundThreads, kCommitBlocksPerSm)
    commit_kernel(const __grid_constant__ CommitPlan<MAXE> plan, unsigned long long *out) {
  constexpr bool kSweep = L::kDigests == 4 || ZERO;  // all but bf16 state without zeroing
  constexpr uint32_t kPad = MIS ? 16 : 0, kStage = stage_bytes<L, MIS>();
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full[L::kStages];
  __shared__ __align__(8) uint64_t empty[L::kStages];
  __shared__ StageDesc desc[L::kStages];
  __shared__ uint64_t red[L::kDigests][L::kThreads / 32];
  __shared__ int abort_flag;

  if (plan.more) chain_start_next();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < L::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], L::kConsumerWarps);
    }
    abort_flag = 0;
    mbar_init_fence();
  }
  __syncthreads();

  Acc a{0, 0, 0, 0};
  if (warp == L::kConsumerWarps) {
    // ------------------------------------------------------------ producer
    const Scalars s{plan.h, plan.pair, plan.limit, plan.one};
    uint32_t phase = 0;
    int stage = 0;
    uint64_t issued = 0;
    if (lane == 0) {
      const uint64_t policy = l2_evict_first();
      const TileWalk w = tile_walk<kSweep>(plan.total_tiles);
      uint32_t cur = w.t0 < w.t1 ? entry_of(plan, 0, w.t0) : 0;
      for (uint64_t tile = w.t0; tile < w.t1; tile += w.ts) {
        if (*(volatile int *)&abort_flag) break;
        cur = next_entry(plan, cur, tile);
        const CommitEntry &E = plan.e[cur];
        const uint64_t start = E.head + (tile - E.tile_begin) * plan.tile;
        const uint32_t cnt = (uint32_t)umin64(plan.tile, E.head + E.body - start);
        if (!mbar_wait(&empty[stage], phase ^ 1)) {
          fail_wait(&abort_flag);
          break;
        }
        uint8_t *st = smem + (size_t)stage * kStage;
        uint8_t *const p = static_cast<uint8_t *>(E.p) + start * L::kES, *const m = static_cast<uint8_t *>(E.m) + start * L::kES,
                *const v = static_cast<uint8_t *>(E.v) + start * L::kES;
        uint16_t *const g = const_cast<uint16_t *>(E.g) + start;
        constexpr uint32_t kRegion = L::kES * (uint32_t)L::kTile + kPad;
        StageDesc sd{p, m, v, L::kDigests == 4 ? E.w + start : nullptr, g, cnt, E.key_base + (uint32_t)start};
        const auto off = [](const void *x) { return (uint32_t)((uintptr_t)x & 15); };
        const auto blocks = [&](const void *x, uint32_t bytes) { return (off(x) + bytes + 15) & ~15u; };
        if (MIS && E.mis == kMisAll) {
          sd.cnt |= kMisTile | off(p) << 16 | off(m) << 20 | off(v) << 24 | off(g) << 28;
          desc[stage] = sd;
          mbar_arrive_expect_tx(&full[stage], blocks(p, cnt * L::kES) + blocks(m, cnt * L::kES) +
                                                  blocks(v, cnt * L::kES) + blocks(g, cnt * 2));
          copy_blocks(st, p, cnt * L::kES, &full[stage], policy);
          copy_blocks(st + kRegion, m, cnt * L::kES, &full[stage], policy);
          copy_blocks(st + 2 * kRegion, v, cnt * L::kES, &full[stage], policy);
          copy_blocks(st + 3 * kRegion, reinterpret_cast<const uint8_t *>(g), cnt * 2, &full[stage], policy);
        } else {
          const bool half = MIS && E.mis == kMisGrad;
          if (half) sd.cnt |= kHalfTile | off(g) << 28;
          desc[stage] = sd;
          mbar_arrive_expect_tx(&full[stage], cnt * 3 * L::kES + (half ? blocks(g, cnt * 2) : cnt * 2));
          bulk_g2s(st, p, cnt * L::kES, &full[stage], policy);
          bulk_g2s(st + kRegion, m, cnt * L::kES, &full[stage], policy);
          bulk_g2s(st + 2 * kRegion, v, cnt * L::kES, &full[stage], policy);
          if (half) copy_blocks(st + 3 * kRegion, reinterpret_cast<const uint8_t *>(g), cnt * 2, &full[stage], policy);
          else bulk_g2s(st + 3 * kRegion, g, cnt * 2, &full[stage], policy);
        }
        ++issued;
        if (++stage == L::kStages) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    __syncwarp();
    // With its copies issued, the producer warp does what the entries hold
    // outside their tiles (at most 31 elements), one entry at a time.
    for (uint32_t e = blockIdx.x; e < plan.count; e += gridDim.x) {
      const CommitEntry &E = plan.e[e];
      if (lane < (uint32_t)(E.n - E.body)) {
        const uint64_t i = lane < E.head ? lane : lane + E.body;
        L::one(E, i, s, a);
        if (ZERO) const_cast<uint16_t *>(E.g)[i] = 0;
      }
    }
    if (lane == 0) {
      // Drain: the last min(issued, stages) copies must have landed before
      // the CTA may exit (normally the consumers already waited for them).
      const int n_drain = (int)umin64(issued, (uint64_t)L::kStages);
      for (int k = 0; k < n_drain; ++k) {
        if (--stage < 0) {
          stage = L::kStages - 1;
          phase ^= 1;
        }
        if (!mbar_wait(&full[stage], phase)) atomicOr(&g_commit_status, (unsigned)APC_ETIMEOUT);
      }
    }
    __syncwarp();
  } else {
    // ----------------------------------------------------------- consumers
    const Scalars s{plan.h, plan.pair, plan.limit, plan.one};
    const int ct = threadIdx.x;  // 0 .. L::kConsumers-1
    uint32_t phase = 0;
    int stage = 0;
    const TileWalk w = tile_walk<kSweep>(plan.total_tiles);
    for (uint64_t tile = w.t0; tile < w.t1; tile += w.ts) {
      if (!mbar_wait(&full[stage], phase)) {
        fail_wait(&abort_flag);
        break;
      }
      if (*(volatile int *)&abort_flag) break;
      const StageDesc sd = desc[stage];
      const uint8_t *st = smem + (size_t)stage * kStage;
      if (MIS && (sd.cnt & kMisTile)) {
        const uint32_t cnt = sd.cnt & kCntMask;
        const typename L::Mis x(st, sd.cnt);
        uint32_t e = ct;
#pragma unroll L::kMisUnroll
        for (; e + L::kConsumers < cnt; e += 2 * L::kConsumers) L::template mis_pair<ZERO>(sd, x, e, s, a);
        if (e < cnt) L::template mis_one<ZERO>(sd, x, e, s, a);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[stage]);
      } else {
        typename L::Regs r[L::kGroups];
        bool ok[L::kGroups];
        const bool half = MIS && (sd.cnt & kHalfTile);
        const uint32_t cnt = MIS ? sd.cnt & kCntMask : sd.cnt;
#pragma unroll
        for (int k = 0; k < L::kGroups; ++k) {
          const uint32_t e = (uint32_t)(k * L::kConsumers + ct) * 4;
          ok[k] = e < cnt;
          if (ok[k]) L::template load<kPad>(st, e, half, sd.cnt >> 28, r[k]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[stage]);
        // this thread's first element in the tile is element 4 * ct
        const uint32_t ob = 4u * (uint32_t)ct;
        const Dst d{sd.p + ob * L::kES, sd.m + ob * L::kES, sd.v + ob * L::kES,
                    L::kDigests == 4 ? sd.w + ob : nullptr, sd.g + ob};
        store_groups<L, ZERO, MIS, 0>(d, sd.G + ob, r, ok, half, s, a);
      }
      if (++stage == L::kStages) {
        stage = 0;
        phase ^= 1;
      }
    }
  }

  // each warp sums its lanes' digests; after one barrier warp d adds the
  // warps' sums of digest d into the output
  const uint64_t sums[4] = {warp_sum(a.p), warp_sum(a.m), warp_sum(a.v), L::kDigests == 4 ? warp_sum(a.w) : 0};
  if (lane == 0)
#pragma unroll
    for (int d = 0; d < L::kDigests; ++d) red[d][warp] = sums[d];
  __syncthreads();
  if (warp < L::kDigests) {
    const bool ok = !*(volatile int *)&abort_flag;
    const uint64_t r = warp_sum(lane < L::kThreads / 32 ? red[warp][lane] : 0);
    chain_wait();
    if (ok && lane == 0 && r) atomicAdd(&out[warp], (unsigned long long)r);
  }
}

// One thread waits on an mbarrier that nothing completes: the bounded wait
// must give up after `limit_ns` and record APC_ETIMEOUT.
__global__ void wait_timeout_kernel(uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  mbar_init(&bar, 1);
  mbar_init_fence();
  if (!mbar_wait(&bar, 0, limit_ns)) atomicOr(&g_commit_status, (unsigned)APC_ETIMEOUT);
}

// The dynamic shared-memory limit of one kernel instantiation, raised once
// per device (the first launch on a device sets it; later launches, for
// example inside a stream capture, only enqueue).
template <class L, int MAXE, bool ZERO, bool MIS>
int ensure_smem_attribute() {
  static std::atomic<uint64_t> done_mask{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  const uint64_t bit = dev < 64 ? (1ull << dev) : 0;
  if (bit && (done_mask.load(std::memory_order_acquire) & bit)) return 0;
  e = cudaFuncSetAttribute(commit_kernel<L, MAXE, ZERO, MIS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem_bytes<L, MIS>());
  if (e != cudaSuccess) return (int)e;
  if (APC_SMEM_CARVEOUT >= 0) {
    e = cudaFuncSetAttribute(commit_kernel<L, MAXE, ZERO, MIS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             APC_SMEM_CARVEOUT);
    if (e != cudaSuccess) return (int)e;
  }
  if (bit) done_mask.fetch_or(bit, std::memory_order_acq_rel);
  return 0;
}

template <class L, int MAXE, bool ZERO, bool MIS>
int launch_t(const CommitPlan<MAXE> &plan, unsigned grid, void *stream, unsigned long long *out) {
  int e = ensure_smem_attribute<L, MAXE, ZERO, MIS>();
  if (e) return e;
  return launch_plan(commit_kernel<L, MAXE, ZERO, MIS>, plan, plan.chained, grid, L::kThreads, smem_bytes<L, MIS>(),
                     stream, out);
}

template <class L, int MAXE>
int launch_l(const CommitPlan<MAXE> &plan, bool zero_grad, unsigned grid, void *stream, unsigned long long *out) {
  bool mis = false;
  for (uint32_t k = 0; k < plan.count; ++k) mis |= plan.e[k].mis != 0;
  if (mis)
    return zero_grad ? launch_t<L, MAXE, true, true>(plan, grid, stream, out)
                     : launch_t<L, MAXE, false, true>(plan, grid, stream, out);
  return zero_grad ? launch_t<L, MAXE, true, false>(plan, grid, stream, out)
                   : launch_t<L, MAXE, false, false>(plan, grid, stream, out);
}

template <class L, int MAXE, bool MIS>
int blocks_m(int *fewest) {
  int n = 0;
  int e = ensure_smem_attribute<L, MAXE, false, MIS>();
  if (e) return e;
  e = (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, commit_kernel<L, MAXE, false, MIS>, L::kThreads,
                                                         smem_bytes<L, MIS>());
  if (n < *fewest) *fewest = n;
  return e;
}

template <int MAXE>
int blocks_n(int *fewest) {
  int e = blocks_m<F32State, MAXE, false>(fewest);
  if (!e) e = blocks_m<F32State, MAXE, true>(fewest);
  if (!e) e = blocks_m<BF16State, MAXE, false>(fewest);
  return e ? e : blocks_m<BF16State, MAXE, true>(fewest);
}

}  // namespace

template <int MAXE>
int launch_commit(const CommitPlan<MAXE> &plan, int layout, bool zero_grad, unsigned grid, void *stream,
                  unsigned long long *out) {
  return layout == kLayoutBF16 ? launch_l<BF16State>(plan, zero_grad, grid, stream, out)
                               : launch_l<F32State>(plan, zero_grad, grid, stream, out);
}
template int launch_commit(const CommitPlan<kCommitSmall> &, int, bool, unsigned, void *, unsigned long long *);
template int launch_commit(const CommitPlan<kCommitMid> &, int, bool, unsigned, void *, unsigned long long *);
template int launch_commit(const CommitPlan<kCommitLarge> &, int, bool, unsigned, void *, unsigned long long *);

int commit_blocks_per_sm(int *out) {
  *out = 1 << 20;
  int e = blocks_n<kCommitSmall>(out);
  if (!e) e = blocks_n<kCommitMid>(out);
  return e ? e : blocks_n<kCommitLarge>(out);
}

int launch_wait_timeout(uint64_t limit_ns, void *stream) {
  wait_timeout_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(limit_ns);
  return (int)cudaGetLastError();
}

int read_commit_status(unsigned *out) {
  cudaError_t e = cudaMemcpyFromSymbol(out, g_commit_status, sizeof(unsigned));
  if (e != cudaSuccess) return (int)e;
  const unsigned zero = 0;
  return (int)cudaMemcpyToSymbol(g_commit_status, &zero, sizeof(unsigned));
}

}  // namespace apc
