// The read-only state digest over a list of buffers (the verification pass
// after recovery): 4 (fp32) or 2 (bf16) bytes read per element and one
// splitmix64 term per element, so the pass is bound by integer issue, not by
// HBM.
//
// Work split: each buffer's 16-byte aligned body is cut into warp tiles of
// 256 * U elements (U = 4, or 2 for little work: kDigestLong, kDigestShort),
// and each CTA of a persistent grid takes one contiguous run of the launch's
// fp32 tiles and one of its bf16 tiles (the CTAs' runs differ by at most one
// tile).  The kWarps warps of a CTA walk a run interleaved, warp w taking its
// tiles w, w + kWarps, ..., each on its own: a warp finds a buffer by a
// binary search when its walk leaves the one before, and inside one only steps
// a pointer and the key.  The CTA as a whole sweeps one region of memory, and
// no step waits for another warp.
//
// Why warp tiles: a table of many small buffers is bound by the latency of
// each buffer's first and last tile, and with tiles of a whole CTA (16,384
// elements) all its warps paid that latency at once, most of them idle in a
// partly filled tile.  1,100 tensors of 136 to 20,557 elements (4,400 buffers,
// 63 MB) took 330 us of kernel time that way and take 56 us by warps.
//
// Loads: a thread's part of a tile is U vectors of 8 words.  The tiles are
// full: they run without per-vector bounds checks, and each thread keeps its
// next tile in flight with cp.async into shared-memory slots that only it
// reads (two stages, no barrier), then folds the current one from there.
// What a buffer holds beyond its full tiles (less than a tile, and the scalar
// head and tail) is loaded straight into registers by one warp, before the
// walks: entry e by warp e / grid of CTA e mod grid.  (A CTA-wide bulk-copy
// pipeline like the commit kernel's measured slower here: its per-tile
// synchronisation costs issue slots, the one resource this pass is short of.)
//
// A thread keeps one running 64-bit sum for the slot of the buffer it is in;
// all lanes of a warp visit the same tiles, so slot changes are warp-uniform
// and the running sum is flushed (shuffle reduce, then a shared-memory
// atomic) only when the warp moves to a buffer of another slot and at exit.
// The host orders a launch's buffers by type and slot, so that is rare.
#include <cuda_runtime.h>

#include <atomic>

#include "../../include/apc.h"
#include "apc_device.cuh"
#include "apc_internal.h"
#include "apc_launch.cuh"

namespace apc {
namespace {

// A lane's words of a tile come in 16-byte groups, group j of all lanes being
// 512 consecutive bytes: kGroups32 groups of 4 fp32 words, kGroups16 of 8
// bf16 words.  (With 32 consecutive bytes per lane instead, each 16-byte copy
// takes half of a 32-byte sector and the other half is fetched again: 3-4%
// slower.)  U is the launch's vectors of 8 words per lane per tile.
constexpr uint32_t kSpan16 = 32 * 8, kSpan32 = 32 * 4;  // elements from a lane's group to its next
constexpr int kWarps = kThreads / 32;

template <int U>
struct Shape {
  static constexpr int kGroups16 = U, kGroups32 = 2 * U;
  static constexpr uint64_t kTile = digest_tile(U);
  // The keys of a thread's terms in a tile lie in [G0, G0 + span - 1]; with
  // the increment's carry their high words lie in [B, B + span].
  static constexpr uint32_t kKeySpan32 = (kGroups32 - 1) * kSpan32 + 4, kKeySpan16 = (kGroups16 - 1) * kSpan16 + 8;
};

// One digest term of this pass, in the fp32 terms' mix of multiplies.
template <uint32_t K>
__device__ __forceinline__ uint64_t term(uint32_t gidx, uint32_t bits, uint32_t one) {
  return digest_term<K, MulWide, MulCompiler>(gidx, bits, one);
}

// The same with SHARED: the caller has checked that all of a thread's terms
// in the tile share the top two bits of the incremented key high word
// (top_bits_shared over the keys of its groups) and passes them as `top`, so
// no term computes hi >> 30 itself.
template <uint32_t K, bool SHARED>
__device__ __forceinline__ uint64_t vterm(uint32_t gidx, uint32_t bits, uint32_t one, uint32_t top) {
  if constexpr (SHARED) return digest_term<K, MulWide, MulCompiler>(gidx, bits, one, top);
  else return digest_term<K, MulWide, MulCompiler>(gidx, bits, one);
}

// A thread's terms of one fp32 tile.
template <bool SHARED, int G>
__device__ __forceinline__ void fold32(const uint4 (&x)[G], const bool (&ok)[G], uint32_t G0,
                                       uint32_t one, uint32_t top, uint64_t &t0, uint64_t &t1) {
#pragma unroll
  for (int j = 0; j < G; ++j) {
    if (!ok[j]) continue;
    const uint32_t g = G0 + j * kSpan32;
    t0 += vterm<0, SHARED>(g, x[j].x, one, top) + vterm<1, SHARED>(g, x[j].y, one, top);
    t1 += vterm<2, SHARED>(g, x[j].z, one, top) + vterm<3, SHARED>(g, x[j].w, one, top);
  }
}

// Group J of a bf16 tile's G groups and those after it, keyed.
template <int J, int G>
__device__ __forceinline__ void fold16_keyed(const uint4 (&x)[G], const bool (&ok)[G], const Key16 (&k)[4],
                                             uint64_t &t0, uint64_t &t1) {
  constexpr uint32_t off = J * kSpan16;
  if (ok[J]) {
    t0 += digest_term_u16<off, 0>(k[0], x[J].x) + digest_term_u16<off, 1>(k[1], x[J].x);
    t1 += digest_term_u16<off, 0>(k[2], x[J].y) + digest_term_u16<off, 1>(k[3], x[J].y);
    t0 += digest_term_u16<off + 4, 0>(k[0], x[J].z) + digest_term_u16<off + 4, 1>(k[1], x[J].z);
    t1 += digest_term_u16<off + 4, 0>(k[2], x[J].w) + digest_term_u16<off + 4, 1>(k[3], x[J].w);
  }
  if constexpr (J + 1 < G) fold16_keyed<J + 1>(x, ok, k, t0, t1);
}

// A thread's terms of one bf16 tile: with SHARED, in the keyed 16-bit form
// (four keys a tile; 1.81 G elements of bf16 state verified in 4,050 us with
// the key's part formed for every term, 3,913 with the keyed form's adds on
// the multiply-add pipe and 3,790 with them left to the compiler).
template <bool SHARED, int G>
__device__ __forceinline__ void fold16(const uint4 (&x)[G], const bool (&ok)[G], uint32_t G0,
                                       uint32_t one, uint32_t top, uint64_t &t0, uint64_t &t1) {
  if constexpr (SHARED) {
    const Key16 k[4] = {key16(G0, one, top), key16(G0 + 1, one, top), key16(G0 + 2, one, top), key16(G0 + 3, one, top)};
    fold16_keyed<0>(x, ok, k, t0, t1);
  } else {
#pragma unroll
    for (int u = 0; u < G; ++u) {
      if (!ok[u]) continue;
      const uint32_t g = G0 + u * kSpan16;
      t0 += term<0>(g, x[u].x & 0xFFFFu, one) + term<1>(g, x[u].x >> 16, one);
      t1 += term<2>(g, x[u].y & 0xFFFFu, one) + term<3>(g, x[u].y >> 16, one);
      t0 += term<4>(g, x[u].z & 0xFFFFu, one) + term<5>(g, x[u].z >> 16, one);
      t1 += term<6>(g, x[u].w & 0xFFFFu, one) + term<7>(g, x[u].w >> 16, one);
    }
  }
}

// A thread's terms of the groups with ok[j] of one tile, straight from memory
// (q: the lane's first group).
template <int G>
__device__ __forceinline__ void tile32(const uint4 *q, const bool (&ok)[G], uint32_t G0, uint32_t one, uint64_t &t0,
                                       uint64_t &t1) {
  uint4 x[G];
#pragma unroll
  for (int j = 0; j < G; ++j)
    if (ok[j]) x[j] = __ldcs(q + j * 32);
  const uint32_t B = G0 + 0x9E3779B9u;
  if (top_bits_shared(B, Shape<G / 2>::kKeySpan32)) fold32<true>(x, ok, G0, one, B >> 30, t0, t1);
  else fold32<false>(x, ok, G0, one, 0, t0, t1);
}

template <int G>
__device__ __forceinline__ void tile16(const uint4 *q, const bool (&ok)[G], uint32_t G0, uint32_t one, uint64_t &t0,
                                       uint64_t &t1) {
  uint4 x[G];
#pragma unroll
  for (int u = 0; u < G; ++u)
    if (ok[u]) x[u] = __ldcs(q + u * 32);
  const uint32_t B = G0 + 0x9E3779B9u;
  if (top_bits_shared(B, Shape<G>::kKeySpan16)) fold16<true>(x, ok, G0, one, B >> 30, t0, t1);
  else fold16<false>(x, ok, G0, one, 0, t0, t1);
}

__device__ __forceinline__ uint32_t word_at(const DigestEntry &E, uint64_t i) {
  return E.dtype == 0 ? reinterpret_cast<const uint32_t *>(E.data)[i]
                      : (uint32_t) reinterpret_cast<const uint16_t *>(E.data)[i];
}

// Which of a lane's groups lie in the first `count` groups of a tile.
template <int G>
__device__ __forceinline__ void groups_ok(uint32_t lane, uint32_t count, bool (&ok)[G]) {
#pragma unroll
  for (int j = 0; j < G; ++j) ok[j] = j * 32 + lane < count;
}

// What an entry holds beyond its full tiles, done by one warp: the body's
// last vectors (fewer than a tile), the scalar head (lanes 0-6) and the scalar
// tail (lanes 8-14).
template <int U>
__device__ __forceinline__ uint64_t remainder(const DigestEntry &E, uint32_t lane, uint32_t one) {
  const uint64_t body = (E.n - E.head) & ~(uint64_t)(kVec - 1);
  const uint64_t begin = E.head + body / Shape<U>::kTile * Shape<U>::kTile;
  const uint32_t rest = (uint32_t)(body % Shape<U>::kTile), G0 = E.key_base + (uint32_t)begin;
  uint64_t t0 = 0, t1 = 0;
  if (E.dtype == 0) {
    bool ok[Shape<U>::kGroups32];
    groups_ok(lane, rest / 4, ok);
    tile32(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint32_t *>(E.data) + begin) + lane, ok,
           G0 + lane * 4, one, t0, t1);
  } else {
    bool ok[Shape<U>::kGroups16];
    groups_ok(lane, rest / 8, ok);
    tile16(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(E.data) + begin) + lane, ok,
           G0 + lane * 8, one, t0, t1);
  }
  const uint64_t i = lane < 8 ? lane : E.head + body + (lane - 8);
  if (i < (lane < 8 ? (uint64_t)E.head : E.n)) t0 += term<0>(E.key_base + (uint32_t)i, word_at(E, i), one);
  return t0 + t1;
}

// Per-thread double buffering of full tiles in shared memory: while a thread
// folds one tile it has the next one in flight with cp.async, into slots that
// only it reads, so no barrier is needed; cp.async.wait_group orders each
// thread's own copies.  Slot k of stage b of thread t is
// stg[(b * slots + k) * kThreads + t]: a warp's 16-byte reads of one slot are
// contiguous.  A stage has kGroups32 slots per thread.
template <int U>
constexpr uint32_t launch_smem() {  // two stages
  return 2u * Shape<U>::kGroups32 * kThreads * 16u + APC_DIGEST_EXTRA_SMEM;
}
static_assert(launch_smem<kDigestLong>() <= 227 * 1024, "shared memory per CTA");

__device__ __forceinline__ void cp16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all_but_newest() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// One walk: the warps' tiles of the fp32 entries (T32) or of the bf16 entries.
// Each kind's tiles are shared out over all CTAs on their own: a bf16 tile
// costs less than an fp32 one, and a CTA with tiles of one kind only would
// finish early or late.
template <bool T32, int U, int MAXE>
__device__ __forceinline__ void walk(const DigestPlan<MAXE> &plan, uint4 *stg, uint32_t stg_t, unsigned long long *s_acc) {
  using S = Shape<U>;
  constexpr int kGroups = T32 ? S::kGroups32 : S::kGroups16, kStageSlots = S::kGroups32;
  constexpr uint64_t kStep = kWarps * S::kTile;  // elements from a warp's tile to its next
  constexpr uint32_t kWords = T32 ? 4 : 8;  // of a group
  constexpr uint32_t kKeySpan = T32 ? S::kKeySpan32 : S::kKeySpan16;
  const uint32_t one = plan.one;
  const uint64_t lo = T32 ? 0 : plan.tiles32, hi = T32 ? plan.tiles32 : plan.total_tiles;
  // this CTA's contiguous run of the kind's tiles, walked by its warps:
  // tile t_begin + r for r = warp, warp + kWarps, ... below len
  // (the bf16 runs are dealt out from the last CTA on, so that the longer runs
  // of both kinds fall on different CTAs)
  const uint32_t c = T32 ? blockIdx.x : gridDim.x - 1 - blockIdx.x;
  const uint64_t per = (hi - lo) / gridDim.x, rem = (hi - lo) % gridDim.x;
  const uint64_t t_begin = lo + c * per + (c < rem ? c : rem);
  const uint32_t len = (uint32_t)(per + (c < rem ? 1 : 0));  // 2^32 tiles are 2^41 elements
  int slot = -1;
  uint64_t acc = 0;
  uint32_t r = threadIdx.x >> 5, cur = 0;
  while (r < len) {
    cur = entry_of(plan, cur, t_begin + r);
    const DigestEntry &E = plan.e[cur];
    const uint64_t left = (cur + 1 < plan.count ? plan.e[cur + 1].tile_begin : plan.total_tiles) - t_begin;
    const uint32_t stop = left < len ? (uint32_t)left : len;
    if ((int)E.slot != slot) {
      flush(acc, slot, s_acc);
      slot = E.slot;
    }
    const uint64_t base = E.head + (t_begin + r - E.tile_begin) * S::kTile;  // the tile's first element
    const uint32_t lane = threadIdx.x & 31;
    const uint4 *q = reinterpret_cast<const uint4 *>(static_cast<const uint8_t *>(E.data) + base * (16 / kWords)) + lane;
    uint32_t G0 = E.key_base + (uint32_t)base + lane * kWords;
    uint64_t t0 = 0, t1 = 0;
    uint32_t b = 0;
    bool all[kGroups];
#pragma unroll
    for (int j = 0; j < kGroups; ++j) {
      all[j] = true;  // a full tile needs no checks
      cp16(stg_t + j * kThreads * 16u, q + j * 32);
    }
    cp_commit();
    for (; r < stop; r += kWarps, q += kStep / kWords, G0 += (uint32_t)kStep) {
      if (r + kWarps < stop) {
        const uint4 *n = q + kStep / kWords;
        const uint32_t dst = stg_t + (b ^ 1) * kStageSlots * kThreads * 16u;
#pragma unroll
        for (int j = 0; j < kGroups; ++j) cp16(dst + j * kThreads * 16u, n + j * 32);
      }
      cp_commit();
      cp_wait_all_but_newest();
      const uint4 *src = stg + b * kStageSlots * kThreads + threadIdx.x;
      uint4 x[kGroups];
#pragma unroll
      for (int j = 0; j < kGroups; ++j) x[j] = src[j * kThreads];
      const uint32_t B = G0 + 0x9E3779B9u;
      const bool shared = top_bits_shared(B, kKeySpan);
      if constexpr (T32) {
        if (shared) fold32<true>(x, all, G0, one, B >> 30, t0, t1);
        else fold32<false>(x, all, G0, one, 0, t0, t1);
      } else {
        if (shared) fold16<true>(x, all, G0, one, B >> 30, t0, t1);
        else fold16<false>(x, all, G0, one, 0, t0, t1);
      }
      b ^= 1;
    }
    acc_add(acc, t0, one);
    acc_add(acc, t1, one);
  }
  flush(acc, slot, s_acc);
}

template <int MAXE, int U>
__global__ void __launch_bounds__(kThreads, APC_DIGEST_MIN_BLOCKS) digest_kernel(const __grid_constant__ DigestPlan<MAXE> plan,
                                                          unsigned long long *out) {
  __shared__ unsigned long long s_acc[APC_MAX_SLOTS];
  extern __shared__ __align__(16) uint4 stg[];
  const uint32_t stg_t = (uint32_t)__cvta_generic_to_shared(stg + threadIdx.x);  // this thread's slot 0, stage 0
  if (plan.more) chain_start_next();
  if (threadIdx.x < APC_MAX_SLOTS) s_acc[threadIdx.x] = 0;
  __syncthreads();
  // what the entries hold beyond their full tiles, one entry per warp
  for (uint32_t e = blockIdx.x + gridDim.x * (threadIdx.x >> 5); e < plan.count; e += gridDim.x * kWarps) {
    uint64_t x = remainder<U>(plan.e[e], threadIdx.x & 31, plan.one);
    flush(x, plan.e[e].slot, s_acc);
  }
  walk<true, U>(plan, stg, stg_t, s_acc);
  walk<false, U>(plan, stg, stg_t, s_acc);
  __syncthreads();
  if (threadIdx.x < APC_MAX_SLOTS) {
    chain_wait();
    if (s_acc[threadIdx.x]) atomicAdd(&out[threadIdx.x], s_acc[threadIdx.x]);
  }
}

// The dynamic shared-memory limit of one instantiation, raised once per
// device (later launches, for example inside a stream capture, only enqueue).
template <int MAXE, int U>
int ensure_stage_attribute() {
  static std::atomic<uint64_t> done_mask{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  const uint64_t bit = dev < 64 ? (1ull << dev) : 0;
  if (bit && (done_mask.load(std::memory_order_acquire) & bit)) return 0;
  e = cudaFuncSetAttribute(digest_kernel<MAXE, U>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)launch_smem<U>());
  if (e != cudaSuccess) return (int)e;
  if (APC_SMEM_CARVEOUT >= 0) {
    e = cudaFuncSetAttribute(digest_kernel<MAXE, U>, cudaFuncAttributePreferredSharedMemoryCarveout, APC_SMEM_CARVEOUT);
    if (e != cudaSuccess) return (int)e;
  }
  if (bit) done_mask.fetch_or(bit, std::memory_order_acq_rel);
  return 0;
}

template <int MAXE, int U>
int launch_u(const DigestPlan<MAXE> &plan, unsigned grid, void *stream, unsigned long long *out) {
  int e = ensure_stage_attribute<MAXE, U>();
  if (e) return e;
  return launch_plan(digest_kernel<MAXE, U>, plan, plan.chained, grid, kThreads, launch_smem<U>(), stream, out);
}

template <int MAXE, int U>
int blocks_u(int *fewest) {
  int n = 0;
  int e = ensure_stage_attribute<MAXE, U>();
  if (e) return e;
  e = (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, digest_kernel<MAXE, U>, kThreads, launch_smem<U>());
  if (n < *fewest) *fewest = n;
  return e;
}

template <int MAXE>
int blocks_n(int *fewest) {
  const int e = blocks_u<MAXE, kDigestShort>(fewest);
  return e ? e : blocks_u<MAXE, kDigestLong>(fewest);
}

}  // namespace

template <int MAXE>
int launch_digest(const DigestPlan<MAXE> &plan, int u, unsigned grid, void *stream, unsigned long long *out) {
  return u == kDigestLong ? launch_u<MAXE, kDigestLong>(plan, grid, stream, out)
                          : launch_u<MAXE, kDigestShort>(plan, grid, stream, out);
}
template int launch_digest(const DigestPlan<kDigestSmall> &, int, unsigned, void *, unsigned long long *);
template int launch_digest(const DigestPlan<kDigestMid> &, int, unsigned, void *, unsigned long long *);
template int launch_digest(const DigestPlan<kDigestLarge> &, int, unsigned, void *, unsigned long long *);

int digest_blocks_per_sm(int *out) {
  *out = 1 << 20;
  int e = blocks_n<kDigestSmall>(out);
  if (!e) e = blocks_n<kDigestMid>(out);
  return e ? e : blocks_n<kDigestLarge>(out);
}

}  // namespace apc
