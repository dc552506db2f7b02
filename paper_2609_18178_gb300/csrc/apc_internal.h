// Launch plans shared by the host side of the C ABI and the kernels.
//
// A plan is a kernel parameter block (__grid_constant__, at most 32,764
// bytes): the chunk table is copied by the driver at launch, so nothing is
// staged in device memory and no allocation is needed.  Tables larger than
// one block are split over several launches that add into the same digests.
#pragma once

#include <stdint.h>

namespace apc {

constexpr int kVec = 8;                    // vector granularity: 16 bytes of bf16, 32 bytes of fp32

// Commit kernel: warp-specialized pipeline.  One producer warp streams each
// tile of p, m, v and g into a ring of shared-memory stages with bulk
// asynchronous copies; the consumer warps compute from shared memory and
// store straight to global memory.
//
// Pipeline shape (compile-time, per state layout; the defaults are the
// measured best on GB300).
//  * fp32 state: 19 consumer warps + 1 producer = 20 warps, 5 per SM
//    sub-partition: each sub-partition's 16,384 registers then give 96 per
//    thread with no spills, the same budget as 16 + 1 warps (whose fifth
//    warp on one sub-partition sets the cap), with three more warps issuing.
//    Each consumer thread takes 2 groups of 4 elements per tile (3 ran 6%
//    slower).
//  * bf16 state stages 8 bytes per element instead of 14 and needs fewer
//    registers: 27 consumer warps + 1 producer = 28 warps at 72 registers
//    with no spills, 3 groups per thread per tile.  That is 3.2% faster than
//    the fp32 layout's shape there (19 warps and 4 groups were 1.8% faster
//    than 19 and 2; 23 warps with 3 groups and 31 with 2 were in between).
#ifndef APC_COMMIT_CONSUMER_WARPS
#define APC_COMMIT_CONSUMER_WARPS 19
#endif
#ifndef APC_COMMIT_CONSUMER_WARPS_BF16
#define APC_COMMIT_CONSUMER_WARPS_BF16 27
#endif
#ifndef APC_COMMIT_GROUPS
#define APC_COMMIT_GROUPS 2
#endif
#ifndef APC_COMMIT_GROUPS_BF16
#define APC_COMMIT_GROUPS_BF16 3
#endif
// Ring stages per CTA: three for fp32 state (0.3% faster than two), two for
// bf16 state (three of its larger tiles exceed a CTA's shared memory).
#ifndef APC_COMMIT_STAGES
#define APC_COMMIT_STAGES 3
#endif
#ifndef APC_COMMIT_BLOCKS_PER_SM
#define APC_COMMIT_BLOCKS_PER_SM 1
#endif
constexpr int kCommitConsumerWarps = APC_COMMIT_CONSUMER_WARPS;
constexpr int kCommitConsumerWarpsBF16 = APC_COMMIT_CONSUMER_WARPS_BF16;
constexpr int kCommitGroups = APC_COMMIT_GROUPS;
constexpr int kCommitGroupsBF16 = APC_COMMIT_GROUPS_BF16;
constexpr uint64_t kCommitTile = (uint64_t)kCommitConsumerWarps * 32 * 4 * kCommitGroups;              // 4,864 elements
constexpr uint64_t kCommitTileBF16 = (uint64_t)kCommitConsumerWarpsBF16 * 32 * 4 * kCommitGroupsBF16;  // 10,368 elements
constexpr int kCommitStages = APC_COMMIT_STAGES;
#ifndef APC_COMMIT_STAGES_BF16
#define APC_COMMIT_STAGES_BF16 2
#endif
constexpr int kCommitStagesBF16 = APC_COMMIT_STAGES_BF16;
constexpr int kCommitBlocksPerSm = APC_COMMIT_BLOCKS_PER_SM;
// Register budget of the fp32-state commit kernel: its launch bound is
// max(block size, APC_COMMIT_BOUND_THREADS) threads, so a build with fewer
// consumer warps can keep the default 96 registers per thread (and leave the
// rest of the SM to a co-resident kernel) instead of growing into them.
#ifndef APC_COMMIT_BOUND_THREADS
#define APC_COMMIT_BOUND_THREADS 0
#endif
// Shared-memory carveout preference (percent of the unified L1/shared
// capacity) given to the commit and digest kernels; -1 leaves the driver's
// default.  100 lets two different kernels' CTAs share an SM.
#ifndef APC_SMEM_CARVEOUT
#define APC_SMEM_CARVEOUT -1
#endif
// A stage holds one tile of p, m, v and g: 14 bytes per element for fp32
// state (66.5 KB, 200 KB per CTA at the defaults), 8 for bf16 state (81 KB,
// 162 KB per CTA).

// State layouts of the commit kernel.
constexpr int kLayoutF32 = 0;   // fp32 p, m, v; bf16 g; bf16 copy w
constexpr int kLayoutBF16 = 1;  // bf16 p, m, v; bf16 g; no copy

constexpr uint64_t commit_tile(int layout) { return layout == kLayoutBF16 ? kCommitTileBF16 : kCommitTile; }

// One chunk-table entry of the commit kernel (72 bytes).
//   p, m, v: fp32 or bf16 state (by the launch's layout); w: the bf16 copy
//         (fp32 layout only).
//   head, body: elements [head, head + body) run in tiles of the plan's `tile`
//         elements, the others (at most 31) one by one.
//   mis:  which buffers are not 16-byte aligned at the body's start: none, g
//         and w (kMisGrad), or any (kMisAll).  Such a buffer is read in the
//         16-byte blocks that hold it, which reach at most 15 bytes over the
//         body on either side; 8 elements are left out there, so the blocks
//         stay inside the buffer.
//   tile_begin: the entry's first tile in the launch's tile space.
//   key_base: global_offset mod 2^32 (the digest key of element 0).
enum CommitMis : uint16_t { kMisNone, kMisGrad, kMisAll };
struct CommitEntry {
  void *p, *m, *v;
  const uint16_t *g;
  uint16_t *w;
  uint64_t n;
  uint64_t body;
  uint64_t tile_begin;
  uint32_t key_base;
  uint16_t head;
  uint16_t mis;
};

// Constants of the commit kernel's packed operations, each in both lanes.
enum CommitPair {
  kPairB1, kPair1B1, kPairB2, kPair1B2,  // b1, 1-b1, b2, 1-b2
  kPairDecay,                            // 1-lr*wd
  kPairRsb2,                             // -1/sqrt(bc2) * 2^-32
  kPairStep,                             // lr/bc1 * 2^-64
  kPairNeg64, kPairNegTiny,              // -2^64, -2^-126
  kPairHalf, kPairOne,                   // 1/2, 1
  kPairs
};

template <int MAXE>
struct CommitPlan {
  float h[8];            // b1, 1-b1, b2, 1-b2, eps, 1-lr*wd, lr/bc1, 1/sqrt(bc2)
  uint64_t pair[kPairs];
  float limit;           // adamw_group's bound, -1 where its form does not apply
  uint32_t pad_;
  uint64_t total_tiles;
  uint32_t count;
  uint32_t one;          // 1: the FMA-pipe carry-add multiplier of the digest
  uint32_t tile;         // elements per tile of this launch (a multiple of 64, at most commit_tile)
  uint16_t more;         // another launch of the same call follows, chained to this one
  uint16_t chained;      // this one is chained to another of the same call before it
  CommitEntry e[MAXE];
};

// Plans of three sizes: a launch copies its whole parameter block, which takes
// 1 to 1.5 us more for 32 KB than for 7 (with_plan).
constexpr int kCommitSmall = 16, kCommitMid = 96, kCommitLarge = 440;
static_assert(sizeof(CommitEntry) == 72, "entry layout");
static_assert(sizeof(CommitPlan<kCommitLarge>) <= 32764, "kernel parameter limit");

// Digest kernel: the loads are issued by the compute warps themselves (the
// pass is bound by its integer pipes): a lane handles U 8-element vectors of
// its warp's tile, whose terms form one block of independent work.  One CTA
// per SM gives each SM one contiguous run of tiles.
//  * 640 threads (5 warps on each of the four schedulers, 96 registers) with
//    U = 4: 453 M elements of fp32 state verify in 1,427 us and 1.81 G of bf16
//    state in 3,675 us, against 1,455 and 3,883 us for 1024 x 2, 1,430 and
//    3,740 for 768 x 3, 1,452 and 3,879 for 512 x 4, 1,446 and 3,888 for
//    640 x 5.  (All before the terms' mixed multiplies, which brought the kept
//    shape to 1,411 and 3,650.)
//  * U = 4 needs several tiles for every warp to be dealt out evenly: with few
//    of them a tile of half the length spreads the work better (1 M elements
//    of fp32 state, 1.3 long tiles per warp: 9.9 us against 12.9).  The long
//    tile is taken from kDigestLongTiles of them per warp on, where the last,
//    partly dealt round costs at most 1 / 8 and typically half of that.
#ifndef APC_DIGEST_THREADS
#define APC_DIGEST_THREADS 640
#endif
constexpr int kThreads = APC_DIGEST_THREADS;     // threads per CTA of the digest kernel
constexpr int kDigestShort = 2, kDigestLong = 4;  // U: vectors per lane per tile
constexpr uint64_t kDigestLongTiles = 8;
constexpr uint64_t digest_tile(int u) { return (uint64_t)32 * kVec * u; }  // elements: 512 and 1,024

// Guard (count) kernel: the same plans and walk with tiles of its own; one
// compare per word leaves it bound by HBM, so its shape is set by the bytes
// each SM keeps in flight: 6 loads a lane (96 KB per SM) read 14.5 GB in
// 1,972 us, 4 in 2,024, 8 in 1,987 (2,001 with 512 threads), 2 in 2,037.
#ifndef APC_COUNT_THREADS
#define APC_COUNT_THREADS 1024
#endif
#ifndef APC_COUNT_GROUPS
#define APC_COUNT_GROUPS 6
#endif
constexpr int kCountThreads = APC_COUNT_THREADS;
constexpr int kCountGroups = APC_COUNT_GROUPS;                   // 16-byte loads per lane per tile
constexpr uint32_t kCountTileBytes = 32 * 16 * kCountGroups;     // one warp's tile
// Minimum resident CTAs per SM the digest kernel is compiled for (its
// register cap: 65,536 / (threads x this)), and extra dynamic shared memory
// per CTA beyond its stages (0 by default; a larger CTA footprint keeps two
// digest CTAs off one SM when another kernel is to share it).
#ifndef APC_DIGEST_MIN_BLOCKS
#define APC_DIGEST_MIN_BLOCKS 1
#endif
#ifndef APC_DIGEST_EXTRA_SMEM
#define APC_DIGEST_EXTRA_SMEM 0
#endif

// One buffer of the digest kernel (32 bytes).
//   head: scalar elements before the first 16-byte boundary (<= 7); then
//         8-element vectors, the whole tiles of which (digest_tile(U) elements
//         for the digest kernel, kCountTileBytes for the count kernel) are
//         counted in tile_begin; then a scalar tail.
struct DigestEntry {
  const void *data;
  uint64_t n;
  uint64_t tile_begin;
  uint32_t key_base;
  uint8_t head;
  uint8_t dtype;        // 0 fp32, 1 bf16
  uint8_t slot;
  uint8_t pad_;
};

template <int MAXE>
struct DigestPlan {
  uint64_t total_tiles;
  uint64_t tiles32;      // tiles of the fp32 entries, which come first (digest kernel)
  uint32_t count;
  uint32_t one;          // 1: the FMA-pipe carry-add multiplier of the digest
  uint16_t more;         // another launch of the same call follows, chained to this one
  uint16_t chained;      // this one is chained to another of the same call before it
  uint32_t pad_;
  DigestEntry e[MAXE];
};

constexpr int kDigestSmall = 16, kDigestMid = 200, kDigestLarge = 1000;
static_assert(sizeof(DigestEntry) == 32, "entry layout");
static_assert(sizeof(DigestPlan<kDigestLarge>) <= 32764, "kernel parameter limit");

// One segment of the upload kernel (48 bytes): bytes [head, head + body) in
// 16-byte words of the destination (dst + head is 16-byte aligned, body a
// multiple of 16), the rest byte by byte.
//   shift: (src + head) % 16: 0 where source and destination are mutually
//          aligned.  Otherwise the words are cut from the source's aligned
//          blocks, of which the first begins `shift` bytes before the body and
//          the last ends up to 16 - shift bytes behind it, both inside the
//          segment.
struct UploadEntry {
  uint8_t *dst;
  const uint8_t *src;   // device-side address of the source
  uint64_t bytes;
  uint64_t body;
  uint64_t tile_begin;   // first full tile of the body (prefix over the launch)
  uint32_t head, shift;
};

template <int MAXE>
struct UploadPlan {
  uint64_t total_tiles;
  uint32_t count;
  uint32_t pad_;
  UploadEntry e[MAXE];
};

#ifndef APC_UPLOAD_THREADS
#define APC_UPLOAD_THREADS 512
#endif
#ifndef APC_UPLOAD_GROUPS
#define APC_UPLOAD_GROUPS 8
#endif
constexpr int kUploadThreads = APC_UPLOAD_THREADS;
constexpr int kUploadGroups = APC_UPLOAD_GROUPS;              // 16-byte words per lane per tile
constexpr uint32_t kUploadTile = 32 * 16 * kUploadGroups;     // one warp's tile: 4 KB
constexpr int kUploadMax = 600;
static_assert(sizeof(UploadEntry) == 48, "entry layout");
static_assert(sizeof(UploadPlan<kUploadMax>) <= 32764, "kernel parameter limit");

// Upload kernel (apc_upload.cu): the plan's segments, on `grid` CTAs.
int launch_upload(const UploadPlan<kUploadMax> &plan, unsigned grid, void *stream);

// Launch wrappers (apc_commit.cu, apc_digest.cu, apc_guard.cu), instantiated for
// the plan sizes above.  They return a cudaError_t value and launch on `stream`
// with `grid` CTAs; u: the digest kernel's vectors per lane per tile.
template <int MAXE>
int launch_commit(const CommitPlan<MAXE> &plan, int layout, bool zero_grad, unsigned grid, void *stream,
                  unsigned long long *out);
template <int MAXE>
int launch_digest(const DigestPlan<MAXE> &plan, int u, unsigned grid, void *stream, unsigned long long *out);
// Per-slot counts of nonzero words over the same buffer plans as the digest.
template <int MAXE>
int launch_count(const DigestPlan<MAXE> &plan, unsigned grid, void *stream, unsigned long long *out);

// Resident CTAs per SM of each kernel (cudaOccupancyMaxActiveBlocksPerMultiprocessor),
// the fewest over its instantiations; those that zero gradients have the threads
// and shared memory of the others, which set it, and are not asked.
int commit_blocks_per_sm(int *out);
int digest_blocks_per_sm(int *out);
int count_blocks_per_sm(int *out);

// Device status word of the kernels of one translation unit on the current
// device: nonzero after a bounded wait gave up.  read_* copies it to the host
// (synchronously) and clears it.
int read_commit_status(unsigned *out);
// Self-test of the bounded wait: one thread waits on an mbarrier that nothing
// completes, gives up after limit_ns and records APC_ETIMEOUT.
int launch_wait_timeout(uint64_t limit_ns, void *stream);

}  // namespace apc
