// The quiescence guard: per-slot counts of nonzero words over a list of
// buffers, read only.  At a committed optimizer boundary the flat-parameter
// gradients have been zeroed (arxiv 2609.18178, Section I), and the recovery
// protocol's guard admits a repair only with zero outstanding gradients
// (Section III-C, phase 2); this kernel is that check on the device.
//
// A word counts when its bit pattern is nonzero (so a -0.0 gradient counts).
// The pass reads 4 (fp32) or 2 (bf16) bytes per element and does one compare
// per element, so it is bound by HBM: by the bytes in flight, and in short
// launches by how soon all SMs have them in flight and how evenly they end.
//
// Same buffer plans as the digest kernel (apc_digest.cu) and the same walk: a
// tile is kCountTileBytes of one buffer's 16-byte aligned body, each CTA of the
// persistent grid takes one contiguous run of the launch's tiles and its warps
// walk it interleaved, each on its own.  A lane issues all its kCountGroups
// 16-byte loads of a tile before it counts, group j of a warp being 512
// consecutive bytes.  What a buffer holds beyond its full tiles goes to one
// warp, before the walks: the CTA's last warps first, as the walk deals them one
// tile fewer (152 M in 146 tensors 50.9 us; 51.4 from the first warp on).
//
// Tiles of a whole CTA (64 KB, dealt out round robin) made its 1,024 threads
// wait for one tile at a time.  Against that, calls over bf16 gradients take:
// 152 M in 146 tensors 51 us (62), 2 M in 100 tensors 9.8 (26), 7.25 G in 291
// tensors 1,972 (2,158), which is 7.35 TB/s.
#include <cuda_runtime.h>

#include "../../include/apc.h"
#include "apc_device.cuh"
#include "apc_internal.h"
#include "apc_launch.cuh"

namespace apc {
namespace {

constexpr int kWarps = kCountThreads / 32;

__device__ __forceinline__ uint32_t nz32(uint4 x) {
  return (uint32_t)(x.x != 0) + (uint32_t)(x.y != 0) + (uint32_t)(x.z != 0) + (uint32_t)(x.w != 0);
}

__device__ __forceinline__ uint32_t nz16(uint32_t w) {
  return (uint32_t)((w & 0xFFFFu) != 0) + (uint32_t)((w >> 16) != 0);
}

__device__ __forceinline__ uint32_t nz(uint4 x, bool f32) {
  return f32 ? nz32(x) : nz16(x.x) + nz16(x.y) + nz16(x.z) + nz16(x.w);
}

template <int MAXE>
__global__ void __launch_bounds__(kCountThreads, 1) count_kernel(const __grid_constant__ DigestPlan<MAXE> plan,
                                                         unsigned long long *out) {
  __shared__ unsigned long long s_acc[APC_MAX_SLOTS];
  if (plan.more) chain_start_next();
  if (threadIdx.x < APC_MAX_SLOTS) s_acc[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // what the entries hold beyond their full tiles: the body's last groups, and
  // the scalar head (lanes 0-6) and tail (lanes 8-14)
  for (uint32_t e = blockIdx.x + gridDim.x * (kWarps - 1 - warp); e < plan.count; e += gridDim.x * kWarps) {
    const DigestEntry &E = plan.e[e];
    const bool f32 = E.dtype == 0;
    const uint32_t es = f32 ? 4 : 2;
    const uint64_t body = (E.n - E.head) & ~(uint64_t)(kVec - 1);
    const uint8_t *d = static_cast<const uint8_t *>(E.data);
    const uint4 *q = reinterpret_cast<const uint4 *>(d + E.head * es + body * es / kCountTileBytes * kCountTileBytes);
    const uint32_t groups = (uint32_t)(body * es % kCountTileBytes) / 16;
    uint64_t c = 0;
#pragma unroll
    for (int j = 0; j < kCountGroups; ++j)
      if (j * 32 + lane < groups) c += nz(__ldcs(q + j * 32 + lane), f32);
    const uint64_t i = lane < 8 ? lane : E.head + body + (lane - 8);
    if (i < (lane < 8 ? (uint64_t)E.head : E.n))
      c += f32 ? reinterpret_cast<const uint32_t *>(d)[i] != 0 : reinterpret_cast<const uint16_t *>(d)[i] != 0;
    flush(c, E.slot, s_acc);
  }
  // this CTA's run of tiles, walked by its warps
  const uint64_t per = plan.total_tiles / gridDim.x, rem = plan.total_tiles % gridDim.x;
  const uint64_t t_begin = blockIdx.x * per + (blockIdx.x < rem ? blockIdx.x : rem);
  const uint32_t len = (uint32_t)(per + (blockIdx.x < rem ? 1 : 0));  // 2^32 tiles are 13 TB
  uint32_t cur = 0, r = warp;
  int slot = -1;
  uint64_t acc = 0;
  while (r < len) {
    cur = entry_of(plan, cur, t_begin + r);
    const DigestEntry &E = plan.e[cur];
    const uint64_t left = (cur + 1 < plan.count ? plan.e[cur + 1].tile_begin : plan.total_tiles) - t_begin;
    const uint32_t stop = left < len ? (uint32_t)left : len;
    if ((int)E.slot != slot) {
      flush(acc, slot, s_acc);
      slot = E.slot;
    }
    const bool f32 = E.dtype == 0;
    const uint4 *q = reinterpret_cast<const uint4 *>(static_cast<const uint8_t *>(E.data) + E.head * (f32 ? 4 : 2) +
                                                     (t_begin + r - E.tile_begin) * kCountTileBytes) + lane;
    for (; r < stop; r += kWarps, q += kWarps * (kCountTileBytes / 16)) {
      uint4 x[kCountGroups];
#pragma unroll
      for (int j = 0; j < kCountGroups; ++j) x[j] = __ldcs(q + j * 32);
      uint32_t c = 0;
#pragma unroll
      for (int j = 0; j < kCountGroups; ++j) c += nz(x[j], f32);
      acc += c;
    }
  }
  flush(acc, slot, s_acc);
  __syncthreads();
  if (threadIdx.x < APC_MAX_SLOTS) {
    chain_wait();
    if (s_acc[threadIdx.x]) atomicAdd(&out[threadIdx.x], s_acc[threadIdx.x]);
  }
}

template <int MAXE>
int blocks_n(int *fewest) {
  int n = 0;
  const int e = (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, count_kernel<MAXE>, kCountThreads, 0);
  if (n < *fewest) *fewest = n;
  return e;
}

}  // namespace

template <int MAXE>
int launch_count(const DigestPlan<MAXE> &plan, unsigned grid, void *stream, unsigned long long *out) {
  return launch_plan(count_kernel<MAXE>, plan, plan.chained, grid, kCountThreads, 0, stream, out);
}
template int launch_count(const DigestPlan<kDigestSmall> &, unsigned, void *, unsigned long long *);
template int launch_count(const DigestPlan<kDigestMid> &, unsigned, void *, unsigned long long *);
template int launch_count(const DigestPlan<kDigestLarge> &, unsigned, void *, unsigned long long *);

int count_blocks_per_sm(int *out) {
  *out = 1 << 20;
  int e = blocks_n<kDigestSmall>(out);
  if (!e) e = blocks_n<kDigestMid>(out);
  return e ? e : blocks_n<kDigestLarge>(out);
}

}  // namespace apc
