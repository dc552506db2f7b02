// Host-to-device upload by the SMs (apc_upload).  On a Grace-Blackwell node
// the GPU reads page-locked (and, where supported, pageable) host memory
// coherently over NVLink-C2C, so plain 16-byte loads of the source, issued
// by a few CTAs, stream it into device memory at the link's rate without a
// DMA copy engine.  The launch is sized by the caller (max_ctas) so that it
// can run beside the step's persistent kernels on SMs they leave free.
//
// Work split: warp tiles of kUploadTile bytes of a segment's body, walked as
// in the digest kernel (one contiguous run of the launch's tiles per CTA, its
// warps interleaved).  Each lane issues all of its kUploadGroups loads of a
// tile before any store, which keeps enough bytes in flight to cover the
// link's latency.  What a segment holds beyond its full tiles is done before the
// walks, by the CTAs' last warps first, which a short launch leaves without a
// tile, the bytes at a segment's ends and its last words by two different
// warps: every part then waits for the link once.  In 7 segments of a packed
// bucket 600 KB take 8.1 us and 2 MB 14.2 (12.4 and 19.7 with one of the first
// warps per segment, 12.2 and 25 when every byte was copied alone).
//
// A segment whose source and destination are not mutually 16-byte aligned (an
// odd-sized tensor in a packed host bucket) is read in the 16-byte blocks of
// the source, each once: a lane's destination word is cut from its own block
// and the next lane's, which comes by shuffle.  The blocks reach up to 15 bytes
// over the words, so 15 to 31 bytes at the start and at least 16 at the end of
// such a segment are copied byte by byte.  40 MB in 146 segments of a packed
// bucket take 198 us (428 when every byte of such a segment was copied alone;
// 190 at the link's 211 GB/s), 1 GB in 20 segments on 16 CTAs 4.8 ms (97.7).
#include <cuda_runtime.h>

#include "../../include/apc.h"
#include "apc_device.cuh"
#include "apc_internal.h"

namespace apc {
namespace {

constexpr int kWarps = kUploadThreads / 32;

// Bytes [shift, shift + 16) of the 32 bytes a, b (shift 1 .. 15).
__device__ __forceinline__ uint4 cut(const uint4 &a, const uint4 &b, uint32_t shift) {
  uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  if (shift & 8) {
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
  }
  if (shift & 4) {
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
  }
  const uint32_t bits = 8 * (shift & 3);
  return make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits),
                    __funnelshift_r(w[2], w[3], bits), __funnelshift_r(w[3], w[4], bits));
}

__device__ __forceinline__ uint4 next_lane(const uint4 &x, uint32_t lane) {
  const int from = (lane + 1) & 31;
  return make_uint4(__shfl_sync(0xFFFFFFFFu, x.x, from), __shfl_sync(0xFFFFFFFFu, x.y, from),
                    __shfl_sync(0xFFFFFFFFu, x.z, from), __shfl_sync(0xFFFFFFFFu, x.w, from));
}

// Two CTAs per SM, so that 16 of them fit on 8 SMs left free by the persistent
// kernels (apc_set_reserved_sms): with 69 registers a thread only one did, and an
// end-to-end step of 14.5 GB of gradients took 79.6 ms instead of 69.2.
__global__ void __launch_bounds__(kUploadThreads, 2) upload_kernel(const __grid_constant__ UploadPlan<kUploadMax> plan) {
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // what the segments hold beyond their full tiles, the bytes at the ends and the
  // last words each by a warp of its own
  for (uint32_t i = blockIdx.x + gridDim.x * (kWarps - 1 - warp); i < 2 * plan.count; i += gridDim.x * kWarps) {
    const UploadEntry &E = plan.e[i >> 1];
    if (i & 1) {
      const uint64_t end = E.head + E.body;
      const uint32_t rest = (uint32_t)(E.bytes - end);  // under 32; the head is under 64
      uint8_t b0 = 0, b1 = 0, b2 = 0;
      if (lane < E.head) b0 = E.src[lane];
      if (lane + 32 < E.head) b1 = E.src[lane + 32];
      if (lane < rest) b2 = E.src[end + lane];
      if (lane < E.head) E.dst[lane] = b0;
      if (lane + 32 < E.head) E.dst[lane + 32] = b1;
      if (lane < rest) E.dst[end + lane] = b2;
      continue;
    }
    const uint64_t at = E.head + E.body / kUploadTile * kUploadTile;
    const uint4 *src = reinterpret_cast<const uint4 *>(E.src + at - E.shift);
    uint4 *dst = reinterpret_cast<uint4 *>(E.dst + at);
    const uint32_t words = (uint32_t)(E.body % kUploadTile) / 16;
    // all loads first here too: one latency of the link, not one per word
    const uint32_t shift = E.shift, blocks = words + (shift != 0);  // at most 256
    uint4 x[kUploadGroups] = {};
#pragma unroll
    for (int j = 0; j < kUploadGroups; ++j)
      if (j * 32 + lane < blocks) x[j] = __ldcs(src + j * 32 + lane);
    if (shift != 0) {
      uint4 n = next_lane(x[0], lane);
#pragma unroll
      for (int j = 0; j < kUploadGroups; ++j) {
        const uint4 after = j + 1 < kUploadGroups ? next_lane(x[j + 1], lane) : n;
        x[j] = cut(x[j], lane < 31 ? n : after, shift);
        n = after;
      }
    }
#pragma unroll
    for (int j = 0; j < kUploadGroups; ++j)
      if (j * 32 + lane < words) dst[j * 32 + lane] = x[j];
  }
  // this CTA's run of tiles, walked by its warps
  const uint64_t per = plan.total_tiles / gridDim.x, rem = plan.total_tiles % gridDim.x;
  const uint64_t t_begin = blockIdx.x * per + (blockIdx.x < rem ? blockIdx.x : rem);
  const uint32_t len = (uint32_t)(per + (blockIdx.x < rem ? 1 : 0));  // 2^32 tiles are 16 TB
  uint32_t cur = 0;
  for (uint32_t r = warp; r < len;) {
    cur = entry_of(plan, cur, t_begin + r);
    const UploadEntry &E = plan.e[cur];
    const uint64_t left = (cur + 1 < plan.count ? plan.e[cur + 1].tile_begin : plan.total_tiles) - t_begin;
    const uint32_t stop = left < len ? (uint32_t)left : len;
    const uint64_t at = E.head + (t_begin + r - E.tile_begin) * kUploadTile;
    const uint32_t shift = E.shift;
    const uint4 *src = reinterpret_cast<const uint4 *>(E.src + at - shift) + lane;
    uint4 *dst = reinterpret_cast<uint4 *>(E.dst + at) + lane;
    for (; r < stop; r += kWarps, src += kWarps * (kUploadTile / 16), dst += kWarps * (kUploadTile / 16)) {
      uint4 x[kUploadGroups + 1];
#pragma unroll
      for (int j = 0; j < kUploadGroups; ++j) x[j] = __ldcs(src + j * 32);
      if (shift == 0) {
#pragma unroll
        for (int j = 0; j < kUploadGroups; ++j) dst[j * 32] = x[j];
      } else {
        // the block behind the tile, for the last lane's last word
        if (lane == 0) x[kUploadGroups] = __ldcs(src + kUploadGroups * 32);
        uint4 n = next_lane(x[0], lane);
#pragma unroll
        for (int j = 0; j < kUploadGroups; ++j) {
          const uint4 after = next_lane(x[j + 1], lane);  // in lane 31: lane 0's block of the next group
          dst[j * 32] = cut(x[j], lane < 31 ? n : after, shift);
          n = after;
        }
      }
    }
  }
}

}  // namespace

int launch_upload(const UploadPlan<kUploadMax> &plan, unsigned grid, void *stream) {
  upload_kernel<<<grid, kUploadThreads, 0, (cudaStream_t)stream>>>(plan);
  return (int)cudaGetLastError();
}

}  // namespace apc
