// Host side of the C ABI declared in include/apc.h: argument validation,
// resolution of the step's binary32 scalars (in double, rounded once),
// conversion of chunk tables, buffer lists and upload segments into launch
// plans, the persistent grid sizes (SM count x residency, less the SMs
// reserved with apc_set_reserved_sms), and the launches.
//
// The library allocates nothing.  Each plan travels in the kernel's
// parameter block; the digests are accumulated with atomics straight into
// the caller's output, which is zeroed on the stream first.
#include <cuda.h>  // attribute names and types; the driver function is looked up at run time
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/apc.h"
#include "apc_internal.h"

#define APC_EXPORT extern "C" __attribute__((visibility("default")))

namespace {

thread_local char g_last_error[512] = "";

apc_status fail(apc_status s, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_last_error, sizeof g_last_error, fmt, ap);
  va_end(ap);
  return s;
}

// An error that is returned is not left pending with the runtime as well.
apc_status cuda_fail(int err, const char *what) {
  cudaGetLastError();
  return fail(APC_ECUDA, "%s: %s", what, cudaGetErrorString((cudaError_t)err));
}

// Scalars of step t (see apc_resolve_hparams).
apc_status resolve(const apc_adamw_hparams *hp, int64_t step, float out[8]) {
  if (!hp) return fail(APC_EINVAL, "hparams pointer is null");
  if (step < 1) return fail(APC_EINVAL, "step %lld < 1", (long long)step);
  const double lr = hp->lr, b1 = hp->beta1, b2 = hp->beta2, eps = hp->eps, wd = hp->weight_decay;
  if (!std::isfinite(lr) || !std::isfinite(b1) || !std::isfinite(b2) || !std::isfinite(eps) || !std::isfinite(wd))
    return fail(APC_EINVAL, "non-finite hyper-parameter");
  if (!(b1 >= 0.0 && b1 < 1.0) || !(b2 >= 0.0 && b2 < 1.0)) return fail(APC_EINVAL, "beta outside [0, 1)");
  if (!(eps > 0.0)) return fail(APC_EINVAL, "eps must be > 0");
  if (lr < 0.0 || wd < 0.0) return fail(APC_EINVAL, "lr and weight_decay must be >= 0");
  // bias corrections in double; each scalar rounded once to binary32
  const double bc1 = 1.0 - std::pow(b1, (double)step);
  const double bc2 = 1.0 - std::pow(b2, (double)step);
  out[0] = (float)b1;
  out[1] = (float)(1.0 - b1);
  out[2] = (float)b2;
  out[3] = (float)(1.0 - b2);
  out[4] = (float)eps;
  out[5] = (float)(1.0 - lr * wd);
  out[6] = (float)(lr / bc1);
  out[7] = (float)(1.0 / std::sqrt(bc2));
  return APC_OK;
}

uint64_t ceil_div(uint64_t a, uint64_t b) { return a / b + (a % b != 0); }

// What a range of a call is: one of a table's five buffers, a buffer of a list
// (kBuffer + its type and slot), an output, or an upload's source or destination.
enum Kind : uint8_t { kP, kM, kV, kG, kW, kSource, kDest, kOut, kBuffer };

// One memory range of a call, [lo, hi), and whether kernels write it; index:
// its entry in the caller's list.
struct Range {
  uintptr_t lo, hi;
  int32_t index;
  uint8_t kind;
  bool written;
};

// The ranges of a call in address order.  A caller's tables usually give each
// kind of buffer in ascending order and each kind has memory of its own, so the
// list, filled kind by kind, is a few ascending runs that do not interleave:
// these are taken in the order of their first addresses (12 us for 5,500
// ranges, where sorting them all takes 60 to 330).  Any other list is sorted.
class Ordered {
 public:
  explicit Ordered(std::vector<Range> &r) : r_(r) {
    size_t begin = 0;
    for (size_t i = 1; i <= r.size() && runs_.size() <= kRuns; ++i)
      if (i == r.size() || r[i].kind != r[i - 1].kind || r[i].lo < r[i - 1].lo) {
        runs_.push_back({begin, i});
        begin = i;
      }
    bool apart = runs_.size() <= kRuns;
    if (apart) {
      std::sort(runs_.begin(), runs_.end(), [&](const auto &a, const auto &b) { return r[a.first].lo < r[b.first].lo; });
      for (size_t k = 1; k < runs_.size() && apart; ++k)
        apart = r[runs_[k - 1].second - 1].lo <= r[runs_[k].first].lo;
    }
    if (!apart) {
      std::sort(r.begin(), r.end(), [](const Range &a, const Range &b) { return a.lo < b.lo; });
      runs_.assign(1, {0, r.size()});
    }
  }

  // f(range) for each range in order until it returns false; whether it never did.
  template <typename F>
  bool each(F f) const {
    for (const auto &run : runs_)
      for (size_t i = run.first; i < run.second; ++i)
        if (!f(r_[i])) return false;
    return true;
  }

 private:
  static constexpr size_t kRuns = 32;
  std::vector<Range> &r_;
  std::vector<std::pair<size_t, size_t>> runs_;
};

// Written ranges must be pairwise disjoint and disjoint from read ranges.
bool overlaps(const Ordered &r) {
  uintptr_t hi_any = 0, hi_written = 0;
  return !r.each([&](const Range &x) {
    if (x.lo < hi_written || (x.written && x.lo < hi_any)) return false;
    hi_any = std::max(hi_any, x.hi);
    if (x.written) hi_written = std::max(hi_written, x.hi);
    return true;
  });
}

struct Device {
  int sms = 0;
  int commit = 0, digest = 0, count = 0;  // resident CTAs per SM
};

constexpr int kMaxDevices = 64;
Device g_devices[kMaxDevices];
std::atomic<bool> g_device_ready[kMaxDevices];
std::mutex g_device_mu;

// SM count and occupancy of the current device, queried once per device.
apc_status device_info(Device *out) {
  int dev = 0;
  int e = (int)cudaGetDevice(&dev);
  if (e) return cuda_fail(e, "cudaGetDevice");
  if (dev >= 0 && dev < kMaxDevices && g_device_ready[dev].load(std::memory_order_acquire)) {
    *out = g_devices[dev];
    return APC_OK;
  }
  Device dd, *d = &dd;
  e = (int)cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, dev);
  if (e) return cuda_fail(e, "cudaDeviceGetAttribute");
  if ((e = apc::commit_blocks_per_sm(&d->commit))) return cuda_fail(e, "occupancy query");
  if ((e = apc::digest_blocks_per_sm(&d->digest))) return cuda_fail(e, "occupancy query");
  if ((e = apc::count_blocks_per_sm(&d->count))) return cuda_fail(e, "occupancy query");
  if (dev >= 0 && dev < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_device_mu);
    if (!g_device_ready[dev].load(std::memory_order_relaxed)) {
      g_devices[dev] = dd;
      g_device_ready[dev].store(true, std::memory_order_release);
    }
  }
  *out = dd;
  return APC_OK;
}

// f(size) with the smallest plan size that holds `count` entries, or the
// largest.  A launch copies its parameter block whole: with the middle size in
// place of 32 KB a commit of 21 tensors takes 9.0 to 10.3 us of host time (10.7),
// one of 50 tensors 10.8 to 11.5 (12.2), their verifications 1 us less too.
template <int SMALL, int MID, int LARGE, typename F>
apc_status with_plan(size_t count, F f) {
  if (count <= (size_t)SMALL) return f(std::integral_constant<int, SMALL>{});
  if (count <= (size_t)MID) return f(std::integral_constant<int, MID>{});
  return f(std::integral_constant<int, LARGE>{});
}

// The launches of a long table go onto their stream as one chain (launch_plan):
// a chain of another thread on the same stream must not mix with them.  (A
// single launch may come in between: it starts nothing early.)  Only where the
// grid may take the whole GPU: the next launch's CTAs would otherwise start on
// the SMs that the caller keeps free (apc_set_reserved_sms, APC_GRID_LIMIT) and
// hold them until the launch before has ended.
std::mutex &chain_lock(const void *stream) {
  static std::mutex locks[64];
  const uintptr_t s = (uintptr_t)stream;
  return locks[(s ^ s >> 6 ^ s >> 12) & 63];
}

// SMs that the persistent kernels leave free (apc_set_reserved_sms).
std::atomic<int> g_reserved_sms{0};

// The persistent grid: one CTA per resident slot on the SMs not reserved
// (at least one SM's worth), capped by APC_GRID_LIMIT (read at every call)
// when that is a positive integer.  `whole`: neither leaves a slot free.  Read
// once a call, so that all its launches agree.
struct Grid {
  unsigned cap;
  bool whole;
};

Grid grid_for(int sms, int per_sm) {
  const int avail = std::max(1, sms - g_reserved_sms.load(std::memory_order_relaxed));
  const uint64_t slots = (uint64_t)std::max(per_sm, 1);
  uint64_t cap = (uint64_t)avail * slots;
  if (const char *lim = std::getenv("APC_GRID_LIMIT")) {
    char *end = nullptr;
    const unsigned long long v = std::strtoull(lim, &end, 10);
    if (end != lim && *end == 0 && v > 0) cap = std::min<uint64_t>(cap, v);
  }
  return {(unsigned)cap, cap == (uint64_t)sms * slots};
}

// The address range of the allocation that holds `p`, if it is an ordinary
// device allocation (cudaMalloc's): one allocation, of one device.  False for
// memory of the virtual-memory interface, whose ranges can hold several
// mappings, and where the driver cannot answer.
bool allocation_of(const void *p, uintptr_t *lo, uintptr_t *hi) {
  static const PFN_cuPointerGetAttributes_v7000 query = [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult st = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &fn, 12000, cudaEnableDefault, &st) != cudaSuccess)
      cudaGetLastError();
    return st == cudaDriverEntryPointSuccess ? (PFN_cuPointerGetAttributes_v7000)fn : nullptr;
  }();
  if (!query) return false;
  CUpointer_attribute names[3] = {CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  unsigned long long ordinary = 0;  // the driver writes a byte or a word of it
  CUdeviceptr start = 0;
  size_t size = 0;
  void *values[3] = {&ordinary, &start, &size};
  if (query(3, names, values, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS || !ordinary || !size) return false;
  *lo = (uintptr_t)start;
  *hi = (uintptr_t)start + size;
  return true;
}

// Every buffer a kernel reads or writes must be memory of the calling
// thread's current device (or managed memory): a pointer into another GPU's
// memory, or host memory, would otherwise be dereferenced by this device's
// copies.  In address order, one attribute query per allocation where its
// range is known, and one per distinct address otherwise: 1,100 tensors' 5,500
// pointers in five arenas take 6 queries instead of 5,500 (0.14 us each).  After
// a failed range query the next 1, 2, 4, ... addresses are taken one by one
// before a range is asked for again, so that a table in virtual memory costs at
// most log2 of its length more than its addresses (5,500 of them in PyTorch's
// expandable segments: 850 us a commit, 1,450 with a range query for each).
// Nothing is kept from one call to the next.  Returns APC_ECUDA if the runtime
// cannot answer (for example, no device) and APC_EINVAL naming the first
// foreign pointer (lowest address first).
apc_status check_device_pointers(const Ordered &ranges, size_t count, const char *out_name) {
  constexpr size_t kFew = 8;  // fewer pointers than this are queried one by one
  int dev = 0;
  int e = (int)cudaGetDevice(&dev);
  if (e) return cuda_fail(e, "cudaGetDevice");
  uintptr_t lo = 0, hi = 0;         // the allocation last queried
  size_t one_by_one = 0, next = 1;  // addresses until a range is asked for again, and after the next failure
  apc_status st = APC_OK;
  ranges.each([&](const Range &o) {
    if (o.lo >= lo && o.lo < hi) return true;
    const void *p = (const void *)o.lo;
    cudaPointerAttributes a;
    e = (int)cudaPointerGetAttributes(&a, p);
    if (e) {
      st = cuda_fail(e, "cudaPointerGetAttributes");
      return false;
    }
    const bool own = (a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged;
    if (!own) {
      static const char *const names[] = {"p", "m", "v", "g", "w"};
      char what[64];
      if (o.kind <= kW) snprintf(what, sizeof what, "table[%d].%s", (int)o.index, names[o.kind]);
      else if (o.kind >= kBuffer) snprintf(what, sizeof what, "bufs[%d].data", (int)o.index);
      else snprintf(what, sizeof what, "%s", out_name);
      st = fail(APC_EINVAL, "%s is not memory of the current device %d (memory type %d, device %d)", what, dev,
                (int)a.type, a.device);
      return false;
    }
    if (count >= kFew && a.type == cudaMemoryTypeDevice) {
      if (one_by_one) {
        --one_by_one;
      } else {
        if (allocation_of(p, &lo, &hi)) return true;
        one_by_one = next;
        next *= 2;
      }
    }
    lo = o.lo;
    hi = o.lo + 1;
    return true;
  });
  return st;
}

// Elements per tile of one launch.  The full tile is what the ring is built
// for, and the launch's time is then set by bandwidth.  In a launch of few
// rounds of them it is set by the CTA with the most to do: 1 M elements are
// 216 full tiles for 152 CTAs, two rounds for 64 of them and one for the rest,
// and 100,000 elements are 21 tiles for 21 CTAs.  So up to kEvenRounds rounds
// the length is chosen that gives that CTA the least work, a tile counting as
// its elements and kTileCost more (its share of the pipeline's latency; 256
// and 1,024 measure the same).  With the kernel's bisection and its one-barrier
// sum, 100,003 elements take 5.5 us of kernel time (9.1 before), 1 M take 11.4
// (13.3), 1,100 entries of 136 to 20,557 take 50 in three launches (130).
constexpr uint64_t kEvenRounds = 8, kTileCost = 512, kTileStep = 64, kTileMin = 256;

uint32_t commit_launch_tile(const apc::CommitEntry *e, size_t count, uint64_t full, uint64_t grid) {
  uint64_t body = 0, longest = 0;
  for (size_t j = 0; j < count; ++j) {
    body += e[j].body;
    longest = std::max(longest, e[j].body);
  }
  if (body > kEvenRounds * grid * full) return (uint32_t)full;
  uint64_t best = full, best_cost = UINT64_MAX;
  const uint64_t fewest = std::max<uint64_t>(1, ceil_div(body, grid * full));
  for (uint64_t rounds = fewest; rounds < fewest + 4; ++rounds) {
    const uint64_t even = ceil_div(ceil_div(body, grid * rounds), kTileStep) * kTileStep;
    const uint64_t tile = std::min(full, std::max(kTileMin, even));
    const double per = 1.0 / (double)tile;  // an estimate will do here
    uint64_t tiles = 0;
    for (size_t j = 0; j < count; ++j) tiles += (uint64_t)((double)(e[j].body + tile - 1) * per);
    const uint64_t cost = ceil_div(tiles, grid) * (std::min(tile, longest) + kTileCost);
    if (cost < best_cost) {
      best_cost = cost;
      best = tile;
    }
  }
  return (uint32_t)best;
}

// The scalars of a launch, and the constants of adamw_group with the bounds
// that its form needs of them.  The root of its 2^-126 addend, which enters den
// as 1/sqrt(bc2) * 2^-95, stays under half an ulp of eps where
// eps >= 1/sqrt(bc2) * 2^-69.  With |m'| + den <= limit = min(2^30, eps * 2^62),
// x is below 2^125, den in [2^-69, 2^30], and a / den <= limit * 2^64 / eps at
// most 2^126.  A nonzero step in [2^-60, 2^20] keeps step * 2^-64 normal and a
// subnormal quotient's term below 2^-106.  Elements beyond take the general
// operations on top of the grouped ones, so the bounds leave out only what no
// job holds: with a fixed limit of 128 and eps >= 2^-50, 30 M elements of fp32
// state took 162 us instead of 138 where gradients are summed instead of
// averaged, or with eps = 1e-16, and of bf16 state 132 instead of 110.
template <int MAXE>
void commit_scalars(const float h[8], apc::CommitPlan<MAXE> *plan) {
  std::memcpy(plan->h, h, sizeof plan->h);
  const float pairs[apc::kPairs] = {h[0],     h[1],       h[2],       h[3], h[5], -h[7] * 0x1p-32f, h[6] * 0x1p-64f,
                                    -0x1p64f, -0x1p-126f, 0.5f, 1.0f};
  for (int k = 0; k < apc::kPairs; ++k) {
    uint32_t bits;
    std::memcpy(&bits, &pairs[k], sizeof bits);
    plan->pair[k] = (uint64_t)bits << 32 | bits;
  }
  const bool fits = h[7] >= 1.0f && h[4] >= h[7] * 0x1p-69f && (h[6] == 0.0f || (h[6] >= 0x1p-60f && h[6] <= 0x1p20f));
  plan->limit = fits ? std::min(0x1p30f, h[4] * 0x1p62f) : -1.0f;
}

// Entries arrive without tile_begin; each batch places their tiles.
template <int MAXE, typename Launch>
apc_status run_commit_batches(const std::vector<apc::CommitEntry> &entries, const float h[8], int layout,
                              bool zero_grad, Grid grid_max, void *stream, unsigned long long *out,
                              Launch launch) {
  std::unique_ptr<apc::CommitPlan<MAXE>> plan(new apc::CommitPlan<MAXE>);  // not cleared: the kernel reads what is filled
  commit_scalars(h, plan.get());
  plan->one = 1;
  const bool chain = grid_max.whole && entries.size() > (size_t)MAXE;
  std::unique_lock<std::mutex> lock;
  if (chain) lock = std::unique_lock<std::mutex>(chain_lock(stream));
  size_t i = 0;
  while (i < entries.size()) {
    const size_t k = std::min(entries.size() - i, (size_t)MAXE);
    const uint32_t tile = commit_launch_tile(&entries[i], k, apc::commit_tile(layout), grid_max.cap);
    uint64_t tiles = 0;
    for (size_t j = 0; j < k; ++j) {
      apc::CommitEntry e = entries[i + j];
      e.tile_begin = tiles;
      tiles += ceil_div(e.body, tile);
      plan->e[j] = e;
    }
    plan->tile = tile;
    plan->count = (uint32_t)k;
    plan->total_tiles = tiles;
    plan->more = chain && i + k < entries.size();
    plan->chained = chain && i > 0;
    const uint64_t want = std::max<uint64_t>(tiles, k);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, grid_max.cap));
    int e = launch(*plan, layout, zero_grad, grid, stream, out);
    if (e) return cuda_fail(e, "commit kernel launch");
    i += k;
  }
  return APC_OK;
}

// Entries arrive with the element count of their vector body in tile_begin;
// tiles_of(body, element size) is the kernel's count of whole tiles in it.
template <int MAXE, typename Tiles, typename Launch>
apc_status run_digest_batches(const std::vector<apc::DigestEntry> &entries, Grid grid_max, const void *stream,
                              Tiles tiles_of, Launch launch, const char *what) {
  std::unique_ptr<apc::DigestPlan<MAXE>> plan(new apc::DigestPlan<MAXE>);
  plan->one = 1;
  const bool chain = grid_max.whole && entries.size() > (size_t)MAXE;
  std::unique_lock<std::mutex> lock;
  if (chain) lock = std::unique_lock<std::mutex>(chain_lock(stream));
  size_t i = 0;
  while (i < entries.size()) {
    const size_t k = std::min(entries.size() - i, (size_t)MAXE);
    uint64_t tiles = 0, tiles32 = 0;
    for (size_t j = 0; j < k; ++j) {
      apc::DigestEntry e = entries[i + j];
      const uint64_t t = tiles_of(e.tile_begin, e.dtype == APC_F32 ? 4 : 2);
      e.tile_begin = tiles;
      tiles += t;
      if (e.dtype == APC_F32) tiles32 = tiles;
      plan->e[j] = e;
    }
    plan->count = (uint32_t)k;
    plan->total_tiles = tiles;
    plan->tiles32 = tiles32;
    plan->more = chain && i + k < entries.size();
    plan->chained = chain && i > 0;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(std::max<uint64_t>(tiles, k), grid_max.cap));
    int e = launch(*plan, grid);
    if (e) return cuda_fail(e, what);
    i += k;
  }
  return APC_OK;
}

}  // namespace

APC_EXPORT apc_status apc_resolve_hparams(const apc_adamw_hparams *hp, int64_t step, float out[8]) {
  g_last_error[0] = 0;
  if (!out) return fail(APC_EINVAL, "output pointer is null");
  return resolve(hp, step, out);
}

namespace {

// One table entry in layout-neutral form.
struct TableRow {
  void *p, *m, *v;
  const uint16_t *g;
  uint16_t *w;  // null for the bf16 layout
  uint64_t n, goff;
};

// Shared by both layouts: validation, scalar resolution, overlap check,
// planning and launches.  nslots digests are zeroed and accumulated.
apc_status commit_common(int layout, const std::vector<TableRow> &rows, const apc_adamw_hparams *hp, int64_t step,
                         uint32_t flags, apc_stream_t stream, uint64_t *out_digests, int nslots) {
  if (flags & ~(uint32_t)APC_COMMIT_ZERO_GRAD) return fail(APC_EINVAL, "unknown flag bits 0x%x", flags);
  const bool zero_grad = (flags & APC_COMMIT_ZERO_GRAD) != 0;
  if (!out_digests) return fail(APC_EINVAL, "out_digests pointer is null");
  if ((uintptr_t)out_digests % 8) return fail(APC_EALIGN, "out_digests not 8-byte aligned");
  float h[8];
  apc_status st = resolve(hp, step, h);
  if (st != APC_OK) return st;
  const uint64_t es = layout == apc::kLayoutF32 ? 4 : 2;  // bytes per state element

  std::vector<apc::CommitEntry> entries;
  entries.reserve(rows.size());
  for (size_t k = 0; k < rows.size(); ++k) {
    const TableRow &t = rows[k];
    if (t.n == 0) continue;
    if (!t.p || !t.m || !t.v || !t.g || (layout == apc::kLayoutF32 && !t.w))
      return fail(APC_EINVAL, "table[%zu]: null buffer pointer", k);
    if (t.n > (UINT64_MAX - t.goff)) return fail(APC_ERANGE, "table[%zu]: global_offset + n overflows", k);
    if (t.n > ((uint64_t)1 << 61)) return fail(APC_ERANGE, "table[%zu]: n too large", k);
    const uintptr_t p = (uintptr_t)t.p, m = (uintptr_t)t.m, v = (uintptr_t)t.v, g = (uintptr_t)t.g,
                    w = (uintptr_t)t.w;
    if (p % es || m % es || v % es)
      return fail(APC_EALIGN, "table[%zu]: state buffer not %u-byte aligned", k, (unsigned)es);
    if (g % 2 || w % 2) return fail(APC_EALIGN, "table[%zu]: bf16 buffer not 2-byte aligned", k);
    // first element at which all buffers sit on a 16-byte boundary
    const uint64_t h0 = ((16 - g % 16) % 16) / 2;
    const bool aligned = (p + es * h0) % 16 == 0 && (m + es * h0) % 16 == 0 && (v + es * h0) % 16 == 0 &&
                         (!t.w || (w + 2 * h0) % 16 == 0);
    apc::CommitEntry e;
    e.p = t.p;
    e.m = t.m;
    e.v = t.v;
    e.g = t.g;
    e.w = t.w;
    e.n = t.n;
    e.key_base = (uint32_t)t.goff;
    // aligned: whole 16-byte vectors from there on.  Otherwise 8 elements are
    // left out on either side, and the body starts where p, m and v sit on a
    // 16-byte boundary if they do so together.
    const uint64_t hp = ((16 - p % 16) % 16) / es;
    const bool state = p % 16 == m % 16 && p % 16 == v % 16;
    const uint64_t head = std::min<uint64_t>(aligned ? h0 : state ? 8 + hp : 8, t.n);
    const uint64_t room = t.n - head - (aligned ? 0 : std::min<uint64_t>(8, t.n - head));
    e.head = (uint16_t)head;
    e.body = t.n < 32 && !aligned ? 0 : room / apc::kVec * apc::kVec;
    e.mis = aligned || !e.body ? apc::kMisNone : state ? apc::kMisGrad : apc::kMisAll;
    entries.push_back(e);
  }
  std::vector<Range> ranges;
  ranges.reserve(entries.size() * 5 + 1);
  const auto add = [&](Kind kind, uint64_t size, bool written, const auto &at) {
    for (size_t k = 0; k < rows.size(); ++k) {
      const uintptr_t lo = (uintptr_t)at(rows[k]);
      if (rows[k].n && lo) ranges.push_back({lo, lo + size * rows[k].n, (int32_t)k, kind, written});
    }
  };
  add(kP, es, true, [](const TableRow &t) { return t.p; });
  add(kM, es, true, [](const TableRow &t) { return t.m; });
  add(kV, es, true, [](const TableRow &t) { return t.v; });
  add(kG, 2, zero_grad, [](const TableRow &t) { return t.g; });
  add(kW, 2, true, [](const TableRow &t) { return t.w; });  // null in the bf16 layout
  const uintptr_t o = (uintptr_t)out_digests;
  ranges.push_back({o, o + (uintptr_t)nslots * sizeof(uint64_t), -1, kOut, true});
  const Ordered ordered(ranges);
  if (overlaps(ordered))
    return fail(APC_EINVAL, "table buffers or out_digests overlap (a written range meets another range)");
  if ((st = check_device_pointers(ordered, ranges.size(), "out_digests")) != APC_OK) return st;

  unsigned long long *out = reinterpret_cast<unsigned long long *>(out_digests);
  Device d;
  if (!entries.empty() && (st = device_info(&d)) != APC_OK) return st;
  int e = (int)cudaMemsetAsync(out, 0, (size_t)nslots * sizeof(uint64_t), (cudaStream_t)stream);
  if (e) return cuda_fail(e, "cudaMemsetAsync(out_digests)");
  if (entries.empty()) return APC_OK;
  const Grid grid_max = grid_for(d.sms, d.commit);
  return with_plan<apc::kCommitSmall, apc::kCommitMid, apc::kCommitLarge>(entries.size(), [&](auto size) {
    return run_commit_batches<size.value>(entries, h, layout, zero_grad, grid_max, stream, out,
                                          apc::launch_commit<size.value>);
  });
}

}  // namespace

APC_EXPORT apc_status apc_commit_step_ex(const apc_tensor *table, int32_t num_tensors,
                                         const apc_adamw_hparams *hp, int64_t step, uint32_t flags,
                                         apc_stream_t stream, uint64_t *out_digests) {
  g_last_error[0] = 0;
  if (num_tensors < 0) return fail(APC_EINVAL, "num_tensors %d < 0", num_tensors);
  if (num_tensors > 0 && !table) return fail(APC_EINVAL, "table pointer is null");
  std::vector<TableRow> rows((size_t)num_tensors);
  for (int32_t k = 0; k < num_tensors; ++k)
    rows[k] = TableRow{table[k].p, table[k].m, table[k].v, table[k].g, table[k].w, table[k].n,
                       table[k].global_offset};
  return commit_common(apc::kLayoutF32, rows, hp, step, flags, stream, out_digests, 4);
}

APC_EXPORT apc_status apc_commit_step(const apc_tensor *table, int32_t num_tensors, const apc_adamw_hparams *hp,
                                      int64_t step, apc_stream_t stream, uint64_t *out_digests) {
  return apc_commit_step_ex(table, num_tensors, hp, step, 0u, stream, out_digests);
}

APC_EXPORT apc_status apc_commit_step_bf16(const apc_tensor_bf16 *table, int32_t num_tensors,
                                           const apc_adamw_hparams *hp, int64_t step, uint32_t flags,
                                           apc_stream_t stream, uint64_t *out_digests) {
  g_last_error[0] = 0;
  if (num_tensors < 0) return fail(APC_EINVAL, "num_tensors %d < 0", num_tensors);
  if (num_tensors > 0 && !table) return fail(APC_EINVAL, "table pointer is null");
  std::vector<TableRow> rows((size_t)num_tensors);
  for (int32_t k = 0; k < num_tensors; ++k)
    rows[k] = TableRow{table[k].p, table[k].m, table[k].v, table[k].g, nullptr, table[k].n,
                       table[k].global_offset};
  return commit_common(apc::kLayoutBF16, rows, hp, step, flags, stream, out_digests, 3);
}

namespace {

// Validate a buffer list and turn it into digest/count plan entries, ordered
// by type, fp32 first, and inside a type by slot (a sum or a count does not
// depend on the order): the digest kernel shares out each type's tiles on
// their own, and a warp's walk over the plan seldom meets another slot and
// flushes its running sum.
apc_status buffer_entries(const apc_buffer *bufs, int32_t num_bufs, int32_t num_slots, uint64_t *out,
                          std::vector<apc::DigestEntry> *entries) {
  if (num_bufs < 0) return fail(APC_EINVAL, "num_bufs %d < 0", num_bufs);
  if (num_bufs > 0 && !bufs) return fail(APC_EINVAL, "bufs pointer is null");
  if (num_slots < 1 || num_slots > APC_MAX_SLOTS)
    return fail(APC_EINVAL, "num_slots %d outside 1..%d", num_slots, APC_MAX_SLOTS);
  if (!out) return fail(APC_EINVAL, "output pointer is null");
  if ((uintptr_t)out % 8) return fail(APC_EALIGN, "output not 8-byte aligned");
  std::vector<Range> ranges;
  size_t at[2 * APC_MAX_SLOTS + 1] = {0};  // first entry of each (type, slot), then the next one to place
  for (int32_t k = 0; k < num_bufs; ++k) {
    const apc_buffer &b = bufs[k];
    if (b.n && b.dtype <= APC_BF16 && b.slot < APC_MAX_SLOTS) ++at[b.dtype * APC_MAX_SLOTS + b.slot + 1];
  }
  for (int g = 0; g < 2 * APC_MAX_SLOTS; ++g) at[g + 1] += at[g];
  entries->resize(at[2 * APC_MAX_SLOTS]);
  ranges.resize(at[2 * APC_MAX_SLOTS] + 1);  // by type and slot like the entries
  for (int32_t k = 0; k < num_bufs; ++k) {
    const apc_buffer &b = bufs[k];
    if (b.dtype != APC_F32 && b.dtype != APC_BF16) return fail(APC_EINVAL, "bufs[%d]: unknown dtype %u", k, b.dtype);
    if (b.slot >= (uint32_t)num_slots) return fail(APC_EINVAL, "bufs[%d]: slot %u >= num_slots", k, b.slot);
    if (b.n == 0) continue;
    if (!b.data) return fail(APC_EINVAL, "bufs[%d]: null data pointer", k);
    if (b.n > (UINT64_MAX - b.global_offset)) return fail(APC_ERANGE, "bufs[%d]: global_offset + n overflows", k);
    if (b.n > ((uint64_t)1 << 61)) return fail(APC_ERANGE, "bufs[%d]: n too large", k);
    const uintptr_t a = (uintptr_t)b.data;
    const uint64_t es = b.dtype == APC_F32 ? 4 : 2;
    if (a % es) return fail(APC_EALIGN, "bufs[%d]: data not %u-byte aligned", k, (unsigned)es);
    apc::DigestEntry e;
    e.data = b.data;
    e.n = b.n;
    e.key_base = (uint32_t)b.global_offset;
    e.head = (uint8_t)std::min<uint64_t>(((16 - a % 16) % 16) / es, b.n);
    e.dtype = (uint8_t)b.dtype;
    e.slot = (uint8_t)b.slot;
    e.pad_ = 0;
    e.tile_begin = (b.n - e.head) / apc::kVec * apc::kVec;  // the vector body, until placed
    const size_t place = at[b.dtype * APC_MAX_SLOTS + b.slot]++;
    (*entries)[place] = e;
    ranges[place] = {a, a + es * b.n, k, (uint8_t)(kBuffer + b.dtype * APC_MAX_SLOTS + b.slot), false};
  }
  const uintptr_t o = (uintptr_t)out;
  ranges.back() = {o, o + (uintptr_t)num_slots * sizeof(uint64_t), -1, kOut, true};
  const Ordered ordered(ranges);
  if (overlaps(ordered)) return fail(APC_EINVAL, "the output overlaps a buffer of the list");
  return check_device_pointers(ordered, ranges.size(), "output");
}

}  // namespace

APC_EXPORT apc_status apc_digest(const apc_buffer *bufs, int32_t num_bufs, int32_t num_slots, apc_stream_t stream,
                                 uint64_t *out_digests) {
  g_last_error[0] = 0;
  std::vector<apc::DigestEntry> entries;
  apc_status st = buffer_entries(bufs, num_bufs, num_slots, out_digests, &entries);
  if (st != APC_OK) return st;
  unsigned long long *out = reinterpret_cast<unsigned long long *>(out_digests);
  Device d;
  if (!entries.empty() && (st = device_info(&d)) != APC_OK) return st;
  int e = (int)cudaMemsetAsync(out, 0, (size_t)num_slots * sizeof(uint64_t), (cudaStream_t)stream);
  if (e) return cuda_fail(e, "cudaMemsetAsync(out_digests)");
  if (entries.empty()) return APC_OK;
  const Grid grid_max = grid_for(d.sms, d.digest);
  // long tiles where every warp of the grid gets several of them in a launch
  uint64_t body = 0;
  for (const apc::DigestEntry &en : entries) body += en.tile_begin;
  const uint64_t warps = (uint64_t)grid_max.cap * (apc::kThreads / 32);
  const uint64_t launches = ceil_div(entries.size(), apc::kDigestLarge);
  const int u = body / apc::digest_tile(apc::kDigestLong) >= apc::kDigestLongTiles * warps * launches ? apc::kDigestLong
                                                                                                       : apc::kDigestShort;
  return with_plan<apc::kDigestSmall, apc::kDigestMid, apc::kDigestLarge>(entries.size(), [&](auto size) {
    return run_digest_batches<size.value>(
        entries, grid_max, stream, [u](uint64_t n, uint64_t) { return n / apc::digest_tile(u); },
        [&](const auto &plan, unsigned grid) { return apc::launch_digest(plan, u, grid, stream, out); },
        "digest kernel launch");
  });
}

APC_EXPORT apc_status apc_count_nonzero(const apc_buffer *bufs, int32_t num_bufs, int32_t num_slots,
                                        apc_stream_t stream, uint64_t *out_counts) {
  g_last_error[0] = 0;
  std::vector<apc::DigestEntry> entries;
  apc_status st = buffer_entries(bufs, num_bufs, num_slots, out_counts, &entries);
  if (st != APC_OK) return st;
  Device d;
  if (!entries.empty() && (st = device_info(&d)) != APC_OK) return st;
  unsigned long long *out = reinterpret_cast<unsigned long long *>(out_counts);
  int e = (int)cudaMemsetAsync(out, 0, (size_t)num_slots * sizeof(uint64_t), (cudaStream_t)stream);
  if (e) return cuda_fail(e, "cudaMemsetAsync(out_counts)");
  if (entries.empty()) return APC_OK;
  const Grid grid_max = grid_for(d.sms, d.count);
  return with_plan<apc::kDigestSmall, apc::kDigestMid, apc::kDigestLarge>(entries.size(), [&](auto size) {
    return run_digest_batches<size.value>(
        entries, grid_max, stream, [](uint64_t n, uint64_t es) { return n * es / apc::kCountTileBytes; },
        [&](const auto &plan, unsigned grid) { return apc::launch_count(plan, grid, stream, out); },
        "count kernel launch");
  });
}

namespace {

// The device-side address of a source the current device `dev` can read:
// its own device memory, managed memory, page-locked host memory mapped for
// the device, or pageable host memory where the device reads it through the
// host's page tables.  Null if the device cannot read it.
const void *device_readable(const void *p, int dev, bool pageable_ok) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // clear the error state of the failed query
    return pageable_ok ? p : nullptr;
  }
  switch (a.type) {
    case cudaMemoryTypeDevice:
      return a.device == dev ? p : nullptr;
    case cudaMemoryTypeManaged:
      return p;
    case cudaMemoryTypeHost:
      return a.devicePointer;
    default:
      return pageable_ok ? p : nullptr;
  }
}

// Device memory of `dev` (or managed memory) that a kernel may write.
bool device_writable(void *p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged;
}

}  // namespace

APC_EXPORT apc_status apc_upload(const apc_segment *segs, int32_t num_segments, int32_t max_ctas,
                                 apc_stream_t stream) {
  g_last_error[0] = 0;
  if (num_segments < 0) return fail(APC_EINVAL, "num_segments %d < 0", num_segments);
  if (num_segments > 0 && !segs) return fail(APC_EINVAL, "segments pointer is null");
  if (max_ctas < 0 || max_ctas > 4096) return fail(APC_EINVAL, "max_ctas %d outside 0..4096", max_ctas);
  std::vector<apc::UploadEntry> entries;
  entries.reserve((size_t)num_segments);
  int dev = 0, pageable = 0;
  bool queried = false;
  for (int32_t k = 0; k < num_segments; ++k) {
    const apc_segment &g = segs[k];
    if (g.bytes == 0) continue;
    if (!g.dst || !g.src) return fail(APC_EINVAL, "segments[%d]: null pointer", k);
    if (g.bytes > UINTPTR_MAX - (uintptr_t)g.dst || g.bytes > UINTPTR_MAX - (uintptr_t)g.src)
      return fail(APC_ERANGE, "segments[%d]: address + bytes overflows", k);
    if (!queried) {
      int e = (int)cudaGetDevice(&dev);
      if (e) return cuda_fail(e, "cudaGetDevice");
      if ((e = (int)cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, dev)))
        return cuda_fail(e, "cudaDeviceGetAttribute");
      queried = true;
    }
    const void *src = device_readable(g.src, dev, pageable != 0);
    if (!src) return fail(APC_EINVAL, "segments[%d]: the current device cannot read the source", k);
    if (!device_writable(g.dst, dev))
      return fail(APC_EINVAL, "segments[%d]: destination is not memory of the current device", k);
    apc::UploadEntry e{};
    e.dst = static_cast<uint8_t *>(g.dst);
    e.src = static_cast<const uint8_t *>(src);
    e.bytes = g.bytes;
    const uintptr_t d = (uintptr_t)e.dst, s = (uintptr_t)e.src;
    const bool aligned = ((d ^ s) & 15) == 0;
    const uint64_t h0 = (16 - (d & 15)) & 15;  // bytes before the destination's first 16-byte boundary
    const uint64_t head = aligned || h0 == 15 ? h0 : h0 + 16, tail = aligned ? 0 : 16;
    e.body = g.bytes > head + tail ? (g.bytes - head - tail) & ~(uint64_t)15 : 0;
    e.head = (uint32_t)(e.body ? head : std::min<uint64_t>(g.bytes, 64));
    e.shift = e.body ? (uint32_t)((s + head) & 15) : 0;
    entries.push_back(e);
  }
  // destinations must not overlap each other or any source (sorted sweep)
  std::vector<Range> rs;
  rs.reserve(2 * entries.size());
  for (const auto &e : entries) {
    rs.push_back(Range{(uintptr_t)e.dst, (uintptr_t)e.dst + e.bytes, 0, kDest, true});
  }
  for (const auto &e : entries) rs.push_back(Range{(uintptr_t)e.src, (uintptr_t)e.src + e.bytes, 0, kSource, false});
  if (overlaps(Ordered(rs))) return fail(APC_EINVAL, "a destination range overlaps another destination or a source");
  if (entries.empty()) return APC_OK;
  Device d;
  apc_status st = device_info(&d);
  if (st != APC_OK) return st;
  const unsigned cap = max_ctas > 0 ? (unsigned)max_ctas : (unsigned)d.sms;
  std::unique_ptr<apc::UploadPlan<apc::kUploadMax>> plan(new apc::UploadPlan<apc::kUploadMax>);
  size_t i = 0;
  while (i < entries.size()) {
    const size_t k = std::min(entries.size() - i, (size_t)apc::kUploadMax);
    uint64_t tiles = 0;
    for (size_t j = 0; j < k; ++j) {
      apc::UploadEntry e = entries[i + j];
      e.tile_begin = tiles;
      tiles += e.body / apc::kUploadTile;
      plan->e[j] = e;
    }
    plan->count = (uint32_t)k;
    plan->total_tiles = tiles;
    const uint64_t want = std::max<uint64_t>(tiles, k);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, cap));
    int e = apc::launch_upload(*plan, grid, stream);
    if (e) return cuda_fail(e, "upload kernel launch");
    i += k;
  }
  return APC_OK;
}

APC_EXPORT apc_status apc_set_reserved_sms(int32_t n) {
  g_last_error[0] = 0;
  if (n < 0 || n > 1024) return fail(APC_EINVAL, "reserved SMs %d outside 0..1024", n);
  g_reserved_sms.store(n, std::memory_order_relaxed);
  return APC_OK;
}

APC_EXPORT apc_status apc_device_status(void) {
  g_last_error[0] = 0;
  int e = (int)cudaDeviceSynchronize();
  if (e) return cuda_fail(e, "cudaDeviceSynchronize");
  unsigned word = 0;
  if ((e = apc::read_commit_status(&word))) return cuda_fail(e, "reading the device status word");
  if (word & APC_ETIMEOUT) return fail(APC_ETIMEOUT, "a bounded wait inside a kernel gave up");
  return APC_OK;
}

APC_EXPORT apc_status apc_selftest_wait_timeout(uint64_t limit_ns, apc_stream_t stream) {
  g_last_error[0] = 0;
  if (limit_ns < 1 || limit_ns > 10000000000ull) return fail(APC_EINVAL, "limit_ns outside 1..1e10");
  int e = apc::launch_wait_timeout(limit_ns, stream);
  if (e) return cuda_fail(e, "self-test kernel launch");
  return APC_OK;
}

APC_EXPORT const char *apc_status_string(apc_status s) {
  switch (s) {
    case APC_OK: return "APC_OK: success";
    case APC_EINVAL: return "APC_EINVAL: invalid argument";
    case APC_EALIGN: return "APC_EALIGN: misaligned pointer";
    case APC_ERANGE: return "APC_ERANGE: index range overflow";
    case APC_ECUDA: return "APC_ECUDA: CUDA runtime error";
    case APC_ETIMEOUT: return "APC_ETIMEOUT: a bounded wait inside a kernel gave up";
  }
  return "unknown apc_status";
}

APC_EXPORT const char *apc_last_error(void) { return g_last_error; }

APC_EXPORT int32_t apc_version(void) { return 3; }
