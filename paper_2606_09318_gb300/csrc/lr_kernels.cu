// lr_kernels.cu -- CUDA kernels of the sparse ruling-set list ranker (sm_103a).
//
// Pipeline of one call (Section 2.1, Algorithm 1 of "Engineering Scalable
// Distributed List Ranking", restated for one GPU):
//   prep0      level-0 pass: range check, has-predecessor bitmap (findInit),
//              pack succ (and the link weight) into per-element records;
//   heads      per level: classify the heads (initial elements) into sampled
//              rulers, extra rulers and resolved singletons, and number the
//              extra rulers after the sampled ones (pickRulers);
//   chase      per level: one thread per ruler walks succ to the next ruler,
//              rewriting each visited record as (ruler id, offset) and
//              emitting one record of the reduced list (ruler chasing);
//   jump       pointer jumping over a whole level in one launch, once a level
//              is small enough (the base case) or stops shrinking;
//   finalize   per level, deepest first: R_l[i] = R_{l+1}[ruler(i)] - offset(i)
//              (ruler propagation).
// The chase records the *next* ruler, so ranks come out relative to the
// terminal directly and the list never has to be reversed (Section 2.1 notes
// that the distributed algorithm needs a reversal or the post-processing of
// Section 2.5; walking succ forward from each ruler makes both unnecessary).
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include "lr_kernels.h"
#include "lr_ordq.h"

namespace lr {

static std::atomic<int64_t> g_launches{0};
void count_launch(int k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
int64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

// A device attribute that never changes, asked for once (every launch sizes
// its grid by it).  Threads that ask at the same time store the same value.
int cached_per_device(CachedInt &c, int (*ask)(int dev, int arg), int arg) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (dev < 0 || dev >= CachedInt::kDevices) return ask(dev, arg);
  int v = c.value[dev].load(std::memory_order_relaxed);
  if (v == 0) {
    v = ask(dev, arg);
    if (v > 0) c.value[dev].store(v, std::memory_order_relaxed);
  }
  return v > 0 ? v : 1;
}

int device_sm_count() {
  static CachedInt cache;
  return cached_per_device(cache, [](int dev, int) {
    int sms = 0;
    return cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? sms : 0;
  }, 0);
}

int stream_grid(uint64_t work_items, int block) {
  // grid-stride kernels: enough CTAs to fill every SM, no more than needed
  uint64_t want = (work_items + block - 1) / block;
  uint64_t full = (uint64_t)device_sm_count() * (2048 / block);
  if (want < 1) want = 1;
  return (int)(want < full ? want : full);
}

// Launch a kernel that starts with after_previous: it may come while the one
// ahead of it is still running, and so does not pay for its own launch after
// it (validated forest of 2^23, 16 launches: 421 to 401 us; one list of 2^20,
// 5 launches: 119.5 to 116).
template <class... P, class... A>
static void launch_after(void (*kernel)(P...), int grid, int block, cudaStream_t s, A &&...args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Kernels that read or write host memory are bound by the link, which a few
// warps per SM keep busy; the rest of the SM is left to other streams.  (1, 2, 4
// and 8 CTAs per SM measure the same within 1 % from 10^3 to 1.7 * 10^7 elements.)
constexpr int kHostCtasPerSm = 2;
static int host_grid(int grid, bool host) { return host ? std::min(grid, kHostCtasPerSm * device_sm_count()) : grid; }

// The same for a kernel whose registers keep 2048 threads off an SM: the CTAs
// that are resident together, so that the equal shares of a grid-stride loop
// end together (at 40 registers 912 CTAs of 256 run first and the other 304 of
// 1216 after them, on a third of the threads).
template <auto Kernel>
static int fit_grid(uint64_t work_items, int block) {
  static CachedInt cache;
  const int per = cached_per_device(cache, [](int, int b) {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, Kernel, b, 0);
    return nb;
  }, block);
  const uint64_t want = std::max<uint64_t>(1, (work_items + block - 1) / block);
  return (int)std::min<uint64_t>(want, (uint64_t)device_sm_count() * per);
}

// ---------------------------------------------------------------- init
__device__ __forceinline__ void init_levels(LevelDesc *desc, const InitParams &p, int l) {
  if (l < p.nlev) {
    LevelDesc x;
    x.mode = l == 0 ? p.mode0 : (uint32_t)kModeOff;
    x.n = l == 0 ? p.n0 : 0u;
    x.f_inv = p.f_inv[l];
    x.r = l == 0 ? (uint32_t)(((uint64_t)p.n0 + p.f_inv[0] - 1) / p.f_inv[0]) : 0u;
    x.k = 0;
    x.h = 0;
    x.visited = 0;
    x.cap = p.cap[l];
    x.seed = p.seed[l];
    x.hsrc = l == 0 ? (uint32_t)kHeadsBitmap : (uint32_t)kHeadsList;
    x.narrow = kNarrowNone;
    x.picked = 0;
    x.nraw = 0;
    x.check = 0;
    desc[l] = x;
  }
}

// Size, rulers and mode of the level below one with r sampled and k extra
// rulers, of which `heads` are heads.
__device__ __forceinline__ void open_level(LevelDesc &e, uint64_t n1, uint32_t heads, bool last, uint32_t base) {
  e.n = (uint32_t)n1;
  e.r = (uint32_t)((n1 + e.f_inv - 1) / e.f_inv);
  e.h = heads;
  e.mode = n1 <= base || last ? kModeBase : kModeSrs;
}

// One warp: the descriptors; and with a single list (one terminal, and the
// other successors are every id but the head's) its head and level 0's choice
// of rulers, which otherwise takes five more launches.  A second warp copies
// the sums to the host meanwhile (InitParams::publish).
__global__ void __launch_bounds__(64)
k_init(LevelDesc *desc, InitParams p, const unsigned long long *__restrict__ acc, const uint32_t *__restrict__ wflags,
       uint32_t *__restrict__ hlist0, uint32_t *__restrict__ ns, uint32_t *__restrict__ hnext) {
  const uint32_t *heads = p.heads;
  after_previous(desc, acc, wflags, heads);
  if (threadIdx.x >= 32) {
    const int i = (int)threadIdx.x - 32;
    if (!p.publish) return;
    if (i < 6) reinterpret_cast<volatile unsigned long long *>(p.publish + 4)[i] = acc[i];
    if (i == 6 && heads) *reinterpret_cast<volatile uint32_t *>(p.publish + 1) = *heads;
    __threadfence_system();
    __syncwarp();
    if (i == 0) *reinterpret_cast<volatile uint32_t *>(p.publish + kHostToken) = p.token;
    return;
  }
  init_levels(desc, p, (int)threadIdx.x);
  __syncwarp();
  if (threadIdx.x != 0) return;
  LevelDesc &d = desc[0];
  if (wflags) d.narrow = narrow_mode(*wflags);
  if (p.err_bits) record_error(p.err, p.err_bits);
  if (!acc || p.nlev < 2) return;
  const unsigned long long n = p.n0, h = n * (n - 1) / 2 - acc[1];
  if (acc[0] != 1 || h >= n || (heads && *heads != 1) || mostly_local(p.check_local, acc, n) ||
      (p.publish && wflags && d.narrow == kNarrowNone)) {
    if (p.publish) d.mode = kModeOff;
    return;
  }
  hlist0[0] = (uint32_t)h;
  d.h = 1;
  d.hsrc = kHeadsList;
  Perm P;
  P.init(p.n0, p.seed[0]);
  const uint32_t id = P.fwd((uint32_t)h);
  const uint32_t r = (uint32_t)((n + p.f_inv[0] - 1) / p.f_inv[0]);
  const bool sampled = id < r;
  if (!sampled) ns[0] = (uint32_t)h;
  hnext[0] = sampled ? id : r;
  d.k = sampled ? 0u : 1u;
  d.picked = 1u;
  open_level(desc[1], (uint64_t)r + d.k, 1u, p.nlev == 2, p.base);
}

cudaError_t launch_init(LevelDesc *desc, const InitParams &p, const unsigned long long *acc, const uint32_t *wflags,
                        uint32_t *hlist0, uint32_t *ns, uint32_t *hnext, cudaStream_t s) {
  launch_after(k_init, 1, p.publish ? 64 : 32, s, desc, p, acc, wflags, hlist0, ns, hnext);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------- prep0
template <int WT>
__device__ __forceinline__ uint64_t load_weight(const void *w, uint32_t i) {
  if constexpr (WT == 1) return (uint64_t)(int64_t)__ldcs(reinterpret_cast<const int *>(w) + i);
  else if constexpr (WT == 2) return (uint64_t)__ldcs(reinterpret_cast<const long long *>(w) + i);
  else return 1u;
}

// Write the records of elements i0 .. i0 + cnt - 1 (cnt <= 4; i0 a multiple of
// 4), whole sectors at a time.
template <int KIND>
__device__ __forceinline__ void store_records(void *work, uint32_t i0, uint32_t cnt, const uint32_t (&s)[4],
                                              const uint64_t (&w)[4]) {
  if constexpr (KIND == kRecKind16) {
    uint4 *out = reinterpret_cast<uint4 *>(work) + i0;
    if (cnt == 4u) {
      st_sector(out, s[0], kUnvisited, (uint32_t)w[0], (uint32_t)(w[0] >> 32),
                s[1], kUnvisited, (uint32_t)w[1], (uint32_t)(w[1] >> 32));
      st_sector(out + 2, s[2], kUnvisited, (uint32_t)w[2], (uint32_t)(w[2] >> 32),
                s[3], kUnvisited, (uint32_t)w[3], (uint32_t)(w[3] >> 32));
    } else {
      for (uint32_t j = 0; j < cnt; ++j)
        __stcs(out + j, make_uint4(s[j], kUnvisited, (uint32_t)w[j], (uint32_t)(w[j] >> 32)));
    }
  } else {
    uint32_t hi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) hi[j] = KIND == kRecKind8w ? (uint32_t)w[j] : kUnvisited;
    uint2 *out = reinterpret_cast<uint2 *>(work) + i0;
    if (cnt == 4u) {
      st_sector(out, s[0], hi[0], s[1], hi[1], s[2], hi[2], s[3], hi[3]);
    } else {
      for (uint32_t j = 0; j < cnt; ++j) out[j] = make_uint2(s[j], hi[j]);
    }
  }
}

// One record of a coalesced run.
template <int KIND>
__device__ __forceinline__ void store_record(void *work, size_t i, uint32_t s, uint64_t w) {
  if constexpr (KIND == kRecKind16)
    __stcs(reinterpret_cast<uint4 *>(work) + i, make_uint4(s, kUnvisited, (uint32_t)w, (uint32_t)(w >> 32)));
  else
    reinterpret_cast<uint2 *>(work)[i] = make_uint2(s, KIND == kRecKind8w ? (uint32_t)w : kUnvisited);
}

// Add a thread's flags to the call's (whole warps).
__device__ __forceinline__ void add_flags(uint32_t *flags, uint32_t mine) {
  mine = __reduce_or_sync(0xFFFFFFFFu, mine);
  if (mine && (threadIdx.x & 31u) == 0) atomicOr(flags, mine);
}

// One pass over the input: check every successor, mark the has-predecessor
// bit of every successor (the complement gives the heads, Algorithm 1's
// findInit), and pack {succ, kUnvisited[, link weight]} records.  A terminal's
// weight is stored as 0, so every deeper computation can treat weights
// inclusively.
// sums != nullptr: accumulate the number of terminals and the sum of the other
// successors (single-list head, see k_init).  Neither: an input small enough
// for the base case, which needs no heads.
// desc != nullptr: also write the level descriptors (saves k_init's launch).
// KIND: the records (unweighted input may have 16-byte ones too, weight 1, when
// they are to carry terminal ids).
template <int WT, int KIND>
__global__ void __launch_bounds__(256)
k_prep0(const uint32_t *__restrict__ succ, const void *__restrict__ weight, uint32_t n,
        void *__restrict__ work, uint32_t *__restrict__ bitmap, uint32_t *__restrict__ err,
        int validate, int vec, const int64_t *__restrict__ offsets, int32_t k,
        unsigned long long *__restrict__ sums, unsigned long long *__restrict__ local,
        WeightScan scan, LevelDesc *__restrict__ desc, InitParams ip) {
  let_next_come();
  if (scan.unless_narrow && narrow_mode(*scan.unless_narrow)) return;
  if (scan.unless_local && mostly_local(kLocalSampled, scan.unless_local, n)) return;
  uint32_t wide = 0;
  if (desc && blockIdx.x == 0) init_levels(desc, ip, (int)threadIdx.x);
  unsigned long long sT = 0, sS = 0, sL = 0;
  uint32_t term = kEnd;
  const uint32_t ngroups = (uint32_t)(((uint64_t)n + 3u) / 4u);
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < ngroups; g += stride) {
    const uint32_t i0 = g * 4u;
    const uint32_t cnt = min(4u, n - i0);
    uint32_t s[4];
    uint64_t w[4];
    if (vec && cnt == 4u) {
      uint4 v = __ldcs(reinterpret_cast<const uint4 *>(succ + i0));
      s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
      if constexpr (WT == 1) {
        int4 q = __ldcs(reinterpret_cast<const int4 *>(reinterpret_cast<const int *>(weight) + i0));
        w[0] = (uint64_t)(int64_t)q.x; w[1] = (uint64_t)(int64_t)q.y;
        w[2] = (uint64_t)(int64_t)q.z; w[3] = (uint64_t)(int64_t)q.w;
      } else if constexpr (WT == 2) {
        const longlong2 *wp = reinterpret_cast<const longlong2 *>(reinterpret_cast<const long long *>(weight) + i0);
        longlong2 a = __ldcs(wp), b = __ldcs(wp + 1);
        w[0] = (uint64_t)a.x; w[1] = (uint64_t)a.y; w[2] = (uint64_t)b.x; w[3] = (uint64_t)b.y;
      } else {
        w[0] = w[1] = w[2] = w[3] = 1u;
      }
    } else {
      for (uint32_t j = 0; j < 4u; ++j) {
        s[j] = j < cnt ? __ldcs(succ + i0 + j) : 0u;
        w[j] = j < cnt ? load_weight<WT>(weight, i0 + j) : 0u;
      }
    }
    if (scan.succ_copy) {
      for (uint32_t j = 0; j < cnt; ++j) {
        scan.succ_copy[i0 + j] = s[j];
        if constexpr (WT == 1) reinterpret_cast<int *>(scan.weight_copy)[i0 + j] = (int)w[j];
        if constexpr (WT == 2) reinterpret_cast<uint64_t *>(scan.weight_copy)[i0 + j] = w[j];
      }
    }
    if (offsets != nullptr) {
      // batched input: instance of i0 by binary search, then walk forward
      int32_t lo = 0, hi = k;
      while (hi - lo > 1) {
        int32_t mid = (lo + hi) >> 1;
        if ((uint64_t)__ldg(offsets + mid) <= i0) lo = mid; else hi = mid;
      }
      uint64_t base = (uint64_t)__ldg(offsets + lo), end = (uint64_t)__ldg(offsets + lo + 1);
      for (uint32_t j = 0; j < cnt; ++j) {
        const uint32_t i = i0 + j;
        while (i >= end && lo + 1 < k) { ++lo; base = end; end = (uint64_t)__ldg(offsets + lo + 1); }
        const uint64_t g = base + s[j];
        if (i < base || i >= end || (uint64_t)s[j] >= end - base || g >= n) {
          record_error(err, kErrRange);   // successor outside its instance (or a bad table)
          s[j] = i;
        } else {
          s[j] = (uint32_t)g;
        }
      }
    } else {
      for (uint32_t j = 0; j < cnt; ++j)
        if (s[j] >= n) { record_error(err, kErrRange); s[j] = i0 + j; }
    }
    for (uint32_t j = 0; j < cnt; ++j) {
      const uint32_t i = i0 + j;
      if (local) sL += s[j] != i && (s[j] >> kContractTileShift) == (i >> kContractTileShift);
      if (s[j] != i) {
        if (sums) sS += s[j];
        if (bitmap) {
          const uint32_t bit = 1u << (s[j] & 31u);
          if (validate) {
            if (atomicOr(bitmap + (s[j] >> 5), bit) & bit) record_error(err, kErrNotList);
          } else {
            atomicOr(bitmap + (s[j] >> 5), bit);
          }
        }
      } else {
        w[j] = 0u;   // a terminal has no outgoing link
        sT += 1;
        term = i;                              // (of use when it is the only one)
      }
    }
    store_records<KIND>(work, i0, cnt, s, w);
    if constexpr (KIND == kRecKind8w)
      for (uint32_t j = 0; j < cnt; ++j) wide |= wide_flags(w[j]);
  }
  if (KIND == kRecKind8w && scan.flags) add_flags(scan.flags, wide);
  if (sums || local) {
    unsigned long long v[3] = {sT, sS, sL};
    unsigned long long *const to[3] = {sums, sums ? sums + 1 : nullptr, local};   // local: decides whether to contract
    block_add(v, to);
    // only a terminal that its CTA has no second of can be the only one
    if (sums && __syncthreads_count(term != kEnd) == 1 && term != kEnd) sums[kSumTerminal] = term;
  }
}

cudaError_t launch_prep0(const uint32_t *succ, const void *weight, int wtype, uint32_t n,
                         void *work, int kind, uint32_t *bitmap, uint32_t *err, int validate,
                         const int64_t *offsets, int32_t k, unsigned long long *sums,
                         unsigned long long *local, const WeightScan &ws, LevelDesc *desc, const InitParams *init,
                         cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  InitParams ip;
  memset(&ip, 0, sizeof(ip));
  if (desc) ip = *init;
  const int block = 256;
  int vec = ((uintptr_t)succ & 15u) == 0;
  if (wtype == 1) vec = vec && ((uintptr_t)weight & 15u) == 0;
  if (wtype == 2) vec = vec && ((uintptr_t)weight & 15u) == 0;
#define LR_PREP0(WT, KIND)                                                                                        \
  k_prep0<WT, KIND><<<host_grid(fit_grid<k_prep0<WT, KIND>>(((uint64_t)n + 3) / 4, block), ws.succ_copy != nullptr), \
                      block, 0, s>>>(                                                                              \
      succ, weight, n, work, bitmap, err, validate, vec, offsets, k, sums, local, ws, desc, ip)
  const bool w8 = kind == kRecKind8w;
  switch (wtype) {
    case 0: if (kind == kRecKind16) LR_PREP0(0, kRecKind16); else LR_PREP0(0, kRecKind8); break;
    case 1: if (w8) LR_PREP0(1, kRecKind8w); else LR_PREP0(1, kRecKind16); break;
    default: if (w8) LR_PREP0(2, kRecKind8w); else LR_PREP0(2, kRecKind16); break;
  }
#undef LR_PREP0
  count_launch();
  return cudaGetLastError();
}

// Links that stay inside their contraction tile, counted over every 16th
// tile (out[0]: local links, out[1]: elements sampled).  It decides the
// automatic tile-local contraction before a first pass that would pack
// records the contraction does not use.
constexpr uint32_t kLocalSampleEvery = 16;

__global__ void __launch_bounds__(256)
k_local_sample(const uint32_t *__restrict__ succ, uint32_t n, unsigned long long *__restrict__ out) {
  constexpr uint32_t kT = 1u << kContractTileShift;
  const uint64_t tiles = ((uint64_t)n + kT - 1) / kT;
  const uint64_t items = (tiles + kLocalSampleEvery - 1) / kLocalSampleEvery * kT;
  unsigned long long loc = 0, cnt = 0;
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < items;
       e += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t i = (e / kT) * kLocalSampleEvery * kT + (e % kT);
    if (i >= n) continue;
    const uint32_t sx = __ldcs(succ + i);
    cnt += 1;
    loc += sx != (uint32_t)i && (sx >> kContractTileShift) == (uint32_t)(i >> kContractTileShift);
  }
  unsigned long long v[2] = {loc, cnt};
  unsigned long long *const to[2] = {out, out + 1};
  block_add(v, to);
}

cudaError_t launch_local_sample(const uint32_t *succ, uint32_t n, unsigned long long *out, cudaStream_t s) {
  const uint64_t tiles = ((uint64_t)n + (1u << kContractTileShift) - 1) >> kContractTileShift;
  const uint64_t items = (tiles + kLocalSampleEvery - 1) / kLocalSampleEvery << kContractTileShift;
  k_local_sample<<<stream_grid(items, 256), 256, 0, s>>>(succ, n, out);
  count_launch();
  return cudaGetLastError();
}

// The instance of element `base` in a table of k nondecreasing offsets with
// offsets[0] = 0 <= base < offsets[k]: the largest j < k with offsets[j] <=
// base, found by the whole warp at once (every lane probes one of 32 points
// spread over the remaining range, the ballot keeps the last probe at or
// below base), in at most 3 rounds for up to 32768 instances.  Warp-uniform.
__device__ __forceinline__ int32_t warp_instance(const int64_t *__restrict__ offsets, int32_t k, uint64_t base,
                                                 uint32_t lane) {
  int32_t lo = 0, hi = k;
  while (hi - lo > 1) {
    const int64_t span = hi - lo;
    const int32_t q = lo + (int32_t)(((int64_t)(lane + 1) * span) / 33);
    const uint32_t le = __ballot_sync(0xFFFFFFFFu, (uint64_t)__ldg(offsets + q) <= base);
    const int t = __popc(le);
    const int32_t nlo = __shfl_sync(0xFFFFFFFFu, q, t > 0 ? t - 1 : 0);
    const int32_t nhi = __shfl_sync(0xFFFFFFFFu, q, t < 32 ? t : 31);
    if (t > 0) lo = max(lo, nlo);
    if (t < 32) hi = nhi;
  }
  return lo;
}

// The per-instance sums of a warp that walks consecutive elements: what its
// lanes have added for the instance `inst` and not yet passed on.
struct InstSums {
  int32_t inst = -1;
  unsigned long long t = 0, s = 0;
};

// Pass them on (whole warps).
__device__ __forceinline__ void flush_sums(InstSums &a, unsigned long long *isums, uint32_t lane) {
  if (!isums || a.inst < 0) return;
  for (int d = 16; d > 0; d >>= 1) {
    a.t += __shfl_down_sync(0xFFFFFFFFu, a.t, d);
    a.s += __shfl_down_sync(0xFFFFFFFFu, a.s, d);
  }
  if (lane == 0) {
    if (a.t) atomicAdd(isums + 2 * (size_t)a.inst, a.t);
    if (a.s) atomicAdd(isums + 2 * (size_t)a.inst + 1, a.s);
  }
  a.t = a.s = 0;
}

// Groups of 128 consecutive elements that a warp takes at a time.
constexpr uint32_t kMaxRun = 16;
static uint32_t run_groups(uint32_t n, int grid, int block) {
  const uint64_t groups = ((uint64_t)n + 127) / 128, warps = (uint64_t)grid * (block / 32);
  return (uint32_t)std::min<uint64_t>(kMaxRun, std::max<uint64_t>(1, (groups + warps - 1) / warps));
}

// Batched prep without per-element atomics.  Each instance j of a batch that
// is one list has exactly one terminal, and its successors are every local id
// but the head's, so head_j = n_j (n_j - 1) / 2 - sum of its non-terminal
// successors (Section 1.1's findInit, by sums).  isums[2 j] counts instance
// j's terminals and isums[2 j + 1] sums its local successors.  Records as in
// k_prep0.
// A warp takes runs of `run` consecutive groups of 128 elements and passes an
// instance's sums on when it leaves the instance: the warps of a grid are
// mostly in one or two large instances, and the atomics of one address come
// one after another (0.6 ns each: with a pair of them for every group they
// bounded the pass, 2.16 ms for 4.6e8 elements with int64 weights; 1.48 ms, 6.3 TB/s, now).
template <int WT, int KIND>
__global__ void __launch_bounds__(256)
k_prep0_sums(const uint32_t *__restrict__ succ, const void *__restrict__ weight, uint32_t n,
             void *__restrict__ work, WeightScan scan, uint32_t *__restrict__ err, int vec, const int64_t *__restrict__ offsets,
             int32_t k, unsigned long long *__restrict__ isums, uint32_t run) {
  let_next_come();
  if (scan.unless_narrow && narrow_mode(*scan.unless_narrow)) return;
  uint32_t wide = 0;
  const uint32_t ngroups = (uint32_t)(((uint64_t)n + 127u) / 128u);
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = gridDim.x * blockDim.x >> 5;
  const uint32_t lane = threadIdx.x & 31u;
  InstSums acc;
  for (uint64_t r0 = (uint64_t)warp * run; r0 < ngroups; r0 += (uint64_t)warps * run) {
    const uint32_t r1 = (uint32_t)min((uint64_t)ngroups, r0 + run);
    int32_t lo0 = -1;                    // instance of the group's first element (warp-uniform)
    uint64_t ib0 = 0, ie0 = 0;
    for (uint32_t g = (uint32_t)r0; g < r1; ++g) {
      const uint32_t base = g * 128u, i0 = base + lane * 4u;
      const uint32_t cnt = i0 < n ? min(4u, n - i0) : 0u;
      uint32_t s[4] = {0, 0, 0, 0};
      uint64_t w[4] = {1, 1, 1, 1};
      if (vec && cnt == 4u) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(succ + i0));
        s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
        if constexpr (WT == 1) {
          const int4 q = __ldcs(reinterpret_cast<const int4 *>(reinterpret_cast<const int *>(weight) + i0));
          w[0] = (uint64_t)(int64_t)q.x; w[1] = (uint64_t)(int64_t)q.y;
          w[2] = (uint64_t)(int64_t)q.z; w[3] = (uint64_t)(int64_t)q.w;
        } else if constexpr (WT == 2) {
          const longlong2 *wp = reinterpret_cast<const longlong2 *>(reinterpret_cast<const long long *>(weight) + i0);
          const longlong2 a = __ldcs(wp), b = __ldcs(wp + 1);
          w[0] = (uint64_t)a.x; w[1] = (uint64_t)a.y; w[2] = (uint64_t)b.x; w[3] = (uint64_t)b.y;
        }
      } else {
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j)
          if (j < cnt) {
            s[j] = __ldcs(succ + i0 + j);
            w[j] = load_weight<WT>(weight, i0 + j);
          }
      }
      if (base >= ie0) {
        lo0 = warp_instance(offsets, k, base, lane);
        ib0 = (uint64_t)__ldg(offsets + lo0);
        ie0 = (uint64_t)__ldg(offsets + lo0 + 1);
      }
      if (base >= ib0 && (uint64_t)base + 128u <= ie0 && ie0 <= n) {      // the whole group in one instance
        if (acc.inst != lo0) {
          flush_sums(acc, isums, lane);
          acc.inst = lo0;
        }
        const uint32_t ib = (uint32_t)ib0, len = (uint32_t)(ie0 - ib0);
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
          const uint32_t l = i0 + j - ib;
          bool term = s[j] == l;
          if (s[j] >= len) {
            record_error(err, kErrRange);     // successor outside its instance
            term = true;
          }
          if (term) { w[j] = 0u; acc.t += 1; s[j] = l; } else acc.s += s[j];
          s[j] += ib;
        }
      } else {
        // each lane walks forward to its own elements' instances, and passes
        // its sums on when it leaves one
        int32_t lo = lo0;
        uint64_t ib = ib0, ie = ie0;
        unsigned long long sT = 0, sS = 0;
        auto pass_on = [&] {
          if (isums && sT) atomicAdd(isums + 2 * (size_t)lo, sT);
          if (isums && sS) atomicAdd(isums + 2 * (size_t)lo + 1, sS);
          sT = sS = 0;
        };
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
          if (j >= cnt) continue;
          const uint32_t i = i0 + j;
          while (i >= ie && lo + 1 < k) { pass_on(); ++lo; ib = ie; ie = (uint64_t)__ldg(offsets + lo + 1); }
          const uint64_t gl = ib + s[j];
          bool term;
          if (i < ib || i >= ie || (uint64_t)s[j] >= ie - ib || gl >= n) {
            record_error(err, kErrRange);   // successor outside its instance (or a bad table)
            s[j] = i;
            term = true;
          } else {
            term = gl == i;
            if (!term) sS += s[j];          // local id
            s[j] = (uint32_t)gl;
          }
          if (term) { w[j] = 0u; sT += 1; }
        }
        pass_on();
      }
      if (cnt) store_records<KIND>(work, i0, cnt, s, w);
      if constexpr (KIND == kRecKind8w) {
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j)
          if (j < cnt) wide |= wide_flags(w[j]);
      }
    }
  }
  flush_sums(acc, isums, lane);
  if (KIND == kRecKind8w && scan.flags) add_flags(scan.flags, wide);
}

cudaError_t launch_prep0_sums(const uint32_t *succ, const void *weight, int wtype, uint32_t n, void *work, int kind,
                              const WeightScan &ws, uint32_t *err, const int64_t *offsets, int32_t k, unsigned long long *isums,
                              cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int block = 256;
  int vec = ((uintptr_t)succ & 15u) == 0;
  if (wtype != 0) vec = vec && ((uintptr_t)weight & 15u) == 0;
#define LR_SUMS(WT, KIND)                                                                                \
  do {                                                                                                  \
    const int grid = fit_grid<k_prep0_sums<WT, KIND>>(((uint64_t)n + 3) / 4, block);                    \
    k_prep0_sums<WT, KIND><<<grid, block, 0, s>>>(succ, weight, n, work, ws, err, vec, offsets, k, isums, \
                                                  run_groups(n, grid, block));                          \
  } while (0)
  const bool w8 = kind == kRecKind8w;
  switch (wtype) {
    case 0: LR_SUMS(0, kRecKind8); break;
    case 1: if (w8) LR_SUMS(1, kRecKind8w); else LR_SUMS(1, kRecKind16); break;
    default: if (w8) LR_SUMS(2, kRecKind8w); else LR_SUMS(2, kRecKind16); break;
  }
#undef LR_SUMS
  count_launch();
  return cudaGetLastError();
}

// Level-0 heads of a batch from its per-instance sums (one CTA): the head of
// every non-empty instance that has exactly one terminal, listed in instance
// order.  If any non-empty instance has another number of terminals, or the
// heads would not fit the list (capacity hcap), the has-predecessor bitmap
// is used instead: the sums are cleared (they share its memory) and
// k_bitmap0_recs fills it.
__global__ void __launch_bounds__(1024)
k_heads0_batch(LevelDesc *desc, unsigned long long *isums, const int64_t *__restrict__ offsets, int32_t k,
               uint32_t *__restrict__ hlist0, uint32_t hcap, uint32_t n) {
  __shared__ uint64_t sm[33];
  LevelDesc &d = desc[0];
  int fallback = 0;
  uint32_t total = 0;
  for (int32_t j0 = 0; j0 < k; j0 += (int32_t)blockDim.x) {
    const int32_t j = j0 + (int32_t)threadIdx.x;
    uint32_t has = 0;
    uint64_t head = 0;
    if (j < k) {
      const int64_t b0 = offsets[j], b1 = offsets[j + 1];
      if (b0 < 0 || b1 < b0 || (uint64_t)b1 > n) {
        fallback = 1;                        // a bad offset table: the prep reported it
      } else if (b1 > b0) {
        const uint64_t b = (uint64_t)b0, nj = (uint64_t)(b1 - b0);
        const unsigned long long T = isums[2 * (size_t)j], S = isums[2 * (size_t)j + 1];
        const unsigned long long h = nj * (nj - 1) / 2 - S;
        if (T == 1 && h < nj) { has = 1; head = b + h; }
        else fallback = 1;
      }
    }
    uint64_t cnt;
    const uint64_t pos = block_exclusive_scan((uint64_t)has, sm, &cnt);
    if (has && total + pos < hcap) hlist0[total + pos] = (uint32_t)head;
    total += (uint32_t)cnt;
    __syncthreads();
  }
  if (total > hcap) fallback = 1;
  fallback = __syncthreads_or(fallback);
  if (fallback) {
    // the sums occupy the start of the bitmap's memory: clear them
    for (int32_t j = (int32_t)threadIdx.x; j < 2 * k; j += (int32_t)blockDim.x) isums[j] = 0ull;
    if (threadIdx.x == 0) d.hsrc = kHeadsBitmap;
  } else if (threadIdx.x == 0) {
    d.h = total;
    d.hsrc = kHeadsList;
  }
}

// Has-predecessor bitmap from the level-0 records (global successors), only
// when k_heads0_batch fell back to it.
__global__ void __launch_bounds__(256)
k_bitmap0_recs(const LevelDesc *__restrict__ desc, const uint32_t *__restrict__ recs, uint32_t words_per_rec,
               uint32_t n, uint32_t *__restrict__ bitmap) {
  if (desc[0].hsrc != kHeadsBitmap) return;
  if (words_per_rec == 0) words_per_rec = desc[0].narrow ? 2u : 4u;      // kind 8w: as the level decided
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t s = __ldcs(recs + (size_t)i * words_per_rec);
    if (s != i) atomicOr(bitmap + (s >> 5), 1u << (s & 31u));
  }
}

// Lists of a batch from its per-instance sums: every list has one terminal.
__global__ void __launch_bounds__(1024)
k_count_batch(const unsigned long long *__restrict__ isums, int32_t k, uint32_t *__restrict__ out) {
  __shared__ uint64_t sm[33];
  uint64_t t = 0;
  for (int32_t j = (int32_t)threadIdx.x; j < k; j += (int32_t)blockDim.x) t += isums[2 * (size_t)j];
  uint64_t total;
  block_exclusive_scan(t, sm, &total);
  if (threadIdx.x == 0) *out = total > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)total;
}

cudaError_t launch_count_batch(const unsigned long long *isums, int32_t k, uint32_t *out, cudaStream_t s) {
  k_count_batch<<<1, 1024, 0, s>>>(isums, k, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_heads0_batch(LevelDesc *desc, unsigned long long *isums, const int64_t *offsets, int32_t k,
                                uint32_t *hlist0, uint32_t hcap, const void *work, int kind, uint32_t n,
                                uint32_t *bitmap, cudaStream_t s) {
  k_heads0_batch<<<1, 1024, 0, s>>>(desc, isums, offsets, k, hlist0, hcap, n);
  k_bitmap0_recs<<<stream_grid(n, 256), 256, 0, s>>>(desc, reinterpret_cast<const uint32_t *>(work),
                                                      kind == kRecKind8w ? 0u : kind == kRecKind16 ? 4u : 2u, n,
                                                      bitmap);
  count_launch(2);
  return cudaGetLastError();
}

// Batched input given as one device pointer per instance (the serving path
// ranks requests where they already live, without gathering them first).
template <int WT, int KIND>
__global__ void __launch_bounds__(256)
k_prep0_ptrs(const uint32_t *const *__restrict__ sptr, const void *const *__restrict__ wptr,
             uint32_t n, void *__restrict__ work, WeightScan scan, uint32_t *__restrict__ bitmap,
             uint32_t *__restrict__ err, int validate, const int64_t *__restrict__ offsets, int32_t k) {
  if (scan.unless_narrow && narrow_mode(*scan.unless_narrow)) return;
  uint32_t wide = 0;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    int32_t lo = 0, hi = k;
    while (hi - lo > 1) {
      int32_t mid = (lo + hi) >> 1;
      if ((uint64_t)__ldg(offsets + mid) <= i) lo = mid; else hi = mid;
    }
    const uint64_t base = (uint64_t)__ldg(offsets + lo), len = (uint64_t)__ldg(offsets + lo + 1) - base;
    const uint64_t loc = i - base;
    uint32_t s = __ldcs(sptr[lo] + loc);
    uint64_t w = 1u;
    if constexpr (WT == 1) w = (uint64_t)(int64_t)__ldcs(reinterpret_cast<const int *>(wptr[lo]) + loc);
    if constexpr (WT == 2) w = (uint64_t)__ldcs(reinterpret_cast<const long long *>(wptr[lo]) + loc);
    if ((uint64_t)s >= len || base + s >= n) { record_error(err, kErrRange); s = i; }
    else s = (uint32_t)(base + s);
    if (s != i) {
      const uint32_t bit = 1u << (s & 31u);
      if (!bitmap) {
      } else if (validate) {
        if (atomicOr(bitmap + (s >> 5), bit) & bit) record_error(err, kErrNotList);
      } else {
        atomicOr(bitmap + (s >> 5), bit);
      }
    } else {
      w = 0u;
    }
    store_record<KIND>(work, i, s, w);
    if constexpr (KIND == kRecKind8w) wide |= wide_flags(w);
  }
  if (KIND == kRecKind8w && scan.flags) add_flags(scan.flags, wide);
}

cudaError_t launch_prep0_ptrs(const uint32_t *const *sptr, const void *const *wptr, int wtype,
                              uint32_t n, void *work, int kind, const WeightScan &ws, uint32_t *bitmap, uint32_t *err,
                              int validate, const int64_t *offsets, int32_t k, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int block = 256;
  const int grid = stream_grid(n, block);
#define LR_PTRS(WT, KIND) \
  k_prep0_ptrs<WT, KIND><<<grid, block, 0, s>>>(sptr, wptr, n, work, ws, bitmap, err, validate, offsets, k)
  const bool w8 = kind == kRecKind8w;
  switch (wtype) {
    case 0: LR_PTRS(0, kRecKind8); break;
    case 1: if (w8) LR_PTRS(1, kRecKind8w); else LR_PTRS(1, kRecKind16); break;
    default: if (w8) LR_PTRS(2, kRecKind8w); else LR_PTRS(2, kRecKind16); break;
  }
#undef LR_PTRS
  count_launch();
  return cudaGetLastError();
}

// Pointer batches without per-element atomics: the per-instance sums of
// k_prep0_sums, with the same runs, read through one pointer per instance.
// Lane l of a warp takes elements l + 32 j of a group, so that loads and
// record stores are coalesced at any alignment.
template <int WT, int KIND>
__global__ void __launch_bounds__(256)
k_prep0_ptrs_sums(const uint32_t *const *__restrict__ sptr, const void *const *__restrict__ wptr,
                  uint32_t n, void *__restrict__ work, WeightScan scan, uint32_t *__restrict__ err,
                  const int64_t *__restrict__ offsets, int32_t k, unsigned long long *__restrict__ isums,
                  uint32_t run) {
  let_next_come();
  if (scan.unless_narrow && narrow_mode(*scan.unless_narrow)) return;
  uint32_t wide = 0;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t ngroups = (uint32_t)(((uint64_t)n + 127u) / 128u);
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = gridDim.x * blockDim.x >> 5;
  InstSums acc;
  for (uint64_t r0 = (uint64_t)warp * run; r0 < ngroups; r0 += (uint64_t)warps * run) {
    const uint32_t r1 = (uint32_t)min((uint64_t)ngroups, r0 + run);
    int32_t lo0 = -1;                    // instance of the group's first element (warp-uniform)
    uint64_t ib0 = 0, ie0 = 0;
    for (uint32_t g = (uint32_t)r0; g < r1; ++g) {
      const uint64_t base = (uint64_t)g * 128u;
      if (base >= ie0) {
        lo0 = warp_instance(offsets, k, base, lane);
        ib0 = (uint64_t)__ldg(offsets + lo0);
        ie0 = (uint64_t)__ldg(offsets + lo0 + 1);
      }
      // each of the lane's four elements: its instance, then all four loads
      // in flight together
      const bool one = base >= ib0 && ie0 >= min(base + 128u, (uint64_t)n);   // warp-uniform
      int32_t inst[4];
      uint64_t ibv[4], iev[4];
      int32_t lo = lo0;
      uint64_t ib = ib0, ie = ie0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t i = base + lane + 32u * j;
        if (!one)
          while (i < n && i >= ie && lo + 1 < k) { ++lo; ib = ie; ie = (uint64_t)__ldg(offsets + lo + 1); }
        inst[j] = lo;
        ibv[j] = ib;
        iev[j] = ie;
      }
      uint32_t sv[4];
      uint64_t wv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t i = base + lane + 32u * j;
        sv[j] = 0u;
        wv[j] = 1u;
        if (i < n && i >= ibv[j] && i < iev[j]) {
          const uint64_t loc = i - ibv[j];
          sv[j] = __ldcs(sptr[inst[j]] + loc);
          if constexpr (WT == 1) wv[j] = (uint64_t)(int64_t)__ldcs(reinterpret_cast<const int *>(wptr[inst[j]]) + loc);
          if constexpr (WT == 2) wv[j] = (uint64_t)__ldcs(reinterpret_cast<const long long *>(wptr[inst[j]]) + loc);
        }
      }
      if (one && acc.inst != lo0) {
        flush_sums(acc, isums, lane);
        acc.inst = lo0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t i = base + lane + 32u * j;
        if (i >= n) continue;
        uint32_t s = sv[j];
        uint64_t w = wv[j];
        const uint64_t ib = ibv[j], ie = iev[j];
        bool term;
        if (i < ib || i >= ie) {
          record_error(err, kErrRange);     // a bad offset table
          s = (uint32_t)i;
          term = true;
        } else if ((uint64_t)s >= ie - ib || ib + s >= n) {
          record_error(err, kErrRange);     // successor outside its instance
          s = (uint32_t)i;
          term = true;
        } else {
          term = (uint64_t)s == i - ib;
          if (!term) {
            if (one) acc.s += s;
            else if (isums) atomicAdd(isums + 2 * (size_t)inst[j] + 1, (unsigned long long)s);
          }
          s = (uint32_t)(ib + s);
        }
        if (term) {
          w = 0u;
          if (one) acc.t += 1;
          else if (isums) atomicAdd(isums + 2 * (size_t)inst[j], 1ull);
        }
        store_record<KIND>(work, i, s, w);
        if constexpr (KIND == kRecKind8w) wide |= wide_flags(w);
      }
    }
  }
  flush_sums(acc, isums, lane);
  if (KIND == kRecKind8w && scan.flags) add_flags(scan.flags, wide);
}

cudaError_t launch_prep0_ptrs_sums(const uint32_t *const *sptr, const void *const *wptr, int wtype, uint32_t n,
                                   void *work, int kind, const WeightScan &ws, uint32_t *err, const int64_t *offsets,
                                   int32_t k, unsigned long long *isums, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int block = 256;
#define LR_PTRS_SUMS(WT, KIND)                                                                           \
  do {                                                                                                  \
    const int grid = fit_grid<k_prep0_ptrs_sums<WT, KIND>>(((uint64_t)n + 3) / 4, block);               \
    k_prep0_ptrs_sums<WT, KIND><<<grid, block, 0, s>>>(sptr, wptr, n, work, ws, err, offsets, k, isums, \
                                                       run_groups(n, grid, block));                     \
  } while (0)
  const bool w8 = kind == kRecKind8w;
  switch (wtype) {
    case 0: LR_PTRS_SUMS(0, kRecKind8); break;
    case 1: if (w8) LR_PTRS_SUMS(1, kRecKind8w); else LR_PTRS_SUMS(1, kRecKind16); break;
    default: if (w8) LR_PTRS_SUMS(2, kRecKind8w); else LR_PTRS_SUMS(2, kRecKind16); break;
  }
#undef LR_PTRS_SUMS
  count_launch();
  return cudaGetLastError();
}

// Number of heads (zero bits of the has-predecessor bitmap below n).
__global__ void k_count_heads(const uint32_t *__restrict__ bitmap, uint32_t n, uint32_t *out) {
  after_previous(bitmap);
  const uint32_t words = (uint32_t)(((uint64_t)n + 31u) / 32u);
  uint32_t c = 0;
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < words; w += gridDim.x * blockDim.x) {
    uint32_t bits = ~__ldcg(bitmap + w);
    if (w == words - 1u && (n & 31u)) bits &= (1u << (n & 31u)) - 1u;
    c += __popc(bits);
  }
  __shared__ uint32_t heads;
  if (threadIdx.x == 0) heads = 0;
  __syncthreads();
  c = __reduce_add_sync(0xFFFFFFFFu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&heads, c);
  __syncthreads();
  if (threadIdx.x == 0 && heads) atomicAdd(out, heads);
}

cudaError_t launch_count_heads(const uint32_t *bitmap, uint32_t n, uint32_t *out, cudaStream_t s) {
  const int block = 256;
  const int grid = stream_grid(((uint64_t)n + 31u) / 32u, block);
  launch_after(k_count_heads, grid, block, s, bitmap, n, out);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------- heads
enum : int { kCatSampled = 0, kCatNew = 1, kCatSingle = 2 };

// Classify head x of a level: a sampled ruler keeps id pi(x); a head that is
// also a terminal is a one-element list whose rank is its own weight
// (resolved here, never chased); any other head becomes an extra ruler.
// (A level of 8-byte weighted records: `narrow` says whether it has them.)
template <class Rec, bool RESOLVE>
__device__ __forceinline__ int classify_head(uint32_t x, const Perm &P, uint32_t r, uint32_t narrow,
                                             const Rec *work, uint32_t *pid, uint64_t *wself) {
  const uint32_t p = P.fwd(x);
  *pid = p;
  if (p < r) return kCatSampled;
  if constexpr (RESOLVE && std::is_same<Rec, Rec8w>::value) {
    const uint32_t s = narrow ? ld_rec(work + x).lo : ld_rec(reinterpret_cast<const Rec16 *>(work) + x).succ;
    if (s == x) { *wself = 0; return kCatSingle; }     // level 0: a terminal weighs 0
  } else if constexpr (RESOLVE) {
    Rec v = ld_rec(work + x);
    if (rec_succ(v) == x) { *wself = rec_weight(v, x); return kCatSingle; }
  }
  return kCatNew;
}

// Visit this thread's heads in a fixed order (deterministic numbering).
template <class F>
__device__ __forceinline__ void for_each_head(const LevelDesc &d, const uint32_t *bitmap,
                                              const uint32_t *hlist, F &&f) {
  if (d.hsrc == kHeadsBitmap) {
    const uint32_t words = (uint32_t)(((uint64_t)d.n + 31u) / 32u);
    const uint32_t per = (words + gridDim.x - 1) / gridDim.x;
    const uint32_t w0 = blockIdx.x * per, w1 = min(words, w0 + per);
    for (uint32_t w = w0 + threadIdx.x; w < w1; w += blockDim.x) {
      uint32_t bits = ~__ldcg(bitmap + w);
      if (w == words - 1u && (d.n & 31u)) bits &= (1u << (d.n & 31u)) - 1u;
      while (bits) {
        const uint32_t b = __ffs(bits) - 1;
        bits &= bits - 1u;
        f(w * 32u + b);
      }
    }
  } else {
    const uint32_t cnt = d.h;
    const uint32_t per = (cnt + gridDim.x - 1) / gridDim.x;
    const uint32_t e0 = blockIdx.x * per, e1 = min(cnt, e0 + per);
    for (uint32_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) f(__ldcg(hlist + e));
  }
}

template <class Rec, bool RESOLVE>
__global__ void __launch_bounds__(kHeadThreads)
k_heads_count(const LevelDesc *__restrict__ desc, int lev, const uint32_t *__restrict__ bitmap,
              const uint32_t *__restrict__ hlist, const Rec *__restrict__ work,
              uint64_t *__restrict__ blockcnt) {
  after_previous(desc);
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || d.picked) return;
  Perm P;
  P.init(d.n, d.seed);
  uint32_t nS = 0, nN = 0;
  for_each_head(d, bitmap, hlist, [&](uint32_t x) {
    uint32_t p;
    uint64_t w;
    const int c = classify_head<Rec, RESOLVE>(x, P, d.r, d.narrow, work, &p, &w);
    nS += c == kCatSampled;
    nN += c == kCatNew;
  });
  uint64_t total;
  block_exclusive_scan(((uint64_t)(nS + nN) << 32) | nN, sm, &total);
  if (threadIdx.x == 0) blockcnt[blockIdx.x] = total;
}

// Exclusive scan of the per-CTA counts; sizes of the next level; its mode.
__global__ void __launch_bounds__(kHeadBlocks)
k_heads_scan(LevelDesc *desc, int lev, int nlev, uint64_t *blockcnt, uint32_t *err,
             uint32_t cutoff, uint32_t hcap) {
  after_previous(desc);
  __shared__ uint64_t sm[33];
  if (desc[lev].mode != kModeSrs || desc[lev].picked) return;
  uint64_t total;
  const uint64_t v = blockcnt[threadIdx.x];
  const uint64_t ex = block_exclusive_scan(v, sm, &total);
  blockcnt[threadIdx.x] = ex;
  if (threadIdx.x == 0) {
    LevelDesc &d = desc[lev];
    LevelDesc &e = desc[lev + 1];
    const uint32_t kNew = (uint32_t)total;
    const uint32_t hNext = (uint32_t)(total >> 32);
    const uint64_t n1 = (uint64_t)d.r + kNew;
    d.k = kNew;
    if (hNext > hcap || n1 > e.cap) {
      record_error(err, kErrCapacity);
      d.mode = kModeOff;      // nothing more runs at this level or below
      return;
    }
    open_level(e, n1, hNext, lev + 1 >= nlev - 1, cutoff);
  }
}

template <class Rec, bool RESOLVE>
__global__ void __launch_bounds__(kHeadThreads)
k_heads_write(LevelDesc *__restrict__ desc, int lev, const uint32_t *__restrict__ bitmap,
              const uint32_t *__restrict__ hlist, Rec *__restrict__ work,
              uint32_t *__restrict__ ns, uint32_t *__restrict__ hnext,
              const uint64_t *__restrict__ blockoff) {
  after_previous(desc);
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || d.picked) return;
  Perm P;
  P.init(d.n, d.seed);
  uint32_t nS = 0, nN = 0;
  for_each_head(d, bitmap, hlist, [&](uint32_t x) {
    uint32_t p;
    uint64_t w;
    const int c = classify_head<Rec, RESOLVE>(x, P, d.r, d.narrow, work, &p, &w);
    nS += c == kCatSampled;
    nN += c == kCatNew;
  });
  const uint64_t mine = block_exclusive_scan(((uint64_t)(nS + nN) << 32) | nN, sm, nullptr);
  const uint64_t base = blockoff[blockIdx.x] + mine;
  uint32_t posN = (uint32_t)base, posH = (uint32_t)(base >> 32), nZ = 0;
  for_each_head(d, bitmap, hlist, [&](uint32_t x) {
    uint32_t p;
    uint64_t w;
    const int c = classify_head<Rec, RESOLVE>(x, P, d.r, d.narrow, work, &p, &w);
    if (c == kCatSampled) {
      hnext[posH++] = p;
    } else if (c == kCatNew) {
      ns[posN] = x;
      hnext[posH++] = d.r + posN;
      ++posN;
    } else {
      if (std::is_same<Rec, Rec8w>::value && !d.narrow)
        st_rec(reinterpret_cast<Rec16 *>(work) + x, kZeroCid, 0);
      else
        st_rec(work + x, kZeroCid, (uint64_t)0 - w);   // R(x) = 0 - (-w) = w
      ++nZ;
    }
  });
  for (int dd = 16; dd > 0; dd >>= 1) nZ += __shfl_down_sync(0xFFFFFFFFu, nZ, dd);
  if ((threadIdx.x & 31) == 0 && nZ) atomicAdd(&desc[lev].visited, nZ);
}

// The same for a level whose few heads come as a list: one CTA, one launch.
constexpr uint32_t kFewHeads = 2048;
template <class Rec>
__global__ void __launch_bounds__(1024)
k_heads_few(LevelDesc *desc, int lev, int nlev, const uint32_t *__restrict__ hlist, Rec *__restrict__ work,
            uint32_t *__restrict__ ns, uint32_t *__restrict__ hnext, uint32_t *__restrict__ err, uint32_t cutoff,
            uint32_t hcap) {
  after_previous(desc);
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || d.picked) return;
  Perm P;
  P.init(d.n, d.seed);
  uint32_t nN = 0, nH = 0, nZ = 0;               // extra rulers, heads below, resolved so far
  for (uint32_t e0 = 0; e0 < d.h; e0 += blockDim.x) {
    const uint32_t e = e0 + threadIdx.x;
    uint32_t x = 0, p = 0;
    uint64_t w = 0;
    int c = -1;
    if (e < d.h) {
      x = __ldcg(hlist + e);
      c = classify_head<Rec, true>(x, P, d.r, d.narrow, work, &p, &w);
    }
    const bool isnew = c == kCatNew, ishead = isnew || c == kCatSampled;
    uint64_t total;
    const uint64_t at = block_exclusive_scan(((uint64_t)ishead << 32) | (isnew ? 1u : 0u), sm, &total);
    const uint32_t posN = nN + (uint32_t)at, posH = nH + (uint32_t)(at >> 32);
    // (the list itself is no longer than hcap, and so is what it leaves)
    if (ishead && posH < hcap) hnext[posH] = isnew ? d.r + posN : p;
    if (isnew && posN < hcap) ns[posN] = x;
    if (c == kCatSingle) st_rec(work + x, kZeroCid, (uint64_t)0 - w);
    nZ += __syncthreads_count(c == kCatSingle);
    nN += (uint32_t)total;
    nH += (uint32_t)(total >> 32);
  }
  if (threadIdx.x == 0) {
    LevelDesc &m = desc[lev];
    LevelDesc &e = desc[lev + 1];
    const uint64_t n1 = (uint64_t)d.r + nN;
    m.k = nN;
    m.visited += nZ;
    if (nH > hcap || n1 > e.cap) {
      record_error(err, kErrCapacity);
      m.mode = kModeOff;
      return;
    }
    open_level(e, n1, nH, lev + 1 >= nlev - 1, cutoff);
  }
}

// A batch of one list per instance: what k_init, k_count_batch,
// k_heads0_batch and the ruler selection do, in one CTA that needs no bitmap
// and whose result the host reads while the chase runs (48 requests, 3 million
// elements: the call 495 us with the seven launches and the wait, 449 with
// this).  The first pass over the instances only looks, so that a batch of
// another kind is left as it was found.
template <class Rec>
__global__ void __launch_bounds__(1024)
k_open_batch(LevelDesc *desc, InitParams p, const unsigned long long *__restrict__ isums,
             const int64_t *__restrict__ offsets, int32_t k, const uint32_t *__restrict__ wflags,
             Rec *__restrict__ work, uint32_t *__restrict__ ns, uint32_t *__restrict__ hnext) {
  after_previous(isums, offsets, wflags);
  __shared__ uint64_t sm[33];
  init_levels(desc, p, (int)threadIdx.x);
  const uint32_t n = p.n0;
  const uint32_t narrow = std::is_same<Rec, Rec8w>::value && wflags ? narrow_mode(*wflags) : kNarrowNone;
  // the head of instance j; false: none (empty), or (ok cleared) not one list
  auto head_of = [&](int32_t j, bool &ok, uint64_t &terms, uint32_t &x) -> bool {
    const int64_t b0 = offsets[j], b1 = offsets[j + 1];
    const unsigned long long T = isums[2 * (size_t)j], S = isums[2 * (size_t)j + 1];
    terms += T;
    if (b0 < 0 || b1 < b0 || (uint64_t)b1 > n) { ok = false; return false; }
    const uint64_t nj = (uint64_t)(b1 - b0), h = nj * (nj - 1) / 2 - S;
    if (nj == 0) return false;
    if (T != 1 || h >= nj) { ok = false; return false; }
    x = (uint32_t)((uint64_t)b0 + h);
    return true;
  };
  bool ok = !(std::is_same<Rec, Rec8w>::value && wflags && narrow == kNarrowNone);
  uint64_t terms = 0, total;
  uint32_t heads = 0;
  for (int32_t j = (int32_t)threadIdx.x; j < k; j += (int32_t)blockDim.x) {
    uint32_t x;
    heads += head_of(j, ok, terms, x);
  }
  block_exclusive_scan(terms, sm, &total);
  ok = __syncthreads_and(ok);
  if (threadIdx.x == 32) {
    volatile uint32_t *w = p.publish;
    w[1] = total > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)total;
    w[2] = ok;
    w[12] = wflags ? *wflags : 0u;
    __threadfence_system();
    w[kHostToken] = p.token;
  }
  LevelDesc &m = desc[0];
  if (!ok) {
    if (threadIdx.x == 0) m.mode = kModeOff;
    return;
  }
  Perm P;
  P.init(n, p.seed[0]);
  const uint32_t r = (uint32_t)(((uint64_t)n + p.f_inv[0] - 1) / p.f_inv[0]);
  uint32_t nN = 0, nH = 0, nZ = 0;               // extra rulers, heads below, resolved so far
  for (int32_t j0 = 0; j0 < k; j0 += (int32_t)blockDim.x) {
    const int32_t j = j0 + (int32_t)threadIdx.x;
    uint32_t x = 0, id = 0;
    uint64_t w = 0, t = 0;
    int c = -1;
    bool fine = true;
    if (j < k && head_of(j, fine, t, x)) c = classify_head<Rec, true>(x, P, r, narrow, work, &id, &w);
    const bool isnew = c == kCatNew, ishead = isnew || c == kCatSampled;
    const uint64_t at = block_exclusive_scan(((uint64_t)ishead << 32) | (isnew ? 1u : 0u), sm, &total);
    const uint32_t posN = nN + (uint32_t)at, posH = nH + (uint32_t)(at >> 32);
    if (ishead) hnext[posH] = isnew ? r + posN : id;      // (the lists hold k)
    if (isnew) ns[posN] = x;
    if (c == kCatSingle) st_rec(work + x, kZeroCid, (uint64_t)0 - w);
    nZ += __syncthreads_count(c == kCatSingle);
    nN += (uint32_t)total;
    nH += (uint32_t)(total >> 32);
  }
  if (threadIdx.x == 0) {
    m.narrow = narrow;
    m.h = nH + nZ;
    m.hsrc = kHeadsList;
    m.k = nN;
    m.visited = nZ;
    m.picked = 1u;
    open_level(desc[1], (uint64_t)r + nN, nH, p.nlev == 2, p.base);
  }
}

cudaError_t launch_open_batch(LevelDesc *desc, const InitParams &p, const unsigned long long *isums,
                              const int64_t *offsets, int32_t k, const uint32_t *wflags, void *work, int kind,
                              uint32_t *ns, uint32_t *hnext, cudaStream_t s) {
#define LR_OPEN(REC)                                                                                              \
  launch_after(k_open_batch<REC>, 1, 1024, s, desc, p, isums, offsets, k, wflags, reinterpret_cast<REC *>(work), ns, hnext)
  if (kind == kRecKind8w) LR_OPEN(Rec8w);
  else if (kind == kRecKind16) LR_OPEN(Rec16);
  else LR_OPEN(Rec8);
#undef LR_OPEN
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_heads(LevelDesc *desc, int lev, int nlev, const uint32_t *bitmap,
                         const uint32_t *hlist, void *work, int rec_kind, uint32_t *ns,
                         uint32_t *hnext, uint64_t *blockcnt, uint32_t *err, uint32_t cutoff,
                         uint32_t hcap, cudaStream_t s) {
  if (lev > 0 && hcap <= kFewHeads) {
    launch_after(k_heads_few<Rec16>, 1, 1024, s, desc, lev, nlev, hlist, reinterpret_cast<Rec16 *>(work), ns, hnext, err,
                                          cutoff, hcap);
    count_launch();
    return cudaGetLastError();
  }
#define LR_HEADS(KERNEL, REC, RES)                                                                \
  launch_after(KERNEL<REC, RES>, kHeadBlocks, kHeadThreads, s,
  switch (rec_kind) {
    case kRecKind8:
      LR_HEADS(k_heads_count, Rec8, true) desc, lev, bitmap, hlist, reinterpret_cast<const Rec8 *>(work), blockcnt);
      break;
    case kRecKind16:
      LR_HEADS(k_heads_count, Rec16, true) desc, lev, bitmap, hlist, reinterpret_cast<const Rec16 *>(work), blockcnt);
      break;
    case kRecKind8w:
      LR_HEADS(k_heads_count, Rec8w, true) desc, lev, bitmap, hlist, reinterpret_cast<const Rec8w *>(work), blockcnt);
      break;
    default:
      LR_HEADS(k_heads_count, Succ4, false) desc, lev, bitmap, hlist, reinterpret_cast<const Succ4 *>(work), blockcnt);
      break;
  }
  launch_after(k_heads_scan, 1, kHeadBlocks, s, desc, lev, nlev, blockcnt, err, cutoff, hcap);
  switch (rec_kind) {
    case kRecKind8:
      LR_HEADS(k_heads_write, Rec8, true) desc, lev, bitmap, hlist, reinterpret_cast<Rec8 *>(work), ns, hnext, blockcnt);
      break;
    case kRecKind16:
      LR_HEADS(k_heads_write, Rec16, true) desc, lev, bitmap, hlist, reinterpret_cast<Rec16 *>(work), ns, hnext, blockcnt);
      break;
    case kRecKind8w:
      LR_HEADS(k_heads_write, Rec8w, true) desc, lev, bitmap, hlist, reinterpret_cast<Rec8w *>(work), ns, hnext, blockcnt);
      break;
    default:
      LR_HEADS(k_heads_write, Succ4, false) desc, lev, bitmap, hlist, reinterpret_cast<Succ4 *>(work), ns, hnext, blockcnt);
      break;
  }
#undef LR_HEADS
  count_launch(3);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- ruler order
// Sampled rulers in element order, for inputs made of contiguous instances
// (a batch; each of its levels keeps every instance's elements together).  A chase that takes its rulers in this order works on
// a few instances at a time, so the records it reads and rewrites at random
// stay within a footprint the L2 can hold, where the default order (ruler
// ids, i.e. random positions) touches the whole input at once.  The sampled
// rulers are the same set (pi(x) < r); only their order and ids change: the
// id of the ruler at position x is the number of sampled rulers before x, so
// the reduced records and the final pass's rank gathers are local too.
//   mark:  bit x of `bits` for every sampled ruler x = pi^{-1}(c), c < r;
//   count: set bits per CTA (a contiguous run of words per thread);
//   scan:  exclusive prefix of the per-CTA counts;
//   write: each thread lists the positions of its run's set bits, in order,
//          and the count before every 256-position block (cum).
__global__ void __launch_bounds__(256)
k_ord_mark(const LevelDesc *__restrict__ desc, int lev, uint32_t *__restrict__ bits) {
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs) return;
  Perm P;
  P.init(d.n, d.seed);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < d.r; c += stride) {
    const uint32_t x = P.inv((uint32_t)c);
    atomicOr(bits + (x >> 5), 1u << (x & 31u));
  }
}

// Words [c0, c1) of this CTA: a contiguous share, read in tiles of one word
// per thread (coalesced).
__device__ __forceinline__ void ord_range(uint32_t words, uint32_t *c0, uint32_t *c1) {
  const uint32_t per_cta = (words + gridDim.x - 1) / gridDim.x;
  *c0 = min(words, blockIdx.x * per_cta);
  *c1 = min(words, *c0 + per_cta);
}

__global__ void __launch_bounds__(kHeadThreads)
k_ord_count(const LevelDesc *__restrict__ desc, int lev, const uint32_t *__restrict__ bits,
            uint64_t *__restrict__ cnt) {
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs) return;
  uint32_t c0, c1, m = 0;
  ord_range((uint32_t)(((uint64_t)d.n + 31u) / 32u), &c0, &c1);
  for (uint32_t w = c0 + threadIdx.x; w < c1; w += blockDim.x) m += __popc(__ldcg(bits + w));
  uint64_t total;
  block_exclusive_scan(m, sm, &total);
  if (threadIdx.x == 0) cnt[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kHeadBlocks)
k_ord_scan(const LevelDesc *__restrict__ desc, int lev, uint64_t *__restrict__ cnt, uint32_t *__restrict__ err) {
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs) return;
  uint64_t total;
  const uint64_t ex = block_exclusive_scan(cnt[threadIdx.x], sm, &total);
  cnt[threadIdx.x] = ex;
  if (threadIdx.x == 0 && total != d.r) record_error(err, kErrInternal);   // pi is a bijection
}

// Tile by tile: each thread one word, the tile's exclusive scan of their
// counts, then each thread lists its word's marks in ascending order.
__global__ void __launch_bounds__(kHeadThreads)
k_ord_write(const LevelDesc *__restrict__ desc, int lev, const uint32_t *__restrict__ bits,
            const uint64_t *__restrict__ cnt, uint32_t *__restrict__ ord, uint32_t *__restrict__ cum) {
  __shared__ uint64_t sm[33];
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs) return;
  uint32_t c0, c1;
  ord_range((uint32_t)(((uint64_t)d.n + 31u) / 32u), &c0, &c1);
  uint64_t base = cnt[blockIdx.x];
  for (uint32_t t0 = c0; t0 < c1; t0 += blockDim.x) {     // uniform trip count in the CTA
    const uint32_t w = t0 + threadIdx.x;
    uint32_t b = w < c1 ? __ldcg(bits + w) : 0u;
    uint64_t tile;
    uint64_t pos = base + block_exclusive_scan(__popc(b), sm, &tile);
    if (w < c1 && (w & 7u) == 0) cum[w >> 3] = (uint32_t)pos;
    while (b) {
      const uint32_t i = __ffs(b) - 1;
      b &= b - 1u;
      if (pos < d.r) ord[pos] = w * 32u + i;
      ++pos;
    }
    base += tile;
  }
}

// Id of the sampled ruler at position y: rulers before y's 256-position
// block plus the marks before y inside it (one 32-byte read of the block's
// eight words).
__device__ __forceinline__ uint32_t ord_id(const uint32_t *__restrict__ bits, const uint32_t *__restrict__ cum,
                                           uint32_t y) {
  const uint32_t b = y >> 8;
  const uint4 *wp = reinterpret_cast<const uint4 *>(bits) + 2 * (size_t)b;
  const uint4 lo = __ldcg(wp), hi = __ldcg(wp + 1);
  uint32_t id = __ldcg(cum + b);
  const uint32_t wi = (y >> 5) & 7u;
  const uint32_t m = (1u << (y & 31u)) - 1u;
  const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i) id += __popc(i < wi ? w[i] : (i == wi ? (w[i] & m) : 0u));
  return id;
}

// The next level's head list named the sampled heads by pi(x); give them
// their ids in element order.
__global__ void __launch_bounds__(256)
k_ord_heads(const LevelDesc *__restrict__ desc, int lev, uint32_t *__restrict__ hnext, OrdArgs oa) {
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs) return;
  Perm P;
  P.init(d.n, d.seed);
  const uint32_t h = desc[lev + 1].h;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < h; e += gridDim.x * blockDim.x) {
    const uint32_t v = hnext[e];
    if (v < d.r) hnext[e] = ord_id(oa.bits, oa.cum, P.inv(v));
  }
}

cudaError_t launch_order(LevelDesc *desc, int lev, uint32_t cap, uint64_t *cnt, const OrdArgs *oa,
                         uint32_t *hnext, uint32_t hcap, uint32_t *err, cudaStream_t s) {
  // whole 256-position blocks, so that a lookup may read all 8 words of one
  cudaError_t e = cudaMemsetAsync(oa->bits, 0, 32 * (((uint64_t)cap + 255u) / 256u), s);
  if (e != cudaSuccess) return e;
  k_ord_mark<<<stream_grid(cap / 8 + 1, 256), 256, 0, s>>>(desc, lev, oa->bits);
  k_ord_count<<<kHeadBlocks, kHeadThreads, 0, s>>>(desc, lev, oa->bits, cnt);
  k_ord_scan<<<1, kHeadBlocks, 0, s>>>(desc, lev, cnt, err);
  k_ord_write<<<kHeadBlocks, kHeadThreads, 0, s>>>(desc, lev, oa->bits, cnt, oa->ord, oa->cum);
  k_ord_heads<<<stream_grid(hcap, 256), 256, 0, s>>>(desc, lev, hnext, *oa);
  count_launch(5);
  return cudaGetLastError();
}

// A CTA's end of the ordered queue (lr_ordq.h), in shared memory.
struct OrdQueue {
  unsigned long long win, next;    // the window; the chunk after it (0: not there)
  uint32_t out;                    // the sequence has run out
};

struct OrdAccess {
  OrdQueue &q;
  uint32_t *counter;
  __device__ __forceinline__ void exchange_window(unsigned long long w) const { atomicExch(&q.win, w); }
  __device__ __forceinline__ unsigned long long window() const { return *(volatile unsigned long long *)&q.win; }
  __device__ __forceinline__ unsigned long long exchange_next(unsigned long long w) const { return atomicExch(&q.next, w); }
  __device__ __forceinline__ uint32_t draw(uint32_t c) const { return atomicAdd(counter, c); }
  __device__ __forceinline__ bool out() const { return *(volatile uint32_t *)&q.out != 0u; }
  __device__ __forceinline__ void set_out() const { *(volatile uint32_t *)&q.out = 1u; }
};

// Position for this lane (total or more: none left); one request for all the
// lanes that ask together.  *fresh: set on the lane that drew a chunk, to the
// chunk's first position.
__device__ __forceinline__ uint32_t ord_take(OrdQueue &q, uint32_t *gq, uint32_t total, uint32_t *fresh) {
  const uint32_t mask = __activemask();
  const uint32_t lane = threadIdx.x & 31u, leader = __ffs(mask) - 1;
  const uint32_t cnt = __popc(mask), mine = __popc(mask & ((1u << lane) - 1u));
  unsigned long long w = 0, more = 0;
  if (lane == leader) {
    w = atomicAdd(&q.win, (unsigned long long)cnt);
    more = ord_ask(OrdAccess{q, gq}, w, cnt, total, fresh);
  }
  w = __shfl_sync(mask, w, leader);
  const uint32_t have = ord_window_has(w, cnt);          // the same in every lane
  if (have < cnt) more = __shfl_sync(mask, more, leader);
  return ord_position(w, have, more, total, mine);
}

// ---------------------------------------------------------------- chase
// Persistent CTAs; CTA b owns a contiguous slice of ruler ids and its threads
// pull ids one at a time from a per-CTA counter (the next id is requested
// while the current chain runs, hiding the atomic's latency).  Each thread
// walks succ from its ruler until it meets the next ruler (pi(y) < r) or a
// terminal, rewriting every visited record as (ruler id, offset).
// Visit one record: return its old contents and rewrite it as (cid, off)
// unless another chase got there first.  XCHG: one atomic exchange at L2;
// otherwise the store is issued only after the load has returned (it depends
// on the loaded tag), so it always hits the sector the load just brought in.
template <bool XCHG, class Rec>
__device__ __forceinline__ Rec visit(Rec *p, uint32_t cid, uint64_t off) {
  if constexpr (XCHG) {
    return xchg_rec(p, cid, off);
  } else {
    Rec v = ld_rec(p);
    if (rec_tag(v) == kUnvisited) st_rec(p, cid, off);
    return v;
  }
}

// A level of one kind of weighted records is none of the other kind's business.
template <class Rec>
__device__ __forceinline__ bool wrong_kind(const LevelDesc &d) {
  return std::is_same<Rec, Rec8w>::value ? !d.narrow : std::is_same<Rec, Rec16>::value && d.narrow;
}

// 8-byte weighted records: a segment of kNarrowSteps elements is cut there,
// so that its offsets fit 32 bits; the walk goes on as a further ruler with
// an id past all others (the next level's size counts them).  With 1/f rulers
// drawn at random this happens once in e^(4096 / f) segments.
//
// TERM: a ruler whose segment ends at a terminal y becomes a terminal of the
// next level; it records y's original id (y itself at level 0, tid_cur[y]
// deeper) in tid_next, so the terminal of every element can be carried back.
//
// SPAWN (Section 2.2, ruler spawning; exchange chase only): a thread whose
// CTA has no queued ruler left claims an unvisited, unsampled element of its
// CTA's slice of ids as a new ruler (one exchange writes the claim mark and
// the thread's reserved id R + k), and chases from it.  A wave that meets a
// claimed element stops there, its next ruler; a queued head that a spawner
// claimed first becomes a zero-weight link to the spawned ruler.  Ids that
// were reserved but never claimed leave holes, removed after the chase.
//
// ORD (ord.ord != nullptr; a level of a batch, no spawning): the rulers come
// in element order instead, from one global queue over the sequence
// heads (ids r .. r+k-1, in head-list order) then ord[0 .. r) (positions of
// the sampled rulers, ascending), so all CTAs advance one front across the
// instances together; the sampled ruler ord[i] has id i (ord_id of its
// position).  The thread that draws a CTA's next rulers also asks L2 for
// the records of the elements its draw covers, pf_lead elements ahead:
// streamed in order, they are mostly in L2 when the chases reach them.
template <class Rec, bool XCHG, bool TERM, bool SPAWN>
__global__ void __launch_bounds__(512)
k_chase(LevelDesc *__restrict__ desc, int lev, Rec *__restrict__ work, Rec16 *__restrict__ next,
        const uint32_t *__restrict__ ns, uint32_t *__restrict__ qctr, uint32_t *__restrict__ err,
        const uint32_t *__restrict__ tid_cur, uint32_t *__restrict__ tid_next, SpawnArgs sp,
        OrdArgs oa) {
  after_previous(desc);
  const uint32_t *__restrict__ ord = oa.ord;
  __shared__ OrdQueue s_q;
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || wrong_kind<Rec>(d)) return;
  const uint32_t n = d.n, r = d.r;
  const uint64_t R = (uint64_t)r + d.k;
  if (ord && threadIdx.x == 0) {               // the CTA's first window and chunk
    const uint32_t first = 2u * blockDim.x, j = atomicAdd(qctr, first);
    s_q.win = j < R ? ord_window(j, (uint32_t)min((uint64_t)j + first, R)) : 0ull;
    s_q.next = 0ull;
    s_q.out = j >= R;
  }
  __syncthreads();
  Perm P;
  P.init(n, d.seed);
  const uint32_t lo = ord ? 0u : (uint32_t)(R * blockIdx.x / gridDim.x);
  const uint64_t hi = ord ? R : (uint32_t)(R * (blockIdx.x + 1) / gridDim.x);
  uint32_t *q = qctr + blockIdx.x;
  // the next position of this thread's ruler sequence: a ruler id, or (ORD)
  // an index of the ordered sequence
  auto take = [&]() -> uint64_t {
    if (ord) {
      uint32_t fresh = 0xFFFFFFFFu;              // first position of a chunk this thread drew
      uint32_t got;
      do got = ord_take(s_q, qctr, (uint32_t)R, &fresh); while (got == kOrdAgain);
      if (const uint64_t j = fresh; fresh != 0xFFFFFFFFu && oa.pf_lead && j >= d.k) {
        // the CTA took the rulers from j on: bring the records of the
        // elements up to its next draw's first ruler, pf_lead elements ahead,
        // into L2 before the front reaches them
        const uint64_t a = (uint64_t)__ldcg(ord + (j - d.k)) + oa.pf_lead;
        const uint64_t jb = j - d.k + kOrdChunk;
        const uint64_t b = (jb < r ? (uint64_t)__ldcg(ord + jb) : (uint64_t)n) + oa.pf_lead;
        if (a < n && b > a) {
          const uintptr_t pa = ((uintptr_t)(work + a) + 15u) & ~(uintptr_t)15u;
          const uintptr_t pb = (uintptr_t)(work + (b < n ? b : n)) & ~(uintptr_t)15u;
          if (pb > pa && pb - pa <= (1u << 20))
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(pa), "r"((uint32_t)(pb - pa)) : "memory");
        }
      }
      return got;
    }
    return (uint64_t)lo + atomicAdd(q, 1u);
  };
  auto ord_pos = [&](uint64_t j) -> uint32_t {
    return (j >= d.k && j < R) ? __ldcg(ord + (j - d.k)) : 0u;
  };
  const uint32_t ncap = desc[lev + 1].cap;             // records of the next level (debug checks)
  uint32_t visited = 0, bad = 0;
  uint32_t myid = kEnd;                                  // SPAWN: reserved, not yet claimed
  const uint32_t slo = (uint32_t)((uint64_t)n * blockIdx.x / gridDim.x);
  const uint32_t shi = (uint32_t)((uint64_t)n * (blockIdx.x + 1) / gridDim.x);
  uint64_t c64 = take();
  uint32_t xo = ord ? ord_pos(c64) : 0u;                 // ORD: position of c64's ruler, loaded ahead
  for (;;) {
    uint32_t c, rho;
    Rec v;
    if (c64 < hi) {
      const uint64_t cnext = take();
      if (!ord) {
        c = (uint32_t)c64;
        rho = c < r ? P.inv(c) : __ldcg(ns + (c - r));
      } else if (c64 < d.k) {
        c = r + (uint32_t)c64;
        rho = __ldcg(ns + c64);
        xo = ord_pos(cnext);
      } else {
        rho = xo;
        c = (uint32_t)(c64 - d.k);
        xo = ord_pos(cnext);
      }
      c64 = cnext;
      if (dbg_fail(rho < n && c < ncap, err)) continue;
      v = visit<XCHG>(work + rho, c, 0);
      if constexpr (SPAWN) {
        if (rec_is_claim(v)) {                           // a spawner took this head first
          const uint32_t cs = rec_tag(v);
          st_rec(work + rho, cs, 0);                     // it stays the spawned ruler's
          __stcg(reinterpret_cast<uint4 *>(next + c), make_uint4(cs, kUnvisited, 0u, 0u));
          continue;
        }
      }
    } else if constexpr (SPAWN) {
      bool got = false;
      for (;;) {
        if (myid == kEnd) {
          const uint32_t k = atomicAdd(sp.ctr, 1u);
          if (k >= sp.cap) break;                        // out of ids: the wave dies
          myid = (uint32_t)R + k;
        }
        const uint32_t u = slo + atomicAdd(sp.cursor + blockIdx.x, 1u);
        if (u >= shi) break;                             // nothing unvisited left here
        if (P.fwd(u) < r) continue;                      // a sampled ruler: the queue chases it
        if (rec_tag(ld_rec(work + u)) != kUnvisited) continue;
        const Rec old = claim_rec(work + u, myid);
        if (rec_tag(old) != kUnvisited) { st_raw(work + u, old); continue; }   // lost it: put it back
        const uint32_t k = myid - (uint32_t)R;
        atomicOr(sp.used + (k >> 5), 1u << (k & 31u));
        c = myid;
        rho = u;
        v = old;
        myid = kEnd;
        got = true;
        break;
      }
      if (!got) break;
    } else {
      break;
    }
    uint64_t o = rec_weight(v, rho, d.narrow);
    uint32_t steps = 1, nxt = c, cut = kNarrowSteps;
    bad |= rec_tag(v) != kUnvisited;
    uint32_t y = rec_succ(v);
    uint32_t tend = (TERM && y == rho && rec_tag(v) == kUnvisited) ? rho : kEnd;
    if (y != rho && rec_tag(v) == kUnvisited) {
      for (;;) {
        if (y >= n) { bad |= 4u; break; }   // never produced by prep or a chase
        const uint32_t p = P.fwd(y);
        if (p < r) {                 // reached the next ruler
          nxt = ord ? ord_id(oa.bits, oa.cum, y) : p;
          if (dbg_fail(nxt < r, err)) nxt = c;
          if (nxt == c) bad |= 2u;   // came back to itself: a cycle
          break;
        }
        if (std::is_same<Rec, Rec8w>::value && steps == cut) {
          const uint32_t more = atomicAdd(&desc[lev + 1].n, 1u);
          if (more >= ncap) { bad |= 8u; break; }
          __stcg(reinterpret_cast<uint4 *>(next + c),
                 make_uint4(more, kUnvisited, (uint32_t)o, (uint32_t)(o >> 32)));
          nxt = c = more;
          o = 0;
          cut = steps + kNarrowSteps;
        }
        v = visit<XCHG>(work + y, c, o);
        if constexpr (SPAWN) {
          if (rec_is_claim(v)) {     // reached a spawned ruler
            const uint32_t cs = rec_tag(v);
            st_rec(work + y, cs, 0);
            nxt = cs;
            if (cs == c) bad |= 2u;  // its own: a cycle
            break;
          }
        }
        ++steps;
        if (rec_tag(v) != kUnvisited) { bad |= 1u; break; }   // second predecessor
        o += rec_weight(v, y, d.narrow);
        const uint32_t s = rec_succ(v);
        if (s == y) {                // terminal: the reduced element is terminal too
          if constexpr (TERM) tend = y;
          break;
        }
        if (steps > n) { bad |= 2u; break; }
        y = s;
      }
    }
    __stcg(reinterpret_cast<uint4 *>(next + c),
           make_uint4(nxt, kUnvisited, (uint32_t)o, (uint32_t)(o >> 32)));
    if constexpr (TERM) {
      if (tend != kEnd) tid_next[c] = tid_cur ? __ldcg(tid_cur + tend) : tend;
    }
    visited += steps;
  }
  if (bad & 1u) record_error(err, kErrNotList);
  if (bad & 2u) record_error(err, kErrCycle);
  if (bad & 4u) record_error(err, kErrInternal);
  if (bad & 8u) record_error(err, kErrCapacity);
  for (int dd = 16; dd > 0; dd >>= 1) visited += __shfl_down_sync(0xFFFFFFFFu, visited, dd);
  if ((threadIdx.x & 31) == 0 && visited) atomicAdd(&desc[lev].visited, visited);
}

cudaError_t launch_chase(LevelDesc *desc, int lev, void *work, int kind, void *next_work,
                         const uint32_t *ns, uint32_t *qctr, int grid, int block, uint32_t *err,
                         int xchg, const uint32_t *tid_cur, uint32_t *tid_next, const SpawnArgs *spawn,
                         const OrdArgs *ord, cudaStream_t s) {
  if (ord && spawn) return cudaErrorInvalidValue;   // spawning needs the per-CTA slices
  Rec16 *nx = reinterpret_cast<Rec16 *>(next_work);
  SpawnArgs sp;
  memset(&sp, 0, sizeof(sp));
  if (spawn) sp = *spawn;
  OrdArgs oa;
  memset(&oa, 0, sizeof(oa));
  if (ord) oa = *ord;
#define LR_CHASE(REC, X, T, SP) \
  launch_after(k_chase<REC, X, T, SP>, grid, block, s, desc, lev, reinterpret_cast<REC *>(work), nx, ns, qctr, err, \
                                                tid_cur, tid_next, sp, oa)
  const bool rec16 = kind == kRecKind16;
  if (kind == kRecKind8w) {
    if (spawn || tid_next || !xchg) return cudaErrorInvalidValue;
    LR_CHASE(Rec8w, true, false, false);
  } else if (spawn) {
    if (rec16) LR_CHASE(Rec16, true, false, true);
    else LR_CHASE(Rec8, true, false, true);
  } else if (tid_next) {
    if (rec16) { if (xchg) LR_CHASE(Rec16, true, true, false); else LR_CHASE(Rec16, false, true, false); }
    else { if (xchg) LR_CHASE(Rec8, true, true, false); else LR_CHASE(Rec8, false, true, false); }
  } else {
    if (rec16) { if (xchg) LR_CHASE(Rec16, true, false, false); else LR_CHASE(Rec16, false, false, false); }
    else { if (xchg) LR_CHASE(Rec8, true, false, false); else LR_CHASE(Rec8, false, false, false); }
  }
#undef LR_CHASE
  count_launch();
  return cudaGetLastError();
}

int chase_occupancy(bool rec16, int block) {
  static CachedInt cache[2][3];                // per record size and block (128, 256, 512)
  return cached_per_device(cache[rec16][block == 128 ? 0 : block == 256 ? 1 : 2], [](int, int arg) {
    int nb = 0;
    if (arg < 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_chase<Rec16, false, false, false>, -arg, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_chase<Rec8, false, false, false>, arg, 0);
    return nb;
  }, rec16 ? -block : block);
}

// ---------------------------------------------------------------- finalize
template <class RT>
__device__ __forceinline__ RT propagate(uint32_t c, uint64_t o, uint32_t nn, const RT *rnext,
                                        uint32_t &bad) {
  RT base = 0;
  if (c < nn) base = __ldcg(rnext + c);
  else if (c != kZeroCid) bad |= c == kUnvisited ? kErrCycle : kErrInternal;
  return (RT)(base - (RT)o);
}

// Terminal of element i at this level: its ruler's, or its own original id
// for a resolved singleton (a head that is its own terminal).
__device__ __forceinline__ uint32_t propagate_term(uint32_t c, uint32_t i, uint32_t nn,
                                                   const uint32_t *tnext, const uint32_t *tid_cur) {
  if (c < nn) return __ldcg(tnext + c);
  if (c == kZeroCid) return tid_cur ? __ldcg(tid_cur + i) : i;
  return kEnd;
}

// A record's last read (evict-first: the lines it frees in L2 serve the
// gathers of the next level's ranks).
template <class Rec>
__device__ __forceinline__ Rec ld_rec_last(const Rec *p) {
  Rec r;
  if constexpr (sizeof(Rec) == 8) {
    const uint2 a = __ldcs(reinterpret_cast<const uint2 *>(p));
    r.lo = a.x;
    r.hi = a.y;
  } else {
    const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(p));
    r.succ = a.x;
    r.tag = a.y;
    r.w = ((uint64_t)a.w << 32) | a.z;
  }
  return r;
}

// Ruler propagation: every element gets its ruler's rank minus its offset
// (TERM: and its ruler's terminal).
template <class Rec, class RT, bool TERM>
__global__ void __launch_bounds__(256)
k_finalize(const LevelDesc *__restrict__ desc, int lev, const Rec *__restrict__ work,
           const RT *__restrict__ rnext, RT *__restrict__ rout, uint32_t *__restrict__ err,
           const uint32_t *__restrict__ tnext, uint32_t *__restrict__ tout,
           const uint32_t *__restrict__ tid_cur) {
  after_previous(desc);
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || wrong_kind<Rec>(d)) return;
  const uint32_t n = d.n, nn = d.nraw ? d.nraw : desc[lev + 1].n;
  uint32_t bad = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) bad |= level_errors(d, desc[lev + 1], err);
  // each warp takes 128 consecutive elements at a time and lane l the
  // elements base + l + 32 j: every record load and rank store of the warp
  // is one contiguous run, and a lane's four gathers are in flight together
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t step = ((uint64_t)gridDim.x * blockDim.x >> 5) * 128u;
  for (uint64_t base = warp * 128u; base < n; base += step) {
    Rec v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint64_t i = base + lane + 32u * j;
      if (i < n) v[j] = ld_rec_last(work + i);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint64_t i = base + lane + 32u * j;
      if (i < n) {
        const RT r = propagate<RT>(done_cid(v[j]), done_off(v[j], d.narrow), nn, rnext, bad);
        if constexpr (TERM) __stcs(tout + i, propagate_term(done_cid(v[j]), (uint32_t)i, nn, tnext, tid_cur));
        __stcs(rout + i, r);
      }
    }
  }
  if (bad) record_error(err, bad);
}

// Level-0 propagation into per-instance output buffers.
template <class Rec, class RT>
__global__ void __launch_bounds__(256)
k_finalize_ptrs(const LevelDesc *__restrict__ desc, const Rec *__restrict__ work,
                const RT *__restrict__ rnext, RT *const *__restrict__ rptr,
                const int64_t *__restrict__ offsets, int32_t k, uint32_t *__restrict__ err) {
  after_previous(desc);
  const LevelDesc d = desc[0];
  if (d.mode != kModeSrs || wrong_kind<Rec>(d)) return;
  const uint32_t n = d.n, nn = desc[1].n;
  uint32_t bad = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) bad |= level_errors(d, desc[1], err);
  // each warp takes 128 consecutive elements (lane l: l + 32 j, coalesced
  // record loads and rank stores); the four records, then the four gathers
  // of the next level's ranks are in flight together, and the instances are
  // found meanwhile (the warp's first by a warp-wide search, the others by
  // walking forward from it).  Element ids and offsets fit 32 bits here.
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t step = ((uint64_t)gridDim.x * blockDim.x >> 5) * 128u;
  for (uint64_t b64 = warp * 128u; b64 < n; b64 += step) {
    const uint32_t base = (uint32_t)b64, rem = n - base;
    Rec v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t t = lane + 32u * j;
      if (t < rem) v[j] = ld_rec_last(work + base + t);
    }
    RT val[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (lane + 32u * j < rem) val[j] = propagate<RT>(done_cid(v[j]), done_off(v[j], d.narrow), nn, rnext, bad);
    }
    int32_t lo = warp_instance(offsets, k, base, lane);
    uint32_t ib = (uint32_t)__ldg(offsets + lo), ie = (uint32_t)__ldg(offsets + lo + 1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t t = lane + 32u * j;
      if (t < rem) {
        const uint32_t i = base + t;
        while (i >= ie && lo + 1 < k) { ++lo; ib = ie; ie = (uint32_t)__ldg(offsets + lo + 1); }
        __stcs(rptr[lo] + (i - ib), val[j]);
      }
    }
  }
  if (bad) record_error(err, bad);
}

cudaError_t launch_finalize_ptrs(LevelDesc *desc, const void *work, int kind, const void *rnext,
                                 void *const *rptr, int rank_bytes, uint32_t cap,
                                 const int64_t *offsets, int32_t k, uint32_t *err, cudaStream_t s) {
  const int block = 256;
#define LR_FINP(REC, RT)                                                                          \
  launch_after(k_finalize_ptrs<REC, RT>, fit_grid<k_finalize_ptrs<REC, RT>>(((uint64_t)cap + 3) / 4, block),  \
                             block, s, desc, reinterpret_cast<const REC *>(work),            \
                                            reinterpret_cast<const RT *>(rnext),                  \
                                            reinterpret_cast<RT *const *>(rptr), offsets, k, err)
  if (kind == kRecKind8w) { if (rank_bytes == 4) LR_FINP(Rec8w, uint32_t); else LR_FINP(Rec8w, unsigned long long); }
  else if (kind == kRecKind16) { if (rank_bytes == 4) LR_FINP(Rec16, uint32_t); else LR_FINP(Rec16, unsigned long long); }
  else { if (rank_bytes == 4) LR_FINP(Rec8, uint32_t); else LR_FINP(Rec8, unsigned long long); }
#undef LR_FINP
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_finalize(LevelDesc *desc, int lev, const void *work, int kind,
                            const void *rnext, void *rout, int rank_bytes, uint32_t cap,
                            uint32_t *err, const uint32_t *tnext, uint32_t *tout,
                            const uint32_t *tid_cur, cudaStream_t s, bool to_host) {
  const int block = 256;
#define LR_FIN(REC, RT, T)                                                                      \
  launch_after(k_finalize<REC, RT, T>, host_grid(fit_grid<k_finalize<REC, RT, T>>(((uint64_t)cap + 3) / 4, block), to_host), \
                           block, s, desc, lev, reinterpret_cast<const REC *>(work),       \
                                          reinterpret_cast<const RT *>(rnext),                  \
                                          reinterpret_cast<RT *>(rout), err, tnext, tout, tid_cur)
  const bool rec16 = kind == kRecKind16;
  if (kind == kRecKind8w) {
    if (tout) return cudaErrorInvalidValue;
    if (rank_bytes == 4) LR_FIN(Rec8w, uint32_t, false); else LR_FIN(Rec8w, unsigned long long, false);
  } else if (tout) {
    if (rec16) { if (rank_bytes == 4) LR_FIN(Rec16, uint32_t, true); else LR_FIN(Rec16, unsigned long long, true); }
    else { if (rank_bytes == 4) LR_FIN(Rec8, uint32_t, true); else LR_FIN(Rec8, unsigned long long, true); }
  } else {
    if (rec16) { if (rank_bytes == 4) LR_FIN(Rec16, uint32_t, false); else LR_FIN(Rec16, unsigned long long, false); }
    else { if (rank_bytes == 4) LR_FIN(Rec8, uint32_t, false); else LR_FIN(Rec8, unsigned long long, false); }
  }
#undef LR_FIN
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------- spawning: compaction
// Spawned ruler ids R + k that were handed out but never claimed leave holes.
// The next level is compacted: id c keeps c below R, and a claimed spawned
// id R + k becomes R + (claimed spawned ids before it).  The ranks are
// scattered back to the original ids before this level's propagation.
__device__ __forceinline__ uint32_t spawn_map(uint32_t c, uint32_t R, const uint32_t *used,
                                              const uint32_t *upre) {
  if (c < R) return c;
  const uint32_t k = c - R;
  return R + __ldg(upre + (k >> 5)) + (uint32_t)__popc(__ldcg(used + (k >> 5)) & ((1u << (k & 31u)) - 1u));
}

// Prefix of the claimed-id bitmap (one CTA) and the next level's size and mode.
__global__ void __launch_bounds__(1024)
k_spawn_scan(LevelDesc *desc, int lev, int nlev, const uint32_t *__restrict__ ctr, uint32_t cap,
             const uint32_t *__restrict__ used, uint32_t *__restrict__ upre, uint32_t cutoff,
             uint32_t *__restrict__ err) {
  __shared__ uint64_t sm[33];
  LevelDesc &d = desc[lev];
  if (d.mode != kModeSrs) return;
  const uint32_t handed = min(*ctr, cap);
  const uint32_t words = (handed + 31) / 32;
  const uint32_t per = (words + blockDim.x - 1) / blockDim.x;
  const uint32_t a = threadIdx.x * per, b = min(words, a + per);
  uint64_t s = 0;
  for (uint32_t w = a; w < b; ++w) s += __popc(used[w]);
  uint64_t total;
  uint64_t run = block_exclusive_scan(s, sm, &total);
  for (uint32_t w = a; w < b; ++w) { upre[w] = (uint32_t)run; run += __popc(used[w]); }
  if (threadIdx.x == 0) {
    LevelDesc &e = desc[lev + 1];
    const uint64_t R = (uint64_t)d.r + d.k;
    const uint64_t n1 = R + total;
    d.nraw = (uint32_t)(R + handed);
    if (n1 > e.cap) { record_error(err, kErrCapacity); d.mode = kModeOff; return; }
    e.n = (uint32_t)n1;
    e.r = (uint32_t)((n1 + e.f_inv - 1) / e.f_inv);
    e.mode = n1 <= cutoff || lev + 1 >= nlev - 1 ? kModeBase : kModeSrs;
  }
}

// The next level's records at compacted ids, successors remapped.
__global__ void k_spawn_compact(const LevelDesc *__restrict__ desc, int lev, const Rec16 *__restrict__ raw,
                                Rec16 *__restrict__ out, const uint32_t *__restrict__ used,
                                const uint32_t *__restrict__ upre) {
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || d.nraw == 0) return;
  const uint32_t R = d.r + d.k;
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < d.nraw; c += gridDim.x * blockDim.x) {
    if (c >= R && !((__ldcg(used + ((c - R) >> 5)) >> ((c - R) & 31u)) & 1u)) continue;   // a hole
    const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(raw + c));
    const uint32_t s = v.x < d.nraw ? spawn_map(v.x, R, used, upre) : v.x;
    __stcg(reinterpret_cast<uint4 *>(out + spawn_map(c, R, used, upre)), make_uint4(s, v.y, v.z, v.w));
  }
}

// Ranks of the compacted next level back at the original ids.
template <class RT>
__global__ void k_spawn_scatter(const LevelDesc *__restrict__ desc, int lev, const RT *__restrict__ rc,
                                RT *__restrict__ rraw, const uint32_t *__restrict__ used,
                                const uint32_t *__restrict__ upre) {
  const LevelDesc d = desc[lev];
  if (d.mode != kModeSrs || d.nraw == 0) return;
  const uint32_t R = d.r + d.k;
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < d.nraw; c += gridDim.x * blockDim.x) {
    if (c >= R && !((__ldcg(used + ((c - R) >> 5)) >> ((c - R) & 31u)) & 1u)) continue;
    rraw[c] = __ldcg(rc + spawn_map(c, R, used, upre));
  }
}

cudaError_t launch_spawn_compact(LevelDesc *desc, int lev, int nlev, const uint32_t *ctr, uint32_t cap,
                                 const uint32_t *used, uint32_t *upre, const void *raw, void *out,
                                 uint32_t raw_cap, uint32_t cutoff, uint32_t *err, cudaStream_t s) {
  k_spawn_scan<<<1, 1024, 0, s>>>(desc, lev, nlev, ctr, cap, used, upre, cutoff, err);
  k_spawn_compact<<<stream_grid(raw_cap, 256), 256, 0, s>>>(desc, lev, reinterpret_cast<const Rec16 *>(raw),
                                                           reinterpret_cast<Rec16 *>(out), used, upre);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_spawn_scatter(LevelDesc *desc, int lev, const void *rc, void *rraw, int rank_bytes,
                                 const uint32_t *used, const uint32_t *upre, uint32_t raw_cap,
                                 cudaStream_t s) {
  const int grid = stream_grid(raw_cap, 256);
  if (rank_bytes == 4)
    k_spawn_scatter<uint32_t><<<grid, 256, 0, s>>>(desc, lev, reinterpret_cast<const uint32_t *>(rc),
                                                   reinterpret_cast<uint32_t *>(rraw), used, upre);
  else
    k_spawn_scatter<unsigned long long><<<grid, 256, 0, s>>>(
        desc, lev, reinterpret_cast<const unsigned long long *>(rc),
        reinterpret_cast<unsigned long long *>(rraw), used, upre);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------- extra outputs (level 0)
// The paper's output also names each element's terminal (Section 1.1) and
// its in-place form counts the terminal's own weight; the head-relative
// (prefix) rank is the list's total minus the rank.  term[] holds global
// terminal ids when these passes run.
//
// Head pass: the total of each list (the rank of its head) is stored at its
// terminal's entry of prefix.
template <class RT>
__global__ void __launch_bounds__(kHeadThreads)
k_out_heads(const LevelDesc *__restrict__ desc, const uint32_t *__restrict__ bitmap,
            const uint32_t *__restrict__ hlist, const uint32_t *__restrict__ term,
            const RT *__restrict__ rank, RT *__restrict__ prefix) {
  const LevelDesc d = desc[0];
  for_each_head(d, bitmap, hlist, [&](uint32_t h) {
    const uint32_t t = __ldcg(term + h);
    if (t < d.n) prefix[t] = __ldcg(rank + h);
  });
}

// Streaming pass: prefix[i] = total - rank[i] (a terminal's entry holds the
// total and keeps it, its rank being 0, so the pass may run in place); the
// inclusive form adds the terminal's weight (weighted input only: unweighted,
// the terminal weighs 0, Section 1.1); in the batched form terminal ids
// become local to their instance.
template <class RT>
__global__ void __launch_bounds__(256)
k_out_fix(uint32_t n, uint32_t *__restrict__ term, RT *__restrict__ rank, RT *__restrict__ prefix,
          int incl, const void *__restrict__ weight, int wtype, const int64_t *__restrict__ offsets,
          int32_t k, int local) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t t = term[i];
    if (t >= n) continue;                       // an error the device already recorded
    const RT r = rank[i];
    if (prefix) prefix[i] = (RT)(__ldcg(prefix + t) - r);
    if (incl) {
      uint64_t wt = 0u;
      if (wtype == 1) wt = (uint64_t)(int64_t)__ldg(reinterpret_cast<const int *>(weight) + t);
      else if (wtype == 2) wt = (uint64_t)__ldg(reinterpret_cast<const long long *>(weight) + t);
      rank[i] = (RT)(r + (RT)wt);
    }
    if (local) {
      int32_t lo = 0, hi = k;
      while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if ((uint64_t)__ldg(offsets + mid) <= i) lo = mid; else hi = mid;
      }
      term[i] = (uint32_t)(t - (uint64_t)__ldg(offsets + lo));
    }
  }
}

// The same for one list, whose terminal and total are two numbers: a single
// streaming pass over the plain ranks, with no terminal ids in the records,
// the levels or a gather per element (2^22 elements with int32 weights,
// terminals and prefix ranks: 85 us of propagation and output passes -> 45).
// total: the rank of the head, a ruler, at the level below.
template <class RT>
__global__ void __launch_bounds__(256)
k_out_one(uint32_t n, uint32_t t, const RT *__restrict__ total, uint32_t *__restrict__ term, RT *__restrict__ rank,
          RT *__restrict__ prefix, int incl, const void *__restrict__ weight, int wtype) {
  after_previous(total, rank, weight);
  const RT all = __ldg(total);
  RT wt = 0;
  if (incl && wtype == 1) wt = (RT)(long long)__ldg(reinterpret_cast<const int *>(weight) + t);
  if (incl && wtype == 2) wt = (RT)__ldg(reinterpret_cast<const long long *>(weight) + t);
  constexpr int kPer = 4;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += stride * kPer) {
    RT r[kPer];
    if (prefix || incl) {
#pragma unroll
      for (int e = 0; e < kPer; ++e)
        if (i0 + stride * e < n) r[e] = rank[i0 + stride * e];
    }
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const uint64_t i = i0 + stride * e;
      if (i >= n) break;
      if (prefix) __stcs(prefix + i, (RT)(all - r[e]));
      if (incl) __stcs(rank + i, (RT)(r[e] + wt));
      if (term) __stcs(term + i, t);
    }
  }
}

cudaError_t launch_out_one(uint32_t n, uint32_t t, const void *total, uint32_t *term, void *rank, void *prefix,
                           int rank_bytes, int incl, const void *weight, int wtype, cudaStream_t s) {
  if (wtype == 0) incl = 0;                     // an unweighted terminal weighs 0
  if (!term && !prefix && !incl) return cudaSuccess;
  const int grid = stream_grid(((uint64_t)n + 3) / 4, 256);
  if (rank_bytes == 4)
    launch_after(k_out_one<uint32_t>, grid, 256, s, n, t, reinterpret_cast<const uint32_t *>(total), term,
                                             reinterpret_cast<uint32_t *>(rank), reinterpret_cast<uint32_t *>(prefix),
                                             incl, weight, wtype);
  else
    launch_after(k_out_one<unsigned long long>, grid, 256, s, 
        n, t, reinterpret_cast<const unsigned long long *>(total), term, reinterpret_cast<unsigned long long *>(rank),
        reinterpret_cast<unsigned long long *>(prefix), incl, weight, wtype);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_outputs(const LevelDesc *desc, const uint32_t *bitmap, const uint32_t *hlist0,
                           uint32_t n, uint32_t *term, void *rank, void *prefix, int rank_bytes,
                           int incl, const void *weight, int wtype, const int64_t *offsets, int32_t k,
                           int local, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (wtype == 0) incl = 0;                     // an unweighted terminal weighs 0
  const int grid = stream_grid(n, 256);
  int launches = 0;
  if (rank_bytes == 4) {
    uint32_t *r = reinterpret_cast<uint32_t *>(rank), *p = reinterpret_cast<uint32_t *>(prefix);
    if (p) { k_out_heads<uint32_t><<<kHeadBlocks, kHeadThreads, 0, s>>>(desc, bitmap, hlist0, term, r, p); ++launches; }
    if (p || incl || local) { k_out_fix<uint32_t><<<grid, 256, 0, s>>>(n, term, r, p, incl, weight, wtype, offsets, k, local); ++launches; }
  } else {
    unsigned long long *r = reinterpret_cast<unsigned long long *>(rank);
    unsigned long long *p = reinterpret_cast<unsigned long long *>(prefix);
    if (p) { k_out_heads<unsigned long long><<<kHeadBlocks, kHeadThreads, 0, s>>>(desc, bitmap, hlist0, term, r, p); ++launches; }
    if (p || incl || local) { k_out_fix<unsigned long long><<<grid, 256, 0, s>>>(n, term, r, p, incl, weight, wtype, offsets, k, local); ++launches; }
  }
  count_launch(launches);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- base case
// Ranks a whole level by pointer jumping over the level's own records, in one
// launch and without barriers.  A record is the state of its element j:
//   untouched  {succ, kUnvisited, w}     as the prep or the chase wrote it
//              (succ == j marks a terminal, which weighs w);
//   moved      {nxt, links, sum}         nxt lies `links` links further on and
//              sum adds up the weights on the way;
//   settled    {kEnd, terminal, rank}.
// Each thread owns up to kJumpElems elements, holds their state in registers
// and repeats: read the record of nxt, append it, publish the result.  Every
// state of a record is a true statement about the list, and one access reads
// or writes a whole record (8 or 16 bytes), so it does not matter how far the
// others have come: where all advance together the pointers double, as in
// rounds with a barrier after each, and where they have not run yet the walk
// is slower but right.  Nobody waits for anybody.  An element appends at
// least one link each time, so one that has gathered more links than the
// level has elements is on a cycle (its links double too: some log2 n steps);
// 8-byte records carry no count and need none, their sum being the count.
//
// Warps take chunks of 32 consecutive elements in a random order.  In element
// order, a list that follows memory would have the first threads walk link by
// link through everything that does not run yet: 51 ms for 700 thousand
// elements in locality order, where the grid holds 623 thousand at once (and
// the same could happen when other kernels keep part of this grid waiting).
//
// What bounds it: the latency of log2 n dependent L2 reads below some 2^17
// elements, the L2's rate of random reads above (n log2 n of them; the
// stores are warp-contiguous).
constexpr int kJumpThreads = 256;
constexpr int kJumpElems = 4;
constexpr int kJumpCtasPerSm = 4;

template <class Rec>
struct JumpState;

template <>
struct JumpState<Rec8> {
  uint32_t nxt, sum;
  __device__ __forceinline__ void load(const Rec8 *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    nxt = (uint32_t)v;
    sum = (uint32_t)(v >> 32);
  }
  __device__ __forceinline__ void store(Rec8 *p) const {
    const unsigned long long v = ((unsigned long long)sum << 32) | nxt;
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
  }
  // own record: false when the element is a terminal (then settled)
  __device__ __forceinline__ bool open(uint32_t self) {
    sum = nxt == self ? 0u : 1u;
    return nxt != self;
  }
  // append record q, read at a = nxt; true once the end of the list is reached
  __device__ __forceinline__ bool append(const JumpState &q, uint32_t a, uint32_t n, uint32_t &bad) {
    if (q.nxt == kEnd) { sum += q.sum; return true; }
    if (q.nxt == a) return true;
    sum += q.sum == kUnvisited ? 1u : q.sum;
    nxt = q.nxt;
    if (sum > n) { bad |= kErrCycle; return true; }
    return false;
  }
  __device__ __forceinline__ void settle() { nxt = kEnd; }
  __device__ __forceinline__ uint64_t rank() const { return sum; }
  __device__ __forceinline__ uint32_t term() const { return kEnd; }
};

template <>
struct JumpState<Rec16> {
  uint32_t nxt, links;
  uint64_t sum;
  __device__ __forceinline__ void load(const Rec16 *p) {
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 d;\n\tld.relaxed.gpu.global.b128 d, [%2];\n\tmov.b128 {%0, %1}, d;\n\t}"
                 : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    nxt = (uint32_t)lo;
    links = (uint32_t)(lo >> 32);
    sum = hi;
  }
  __device__ __forceinline__ void store(Rec16 *p) const {
    const unsigned long long lo = ((unsigned long long)links << 32) | nxt, hi = sum;
    asm volatile("{\n\t.reg .b128 d;\n\tmov.b128 d, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], d;\n\t}"
                 :: "l"(p), "l"(lo), "l"(hi) : "memory");
  }
  __device__ __forceinline__ bool open(uint32_t self) {
    const bool inner = nxt != self;
    links = inner ? 1u : self;                 // settled: the terminal
    return inner;
  }
  __device__ __forceinline__ bool append(const JumpState &q, uint32_t a, uint32_t n, uint32_t &bad) {
    sum += q.sum;
    if (q.nxt == kEnd) { links = q.links; return true; }
    if (q.nxt == a) { links = a; return true; }
    const uint64_t l = (uint64_t)links + (q.links == kUnvisited ? 1u : q.links);
    nxt = q.nxt;
    links = (uint32_t)l;
    if (l > n) { bad |= kErrCycle; links = kEnd; return true; }
    return false;
  }
  __device__ __forceinline__ void settle() { nxt = kEnd; }
  __device__ __forceinline__ uint64_t rank() const { return sum; }
  __device__ __forceinline__ uint32_t term() const { return links; }
};

// A level below the first holds every element once among the successors of
// its non-terminals and its heads, or some element has two predecessors.
// Both sides are compared as sums of this hash (check in LevelDesc,
// examined by the propagation that reads the level's ranks).
__device__ __forceinline__ uint64_t jump_hash(uint32_t x, uint64_t seed) {
  return splitmix64(seed ^ ((uint64_t)x * 0xD1342543DE82EF95ull));
}

// Level 0 (JumpInput): heads are not needed; with a bound on the lists, they
// are counted from the has-predecessor bitmap, as many as the ruling set would
// have to provide for.  PTRS: ranks go to one buffer per instance.
template <class Rec, class RT, bool TERM, bool PTRS>
__global__ void __launch_bounds__(kJumpThreads, kJumpCtasPerSm)
k_jump(LevelDesc *__restrict__ desc, int lev, Rec *work, RT *__restrict__ rout, uint32_t *__restrict__ err,
       const uint32_t *__restrict__ heads, const uint32_t *__restrict__ tid, uint32_t *__restrict__ tout,
       JumpInput in) {
  after_previous(desc);
  const LevelDesc d = desc[lev];
  if (d.mode != kModeBase) return;
  const uint32_t n = d.n;
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t bad = 0, lists = 0;
  uint64_t chk = 0;
  if (heads)
    for (uint64_t e = t; e < d.h; e += stride) chk += jump_hash(__ldcg(heads + e), d.seed);
  const uint32_t chunks = (uint32_t)(((uint64_t)n + 31u) / 32u), warps = (uint32_t)(stride >> 5);
  Perm P;
  P.init(chunks, d.seed);
  for (uint64_t c0 = t >> 5; c0 < chunks; c0 += (uint64_t)warps * kJumpElems) {   // uniform in the warp
    JumpState<Rec> x[kJumpElems];
    uint32_t idx[kJumpElems];                  // this lane's element of each chunk, or kEnd
    uint32_t pend = 0;                         // bit e: element e is not settled yet
#pragma unroll
    for (int e = 0; e < kJumpElems; ++e) {
      const uint64_t c = c0 + (uint64_t)warps * e;
      const uint64_t i = c < chunks ? (uint64_t)P.fwd((uint32_t)c) * 32u + lane : n;
      idx[e] = i < n ? (uint32_t)i : kEnd;
      if (i < n) x[e].load(work + i);
    }
#pragma unroll
    for (int e = 0; e < kJumpElems; ++e) {
      const uint32_t i = idx[e];
      if (i == kEnd) continue;
      const uint32_t s = x[e].nxt;
      if (x[e].open(i)) {
        if (s < n) pend |= 1u << e;
        else bad |= kErrInternal;              // never written by a prep or a chase
        if (heads) chk += jump_hash(s, d.seed);
        if (in.max_lists) lists += !((__ldcg(in.bitmap + (i >> 5)) >> (i & 31u)) & 1u);
      } else if (in.max_lists && !((__ldcg(in.bitmap + (i >> 5)) >> (i & 31u)) & 1u)) {
        Perm Q;                                // a list of one: the ruling set takes it for a
        Q.init(n, d.seed);                     // list if it is a sampled ruler
        lists += Q.fwd(i) < d.r;
      }
      if (heads) chk -= jump_hash(i, d.seed);
    }
    if (in.clear) {                            // this warp was its chunks' marks' last reader
      __syncwarp();
#pragma unroll
      for (int e = 0; e < kJumpElems; ++e) {
        const uint32_t first = __shfl_sync(0xFFFFFFFFu, idx[e], 0);
        if (lane == 0 && first != kEnd) in.clear[first >> 5] = 0u;
      }
    }
    while (pend) {
      JumpState<Rec> q[kJumpElems];
#pragma unroll
      for (int e = 0; e < kJumpElems; ++e)
        if (pend >> e & 1u) q[e].load(work + x[e].nxt);
#pragma unroll
      for (int e = 0; e < kJumpElems; ++e) {
        if (!(pend >> e & 1u)) continue;
        const uint32_t self = idx[e];
        bool done = x[e].append(q[e], x[e].nxt, n, bad);
        if (!done && x[e].nxt >= n) { bad |= kErrInternal; done = true; }
        // back at itself: a cycle (published, it would read as a terminal)
        if (!done && x[e].nxt == self) { bad |= kErrCycle; done = true; }
        if (done) {
          x[e].settle();
          pend &= ~(1u << e);
        }
        x[e].store(work + self);
      }
    }
    if constexpr (PTRS) {
#pragma unroll
      for (int e = 0; e < kJumpElems; ++e) {
        const uint32_t i = idx[e];
        const uint32_t first = __shfl_sync(0xFFFFFFFFu, i, 0);
        if (first == kEnd) continue;           // no such chunk (uniform in the warp)
        int32_t lo = warp_instance(in.offsets, in.k, first, lane);
        uint64_t ib = (uint64_t)__ldg(in.offsets + lo), ie = (uint64_t)__ldg(in.offsets + lo + 1);
        if (i != kEnd) {
          while (i >= ie && lo + 1 < in.k) { ++lo; ib = ie; ie = (uint64_t)__ldg(in.offsets + lo + 1); }
          reinterpret_cast<RT *>(in.rptr[lo])[i - ib] = (RT)x[e].rank();
        }
      }
    } else {
#pragma unroll
      for (int e = 0; e < kJumpElems; ++e) {
        const uint32_t i = idx[e];
        if (i == kEnd) continue;
        rout[i] = (RT)x[e].rank();
        if constexpr (TERM) {
          const uint32_t z = x[e].term();
          tout[i] = z >= n ? kEnd : (tid ? __ldcg(tid + z) : z);
        }
      }
    }
  }
  if (in.max_lists) {
    lists = __reduce_add_sync(0xFFFFFFFFu, lists);
    if (lane == 0 && lists && (uint64_t)atomicAdd(in.count, lists) + lists > in.max_lists) bad |= kErrCapacity;
  }
  if (bad) record_error(err, bad);
  if (heads) {
    for (int dd = 16; dd > 0; dd >>= 1) chk += __shfl_down_sync(0xFFFFFFFFu, chk, dd);
    if (lane == 0 && chk) atomicAdd(&desc[lev].check, (unsigned long long)chk);
  }
  if (t == 0) desc[lev].visited = n;
  if (in.ticket) {
    // the last CTA reports the call's error bits and leaves the words at zero
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(in.ticket, 1u) == gridDim.x - 1u) {
        __threadfence();
        *in.status = atomicExch(err, 0u);
        *in.count = 0u;
        *in.ticket = 0u;
      }
    }
  }
}

cudaError_t launch_jump(LevelDesc *desc, int lev, void *work, bool rec16, void *rout, int rank_bytes,
                        uint32_t cap, uint32_t *err, const uint32_t *heads, const uint32_t *tid,
                        uint32_t *tout, const JumpInput *input, cudaStream_t s) {
  JumpInput in;
  memset(&in, 0, sizeof(in));
  if (input) in = *input;
  const uint64_t ctas = ((uint64_t)cap + kJumpThreads - 1) / kJumpThreads;
  const uint64_t full = (uint64_t)device_sm_count() * kJumpCtasPerSm;
  const int grid = (int)std::max<uint64_t>(1, std::min(ctas, full));
#define LR_JUMP(REC, T, P)                                                                             \
  do {                                                                                                 \
    if (rank_bytes == 4)                                                                               \
      launch_after(k_jump<REC, uint32_t, T, P>, grid, kJumpThreads, s,                                        \
          desc, lev, reinterpret_cast<REC *>(work), reinterpret_cast<uint32_t *>(rout), err, heads, tid, tout, in); \
    else                                                                                               \
      launch_after(k_jump<REC, unsigned long long, T, P>, grid, kJumpThreads, s,                              \
          desc, lev, reinterpret_cast<REC *>(work), reinterpret_cast<unsigned long long *>(rout), err, heads, tid, \
          tout, in);                                                                                   \
  } while (0)
  if (tout) {
    if (!rec16) return cudaErrorInvalidValue;   // an 8-byte record has no room for the terminal
    LR_JUMP(Rec16, true, false);
  } else if (in.rptr) {
    if (rec16) LR_JUMP(Rec16, false, true); else LR_JUMP(Rec8, false, true);
  } else {
    if (rec16) LR_JUMP(Rec16, false, false); else LR_JUMP(Rec8, false, false);
  }
#undef LR_JUMP
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------- small lists
// A single list or forest of at most kSmallMax elements, whole call in one
// launch: one CTA reads the successors, doubles pointers in shared memory and
// writes the ranks, and the status straight to the host's status word.  At
// these sizes a call is all latency: as a clear, a packing pass, k_jump and a
// status copy it took 54 us at n = 1000, of which the kernels were 16.
//
// One 32-bit word holds an element's pointer and the links up to it,
// links << 16 | settled | pointer; the settled bit is set once the pointer is
// a terminal and travels with it.  A round adds the word (weighted: and the
// sum) of the element pointed to, from one buffer into the other; a list
// settles in log2 n rounds, a cycle never does.
constexpr uint32_t kSmallMax = 4096;
constexpr int kSmallThreads = 1024;
constexpr int kSmallElems = (int)kSmallMax / kSmallThreads;
constexpr uint32_t kSmallSettled = 0x8000u, kSmallPtr = kSmallMax - 1u;
constexpr int kSmallRounds = 13;               // links double each round: 2^13 fits their 16 bits

template <int WT, class RT>
__global__ void __launch_bounds__(kSmallThreads)
k_small(const uint32_t *__restrict__ succ, const void *__restrict__ weight, uint32_t n, RT *__restrict__ rank,
        int validate, LevelDesc *__restrict__ desc, InitParams ip, uint32_t *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  __shared__ uint32_t s_bad, s_pred[kSmallMax / 32];
  init_levels(desc, ip, (int)threadIdx.x);
  RT *sum = reinterpret_cast<RT *>(small_smem);                                    // [2][n], weighted only
  uint32_t *word = reinterpret_cast<uint32_t *>(small_smem + (WT ? 2 * n * sizeof(RT) : 0));   // [2][n]
  if (threadIdx.x == 0) s_bad = 0;
  for (uint32_t w = threadIdx.x; w < kSmallMax / 32; w += blockDim.x) s_pred[w] = 0;
  __syncthreads();
  uint32_t x[kSmallElems], bad = 0;
  RT v[kSmallElems];
#pragma unroll
  for (int e = 0; e < kSmallElems; ++e) {
    const uint32_t j = threadIdx.x + e * blockDim.x;
    x[e] = kSmallSettled;
    v[e] = 0;
    if (j >= n) continue;
    const uint32_t s = __ldg(succ + j);
    const bool inner = s != j && s < n;
    if (s >= n) bad |= kErrRange;
    x[e] = inner ? 1u << 16 | s : kSmallSettled | j;
    word[j] = x[e];
    if constexpr (WT != 0) {
      v[e] = inner ? (RT)load_weight<WT>(weight, j) : (RT)0;
      sum[j] = v[e];
    }
    if (validate && inner && (atomicOr(&s_pred[s >> 5], 1u << (s & 31u)) >> (s & 31u) & 1u)) bad |= kErrNotList;
  }
  __syncthreads();
  uint32_t b = 0, all;
  for (int round = 0; round < kSmallRounds; ++round) {
    const uint32_t *wcur = word + b * n;
    const RT *scur = sum + b * n;
    uint32_t *wnxt = word + (b ^ 1u) * n;
    RT *snxt = sum + (b ^ 1u) * n;
    all = kSmallSettled;
#pragma unroll
    for (int e = 0; e < kSmallElems; ++e) {
      const uint32_t j = threadIdx.x + e * blockDim.x;
      if (j >= n) continue;
      if (!(x[e] & kSmallSettled)) {
        const uint32_t a = x[e] & kSmallPtr;
        x[e] = (x[e] & 0xFFFF0000u) + wcur[a];
        if constexpr (WT != 0) v[e] += scur[a];
      }
      all &= x[e];
      wnxt[j] = x[e];
      if constexpr (WT != 0) snxt[j] = v[e];
    }
    b ^= 1u;
    if (__syncthreads_and((all & kSmallSettled) != 0)) break;
  }
#pragma unroll
  for (int e = 0; e < kSmallElems; ++e) {
    const uint32_t j = threadIdx.x + e * blockDim.x;
    if (j >= n) continue;
    if (!(x[e] & kSmallSettled)) bad |= kErrCycle;
    rank[j] = WT != 0 ? v[e] : (RT)(x[e] >> 16);
  }
  if (bad) atomicOr(&s_bad, bad);
  __syncthreads();
  if (threadIdx.x == 0) {
    *status = s_bad;
    desc[0].visited = n;
  }
}

uint32_t small_max() { return kSmallMax; }

cudaError_t small_setup() {
  const int most = 2 * kSmallMax * (8 + 4);
  cudaError_t e = cudaFuncSetAttribute(k_small<1, uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small<1, unsigned long long>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small<2, uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small<2, unsigned long long>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  return e;
}

cudaError_t launch_small(const uint32_t *succ, const void *weight, int wtype, uint32_t n, void *rank, int rank_bytes,
                         int validate, LevelDesc *desc, const InitParams &ip, uint32_t *status, cudaStream_t s) {
  if (n == 0 || n > kSmallMax) return cudaErrorInvalidValue;
  const int block = (int)std::min<uint32_t>(kSmallThreads, (n + 31u) / 32u * 32u);
  const size_t smem = 2 * (size_t)n * (4 + (wtype ? rank_bytes : 0));
#define LR_SMALL(W)                                                                                             \
  do {                                                                                                          \
    if (rank_bytes == 4)                                                                                        \
      k_small<W, uint32_t><<<1, block, smem, s>>>(succ, weight, n, reinterpret_cast<uint32_t *>(rank), validate, desc, \
                                                  ip, status);                                                  \
    else                                                                                                        \
      k_small<W, unsigned long long><<<1, block, smem, s>>>(                                                    \
          succ, weight, n, reinterpret_cast<unsigned long long *>(rank), validate, desc, ip, status);           \
  } while (0)
  if (wtype == 0) LR_SMALL(0);
  else if (wtype == 1) LR_SMALL(1);
  else LR_SMALL(2);
#undef LR_SMALL
  count_launch();
  return cudaGetLastError();
}

}  // namespace lr
