// lr_engine.cu -- host engine of liblr.so: argument checks, the static level
// plan, workspace layout, per-stream contexts, launch sequence, device status
// and profiling.  Implements the C ABI declared in include/lr.h.
//
// Recursion plan (Section 2.1: rank the rulers' list recursively, then
// propagate; Section 3 runs a few sparse ruling-set rounds before pointer
// doubling).  The number of levels and every array size are fixed on the host
// from n and a bound h on the number of lists:
//   cap_0 = n,  cap_{l+1} = min(cap_l, ceil(cap_l / f_l) + h),
// until a level is small enough for the base case (k_jump).  The actual sizes are decided
// on the device (each level's head scan writes the next level's size and
// mode), so a call never waits for the device unless h has to be counted
// first, and a call with a known bound can be captured in a CUDA graph.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <nvtx3/nvToolsExt.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "lr.h"
#include "lr_engine.h"
#include "lr_hostview.h"
#include "lr_kernels.h"

namespace lr {

// ---------------------------------------------------------------- tuning
static uint32_t env_u32(const char *spec, const char *key, uint32_t dflt) {
  if (!spec) return dflt;
  std::string s(spec), k = std::string(key) + "=";
  size_t p = 0;
  while ((p = s.find(k, p)) != std::string::npos) {
    if (p == 0 || s[p - 1] == ',') return (uint32_t)strtoul(s.c_str() + p + k.size(), nullptr, 10);
    p += k.size();
  }
  return dflt;
}

// Default ruler fraction at level 0 by size (measured on GB300, random order;
// a single list, int32 weights / unweighted where both are given).
//  - Up to 4.7 million elements the rulers' list goes straight to the base
//    case (k_jump), whose time grows with its size, and the chase is bound by
//    the latency of its longest segment, about f ln(n / f) dependent steps:
//    the two balance near 200 to 400 thousand rulers (2^20: 172 us a call at
//    1/3 to 1/8, 199 at 1/12; 2^21: 189 at 1/8, 207 at 1/4, 211 at 1/16).
//  - Then one more level stands between them and rulers get cheaper: 7
//    million 377 / 296 us at 1/8, 393 / 326 at 1/16; 20 million 1033 / 822 at
//    1/12, 1066 / 849 at 1/16, 1098 / 860 at 1/24.
//  - Beyond L2 the chase is bound by the random-access rate; fewer rulers
//    shrink the recursion and the final pass's gathers more than their longer
//    segments lengthen the chase's tail: 2^26 3.11 / 2.29 ms at 1/24, 3.13 /
//    2.35 at 1/16; 2^27 4.84 at 1/48, 4.94 at 1/24; 2^28 10.10 at 1/64, 10.20
//    at 1/48, 11.00 at 1/16; 2^30 43.1 at 1/96, 43.6 at 1/64.
struct F0Step { int64_t below; uint32_t f0_inv; };
static const F0Step kF0Steps[] = {
    {3ll << 18, 4}, {5ll << 18, 6}, {5ll << 19, 8}, {9ll << 19, 12}, {1ll << 23, 8}, {3ll << 23, 12},
    {5ll << 23, 16}, {3ll << 25, 24}, {1ll << 27, 32}, {3ll << 26, 48}, {1ll << 29, 64}};

static uint32_t default_f0_inv(int64_t n) {
  for (const F0Step &t : kF0Steps)
    if (n < t.below) return t.f0_inv;
  return 96;
}

// A batch beyond L2 chases level 0 in element order: its records stay in L2
// only if the front (threads x ruler spacing) is narrow (1024 instances,
// 4.7e8 elements: 15.9 ms at 1/12, 16.1 at 1/16, 17.4 at 1/8, 17.7 at 1/24;
// 22 million elements 1.00 / 1.03 / 1.04 / 1.14 ms).
constexpr int64_t kOrdSpacingFrom = 1ll << 24;
static uint32_t default_f0_inv_batch(int64_t n) {
  if (n < (1ll << 23)) return default_f0_inv(n);
  return n < kOrdSpacingFrom ? 16 : 12;
}

// Largest level below the first that the base case ranks (k_jump), unless the
// caller sets a smaller bound: with 262 / 350 / 524 thousand elements it takes
// 25 / 35 / 65 us, one more level in front of it (chase at 1/4, selection,
// propagation) about 60 us less the smaller base case's 18.
constexpr uint32_t kJumpMax = 3u << 17;

// Largest level 0 that the base case ranks (k_jump needs no heads, no count of
// the lists and so no wait, and no further launches, but reads n log2 n
// records where the ruling set's chase reads n).  Random order, a whole call,
// base case / ruling set: 131 thousand elements 70 / 145 us, 2^19 108 / 165,
// 2^20 177 / 197, 1.5 million 226 / 211.  Beyond some 620 thousand elements
// not all of them are held by running threads, which costs lists in memory
// order most (1.5 million in locality order 467 / 143 us).
constexpr uint32_t kBase0Max = 1u << 19;

// Default ruler fraction below level 0: 1/4 where that already reaches the
// base case (2^24, 10^6 rulers: 900 us a call at 1/4, 907 at 1/6, 912 at 1/8).
static uint32_t default_f_inv(int64_t n, uint32_t f0_inv) {
  return n / f0_inv <= 4ll * kJumpMax ? 4 : 8;
}

Tuning resolve_tuning_builtin(int64_t n, bool weighted, bool batch) {
  (void)weighted;
  Tuning u;
  u.f0_inv = batch ? default_f0_inv_batch(n) : default_f0_inv(n);
  u.f_inv = default_f_inv(n, u.f0_inv);
  u.cutoff = kMaxCutoff;
  u.block = 256;
  u.ctas = 0;
  u.xchg = 1;
  u.chase0 = LR_CHASE0_AUTO;
  u.algo = LR_ALGO_SRS;
  u.contract = LR_CONTRACT_AUTO;
  u.spawn = 0;
  u.ord = 2;              // batches: every level of more than kOrdMinBytes in element order
  u.base0 = kBase0Max;
  u.base = kJumpMax;
  u.pf = 4;               // ... prefetching its records 4K elements ahead of each draw
  return u;
}

Tuning resolve_tuning(const lr_tuning *t, int64_t n, bool weighted, bool batch) {
  Tuning u = resolve_tuning_builtin(n, weighted, batch);
  const uint32_t f0_builtin = u.f0_inv;
  u.f_inv = 0;
  lr_tuning tt;
  if (tuned_lookup(n, weighted, batch, &tt)) {
    if (tt.f0_inv) u.f0_inv = tt.f0_inv;
    if (tt.f_inv) u.f_inv = tt.f_inv;
    // (not its cutoff: entries saved before the base case jumped pointers hold
    // bounds of 12288 and less, which would take it away from whole octaves)
    if (tt.chase_block) u.block = tt.chase_block;
    if (tt.chase_ctas) u.ctas = tt.chase_ctas;
  }
  const char *env = getenv("LR_TUNING");
  u.f0_inv = env_u32(env, "f0", u.f0_inv);
  u.f_inv = env_u32(env, "f", u.f_inv);
  u.cutoff = env_u32(env, "cutoff", u.cutoff);
  u.block = env_u32(env, "block", u.block);
  u.ctas = env_u32(env, "ctas", u.ctas);
  u.xchg = env_u32(env, "xchg", 1);
  const uint32_t env_log = env_u32(env, "log", 2);      // log=1 / log=0: force a level-0 form
  if (env_log < 2) u.chase0 = env_log ? LR_CHASE0_LOG : LR_CHASE0_EXCHANGE;
  u.algo = env_u32(env, "algo", LR_ALGO_SRS);
  u.contract = env_u32(env, "contract", u.contract);
  u.spawn = env_u32(env, "spawn", u.spawn);
  u.ord = env_u32(env, "ord", u.ord);
  u.pf = env_u32(env, "pf", u.pf);
  if (t) {
    if (t->spawn) u.spawn = t->spawn;
    if (t->chase0) u.chase0 = t->chase0;
    if (t->algorithm) u.algo = t->algorithm;
    if (t->contract) u.contract = t->contract;
    if (t->f0_inv) u.f0_inv = t->f0_inv;
    if (t->f_inv) u.f_inv = t->f_inv;
    if (t->cutoff) u.cutoff = t->cutoff;
    if (t->chase_block) u.block = t->chase_block;
    if (t->chase_ctas) u.ctas = t->chase_ctas;
  }
  u.f0_inv = std::max<uint32_t>(2, u.f0_inv);
  u.f_inv = u.f_inv ? std::max<uint32_t>(2, u.f_inv) : default_f_inv(n, u.f0_inv);
  u.cutoff = std::min<uint32_t>(std::max<uint32_t>(u.cutoff, 64), kMaxCutoff);
  if (u.block != 128 && u.block != 256 && u.block != 512) u.block = 256;
  // what asks for the ruling set itself keeps level 0 to it; a caller's
  // spacing does unless it is the default, as the autotuner hands it out
  const bool srs = u.cutoff < kMaxCutoff || u.spawn || u.chase0 != LR_CHASE0_AUTO || env_u32(env, "f0", 0) ||
                   (t && t->f0_inv && t->f0_inv != f0_builtin);
  u.base0 = srs ? u.cutoff : kBase0Max;
  u.base = u.cutoff >= kMaxCutoff ? kJumpMax : u.cutoff;
  return u;
}

// Level-0 chase form: the log form (lr_log.cu) needs an unweighted single
// instance with int32 ranks and n <= 2^30; auto takes it from 2^25 on, where
// its one random access per element beats the exchange form's two, unless
// spawning (an exchange-form feature) was asked for.
constexpr uint64_t kLogAutoMin = 1ull << 25;
static bool use_log0(const Tuning &u, uint64_t n, bool weighted, int rank_bytes, bool extras, bool multi) {
  if (weighted || rank_bytes != 4 || extras || multi || n <= u.base0 || n > (1ull << 30) || !u.xchg)
    return false;
  if (u.chase0 == LR_CHASE0_LOG) return true;
  return u.chase0 == LR_CHASE0_AUTO && n >= kLogAutoMin && !u.spawn;
}

// Level 0 of a set of contiguous instances (a batch) chases its rulers in
// element order: a front that crosses the instances a few at a time keeps
// the records it touches, the reduced records it writes and, in the final
// pass, the rank gathers within a footprint the L2 holds.
// While the level's records fit L2 anyway, the order only costs: five launches
// to build it and half the threads (3.8 million weighted elements 249 us
// without, 306 with it; 15 million unweighted 586 / 663; 22 million weighted,
// 355 MB of records, 1237 / 1016).
// (Deeper levels of a batch keep each instance's rulers together too, and are
// chased in order by the same rule; LR_TUNING ord=1: level 0 only; ord=0: no
// level.)
constexpr uint64_t kOrdMinBytes = 128ull << 20;
static bool use_ord0(const Tuning &u, uint64_t n, bool rec16, bool log0, bool spawn0, bool extras, bool multi) {
  return u.ord != 0 && multi && !log0 && !spawn0 && !extras && n <= 0x7FFFFFFFull &&
         n * (rec16 ? 16 : 8) > kOrdMinBytes;
}

static size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

// CTAs of 256 threads per SM for the chase in element order: the front's
// width (threads x ruler spacing) must stay small enough that the instances
// it crosses fit in L2 (7.5e7 elements at 1/12, 4 / 6 / 8 CTAs: weighted 1.21 /
// 1.31 / 1.55 ms, unweighted 1.37 / 1.06 / 1.06; 4.7e8 weighted 6.7 / 7.7 / 9.4).
constexpr int kOrdCtasWeighted = 4, kOrdCtasUnweighted = 6;
// Below this size the packing pass counts the links that stay in their tiles
// itself, instead of a sample and a wait of its own before it.
constexpr uint64_t kPackFirst = 1ull << 22;

int chase_grid_for(const Tuning &u, bool rec16, bool log0, bool ord0, bool weighted) {
  int per = u.ctas ? (int)u.ctas : (log0 ? chase_log_occupancy((int)u.block) : chase_occupancy(rec16, (int)u.block));
  if (ord0 && !u.ctas) per = std::min(per, (weighted ? kOrdCtasWeighted : kOrdCtasUnweighted) * 256 / (int)u.block);
  return device_sm_count() * std::max(1, per);
}

// Level 0 of a weighted call tries 8-byte records (Rec8w): half the bytes of
// every pass over them, and of the footprint that sets the rate of the chase's
// random exchanges (2^24 elements: 128 MiB and 61 G/s against 256 MiB and 35).
// The packing pass finds out whether the weights allow it.  A call that waits
// for its list count learns the answer there; another launches the kernels of
// both kinds, of which those of the wrong one return at once, so it tries from
// a size on where their 10 us do not count.
constexpr uint64_t kNarrowAsyncMin = 1ull << 22;
static bool use_narrow(const Tuning &u, uint64_t n, bool weighted, bool spawn0, bool extras, bool waits) {
  return weighted && !extras && !spawn0 && u.xchg && n > u.base0 && n <= 0x7FFFFF00ull &&
         (waits || n >= kNarrowAsyncMin);
}

// Static plan for n elements and at most h lists.
// Spawned rulers provided for at level 0: t waves leave about t ln(n/t)
// rulers in all (Section 2.5 cites this for spawning); a few t more as slack.
static uint32_t spawn_capacity(uint64_t n, uint64_t threads) {
  if (threads == 0) threads = 1;
  const double ratio = n > threads ? (double)n / (double)threads : 1.0;
  const double want = (double)threads * (std::ceil(std::log(ratio)) + 4.0);
  return (uint32_t)std::min<double>((double)n, want);
}

Plan make_plan(uint64_t n, uint64_t h, const Tuning &u, bool rec16_0, int rank_bytes,
               uint64_t seed, int chase_grid, bool log0, bool term, bool t0ws, bool spawn0, bool ord0,
               bool narrow) {
  Plan p;
  memset(&p, 0, sizeof(p));
  p.n = n;
  p.rec16_0 = rec16_0;
  p.log0 = log0;
  p.rank_bytes = rank_bytes;
  p.base = u.base;
  p.chase_grid = chase_grid;
  p.chase_block = (int)u.block;
  p.hcap = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(h, std::max<uint64_t>(n, 1)));
  p.cap[0] = (uint32_t)n;
  p.f_inv[0] = u.f0_inv;
  int L = 0;
  p.low[0] = n;
  const bool sp = spawn0 && (n > u.base0);
  p.spawn_cap = sp ? spawn_capacity(n, (uint64_t)chase_grid * u.block) : 0;
  if (n > u.base0) {
    for (;;) {
      const uint64_t r = (p.cap[L] + p.f_inv[L] - 1) / p.f_inv[L];
      uint64_t nc = std::min<uint64_t>(p.cap[L], r + p.hcap);
      if (L == 0 && sp) {
        p.raw_cap = (uint32_t)std::min<uint64_t>(0xFFFFFFF0ull, nc + p.spawn_cap);
        nc = std::min<uint64_t>(p.cap[0], nc + p.spawn_cap);
      }
      if (L == 0 && narrow) nc += n / kNarrowSteps + 1;
      ++L;
      p.cap[L] = (uint32_t)nc;
      p.low[L] = (p.low[L - 1] + p.f_inv[L - 1] - 1) / p.f_inv[L - 1];   // the sampled rulers alone
      p.f_inv[L] = u.f_inv;
      if (nc <= u.base) break;
      if (L == kMaxLevels) break;
      if (L >= 3 && (uint64_t)p.cap[L] * 4 > (uint64_t)p.cap[L - 1] * 3) break;  // stalled
    }
  }
  p.nlev = L + 1;
  for (int l = 0; l <= L; ++l) p.seed[l] = splitmix64(seed + 0x9E37ull * (uint64_t)(l + 1));

  // fixed part: independent of h
  size_t o = 0;
  p.off_desc = o; o = align_up(o + sizeof(LevelDesc) * (kMaxLevels + 1));
  p.off_zero = o;
  p.off_err = o; o = align_up(o + 16);
  p.off_hcount = o; o = align_up(o + 16);
  p.off_acc = o; o = align_up(o + 48);        // sums of terminals, successors; local links, sample; flags;
                                              // a terminal
  p.off_logctr = o; o = align_up(o + 16);
  p.off_bctr = o; o = align_up(o + sizeof(uint32_t) * 256);
  p.off_q = o; o = align_up(o + sizeof(uint32_t) * (size_t)chase_grid * kMaxLevels);
  p.off_bcnt = o; o = align_up(o + sizeof(uint64_t) * kHeadBlocks);
  p.zero_bytes = o - p.off_zero;
  p.off_bitmap = o; o = align_up(o + sizeof(uint32_t) * ((n + 31) / 32));
  if (!log0) { p.off_work[0] = o; o = align_up(o + (rec16_0 ? 16 : 8) * (size_t)n); }
  p.fixed_bytes = o;
  // variable part
  o = 0;
  for (int l = 1; l <= L; ++l) {
    p.off_work[l] = o; o = align_up(o + 16 * (size_t)p.cap[l]);
    p.off_R[l] = o; o = align_up(o + (size_t)rank_bytes * p.cap[l]);
  }
  if (log0) {
    // log entries: every element once plus one mark per ruler, in 32-entry
    // chunks handed out from one counter; each thread leaves at most one
    // chunk partly filled, and each CTA at most the rest of one window of
    // kLogWindow chunks, however long the segments are
    const uint64_t rulers = (n + p.f_inv[0] - 1) / p.f_inv[0] + p.hcap;
    const uint64_t need = (n + rulers + 31) / 32;
    const uint64_t threads = (uint64_t)chase_grid * u.block;
    const uint64_t total = need + threads + (uint64_t)chase_grid * kLogWindow + 4096;
    p.total_chunks = (uint32_t)std::min<uint64_t>(total, 0xFFFFFFF0ull);
    uint32_t lg = 0;
    while ((1ull << lg) < n) ++lg;
    p.shift = lg > 8 ? lg - 8 : 0;
    p.off_log = o; o = align_up(o + (size_t)p.total_chunks * 32 * 4);
    p.off_hdr = o; o = align_up(o + (size_t)p.total_chunks * 8);
    p.lg = log_geometry((uint32_t)n);
    p.off_pairs = o; o = align_up(o + (size_t)p.lg.na * p.lg.capA * 8);
    p.off_pairsB = o; o = align_up(o + (size_t)p.lg.nw * p.lg.capB * 8);
    p.off_cur = o;
    p.cur_bytes = 4 * ((size_t)p.lg.na + p.lg.nbB);           // claimed slots per region
    o = align_up(o + p.cur_bytes);
  }
  p.off_hA = o; o = align_up(o + 4 * (size_t)p.hcap);
  p.off_hB = o; o = align_up(o + 4 * (size_t)p.hcap);
  p.off_ns = o; o = align_up(o + 4 * (size_t)p.hcap);
  if (p.spawn_cap) {
    const size_t words = (p.spawn_cap + 31) / 32;
    p.off_sraw = o; o = align_up(o + 16 * (size_t)p.raw_cap);
    p.off_srraw = o; o = align_up(o + (size_t)rank_bytes * p.raw_cap);
    p.off_supre = o; o = align_up(o + 4 * words);
    p.off_sctr = o; o = align_up(o + 16 + 4 * (size_t)chase_grid);
    p.off_sused = o; o = align_up(o + 4 * words);
    p.spawn_zero = o - p.off_sctr;                // counter, cursors, claimed bitmap
  }
  p.ord0 = ord0 && p.nlev > 1;
  if (p.ord0) {
    // one set of arrays serves every level chased in order, one at a time:
    // marks and block counts for level 0's n, positions for the most
    // sampled rulers of any level
    uint64_t rmax = 0;
    for (int l = 0; l < L; ++l) rmax = std::max<uint64_t>(rmax, (p.cap[l] + p.f_inv[l] - 1) / p.f_inv[l]);
    p.off_ord = o; o = align_up(o + 4 * (size_t)rmax);
    p.off_cum = o; o = align_up(o + 4 * (size_t)((n + 255) / 256));
  }
  p.term = term;
  if (term) {
    for (int l = 1; l <= L; ++l) {
      p.off_T[l] = o; o = align_up(o + 4 * (size_t)p.cap[l]);
      p.off_tid[l] = o; o = align_up(o + 4 * (size_t)p.cap[l]);
    }
    p.off_hC = o; o = align_up(o + 4 * (size_t)p.hcap);   // keeps level 0's head list intact
    if (t0ws) { p.off_T0 = o; o = align_up(o + 4 * (size_t)n); }
  }
  p.var_bytes = std::max<size_t>(o, 256);
  return p;
}

// ---------------------------------------------------------------- contexts
static std::mutex g_mu;
static std::map<std::pair<int, uintptr_t>, Ctx *> g_ctx;
static bool g_setup_done[64];

static lr_status from_cuda(cudaError_t e) {
  if (e == cudaSuccess) return LR_OK;
  if (e == cudaErrorMemoryAllocation) return LR_ERR_OUT_OF_MEMORY;
  if (e == cudaErrorStreamCaptureUnsupported || e == cudaErrorStreamCaptureInvalidated)
    return LR_ERR_CAPTURE;
  return LR_ERR_CUDA;
}

// (with g_mu held)
static lr_status setup_device_locked(int dev) {
  cudaError_t e = cudaSuccess;
  if (dev >= 0 && dev < 64 && !g_setup_done[dev]) {
    e = small_setup();
    if (e == cudaSuccess) e = log_setup();
    if (e == cudaSuccess) e = lc_setup();
    if (e != cudaSuccess) return from_cuda(e);
    // Place lr_rank_noalloc's scratch array on this device now, while the
    // process can still spare its 64 MiB: under lazy module loading it would
    // otherwise be placed only at the first lr_rank_noalloc call, which may
    // come after the caller's allocator has taken all free memory.  Best
    // effort: a failure here surfaces at that call, with its status.
    (void)noalloc_resolve_scratch();
    g_setup_done[dev] = true;
  }
  return LR_OK;
}

lr_status setup_device_once() {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return from_cuda(e);
  std::lock_guard<std::mutex> g(g_mu);
  return setup_device_locked(dev);
}

Ctx *get_ctx(cudaStream_t stream, lr_status *st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) { *st = from_cuda(e); return nullptr; }
  std::lock_guard<std::mutex> g(g_mu);
  *st = setup_device_locked(dev);
  if (*st != LR_OK) return nullptr;
  auto key = std::make_pair(dev, (uintptr_t)stream);
  auto it = g_ctx.find(key);
  if (it != g_ctx.end()) { *st = LR_OK; return it->second; }
  Ctx *c = new Ctx();
  c->device = dev;
  e = cudaMallocHost((void **)&c->host_words, kHostWordsBytes);
  if (e != cudaSuccess) { delete c; *st = LR_ERR_OUT_OF_MEMORY; return nullptr; }
  memset(c->host_words, 0, kHostWordsBytes);
  g_ctx[key] = c;
  *st = LR_OK;
  return c;
}

void release_ctx(cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  Ctx *c = nullptr;
  {
    std::lock_guard<std::mutex> g(g_mu);
    auto it = g_ctx.find(std::make_pair(dev, (uintptr_t)stream));
    if (it == g_ctx.end()) return;
    c = it->second;
    g_ctx.erase(it);
  }
  cudaStreamSynchronize(stream);
  if (c->fixed) cudaFree(c->fixed);
  if (c->var) cudaFree(c->var);
  if (c->hostpath) cudaFree(c->hostpath);
  if (c->contract) cudaFree(c->contract);
  if (c->contract2) cudaFree(c->contract2);
  if (c->direct) cudaFree(c->direct);
  cudaFreeHost(c->host_words);
  delete c;
}

static bool stream_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) return false;
  return cs != cudaStreamCaptureStatusNone;
}

// Grow-only device buffer.
// Fault injection on the host (tests): with LR_INJECT_ALLOC_FAIL=1 in the
// environment every request for library workspace fails as a cudaMalloc
// that ran out of memory would, whether or not the arena had to grow, and
// without calling it.
static bool inject_alloc_failure() {
  const char *v = getenv("LR_INJECT_ALLOC_FAIL");
  return v && v[0] == '1';
}

// In a debug build LR_INJECT_LAUNCH_FAIL=1 makes the base case of an input fail
// between its two launches, as if the second had been refused.
static bool inject_launch_failure() {
  const char *v = kDebugChecks ? getenv("LR_INJECT_LAUNCH_FAIL") : nullptr;
  return v && v[0] == '1';
}

lr_status ensure_buffer(void **buf, size_t *cur, size_t want, cudaStream_t s) {
  if (inject_alloc_failure()) return LR_ERR_OUT_OF_MEMORY;
  if (*cur >= want && *buf) return LR_OK;
  if (stream_capturing(s)) return LR_ERR_CAPTURE;
  if (*buf) {
    cudaStreamSynchronize(s);
    cudaFree(*buf);
    *buf = nullptr;
    *cur = 0;
  }
  size_t sz = std::max(want, (size_t)1 << 20);
  cudaError_t e = cudaMalloc(buf, sz);
  if (e != cudaSuccess) { cudaGetLastError(); *buf = nullptr; return LR_ERR_OUT_OF_MEMORY; }
  *cur = sz;
  return LR_OK;
}

// ---------------------------------------------------------------- profiling
static bool g_prof = false;
struct ProfMark { cudaEvent_t ev; int phase; };  // phase of the interval ending here
struct ProfCall { std::vector<ProfMark> marks; int64_t n; int64_t launches; bool log0 = false; };
static std::vector<ProfCall> g_prof_pending;
static lr_profile g_prof_acc;

// Per call: an NVTX range (always; free without an attached tool) whose
// payload is n, NVTX marks at the phase boundaries, and, when profiling is
// on, CUDA events at the same boundaries for lr_profile_read.
static const char *const kPhaseNames[] = {"lr.prep", "lr.select", "lr.chase0", "lr.chase",
                                          "lr.base", "lr.finalize"};

struct Profiler {
  bool on = false;
  bool ranged = false;
  ProfCall call;
  cudaStream_t s = nullptr;
  void begin(cudaStream_t st, int64_t n) {
    nvtxEventAttributes_t a;
    memset(&a, 0, sizeof(a));
    a.version = NVTX_VERSION;
    a.size = NVTX_EVENT_ATTRIB_STRUCT_SIZE;
    a.messageType = NVTX_MESSAGE_TYPE_ASCII;
    a.message.ascii = "lr.call";
    a.payloadType = NVTX_PAYLOAD_TYPE_INT64;
    a.payload.llValue = n;
    nvtxRangePushEx(&a);
    ranged = true;
    on = g_prof && !stream_capturing(st);
    s = st;
    if (!on) return;
    call.n = n;
    call.launches = launch_count();
    mark(-1);
  }
  void mark(int phase) {
    note(phase);
    record(phase);
  }
  void note(int phase) {
    if (ranged && phase >= 0) nvtxMarkA(kPhaseNames[phase]);
  }
  void record(int phase) {
    if (!on) return;
    ProfMark m;
    m.phase = phase;
    cudaEventCreate(&m.ev);
    cudaEventRecord(m.ev, s);
    call.marks.push_back(m);
  }
  void end() {
    if (ranged) { nvtxRangePop(); ranged = false; }
    if (!on) return;
    on = false;
    call.launches = launch_count() - call.launches;
    std::lock_guard<std::mutex> g(g_mu);
    g_prof_pending.push_back(call);
  }
  // take back the marks from the k-th on (work that turned out not to be done)
  void drop_from(size_t k) {
    for (size_t i = k; i < call.marks.size(); ++i) cudaEventDestroy(call.marks[i].ev);
    if (call.marks.size() > k) call.marks.resize(k);
  }
  // drop a call that turned out not to happen (its marks are not recorded)
  void cancel() {
    if (ranged) { nvtxRangePop(); ranged = false; }
    if (!on) return;
    for (auto &m : call.marks) cudaEventDestroy(m.ev);
    call.marks.clear();
    on = false;
  }
  // a call that returns early (an error) closes its range and drops its marks
  ~Profiler() { cancel(); }
};
enum { PH_PREP = 0, PH_SELECT, PH_CHASE0, PH_CHASE, PH_BASE, PH_FINAL };

// ---------------------------------------------------------------- the run
// Pinned host buffers, as the device sees them (or null): the inputs, of which
// Inputs::succ and weight are then device memory to hold a copy where one is
// needed, and where the ranks go; *ranks_out is set if they went there rather
// than to Inputs::rank.
struct HostBuffers {
  const uint32_t *succ;
  const void *weight;
  void *rank;
  bool *ranks_out;
};

struct Inputs {
  const uint32_t *succ;
  const void *weight;
  int wtype;          // 0 none, 1 i32, 2 i64
  void *rank;
  int rank_bytes;
  uint64_t n;
  const int64_t *offsets;  // batched form
  int32_t k;
  int validate;
  uint64_t seed;
  int64_t max_lists;
  int sync;
  void *ws;
  size_t ws_bytes;
  const uint32_t *const *sptr;   // per-instance pointer tables (device), or null
  const void *const *wptr;
  void *const *rptr;
  Ctx *ctx;                      // use this context instead of the per-stream one
  int count_in_ws;               // caller workspace, but still count the lists first
  uint32_t *term;                // extra outputs (device, optional): terminal ids,
  void *prefix;                  // head-relative ranks,
  int incl;                      // inclusive-tail ranks
  uint32_t *err_ext;             // record device errors here (and do not clear it)
  int no_contract;               // never contract (the contracted list itself)
  int builtin_tuning;            // ignore LR_TUNING and the autotuned table
  HostBuffers h;
};

static lr_status map_device_bits(uint32_t bits) {
  if (bits & kErrDebug) return LR_ERR_INTERNAL;      // a debug build's index check
  if (bits & kErrRange) return LR_ERR_OUT_OF_RANGE;
  if (bits & kErrNotList) return LR_ERR_NOT_A_LIST;
  if (bits & kErrCycle) return LR_ERR_CYCLE;
  if (bits & kErrCapacity) return LR_ERR_CAPACITY;
  if (bits & kErrInternal) return LR_ERR_NOT_A_LIST;
  return LR_OK;
}

#define LR_TRY(expr)                                   \
  do {                                                 \
    cudaError_t e__ = (expr);                          \
    if (e__ != cudaSuccess) return from_cuda(e__);     \
  } while (0)

// Wait for a kernel on stream s to write `token` to the pinned word *w.  The
// stream's state is looked at now and then, so that the wait ends whatever
// becomes of the kernel; and a caller that has asked for waits which give up
// their core (cudaSetDeviceFlags: blocking, yield) gets one, for the stream.
static lr_status wait_word(const uint32_t *w, uint32_t token, cudaStream_t s) {
  bool asked = false;
  for (uint32_t spin = 1; __atomic_load_n(w, __ATOMIC_ACQUIRE) != token; ++spin) {
    if (spin % 4096 != 0) continue;
    unsigned flags = 0;
    if (!asked && cudaGetDeviceFlags(&flags) == cudaSuccess &&
        (flags & (cudaDeviceScheduleYield | cudaDeviceScheduleBlockingSync)))
      LR_TRY(cudaStreamSynchronize(s));
    asked = true;
    const cudaError_t e = cudaStreamQuery(s);
    if (e == cudaErrorNotReady) continue;
    LR_TRY(e);
    return __atomic_load_n(w, __ATOMIC_ACQUIRE) == token ? LR_OK : LR_ERR_INTERNAL;
  }
  return LR_OK;
}

// Copy the call's device error word to the context's pinned status word;
// with sync, wait and return the status it encodes.  err == nullptr: a kernel
// has written the status word itself.
static lr_status finish_call(Ctx *c, const uint32_t *err, int sync, cudaStream_t s) {
  if (err) LR_TRY(cudaMemcpyAsync(c->host_words, err, 4, cudaMemcpyDeviceToHost, s));
  c->pending_status = true;
  if (sync) {
    LR_TRY(cudaStreamSynchronize(s));
    c->pending_status = false;
    const uint32_t bits = c->host_words[0];
    c->host_words[0] = 0;
    return map_device_bits(bits);
  }
  return LR_OK;
}

// Workspace of the pointer-doubling algorithm: error word and scratch sums,
// the has-predecessor bitmap (validation), two record arrays.
struct WyPlan {
  size_t off_err, off_sums, off_bitmap, off_a, off_b, zero_bytes, bytes;
};

static WyPlan wyllie_plan(uint64_t n, bool w16) {
  WyPlan q;
  size_t o = 0;
  q.off_err = o; o = align_up(o + 16);
  q.off_sums = o; o = align_up(o + 48);
  q.zero_bytes = o;
  q.off_bitmap = o; o = align_up(o + sizeof(uint32_t) * ((n + 31) / 32));
  q.off_a = o; o = align_up(o + (w16 ? 16 : 8) * n);
  q.off_b = o; o = align_up(o + (w16 ? 16 : 8) * n);
  q.bytes = o;
  return q;
}

// 16-byte records exactly when weighted: the layout k_prep0 writes.
static bool wyllie_w16(const Inputs &in) { return in.wtype != 0; }

// Whole-list pointer doubling (lr_wyllie.cu) on the same inputs and outputs.
static lr_status run_wyllie(const Inputs &in, Ctx *c, cudaStream_t s) {
  c->last_nlev = 0;
  const bool w16 = wyllie_w16(in);
  const WyPlan q = wyllie_plan(in.n, w16);
  char *base = nullptr;
  if (in.ws) {
    if (in.ws_bytes < q.bytes) return LR_ERR_INVALID_ARGUMENT;
    base = (char *)in.ws;
  } else {
    const lr_status st = ensure_buffer(&c->var, &c->var_bytes, q.bytes, s);
    if (st != LR_OK) return st;
    base = (char *)c->var;
  }
  uint32_t *err = (uint32_t *)(base + q.off_err);
  uint32_t *bitmap = (uint32_t *)(base + q.off_bitmap);
  unsigned long long *sums = (unsigned long long *)(base + q.off_sums);
  void *A = base + q.off_a, *B = base + q.off_b;
  Profiler prof;
  if (!in.ctx) prof.begin(s, (int64_t)in.n);
  LR_TRY(cudaMemsetAsync(base, 0, in.validate ? q.off_a : q.zero_bytes, s));
  // without validation the scratch sums stand in for the bitmap, so the
  // pass issues no per-element atomics
  LR_TRY(launch_prep0(in.succ, in.weight, in.wtype, (uint32_t)in.n, A, w16 ? kRecKind16 : kRecKind8, in.validate ? bitmap : nullptr, err,
                      in.validate, in.offsets, in.k, in.validate ? nullptr : sums, nullptr, WeightScan{}, nullptr,
                      nullptr, s));
  prof.mark(PH_PREP);
  LR_TRY(launch_wyllie(A, B, w16, (uint32_t)in.n, in.rank, in.rank_bytes, err, s));
  prof.mark(PH_BASE);
  prof.end();
  return finish_call(c, err, in.sync, s);
}

lr_status run(const Inputs &in, const lr_tuning *tuning, cudaStream_t s);

static InitParams init_params(const Plan &p) {
  InitParams ip;
  memset(&ip, 0, sizeof(ip));
  ip.nlev = p.nlev;
  ip.n0 = (uint32_t)p.n;
  ip.mode0 = p.nlev == 1 ? kModeBase : kModeSrs;
  for (int l = 0; l < p.nlev; ++l) {
    ip.f_inv[l] = p.f_inv[l];
    ip.cap[l] = p.cap[l];
    ip.seed[l] = p.seed[l];
  }
  ip.hcap = p.hcap;
  ip.base = p.base;
  return ip;
}

// The words that run_base's two launches share, while a call uses them.  A call
// that fails between the launches clears them itself, so that neither the next
// call nor a graph captured before finds what it left.  A captured call has
// not run: it leaves the context's note of them alone.
struct OwnWords {
  Ctx *ctx;                                    // null: not used (or captured)
  size_t bytes;
  cudaStream_t s;
  void left_clean() {
    if (ctx) ctx->direct_clean = true;
    ctx = nullptr;
  }
  ~OwnWords() {
    if (ctx) ctx->direct_clean = cudaMemsetAsync(ctx->direct, 0, bytes, s) == cudaSuccess;
  }
};

// An input that the base case ranks as it is: one pass that packs the records,
// then k_jump, which needs no heads.  From `checked` elements on (and for a
// batch of separate buffers) two predecessors and a broken promise of
// max_lists are looked for, as the ruling set notices them there.
static lr_status run_base(const Inputs &in, const Plan &p, bool checked, bool capturing, char *fixed, char *var,
                          Ctx *c, cudaStream_t s) {
  const uint32_t n = (uint32_t)in.n;
  const bool extras = p.term, marks = checked || in.validate || in.prefix != nullptr;
  LevelDesc *desc = (LevelDesc *)(fixed + p.off_desc);
  uint32_t *err = in.err_ext ? in.err_ext : (uint32_t *)(fixed + p.off_err);
  uint32_t *bitmap = (uint32_t *)(fixed + p.off_bitmap);
  void *work = fixed + p.off_work[0];
  uint32_t *T0 = extras ? (in.term ? in.term : (uint32_t *)(var + p.off_T0)) : nullptr;
  Profiler prof;
  if (!in.ctx) prof.begin(s, (int64_t)in.n);
  // (a context passed in, or a shared error word, has no status word of its
  // own that the device can write)
  if (n <= small_max() && !in.sptr && !in.offsets && !extras && !in.ctx && !in.err_ext) {
    LR_TRY(launch_small(in.succ, in.weight, in.wtype, n, in.rank, p.rank_bytes, in.validate, desc, init_params(p),
                        c->host_words, s));
    c->last_desc = desc;
    c->last_nlev = 1;
    prof.mark(PH_BASE);
    prof.end();
    return finish_call(c, nullptr, in.sync, s);
  }
  // The error word, the list count and the marks start at zero.  The stream's
  // own ones are left so by k_jump, which also reports the status: a call is
  // two launches, where a clear before and a copy after them took another 9
  // us.  Memory that is not the stream's own (or cannot be had now) is cleared.
  JumpInput ji;
  memset(&ji, 0, sizeof(ji));
  bool own = !in.ws && !in.ctx && !in.err_ext && !extras && n <= kBase0Max;
  const size_t own_bytes = 256 + kBase0Max / 8;
  OwnWords words_used = {nullptr, own_bytes, s};
  if (own && !c->direct) own = !capturing && ensure_buffer(&c->direct, &c->direct_bytes, own_bytes, s) == LR_OK;
  if (own) {
    if (!c->direct_clean) LR_TRY(cudaMemsetAsync(c->direct, 0, own_bytes, s));       // new
    if (!capturing) words_used.ctx = c;
    uint32_t *words = (uint32_t *)c->direct;
    err = words;
    ji.count = words + 16;
    ji.ticket = words + 32;
    ji.status = c->host_words;
    bitmap = words + 64;
    if (marks || in.sptr) ji.clear = bitmap;
  } else {
    // the bitmap follows the words that start at zero
    LR_TRY(cudaMemsetAsync(fixed + p.off_zero, 0,
                           p.off_bitmap - p.off_zero + (marks ? 4 * (((size_t)n + 31) / 32) : 0), s));
    ji.count = (uint32_t *)(fixed + p.off_hcount);
  }
  const InitParams ip = init_params(p);
  const int kind = p.rec16_0 ? kRecKind16 : kRecKind8;
  if (in.sptr) {
    LR_TRY(launch_init(desc, ip, nullptr, nullptr, nullptr, nullptr, nullptr, s));
    LR_TRY(launch_prep0_ptrs(in.sptr, in.wptr, in.wtype, n, work, kind, WeightScan{}, bitmap, err, 1, in.offsets,
                             in.k, s));
  } else {
    LR_TRY(launch_prep0(in.succ, in.weight, in.wtype, n, work, kind, marks ? bitmap : nullptr, err,
                        checked || in.validate, in.offsets, in.k, nullptr, nullptr, WeightScan{}, desc, &ip, s));
  }
  if (!in.ctx) { c->last_desc = desc; c->last_nlev = 1; }
  prof.mark(PH_PREP);
  if (inject_launch_failure()) return LR_ERR_CUDA;
  if (checked && in.max_lists > 0) {
    ji.max_lists = (uint64_t)in.max_lists;
    ji.bitmap = bitmap;
  }
  ji.rptr = in.rptr;
  ji.offsets = in.offsets;
  ji.k = in.k;
  LR_TRY(launch_jump(desc, 0, work, p.rec16_0, in.rank, p.rank_bytes, n, err, nullptr, nullptr, T0, &ji, s));
  words_used.left_clean();
  prof.mark(PH_BASE);
  if (extras)
    LR_TRY(launch_outputs(desc, bitmap, nullptr, n, T0, in.rank, in.prefix, p.rank_bytes, in.incl, in.weight,
                          in.wtype, in.offsets, in.k, in.offsets != nullptr && in.term != nullptr, s));
  prof.mark(PH_FINAL);
  prof.end();
  return finish_call(c, own ? nullptr : err, in.sync, s);
}

// Tile-local contraction (lr_contract.cu) around the ruling set: count the
// local heads of every tile, build the contracted list, rank it (inclusive
// form, through run() itself), restore every element.  Returns
// LR_ERR_NOT_FOUND (nothing enqueued that writes outputs) when the exact
// count shows that contraction would not shrink the list enough.
static lr_status run_contracted(const Inputs &in, const lr_tuning *tuning, Ctx *c, bool forced,
                                cudaStream_t s) {
  const uint32_t n = (uint32_t)in.n;
  const uint32_t nt = lc_tiles(n);
  const size_t words = (size_t)nt * lc_tile_words();
  size_t o = 0;
  const size_t off_err = o; o = align_up(o + 16);
  const size_t off_hb = o; o = align_up(o + 4 * words);
  const size_t off_wpre = o; o = align_up(o + 2 * words);
  const size_t off_tcnt = o; o = align_up(o + 4 * (size_t)nt);
  const size_t off_tpre = o; o = align_up(o + 4 * ((size_t)nt + 1));
  const size_t off_tail = o; o = align_up(o + 2 * (size_t)n);
  lr_status st = ensure_buffer(&c->contract, &c->contract_bytes, o, s);
  if (st != LR_OK) return st;
  char *b = (char *)c->contract;
  uint32_t *err = (uint32_t *)(b + off_err);
  LR_TRY(cudaMemsetAsync(b, 0, off_hb, s));
  Profiler prof;
  prof.begin(s, (int64_t)in.n);
  c->last_nlev = 0;
  uint32_t *hb = (uint32_t *)(b + off_hb);
  uint16_t *wpre = (uint16_t *)(b + off_wpre);
  uint32_t *tcnt = (uint32_t *)(b + off_tcnt);
  uint32_t *tpre = (uint32_t *)(b + off_tpre);
  uint16_t *tail16 = (uint16_t *)(b + off_tail);
  LR_TRY(launch_lc_solve(in.succ, in.weight, in.wtype, n, in.rank, in.rank_bytes, tail16, hb, wpre, tcnt,
                         tpre, err, c->host_words, ++c->token, s));
  st = wait_word(c->host_words + kHostToken, c->token, s);
  if (st != LR_OK) return st;
  const uint64_t m = c->host_words[1];
  if (!forced && m * 5 > (uint64_t)n * 3) { prof.cancel(); return LR_ERR_NOT_FOUND; }
  // the contracted list: successors, weights (int32 unweighted: at most one
  // tile's links; int64 weighted), ranks in the caller's type
  const int wc = in.wtype == 0 ? 1 : 2;
  const size_t wb = wc == 1 ? 4 : 8;
  size_t o2 = 0;
  const size_t off_sc = o2; o2 = align_up(o2 + 4 * std::max<uint64_t>(m, 1));
  const size_t off_wc = o2; o2 = align_up(o2 + wb * std::max<uint64_t>(m, 1));
  const size_t off_rc = o2; o2 = align_up(o2 + (size_t)in.rank_bytes * std::max<uint64_t>(m, 1));
  st = ensure_buffer(&c->contract2, &c->contract2_bytes, o2, s);
  if (st != LR_OK) return st;
  char *b2 = (char *)c->contract2;
  LR_TRY(launch_lc_nodes(in.succ, in.weight, in.wtype, n, in.rank, in.rank_bytes, tail16, hb, wpre, tpre,
                         (uint32_t *)(b2 + off_sc), b2 + off_wc, err, s));
  prof.mark(PH_PREP);
  if (m > 0) {
    Inputs sub;
    memset(&sub, 0, sizeof(sub));
    sub.succ = (const uint32_t *)(b2 + off_sc);
    sub.weight = b2 + off_wc;
    sub.wtype = wc;
    sub.rank = b2 + off_rc;
    sub.rank_bytes = in.rank_bytes;
    sub.n = m;
    sub.validate = in.validate;
    sub.seed = in.seed;
    sub.ctx = c;
    sub.incl = 1;
    sub.err_ext = err;
    sub.no_contract = 1;
    st = run(sub, tuning, s);
    if (st != LR_OK) return st;
  }
  prof.mark(PH_CHASE0);
  LR_TRY(launch_lc_finish(in.succ, in.weight, in.wtype, n, in.rank, in.rank_bytes, tail16, hb, wpre, tpre,
                          b2 + off_rc, s));
  prof.mark(PH_FINAL);
  prof.end();
  return finish_call(c, err, in.sync, s);
}

lr_status run(const Inputs &given, const lr_tuning *tuning, cudaStream_t s) {
  Inputs in = given;
  const bool ptrs = in.sptr != nullptr;
  lr_status st = LR_OK;
  Ctx *c = in.ctx ? in.ctx : get_ctx(s, &st);
  if (!c) return st;
  if (in.n == 0) {
    // nothing to rank; still clear the stream's recorded status
    c->host_words[0] = 0;
    c->pending_status = false;
    return LR_OK;
  }
  // Inputs in host memory: the base case and the first pass of the exchange
  // form, which read them once, read them where they are; the other forms
  // copy them first.
  auto fetch = [&]() -> cudaError_t {
    if (!in.h.succ) return cudaSuccess;
    cudaError_t e = cudaMemcpyAsync((void *)in.succ, in.h.succ, 4 * in.n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && in.wtype)
      e = cudaMemcpyAsync((void *)in.weight, in.h.weight, (in.wtype == 1 ? 4 : 8) * in.n, cudaMemcpyHostToDevice, s);
    in.h.succ = nullptr;
    return e;
  };
  const bool capturing = stream_capturing(s);
  const Tuning u = in.builtin_tuning ? resolve_tuning_builtin((int64_t)in.n, in.wtype != 0, false)
                                     : resolve_tuning(tuning, (int64_t)in.n, in.wtype != 0,
                                                      in.offsets != nullptr || ptrs);
  if (u.algo == LR_ALGO_WYLLIE && !ptrs) {
    if (in.term || in.prefix || in.incl) return LR_ERR_INVALID_ARGUMENT;   // default algorithm only
    LR_TRY(fetch());
    return run_wyllie(in, c, s);
  }
  if (u.algo != LR_ALGO_SRS && u.algo != LR_ALGO_WYLLIE) return LR_ERR_INVALID_ARGUMENT;
  const bool outputs = in.term != nullptr || in.prefix != nullptr || in.incl != 0;
  bool extras = outputs;                       // to be carried through the levels
  // 16-byte level-0 records: weighted, or ranked at level 0 with terminal ids
  const bool rec16_0 = in.wtype != 0 || (extras && in.n <= u.base0);
  if (extras && ptrs) return LR_ERR_INVALID_ARGUMENT;
  const bool log0 = use_log0(u, in.n, in.wtype != 0, in.rank_bytes, extras, ptrs || in.offsets != nullptr);
  bool t0ws = extras && in.term == nullptr;
  const bool spawn0 = u.spawn != 0 && u.xchg != 0 && !log0 && !extras && !ptrs;
  // a batch chases its level-0 rulers in element order (the has-predecessor
  // bitmap, free once the heads are chosen, holds the ruler marks; level 1's
  // rank array, written only after the chase, holds the order)
  const bool ord0 = use_ord0(u, in.n, rec16_0, log0, spawn0, extras, ptrs || in.offsets != nullptr);
  // tile-local contraction: forced, or decided from the count of links that
  // stay inside their tile (the log form's first pass counts them and they
  // are read with the list count; otherwise a sample of the tiles decides)
  const bool contractible = u.contract != LR_CONTRACT_OFF && !in.no_contract && !ptrs &&
                            in.offsets == nullptr && !extras && in.ws == nullptr && in.ctx == nullptr &&
                            !capturing && in.max_lists <= 0 && in.n >= 16384 && in.n <= 0xFFFFFFFEull;
  if (contractible && u.contract == LR_CONTRACT_ON) {
    LR_TRY(fetch());
    const lr_status cs = run_contracted(in, tuning, c, true, s);
    if (cs != LR_ERR_NOT_FOUND) return cs;
  }
  const bool count_local = contractible && u.contract == LR_CONTRACT_AUTO && in.n > u.base0;
  // Counting the lists needs a wait.  The base case ranks level 0 without a
  // count, but a call above the smallest sizes is not capturable without a
  // promise of max_lists whichever way it is ranked.
  const bool checked = in.n > u.cutoff || ptrs;
  const bool may_count = in.max_lists <= 0 && (in.ws == nullptr || in.count_in_ws);
  if (may_count && checked && capturing) return LR_ERR_CAPTURE;
  const bool need_count = may_count && in.n > u.base0;
  const bool narrow = use_narrow(u, in.n, in.wtype != 0, spawn0, extras, need_count);
  // the element order, where the records that level 0 really has call for it
  const bool rec16_used = rec16_0 && !narrow;
  const bool ord_used = ord0 && in.n * (rec16_used ? 16 : 8) > kOrdMinBytes;
  const int grid = chase_grid_for(u, rec16_used, log0, ord_used, in.wtype != 0);
  uint64_t hb = in.max_lists > 0 ? (uint64_t)in.max_lists : in.n;
  Plan p = make_plan(in.n, hb, u, rec16_0, in.rank_bytes, in.seed, grid, log0, extras, t0ws, spawn0, ord0, narrow);

  // fixed part (level 0)
  char *fixed = nullptr;
  char *var = nullptr;
  if (in.ws) {
    if (in.ws_bytes < p.fixed_bytes + (need_count ? 0 : p.var_bytes)) return LR_ERR_INVALID_ARGUMENT;
    fixed = (char *)in.ws;
    var = fixed + p.fixed_bytes;
  } else {
    st = ensure_buffer(&c->fixed, &c->fixed_bytes, p.fixed_bytes, s);
    if (st != LR_OK) return st;
    fixed = (char *)c->fixed;
  }
  if (p.nlev == 1) {
    if (!in.ws) {
      st = ensure_buffer(&c->var, &c->var_bytes, p.var_bytes, s);
      if (st != LR_OK) return st;
      var = (char *)c->var;
    }
    if (in.h.succ) {
      in.succ = in.h.succ;
      in.weight = in.h.weight;
    }
    if (in.h.rank) {
      in.rank = in.h.rank;
      *in.h.ranks_out = true;
    }
    return run_base(in, p, checked, capturing, fixed, var, c, s);
  }
  if (log0) LR_TRY(fetch());
  // (the log form's last pass would hold every SM for the time of the link)
  const bool ranks_to_host = in.h.rank && !log0;
  LevelDesc *desc = (LevelDesc *)(fixed + p.off_desc);
  uint32_t *err = in.err_ext ? in.err_ext : (uint32_t *)(fixed + p.off_err);
  uint32_t *hcount = (uint32_t *)(fixed + p.off_hcount);
  uint32_t *qctr = (uint32_t *)(fixed + p.off_q);
  uint64_t *bcnt = (uint64_t *)(fixed + p.off_bcnt);
  uint32_t *bitmap = (uint32_t *)(fixed + p.off_bitmap);
  void *work0 = fixed + p.off_work[0];

  // Single instance, no validation: heads from the streaming sums (one list)
  // with the bitmap as the fallback, instead of atomics for every element.
  const bool sums0 = !log0 && !ptrs && in.offsets == nullptr && !in.validate;
  // With validation and a count: both, and no mark has to tell whether it was
  // set before.  As many heads (elements without a mark) as terminals means
  // that the other elements' successors are all distinct.  (A mark that must
  // return its word holds its thread for the round trip: 2^23 elements in
  // forests packed in 79 us that way, in 55 with marks and sums.)
  const bool sumsv = !log0 && !ptrs && in.offsets == nullptr && in.validate && need_count;
  // A batch (contiguous or one pointer per instance): per-instance sums (kept
  // at the start of the bitmap's memory, which must hold 16 bytes per
  // instance) give one head per instance and the number of lists, with the
  // bitmap as the fallback for the heads.
  const bool sums0b = !log0 && in.offsets != nullptr && !in.validate && !extras && !spawn0 &&
                      in.k > 0 && (uint64_t)in.k * 16 <= 4 * ((in.n + 31) / 32);
  Profiler prof;
  if (!in.ctx) prof.begin(s, (int64_t)in.n);
  unsigned long long *acc = (unsigned long long *)(fixed + p.off_acc);
  const size_t bitmap_bytes = sizeof(uint32_t) * ((in.n + 31) / 32);
  // A single instance needs the bitmap only if it turns out not to be one
  // list; otherwise it is cleared here with the words that start at zero,
  // which it follows.
  const bool late_bitmap = (log0 || sums0) && need_count && !in.validate;
  LR_TRY(cudaMemsetAsync(fixed + p.off_zero, 0, p.zero_bytes + (late_bitmap ? 0 : bitmap_bytes), s));
  // A first pass that packs records (the exchange form) would pack them in
  // vain for an input that is then contracted: from kPackFirst elements on,
  // decide from a sample of the tiles first.  (The log form's first pass only
  // reads succ, and counts every tile on the way; a shorter list is packed
  // sooner than the wait for the sample takes.)
  const bool local_exact = count_local && (log0 || ((sums0 || sumsv) && in.n < kPackFirst));
  // Most single instances are one list: its descriptors and level-0 chase are
  // queued before the sums are read, and do nothing if the device finds it is
  // not one (or that the sample says to contract it: then nor does the first
  // pass).  The sums come by a pinned word that the host watches, while the
  // chase runs.  (2^20 elements: the device sat idle for 13 of the call's 131
  // us, and 9 more of 737 in the wait for the sample at 2^24.)
  // Likewise a batch, as one list per instance.
  const bool guess_batch = sums0b && in.k <= kMaxOpenBatch && !ord_used;
  const bool guess = need_count && (sums0 || sumsv || guess_batch) && !in.ws && !spawn0;
  const uint64_t guess_lists = guess_batch ? (uint64_t)in.k : 1;
  const uint32_t ask_local = local_exact ? kLocalCounted : count_local && guess ? kLocalSampled : kLocalUnasked;
  if (count_local && !local_exact)
    LR_TRY(launch_local_sample(in.h.succ ? in.h.succ : in.succ, (uint32_t)in.n, acc + 2, s));
  if (count_local && !local_exact && !guess) {
    LR_TRY(cudaMemcpyAsync(c->host_words + 4, acc + 2, 16, cudaMemcpyDeviceToHost, s));
    LR_TRY(cudaStreamSynchronize(s));
    uint64_t smp[2];
    memcpy(smp, c->host_words + 4, 16);
    if (smp[0] * 2 >= smp[1]) {                // at least half the sampled links stay in their tile
      LR_TRY(fetch());
      prof.cancel();
      const lr_status cs = run_contracted(in, tuning, c, false, s);
      if (cs != LR_ERR_NOT_FOUND) return cs;
      prof.begin(s, (int64_t)in.n);            // not contracted after all: carry on
    }
  }
  // flags of weights too wide for 8-byte records (int32 ranks: none is)
  uint32_t *wflags = narrow ? reinterpret_cast<uint32_t *>(acc + 4) : nullptr;
  // The pass that packs level 0's records.  `again`: only the records, in 16
  // bytes, after a pass whose flags forbid 8-byte ones (unless_narrow: if they do).
  auto pack = [&](int kind, bool again, const uint32_t *unless_narrow) -> cudaError_t {
    const uint32_t n = (uint32_t)in.n;
    WeightScan scan;
    scan.flags = kind == kRecKind8w && in.rank_bytes == 8 ? wflags : nullptr;
    scan.unless_narrow = unless_narrow;
    scan.unless_local = ask_local == kLocalSampled && !again ? acc : nullptr;
    const bool host = in.h.succ && !again;
    scan.succ_copy = host ? (uint32_t *)in.succ : nullptr;
    scan.weight_copy = host ? (void *)in.weight : nullptr;
    unsigned long long *isums = again ? nullptr : reinterpret_cast<unsigned long long *>(bitmap);
    uint32_t *marks = again || sums0 ? nullptr : bitmap;
    if (ptrs && sums0b)
      return launch_prep0_ptrs_sums(in.sptr, in.wptr, in.wtype, n, work0, kind, scan, err, in.offsets, in.k, isums, s);
    if (ptrs)
      return launch_prep0_ptrs(in.sptr, in.wptr, in.wtype, n, work0, kind, scan, marks, err, in.validate, in.offsets,
                               in.k, s);
    if (sums0b)
      return launch_prep0_sums(in.succ, in.weight, in.wtype, n, work0, kind, scan, err, in.offsets, in.k, isums, s);
    const bool sums = (sums0 || sumsv) && !again;
    return launch_prep0(host ? in.h.succ : in.succ, host ? in.h.weight : in.weight, in.wtype, n, work0, kind, marks, err, in.validate && !sumsv, in.offsets,
                        in.k, sums ? acc : nullptr, sums && local_exact ? acc + 2 : nullptr, scan, nullptr, nullptr, s);
  };
  int kind0 = narrow ? kRecKind8w : rec16_0 ? kRecKind16 : kRecKind8;
  bool both = narrow && !need_count;           // 8- or 16-byte records: the device decides
  if (log0)
    LR_TRY(launch_sum0(in.succ, (uint32_t)in.n, acc, local_exact ? acc + 2 : nullptr, err, s));
  else
    LR_TRY(pack(kind0, false, nullptr));
  if (both) LR_TRY(pack(kRecKind16, true, wflags));
  uint32_t found = 0;                          // errors the count shows
  uint64_t one_head = 0;
  uint32_t one_term = 0;
  bool one_list = false;                       // the host has seen that level 0 is one list
  bool chased = false;                         // and it was one
  const size_t marks_before = prof.call.marks.size();
  if (guess) {
    const Plan g = make_plan(in.n, guess_lists, u, rec16_0, in.rank_bytes, in.seed, grid, log0, false, false, spawn0, ord0, narrow);
    st = ensure_buffer(&c->var, &c->var_bytes, g.var_bytes, s);
    if (st != LR_OK) return st;
    char *v = (char *)c->var;
    InitParams ip = init_params(g);
    ip.publish = c->host_words;
    ip.token = ++c->token;
    ip.check_local = ask_local;
    if (sumsv) {
      ip.heads = hcount;
      LR_TRY(launch_count_heads(bitmap, (uint32_t)in.n, hcount, s));
    }
    uint32_t *ns = (uint32_t *)(v + g.off_ns);
    if (guess_batch)
      LR_TRY(launch_open_batch(desc, ip, reinterpret_cast<const unsigned long long *>(bitmap), in.offsets, in.k,
                               kind0 == kRecKind8w ? wflags : nullptr, work0, kind0, ns,
                               (uint32_t *)(v + g.off_hB), s));
    else
      LR_TRY(launch_init(desc, ip, acc, kind0 == kRecKind8w ? wflags : nullptr, (uint32_t *)(v + g.off_hA), ns,
                         (uint32_t *)(v + g.off_hB), s));
    prof.record(PH_PREP);
    LR_TRY(launch_chase(desc, 0, work0, kind0, v + g.off_work[1], ns, qctr, g.chase_grid, g.chase_block, err,
                        (int)u.xchg, nullptr, nullptr, nullptr, nullptr, s));
    prof.record(PH_CHASE0);
    st = wait_word(c->host_words + kHostToken, ip.token, s);
    if (st != LR_OK) return st;
  }
  if (need_count) {
    // count the lists (one wait), then size the recursion for exactly that many:
    // a single-instance pass counts terminals in its reduction, a batch adds
    // its instances' terminal counts, the other passes count zero bits of the
    // has-predecessor bitmap
    unsigned long long sums[6];                // terminals, other successors, local links, (sample), flags,
                                               // a terminal
    const bool acc_read = log0 || sums0 || sumsv;
    if (acc_read && !guess)
      LR_TRY(cudaMemcpyAsync(c->host_words + 4, acc, sizeof(sums), cudaMemcpyDeviceToHost, s));
    if (log0 || sums0 || guess) {
    } else if (sums0b) {
      LR_TRY(launch_count_batch(reinterpret_cast<const unsigned long long *>(bitmap), in.k, hcount, s));
      LR_TRY(cudaMemcpyAsync(c->host_words + 1, hcount, 4, cudaMemcpyDeviceToHost, s));
    } else {
      LR_TRY(launch_count_heads(bitmap, (uint32_t)in.n, hcount, s));
      LR_TRY(cudaMemcpyAsync(c->host_words + 1, hcount, 4, cudaMemcpyDeviceToHost, s));
    }
    if (narrow && !acc_read && !guess) LR_TRY(cudaMemcpyAsync(c->host_words + 12, wflags, 4, cudaMemcpyDeviceToHost, s));
    if (!guess) LR_TRY(cudaStreamSynchronize(s));
    if (acc_read) {
      memcpy(sums, c->host_words + 4, sizeof(sums));
      if (!sumsv) c->host_words[1] = (uint32_t)sums[0];
      else if (sums[0] != c->host_words[1]) found = kErrNotList;
      one_head = in.n * (in.n - 1) / 2 - sums[1];
      one_list = (late_bitmap || sumsv) && sums[0] == 1 && c->host_words[1] == 1 && one_head < in.n;
      one_term = (uint32_t)sums[5];
      if (one_list && !log0) extras = t0ws = false;    // one terminal, one total: added at the end
      chased = guess && one_list;
    } else if (guess) {
      chased = c->host_words[2] != 0;
    }
    if (mostly_local(ask_local, sums, in.n)) {
      chased = false;
      prof.cancel();
      if (ask_local == kLocalSampled) LR_TRY(fetch());
      const lr_status cs = run_contracted(in, tuning, c, false, s);
      if (cs != LR_ERR_NOT_FOUND) return cs;
      if (ask_local == kLocalSampled) {        // not contracted after all: nothing is packed yet
        Inputs again = in;
        again.no_contract = 1;
        return run(again, tuning, s);
      }
      prof.begin(s, (int64_t)in.n);            // the same: carry on
    }
    if (narrow && narrow_mode(c->host_words[12]) == kNarrowNone) {      // (the flags, either way)
      kind0 = kRecKind16;
      chased = false;
      LR_TRY(pack(kind0, true, nullptr));
    }
    hb = chased ? guess_lists : std::max<uint64_t>(1, c->host_words[1]);
    p = make_plan(in.n, hb, u, rec16_0, in.rank_bytes, in.seed, grid, log0, extras, t0ws, spawn0, ord0, narrow);
  }
  if (!in.ws) {
    st = ensure_buffer(&c->var, &c->var_bytes, p.var_bytes, s);
    if (st != LR_OK) return st;
    var = (char *)c->var;
  } else if (in.ws_bytes < p.fixed_bytes + p.var_bytes) {
    LR_TRY(cudaStreamSynchronize(s));     // nothing else may still write the caller's memory
    return LR_ERR_CAPACITY;               // the lists need more workspace than was given
  }
  if (!chased) {
    prof.drop_from(marks_before);
    prof.record(PH_PREP);
  }
  prof.note(PH_PREP);

  uint32_t *hA = (uint32_t *)(var + p.off_hA);
  uint32_t *hB = (uint32_t *)(var + p.off_hB);
  uint32_t *hC = extras ? (uint32_t *)(var + p.off_hC) : hA;
  uint32_t *ns = (uint32_t *)(var + p.off_ns);
  const bool acc_heads = ((log0 || sums0) && !in.validate) || (sumsv && one_list);
  InitParams ip = init_params(p);
  ip.err = err;
  ip.err_bits = found;
  if (!chased)
    LR_TRY(launch_init(desc, ip, acc_heads ? acc : nullptr, kind0 == kRecKind8w ? wflags : nullptr, hA, ns,
                       hB, s));
  if (!in.ctx) { c->last_desc = desc; c->last_nlev = p.nlev; }
  if (p.spawn_cap) LR_TRY(cudaMemsetAsync(var + p.off_sctr, 0, p.spawn_zero, s));
  SpawnArgs spa;
  memset(&spa, 0, sizeof(spa));
  if (p.spawn_cap) {
    spa.ctr = (uint32_t *)(var + p.off_sctr);
    spa.cap = p.spawn_cap;
    spa.used = (uint32_t *)(var + p.off_sused);
    spa.cursor = (uint32_t *)(var + p.off_sctr + 16);
  }
  if (log0) {
    LR_TRY(cudaMemsetAsync(var + p.off_hdr, 0xFF, (size_t)p.total_chunks * 8, s));
    LR_TRY(cudaMemsetAsync(var + p.off_cur, 0, p.cur_bytes, s));
  }
  if ((log0 || sums0) && !one_list) {
    if (late_bitmap) LR_TRY(cudaMemsetAsync(bitmap, 0, bitmap_bytes, s));
    LR_TRY(launch_bitmap0(desc, in.succ, (uint32_t)in.n, bitmap, err, in.validate, s));
  } else if (sums0b && !chased)
    LR_TRY(launch_heads0_batch(desc, reinterpret_cast<unsigned long long *>(bitmap), in.offsets, in.k, hA,
                               p.hcap, work0, kind0, (uint32_t)in.n, bitmap, s));

  auto work_of = [&](int l) -> void * { return l == 0 ? work0 : (void *)(var + p.off_work[l]); };
  auto R_of = [&](int l) -> void * { return l == 0 ? (ranks_to_host ? in.h.rank : in.rank) : (void *)(var + p.off_R[l]); };
  // terminal ids: T_l of every element of level l (the caller's array, or
  // workspace, at level 0), tid_l of every terminal of level l >= 1
  uint32_t *T0 = extras ? (in.term ? in.term : (uint32_t *)(var + p.off_T0)) : nullptr;
  auto T_of = [&](int l) -> uint32_t * {
    if (!extras) return nullptr;
    return l == 0 ? T0 : (uint32_t *)(var + p.off_T[l]);
  };
  auto tid_of = [&](int l) -> uint32_t * {
    return (extras && l > 0) ? (uint32_t *)(var + p.off_tid[l]) : nullptr;
  };
  // head lists alternate between buffers; with extra outputs level 0's list
  // (hA) stays intact for the prefix pass
  auto head_list = [&](int l) -> uint32_t * { return l == 0 ? hA : ((l & 1) ? hB : hC); };
  const int L = p.nlev - 1;
  for (int l = 0; l < L; ++l) {
    const bool r16 = l > 0 || rec16_0;
    uint32_t *hin = head_list(l), *hout = head_list(l + 1);
    if (l > 0) {
      if (p.low[l] <= p.base) {
        LR_TRY(launch_jump(desc, l, work_of(l), r16, R_of(l), p.rank_bytes, p.cap[l], err, hin, tid_of(l),
                           T_of(l), nullptr, s));
        prof.mark(PH_BASE);
      }
    }
    const int kind = (l == 0 && log0) ? kRecKindSucc : l == 0 ? kind0 : kRecKind16;
    if (l > 0 || !(one_list || chased))
      LR_TRY(launch_heads(desc, l, p.nlev, bitmap, hin, (l == 0 && log0) ? (void *)in.succ : work_of(l),
                        kind, ns, hout, bcnt, err, p.base, p.hcap, s));
    const bool recorded = l == 0 && chased;
    prof.note(PH_SELECT);
    if (!recorded) prof.record(PH_SELECT);
    if (l == 0 && chased) {
      // (queued before the wait)
    } else if (l == 0 && log0)
      LR_TRY(launch_chase_log(desc, in.succ, work_of(1), ns, qctr, p.chase_grid, p.chase_block, err,
                              (uint32_t *)(var + p.off_log), (uint2 *)(var + p.off_hdr),
                              p.total_chunks, (uint32_t *)(fixed + p.off_logctr), s));
    else if (l == 0 && p.spawn_cap) {
      // spawning: reduced records at uncompacted ids, then compacted into level 1
      LR_TRY(launch_chase(desc, 0, work0, kind, var + p.off_sraw, ns, qctr, p.chase_grid, p.chase_block,
                          err, (int)u.xchg, nullptr, nullptr, &spa, nullptr, s));
      LR_TRY(launch_spawn_compact(desc, 0, p.nlev, spa.ctr, spa.cap, spa.used, (uint32_t *)(var + p.off_supre),
                                  var + p.off_sraw, work_of(1), p.raw_cap, p.base, err, s));
    } else {
      OrdArgs oa;
      memset(&oa, 0, sizeof(oa));
      if (p.ord0 && ord_used && (l == 0 || (u.ord >= 2 && 16ull * p.cap[l] > kOrdMinBytes))) {
        oa.ord = (uint32_t *)(var + p.off_ord);
        oa.cum = (uint32_t *)(var + p.off_cum);
        oa.bits = bitmap;        // the has-predecessor bitmap is free once level 0's heads are chosen
        oa.pf_lead = u.pf << 10;
        LR_TRY(launch_order(desc, l, p.cap[l], bcnt, &oa, hout, p.hcap, err, s));
      }
      LR_TRY(launch_chase(desc, l, work_of(l), kind, work_of(l + 1), ns,
                          qctr + (size_t)l * p.chase_grid, p.chase_grid, p.chase_block, err,
                          (int)u.xchg, tid_of(l), tid_of(l + 1), nullptr, oa.ord ? &oa : nullptr, s));
      if (l == 0 && both)
        LR_TRY(launch_chase(desc, 0, work0, kRecKind16, work_of(1), ns, qctr, p.chase_grid, p.chase_block, err,
                            (int)u.xchg, nullptr, nullptr, nullptr, oa.ord ? &oa : nullptr, s));
    }
    if (l == 0) prof.call.log0 = log0;
    prof.note(l == 0 ? PH_CHASE0 : PH_CHASE);
    if (!recorded) prof.record(l == 0 ? PH_CHASE0 : PH_CHASE);
  }
  LR_TRY(launch_jump(desc, L, work_of(L), true, R_of(L), p.rank_bytes, p.cap[L], err, head_list(L),
                     tid_of(L), T_of(L), nullptr, s));
  prof.mark(PH_BASE);
  for (int l = L - 1; l >= 0; --l) {
    if (l == 0 && log0)
      LR_TRY(launch_finalize_log(desc, (const uint32_t *)(var + p.off_log), (const uint2 *)(var + p.off_hdr),
                                 p.total_chunks, (const uint32_t *)(fixed + p.off_logctr), R_of(1),
                                 (uint2 *)(var + p.off_pairs),
                                 (uint2 *)(var + p.off_pairsB), (uint32_t *)(var + p.off_cur),
                                 (uint32_t *)(var + p.off_cur) + p.lg.na, p.lg, (uint32_t *)in.rank, err, s));
    else if (l == 0 && ptrs)
      LR_TRY(launch_finalize_ptrs(desc, work0, kind0, R_of(1), in.rptr, p.rank_bytes, p.cap[0],
                                  in.offsets, in.k, err, s));
    else if (l == 0 && p.spawn_cap) {
      LR_TRY(launch_spawn_scatter(desc, 0, R_of(1), var + p.off_srraw, p.rank_bytes, spa.used,
                                  (uint32_t *)(var + p.off_supre), p.raw_cap, s));
      LR_TRY(launch_finalize(desc, 0, work0, kind0, var + p.off_srraw, R_of(0), p.rank_bytes, p.cap[0],
                             err, nullptr, nullptr, nullptr, s, ranks_to_host));
    } else
      LR_TRY(launch_finalize(desc, l, work_of(l), l > 0 ? (int)kRecKind16 : kind0, R_of(l + 1), R_of(l),
                             p.rank_bytes, p.cap[l], err, T_of(l + 1), T_of(l), tid_of(l), s, l == 0 && ranks_to_host));
    if (l == 0 && both) {
      if (ptrs)
        LR_TRY(launch_finalize_ptrs(desc, work0, kRecKind16, R_of(1), in.rptr, p.rank_bytes, p.cap[0], in.offsets,
                                    in.k, err, s));
      else
        LR_TRY(launch_finalize(desc, 0, work0, kRecKind16, R_of(1), R_of(0), p.rank_bytes, p.cap[0], err, nullptr,
                               nullptr, nullptr, s, ranks_to_host));
    }
  }
  if (ranks_to_host) *in.h.ranks_out = true;
  if (outputs && !extras) {
    Perm P;                                    // the head is a ruler: its rank at level 1
    P.init((uint32_t)in.n, p.seed[0]);
    const uint32_t id = P.fwd((uint32_t)one_head);
    const uint32_t r = (uint32_t)((in.n + p.f_inv[0] - 1) / p.f_inv[0]);
    LR_TRY(launch_out_one((uint32_t)in.n, one_term, (const char *)R_of(1) + (size_t)p.rank_bytes * std::min(id, r),
                          in.term, in.rank, in.prefix, p.rank_bytes, in.incl, in.weight, in.wtype, s));
  }
  if (extras)
    LR_TRY(launch_outputs(desc, bitmap, hA, (uint32_t)in.n, T0, in.rank, in.prefix, p.rank_bytes,
                          in.incl, in.weight, in.wtype, in.offsets, in.k,
                          in.offsets != nullptr && in.term != nullptr, s));
  prof.mark(PH_FINAL);
  prof.end();
  return finish_call(c, err, in.sync, s);
}

lr_status run_fixed_scratch(const uint32_t *succ, int64_t n, int32_t *rank, void *scratch,
                            size_t scratch_bytes, Ctx *ctx, cudaStream_t s) {
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.succ = succ;
  in.rank = rank;
  in.rank_bytes = 4;
  in.n = (uint64_t)n;
  in.seed = 0x5eedull;
  in.sync = 1;
  in.ws = scratch;
  in.ws_bytes = scratch_bytes;
  in.ctx = ctx;
  in.count_in_ws = 1;
  // fixed settings: whether a valid list fits the scratch must not depend on
  // LR_TUNING or on what the autotuner stored in this process
  in.builtin_tuning = 1;
  return run(in, nullptr, s);
}

lr_status run_single(const uint32_t *succ, const void *weight, int wtype, void *rank, int rank_bytes,
                     int64_t n, uint64_t seed, cudaStream_t s) {
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.succ = succ;
  in.weight = weight;
  in.wtype = wtype;
  in.rank = rank;
  in.rank_bytes = rank_bytes;
  in.n = (uint64_t)n;
  in.seed = seed;
  in.sync = 1;
  return run(in, nullptr, s);
}

lr_status run_ptr_batch(const int64_t *offsets, int32_t k, int64_t n_total,
                        const uint32_t *const *sptr, const void *const *wptr, void *const *rptr,
                        int wtype, int rank_bytes, uint64_t seed, cudaStream_t s) {
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.n = (uint64_t)n_total;
  in.offsets = offsets;
  in.k = k;
  in.sptr = sptr;
  in.wptr = wptr;
  in.rptr = rptr;
  in.wtype = wtype;
  in.rank_bytes = rank_bytes;
  in.seed = seed;
  in.sync = 1;
  return run(in, nullptr, s);
}

lr_status status_from_bits(uint32_t bits) { return map_device_bits(bits); }

lr_status device_status(cudaStream_t s) {
  lr_status st;
  Ctx *c = get_ctx(s, &st);
  if (!c) return st;
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return from_cuda(e);
  const uint32_t bits = c->host_words[0];
  c->host_words[0] = 0;
  c->pending_status = false;
  return map_device_bits(bits);
}

}  // namespace lr

// ================================================================ C ABI
using namespace lr;

extern "C" {

void lr_opts_default(lr_opts *o) {
  if (!o) return;
  memset(o, 0, sizeof(*o));
  o->wtype = LR_NONE;
  o->rtype = LR_I32;
  o->seed = 0x5eedull;
}

const char *lr_version(void) { return "lr-gb300 0.1 (sparse ruling set, sm_103a)"; }

const char *lr_status_string(lr_status s) {
  switch (s) {
    case LR_OK: return "LR_OK";
    case LR_ERR_INVALID_ARGUMENT: return "LR_ERR_INVALID_ARGUMENT";
    case LR_ERR_OUT_OF_RANGE: return "LR_ERR_OUT_OF_RANGE";
    case LR_ERR_CYCLE: return "LR_ERR_CYCLE";
    case LR_ERR_NOT_A_LIST: return "LR_ERR_NOT_A_LIST";
    case LR_ERR_OUT_OF_MEMORY: return "LR_ERR_OUT_OF_MEMORY";
    case LR_ERR_BUDGET: return "LR_ERR_BUDGET";
    case LR_ERR_TIMEOUT: return "LR_ERR_TIMEOUT";
    case LR_ERR_CUDA: return "LR_ERR_CUDA";
    case LR_ERR_CAPACITY: return "LR_ERR_CAPACITY";
    case LR_ERR_NOT_FOUND: return "LR_ERR_NOT_FOUND";
    case LR_ERR_CANCELLED: return "LR_ERR_CANCELLED";
    case LR_ERR_CAPTURE: return "LR_ERR_CAPTURE";
    case LR_ERR_INTERNAL: return "LR_ERR_INTERNAL";
  }
  return "LR_ERR_UNKNOWN";
}

static lr_status check_types(const void *weight, lr_dtype wtype, lr_dtype rtype, int *wcode, int *rbytes) {
  if (rtype != LR_I32 && rtype != LR_I64) return LR_ERR_INVALID_ARGUMENT;
  if (wtype != LR_NONE && wtype != LR_I32 && wtype != LR_I64) return LR_ERR_INVALID_ARGUMENT;
  if ((wtype == LR_NONE) != (weight == nullptr)) return LR_ERR_INVALID_ARGUMENT;
  *wcode = (int)wtype;
  *rbytes = rtype == LR_I32 ? 4 : 8;
  return LR_OK;
}

static void set_outputs(Inputs &in, const lr_outputs *outs) {
  if (!outs) return;
  in.term = outs->term;
  in.prefix = outs->prefix;
  in.incl = outs->inclusive_tail != 0;
}

static lr_status rank_ex_impl(const uint32_t *succ, const void *weight, int64_t n, void *rank,
                              const lr_outputs *outs, const lr_opts *opts, lr_stream stream,
                              const HostBuffers *host = nullptr) {
  lr_opts d;
  if (!opts) { lr_opts_default(&d); if (weight) { d.wtype = LR_I64; d.rtype = LR_I64; } opts = &d; }
  if (n < 0 || n > LR_MAX_N) return LR_ERR_INVALID_ARGUMENT;
  if (n > 0 && (!succ || !rank)) return LR_ERR_INVALID_ARGUMENT;
  int wc, rb;
  lr_status st = check_types(n > 0 ? weight : (opts->wtype ? (const void *)1 : nullptr),
                             opts->wtype, opts->rtype, &wc, &rb);
  if (st != LR_OK) return st;
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.succ = succ;
  in.weight = weight;
  in.wtype = wc;
  in.rank = rank;
  in.rank_bytes = rb;
  in.n = (uint64_t)n;
  in.validate = opts->validate;
  in.seed = opts->seed;
  in.max_lists = opts->max_lists;
  in.sync = opts->sync;
  in.ws = opts->workspace;
  in.ws_bytes = opts->ws_bytes;
  if (host) in.h = *host;
  set_outputs(in, outs);
  return run(in, opts->tuning, (cudaStream_t)stream);
}

lr_status lr_rank_ex(const uint32_t *succ, const void *weight, int64_t n, void *rank,
                     const lr_opts *opts, lr_stream stream) {
  return rank_ex_impl(succ, weight, n, rank, nullptr, opts, stream);
}

lr_status lr_rank_outputs(const uint32_t *succ, const void *weight, int64_t n, void *rank,
                          const lr_outputs *outs, const lr_opts *opts, lr_stream stream) {
  return rank_ex_impl(succ, weight, n, rank, outs, opts, stream);
}

lr_status lr_rank(const uint32_t *succ, const void *weight, int64_t n, void *rank, lr_stream stream) {
  lr_opts o;
  lr_opts_default(&o);
  if (weight) { o.wtype = LR_I64; o.rtype = LR_I64; }
  else if (n >= ((int64_t)1 << 31)) return LR_ERR_INVALID_ARGUMENT;  // int32 ranks
  return lr_rank_ex(succ, weight, n, rank, &o, stream);
}

// The element total of a batch: n_total when given (> 0), else offsets[k]
// read back from the device (one wait on the stream).
static lr_status batch_total(const int64_t *offsets, int32_t k, int64_t n_total, cudaStream_t s, int64_t *n) {
  if (n_total > 0) {
    *n = n_total;
    return LR_OK;
  }
  if (stream_capturing(s)) return LR_ERR_CAPTURE;
  lr_status st;
  Ctx *c = get_ctx(s, &st);
  if (!c) return st;
  int64_t *h = (int64_t *)(c->host_words + 8);
  cudaError_t e = cudaMemcpyAsync(h, offsets + k, 8, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return from_cuda(e);
  *n = *h;
  return LR_OK;
}

static lr_status rank_batch_impl(const int64_t *offsets, const uint32_t *succ, const void *weight,
                                 void *rank, int32_t k, const lr_outputs *outs, const lr_opts *opts,
                                 lr_stream stream) {
  lr_opts d;
  if (!opts) { lr_opts_default(&d); if (weight) { d.wtype = LR_I64; d.rtype = LR_I64; } opts = &d; }
  if (k < 0 || (k > 0 && !offsets)) return LR_ERR_INVALID_ARGUMENT;
  if (k == 0) return LR_OK;
  cudaStream_t s = (cudaStream_t)stream;
  int64_t n = 0;
  const lr_status nst = batch_total(offsets, k, opts->n_total, s, &n);
  if (nst != LR_OK) return nst;
  if (n < 0 || n > LR_MAX_N) return LR_ERR_INVALID_ARGUMENT;
  if (n > 0 && (!succ || !rank)) return LR_ERR_INVALID_ARGUMENT;
  int wc, rb;
  lr_status st = check_types(n > 0 ? weight : (opts->wtype ? (const void *)1 : nullptr),
                             opts->wtype, opts->rtype, &wc, &rb);
  if (st != LR_OK) return st;
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.succ = succ;
  in.weight = weight;
  in.wtype = wc;
  in.rank = rank;
  in.rank_bytes = rb;
  in.n = (uint64_t)n;
  in.offsets = offsets;
  in.k = k;
  in.validate = opts->validate;
  in.seed = opts->seed;
  in.max_lists = opts->max_lists;
  in.sync = opts->sync;
  in.ws = opts->workspace;
  in.ws_bytes = opts->ws_bytes;
  set_outputs(in, outs);
  return run(in, opts->tuning, s);
}

lr_status lr_rank_batch_ex(const int64_t *offsets, const uint32_t *succ, const void *weight,
                           void *rank, int32_t k, const lr_opts *opts, lr_stream stream) {
  return rank_batch_impl(offsets, succ, weight, rank, k, nullptr, opts, stream);
}

lr_status lr_rank_batch_outputs(const int64_t *offsets, const uint32_t *succ, const void *weight,
                                void *rank, int32_t k, const lr_outputs *outs, const lr_opts *opts,
                                lr_stream stream) {
  return rank_batch_impl(offsets, succ, weight, rank, k, outs, opts, stream);
}

lr_status lr_rank_batch(const int64_t *offsets, const uint32_t *succ, const void *weight,
                        void *rank, int32_t k, lr_stream stream) {
  lr_opts o;
  lr_opts_default(&o);
  if (weight) { o.wtype = LR_I64; o.rtype = LR_I64; }
  return lr_rank_batch_ex(offsets, succ, weight, rank, k, &o, stream);
}

lr_status lr_rank_batch_ptrs(const int64_t *offsets, const uint32_t *const *succ_ptrs,
                             const void *const *weight_ptrs, void *const *rank_ptrs, int32_t k,
                             const lr_opts *opts, lr_stream stream) {
  lr_opts d;
  if (!opts) {
    lr_opts_default(&d);
    if (weight_ptrs) { d.wtype = LR_I64; d.rtype = LR_I64; }
    opts = &d;
  }
  if (k < 0 || (k > 0 && (!offsets || !succ_ptrs || !rank_ptrs))) return LR_ERR_INVALID_ARGUMENT;
  if (k == 0) return LR_OK;
  if (opts->workspace) return LR_ERR_INVALID_ARGUMENT;   // the pointer form keeps its own workspace
  cudaStream_t s = (cudaStream_t)stream;
  // the kernels index the caller's buffers through the offset table, so it is
  // read back and checked here before any of them runs (one wait)
  if (stream_capturing(s)) return LR_ERR_CAPTURE;
  std::vector<int64_t> h((size_t)k + 1);
  cudaError_t e = cudaMemcpyAsync(h.data(), offsets, 8 * ((size_t)k + 1), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return from_cuda(e);
  if (h[0] != 0) return LR_ERR_INVALID_ARGUMENT;
  for (int32_t j = 0; j < k; ++j)
    if (h[j + 1] < h[j]) return LR_ERR_INVALID_ARGUMENT;
  const int64_t n = h[k];
  if (n > LR_MAX_N || (opts->n_total > 0 && opts->n_total != n)) return LR_ERR_INVALID_ARGUMENT;
  int wc, rb;
  lr_status st = check_types(weight_ptrs, opts->wtype, opts->rtype, &wc, &rb);
  if (st != LR_OK) return st;
  if (n == 0) return LR_OK;
  Inputs in;
  memset(&in, 0, sizeof(in));
  in.sptr = succ_ptrs;
  in.wptr = weight_ptrs;
  in.rptr = rank_ptrs;
  in.wtype = wc;
  in.rank_bytes = rb;
  in.n = (uint64_t)n;
  in.offsets = offsets;
  in.k = k;
  in.validate = opts->validate;
  in.seed = opts->seed;
  in.max_lists = opts->max_lists;
  in.sync = opts->sync;
  return run(in, opts->tuning, s);
}

// Enqueue copy-in, ranking and copy-out on `stream` through the stream's own
// device staging buffers; `sync` waits and returns the final status.
static lr_status rank_host_impl(const uint32_t *succ_host, const void *weight_host, int64_t n,
                                void *rank_host, const lr_opts *opts, lr_stream stream, bool sync);

lr_status lr_rank_host(const uint32_t *succ_host, const void *weight_host, int64_t n,
                       void *rank_host, const lr_opts *opts, lr_stream stream) {
  return rank_host_impl(succ_host, weight_host, n, rank_host, opts, stream, true);
}

lr_status lr_rank_host_async(const uint32_t *succ_host, const void *weight_host, int64_t n,
                             void *rank_host, const lr_opts *opts, lr_stream stream) {
  return rank_host_impl(succ_host, weight_host, n, rank_host, opts, stream, false);
}

// The pinned piece of host memory around q (pinned_view).
static bool pinned_piece(const void *q, PinnedPiece &piece) {
  using Ask = CUresult (*)(void *, CUpointer_attribute, CUdeviceptr);
  static const Ask ask = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult got;
    if (cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &f, 12000, cudaEnableDefault, &got) != cudaSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return reinterpret_cast<Ask>(f);
  }();
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, q) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (!ask || a.type != cudaMemoryTypeHost || !a.devicePointer) return false;
  CUdeviceptr start = 0;
  size_t size = 0;
  const CUdeviceptr d = reinterpret_cast<CUdeviceptr>(a.devicePointer);
  if (ask(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, d) != CUDA_SUCCESS ||
      ask(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, d) != CUDA_SUCCESS || d < start || d - start >= size)
    return false;
  piece.device = a.devicePointer;
  piece.left = size - (size_t)(d - start);
  return true;
}

// What the device calls a host buffer that it can read and write in place
// (null: not pinned throughout, or not aligned to its elements, which a copy
// may be).
static void *device_view(const void *p, size_t elems, size_t bytes) {
  return (uintptr_t)p % bytes ? nullptr : pinned_view(p, elems * bytes, pinned_piece);
}

static lr_status rank_host_impl(const uint32_t *succ_host, const void *weight_host, int64_t n,
                                void *rank_host, const lr_opts *opts, lr_stream stream, bool sync) {
  lr_opts d;
  if (!opts) { lr_opts_default(&d); if (weight_host) { d.wtype = LR_I64; d.rtype = LR_I64; } opts = &d; }
  if (n < 0 || n > LR_MAX_N) return LR_ERR_INVALID_ARGUMENT;
  if (n == 0) return LR_OK;
  if (!succ_host || !rank_host) return LR_ERR_INVALID_ARGUMENT;
  int wc, rb;
  lr_status st = check_types(weight_host, opts->wtype, opts->rtype, &wc, &rb);
  if (st != LR_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  if (stream_capturing(s)) return LR_ERR_CAPTURE;
  Ctx *c = get_ctx(s, &st);
  if (!c) return st;
  const size_t wb = wc == 0 ? 0 : (wc == 1 ? 4 : 8);
  const size_t bs = align_up(4 * (size_t)n), bw = align_up(wb * (size_t)n), br = align_up((size_t)rb * n);
  st = ensure_buffer(&c->hostpath, &c->hostpath_bytes, bs + bw + br, s);
  if (st != LR_OK) return st;
  char *b = (char *)c->hostpath;
  uint32_t *dsucc = (uint32_t *)b;
  void *dw = wb ? (void *)(b + bs) : nullptr;
  void *drank = b + bs + bw;
  // A call that waits reads and writes pinned buffers in place: a copy before
  // and after it would each take the link's time, in which the first and the
  // last pass are done on the way (4 million elements: 371 us with the copies, 340
  // without).  Streams that overlap calls keep the copies, which need no SM.
  HostBuffers h;
  memset(&h, 0, sizeof(h));
  bool ranks_out = false;
  h.ranks_out = &ranks_out;
  if (sync) {
    h.succ = (const uint32_t *)device_view(succ_host, (size_t)n, 4);
    if (wb) h.weight = device_view(weight_host, (size_t)n, wb);
    if (wb && !h.weight) h.succ = nullptr;
    h.rank = device_view(rank_host, (size_t)n, (size_t)rb);
  }
  if (!h.succ) {
    LR_TRY(cudaMemcpyAsync(dsucc, succ_host, 4 * (size_t)n, cudaMemcpyHostToDevice, s));
    if (wb) LR_TRY(cudaMemcpyAsync(dw, weight_host, wb * (size_t)n, cudaMemcpyHostToDevice, s));
  }
  lr_opts o = *opts;
  o.sync = 0;
  st = rank_ex_impl(dsucc, dw, n, drank, nullptr, &o, stream, &h);
  if (st != LR_OK) return st;
  if (!ranks_out) LR_TRY(cudaMemcpyAsync(rank_host, drank, (size_t)rb * n, cudaMemcpyDeviceToHost, s));
  return sync ? device_status(s) : LR_OK;
}

}  // extern "C"

namespace lr {
// Bytes of workspace for a call of exactly this size.
static size_t workspace_exact(int64_t n_total, int32_t k, const lr_outputs *outs, const lr_opts *opts, const Tuning &u) {
  // The chase grid depends on the device; size for a generous upper bound so
  // the answer needs no GPU: 256 SMs x 16 CTAs.
  if (u.algo == LR_ALGO_WYLLIE) {
    Inputs in;
    memset(&in, 0, sizeof(in));
    in.wtype = opts->wtype != LR_NONE;
    in.rank_bytes = opts->rtype == LR_I64 ? 8 : 4;
    return wyllie_plan((uint64_t)n_total, wyllie_w16(in)).bytes;
  }
  const uint64_t h = opts->max_lists > 0 ? (uint64_t)opts->max_lists : (uint64_t)n_total;
  const bool extras = outs && (outs->term || outs->prefix || outs->inclusive_tail);
  const bool log0 = use_log0(u, (uint64_t)n_total, opts->wtype != LR_NONE, opts->rtype == LR_I64 ? 8 : 4,
                             extras, k != 0);
  const bool spawn0 = u.spawn != 0 && u.xchg != 0 && !log0 && !extras;
  const bool ord0 = use_ord0(u, (uint64_t)n_total, opts->wtype != LR_NONE, log0, spawn0, extras, k != 0);
  Plan p = make_plan((uint64_t)n_total, h, u,
                     opts->wtype != LR_NONE || (extras && (uint64_t)n_total <= u.base0),
                     opts->rtype == LR_I64 ? 8 : 4, opts->seed, 256 * 16, log0, extras,
                     extras && !outs->term, spawn0, ord0,
                     use_narrow(u, (uint64_t)n_total, opts->wtype != LR_NONE, spawn0, extras, true));
  return p.fixed_bytes + p.var_bytes;
}

// Sizes from which on a call may need less workspace than just below them:
// with n growing, the need grows except where a rule on n gives fewer rulers,
// fewer bytes an element or another form of level 0.  (Fewer rulers below
// level 0: workspace_rulers_end; the log form's partition: log_geometry_step.
// Powers of two: tuned entries are kept by them, and the partition's buckets
// widen after them.)
template <class F>
static void workspace_steps(uint32_t base0, F &&step) {
  for (const F0Step &t : kF0Steps) step(t.below);
  step(1ll << 23);                               // default_f0_inv_batch
  step(kOrdSpacingFrom);
  step((int64_t)base0 + 1);                      // the base case: terminal ids make its records larger
  step((int64_t)kLogAutoMin);                    // the log form at level 0, and its end
  step((1ll << 30) + 1);
  step(0x7FFFFF01ll);                            // 8-byte weighted records (room for cut segments) end
  for (int b = 1; b < 33; ++b) { step(1ll << b); step((1ll << b) + 1); }
}

// The largest size with ruler fraction f0_inv for which default_f_inv takes
// the larger share of rulers below level 0.
static int64_t workspace_rulers_end(uint32_t f0_inv) { return (int64_t)f0_inv * (4ll * kJumpMax + 1) - 1; }
}  // namespace lr

extern "C" {

size_t lr_workspace_size(int64_t n_total, int32_t k, const lr_opts *opts) {
  return lr_workspace_size_outputs(n_total, k, nullptr, opts);
}

size_t lr_workspace_size_outputs(int64_t n_total, int32_t k, const lr_outputs *outs,
                                 const lr_opts *opts) {
  lr_opts d;
  if (!opts) { lr_opts_default(&d); opts = &d; }
  if (n_total <= 0) return 0;
  const bool weighted = opts->wtype != LR_NONE;
  const uint32_t base0 = resolve_tuning(opts->tuning, n_total, weighted, k > 0).base0;
  // enough for every size up to n_total: for it, and for the last size of
  // each stretch below it over which the need grows (at any ruler fraction an
  // element takes 8 bytes at least and 64 at most, so an eighth of n_total
  // never needs more than n_total)
  size_t most = 0;
  auto at = [&](int64_t m) {
    const Tuning v = resolve_tuning(opts->tuning, m, weighted, k > 0);
    most = std::max(most, workspace_exact(m, k, outs, opts, v));
    return v.f0_inv;
  };
  auto consider = [&](int64_t m) {
    if (m <= n_total / 8 || m > n_total) return;
    const uint32_t f0 = at(m);
    const int64_t rulers = workspace_rulers_end(f0), part = log_geometry_step(m);
    if (rulers < m) at(rulers);
    if (part > 0) at(part);
  };
  consider(n_total);
  workspace_steps(base0, [&](int64_t from) { if (from <= n_total) consider(from - 1); });
  return most;
}

lr_status lr_get_device_status(lr_stream stream) { return device_status((cudaStream_t)stream); }

int32_t lr_level_sizes(lr_stream stream, int64_t *sizes, int32_t max_levels) {
  lr_status st;
  Ctx *c = get_ctx((cudaStream_t)stream, &st);
  if (!c || !c->last_desc || c->last_nlev <= 0) return 0;
  LevelDesc d[kMaxLevels + 1];
  if (cudaMemcpyAsync(d, c->last_desc, sizeof(LevelDesc) * c->last_nlev, cudaMemcpyDeviceToHost,
                      (cudaStream_t)stream) != cudaSuccess ||
      cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
    return -1;
  int32_t used = 0;
  for (int l = 0; l < c->last_nlev; ++l) {
    if (d[l].mode == kModeOff) break;
    if (sizes && used < max_levels) sizes[used] = d[l].n;
    ++used;
  }
  return used;
}

lr_status lr_profile_enable(int32_t on) {
  std::lock_guard<std::mutex> g(g_mu);
  g_prof = on != 0;
  return LR_OK;
}

lr_status lr_profile_read(lr_profile *out, int32_t reset) {
  std::vector<ProfCall> pend;
  {
    std::lock_guard<std::mutex> g(g_mu);
    pend.swap(g_prof_pending);
  }
  for (auto &call : pend) {
    for (size_t i = 1; i < call.marks.size(); ++i) {
      float ms = 0.f;
      cudaEventSynchronize(call.marks[i].ev);
      cudaEventElapsedTime(&ms, call.marks[i - 1].ev, call.marks[i].ev);
      switch (call.marks[i].phase) {
        case PH_PREP: g_prof_acc.ms_prep += ms; break;
        case PH_SELECT: g_prof_acc.ms_select += ms; break;
        case PH_CHASE0:
          g_prof_acc.ms_chase0 += ms;
          g_prof_acc.chase0_launches += 1;
          g_prof_acc.chase0_log_launches += call.log0 ? 1 : 0;
          break;
        case PH_CHASE: g_prof_acc.ms_chase_rest += ms; break;
        case PH_BASE: g_prof_acc.ms_base += ms; break;
        case PH_FINAL: g_prof_acc.ms_finalize += ms; break;
      }
    }
    for (auto &m : call.marks) cudaEventDestroy(m.ev);
    g_prof_acc.calls += 1;
    g_prof_acc.kernel_launches += call.launches;
    g_prof_acc.elements += call.n;
  }
  if (out) *out = g_prof_acc;
  if (reset) memset(&g_prof_acc, 0, sizeof(g_prof_acc));
  return LR_OK;
}

int64_t lr_kernel_launch_count(void) { return launch_count(); }

}  // extern "C"
