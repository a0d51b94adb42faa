// KADABRA adaptive sampling loop for GB300 (sm_103a): kernels, host runtime
// and C ABI.
//
// Paper: Borassi & Natale, "KADABRA is an ADaptive Algorithm for Betweenness
// via Random Approximation".  The method (Alg. 1) samples shortest paths
// between uniform node pairs and stops once every node's estimate b~(v) is
// within lambda with probability 1-delta:
//   * k_sample      -- one sample per CTA (Sec. 4; 128 to 1,024 threads by
//                      tier and layout): (s,t) draw, balanced
//                      bidirectional BFS with exact uint64
//                      sigma, candidate-edge choice proportional to
//                      sigma_sv*sigma_wt, backtracking to a uniform shortest
//                      path, hit counters (Alg. 1).
//   * k_sample_warp -- the same sample by one warp, for small searches.
//   * k_check_tab   -- the all-nodes stop test: f and g of Thm. 2 in FP64,
//                      rule f <= lambda and g <= lambda; k_topk_* the
//                      top-k test (Sec. 5, Alg. 3).
//   * host code     -- omega (Alg. 1), computeDelta (Alg. 2, App. D), the
//                      batch / test schedule (host rounds or a CUDA graph
//                      loop), VD bound (condensation into strongly
//                      connected components), CSR validation, the autotuner,
//                      batched runs and the serving engine.
//
// Sampler design (GB300-first, not the paper's CPU design):
//   * A persistent grid, sized to the SMs, pulls sample indices from a device
//     counter; the counter-based Philox4x32-10 RNG keyed by (seed, sample
//     index) makes results independent of the schedule, and hit counts are
//     integer atomics.
//   * Both searches' visited sets share one open-addressing hash table in
//     shared memory, one packed 64-bit word per node (node | side | depth |
//     sigma); level lists hold 16-bit hash positions (the node id is in the
//     hash word).  Four CTAs of 256 threads fit per SM in the default layout,
//     five of 192 and seven of 128 in the smaller ones, one of 1,024 in tier B.
//   * Every level runs pass 1 (touch test against the other search; most
//     arcs lie in the touching level, which only reads the table, and a bit
//     filter of the other side's frontier rejects most heads before the
//     probe), and only a level that does not touch runs pass 2 (first
//     discoverers insert with a CAS, every discoverer adds its sigma
//     atomically).
//   * The two backtracking walks (v -> s, w -> t) take disjoint Philox
//     blocks, so two warps walk them at the same time.
//   * Each warp scans a contiguous slice of the level's flattened arc range:
//     pass 1 with 32 * TOUCH_DEPTH arcs in flight, pass 2 in windows of 32
//     arcs, the next one's loads issued before the current one is processed.
//     For graphs beyond the L2, pass 1 searches long rows instead.
//     Candidate edges are chosen in (x, y) order without a sort (quadratic
//     ranking or a weighted radix selection).
//   * The kernel is short of issue slots and instruction fetch, not of
//     bandwidth: loops of the sampler are not unrolled unless it says so
//     (130 KB of code against 72 KB: the Chung-Lu graph's batch 4.50 -> 3.87
//     ms), and what one thread does while the others wait is kept short.
//   * A sample that outgrows its table moves on to bigger tables (tier B in
//     shared memory, then global-memory tiers M and L) with identical
//     results.
//
// Sections: constants, Philox, tables, parameters, block helpers, one sample
// (tiers S and B), tier W, stop test, top-k stop test, graph checks and VD,
// host side (omega, computeDelta, autotuner, device-driven loop, Alg. 1
// runner, top-k runner), serving, the sampler without device allocation, C
// ABI.

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <deque>
#include <memory>
#include <thread>
#include <type_traits>
#include <cstdint>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/kadabra.h"

namespace {

// ============================================================== constants
// Tuning constants (overridable at build time with -D for sweeps).
#ifndef KD_NT
#define KD_NT 256
#endif
#ifndef KD_U
#define KD_U 1
#endif
#ifndef KD_FAST_HLOG
#define KD_FAST_HLOG 12
#endif
#ifndef KD_MIN_BLOCKS
#define KD_MIN_BLOCKS 4
#endif
#ifndef KD_NT_BIG
#define KD_NT_BIG 1024
#endif
// Warps per sampler CTA.  Tiers S and L: 8.
// Tier B (with M): 32 on one CTA per SM with 16,384 slots, since its samples are
// few and large, so that a sample's latency counts.  Its launch per batch,
// against 8 warps on two CTAs with 8,192 slots: ER 3.4 M nodes (1,100 samples)
// 0.83 -> 0.25 ms, R-MAT scale 24 (65,536) 2.28 -> 1.22 ms.
// The compact tier-S layout: 6, which leaves five CTAs per SM 64 registers a
// thread; with 8 warps (48 registers) it spilled: 65,536 samples on the
// Chung-Lu graph of 10^6 nodes 3.45 -> 2.97 ms.
// The small tier-S layout, the compact one's place on graphs of few nodes: 4,
// with 2048 slots and seven CTAs per SM, so that a batch of 1,000 samples runs
// at once and a sample's barriers join fewer warps.  The line: runs at K near
// 1,000 with the compact layout and with it, ER of 2,000 nodes 1.02 -> 0.91 ms,
// of 8,000 1.14 -> 1.01, of 32,000 1.28 -> 1.28, of 3.4 M 7.9 -> 8.4.  On dense
// graphs of 4,000 to 16,000 nodes (mean degree 40 to 800) the compact layout was
// at most 2 % ahead of the better of the small and the default one.
constexpr int NW_S = KD_NT / 32;
constexpr int NW_CMP = 6;
constexpr int NW_TINY = 4;
constexpr int TINY_NODES = 16384;  // largest graph whose launches take it
constexpr int NW_BIG = KD_NT_BIG / 32;
constexpr int U = KD_U;            // independent items per thread per step (memory-level parallelism)
// Tiers of per-sample tables.  A sample starts in a small shared-memory
// table (tier S, main launch, four or five CTAs per SM; optionally tier W,
// one warp per sample, before it).  If it outgrows it, it is queued for a
// second launch with one CTA per SM and a large shared-memory table (tier
// B); beyond that the same CTA retries it on medium global tables (tier M),
// and beyond those it is queued for a last launch with n-sized global tables
// (tier L).  Every tier gives the same result.
constexpr int FAST_HLOG = KD_FAST_HLOG;        // tier S: 2^FAST_HLOG hash slots
// tier B: 2^KD_BIG_EXTRA times tier S's slots
#ifndef KD_BIG_EXTRA
#define KD_BIG_EXTRA 2
#endif
constexpr int BIG_HLOG = FAST_HLOG + KD_BIG_EXTRA;
#ifndef KD_FAST_MAXD
#define KD_FAST_MAXD 126
#endif
constexpr int FAST_MAXD = KD_FAST_MAXD;  // levels per side in shared memory (at most 126: the packed entry's dist field)
constexpr int MED_HLOG = 16;       // tier M, global memory per CTA: 65536 hash slots
constexpr int MED_LCAP = 32768;    //   level lists: 32768 nodes
constexpr int MED_MAXD = 1022;     //   levels per side
constexpr int GM_MAXD = 65534;     // tier L, global memory, hash >= 2n slots, lists of n
constexpr int PI_SEGS = 16;        // a sample's candidate edges: PI_SEGS * pcap entries in global memory,
constexpr int FAST_PCAP = 2048;    //   pcap in tiers S, B and M
constexpr int QUAD_PICK_MAX = 256;  // global-memory tiers: candidate sets ranked quadratically up to this size
constexpr size_t RADIX_HIST = 256 * (sizeof(unsigned long long) + sizeof(unsigned));  // larger sets: the selection's histogram
constexpr unsigned long long EMPTY = ~0ull;
constexpr unsigned FULL = 0xFFFFFFFFu;

// sample flags
constexpr int F_CAP = 1;       // a capacity bound was hit
constexpr int F_SIGMA = 2;     // sigma overflowed uint64
constexpr int F_INTERNAL = 4;  // an invariant failed
// a level's failures, kept apart from the sample's flags until the level is
// known not to touch
constexpr int LF_SIGMA = 1;        // a sigma overflowed uint64
constexpr int LF_CAP = 2;          // the lists, the table or a packed sigma ran out of room
constexpr int LF_TOUCH_SIGMA = 4;  // a candidate edge's weight overflowed uint64

// ============================================================== Philox
// Philox4x32-10, Salmon, Moraes, Dror, Shaw (SC'11): ten rounds of two
// 32x32 multiplications (counter words 0 and 2) whose high halves are
// xor-ed into the other words with the round key; Weyl key schedule.
__device__ __forceinline__ uint4 philox(uint32_t k0, uint32_t k1, uint4 x) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * x.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, x.x);
    const uint32_t lo1 = 0xCD9E8D57u * x.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, x.z);
    x = make_uint4(hi1 ^ x.y ^ k0, lo1, hi0 ^ x.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return x;
}

__device__ __forceinline__ uint4 draw(uint64_t seed, uint32_t domain, uint64_t idx, uint32_t j) {
  return philox((uint32_t)seed, (uint32_t)(seed >> 32),
                make_uint4((uint32_t)idx, (uint32_t)(idx >> 32), j, domain));
}

// the blocks beyond a sample's first 32 (long paths only): not inlined, the
// sampler's code is long for the instruction caches
__device__ __noinline__ uint4 draw_late(uint64_t seed, uint32_t domain, uint64_t idx, uint32_t j) {
  return draw(seed, domain, idx, j);
}

// the ordered pair s != t of a sample's block 0
__device__ __forceinline__ void draw_pair(uint4 b, int32_t n, int* s, int* t) {
  const uint64_t u = (uint64_t)b.x | ((uint64_t)b.y << 32);
  const uint64_t u2 = (uint64_t)b.z | ((uint64_t)b.w << 32);
  *s = (int)__umul64hi(u, (uint64_t)n);
  const int tp = (int)__umul64hi(u2, (uint64_t)(n - 1));
  *t = tp + (tp >= *s ? 1 : 0);
}

// floor(U * S / 2^128) for the 128-bit block U (x least significant)
__device__ __forceinline__ uint64_t below128(uint4 b, uint64_t S) {
  const uint64_t lo = (uint64_t)b.x | ((uint64_t)b.y << 32);
  const uint64_t hi = (uint64_t)b.z | ((uint64_t)b.w << 32);
  const uint64_t carry_in = __umul64hi(lo, S);
  const uint64_t hl = hi * S;
  const uint64_t hh = __umul64hi(hi, S);
  const uint64_t sum = hl + carry_in;
  return hh + (sum < hl ? 1ull : 0ull);
}

// ============================================================== checked build
// With KADABRA_CHECKED defined, the sampler checks the index of every list,
// frontier-array, level-bound, adjacency and hit-counter access.  A failing
// check records (site << 40 | index) in g_checked once, redirects the access
// to index 0 (so nothing outside the arrays is touched), and the sample then
// fails with KADABRA_ERR_INTERNAL, whose message names the site and index.
// It also delays warps where several work at once between two barriers.
// Without the flag the checks compile to nothing.
#ifdef KADABRA_CHECKED
__device__ unsigned long long g_checked;
__device__ __forceinline__ int64_t kchk(int64_t i, int64_t bound, int site) {
  if (i >= 0 && i < bound) return i;
  atomicCAS(&g_checked, 0ull, ((unsigned long long)site << 40) | ((unsigned long long)i & ((1ull << 40) - 1)));
  return 0;
}
#define KIDX(i, bound, site) ((std::decay_t<decltype(i)>)kchk((int64_t)(i), (int64_t)(bound), (site)))
// holds the warps for which `late` is true back by some microseconds, so that
// a value they read without a barrier is seen to change under them
#define KSTAGGER(late)             \
  do {                             \
    if (late) __nanosleep(20000u); \
  } while (0)
#else
#define KIDX(i, bound, site) (i)
#define KSTAGGER(late)
#endif

// ============================================================== tables
struct alignas(16) PiEntry {
  int32_t x, y;          // x on the expanding side, y the scanned neighbour
  unsigned long long w;  // sigma_x * sigma_y (exact; overflow flagged)
};

// Per-sample state.  The hash maps a visited node to (side, dist) in hkv
// and keeps its shortest-path count at the same position in hsig; the
// level lists hold, level after level, each node and the position of its
// hash entry; lvl holds each side's level bounds in the lists.
struct Tables {
  unsigned long long* hkv;  // (node << 32) | (side << 31 | dist), EMPTY = free
  unsigned long long* hsig; // sigma of the node at the same position
  uint32_t hmask;
  int hlog;
  int32_t* lnode;           // level lists: node ids (global-memory tiers; null in the packed tiers)
  uint32_t* lpos;           // level lists: hash positions (global-memory tiers)
  uint16_t* lpos16;         //   the same, 16 bits, in the shared-memory tiers (2^HLOG <= 2^16 slots)
  int2* pr;                 // frontier: {degree prefix, row start}; frcap+1 entries
  int lcap;
  int frcap;                // frontier nodes per scan segment (the frontier array's capacity)
  uint32_t* bits;           // filter of the other side's frontier (shared-memory tiers), else null
  int fwords, fshift;       //   its 32-bit words and 32 - log2(its bits)
  struct LongRows* lr;      // long rows of the segment (shared memory; null in the compact layout)
  int* lvl;                 // [side][lo|hi][maxd+2]
  int maxd;
  PiEntry* pi;              // candidate edges beyond shared memory: PI_SEGS * pcap entries
  int pcap;
};

__device__ __forceinline__ int& lvl_lo(const Tables& T, int side, int d) {
  return T.lvl[KIDX((2 * side) * (T.maxd + 2) + d, 4 * (T.maxd + 2), 1)];
}
__device__ __forceinline__ int& lvl_hi(const Tables& T, int side, int d) {
  return T.lvl[KIDX((2 * side + 1) * (T.maxd + 2) + d, 4 * (T.maxd + 2), 2)];
}

// list entry i's hash position (16-bit in the shared-memory tiers: PK)
template <bool PK>
__device__ __forceinline__ uint32_t lpos_get(const Tables& T, int i) {
  return PK ? (uint32_t)T.lpos16[KIDX(i, T.lcap, 3)] : T.lpos[KIDX(i, T.lcap, 3)];
}
// list entry i's node: the packed tiers keep no id list and read it from the
// entry's hash word (its high half never changes once published)
template <bool PK>
__device__ __forceinline__ int32_t list_node(const Tables& T, int i) {
  if (PK) return (int32_t)(T.hkv[KIDX((uint32_t)T.lpos16[KIDX(i, T.lcap, 5)], T.hmask + 1u, 6)] >> 32);
  return T.lnode[KIDX(i, T.lcap, 5)];
}
template <bool PK>
__device__ __forceinline__ void lpos_set(const Tables& T, int i, uint32_t pos) {
  if (PK)
    T.lpos16[KIDX(i, T.lcap, 4)] = (uint16_t)pos;
  else
    T.lpos[KIDX(i, T.lcap, 4)] = pos;
}

__device__ __forceinline__ uint32_t pack_val(int side, int dist) { return ((uint32_t)side << 31) | (uint32_t)dist; }
__device__ __forceinline__ int val_side(uint32_t v) { return (int)(v >> 31); }

// Two entry formats.  Split (tiers M, L): the hkv word is
// node << 32 | side << 31 | dist and sigma sits in hsig at the same
// position.  Packed (tier S): one word node << 32 | side << 31 | dist << 24 |
// sigma, with dist < 128 and sigma < 2^24; a sigma that would not fit sends
// the sample on to the split tiers, so results do not depend on the format.
constexpr unsigned long long PK_SIG_MASK = (1ull << 24) - 1;

template <bool PK>
__device__ __forceinline__ uint32_t ent_val(unsigned long long w) {
  if (PK) {
    const uint32_t lo = (uint32_t)w;
    return (lo & 0x80000000u) | ((lo >> 24) & 0x7Fu);
  }
  return (uint32_t)w;
}

template <bool PK>
__device__ __forceinline__ unsigned long long ent_sig(const Tables& T, unsigned long long w, uint32_t pos) {
  return PK ? (w & PK_SIG_MASK) : T.hsig[pos];
}

// the word a first discoverer publishes (packed: with its sigma included)
template <bool PK>
__device__ __forceinline__ unsigned long long ent_word(int32_t node, uint32_t val, unsigned long long sig0) {
  const unsigned long long hi = (unsigned long long)(uint32_t)node << 32;
  if (PK) return hi | (val & 0x80000000u) | ((unsigned long long)(val & 0x7Fu) << 24) | sig0;
  return hi | val;
}

// adds to a node's sigma; returns false if the sum no longer fits the format
template <bool PK>
__device__ __forceinline__ bool ent_add(const Tables& T, uint32_t pos, unsigned long long add) {
  if (PK) {
    const unsigned long long o = atomicAdd(&T.hkv[pos], add);
    return (o & PK_SIG_MASK) + add <= PK_SIG_MASK;
  }
  const unsigned long long o = atomicAdd(&T.hsig[pos], add);
  return o + add >= o;
}

__device__ __forceinline__ uint32_t hash_pos(int32_t v, int hlog) {
  return ((uint32_t)v * 2654435761u) >> (32 - hlog);
}

// A level can touch the other search only at nodes of the other side's
// current frontier: a node the other side reached earlier was expanded by it
// before this side reached x, and would have touched then (or claimed x).
// The shared-memory tiers keep a one-bit-per-slot filter of that frontier
// (2^FILTER_LOG slots, a different hash than the table's), so that most heads
// of a scanned arc are rejected by one shared load instead of a probe.
#ifndef KD_FILTER_LOG
#define KD_FILTER_LOG 15
#endif
constexpr int FILTER_LOG = KD_FILTER_LOG;  // the default layout's filter: 2^FILTER_LOG bits
// fshift = 32 - log2(the filter's bits)
__device__ __forceinline__ uint32_t filter_slot(int32_t v, int fshift) { return ((uint32_t)v * 0x9E3779B1u) >> fshift; }

// position of v's entry (its word in *wout), or -1
__device__ __forceinline__ int tab_probe(const Tables& T, int32_t v, unsigned long long* wout) {
  uint32_t pos = hash_pos(v, T.hlog);
#pragma unroll 1
  for (uint32_t k = 0; k <= T.hmask; ++k) {
    const unsigned long long w = T.hkv[pos];
    if (w == EMPTY) return -1;
    if ((int32_t)(w >> 32) == v) {
      *wout = w;
      return (int)pos;
    }
    pos = (pos + 1) & T.hmask;
  }
  return -1;
}

// position of v's entry, or -1
__device__ __forceinline__ int tab_find_pos(const Tables& T, int32_t v) {
  uint32_t pos = hash_pos(v, T.hlog);
#pragma unroll 1
  for (uint32_t k = 0; k <= T.hmask; ++k) {
    const unsigned long long w = T.hkv[pos];
    if (w == EMPTY) return -1;
    if ((int32_t)(w >> 32) == v) return (int)pos;
    pos = (pos + 1) & T.hmask;
  }
  return -1;
}

// 1 = inserted at *pos_out, 0 = already present at *pos_out, -1 = table full
__device__ __forceinline__ int tab_insert(const Tables& T, int32_t v, unsigned long long want, uint32_t* pos_out) {
  uint32_t pos = hash_pos(v, T.hlog);
#pragma unroll 1
  for (uint32_t k = 0; k <= T.hmask; ++k) {
    unsigned long long w = T.hkv[pos];
    if (w == EMPTY) {
      const unsigned long long old = atomicCAS(&T.hkv[pos], EMPTY, want);
      if (old == EMPTY) {
        *pos_out = pos;
        return 1;
      }
      w = old;
    }
    if ((int32_t)(w >> 32) == v) {
      *pos_out = pos;
      return 0;
    }
    pos = (pos + 1) & T.hmask;
  }
  return -1;
}

// ============================================================== parameters
struct GraphDev {
  int32_t n;
  int64_t m;
  const int32_t* rp;   // out-arc offsets
  const int32_t* ci;   // out-arc targets
  const int32_t* rrp;  // in-arc offsets
  const int32_t* rci;  // in-arc sources
};

// One graph's share of a sampler launch: samples [first_idx, first_idx+count)
// of one RNG domain, numbered work_begin.. in the launch's work index space.
struct Job {
  GraphDev g;
  uint64_t seed;
  uint32_t domain;
  uint32_t pad;
  uint64_t first_idx;
  uint64_t count;
  uint32_t* counts;                 // hit counters (n) or null
  long long* totals;                // KADABRA_NSTAT work counters or null
  uint64_t work_begin;
};

struct SampleParams {
  Job job0;                         // the job, when the launch has only one
  const Job* jobs;                  // device array of njobs jobs, or null (then job0)
  int njobs;
  uint64_t total_work;              // sum of the jobs' counts
  const unsigned long long* total_dev;  // if set: the sum, read from device memory at launch
  unsigned long long* ctr;          // queue counters, Q_*
  unsigned long long* qb;           // sample indices queued for tier B
  unsigned long long* ql;           // sample indices queued for tier L
  unsigned long long* q0;           // if set: tier S takes its samples from this queue (filled by tier W)
  uint64_t deferred_cap;            // capacity of each queue
  int32_t* status;                  // run-wide error word (kadabra_status values)
  int tier_flags;                   // TF_* test switches for the table tiers
  // per-sample outputs (test hook) or null
  int32_t* st_out;
  int32_t* path_len;
  int32_t* paths;
  int32_t max_len;
  long long* stats;
  int32_t* sstatus;
  // tables
  PiEntry* pi_base;                 // per CTA: PI_SEGS * pcap entries
  int pcap;
  unsigned char* med_base;          // tier M tables, per CTA of the large-table launch
  size_t med_stride;
  int med_hlog, med_lcap;           //   their hash slots (log2) and list capacity
  unsigned char* gm_base;           // tier L tables, per CTA of the deferred launch
  size_t gm_stride;
  int gm_hlog;
  int gm_lcap;
};

// Long rows of a level (the scan variant for graphs beyond the L2 only).
// Every arc that can touch joins the two current frontiers, so a frontier
// row x of deg arcs holds a touch arc for each node of the other frontier
// (k nodes) that it contains.  Rows are sorted, so k searches in the row
// find them all; pass 1 takes them instead of scanning the row when
// deg > k * log2(deg) * W / 16.  A search's loads depend on one another while
// a scan streams, so W = 16 (measured: R-MAT scale 22, W = 4, 8, 16 gave
// 2.70, 2.61, 2.52 ms per batch against 2.98 ms with no searches; on the
// L2-resident Chung-Lu graph searches gained nothing and the extra code cost
// 4 %).  Up to one row per 32 nodes of a frontier segment and LONG_CAP in
// all (16 rows in all measured 2 % slower on R-MAT scale 22); the work
// counter still counts every arc.
#ifndef KD_LONG_CAP
#define KD_LONG_CAP 32
#endif
#ifndef KD_MEMB_W
#define KD_MEMB_W 16
#endif
#ifndef KD_LONG_MIN
#define KD_LONG_MIN 32
#endif
constexpr int LONG_CAP = KD_LONG_CAP;
#ifndef KD_FUSE_MAX
#define KD_FUSE_MAX 256
#endif
#ifndef KD_TD
#define KD_TD 6
#endif
// Pass 1: arcs per lane in flight.  Batches of 65,536 samples on the Chung-Lu
// graph of 10^6 nodes and the run of 64 BA graphs with 4 and 6: 2.85 and 2.81,
// 93.4 and 92.0 ms; the small ER graph's runs 1.07 ms with either.
constexpr int TOUCH_DEPTH = KD_TD;
constexpr int FUSE_MAX = KD_FUSE_MAX;  // levels of at most this many arcs insert and test for touches in one pass
__device__ __forceinline__ bool row_is_long(int deg, int k) {
  if (KD_MEMB_W <= 0 || k <= 0 || deg < KD_LONG_MIN) return false;
  const int lg = 32 - __clz(deg);  // bits of deg: the search steps
  return (long long)deg * 16 > (long long)k * lg * KD_MEMB_W;
}

struct LongRows {
  int start[LONG_CAP], deg[LONG_CAP];  // row start and degree
  uint16_t pos[LONG_CAP];              // position in the frontier segment
};

// per-CTA control block in shared memory
template <int NW>
struct Ctl {
  Job job;        // the job of the current sample
  int tot_job;    // the job that tot accumulates for (-1: none)
  long long stat[KADABRA_NSTAT];  // per sample; but for BT_SCANNED, adds go to the low words (32 bits hold them)
  long long tot[KADABRA_NSTAT];
  unsigned long long wsum[NW];
  unsigned long long wsum_hi[NW];
  unsigned long long u64tmp[NW];
  unsigned long long r;
  unsigned cost[2];   // frontier degree sums of the two roots
  unsigned acc[2];    // degree sum of the nodes a level inserts, by level parity
  unsigned hacc[2];   //   and its repeat discoveries
  int scan_tmp[2][NW];
  int s, t;
  int nlist;
  int npi;            // candidate (touch) edges found
  int flags;
  int lvl_flags;      // failures of the level that is being inserted (LF_*)
  int2 fr[2][32];     // row bounds {start, arcs} of each side's frontier, if it has at most 32 nodes
  int fside, fdepth;  // the frontier the filter in T.bits was built for (fside -1: none)
  int nlong;          // frontier rows of the current segment searched instead of scanned (T.lr)
  int ecount;     // backtracking: candidates found in the previous level
  int bt_flag;    // backtracking: an invariant failed at this step
  uint4 draws[32];  // the sample's Philox blocks j = 0..31, drawn by warp 0 at its start
  int pick;
  int mode;       // backtracking: 0 = scan the row of x, 1 = scan the previous level
  int cand[2];               // the chosen candidate edge: v on the s side, w on the t side
  int bt_x[2], bt_dx[2];     // backtracking walkers (0: v -> s, 1: w -> t): node, depth
  uint32_t bt_j[2];          //   and the next Philox block of each
  unsigned long long cur, k;  // the launch's running index, the sample's work index
  unsigned long long ntotal;
  // weighted radix selection (block_pick_radix; its histogram lives in the
  // frontier array, which is free while a candidate edge is chosen)
  unsigned long long rsel_r;
  int rsel_digit;
  unsigned rsel_cnt;
};

// adds to a per-sample counter (no thread waits for the sum)
template <int NW>
__device__ __forceinline__ void stat_add(Ctl<NW>& c, int q, unsigned x) {
  atomicAdd(reinterpret_cast<unsigned*>(&c.stat[q]), x);
}

// ============================================================== block helpers
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }

// exclusive scan of one int per thread; *total gets the block sum.  One
// barrier: calls that follow each other alternate between two tmp arrays.
template <int NW>
__device__ __forceinline__ int block_exscan(int x, int* tmp, int* total) {
  const int lane = lane_id(), w = warp_id();
  int v = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) tmp[w] = v;
  __syncthreads();
  int wpre = 0, tot = 0;
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int t = tmp[i];
    if (i < w) wpre += t;
    tot += t;
  }
  *total = tot;
  return wpre + v - x;
}

// inclusive scan of one u64 per thread; *total gets the block sum
template <int NW>
__device__ __forceinline__ unsigned long long block_inscan_u64(unsigned long long x, unsigned long long* tmp,
                                                               unsigned long long* total) {
  const int lane = lane_id(), w = warp_id();
  unsigned long long v = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) tmp[w] = v;
  __syncthreads();
  unsigned long long wpre = 0, tot = 0;
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const unsigned long long t = tmp[i];
    if (i < w) wpre += t;
    tot += t;
  }
  __syncthreads();
  *total = tot;
  return wpre + v;
}

// largest p in [0, cnt) with pr[p].x <= e (prefixes non-decreasing, pr[0].x = 0)
__device__ __forceinline__ int frontier_pos(const int2* pr, int cnt, int e) {
  int lo = 0, hi = cnt;
#pragma unroll 1
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pr[mid].x <= e)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// largest p in [a, cnt) with pr[p].x <= e, given pr[a].x <= e < pr[cnt].x:
// a window of 32 arcs from a row start reaches at most 32 rows further unless
// rows are empty, so the next 32 rows are searched first
__device__ __forceinline__ int frontier_next(const int2* pr, int a, int cnt, int e) {
  int b = min(a + 32, cnt);
  if (pr[b].x <= e) {
    a = b;
    b = cnt;
  }
#pragma unroll 1
  while (b - a > 1) {
    const int mid = (a + b) >> 1;
    if (pr[mid].x <= e)
      a = mid;
    else
      b = mid;
  }
  return a;
}

// first position of y in the sorted row col[a, b) (b if absent)
__device__ __forceinline__ int lower_bound_row(const int32_t* col, int a, int b, int32_t y) {
#pragma unroll 1
  while (a < b) {
    const int mid = a + ((b - a) >> 1);  // a + b may pass 2^31
    if (__ldg(&col[mid]) < y)
      a = mid + 1;
    else
      b = mid;
  }
  return a;
}

// One round of a four-way lower-bound search: pivots v1..v3 at a + s,
// a + 2s, a + 3s (s = (b - a) / 4 > 0) narrow [a, b] to a quarter.
__device__ __forceinline__ void lb4_update(int& a, int& b, int s, int32_t v1, int32_t v2, int32_t v3, int32_t y) {
  if (v3 < y) {
    a += 3 * s + 1;
  } else if (v2 < y) {
    b = a + 3 * s;
    a += 2 * s + 1;
  } else if (v1 < y) {
    b = a + 2 * s;
    a += s + 1;
  } else {
    b = a + s;
  }
}

// First positions of y0 in the sorted row col[a0, b0) and of y1 in
// col[a1, b1) (the row end if absent), searched together: each round loads
// three pivots of each range, six independent loads, and narrows both
// four-fold, so a 10^4-arc row takes seven rounds of one L2 round trip each
// instead of fourteen dependent loads per search.
__device__ __forceinline__ void lower_bound_rows2(const int32_t* col, int& a0, int b0, int32_t y0, int& a1, int b1,
                                                  int32_t y1) {
#pragma unroll 1
  for (;;) {
    const bool w0 = b0 - a0 > 3, w1 = b1 - a1 > 3;
    if (!w0 && !w1) break;
    const int s0 = (b0 - a0) >> 2, s1 = (b1 - a1) >> 2;
    int32_t u1 = 0, u2 = 0, u3 = 0, v1 = 0, v2 = 0, v3 = 0;
    if (w0) {
      u1 = __ldg(&col[a0 + s0]);
      u2 = __ldg(&col[a0 + 2 * s0]);
      u3 = __ldg(&col[a0 + 3 * s0]);
    }
    if (w1) {
      v1 = __ldg(&col[a1 + s1]);
      v2 = __ldg(&col[a1 + 2 * s1]);
      v3 = __ldg(&col[a1 + 3 * s1]);
    }
    if (w0) lb4_update(a0, b0, s0, u1, u2, u3, y0);
    if (w1) lb4_update(a1, b1, s1, v1, v2, v3, y1);
  }
#pragma unroll 1
  while (a0 < b0 || a1 < b1) {  // at most two more rounds
    const int m0 = a0 + ((b0 - a0) >> 1), m1 = a1 + ((b1 - a1) >> 1);
    const bool w0 = a0 < b0, w1 = a1 < b1;
    const int32_t u = w0 ? __ldg(&col[m0]) : 0, v = w1 ? __ldg(&col[m1]) : 0;
    if (w0) {
      if (u < y0)
        a0 = m0 + 1;
      else
        b0 = m0;
    }
    if (w1) {
      if (v < y1)
        a1 = m1 + 1;
      else
        b1 = m1;
    }
  }
}

// lower_bound over a sorted row by one warp: 32 pivots per round narrow the
// range 32-fold, so a 10^4-entry row takes three rounds of loads instead of
// fourteen dependent ones.  All lanes get the result.
__device__ __forceinline__ int warp_lower_bound(const int32_t* col, int a, int b, int32_t y) {
  const int lane = lane_id();
#pragma unroll 1
  while (b - a > 32) {
    const long long span = b - a;
    const int piv = a + (int)((span * lane) / 32);
    const bool less = __ldg(&col[piv]) < y;
    const unsigned m = __ballot_sync(FULL, less);
    // pivots are non-decreasing in lane order: the first lane whose pivot is
    // not below y bounds the answer
    const int k = m == FULL ? 32 : __ffs(~m) - 1;
    const int na = k == 0 ? a : a + (int)((span * (k - 1)) / 32) + 1;
    const int nb = k == 32 ? b : a + (int)((span * k) / 32);
    a = na;
    b = nb;
  }
  const bool less = lane < b - a && __ldg(&col[a + lane]) < y;
  const unsigned m = __ballot_sync(FULL, less);
  return a + __popc(m);
}

// Weighted choice over items 0..N-1 in order: the first item whose inclusive
// prefix sum of weights exceeds r (r < total weight).  Each thread weighs U
// consecutive items per step so their memory accesses overlap.  Returns the
// item index (all threads), or -1 if r is not below the total.
template <int NW, class WF>
__device__ __forceinline__ int block_pick(int N, unsigned long long r, Ctl<NW>& c, WF wf) {
  constexpr int NT = 32 * NW;
  const int tid = threadIdx.x;
  if (tid == 0) c.pick = -1;
  __syncthreads();
  unsigned long long carry = 0;
#pragma unroll 1
  for (int base = 0; base < N; base += NT * U) {
    unsigned long long w[U];
    unsigned long long tsum = 0;
    wf(base + tid * U, N, w);
#pragma unroll
    for (int k = 0; k < U; ++k) tsum += w[k];
    unsigned long long tot;
    const unsigned long long incl = block_inscan_u64<NW>(tsum, c.u64tmp, &tot);
    const unsigned long long excl = incl - tsum;
    if (tsum != 0 && carry + excl <= r && r < carry + incl) {
      unsigned long long acc = carry + excl;
#pragma unroll
      for (int k = 0; k < U; ++k) {
        acc += w[k];
        if (acc > r) {
          c.pick = base + tid * U + k;
          break;
        }
      }
    }
    carry += tot;
    if (carry > r) break;
  }
  __syncthreads();
  return c.pick;
}

// ============================================================== one sample
// Arcs per warp of a level of E arcs: whole windows of 32, so that a small
// level issues few full windows instead of one per warp with a few lanes each.
template <int NW>
__device__ __forceinline__ int warp_slice(int E) {
  return max(1, (int)(((unsigned)E + 32u * NW - 1u) / (32u * NW))) * 32;
}

// The warp's slice [c0, c1) of the level's E arcs.  (E may be close to 2^31:
// no sum of arc indices beyond it is taken as an int, and the scans below
// count down the arcs left instead of comparing ends.)
template <int NW>
__device__ __forceinline__ void take_slice(int E, int& c0, int& c1) {
  const unsigned per = (unsigned)warp_slice<NW>(E);
  const unsigned a = min((unsigned)E, (unsigned)warp_id() * per);
  c0 = (int)a;
  c1 = (int)min((unsigned)E, a + per);
}

// Frontier positions p[k] of the tails of arcs wb + 32 k + lane (k < D; the
// next `rem` of them matter), given row pcur with its start <= wb < the next
// row's start.  Each lane takes one of the next 32 rows and sets a bit where it
// starts; a lane's row is pcur plus the bits up to its arc.  That is one
// shared load and a few warp reductions instead of a binary search per lane.
// Rows without arcs share a start, and more than 32 rows may start in the
// step: then the lanes search.
template <int D>
__device__ __forceinline__ void rows_of_step(const Tables& T, int pcur, int fcount, int wb, int rem, int (&p)[D]) {
  const int lane = lane_id();
  const int q = pcur + 1 + lane;
  const int st = T.pr[KIDX(min(q, fcount), T.frcap + 1, 7)].x - wb;  // at least 1
  const bool in = q < fcount && st < 32 * D;
  const unsigned who = __ballot_sync(FULL, in);
  unsigned w[D];
  int rows = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    w[k] = __reduce_or_sync(FULL, in && (st >> 5) == k ? 1u << (st & 31) : 0u);
    rows += __popc(w[k]);
  }
  if (rows == __popc(who) && !(who >> 31)) {
    int at = pcur;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      p[k] = at + __popc(w[k] & (FULL >> (31 - lane)));
      at += __popc(w[k]);
    }
  } else {
#pragma unroll 1
    for (int k = 0; k < D; ++k) {
      const int f = 32 * k + lane < rem ? frontier_next(T.pr, pcur, fcount, wb + 32 * k + lane) : pcur;
#pragma unroll
      for (int j = 0; j < D; ++j)
        if (j == k) p[j] = f;
    }
  }
}

// Pass 1 of a level: looks for touch arcs among its E arcs.  Each warp takes
// a contiguous slice of the flattened arc range and walks it 32 D arcs at a
// time, every lane with D independent loads in flight (coalesced within rows,
// of any alignment), whether the step lies in one row or in many.  Hardly any
// arc touches, and in the shared-memory tiers one filter load rejects most
// heads, so a step tests its heads against the filter only; the lanes that
// pass then probe the table together.  Calls emit(touch, x's frontier
// position, y, y's table position and word) with all lanes of the warp, in
// no particular order.  Bound by instruction issue and by the slowest warp at
// the barrier after it: windows of 32 arcs with a probe each, and short rows
// one window at a time, took 23.2 k of 74 k cycles per sample on the Chung-Lu
// graph of 10^6 nodes; this takes 16 k of 57 k.  Run twice, it adds 36 % to a
// batch's instructions and 35 % to its time; without the branches around each
// filter test a batch of 65,536 went 2.97 -> 2.85 ms.
template <bool PK, int D, int NW, class EM>
__device__ __forceinline__ void touch_pass(const Tables& T, int side, int fcount, int E, const int32_t* cols,
                                           int64_t ncols, EM emit) {
  const int lane = lane_id();
  int c0, c1;
  take_slice<NW>(E, c0, c1);
  if (c0 >= c1) return;
  int pcur = frontier_pos(T.pr, fcount, c0);  // warp-uniform
  int2 cur = T.pr[KIDX(pcur, T.frcap + 1, 7)];  // {first arc index, row start}
  int nxt = T.pr[KIDX(pcur + 1, T.frcap + 1, 7)].x;  // first arc index of the next row
#pragma unroll 1
  for (int rem = c1 - c0; rem > 0; rem -= 32 * D) {
    const int wb = c1 - rem;
    if (nxt <= wb) {  // the next arc lies in a later row
      pcur = frontier_next(T.pr, pcur + 1, fcount, wb);
      cur = T.pr[KIDX(pcur, T.frcap + 1, 7)];
      nxt = T.pr[KIDX(pcur + 1, T.frcap + 1, 7)].x;
    }
    int a[D];  // the arcs' places in the column array
    if (nxt - wb >= min(rem, 32 * D)) {  // one row
#pragma unroll
      for (int k = 0; k < D; ++k) a[k] = cur.y + (wb - cur.x) + lane + 32 * k;
    } else {
      int p[D];
      rows_of_step<D>(T, pcur, fcount, wb, rem, p);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int2 q = T.pr[KIDX(p[k], T.frcap + 1, 7)];
        a[k] = q.y + (wb + 32 * k + lane - q.x);
      }
    }
    const int left = rem - lane;  // the lane's arc k exists if left > 32 k
    int y[D];
#pragma unroll
    for (int k = 0; k < D; ++k)
      y[k] = left > 32 * k ? __ldg(&cols[KIDX((int64_t)a[k], ncols, 8)]) : 0;
    // bit k: head y[k] may touch (tested without branches; the heads of lanes
    // beyond the slice are masked)
    unsigned hit = PK ? 0u : (1u << D) - 1u;
    if (PK) {
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const uint32_t h = filter_slot(y[k], T.fshift);
        hit |= (__funnelshift_r(T.bits[h >> 5], 0u, h) & 1u) << k;
      }
    }
    if (left <= 32 * (D - 1)) hit &= left > 0 ? (2u << ((left - 1) >> 5)) - 1u : 0u;
#pragma unroll 1
    while (__any_sync(FULL, hit != 0)) {
      bool touch = false;
      int yy = 0, pos = -1, p = 0;
      unsigned long long hy = 0;
      if (hit) {
        const int k = __ffs(hit) - 1;
        hit &= hit - 1;
        yy = y[0];
#pragma unroll
        for (int j = 1; j < D; ++j)
          if (k == j) yy = y[j];
        pos = tab_probe(T, yy, &hy);
        touch = pos >= 0 && val_side(ent_val<PK>(hy)) != side;
        if (touch) {
          const int e = wb + 32 * k + lane;
          p = e < nxt ? pcur : frontier_next(T.pr, pcur + 1, fcount, e);
        }
      }
      emit(touch, p, yy, pos, hy);
    }
  }
}

// The level scan of pass 2: each warp walks its slice in windows of 32 arcs,
// software-pipelined (the loads of the next window are issued before the
// current one is processed, so their latency overlaps its probes).  For every
// window it calls f(ok, p, y): ok = the lane holds an arc, p = frontier
// position of its tail, y = its head.  All lanes of the warp call f together.
template <int NW, class F>
__device__ __forceinline__ void scan_level(const Tables& T, int fcount, int E, const int32_t* cols, int64_t ncols,
                                           F f) {
  const int lane = lane_id();
  int c0, c1;
  take_slice<NW>(E, c0, c1);
  if (c0 >= c1) return;
  int pcur = frontier_pos(T.pr, fcount, c0);  // warp-uniform
  int2 cur = T.pr[KIDX(pcur, T.frcap + 1, 7)];  // {first arc index, row start}
  int nxt = T.pr[KIDX(pcur + 1, T.frcap + 1, 7)].x;  // first arc index of the next row
  // the window of the last `rem` arcs: its lanes' frontier positions and heads (loads issued)
  auto fetch = [&](int rem, bool& ok, int& p, int& y) {
    ok = false;
    p = y = 0;
    if (rem <= 0) return;
    const int wb = c1 - rem;
    if (nxt <= wb) {  // the window starts in a later row
      pcur = frontier_next(T.pr, pcur + 1, fcount, wb);
      cur = T.pr[KIDX(pcur, T.frcap + 1, 7)];
      nxt = T.pr[KIDX(pcur + 1, T.frcap + 1, 7)].x;
    }
    int2 q = cur;
    p = pcur;
    if (nxt - wb < min(rem, 32)) {
      int pk[1];
      rows_of_step<1>(T, pcur, fcount, wb, rem, pk);
      p = pk[0];
      q = T.pr[KIDX(p, T.frcap + 1, 7)];
    }
    ok = lane < rem;
    if (ok) y = __ldg(&cols[KIDX((int64_t)q.y + (wb - q.x) + lane, ncols, 8)]);
  };
  bool ok0 = false, ok1;
  int p0 = 0, p1, y0 = 0, y1;
#pragma unroll 1
  for (int rem = c1 - c0 + 32; rem > 0; rem -= 32) {  // the first round only fetches
    fetch(rem - 32, ok1, p1, y1);
    if (rem <= c1 - c0) f(ok0, p0, y0);
    ok0 = ok1;
    p0 = p1;
    y0 = y1;
  }
}

// Weighted choice among n items held in any order, in the order of their
// 64-bit keys (distinct): the item whose key-order prefix interval contains r.
// Quadratic in n: each thread ranks its items against all others.  c.pick
// must be -1 before a barrier that precedes the call.
template <int NW, class KF, class WF>
__device__ __forceinline__ int block_pick_by_key(int n, unsigned long long r, Ctl<NW>& c, KF key, WF w) {
  constexpr int NT = 32 * NW;
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += NT) {
    const unsigned long long ki = key(i);
    const unsigned long long wi = w(i);
    if (wi == 0) continue;
    unsigned long long below = 0;
#pragma unroll 1
    for (int j = 0; j < n; ++j)
      if (key(j) < ki) below += w(j);
    if (below <= r && r - below < wi) c.pick = i;
  }
  __syncthreads();
  return c.pick;
}

// Weighted choice among n candidate edges in the order of their keys
// (x << 32 | y, distinct) without sorting them: most-significant-byte radix
// selection.  Each pass sums, per value of the next key byte, the weights
// (and the number) of the candidates that share the bytes fixed so far; the
// byte whose cumulative weight first exceeds r is fixed and r is reduced by
// the weight below it.  Once a single candidate shares the fixed bytes it is
// the pick.  Each thread reads a contiguous run of candidates and adds to the
// shared histogram once per run of equal bytes: candidates of one tail x are
// contiguous and sorted by y, so runs are long.  Returns the candidate's
// index (all threads), or -1 if r is not below the total weight.
template <int NW>
__device__ __noinline__ int block_pick_radix(const PiEntry* buf, int n, unsigned long long r, Ctl<NW>& c,
                                unsigned long long* rhist, unsigned* rcnt) {
  constexpr int NT = 32 * NW;
  const int tid = threadIdx.x, lane = lane_id();
  auto key = [&](int i) { return ((unsigned long long)(uint32_t)buf[i].x << 32) | (uint32_t)buf[i].y; };
  const int chunk = (n + NT - 1) / NT;
  const int a = min(n, tid * chunk), b = min(n, a + chunk);
  unsigned long long fixed = 0;  // the key bytes above `shift` chosen so far
#pragma unroll 1
  for (int shift = 56; shift >= 0; shift -= 8) {
#pragma unroll 1
    for (int i = tid; i < 256; i += NT) {
      rhist[i] = 0ull;
      rcnt[i] = 0u;
    }
    __syncthreads();
    int cur = -1;
    unsigned long long acc = 0;
    unsigned cnt = 0;
#pragma unroll 1
    for (int i = a; i < b; ++i) {
      const unsigned long long k = key(i);
      if (shift < 56 && (k >> (shift + 8)) != fixed) continue;
      const int d = (int)((k >> shift) & 255ull);
      if (d != cur) {
        if (cur >= 0) {
          atomicAdd(&rhist[cur], acc);
          atomicAdd(&rcnt[cur], cnt);
        }
        cur = d;
        acc = 0;
        cnt = 0;
      }
      acc += buf[i].w;
      ++cnt;
    }
    if (cur >= 0) {
      atomicAdd(&rhist[cur], acc);
      atomicAdd(&rcnt[cur], cnt);
    }
    __syncthreads();
    if (tid < 32) {  // warp 0: the byte whose cumulative weight first exceeds r
      unsigned long long s8 = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) s8 += rhist[8 * lane + q];
      unsigned long long incl = s8;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 0) c.rsel_digit = -1;
      __syncwarp();
      const unsigned long long excl = incl - s8;
      if (excl <= r && r < incl) {
        unsigned long long below = excl;
#pragma unroll 1
        for (int q = 0; q < 8; ++q) {
          const unsigned long long h = rhist[8 * lane + q];
          if (r < below + h) {
            c.rsel_digit = 8 * lane + q;
            c.rsel_r = r - below;
            c.rsel_cnt = rcnt[8 * lane + q];
            break;
          }
          below += h;
        }
      }
      if (lane == 0) c.pick = -1;
    }
    __syncthreads();
    const int d = c.rsel_digit;
    if (d < 0) return -1;
    r = c.rsel_r;
    fixed = (fixed << 8) | (unsigned long long)d;
    if (c.rsel_cnt == 1u || shift == 0) {
#pragma unroll 1
      for (int i = tid; i < n; i += NT)
        if ((key(i) >> shift) == fixed) c.pick = i;
      __syncthreads();
      return c.pick;
    }
    // the next pass clears the histogram only: the selection fields read
    // above are rewritten after two more barriers
  }
  return -1;
}

// Records a backtracking pick y (now at depth dn on side `half`, at position
// pos of the scanned row): the work counter, its hit (interior nodes only)
// and its place on the path.  One thread.
template <bool PK, int NW>
__device__ __forceinline__ void bt_record(const SampleParams& P, const Job& J, Ctl<NW>& c, int half, int dn, int y, int pos,
                                          int64_t out_i, int dv, int dw, bool want_path) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&c.stat[KADABRA_STAT_BT_SCANNED]), (unsigned long long)(pos + 1));
  if (dn > 0 && J.counts) atomicAdd(&J.counts[KIDX(y, J.g.n, 11)], 1u);
  if (want_path) {
    const int at = half == 0 ? dn : (dv + 1) + (dw - dn);
    if (at < P.max_len) P.paths[out_i * (int64_t)P.max_len + at] = y;
  }
}

#ifndef KD_WARP_BT_ROW
#define KD_WARP_BT_ROW 256
#endif
constexpr int WARP_BT_ROW = KD_WARP_BT_ROW;  // rows up to this length: the step stays with its warp

// One warp's backtracking steps for walker `half` (0: from v towards s over
// predecessors, 1: from w towards t over successors), from its state in
// c.bt_*[half] until it reaches its root or a step with more candidates than
// a warp takes comes up (left in c.bt_*[half] for the block).  The draw, the
// candidate order and the pick are those of the block's steps: the first
// neighbour one level closer, in row order, whose cumulative sigma exceeds r.
// A row is read four windows of 32 at a time.
template <bool PK, int NW>
__device__ void bt_warp_steps(const SampleParams& P, const Job& J, const Tables& T, Ctl<NW>& c, uint64_t idx,
                              int64_t out_i, int dv, int dw, bool want_path, int half) {
  const int lane = lane_id();
  const GraphDev& G = J.g;
  int x = c.bt_x[half], dx = c.bt_dx[half];
  if (dx <= 0) return;
  uint32_t j = c.bt_j[half];
  const int32_t* brow = half == 0 ? G.rrp : G.rp;
  const int32_t* bcol = half == 0 ? G.rci : G.ci;
  unsigned long long sx = 0;  // sigma of x
  {
    const int px = tab_find_pos(T, x);
    const unsigned long long hx = px >= 0 ? T.hkv[px] : 0ull;
    if (px < 0 || ent_val<PK>(hx) != pack_val(half, dx)) {
      if (lane == 0) c.bt_flag = 1;
      return;
    }
    sx = ent_sig<PK>(T, hx, (uint32_t)px);
  }
#pragma unroll 1
  while (dx > 0) {
    const int plo = lvl_lo(T, half, dx - 1), phi = lvl_hi(T, half, dx - 1);
    const int r0 = __ldg(&brow[x]), deg = __ldg(&brow[x + 1]) - r0;
    const bool single = phi - plo == 1;
    const bool by_level = phi - plo <= 32 && (phi - plo) * 16 < deg;
    if (!single && !by_level && deg > WARP_BT_ROW) break;  // the block takes this step
    int y = -1, pos = -1;
    if (single) {
      // a single node one level closer: it is x's only predecessor
      y = list_node<PK>(T, plo);
      const uint32_t q = lpos_get<PK>(T, plo);
      sx = ent_sig<PK>(T, T.hkv[q], q);
    } else if (by_level) {
      // the previous level's nodes, one per lane: those adjacent to x are the
      // candidates, in id order (a long row of x takes more steps to scan)
      const unsigned long long r = below128(j < 32 ? c.draws[j] : draw_late(J.seed, J.domain, idx, j), sx);
      const int32_t* frow = half == 0 ? G.rp : G.rrp;
      const int32_t* fcol = half == 0 ? G.ci : G.rci;
      int yy = 0x7FFFFFFF;
      unsigned long long w = 0;
      if (plo + lane < phi) {
        yy = list_node<PK>(T, plo + lane);
        const int b = __ldg(&frow[yy + 1]);
        const int at = lower_bound_row(fcol, __ldg(&frow[yy]), b, x);
        if (at < b && __ldg(&fcol[KIDX((int64_t)at, G.m, 12)]) == x) {
          const uint32_t q = lpos_get<PK>(T, plo + lane);
          w = ent_sig<PK>(T, T.hkv[q], q);
        }
      }
      unsigned long long below = 0;
      for (unsigned m = __ballot_sync(FULL, w != 0); m; m &= m - 1) {
        const int k = __ffs(m) - 1;
        const int yk = __shfl_sync(FULL, yy, k);
        const unsigned long long wk = __shfl_sync(FULL, w, k);
        if (yk < yy) below += wk;
      }
      const unsigned hit = __ballot_sync(FULL, w != 0 && below <= r && r - below < w);
      if (hit) {
        y = __shfl_sync(FULL, yy, __ffs(hit) - 1);
        sx = __shfl_sync(FULL, w, __ffs(hit) - 1);
      }
    } else {
      const unsigned long long r = below128(j < 32 ? c.draws[j] : draw_late(J.seed, J.domain, idx, j), sx);
      const uint32_t want = pack_val(half, dx - 1);
      unsigned long long carry = 0;
#pragma unroll 1
      for (int base = 0; base < deg && y < 0; base += 128) {
        int ys[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = base + 32 * k + lane;
          ys[k] = i < deg ? __ldg(&bcol[KIDX((int64_t)r0 + i, G.m, 12)]) : -1;
        }
#pragma unroll 1
        for (int k = 0; k < 4 && base + 32 * k < deg; ++k) {
          const int yy = k == 0 ? ys[0] : k == 1 ? ys[1] : k == 2 ? ys[2] : ys[3];
          unsigned long long w = 0;
          if (yy >= 0) {
            unsigned long long hw = 0;
            const int q = tab_probe(T, yy, &hw);
            if (q >= 0 && ent_val<PK>(hw) == want) w = ent_sig<PK>(T, hw, (uint32_t)q);
          }
          if (!__any_sync(FULL, w != 0)) continue;
          unsigned long long inc = w;  // inclusive scan (partial sums stay below sigma(x))
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += v;
          }
          const bool hit = w != 0 && carry + inc - w <= r && r < carry + inc;
          const unsigned m = __ballot_sync(FULL, hit);
          if (m) {
            const int from = __ffs(m) - 1;
            pos = base + 32 * k + from;
            y = __shfl_sync(FULL, yy, from);
            sx = __shfl_sync(FULL, w, from);
            break;
          }
          carry += __shfl_sync(FULL, inc, 31);
        }
      }
    }
    ++j;
    if (y < 0) {
      if (lane == 0) c.bt_flag = 1;
      return;
    }
    if (pos < 0) pos = warp_lower_bound(bcol, r0, r0 + deg, y) - r0;
    if (lane == 0) bt_record<PK>(P, J, c, half, dx - 1, y, pos, out_i, dv, dw, want_path);
    x = y;
    dx -= 1;
  }
  if (lane == 0) {
    c.bt_x[half] = x;
    c.bt_dx[half] = dx;
    c.bt_j[half] = j;
  }
}

// The touch arcs of the long rows of a frontier segment (T.lr, nl of
// them): item q = (row q / kother, node q % kother of the other frontier,
// list entries [ob, ob + kother)); a thread searches two items at a time.
// Calls emit as touch_pass does.  All lanes of every warp call it.
#ifdef KD_MEMB_NOINLINE
#define KD_MEMB_ATTR __device__ __noinline__
#else
#define KD_MEMB_ATTR __device__ __forceinline__
#endif
template <bool PK, int NW, class EM>
KD_MEMB_ATTR void search_long_rows(const Tables& T, const Ctl<NW>& c, const int32_t* cols, int64_t m, int ob,
                                   int kother, int nl, EM emit) {
  constexpr int NT = 32 * NW;
  const int lane = lane_id(), wid = warp_id();
  const long long items = (long long)nl * kother;
#pragma unroll 1
  for (long long qb = (long long)wid * 32; qb < items; qb += 2 * NT) {
    int r[2], a[2], e[2];
    uint32_t py[2];
    unsigned long long hy[2];
    int32_t y[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long q = qb + h * NT + lane;
      r[h] = -1;
      a[h] = e[h] = 0;
      y[h] = 0;
      py[h] = 0;
      hy[h] = 0;
      if (q < items) {
        r[h] = (int)(q / kother);
        const int yi = (int)(q - (long long)r[h] * kother);
        py[h] = lpos_get<PK>(T, ob + yi);
        hy[h] = T.hkv[KIDX(py[h], T.hmask + 1u, 14)];
        y[h] = (int32_t)(hy[h] >> 32);
        a[h] = T.lr->start[KIDX(r[h], LONG_CAP, 16)];
        e[h] = a[h] + T.lr->deg[r[h]];
      }
    }
    int b0 = e[0], b1 = e[1];
    lower_bound_rows2(cols, a[0], b0, y[0], a[1], b1, y[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool touch = r[h] >= 0 && a[h] < e[h] && __ldg(&cols[KIDX((int64_t)a[h], m, 8)]) == y[h];
      emit(touch, touch ? (int)T.lr->pos[r[h]] : 0, y[h], (int)py[h], hy[h]);
    }
  }
}

// One sample, from the state begin_sample and insert_roots left (warp 0's
// insertions need no barrier: the first level's frontier is read by warp 0,
// and the other warps read the table only after that level's first barrier).
// The caller puts a barrier after it.
//
// What a level costs beside its arcs is barriers and the latency of the steps
// one thread or warp takes while the others wait, so a level has as few of
// both as its data flow allows: the search's scalars live in every thread's
// registers (equal in all of them), counters are added without waiting for
// the sum, and a level has one barrier after its degree prefix, one after the
// filter if it is rebuilt, one after pass 1 and one after pass 2.  Candidate
// edges stay in shared memory, and so do the row bounds of small frontiers.
// With the scans above and the shorter code, batches of 65,536 samples went
// 4.41 -> 3.37 ms on the Chung-Lu graph of 10^6 nodes (2.49 -> 1.85 G warp
// instructions) and 2.70 -> 2.21 ms on R-MAT scale 22; a 3.4 M-node ER graph's
// run 18.3 -> 15.4 ms.
template <bool PK, bool RG, int NW>
__device__ __forceinline__ void run_sample(const SampleParams& P, const Job& J, const Tables& T, Ctl<NW>& c, uint64_t idx,
                                           int64_t out_i) {
  constexpr int NT = 32 * NW;
  const int tid = threadIdx.x, lane = lane_id(), wid = warp_id();
  const GraphDev& G = J.g;

  // ------------------------------------------------ bb-BFS (Sec. 4)
  int cost0 = (int)c.cost[0], cost1 = (int)c.cost[1];  // frontier degree sums
  int depth0 = 0, depth1 = 0;
  int last = -1;  // the side expanded by the previous level, whose bounds end at the lists' end
  bool touched = false;
  int side = 0;  // the side a level expands (after the search: the side that touched)
  int cand_at = 0, cand_cap = 0;  // where the level's candidate edges start in T.pr, and how many fit there
  const int pi_cap = PI_SEGS * T.pcap;  // candidate edges a sample may have
#pragma unroll 1
  for (int iter = 0; iter <= 2 * T.maxd + 2; ++iter) {
    const int par = iter & 1;
    side = cost0 <= cost1 ? 0 : 1;
    const int E = side == 0 ? cost0 : cost1;  // the level's arcs
    const int dcur = side == 0 ? depth0 : depth1, od = side == 0 ? depth1 : depth0;
    const int list_before = c.nlist;
    const int f0 = lvl_lo(T, side, dcur);
    const int fcount = (side == last ? list_before : lvl_hi(T, side, dcur)) - f0;
    // the other side's current frontier: the only nodes a touch arc reaches
    const int ob = lvl_lo(T, 1 - side, od);
    const int kother = (1 - side == last ? list_before : lvl_hi(T, 1 - side, od)) - ob;
    if (tid == NT - 32) {  // a warp that waits for the first one's prefix
      stat_add(c, KADABRA_STAT_LEVELS, 1u);
      stat_add(c, KADABRA_STAT_EXPANDED, (unsigned)fcount);
      stat_add(c, KADABRA_STAT_EDGES, (unsigned)E);
    }
    if (E == 0) return;  // no arc leaves this side: s and t are not connected
    const int dnew = dcur + 1;
    const int32_t* rowp = side == 0 ? G.rp : G.rrp;
    const int32_t* cols = side == 0 ? G.ci : G.rci;
    const int nseg = (fcount + T.frcap - 1) / T.frcap;
    // A level of at most FUSE_MAX arcs that cannot fill the lists skips pass
    // 1: pass 2 then tests for touches while it inserts, and undoes its
    // insertions if it finds one.
    const bool fused = E <= FUSE_MAX && nseg == 1 && list_before + E <= T.lcap;
    // pass 1 uses a filter of the other side's frontier, kept while that
    // frontier stays the same
    const bool new_filter = PK && !fused && (c.fside != 1 - side || c.fdepth != od);
    // Candidate edges go behind the frontier prefix in T.pr while they fit
    // (shared-memory tiers, one segment), then to T.pi, at their running index.
    cand_at = (fcount + 2) & ~1;
    cand_cap = PK && nseg == 1 ? max(0, T.frcap + 1 - cand_at) / 2 : 0;

    // Degree prefix and row starts over frontier nodes [fb, fb + cnt) into
    // T.pr.  A frontier of more than T.frcap nodes is scanned in segments of
    // T.frcap: the touch test and the insertion treat a level's arcs as a
    // set, so segments give the same result.
    // With kl > 0 (pass 1), rows that row_is_long picks for searches of the
    // other frontier's kl nodes go to T.lr (long_cap at most: one per 32
    // nodes of a segment, up to LONG_CAP; c.nlong must be 0) and count 0
    // arcs in the prefix.
    const int long_cap = min(LONG_CAP, max(1, T.frcap >> 5));
    auto take_long = [&](int deg, int kl, int seg_pos, int rs) {
      if (RG && row_is_long(deg, kl)) {
        const int q = atomicAdd(&c.nlong, 1);
        if (q < long_cap) {
          T.lr->pos[KIDX(q, LONG_CAP, 16)] = (uint16_t)seg_pos;
          T.lr->start[q] = rs;
          T.lr->deg[q] = deg;
          deg = 0;
        }
      }
      return deg;
    };
    auto build_prefix = [&](int fb, int cnt, int kl, bool clear_filter) {
      if (fcount <= 32) {  // one warp: shuffles only; the others clear the filter
        if (wid == 0) {
          int deg = 0, rs = 0;
          if (lane < cnt) {
            const int2 b = c.fr[side][KIDX(lane, 32, 17)];  // the rows' bounds, kept when the nodes were inserted
            rs = b.x;
            deg = take_long(b.y, kl, lane, rs);
          }
          int v = deg;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += u;
          }
          if (lane < cnt) T.pr[KIDX(lane, T.frcap + 1, 10)] = make_int2(v - deg, rs);
          if (lane == cnt - 1) T.pr[KIDX(cnt, T.frcap + 1, 10)] = make_int2(v, 0);
        } else if (PK && clear_filter) {
          int4* b = reinterpret_cast<int4*>(T.bits);
#pragma unroll 1
          for (int i = tid - 32; i < T.fwords / 4; i += NT - 32) b[i] = make_int4(0, 0, 0, 0);
        }
      } else {
        if (PK && clear_filter) {
          int4* b = reinterpret_cast<int4*>(T.bits);
#pragma unroll 1
          for (int i = tid; i < T.fwords / 4; i += NT) b[i] = make_int4(0, 0, 0, 0);
        }
        int carry = 0;
#pragma unroll 1
        for (int base = 0, h = 0; base < cnt; base += NT, h ^= 1) {
          const int i = base + tid;
          int deg = 0, rs = 0;
          if (i < cnt) {
            const int x = KIDX(list_node<PK>(T, fb + i), G.n, 9);
            rs = __ldg(&rowp[x]);
            deg = take_long(__ldg(&rowp[x + 1]) - rs, kl, i, rs);
          }
          int tot;
          const int ex = block_exscan<NW>(deg, c.scan_tmp[h], &tot);
          if (i < cnt) T.pr[KIDX(i, T.frcap + 1, 10)] = make_int2(carry + ex, rs);
          carry += tot;
        }
        if (tid == 0) T.pr[KIDX(cnt, T.frcap + 1, 10)] = make_int2(carry, 0);
      }
      __syncthreads();
    };

    // appends a warp's touch arcs (frontier position p, head y at table
    // position pos with word hy) with weight sigma_x * sigma_y
    bool sigma_of = false;
    auto emit = [&](int fb, bool touch, int p, int y, int pos, unsigned long long hy) {
      const unsigned m = __ballot_sync(FULL, touch);
      if (m == 0) return;
      int at = 0;
      if (lane == 0) at = atomicAdd(&c.npi, __popc(m));
      at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (touch) {
        const uint32_t px = lpos_get<PK>(T, fb + p);
        const unsigned long long hx = T.hkv[px];
        const unsigned long long sx = ent_sig<PK>(T, hx, px), sy = ent_sig<PK>(T, hy, (uint32_t)pos);
        if (!PK && __umul64hi(sx, sy) != 0ull) sigma_of = true;
        PiEntry e;
        e.x = (int32_t)(hx >> 32);
        e.y = y;
        e.w = sx * sy;
        if (at < cand_cap)  // entries cand_at + 2 at and the next one of T.pr
          *reinterpret_cast<PiEntry*>(T.pr + (KIDX(cand_at + 2 * at + 1, T.frcap + 1, 18) - 1)) = e;
        else if (at < pi_cap)
          T.pi[KIDX(at, pi_cap, 15)] = e;
      }
    };

    // Pass 1 is the touch test against the other search.  Pass 2 makes the
    // next level: the first discoverer of an unvisited head y publishes (y,
    // side, dist) with one CAS and appends y to the level list; every
    // discoverer adds sigma_x to the sigma field of y's hash entry (zero
    // until then), so the order of discoveries does not matter.  (One loop
    // over both, so that the prefix is built at one place in the code: the
    // kernel is long for the instruction caches.)
    bool had_long = false;  // pass 1 searched rows that pass 2 must scan
    int Eseg = E;           // arcs of the segment in T.pr
    unsigned hits = 0, cost = 0;
    bool of = false, cap = false;
    const uint32_t want_val = pack_val(side, dnew);
    const volatile int* nlist_now = &c.nlist;
#pragma unroll 1
    for (int pass = fused ? 2 : 1; pass <= 2; ++pass) {
      if (pass == 2 && dnew > T.maxd) {
        if (tid == 0) c.flags |= F_CAP;
        return;
      }
#pragma unroll 1
      for (int sg = 0; sg < nseg; ++sg) {
        const int fb = f0 + sg * T.frcap, cnt = min(T.frcap, fcount - sg * T.frcap);
        // pass 2, one segment without long rows: pass 1's prefix is still there
        if (pass == 1 || fused || nseg > 1 || had_long) {
          const bool nf = new_filter && pass == 1 && sg == 0;
          build_prefix(fb, cnt, RG && pass == 1 ? kother : 0, nf);
          if (PK && nf) {
#pragma unroll 1
            for (int i = ob + tid; i < ob + kother; i += NT) {
              const uint32_t h = filter_slot(list_node<PK>(T, i), T.fshift);
              atomicOr(&T.bits[h >> 5], 1u << (h & 31));
            }
            if (tid == 0) {
              c.fside = 1 - side;
              c.fdepth = od;
            }
            __syncthreads();
          }
          Eseg = T.pr[cnt].x;
        }
        if (pass == 1) {
          touch_pass<PK, TOUCH_DEPTH, NW>(
              T, side, cnt, Eseg, cols, G.m,
              [&](bool touch, int p, int y, int pos, unsigned long long hy) { emit(fb, touch, p, y, pos, hy); });
          // the long rows: one search per (row, other-frontier node)
          if constexpr (RG) {
            const int nl = min(c.nlong, long_cap);
            if (nl > 0) {
              had_long = true;
              search_long_rows<PK>(
                  T, c, cols, G.m, ob, kother, nl,
                  [&](bool touch, int p, int y, int pos, unsigned long long hy) { emit(fb, touch, p, y, pos, hy); });
            }
          }
        } else {
          scan_level<NW>(T, cnt, Eseg, cols, G.m, [&](bool ok, int p, int y) {
            int res = 0;  // 1 = inserted, 2 = a touch arc (fused)
            int ydeg = 0, ylo = 0;
            uint32_t pos = 0;
            unsigned long long add = 0, w = 0;
            if (ok && (fused || !cap)) {
              // the head's row bounds (its degree joins the new frontier's cost
              // if it is new), loaded before the probe so the load overlaps it
              ylo = __ldg(&rowp[KIDX(y, G.n, 13)]);
              const int yhi = __ldg(&rowp[KIDX(y, G.n, 13) + 1]);
              const uint32_t px = lpos_get<PK>(T, fb + p);
              add = ent_sig<PK>(T, T.hkv[px], px);
              pos = hash_pos(y, T.hlog);
              uint32_t k = 0;
#pragma unroll 1
              for (; k <= T.hmask; ++k) {
                w = T.hkv[pos];
                if (w == EMPTY) {
                  // stop inserting once the lists are full, so the table never
                  // fills beyond lcap + NT keys and probes stay short
                  if (*nlist_now >= T.lcap) {
                    cap = true;
                    break;
                  }
                  w = atomicCAS(&T.hkv[pos], EMPTY, ent_word<PK>(y, want_val, PK ? add : 0ull));
                  if (w == EMPTY) {
                    res = 1;
                    ydeg = yhi - ylo;
                    break;
                  }
                }
                if ((int32_t)(w >> 32) == y) {
                  const uint32_t v = ent_val<PK>(w);
                  if (v == want_val) {  // also discovered at this level
                    ++hits;
                    if (!ent_add<PK>(T, pos, add)) {
                      if (PK)
                        cap = true;  // sigma outgrew the packed field
                      else
                        of = true;
                    }
                  } else if (fused && val_side(v) != side) {
                    res = 2;
                  }
                  break;
                }
                pos = (pos + 1) & T.hmask;
              }
              if (k > T.hmask) cap = true;  // table full
            }
            const unsigned ins = __ballot_sync(FULL, res == 1);
            if (ins) {
              int at = 0;
              if (lane == 0) at = atomicAdd(&c.nlist, __popc(ins));
              at = __shfl_sync(FULL, at, 0) + __popc(ins & ((1u << lane) - 1u));
              if (res == 1) {
                if (at >= T.lcap) {
                  cap = true;
                } else {
                  if (!PK) T.lnode[at] = y;
                  lpos_set<PK>(T, at, pos);
                  cost += (unsigned)ydeg;
                  if (at - list_before < 32) c.fr[side][KIDX(at - list_before, 32, 17)] = make_int2(ylo, ydeg);
                  if (!PK && !ent_add<PK>(T, pos, add)) of = true;
                }
              }
            }
            if (fused) emit(fb, res == 2, p, y, (int)pos, w);
          });
        }
        if (sg + 1 < nseg) {
          __syncthreads();  // the next segment's prefix overwrites T.pr and the long rows
          if (RG && pass == 1) {
            if (tid == 0) c.nlong = 0;
            __syncthreads();
          }
        }
      }
      if (pass == 1) {
        if (!PK && __any_sync(FULL, sigma_of) && lane == 0) atomicOr(&c.lvl_flags, LF_TOUCH_SIGMA);
        __syncthreads();
        if (RG && tid == 0) c.nlong = 0;  // every thread has passed its last read of the long rows
        touched = c.npi > 0;
        if (touched) break;
      }
    }
    if (!touched) {
      if (tid == NT - 32) {
        if (last >= 0) lvl_hi(T, last, last == 0 ? depth0 : depth1) = list_before;
        lvl_lo(T, side, dnew) = list_before;
        c.acc[par ^ 1] = 0;  // the next level's
        c.hacc[par ^ 1] = 0;
      }
      cost = __reduce_add_sync(FULL, cost);
      hits = __reduce_add_sync(FULL, hits);
      if (lane == 0) {
        if (cost) atomicAdd(&c.acc[par], cost);
        if (hits) atomicAdd(&c.hacc[par], hits);
      }
      const int lf = (of ? LF_SIGMA : 0) | (cap ? LF_CAP : 0) | (sigma_of ? LF_TOUCH_SIGMA : 0);
      if (lf) atomicOr(&c.lvl_flags, lf);
      __syncthreads();
      if (PK && c.lvl_flags) {
        // (Packed levels only run out of room.)  A sigma that ran out of its
        // bits has carried into its entry's depth and side, so a one-pass
        // level's touches may be false: the next tier takes the sample, touch
        // or not.
        if (tid == 0) c.flags |= F_CAP;
        return;
      }
      if (fused && c.npi > 0) {
        // the level touches: undo its insertions (slots that were empty
        // before it) and choose among its touch arcs, as after pass 1
#pragma unroll 1
        for (int i = list_before + tid; i < c.nlist; i += NT) {
          const uint32_t q = lpos_get<PK>(T, i);
          T.hkv[q] = EMPTY;
          if (!PK) T.hsig[q] = 0ull;
        }
        __syncthreads();
        if (tid == 0) c.nlist = list_before;
        touched = true;
      }
    }
    if (touched) {
      if (tid == 0 && last >= 0) lvl_hi(T, last, last == 0 ? depth0 : depth1) = list_before;
      break;
    }
    const int lf = PK ? 0 : c.lvl_flags, nl = c.nlist;
    if (lf) {
      if (tid == 0) c.flags |= ((lf & LF_SIGMA) ? F_SIGMA : 0) | ((lf & LF_CAP) ? F_CAP : 0);
      return;
    }
    if (nl == list_before) return;  // frontier exhausted: s and t are not connected
    if (tid == NT - 32) {
      stat_add(c, KADABRA_STAT_NEW, (unsigned)(nl - list_before));
      stat_add(c, KADABRA_STAT_SIGMA_ADDS, c.hacc[par]);
    }
    if (side == 0) {
      depth0 = dnew;
      cost0 = (int)c.acc[par];
    } else {
      depth1 = dnew;
      cost1 = (int)c.acc[par];
    }
    last = side;
  }
  if (!touched) {  // loop bound reached (cannot happen within maxd levels)
    if (tid == 0) c.flags |= F_CAP;
    return;
  }

  // ------------------------------------------------ candidate-edge choice
  // Candidates are ordered by (x, y), x on the expanding side.
  const int total = c.npi;
  if (total > pi_cap || (!PK && (c.lvl_flags & LF_TOUCH_SIGMA))) {
    if (tid == 0) c.flags |= (total > pi_cap ? F_CAP : 0) | ((c.lvl_flags & LF_TOUCH_SIGMA) ? F_SIGMA : 0);
    return;
  }
  const int dv = depth0, dw = depth1;
  {
    PiEntry* const sh = reinterpret_cast<PiEntry*>(T.pr + cand_at);
    const int in_sh = PK ? min(total, cand_cap) : 0;  // the first of them are in shared memory
    if (tid == 0) {
      c.bt_dx[0] = dv;
      c.bt_dx[1] = dw;
      c.bt_j[0] = 2;
      c.bt_j[1] = 2 + (uint32_t)dv;
      stat_add(c, KADABRA_STAT_PI, (unsigned)total);
    }
    if (PK && total <= min(in_sh, NT)) {
      // Ranked quadratically in shared memory, all pairs spread over the
      // block: 2^sl neighbouring lanes share a candidate and each adds up
      // every 2^sl-th weight, both the total and that of the smaller keys, so
      // the draw's range needs no pass (and no barrier) of its own.  A packed
      // sigma has 24 bits: the sums fit 64.
      const int sl = total <= NT / 8 ? 3 : total <= NT / 4 ? 2 : total <= NT / 2 ? 1 : 0;
      const int i = tid >> sl;
      if (wid * 32 < total << sl) {
        const int4 me = reinterpret_cast<const int4*>(sh)[min(i, total - 1)];
        const unsigned long long key = ((unsigned long long)(uint32_t)me.x << 32) | (uint32_t)me.y;
        const unsigned long long mw = ((unsigned long long)(uint32_t)me.w << 32) | (uint32_t)me.z;
        unsigned long long all = 0, below = 0;
#pragma unroll 2
        for (int j = tid & ((1 << sl) - 1); j < total; j += 1 << sl) {
          const int4 e = reinterpret_cast<const int4*>(sh)[j];
          const unsigned long long w = ((unsigned long long)(uint32_t)e.w << 32) | (uint32_t)e.z;
          all += w;
          if ((((unsigned long long)(uint32_t)e.x << 32) | (uint32_t)e.y) < key) below += w;
        }
#pragma unroll 1
        for (int o = 1; o < 1 << sl; o <<= 1) {
          all += __shfl_xor_sync(FULL, all, o);
          below += __shfl_xor_sync(FULL, below, o);
        }
        const unsigned long long r = below128(c.draws[1], all);
        if (i < total && (tid & ((1 << sl) - 1)) == 0 && below <= r && r - below < mw) {
          c.pick = i;
          c.cand[0] = c.bt_x[0] = side == 0 ? me.x : me.y;
          c.cand[1] = c.bt_x[1] = side == 0 ? me.y : me.x;
          c.stat[KADABRA_STAT_SIGMA_LO] = (long long)(all & 0xFFFFFFFFull);
          c.stat[KADABRA_STAT_SIGMA_HI] = (long long)(all >> 32);
        }
      }
    } else {
      // the weights' 128-bit sum
#pragma unroll 1
      for (int i = tid; i < in_sh; i += NT) T.pi[i] = sh[i];
      unsigned long long lo = 0, hi = 0;
#pragma unroll 1
      for (int i = tid; i < total; i += NT) {
        const unsigned long long w = i < in_sh ? sh[i].w : T.pi[KIDX(i, pi_cap, 15)].w;
        lo += w;
        if (lo < w) ++hi;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long lo2 = __shfl_xor_sync(FULL, lo, o);
        hi += __shfl_xor_sync(FULL, hi, o);
        lo += lo2;
        if (lo < lo2) ++hi;
      }
      if (lane == 0) {
        c.wsum[wid] = lo;
        c.wsum_hi[wid] = hi;
      }
      __syncthreads();
      lo = hi = 0;
#pragma unroll 1
      for (int w = 0; w < NW; ++w) {
        lo += c.wsum[w];
        hi += c.wsum_hi[w] + (lo < c.wsum[w] ? 1ull : 0ull);
      }
      if (hi != 0) {
        if (tid == 0) c.flags |= F_SIGMA;
        return;
      }
      const unsigned long long r = below128(c.draws[1], lo);
      int pick;
      if (!PK && total <= QUAD_PICK_MAX) {
        pick = block_pick_by_key(
            total, r, c, [&](int i) { return ((unsigned long long)(uint32_t)T.pi[i].x << 32) | (uint32_t)T.pi[i].y; },
            [&](int i) { return T.pi[i].w; });
      } else {
        // its histogram (256 u64 weights, then 256 counts) takes the frontier array
        unsigned long long* kw = reinterpret_cast<unsigned long long*>(T.pr);
        pick = block_pick_radix(T.pi, total, r, c, kw, reinterpret_cast<unsigned*>(kw + 256));
      }
      if (tid == 0) {
        c.stat[KADABRA_STAT_SIGMA_LO] = (long long)(lo & 0xFFFFFFFFull);
        c.stat[KADABRA_STAT_SIGMA_HI] = (long long)(lo >> 32);
        c.pick = pick;
        if (pick >= 0) {
          const PiEntry e = T.pi[pick];
          c.cand[0] = c.bt_x[0] = side == 0 ? e.x : e.y;
          c.cand[1] = c.bt_x[1] = side == 0 ? e.y : e.x;
        }
      }
    }
  }
  __syncthreads();
  if (c.pick < 0) {
    if (tid == 0) c.flags |= F_INTERNAL;
    return;
  }

  // ------------------------------------------------ backtracking
  // The candidate edge joins the two current frontiers, so v is at depth0
  // on the s side and w at depth1 on the t side.
  const bool want_path = P.paths != nullptr && out_i >= 0;
  KSTAGGER(wid >= 2);
  if (tid == NT - 1) {  // a warp that does not walk; the walkers change bt_x meanwhile
    const int cv = c.cand[0], cw = c.cand[1];
    c.stat[KADABRA_STAT_DIST] = dv + 1 + dw;
    c.stat[KADABRA_STAT_PATH_NODES] = dv + dw + 2;
    if (want_path) {
      int32_t* row = P.paths + out_i * (int64_t)P.max_len;
      if (dv < P.max_len) row[dv] = cv;
      if (dv + 1 < P.max_len) row[dv + 1] = cw;
    }
    if (J.counts) {
      if (dv > 0) atomicAdd(&J.counts[KIDX(cv, J.g.n, 11)], 1u);
      if (dw > 0) atomicAdd(&J.counts[KIDX(cw, J.g.n, 11)], 1u);
    }
  }
  // Steps go one node at a time, v -> s over predecessors (walker 0, weights
  // sigma_s) and w -> t over successors (walker 1).  The s side takes the
  // Philox blocks 2 .. dv + 1 and the t side the next dw, so the two walkers
  // are independent: warp 0 walks the first and warp 1 the second, at the
  // same time, taking the steps whose candidates are few (a single node one
  // level closer, or a row of up to WARP_BT_ROW arcs) with warp scans only.
  // A longer step goes to the whole block.  Both choose the same node with
  // the same draw.  The state between them (node, depth, next draw) lives in
  // c.bt_*[walker].
#pragma unroll 1
  for (;;) {
    if (wid < 2) bt_warp_steps<PK>(P, J, T, c, idx, out_i, dv, dw, want_path, wid);
    __syncthreads();
    if (c.bt_flag) {
      if (tid == 0) c.flags |= F_INTERNAL;
      return;
    }
    const int half = c.bt_dx[0] > 0 ? 0 : c.bt_dx[1] > 0 ? 1 : -1;
    if (half < 0) break;
    // one long step of that walker, by the whole block
    const int x = c.bt_x[half], dx = c.bt_dx[half];
    const uint32_t j = c.bt_j[half];
    // the row of x that holds its neighbours one level closer to the root
    const int32_t* brow = half == 0 ? G.rrp : G.rp;
    const int32_t* bcol = half == 0 ? G.rci : G.ci;
    // the opposite direction, to test adjacency from a previous-level node
    const int32_t* frow = half == 0 ? G.rp : G.rrp;
    const int32_t* fcol = half == 0 ? G.ci : G.rci;
    const int plo = lvl_lo(T, half, dx - 1), phi = lvl_hi(T, half, dx - 1);
    const uint32_t want = pack_val(half, dx - 1);
    const int r0 = __ldg(&brow[x]), deg = __ldg(&brow[x + 1]) - r0;
    __syncthreads();  // every thread has read c.bt_*[half] before thread 0 writes below
    if (tid == 0) {
      const int px = tab_find_pos(T, x);
      if (px < 0) {
        c.bt_flag = 1;  // reported below, after every thread has decided
        c.r = 0;
      } else {
        c.r = below128(j < 32 ? c.draws[j] : draw_late(J.seed, J.domain, idx, j),
                       ent_sig<PK>(T, T.hkv[px], (uint32_t)px));
      }
      // scan whichever is shorter: the row of x, or the previous level
      c.mode = ((long long)(phi - plo) * 16 < (long long)deg) ? 1 : 0;
      c.ecount = 0;  // candidates found in the previous level (mode 1)
      c.pick = -1;
    }
    __syncthreads();
    if (c.bt_flag) {
      if (tid == 0) c.flags |= F_INTERNAL;
      return;
    }
    const unsigned long long r = c.r;
    bool by_level = c.mode == 1;
    if (by_level) {
      // previous-level nodes adjacent to x, collected as (node, hash position)
#pragma unroll 1
      for (int i = plo + tid; i < phi; i += NT) {
        const int y = list_node<PK>(T, i);
        const int a = __ldg(&frow[y]), b = __ldg(&frow[y + 1]);
        const int at = lower_bound_row(fcol, a, b, x);
        if (at < b && __ldg(&fcol[at]) == x) {
          const int q = atomicAdd(&c.ecount, 1);
          if (q < T.frcap) T.pr[q] = make_int2(y, (int)lpos_get<PK>(T, i));
        }
      }
      __syncthreads();
      if (c.ecount > min(T.frcap, 128)) by_level = false;  // many predecessors: scan the row instead
    }
    int y_pick = -1, pos_pick = 0;
    if (by_level) {
      const int nc = c.ecount;
      const int pick = block_pick_by_key(
          nc, r, c, [&](int i) { return (unsigned long long)(uint32_t)T.pr[i].x; },
          [&](int i) {
            const uint32_t q = (uint32_t)T.pr[i].y;
            return ent_sig<PK>(T, T.hkv[q], q);
          });
      if (pick >= 0) y_pick = T.pr[pick].x;
      if (wid == 0 && pick >= 0) pos_pick = warp_lower_bound(bcol, r0, r0 + deg, y_pick) - r0;
    } else {
      const int pick = block_pick(deg, r, c, [&](int i0, int N, unsigned long long* w) {
        int ys[U];
#pragma unroll
        for (int k = 0; k < U; ++k) ys[k] = (i0 + k < N) ? __ldg(&bcol[r0 + i0 + k]) : -1;
#pragma unroll
        for (int k = 0; k < U; ++k) {
          w[k] = 0;
          if (ys[k] >= 0) {
            const int pos = tab_find_pos(T, ys[k]);
            if (pos >= 0) {
              const unsigned long long hw = T.hkv[pos];
              if (ent_val<PK>(hw) == want) w[k] = ent_sig<PK>(T, hw, (uint32_t)pos);
            }
          }
        }
      });
      if (pick >= 0) {
        y_pick = __ldg(&bcol[r0 + pick]);
        pos_pick = pick;
      }
    }
    if (y_pick < 0) {
      if (tid == 0) c.flags |= F_INTERNAL;
      return;
    }
    if (tid == 0) {
      bt_record<PK>(P, J, c, half, dx - 1, y_pick, pos_pick, out_i, dv, dw, want_path);
      c.bt_x[half] = y_pick;
      c.bt_dx[half] = dx - 1;
      c.bt_j[half] = j + 1;
    }
    __syncthreads();
  }
}

// Clears what the last sample left in the hash table of a global-memory tier
// (key and sigma of every entry it inserted): the whole table after a
// capacity failure (entries beyond the lists), else the entries at the
// positions the lists recorded.
template <int NW>
__device__ void reset_tables(const Tables& T, Ctl<NW>& c) {
  constexpr int NT = 32 * NW;
  const int tid = threadIdx.x;
  if (c.flags & F_CAP) {
#pragma unroll 1
    for (uint32_t i = tid; i <= T.hmask; i += NT) {
      T.hkv[i] = EMPTY;
      T.hsig[i] = 0ull;
    }
  } else {
    const int nl = min(c.nlist, T.lcap);
#pragma unroll 1
    for (int i = tid; i < nl; i += NT) {
      const uint32_t pos = lpos_get<false>(T, i);
      T.hkv[pos] = EMPTY;
      T.hsig[pos] = 0ull;
    }
  }
  __syncthreads();
}

// Empties a shared-memory table (cheaper than locating a sample's entries):
// every warp but the first, which meanwhile sets up the next sample.
template <int NW>
__device__ __forceinline__ void clear_table(const Tables& T) {
  constexpr int NT = 32 * NW;
  int4* h = reinterpret_cast<int4*>(T.hkv);
#pragma unroll 1
  for (uint32_t i = threadIdx.x - 32; i < (T.hmask + 1) / 2; i += NT - 32) h[i] = make_int4(-1, -1, -1, -1);
}

// The draw and control state of a sample (warp 0; the roots go into the
// table afterwards).  Every lane draws one of the sample's first 32 Philox
// blocks ((s,t), candidate edge, backtracking steps), so the serial steps
// only read them.
template <int NW>
__device__ __forceinline__ void begin_sample(const SampleParams& P, const Tables& T, Ctl<NW>& c, uint64_t idx,
                                             int64_t out_i) {
  const int lane = lane_id();
  const GraphDev& G = c.job.g;
  const uint4 b = draw(c.job.seed, c.job.domain, idx, (uint32_t)lane);
  c.draws[lane] = b;
  int s, t;
  draw_pair(make_uint4(__shfl_sync(FULL, b.x, 0), __shfl_sync(FULL, b.y, 0), __shfl_sync(FULL, b.z, 0),
                       __shfl_sync(FULL, b.w, 0)),
            G.n, &s, &t);
  int bound = 0;  // lanes 0..3: the two roots' row bounds
  if (lane < 4) bound = __ldg((lane < 2 ? G.rp + s : G.rrp + t) + (lane & 1));
  if (lane < KADABRA_NSTAT) c.stat[lane] = lane == KADABRA_STAT_DIST ? -1 : 0;
  const int deg = __shfl_down_sync(FULL, bound, 1) - bound;
  if (lane == 0) {
    c.s = s;
    c.t = t;
    c.flags = 0;
    c.lvl_flags = 0;
    c.bt_flag = 0;
    c.npi = 0;
    c.pick = -1;
    c.acc[0] = c.acc[1] = c.hacc[0] = c.hacc[1] = 0;
    c.nlist = 2;
    lvl_lo(T, 0, 0) = 0;
    lvl_hi(T, 0, 0) = 1;
    lvl_lo(T, 1, 0) = 1;
    lvl_hi(T, 1, 0) = 2;
    c.fside = -1;
    c.nlong = 0;
    c.cost[0] = (unsigned)deg;
  }
  if (lane == 0 || lane == 2) c.fr[lane >> 1][0] = make_int2(bound, deg);
  if (lane == 2) c.cost[1] = (unsigned)deg;
  if (out_i >= 0 && P.paths)
#pragma unroll 1
    for (int q = lane; q < P.max_len; q += 32) P.paths[out_i * (int64_t)P.max_len + q] = -1;
  __syncwarp();
}

// s and t into the (empty) table: the level 0 of both sides (warp 0)
template <bool PK, int NW>
__device__ __forceinline__ void insert_roots(const Tables& T, Ctl<NW>& c) {
  if (threadIdx.x == 0) {
    uint32_t ps = 0, pt = 0;
    if (tab_insert(T, c.s, ent_word<PK>(c.s, pack_val(0, 0), 1ull), &ps) != 1) c.flags |= F_INTERNAL;
    if (tab_insert(T, c.t, ent_word<PK>(c.t, pack_val(1, 0), 1ull), &pt) != 1) c.flags |= F_INTERNAL;
    if (!PK) {
      T.hsig[ps] = 1ull;
      T.hsig[pt] = 1ull;
      T.lnode[0] = c.s;
      T.lnode[1] = c.t;
    }
    lpos_set<PK>(T, 0, ps);
    lpos_set<PK>(T, 1, pt);
  }
  __syncwarp();
}

// global-memory tiers share one body per scan kind, compiled outside the kernel
template <bool RG, int NW>
__device__ __noinline__ void run_sample_global(const SampleParams& P, const Job& J, const Tables& T, Ctl<NW>& c,
                                               uint64_t idx, int64_t out_i) {
  if (warp_id() == 0) {
    begin_sample(P, T, c, idx, out_i);
    insert_roots<false>(T, c);
  }
  __syncthreads();
  run_sample<false, RG>(P, J, T, c, idx, out_i);
  __syncthreads();
}

// layout of one CTA's tables in global memory (tiers M and L)
__host__ __device__ inline size_t gm_layout(int hlog, int lcap, int maxd, size_t* off_pr, size_t* off_lnode,
                                            size_t* off_lpos, size_t* off_lvl) {
  size_t o = (2 * sizeof(unsigned long long)) << hlog;  // hkv, then hsig
  *off_pr = o;
  // the radix selection's histogram (RADIX_HIST) takes the frontier array, whatever the lists' capacity
  const size_t frontier = sizeof(int2) * ((size_t)lcap + 1);
  o += frontier > RADIX_HIST ? frontier : RADIX_HIST;
  *off_lnode = o;
  o += sizeof(int32_t) * (size_t)lcap;
  *off_lpos = o;
  o += sizeof(uint32_t) * (size_t)lcap;
  *off_lvl = o;
  o += sizeof(int) * 4 * (size_t)(maxd + 2);
  return (o + 255) & ~size_t(255);
}

__device__ inline Tables gm_tables(unsigned char* base, int hlog, int lcap, int maxd) {
  size_t o_pr, o_lnode, o_lpos, o_lvl;
  gm_layout(hlog, lcap, maxd, &o_pr, &o_lnode, &o_lpos, &o_lvl);
  Tables T;
  T.hkv = reinterpret_cast<unsigned long long*>(base);
  T.hsig = reinterpret_cast<unsigned long long*>(base + (sizeof(unsigned long long) << hlog));
  T.pr = reinterpret_cast<int2*>(base + o_pr);
  T.lnode = reinterpret_cast<int32_t*>(base + o_lnode);
  T.lpos = reinterpret_cast<uint32_t*>(base + o_lpos);
  T.lvl = reinterpret_cast<int*>(base + o_lvl);
  T.hlog = hlog;
  T.hmask = (1u << hlog) - 1u;
  T.lcap = lcap;
  T.frcap = lcap;
  T.lpos16 = nullptr;
  T.lr = nullptr;  // set by the kernel
  T.bits = nullptr;
  T.fwords = 0;
  T.fshift = 32;
  T.maxd = maxd;
  return T;
}

// shared-memory layout of a packed tier after the control block: 2^HLOG
// hash slots, lists of L8 eighths of the slots (hash positions), frontier
// segments of FSEG nodes (the frontier array's capacity), a 2^FLOG-bit
// filter and MAXD levels per side.  The scan variant for graphs beyond the
// L2 has the same layout.
#ifndef KD_FRONTIER_SEG
#define KD_FRONTIER_SEG 1024
#endif
constexpr int FRONTIER_SEG = KD_FRONTIER_SEG;
#ifndef KD_LOAD_QUARTERS
#define KD_LOAD_QUARTERS 3
#endif
template <int NW>
constexpr size_t CTL_BYTES = (sizeof(Ctl<NW>) + 15) & ~size_t(15);
template <int NW, int HLOG, int L8, int FSEG, int FLOG, int MAXD, bool LR>
struct SLayout {
  static constexpr int SLOTS_LOG = HLOG;
  // nodes a table takes before the sample moves on to the next tier (the
  // probes stay short)
  static constexpr int LCAP = (L8 << HLOG) / 8;
  static_assert(LCAP + 32 * NW < (1 << HLOG), "a full list leaves free slots");
  static constexpr int FRCAP = LCAP < FSEG ? LCAP : FSEG;
  static constexpr int FWORDS = (1 << FLOG) / 32;
  static constexpr int FSHIFT = 32 - FLOG;
  static constexpr int LEVELS = MAXD;
  static_assert(MAXD <= 126, "the packed entry's dist field");
  static constexpr size_t HKV = CTL_BYTES<NW>;
  static constexpr size_t PR = HKV + (sizeof(unsigned long long) << HLOG);
  static constexpr size_t LPOS = PR + sizeof(int2) * (FRCAP + 1);
  static constexpr size_t LVL = LPOS + sizeof(uint16_t) * LCAP;
  static constexpr size_t BITS = (LVL + sizeof(int) * 4 * (MAXD + 2) + 15) & ~size_t(15);
  static constexpr size_t LONG = BITS + sizeof(uint32_t) * FWORDS;
  static constexpr size_t BYTES = LONG + (LR ? sizeof(LongRows) : 0);
  static_assert(HLOG <= 16, "16-bit list positions");
  // the radix selection's histogram (256 u64 + 256 u32) in the frontier array
  static_assert(sizeof(int2) * (FRCAP + 1) >= RADIX_HIST,
                "frontier array holds the selection histogram");
};
// tier S at KD_MIN_BLOCKS CTAs per SM; tier S compact (one more CTA per SM:
// half-full lists, 512-node segments, a 2^14-bit filter, 38 levels per
// side; 45,328 B, of which five fit an SM's shared memory up to 45,408 B);
// tier B (four times the slots, one CTA per SM); the small layout.
#ifndef KD_CMP_L8
#define KD_CMP_L8 4
#endif
#ifndef KD_CMP_FLOG
#define KD_CMP_FLOG 14
#endif
#ifndef KD_CMP_MAXD
#define KD_CMP_MAXD 38
#endif
using FastLayout = SLayout<NW_S, FAST_HLOG, 2 * KD_LOAD_QUARTERS, FRONTIER_SEG, FILTER_LOG, FAST_MAXD, true>;
using CompactLayout = SLayout<NW_CMP, FAST_HLOG, KD_CMP_L8, 512, KD_CMP_FLOG, KD_CMP_MAXD, false>;
using BigLayout = SLayout<NW_BIG, BIG_HLOG, 2 * KD_LOAD_QUARTERS, FRONTIER_SEG, FILTER_LOG, FAST_MAXD, true>;
using TinyLayout = SLayout<NW_TINY, 11, 6, 512, 13, KD_CMP_MAXD, false>;
// the tier-S layout a k_sample instance uses (SL)
constexpr int SL_FAST = 0;
constexpr int SL_COMPACT = 1;
constexpr int SL_TINY = 2;
template <int SL>
using TierSLayout = std::conditional_t<SL == SL_FAST, FastLayout, std::conditional_t<SL == SL_TINY, TinyLayout, CompactLayout>>;

template <class L>
__device__ inline Tables smem_tables(unsigned char* smem) {
  Tables T;
  T.hkv = reinterpret_cast<unsigned long long*>(smem + L::HKV);
  T.hsig = nullptr;  // packed entries
  T.pr = reinterpret_cast<int2*>(smem + L::PR);
  T.lnode = nullptr;  // node ids come from the hash words
  T.lpos = nullptr;
  T.lpos16 = reinterpret_cast<uint16_t*>(smem + L::LPOS);
  T.lvl = reinterpret_cast<int*>(smem + L::LVL);
  T.bits = reinterpret_cast<uint32_t*>(smem + L::BITS);
  T.lr = L::BYTES > L::LONG ? reinterpret_cast<LongRows*>(smem + L::LONG) : nullptr;
  T.fwords = L::FWORDS;
  T.fshift = L::FSHIFT;
  T.hlog = L::SLOTS_LOG;
  T.hmask = (1u << L::SLOTS_LOG) - 1u;
  T.lcap = L::LCAP;
  T.frcap = L::FRCAP;
  T.maxd = L::LEVELS;
  return T;
}

// flags of SampleParams::tier_flags (test switches: skip tiers)
constexpr int TF_SKIP_S = 1;
constexpr int TF_SKIP_B = 2;
constexpr int TF_SKIP_M = 4;
constexpr int TF_WARP = 8;  // tier W first, whatever the launch's variant
constexpr int TF_VEC = 16;  // pass 1 searches long rows (graphs beyond the L2)
constexpr int TF_SEG64 = 32;  // shared-memory tiers scan frontiers in 64-node segments (tests)
constexpr int TF_COMPACT = 64;  // tier S in the compact layout, whatever the launch's variant
constexpr int TF_SCREEN = 128;  // k_screen first: tier S takes only the samples whose roots have arcs
constexpr int TF_TINY = 256;  // the small layout where the launch's variant asks for the compact one

// queue counters in SampleParams::ctr
constexpr int Q_NEXT_A = 0;   // next sample index of the batch
constexpr int Q_NEXT_B = 1;   // next entry of the tier-B queue
constexpr int Q_SIZE_B = 2;   // entries in the tier-B queue
constexpr int Q_NEXT_L = 3;   // next entry of the tier-L queue
constexpr int Q_SIZE_L = 4;   // entries in the tier-L queue
constexpr int Q_NEXT_W = 5;   // next sample index of tier W
constexpr int Q_SIZE_S = 6;   // entries tier W queued for tier S
constexpr int Q_COUNT = 8;

__device__ void enqueue(const SampleParams& P, int size_ctr, unsigned long long* q, uint64_t idx) {
  const unsigned long long d = atomicAdd(&P.ctr[size_ctr], 1ull);
  if (d < P.deferred_cap)
    q[d] = idx;
  else
    atomicCAS(P.status, 0, (int)KADABRA_ERR_CAPACITY);
}

// Adds the CTA's accumulated work counters to their job's totals (warp 0).
template <int NW>
__device__ void flush_totals(const SampleParams& P, Ctl<NW>& c) {
  const int q = lane_id();
  if (q < KADABRA_NSTAT) {
    if (c.tot_job >= 0) {
      long long* t = P.jobs ? P.jobs[c.tot_job].totals : P.job0.totals;
      if (t && c.tot[q]) atomicAdd((unsigned long long*)&t[q], (unsigned long long)c.tot[q]);
    }
    c.tot[q] = 0;
  }
  __syncwarp();
}

// The job of work index k into c.job (warp 0).
template <int NW>
__device__ __forceinline__ void take_job(const SampleParams& P, Ctl<NW>& c, unsigned long long k) {
  int j = 0;
  if (P.jobs) {
    int lo = 0, hi = P.njobs;
#pragma unroll 1
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (P.jobs[mid].work_begin <= k)
        lo = mid;
      else
        hi = mid;
    }
    j = lo;
  }
  if (j == c.tot_job) return;
  flush_totals(P, c);  // the counters so far belong to another job
  static_assert(sizeof(Job) % 4 == 0 && sizeof(Job) / 4 <= 32, "a lane copies one word");
  const int q = lane_id();
  if (q < (int)(sizeof(Job) / 4))
    reinterpret_cast<uint32_t*>(&c.job)[q] = reinterpret_cast<const uint32_t*>(P.jobs ? &P.jobs[j] : &P.job0)[q];
  if (q == 0) c.tot_job = j;
  __syncwarp();
}

// Records the outcome of one sample (per-sample outputs, totals, status; warp 0).
template <int NW>
__device__ void finish_sample(const SampleParams& P, Ctl<NW>& c, int64_t out_i) {
  int flags = c.flags;
#ifdef KADABRA_CHECKED
  if (*(volatile unsigned long long*)&g_checked) flags |= F_INTERNAL;
#endif
  int st = KADABRA_OK;
  if (flags & F_INTERNAL)
    st = KADABRA_ERR_INTERNAL;
  else if (flags & F_SIGMA)
    st = KADABRA_ERR_SIGMA_OVERFLOW;
  else if (flags & F_CAP)
    st = KADABRA_ERR_CAPACITY;
  const int q = lane_id();
  if (q == 0 && st != KADABRA_OK) atomicCAS(P.status, 0, st);
  if (q < KADABRA_NSTAT) {
    const long long x = c.stat[q];
    if (q != KADABRA_STAT_SIGMA_LO && q != KADABRA_STAT_SIGMA_HI && q != KADABRA_STAT_DIST) c.tot[q] += x;
    if (out_i >= 0 && P.stats) P.stats[out_i * KADABRA_NSTAT + q] = x;
  }
  if (q == 0 && out_i >= 0) {
    P.st_out[2 * out_i] = c.s;
    P.st_out[2 * out_i + 1] = c.t;
    if (P.path_len) P.path_len[out_i] = (int32_t)c.stat[KADABRA_STAT_PATH_NODES];
    if (P.sstatus) P.sstatus[out_i] = st;
  }
  __syncwarp();
}

// MODE 0: every sample of the batch, on tier S; overflow -> tier-B queue.
// MODE 2: the tier-B queue, on tier B, then tier M; overflow -> tier-L queue.
// MODE 1: the tier-L queue, on tier L.
// SL: the tier-S layout of MODE 0; the compact and the small one fit more CTAs
// per SM and give the same results (samples that outgrow them go on to tier B
// as usual).  RG (the default layout only): pass 1 searches long rows (for
// graphs whose CSR exceeds L2); same results.
template <int MODE, int SL = SL_FAST>
constexpr int MODE_NW = MODE == 2 ? NW_BIG : SL == SL_COMPACT ? NW_CMP : SL == SL_TINY ? NW_TINY : NW_S;
template <int MODE, int SL>
constexpr int MODE_CTAS =
    MODE == 2 ? 1 : MODE == 1 ? 2 : SL == SL_FAST ? KD_MIN_BLOCKS : SL == SL_TINY ? 7 : KD_MIN_BLOCKS + 1;
template <int MODE, int SL = SL_FAST, bool RG = false>
__global__ void __launch_bounds__(32 * MODE_NW<MODE, SL>, MODE_CTAS<MODE, SL>)
    k_sample(SampleParams P) {
  static_assert(!RG || SL == SL_FAST, "the beyond-L2 scan has no compact-layout instance");
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NW = MODE_NW<MODE, SL>;
  Ctl<NW>& c = *reinterpret_cast<Ctl<NW>*>(smem);
  Tables TS, TM;
  PiEntry* pi = P.pi_base + (size_t)blockIdx.x * PI_SEGS * P.pcap;
  if (MODE == 0) TS = smem_tables<TierSLayout<SL>>(smem);
  if (MODE == 2) {
    TS = smem_tables<BigLayout>(smem);
    TM = gm_tables(P.med_base + (size_t)blockIdx.x * P.med_stride, P.med_hlog, P.med_lcap, MED_MAXD);
  }
  if (MODE == 1) TM = gm_tables(P.gm_base + (size_t)blockIdx.x * P.gm_stride, P.gm_hlog, P.gm_lcap, GM_MAXD);
  if (MODE == 2) TM.lr = TS.lr;
  if (MODE == 1) TM.lr = reinterpret_cast<LongRows*>(smem + CTL_BYTES<NW>);
  TS.pi = TM.pi = pi;
  TS.pcap = TM.pcap = P.pcap;
  if (MODE != 1 && (P.tier_flags & TF_SEG64)) TS.frcap = min(TS.frcap, 64);

  const int tid = threadIdx.x;
  if (tid == 0) {
#pragma unroll 1
    for (int k = 0; k < KADABRA_NSTAT; ++k) c.tot[k] = 0;
    c.tot_job = -1;
    c.ntotal = MODE == 0 ? (P.q0 ? min(P.ctr[Q_SIZE_S], (unsigned long long)P.deferred_cap)
                                 : (P.total_dev ? *P.total_dev : P.total_work))
               : MODE == 2 ? min(P.ctr[Q_SIZE_B], (unsigned long long)P.deferred_cap)
                           : min(P.ctr[Q_SIZE_L], (unsigned long long)P.deferred_cap);
  }
  __syncthreads();
  const unsigned long long ntotal = c.ntotal;
  if (ntotal == 0) return;  // nothing queued for this tier: skip the table set-up (the whole block)

  // Between two samples (two barriers) warp 0 records the last one, takes
  // the next index and sets its sample up, while the other warps empty the
  // shared-memory table.
  bool finish = false;       // a sample to record (warp 0)
#pragma unroll 1
  for (;;) {
    if (tid < 32) {
      unsigned long long cur = 0;
      if (tid == 0) cur = atomicAdd(&P.ctr[MODE == 0 ? Q_NEXT_A : MODE == 2 ? Q_NEXT_B : Q_NEXT_L], 1ull);
      if (finish) {
        const unsigned long long k = c.k;  // the sample's index in the launch's work space
        if (MODE != 1 && c.flags == F_CAP) {  // to the next tier
          if (tid == 0) enqueue(P, MODE == 0 ? Q_SIZE_B : Q_SIZE_L, MODE == 0 ? P.qb : P.ql, k);
        } else {
          finish_sample(P, c, P.st_out ? (int64_t)k : -1);
        }
      }
      finish = true;
      cur = __shfl_sync(FULL, cur, 0);
      if (cur < ntotal) {
        const unsigned long long k = MODE == 0 ? (P.q0 ? P.q0[cur] : cur) : MODE == 2 ? P.qb[cur] : P.ql[cur];
        take_job(P, c, k);
        if (MODE != 1) begin_sample(P, TS, c, c.job.first_idx + (k - c.job.work_begin), P.st_out ? (int64_t)k : -1);
        if (tid == 0) c.k = k;
      }
      if (tid == 0) c.cur = cur;
    } else if (MODE != 1) {
      clear_table<NW>(TS);
    }
    __syncthreads();
    if (c.cur >= ntotal) break;
    const uint64_t idx = c.job.first_idx + (c.k - c.job.work_begin);
    const int64_t out_i = P.st_out ? (int64_t)c.k : -1;
    if (MODE == 0) {
      if (!(P.tier_flags & TF_SKIP_S)) {
        if (tid < 32) insert_roots<true>(TS, c);
        run_sample<true, RG>(P, c.job, TS, c, idx, out_i);
      } else if (tid == 0) {
        c.flags = F_CAP;
      }
      __syncthreads();
    } else if (MODE == 2) {
      bool done = false;
      if (!(P.tier_flags & TF_SKIP_B)) {
        if (tid < 32) insert_roots<true>(TS, c);
        run_sample<true, RG>(P, c.job, TS, c, idx, out_i);
        __syncthreads();
        done = c.flags != F_CAP;
        __syncthreads();
      }
      if (!done && !(P.tier_flags & TF_SKIP_M)) {
        run_sample_global<RG>(P, c.job, TM, c, idx, out_i);
        reset_tables(TM, c);
      } else if (!done) {
        if (tid == 0) c.flags = F_CAP;
        __syncthreads();
      }
    } else {
      run_sample_global<RG>(P, c.job, TM, c, idx, out_i);
      reset_tables(TM, c);
    }
  }
  if (tid < 32) flush_totals(P, c);
}

// ============================================================== screening
// The samples whose s has no out-arc or whose t has no in-arc end at their
// first level: one level, one expanded node, no arc.  One thread draws and
// records such a sample; the others' work indices go to tier S's queue.  On
// directed graphs with many such nodes most samples end here (R-MAT scale 22:
// 65,536 samples 1.81 -> 1.65 ms).
__global__ void __launch_bounds__(256) k_screen(const __grid_constant__ SampleParams P) {
  const int lane = lane_id();
  const unsigned long long ntotal = P.total_dev ? *P.total_dev : P.total_work;
  for (unsigned long long base = blockIdx.x * 256ull; base < ntotal; base += gridDim.x * 256ull) {
    const unsigned long long k = base + threadIdx.x;
    bool idle = false, push = false;
    int j = 0;
    if (k < ntotal) {
      if (P.jobs) {
        int lo = 0, hi = P.njobs;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (P.jobs[mid].work_begin <= k)
            lo = mid;
          else
            hi = mid;
        }
        j = lo;
      }
      const Job& J = P.jobs ? P.jobs[j] : P.job0;
      int s, t;
      draw_pair(draw(J.seed, J.domain, J.first_idx + (k - J.work_begin), 0), J.g.n, &s, &t);
      idle = __ldg(&J.g.rp[s]) == __ldg(&J.g.rp[s + 1]) || __ldg(&J.g.rrp[t]) == __ldg(&J.g.rrp[t + 1]);
      push = !idle;
      if (idle && P.st_out) {
        P.st_out[2 * k] = s;
        P.st_out[2 * k + 1] = t;
        if (P.path_len) P.path_len[k] = 0;
        if (P.paths)
          for (int q = 0; q < P.max_len; ++q) P.paths[(int64_t)k * P.max_len + q] = -1;
        if (P.stats)
          for (int q = 0; q < KADABRA_NSTAT; ++q)
            P.stats[(int64_t)k * KADABRA_NSTAT + q] =
                q == KADABRA_STAT_LEVELS || q == KADABRA_STAT_EXPANDED ? 1 : q == KADABRA_STAT_DIST ? -1 : 0;
        if (P.sstatus) P.sstatus[k] = KADABRA_OK;
      }
    }
    const unsigned go = __ballot_sync(FULL, push);
    if (go) {
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(&P.ctr[Q_SIZE_S], (unsigned long long)__popc(go));
      at = __shfl_sync(FULL, at, 0) + __popc(go & ((1u << lane) - 1u));
      if (push) {
        if (at < P.deferred_cap)
          P.q0[at] = k;
        else
          atomicCAS(P.status, 0, (int)KADABRA_ERR_CAPACITY);
      }
    }
    // the idle samples' counters, once per warp and job
    const unsigned same = __match_any_sync(FULL, idle ? j : -1);
    if (idle && lane == __ffs(same) - 1) {
      long long* tot = P.jobs ? P.jobs[j].totals : P.job0.totals;
      if (tot) {
        atomicAdd((unsigned long long*)&tot[KADABRA_STAT_LEVELS], (unsigned long long)__popc(same));
        atomicAdd((unsigned long long*)&tot[KADABRA_STAT_EXPANDED], (unsigned long long)__popc(same));
      }
    }
  }
}

// ============================================================== tier W: one warp per sample
// Eight independent samples per CTA, one per warp, each on a small packed
// table in shared memory, synchronised by warp only.  For graphs whose
// searches stay small, this gives more samples in flight and no block
// barriers.  A sample that outgrows the table (more nodes, candidate edges
// or levels than below, or a sigma beyond the packed field) is queued
// for tier S, which gives the same result; hits are counted only in the
// backtracking, which never escalates, so nothing is counted twice.
constexpr int WT_HLOG = 9;
constexpr int WT_HSIZE = 1 << WT_HLOG;  // 512 hash slots
constexpr int WT_LCAP = 256;            // level-list nodes
constexpr int WT_PCAP = 128;            // candidate edges
constexpr int WT_MAXD = FAST_MAXD;      // levels per side (the packed dist field)
constexpr int WT_WARPS = 8;             // samples per CTA

struct WSlot {  // one warp's shared memory
  unsigned long long hkv[WT_HSIZE];  // packed entries, as in tier S
  int2 pr[WT_LCAP + 1];              // frontier: {degree prefix, row start}
  int32_t lnode[WT_LCAP];
  uint32_t lpos[WT_LCAP];
  PiEntry pi[WT_PCAP];
  Job job;
  long long stat[KADABRA_NSTAT];
  long long tot[KADABRA_NSTAT];
  int tot_job;
  int s, t;
};

__device__ __forceinline__ int wt_probe(const unsigned long long* h, int32_t v, unsigned long long* wo) {
  uint32_t pos = hash_pos(v, WT_HLOG);
  for (int k = 0; k < WT_HSIZE; ++k) {
    const unsigned long long w = h[pos];
    if (w == EMPTY) return -1;
    if ((int32_t)(w >> 32) == v) {
      *wo = w;
      return (int)pos;
    }
    pos = (pos + 1) & (WT_HSIZE - 1);
  }
  return -1;
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// One sample by one warp (all lanes call it); the same search, choices and
// random draws as run_sample.  Returns 0, or F_CAP (escalate to tier S), or
// F_INTERNAL.  Leaves the work counters in S.stat.
__device__ int run_sample_warp(const SampleParams& P, const Job& J, WSlot& S, uint64_t idx, int64_t out_i) {
  const int lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  const GraphDev& G = J.g;
  const uint4 myd = draw(J.seed, J.domain, idx, (uint32_t)lane);  // this lane's block j = lane
  auto dr = [&](uint32_t j) {  // block j, same j in all lanes
    uint4 b;
    if (j < 32u) {
      b.x = __shfl_sync(FULL, myd.x, (int)j);
      b.y = __shfl_sync(FULL, myd.y, (int)j);
      b.z = __shfl_sync(FULL, myd.z, (int)j);
      b.w = __shfl_sync(FULL, myd.w, (int)j);
    } else {
      b = draw(J.seed, J.domain, idx, j);
    }
    return b;
  };
  if (lane < KADABRA_NSTAT) S.stat[lane] = lane == KADABRA_STAT_DIST ? -1 : 0;
  const uint4 b0 = dr(0);
  const uint64_t u = (uint64_t)b0.x | ((uint64_t)b0.y << 32);
  const uint64_t u2 = (uint64_t)b0.z | ((uint64_t)b0.w << 32);
  const int s = (int)__umul64hi(u, (uint64_t)G.n);
  const int tp = (int)__umul64hi(u2, (uint64_t)(G.n - 1));
  const int t = tp + (tp >= s ? 1 : 0);
  if (lane == 0) {
    S.s = s;
    S.t = t;
    uint32_t ps = hash_pos(s, WT_HLOG);
    while (S.hkv[ps] != EMPTY) ps = (ps + 1) & (WT_HSIZE - 1);
    S.hkv[ps] = ent_word<true>(s, pack_val(0, 0), 1ull);
    uint32_t pt = hash_pos(t, WT_HLOG);
    while (S.hkv[pt] != EMPTY) pt = (pt + 1) & (WT_HSIZE - 1);
    S.hkv[pt] = ent_word<true>(t, pack_val(1, 0), 1ull);
    S.lnode[0] = s;
    S.lpos[0] = ps;
    S.lnode[1] = t;
    S.lpos[1] = pt;
  }
  __syncwarp();
  int dep[2] = {0, 0}, flo[2] = {0, 1}, fhi[2] = {1, 2};
  long long cst[2] = {G.rp[s + 1] - G.rp[s], G.rrp[t + 1] - G.rrp[t]};
  int nlist = 2, done = 0, side = 0, npi = 0;
  long long n_lev = 0, n_exp = 0, n_edges = 0, n_new = 0, n_adds = 0;

  // ------------------------------------------------ bb-BFS (Sec. 4)
  for (int iter = 0; iter <= 2 * WT_MAXD + 2; ++iter) {
    side = cst[0] <= cst[1] ? 0 : 1;
    const int f0 = flo[side], fc = fhi[side] - f0;
    ++n_lev;
    n_exp += fc;
    const int32_t* rowp = side == 0 ? G.rp : G.rrp;
    const int32_t* cols = side == 0 ? G.ci : G.rci;
    int E = 0;
    for (int base = 0; base < fc; base += 32) {
      const int i = base + lane;
      int deg = 0, rs = 0;
      if (i < fc) {
        const int x = S.lnode[f0 + i];
        rs = __ldg(&rowp[x]);
        deg = __ldg(&rowp[x + 1]) - rs;
      }
      int inc = deg;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += y;
      }
      if (i < fc) S.pr[i] = make_int2(E + inc - deg, rs);
      E += __shfl_sync(FULL, inc, 31);
    }
    if (lane == 0) S.pr[fc] = make_int2(E, 0);
    __syncwarp();
    n_edges += E;
    // pass 1: touch test against the other search
    npi = 0;
    for (int rem = E; rem > 0; rem -= 32) {
      const int e = lane < rem ? E - rem + lane : E;
      bool touch = false;
      int x = 0, y = 0;
      unsigned long long wgt = 0;
      if (e < E) {
        const int p = frontier_pos(S.pr, fc, e);
        const int2 q = S.pr[p];
        y = __ldg(&cols[q.y + (e - q.x)]);
        unsigned long long hy = 0;
        if (wt_probe(S.hkv, y, &hy) >= 0 && val_side(ent_val<true>(hy)) != side) {
          touch = true;
          x = S.lnode[f0 + p];
          wgt = (S.hkv[S.lpos[f0 + p]] & PK_SIG_MASK) * (hy & PK_SIG_MASK);  // < 2^48: no overflow
        }
      }
      const unsigned m = __ballot_sync(FULL, touch);
      if (touch) {
        const int at = npi + __popc(m & lt);
        if (at < WT_PCAP) {
          S.pi[at].x = x;
          S.pi[at].y = y;
          S.pi[at].w = wgt;
        }
      }
      npi += __popc(m);
    }
    if (npi > WT_PCAP) return F_CAP;
    if (npi > 0) {
      done = 1;
      break;
    }
    // pass 2: the next level (first discoverer inserts, every discoverer adds sigma)
    const int dnew = dep[side] + 1;
    if (dnew > WT_MAXD) return F_CAP;
    const uint32_t want_val = pack_val(side, dnew);
    const int list_before = nlist;
    long long fresh = 0, hits = 0, cost = 0;
    bool cap = false;
    for (int rem = E; rem > 0 && !cap; rem -= 32) {
      const int e = lane < rem ? E - rem + lane : E;
      bool ins = false, bad = false;
      uint32_t ipos = 0;
      int yy = 0, ydeg = 0;
      if (e < E) {
        const int p = frontier_pos(S.pr, fc, e);
        const int2 q = S.pr[p];
        const int y = __ldg(&cols[q.y + (e - q.x)]);
        const int ylo = __ldg(&rowp[y]), yhi = __ldg(&rowp[y + 1]);
        const unsigned long long add = S.hkv[S.lpos[f0 + p]] & PK_SIG_MASK;
        uint32_t pos = hash_pos(y, WT_HLOG);
        int k = 0;
        for (; k < WT_HSIZE; ++k) {
          unsigned long long w = S.hkv[pos];
          if (w == EMPTY) {
            const unsigned long long old = atomicCAS(&S.hkv[pos], EMPTY, ent_word<true>(y, want_val, add));
            if (old == EMPTY) {
              ins = true;
              ipos = pos;
              yy = y;
              ydeg = yhi - ylo;
              break;
            }
            w = old;
          }
          if ((int32_t)(w >> 32) == y) {
            if (ent_val<true>(w) == want_val) {  // also discovered at this level
              ++hits;
              const unsigned long long o = atomicAdd(&S.hkv[pos], add);
              if ((o & PK_SIG_MASK) + add > PK_SIG_MASK) bad = true;  // sigma outgrew the packed field
            }
            break;
          }
          pos = (pos + 1) & (WT_HSIZE - 1);
        }
        if (k == WT_HSIZE) bad = true;  // table full
      }
      const unsigned m = __ballot_sync(FULL, ins);
      if (ins) {
        const int slot = nlist + __popc(m & lt);
        if (slot < WT_LCAP) {
          S.lnode[slot] = yy;
          S.lpos[slot] = ipos;
        } else {
          bad = true;
        }
        ++fresh;
        cost += ydeg;
      }
      nlist += __popc(m);
      if (__any_sync(FULL, bad)) cap = true;
    }
    if (cap) return F_CAP;
    fresh = (long long)warp_sum_u64((unsigned long long)fresh);
    hits = (long long)warp_sum_u64((unsigned long long)hits);
    cost = (long long)warp_sum_u64((unsigned long long)cost);
    if (fresh == 0) {  // frontier exhausted: s and t are not connected
      done = 2;
      break;
    }
    dep[side] = dnew;
    flo[side] = list_before;
    fhi[side] = nlist;
    cst[side] = cost;
    n_new += fresh;
    n_adds += hits;
    __syncwarp();
  }
  if (done == 0) return F_CAP;
  if (lane == 0) {
    S.stat[KADABRA_STAT_LEVELS] = n_lev;
    S.stat[KADABRA_STAT_EXPANDED] = n_exp;
    S.stat[KADABRA_STAT_EDGES] = n_edges;
    S.stat[KADABRA_STAT_NEW] = n_new;
    S.stat[KADABRA_STAT_SIGMA_ADDS] = n_adds;
    if (done == 1) S.stat[KADABRA_STAT_PI] = npi;
  }
  __syncwarp();
  if (done == 2) return 0;  // disconnected: no hits

  // ------------------------------------------------ candidate-edge choice
  // Weights sigma_sv * sigma_wt < 2^48 each, at most WT_PCAP of them: the
  // total fits 64 bits.  Candidates are ranked by (x, y), x on the expanding side.
  unsigned long long tot = 0;
  for (int i = lane; i < npi; i += 32) tot += S.pi[i].w;
  tot = warp_sum_u64(tot);
  if (lane == 0) {
    S.stat[KADABRA_STAT_SIGMA_LO] = (long long)(tot & 0xFFFFFFFFull);
    S.stat[KADABRA_STAT_SIGMA_HI] = (long long)(tot >> 32);
  }
  const unsigned long long r = below128(dr(1), tot);
  int pick = -1;
  for (int i = lane; i < npi; i += 32) {
    const unsigned long long ki = ((unsigned long long)(uint32_t)S.pi[i].x << 32) | (uint32_t)S.pi[i].y;
    const unsigned long long wi = S.pi[i].w;
    unsigned long long below = 0;
    for (int q = 0; q < npi; ++q) {
      const unsigned long long kq = ((unsigned long long)(uint32_t)S.pi[q].x << 32) | (uint32_t)S.pi[q].y;
      if (kq < ki) below += S.pi[q].w;
    }
    if (below <= r && r - below < wi) pick = i;
  }
  pick = (int)__reduce_max_sync(FULL, (unsigned)(pick + 1)) - 1;
  if (pick < 0) return F_INTERNAL;
  const int cv = side == 0 ? S.pi[pick].x : S.pi[pick].y;
  const int cw = side == 0 ? S.pi[pick].y : S.pi[pick].x;

  // ------------------------------------------------ backtracking
  const int dv = dep[0], dw = dep[1];
  const bool want_path = P.paths != nullptr && out_i >= 0;
  int32_t* row = want_path ? P.paths + out_i * (int64_t)P.max_len : nullptr;
  if (lane == 0) {
    S.stat[KADABRA_STAT_DIST] = dv + 1 + dw;
    S.stat[KADABRA_STAT_PATH_NODES] = dv + dw + 2;
    if (want_path) {
      if (dv < P.max_len) row[dv] = cv;
      if (dv + 1 < P.max_len) row[dv + 1] = cw;
    }
    if (J.counts) {
      if (dv > 0) atomicAdd(&J.counts[cv], 1u);
      if (dw > 0) atomicAdd(&J.counts[cw], 1u);
    }
  }
  uint32_t j = 2;
  long long bts = 0;
  for (int half = 0; half < 2; ++half) {
    int x = half == 0 ? cv : cw;
    int dx = half == 0 ? dv : dw;
    const int32_t* brow = half == 0 ? G.rrp : G.rp;
    const int32_t* bcol = half == 0 ? G.rci : G.ci;
    while (dx > 0) {
      const uint32_t want = pack_val(half, dx - 1);
      unsigned long long hx = 0;
      if (wt_probe(S.hkv, x, &hx) < 0) return F_INTERNAL;
      const unsigned long long rr = below128(dr(j), hx & PK_SIG_MASK);
      ++j;
      const int r0 = __ldg(&brow[x]), deg = __ldg(&brow[x + 1]) - r0;
      unsigned long long carry = 0;
      int pk = -1;
      for (int base = 0; base < deg && pk < 0; base += 32) {
        const int i = base + lane;
        unsigned long long w = 0;
        if (i < deg) {
          const int y = __ldg(&bcol[r0 + i]);
          unsigned long long hw = 0;
          if (wt_probe(S.hkv, y, &hw) >= 0 && ent_val<true>(hw) == want) w = hw & PK_SIG_MASK;
        }
        unsigned long long inc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned long long v = __shfl_up_sync(FULL, inc, o);
          if (lane >= o) inc += v;
        }
        const bool hit = w != 0 && carry + inc - w <= rr && rr < carry + inc;
        const unsigned m = __ballot_sync(FULL, hit);
        if (m) pk = base + __ffs(m) - 1;
        carry += __shfl_sync(FULL, inc, 31);
      }
      if (pk < 0) return F_INTERNAL;
      const int y = __ldg(&bcol[r0 + pk]);
      bts += pk + 1;
      const int dn = dx - 1;
      if (lane == 0) {
        if (dn > 0 && J.counts) atomicAdd(&J.counts[y], 1u);
        if (want_path) {
          const int at = half == 0 ? dn : (dv + 1) + (dw - dn);
          if (at < P.max_len) row[at] = y;
        }
      }
      x = y;
      dx = dn;
    }
  }
  if (lane == 0) S.stat[KADABRA_STAT_BT_SCANNED] = bts;
  __syncwarp();
  return 0;
}

__device__ void wt_flush(const SampleParams& P, WSlot& S) {  // lane 0
  if (S.tot_job >= 0) {
    long long* t = P.jobs ? P.jobs[S.tot_job].totals : P.job0.totals;
    if (t)
      for (int q = 0; q < KADABRA_NSTAT; ++q)
        if (S.tot[q]) atomicAdd((unsigned long long*)&t[q], (unsigned long long)S.tot[q]);
  }
  for (int q = 0; q < KADABRA_NSTAT; ++q) S.tot[q] = 0;
}

__global__ void __launch_bounds__(32 * WT_WARPS) k_sample_warp(SampleParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  WSlot& S = reinterpret_cast<WSlot*>(smem)[warp_id()];
  const int lane = lane_id();
  for (int i = lane; i < WT_HSIZE; i += 32) S.hkv[i] = EMPTY;
  if (lane == 0) {
    S.tot_job = -1;
    for (int q = 0; q < KADABRA_NSTAT; ++q) S.tot[q] = 0;
  }
  __syncwarp();
  const unsigned long long ntotal = P.total_dev ? *P.total_dev : P.total_work;
  for (;;) {
    unsigned long long k = 0;
    if (lane == 0) k = atomicAdd(&P.ctr[Q_NEXT_W], 1ull);
    k = __shfl_sync(FULL, k, 0);
    if (k >= ntotal) break;
    if (lane == 0) {
      int j = 0;
      if (P.jobs) {
        int lo = 0, hi = P.njobs;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (P.jobs[mid].work_begin <= k)
            lo = mid;
          else
            hi = mid;
        }
        j = lo;
      }
      if (j != S.tot_job) {
        wt_flush(P, S);
        S.tot_job = j;
      }
      S.job = P.jobs ? P.jobs[j] : P.job0;
    }
    __syncwarp();
    const uint64_t idx = S.job.first_idx + (k - S.job.work_begin);
    const int64_t out_i = P.st_out ? (int64_t)k : -1;
    if (out_i >= 0 && P.paths)
      for (int q = lane; q < P.max_len; q += 32) P.paths[out_i * (int64_t)P.max_len + q] = -1;
    __syncwarp();
    const int fl = run_sample_warp(P, S.job, S, idx, out_i);
    __syncwarp();
    if (lane == 0) {
      if (fl == F_CAP) {
        if (P.q0)
          enqueue(P, Q_SIZE_S, P.q0, k);
        else
          atomicCAS(P.status, 0, (int)KADABRA_ERR_INTERNAL);
      } else {
        const int st = fl ? KADABRA_ERR_INTERNAL : KADABRA_OK;
        if (st != KADABRA_OK) atomicCAS(P.status, 0, st);
        for (int q = 0; q < KADABRA_NSTAT; ++q)
          if (q != KADABRA_STAT_SIGMA_LO && q != KADABRA_STAT_SIGMA_HI && q != KADABRA_STAT_DIST) S.tot[q] += S.stat[q];
        if (out_i >= 0) {
          P.st_out[2 * out_i] = S.s;
          P.st_out[2 * out_i + 1] = S.t;
          if (P.path_len) P.path_len[out_i] = (int32_t)S.stat[KADABRA_STAT_PATH_NODES];
          if (P.stats)
            for (int q = 0; q < KADABRA_NSTAT; ++q) P.stats[out_i * KADABRA_NSTAT + q] = S.stat[q];
          if (P.sstatus) P.sstatus[out_i] = st;
        }
      }
    }
    for (int i = lane; i < WT_HSIZE; i += 32) S.hkv[i] = EMPTY;
    __syncwarp();
  }
  if (lane == 0) wt_flush(P, S);
}

size_t warp_tier_smem_bytes() { return sizeof(WSlot) * WT_WARPS; }

size_t fast_smem_bytes() { return FastLayout::BYTES; }
size_t compact_smem_bytes() { return CompactLayout::BYTES; }
size_t tiny_smem_bytes() { return TinyLayout::BYTES; }
size_t big_smem_bytes() { return BigLayout::BYTES; }

// ============================================================== stop test
struct CheckOut {
  unsigned long long max_f_bits;
  unsigned long long max_g_bits;
  unsigned int fail;
  unsigned int pad;
};

// f and g of Thm. 2; this expression tree is part of the specification
// (FP64, no contraction: the file is compiled with --fmad=false).
__device__ __forceinline__ void f_and_g(uint32_t count, double t, double omega, double lnL, double lnU, double* f,
                                        double* g) {
  const double b = (double)count / t;
  const double aL = (1.0 / 3.0) - omega / t;
  const double aU = (1.0 / 3.0) + omega / t;
  *f = (lnL / t) * (aL + sqrt(aL * aL + ((2.0 * b) * omega) / lnL));
  *g = (lnU / t) * (aU + sqrt(aU * aU + ((2.0 * b) * omega) / lnU));
}

__global__ void __launch_bounds__(256) k_check(const uint32_t* __restrict__ counts, const double* __restrict__ lnL,
                                               const double* __restrict__ lnU, int64_t n, uint64_t tau,
                                               double omega, double lambda, CheckOut* out) {
  const double t = (double)tau;
  unsigned long long mf = 0, mg = 0;
  unsigned fail = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    double f, g;
    f_and_g(counts[v], t, omega, lnL[v], lnU[v], &f, &g);
    if (!(f <= lambda) || !(g <= lambda)) fail = 1;
    const unsigned long long fb = (unsigned long long)__double_as_longlong(f);
    const unsigned long long gb = (unsigned long long)__double_as_longlong(g);
    mf = fb > mf ? fb : mf;
    mg = gb > mg ? gb : mg;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(FULL, mf, o);
    const unsigned long long b = __shfl_xor_sync(FULL, mg, o);
    mf = a > mf ? a : mf;
    mg = b > mg ? b : mg;
    fail |= __shfl_xor_sync(FULL, fail, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (mf) atomicMax(&out->max_f_bits, mf);
    if (mg) atomicMax(&out->max_g_bits, mg);
    if (fail) atomicOr(&out->fail, 1u);
  }
}

// Stop test of several graphs in all-nodes mode, where ln(1/delta_L(v)) =
// ln(1/delta_U(v)) depends only on v's warm-up count: lnT[count0[v]].  A
// node with no hit has f = 0 exactly (a_L < 0, so a_L + sqrt(a_L^2) = +0) and
// g = (L/t)(a_U + a_U), increasing in L, so the block evaluates g once, at
// the largest L among its unhit nodes; hit nodes take the full formula.  The
// maxima and the decision equal those of the per-node evaluation bit for bit.
// fail_fast: the caller reads the maxima only if the test holds, so once a
// node fails (here or in another block) the rest of the nodes are skipped;
// a test that holds finds no failure and evaluates every node.
struct CheckTabJob {
  const uint32_t* counts;
  const uint32_t* count0;
  const double* lnT;
  int64_t n;
  uint64_t tau;
  double omega;
  double lambda;
  CheckOut* out;
  int fail_fast;
};

// one block's share of the test of graph J (blocks over blockIdx.x)
__device__ __forceinline__ void check_tab_block(const CheckTabJob J) {
  __shared__ unsigned long long s_u[8];
  const double t = (double)J.tau;
  unsigned long long mf = 0, mg = 0, mu = 0;  // bit patterns of non-negative doubles
  unsigned fail = 0;
  int it = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < J.n; v += (int64_t)gridDim.x * blockDim.x) {
    if (J.fail_fast) {
      if (fail) {
        atomicOr(&J.out->fail, 1u);
        break;
      }
      if ((++it & 7) == 0 && *(volatile const unsigned*)&J.out->fail) break;
    }
    const uint32_t cnt = J.counts[v];
    const double L = J.lnT[J.count0[v]];
    if (cnt == 0) {
      const unsigned long long lb = (unsigned long long)__double_as_longlong(L);
      mu = lb > mu ? lb : mu;
      continue;
    }
    double f, g;
    f_and_g(cnt, t, J.omega, L, L, &f, &g);
    if (!(f <= J.lambda) || !(g <= J.lambda)) fail = 1;
    const unsigned long long fb = (unsigned long long)__double_as_longlong(f);
    const unsigned long long gb = (unsigned long long)__double_as_longlong(g);
    mf = fb > mf ? fb : mf;
    mg = gb > mg ? gb : mg;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(FULL, mf, o);
    const unsigned long long b = __shfl_xor_sync(FULL, mg, o);
    const unsigned long long u = __shfl_xor_sync(FULL, mu, o);
    mf = a > mf ? a : mf;
    mg = b > mg ? b : mg;
    mu = u > mu ? u : mu;
    fail |= __shfl_xor_sync(FULL, fail, o);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) s_u[w] = mu;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long u = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) u = s_u[i] > u ? s_u[i] : u;
    if (u) {  // some node of this block has no hit: g at its largest L (f is 0)
      double f0, g0;
      f_and_g(0u, t, J.omega, __longlong_as_double((long long)u), __longlong_as_double((long long)u), &f0, &g0);
      const unsigned long long gb = (unsigned long long)__double_as_longlong(g0);
      atomicMax(&J.out->max_g_bits, gb);
      if (!(f0 <= J.lambda) || !(g0 <= J.lambda)) atomicOr(&J.out->fail, 1u);
    }
  }
  if (lane == 0) {
    if (mf) atomicMax(&J.out->max_f_bits, mf);
    if (mg) atomicMax(&J.out->max_g_bits, mg);
    if (fail) atomicOr(&J.out->fail, 1u);
  }
}

__global__ void __launch_bounds__(256) k_check_tab(const CheckTabJob* __restrict__ jobs) {
  check_tab_block(jobs[blockIdx.y]);
}

// Device-driven main loop of all-nodes runs (Alg. 1) on G graphs at once: a
// CUDA graph whose while node repeats {one sampler launch over every
// unfinished graph's next batch, one stop-test launch over those graphs},
// with the loop state in device memory, so no host round trip separates the
// rounds.  Device memory: LoopState, then G LoopGraph, G Job, G CheckTabJob.
struct LoopState {
  unsigned long long total_work;  // samples of the round over all graphs (the sampler reads it)
  int G;
  unsigned arrive;  // blocks of the round's test that have finished
};
struct LoopGraph {
  unsigned long long tau, cap, K, B, checks;
  int64_t n;
  unsigned stopped, done;
  CheckOut co;
};

__device__ __forceinline__ LoopGraph* loop_graphs(LoopState* s) { return reinterpret_cast<LoopGraph*>(s + 1); }
__device__ __forceinline__ Job* loop_jobs(LoopState* s) {
  return reinterpret_cast<Job*>(loop_graphs(s) + s->G);
}
__device__ __forceinline__ CheckTabJob* loop_checks(LoopState* s) {
  return reinterpret_cast<CheckTabJob*>(loop_jobs(s) + s->G);
}

// the next round's sample ranges, test descriptors and queue counters (one thread)
__device__ void loop_begin(LoopState* s, unsigned long long* ctr) {
  LoopGraph* lg = loop_graphs(s);
  Job* job = loop_jobs(s);
  CheckTabJob* cj = loop_checks(s);
  unsigned long long total = 0;
  for (int i = 0; i < s->G; ++i) {
    LoopGraph& L = lg[i];
    job[i].work_begin = total;
    if (L.done) {
      L.B = 0ull;
      job[i].count = 0ull;
      cj[i].n = 0;
      continue;
    }
    const unsigned long long rest = L.cap - L.tau;
    const unsigned long long B = L.K < rest ? L.K : rest;
    L.B = B;
    job[i].first_idx = L.tau;
    job[i].count = B;
    total += B;
    L.co.max_f_bits = 0ull;
    L.co.max_g_bits = 0ull;
    L.co.fail = 0u;
    cj[i].tau = L.tau + B;
    cj[i].n = (L.tau + B >= L.cap) ? 0 : L.n;  // no test once ceil(omega) is reached
  }
  s->total_work = total;
  for (int q = 0; q < Q_COUNT; ++q) ctr[q] = 0ull;
}

// the first round's setup, launched before the loop's graph
__global__ void k_loop_begin(LoopState* s, unsigned long long* ctr) { loop_begin(s, ctr); }

// The round's stop tests (graph blockIdx.y); the last block to finish then
// closes the round for every graph (advance tau, count the test, decide
// whether it goes on) and sets up the next one, so no single-thread kernels
// separate the rounds.  Each block publishes its test results (atomics)
// before it signs in on `arrive`.
__global__ void __launch_bounds__(256) k_loop_check(LoopState* s, unsigned long long* ctr, const int32_t* status,
                                                    cudaGraphConditionalHandle h) {
  check_tab_block(loop_checks(s)[blockIdx.y]);
  __shared__ unsigned last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&s->arrive, 1u) == gridDim.x * gridDim.y - 1 ? 1u : 0u;
  __syncthreads();
  if (!last || threadIdx.x != 0) return;
  __threadfence();
  s->arrive = 0u;
  LoopGraph* lg = loop_graphs(s);
  unsigned keep = 0u;
  for (int i = 0; i < s->G; ++i) {
    LoopGraph& L = lg[i];
    if (L.done) continue;
    L.tau += L.B;
    if (L.tau >= L.cap) {
      L.done = 1u;
      continue;
    }
    L.checks += 1ull;
    if (!*(volatile const unsigned*)&L.co.fail) {
      L.stopped = 1u;
      L.done = 1u;
      continue;
    }
    keep = 1u;
  }
  if (*(volatile const int32_t*)status != 0) keep = 0u;
  if (keep) loop_begin(s, ctr);
  cudaGraphSetConditional(h, keep);
}

// Stable compaction of the non-zero warm-up counts of several graphs, in
// node order (graph = blockIdx.y; each block owns a contiguous chunk).
struct NzJob {
  const uint32_t* count0;
  int64_t n;
  uint32_t* out;     // non-zero values, node order
  unsigned* blk;     // per-block counts, then exclusive offsets (gridDim.x entries)
  unsigned* total;
  uint32_t* out_idx; // optional: their node ids
  const uint32_t* aux;  // optional: a second per-node array ...
  uint32_t* out_aux;    // ... gathered at the same nodes
};

__global__ void __launch_bounds__(256) k_nz_count(const NzJob* __restrict__ jobs) {
  __shared__ int tmp[8];
  const NzJob J = jobs[blockIdx.y];
  const int64_t chunk = (J.n + gridDim.x - 1) / gridDim.x;
  const int64_t a = min(J.n, (int64_t)blockIdx.x * chunk), b = min(J.n, a + chunk);
  int c = 0;
#pragma unroll 8
  for (int64_t v = a + threadIdx.x; v < b; v += blockDim.x) c += J.count0[v] != 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
  if ((threadIdx.x & 31) == 0) tmp[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += tmp[i];
    J.blk[blockIdx.x] = (unsigned)s;
  }
}

// one block per graph: exclusive offsets of the per-block counts
__global__ void k_nz_offsets(const NzJob* __restrict__ jobs, int nblk) {
  const NzJob J = jobs[blockIdx.x];
  if (threadIdx.x == 0) {
    unsigned s = 0;
    for (int i = 0; i < nblk; ++i) {
      const unsigned c = J.blk[i];
      J.blk[i] = s;
      s += c;
    }
    *J.total = s;
  }
}

// A block takes NZ_ROWS rows of 256 nodes at a time, the loads of all of them
// in flight, and two barriers for all: 16.8 M nodes 0.40 -> 0.12 ms.
constexpr int NZ_ROWS = 8;
__global__ void __launch_bounds__(256) k_nz_scatter(const NzJob* __restrict__ jobs) {
  __shared__ int tmp[NZ_ROWS * 8];  // non-zero counts by row and warp
  const NzJob J = jobs[blockIdx.y];
  const int64_t chunk = (J.n + gridDim.x - 1) / gridDim.x;
  const int64_t a = min(J.n, (int64_t)blockIdx.x * chunk), b = min(J.n, a + chunk);
  unsigned base = J.blk[blockIdx.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t t0 = a; t0 < b; t0 += 256 * NZ_ROWS) {
    uint32_t x[NZ_ROWS];
    unsigned m[NZ_ROWS];
#pragma unroll
    for (int r = 0; r < NZ_ROWS; ++r) {
      const int64_t v = t0 + 256 * r + threadIdx.x;
      x[r] = v < b ? J.count0[v] : 0u;
    }
#pragma unroll
    for (int r = 0; r < NZ_ROWS; ++r) {
      m[r] = __ballot_sync(FULL, x[r] != 0);
      if (lane == 0) tmp[8 * r + w] = __popc(m[r]);
    }
    __syncthreads();
    // every warp: the exclusive prefix of the 64 counts, two per lane
    const int c0 = tmp[2 * lane], c1 = tmp[2 * lane + 1];
    int incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int pre = incl - c0 - c1;
#pragma unroll
    for (int r = 0; r < NZ_ROWS; ++r) {
      const int q = 8 * r + w;  // before (row r, warp w)
      const int p0 = __shfl_sync(FULL, pre, q >> 1), p1 = __shfl_sync(FULL, pre + c0, q >> 1);
      if (x[r] != 0) {
        const int64_t v = t0 + 256 * r + threadIdx.x;
        const unsigned at = base + (unsigned)((q & 1) ? p1 : p0) + __popc(m[r] & ((1u << lane) - 1u));
        J.out[at] = x[r];
        if (J.out_idx) J.out_idx[at] = (uint32_t)v;
        if (J.aux) J.out_aux[at] = J.aux[v];
      }
    }
    base += (unsigned)__shfl_sync(FULL, incl, 31);
    __syncthreads();  // the next rows overwrite tmp
  }
}

// ============================================================== top-k stop test (Alg. 3)
// Nodes are ranked by b~ decreasing, ties by id increasing; with one tau for
// all nodes that is the order of the 64-bit key (count << 32 | ~id), whose
// values are distinct.  A check selects the k+1 largest keys in two stages
// (per-block, then one block over the blocks' survivors), evaluates Alg. 3 on
// them, then tests every other node against the k-th node's lower end.
constexpr int TOPK_MAX = 256;   // largest k of top-k mode
constexpr int TK_SORT = 2048;   // keys one block holds at most (256 + 2 (k + 1) and one row of 256)
constexpr int TK_BLOCKS = 304;  // first-stage selection blocks
constexpr int TK_ROWS = 8;      // rows of 256 nodes a first-stage block reads at a time (16.8 M nodes, with the short sorts: 176 -> 78 us)

__device__ __forceinline__ unsigned long long rank_key(uint32_t count, int64_t v) {
  return ((unsigned long long)count << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)v);
}
__device__ __forceinline__ uint32_t key_node(unsigned long long key) { return 0xFFFFFFFFu - (uint32_t)key; }
__device__ __forceinline__ uint32_t key_count(unsigned long long key) { return (uint32_t)(key >> 32); }

// Block-wide selection of the k1 largest keys.  buf[0, *nb) holds the best so
// far (sorted, descending) followed by pending candidates; keys at or below
// *thr (the k1-th best once k1 are known, else 0) are dropped on arrival.
struct TopSel {
  unsigned long long* buf;  // TK_SORT keys
  int* nb;
  unsigned long long* thr;
  int k1;
};

// sorts buf descending (zero padding beyond *nb, to a power of two), keeps k1, updates thr
__device__ void topsel_compact(const TopSel& S) {
  const int n0 = *S.nb;
  int full = 2;
  while (full < n0) full <<= 1;
  for (int i = n0 + threadIdx.x; i < full; i += blockDim.x) S.buf[i] = 0ull;
  __syncthreads();
  for (int size = 2; size <= full; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < full / 2; i += blockDim.x) {
        const int lo = 2 * i - (i & (stride - 1));
        const int hi = lo + stride;
        const bool desc = (lo & size) == 0;
        const unsigned long long a = S.buf[lo], b = S.buf[hi];
        if ((a < b) == desc) {
          S.buf[lo] = b;
          S.buf[hi] = a;
        }
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    int keep = n0 < S.k1 ? n0 : S.k1;
    while (keep > 0 && S.buf[keep - 1] == 0ull) --keep;  // padding is not a key
    *S.nb = keep;
    *S.thr = keep == S.k1 ? S.buf[S.k1 - 1] : 0ull;
  }
  __syncthreads();
}

// offers one key per thread (0 = none); all threads of the block call it
__device__ void topsel_offer(const TopSel& S, unsigned long long key) {
  const bool pass = key > *S.thr;
  const unsigned m = __ballot_sync(FULL, pass);
  int base = 0;
  if ((threadIdx.x & 31) == 0 && m) base = atomicAdd(S.nb, __popc(m));
  base = __shfl_sync(FULL, base, 0);
  if (pass) S.buf[base + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = key;
  __syncthreads();
  const int cur = *S.nb;
  __syncthreads();  // every thread has read nb before the next offer adds to it
  // early enough that the sort is short and the threshold stands soon
  if (cur > 256 + 2 * S.k1) topsel_compact(S);
}

// stage 1: the k1 largest keys of a contiguous chunk of nodes per block
__global__ void __launch_bounds__(256) k_topk_block(const uint32_t* __restrict__ counts, int64_t n, int k1,
                                                    unsigned long long* __restrict__ out) {
  __shared__ unsigned long long buf[TK_SORT];
  __shared__ int nb;
  __shared__ unsigned long long thr;
  if (threadIdx.x == 0) {
    nb = 0;
    thr = 0ull;
  }
  __syncthreads();
  const TopSel S{buf, &nb, &thr, k1};
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t a = min(n, (int64_t)blockIdx.x * chunk), b = min(n, a + chunk);
  // TK_ROWS rows of 256 nodes at a time; once the threshold stands, hardly any
  // holds a key above it, and one barrier settles them all
  for (int64_t t0 = a; t0 < b; t0 += 256 * TK_ROWS) {
    uint32_t x[TK_ROWS];
    bool any = false;
    const unsigned long long floor = thr;
#pragma unroll
    for (int r = 0; r < TK_ROWS; ++r) {
      const int64_t v = t0 + 256 * r + threadIdx.x;
      x[r] = v < b ? counts[v] : 0u;
    }
#pragma unroll
    for (int r = 0; r < TK_ROWS; ++r) {
      const int64_t v = t0 + 256 * r + threadIdx.x;
      any |= v < b && rank_key(x[r], v) > floor;
    }
    if (!__syncthreads_or(any)) continue;
#pragma unroll 1
    for (int r = 0; r < TK_ROWS; ++r) {
      const int64_t v = t0 + 256 * r + threadIdx.x;
      uint32_t c = x[0];
#pragma unroll
      for (int q = 1; q < TK_ROWS; ++q)
        if (r == q) c = x[q];
      topsel_offer(S, v < b ? rank_key(c, v) : 0ull);
    }
  }
  topsel_compact(S);
  for (int i = threadIdx.x; i < k1; i += blockDim.x) out[(size_t)blockIdx.x * k1 + i] = i < nb ? buf[i] : 0ull;
}

struct TopkOut {
  unsigned long long keys[TOPK_MAX + 1];  // the k1 first nodes of the ranking
  int nk;                                 // how many (min(k + 1, n))
  unsigned fail;                          // Alg. 3 returns false
  unsigned long long max_f_bits, max_g_bits;
  double lower_k;                         // b~(v_k) - f(v_k)
  unsigned long long key_k;               // key of v_k
};

struct TopkJob {
  const uint32_t* counts;
  const double* lnL;
  const double* lnU;
  int64_t n;
  uint64_t tau;
  double omega;
  double lambda;
  int k;                                  // min(k, n)
  int k1;                                 // min(k + 1, n)
  const unsigned long long* cand;         // TK_BLOCKS * k1 keys of stage 1
  int select_only;                        // 1: only the selection (keys, nk)
  int fail_fast;                          // the maxima are read only if the test holds: stop at a failure
  TopkOut* out;
};

// stage 2 (one block): the k1 first nodes, then Alg. 3's test of the k first
__global__ void __launch_bounds__(256) k_topk_final(const TopkJob* __restrict__ jp) {
  __shared__ unsigned long long buf[TK_SORT];
  __shared__ int nb;
  __shared__ unsigned long long thr;
  __shared__ double sb[TOPK_MAX + 1], sf[TOPK_MAX + 1], sg[TOPK_MAX + 1];
  const TopkJob J = *jp;
  if (threadIdx.x == 0) {
    nb = 0;
    thr = 0ull;
  }
  __syncthreads();
  const TopSel S{buf, &nb, &thr, J.k1};
  const int total = TK_BLOCKS * J.k1;
  for (int t0 = 0; t0 < total; t0 += blockDim.x) {
    const int i = t0 + threadIdx.x;
    topsel_offer(S, i < total ? J.cand[i] : 0ull);
  }
  topsel_compact(S);
  const int nk = nb;
  for (int i = threadIdx.x; i < nk; i += blockDim.x) J.out->keys[i] = buf[i];
  if (threadIdx.x == 0) J.out->nk = nk;
  if (J.select_only) return;
  // f, g and b~ of the k1 first nodes
  const double t = (double)J.tau;
  for (int i = threadIdx.x; i < nk; i += blockDim.x) {
    const uint32_t v = key_node(buf[i]), cnt = key_count(buf[i]);
    double f, g;
    f_and_g(cnt, t, J.omega, J.lnL[v], J.lnU[v], &f, &g);
    sb[i] = (double)cnt / t;
    sf[i] = f;
    sg[i] = g;
  }
  __syncthreads();
  // the k first nodes (Alg. 3 first loop); v_0 - f = +inf, v_{n+1} + g = -inf
  for (int i = threadIdx.x; i < J.k && i < nk; i += blockDim.x) {
    const bool loose = sf[i] > J.lambda || sg[i] > J.lambda;
    bool bad = false;
    if (loose) {
      if (i > 0 && sb[i - 1] - sf[i - 1] < sb[i] + sg[i]) bad = true;
      if (i + 1 < nk && sb[i] - sf[i] < sb[i + 1] + sg[i + 1]) bad = true;
    }
    if (bad) atomicOr(&J.out->fail, 1u);
    atomicMax(&J.out->max_f_bits, (unsigned long long)__double_as_longlong(sf[i]));
    atomicMax(&J.out->max_g_bits, (unsigned long long)__double_as_longlong(sg[i]));
  }
  if (threadIdx.x == 0 && J.k >= 1 && J.k <= nk) {
    J.out->lower_k = sb[J.k - 1] - sf[J.k - 1];
    J.out->key_k = buf[J.k - 1];
  }
}

// the other nodes (Alg. 3 second loop): a node below v_k whose f or g exceeds
// lambda must lie below b~(v_k) - f(v_k).  Unhit nodes have f = 0 and g
// increasing in ln(1/delta_U), so each block evaluates g once for them, at
// the largest ln(1/delta_U) among its unhit nodes.
__global__ void __launch_bounds__(256) k_topk_rest(const TopkJob* __restrict__ jp) {
  __shared__ unsigned long long s_u[8];
  const TopkJob J = *jp;
  const double t = (double)J.tau;
  const double lower_k = J.out->lower_k;
  const unsigned long long key_k = J.out->key_k;
  unsigned long long mf = 0, mg = 0, mu = 0;
  unsigned fail = 0;
  int it = 0;
  // fail_fast: nothing to do once the k first nodes or another block failed
  const bool skip = J.fail_fast && *(volatile const unsigned*)&J.out->fail;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < J.n && !skip;
       v += (int64_t)gridDim.x * blockDim.x) {
    if (J.fail_fast) {
      if (fail) {
        atomicOr(&J.out->fail, 1u);
        break;
      }
      if ((++it & 7) == 0 && *(volatile const unsigned*)&J.out->fail) break;
    }
    const uint32_t cnt = J.counts[v];
    if (rank_key(cnt, v) >= key_k) continue;  // one of the k first nodes
    if (cnt == 0) {
      const unsigned long long ub = (unsigned long long)__double_as_longlong(J.lnU[v]);
      mu = ub > mu ? ub : mu;
      continue;
    }
    double f, g;
    f_and_g(cnt, t, J.omega, J.lnL[v], J.lnU[v], &f, &g);
    const double b = (double)cnt / t;
    if ((f > J.lambda || g > J.lambda) && lower_k < b + g) fail = 1;
    const unsigned long long fb = (unsigned long long)__double_as_longlong(f);
    const unsigned long long gb = (unsigned long long)__double_as_longlong(g);
    mf = fb > mf ? fb : mf;
    mg = gb > mg ? gb : mg;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(FULL, mf, o);
    const unsigned long long b = __shfl_xor_sync(FULL, mg, o);
    const unsigned long long u = __shfl_xor_sync(FULL, mu, o);
    mf = a > mf ? a : mf;
    mg = b > mg ? b : mg;
    mu = u > mu ? u : mu;
    fail |= __shfl_xor_sync(FULL, fail, o);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) s_u[w] = mu;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long u = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) u = s_u[i] > u ? s_u[i] : u;
    if (u) {
      const double L = __longlong_as_double((long long)u);
      double f0, g0;
      f_and_g(0u, t, J.omega, L, L, &f0, &g0);
      atomicMax(&J.out->max_g_bits, (unsigned long long)__double_as_longlong(g0));
      if ((f0 > J.lambda || g0 > J.lambda) && lower_k < 0.0 + g0) atomicOr(&J.out->fail, 1u);
    }
  }
  if (lane == 0) {
    if (mf) atomicMax(&J.out->max_f_bits, mf);
    if (mg) atomicMax(&J.out->max_g_bits, mg);
    if (fail) atomicOr(&J.out->fail, 1u);
  }
}

__global__ void k_fill2(double* __restrict__ a, double* __restrict__ b, int64_t n, double x) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    a[v] = b[v] = x;
}

__global__ void k_scatter2(double* __restrict__ a, double* __restrict__ b, const uint32_t* __restrict__ idx,
                           const double* __restrict__ va, const double* __restrict__ vb, int64_t m) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    a[idx[i]] = va[i];
    b[idx[i]] = vb[i];
  }
}

// 32 row offsets and 32 adjacency entries at evenly spaced positions
__global__ void k_fingerprint(const int32_t* rp, const int32_t* ci, int32_t n, int64_t m, int32_t* out) {
  const int i = threadIdx.x;
  if (i < 32) out[i] = rp[(int64_t)n * i / 32];
  else if (i < 64) out[i] = m > 0 ? ci[m * (i - 32) / 32] : 0;
}

// Measurement helper: re-reads a buffer `reps` times, caching in L2 only
// (ld.global.cg), so a buffer that fits in L2 measures the L2's read rate.
__global__ void k_l2_read(const float4* __restrict__ buf, size_t n4, int reps, float* sink) {
  float acc = 0.f;
  for (int r = 0; r < reps; ++r)
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
      const float4 v = __ldcg(&buf[i]);
      acc += (v.x + v.y) + (v.z + v.w);
    }
  if (acc == -1.f) sink[0] = acc;  // never true for the zero buffer; keeps the loads
}

// b~ = count / tau.  FP64 division is slow on this GPU and most counts are small
// or zero, so each block divides the counts below 256 once and looks them up:
// 16.8 M nodes 0.63 -> 0.07 ms.
__global__ void __launch_bounds__(256) k_btilde(const uint32_t* __restrict__ counts, int64_t n, uint64_t tau,
                                                double* __restrict__ out) {
  __shared__ double small[256];
  const double t = (double)tau;
  small[threadIdx.x] = (double)threadIdx.x / t;
  __syncthreads();
  for (int64_t v = blockIdx.x * 256ll + threadIdx.x; v < n; v += gridDim.x * 256ll) {
    const uint32_t c = counts[v];
    out[v] = c < 256u ? small[c] : (double)c / t;
  }
}

__global__ void k_philox(uint64_t seed, uint32_t domain, uint32_t j, uint64_t first, uint32_t count, uint4* out) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) out[i] = draw(seed, domain, first + i, j);
}

// ============================================================== graph checks, VD
// error bits: 1 offsets, 2 id range, 4 order/duplicate, 8 self-loop, 16 reverse mismatch
//
// The arc passes run arc-parallel: a warp takes ARC_CHUNK consecutive arcs,
// one per lane at a time, so the column array is read coalesced and a hub's
// row is spread over many warps.
// R-MAT scale 24's row checks, two passes of 263 M arcs: 16 arcs per thread
// read with a stride of 64 bytes 3.09 ms; chunks of 128, 256, 512 arcs per
// warp 2.94, 2.46, 2.18 ms (each chunk searches its first row).
constexpr int ARC_CHUNK = 512;

// offsets: 0 <= rp[v] <= rp[v+1] <= m (rp[0] = 0 and rp[n] = m are checked on the host)
__global__ void k_validate_offsets(const int32_t* rp, int32_t n, int64_t m, unsigned* err) {
  bool bad = false;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = rp[v], b = rp[v + 1];
    if (a < 0 || b < a || b > m) bad = true;
  }
  if (__any_sync(FULL, bad) && lane_id() == 0) atomicOr(err, 1u);
}

// The row u that holds arc e: the largest u with rp[u] <= e (rp monotone,
// e < rp[n]), by one warp, 32 offsets per round.
__device__ __forceinline__ int32_t warp_row_of_arc(const int32_t* rp, int32_t n, int64_t e) {
  int32_t lo = 0, hi = n;  // rp[lo] <= e, and e < rp[hi]
  while (hi - lo > 1) {
    const int32_t step = (hi - lo + 31) / 32;
    const int64_t i = lo + (int64_t)(lane_id() + 1) * step;
    const int k = __popc(__ballot_sync(FULL, i < hi && __ldg(&rp[i]) <= e));
    lo += k * step;
    hi = min((int64_t)hi, (int64_t)lo + step);
  }
  return lo;
}

// Calls f(ok, u, e, v) for arcs e[k] = (u[k], v[k]), D per lane (32 apart;
// ok[k] = there is one), with all lanes of the warp.  The lanes' rows come
// from the starts of the next rows, 32 at a time, counted by a search over
// the lanes' registers (several rounds only where rows are so short, or
// empty, that more than 32 start in a window).  Starts count from the step's
// first arc, since a window's end may lie behind arc 2^31 - 1, the largest
// start and the one that stands for "no more rows".
template <int D, class F>
__device__ __forceinline__ void for_each_arc(const int32_t* rp, const int32_t* ci, int32_t n, int64_t m, F f) {
  const int lane = lane_id();
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  if (m <= 0) return;  // no chunk
  // a graph with less than ARC_CHUNK arcs per warp is spread over all of them
  const int64_t per = (m + nwarps - 1) / nwarps;
  const int64_t chunk = per < ARC_CHUNK ? (per + 31) / 32 * 32 : ARC_CHUNK;
  const int64_t chunks = (m + chunk - 1) / chunk;
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < chunks; c += nwarps) {
    const int64_t e1 = min(m, (c + 1) * chunk);
    int32_t row = warp_row_of_arc(rp, n, c * chunk);
    for (int64_t base = c * chunk; base < e1; base += 32 * D) {
      bool ok[D];
      int32_t u[D], v[D];
      int64_t e[D];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        e[k] = base + 32 * k + lane;
        ok[k] = e[k] < e1;
        v[k] = ok[k] ? __ldg(&ci[e[k]]) : 0;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int32_t at = 32 * k + lane, last = 32 * k + 31;
        u[k] = row;
        for (int32_t r = row;; r += 32) {
          const int32_t st = r + 1 + lane < n ? __ldg(&rp[r + 1 + lane]) - (int32_t)base : 0x7FFFFFFF;
          if (!__any_sync(FULL, st <= last)) break;
          int q = 0;  // how many of the 32 rows start at e or before
#pragma unroll
          for (int h = 16; h > 0; h >>= 1)
            if (__shfl_sync(FULL, st, q + h - 1) <= at) q += h;
          if (__shfl_sync(FULL, st, q) <= at) ++q;
          if (q > 0) u[k] = r + q;
          if (__shfl_sync(FULL, st, 31) > last) break;
        }
        row = __shfl_sync(FULL, u[k], 31);
      }
      f(ok, u, e, v);
    }
  }
}

// ids in range, rows strictly increasing (sorted, no repeats), no self-loops
__global__ void __launch_bounds__(256) k_validate_arcs(const int32_t* rp, const int32_t* ci, int32_t n, int64_t m,
                                                       unsigned* err) {
  if (*(volatile const unsigned*)err & 1u) return;  // needs valid offsets
  unsigned bits = 0;
  for_each_arc<4>(rp, ci, n, m, [&](const bool* ok, const int32_t* u, const int64_t* e, const int32_t* v) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      int32_t before = __shfl_up_sync(FULL, v[k], 1);
      if (!ok[k]) continue;
      const bool first = e[k] == __ldg(&rp[u[k]]);
      if (lane_id() == 0 && !first) before = __ldg(&ci[e[k] - 1]);
      if (v[k] < 0 || v[k] >= n) bits |= 2u;
      if (!first && v[k] <= before) bits |= 4u;
      if (v[k] == u[k]) bits |= 8u;
    }
  });
  bits = __reduce_or_sync(FULL, bits);
  if (bits && lane_id() == 0) atomicOr(err, bits);
}

// An 8-ary tree over the column array that the mirror test searches, for
// graphs beyond the L2: level k holds every (2^TREE_SHIFT * 8^k)-th entry, and
// an aligned group of 8 of them, one 32-byte load, settles one octal digit of
// a position.
// What bounds the test is the number of scattered loads per arc: each lane's
// goes to another line, and L1 takes one line per cycle.  A binary search
// costs one per bit, the tree one per three bits, and the two levels that are
// not L2-resident cost HBM one sector each.  The mirror test of R-MAT scale 24
// (263 M arcs): binary search 32 to 33 ms (one, two or four searches per lane
// at once), binary over every 32nd entry first 15.6, this tree 9.6 ms (L1 at
// 68 %, L2 62 %, issue 59 % on scale 22); with a last block of 16 or 32
// entries (TREE_SHIFT 4, 5) 11.6, 14.0 ms.  Graphs within the L2 have no
// tree: building it costs more than it saves (Chung-Lu 10^6 nodes 0.18 -> 0.23 ms).
#ifndef KD_TREE_SHIFT
#define KD_TREE_SHIFT 3
#endif
constexpr int TREE_SHIFT = KD_TREE_SHIFT;  // at least 3
constexpr int TREE_LEVELS = (31 - TREE_SHIFT + 2) / 3;
struct RowTree {
  int32_t* lv[TREE_LEVELS];  // 32-byte aligned, whole groups of 8
  int32_t levels;            // 0: no tree
  int32_t groups;            // whole groups of 8 of the column array itself, 0 if it is not 32-byte aligned
};

__global__ void k_row_tree(const int32_t* ci, int64_t m, const __grid_constant__ RowTree t) {
  const int64_t c = (m + (1ll << TREE_SHIFT) - 1) >> TREE_SHIFT;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < c; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = ci[i << TREE_SHIFT];
    t.lv[0][i] = x;
    int64_t q = i;
    for (int k = 1; k < t.levels && (q & 7) == 0; ++k) {
      q >>= 3;
      t.lv[k][q] = x;
    }
  }
}

// p: 32-byte aligned
__device__ __forceinline__ void ldg8(const int32_t* p, int32_t (&w)[8]) {
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
      : "l"(p));
}

// entries [a, b], not none, of a sorted row have y
__device__ __forceinline__ bool tree_has(const int32_t* ci, const RowTree& t, int32_t a, int32_t b, int32_t y) {
  int32_t w[8];
  const uint32_t diff = (uint32_t)(a ^ b) >> TREE_SHIFT;
  for (int k = diff ? (31 - __clz(diff)) / 3 : -1; k >= 0; --k) {
    // a and b lie under one group of this level; y, if it is there, lies under
    // the last entry of the group within (a, b] that is not above it, or under a's
    const int sh = TREE_SHIFT + 3 * k;
    const int32_t pa = a >> sh, pb = b >> sh;
    if (pa == pb) continue;
    ldg8(t.lv[k] + (pa & ~7), w);
    uint32_t le = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) le |= (w[q] <= y ? 1u : 0u) << q;
    const int32_t i = pa + __popc(le & ((2u << (pb & 7)) - (2u << (pa & 7))));
    if (i > pa) a = i << sh;
    if (i < pb) b = ((i + 1) << sh) - 1;
  }
  while ((a >> 3) != (b >> 3)) {  // TREE_SHIFT > 3: groups of 8 of the last block
    const int32_t mid = ((a >> 3) + (b >> 3) + 1) >> 1;
    if (__ldg(&ci[8 * mid]) <= y)
      a = 8 * mid;
    else
      b = 8 * mid - 1;
  }
  if ((a >> 3) < t.groups) {
    ldg8(ci + (a & ~7), w);
    uint32_t eq = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) eq |= (w[q] == y ? 1u : 0u) << q;
    return (eq & ((2u << (b & 7)) - (1u << (a & 7)))) != 0;
  }
  bool found = false;
  for (; a <= b; ++a) found |= __ldg(&ci[a]) == y;
  return found;
}

// row v of a sorted CSR has y
__device__ __forceinline__ bool row_has(const int32_t* rp, const int32_t* ci, const RowTree& t, int32_t v, int32_t y) {
  int32_t lo = __ldg(&rp[v]), hi = __ldg(&rp[v + 1]);
  if (t.levels) return lo < hi && tree_has(ci, t, lo, hi - 1, y);
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    const int32_t z = __ldg(&ci[mid]);
    if (z == y) return true;
    if (z < y)
      lo = mid + 1;
    else
      hi = mid;
  }
  return false;
}

// Every arc (u, v) of the forward CSR must appear as u in row v of the
// reverse CSR.  Both hold m arcs with no repeats (rows strictly increasing),
// so this injection is a bijection and the two CSRs are mirrors.  An
// undirected graph is its own mirror: there only arcs with u < v are looked
// up, and the arcs with u < v and u > v are counted (lt_gt[0], lt_gt[1]);
// equal counts make the injection from the first kind into the second a
// bijection, which is symmetry.
// For a directed graph the same pass counts, per node u that can be the root
// r below, the arcs (u, v) whose reverse arc (v, u) exists (recip[u]): the
// degree in the underlying undirected graph is at least max(out, in) and at
// most out + in, so only the nodes whose out + in reaches the largest
// max(out, in) of any node (*floor_deg) can be it.
__global__ void __launch_bounds__(256) k_validate_mirror(const int32_t* rp, const int32_t* ci, const int32_t* rrp,
                                                         const int32_t* rci, int32_t n, int64_t m, int undirected,
                                                         unsigned* err, unsigned long long* lt_gt, uint32_t* recip,
                                                         const int32_t* floor_deg, const __grid_constant__ RowTree tree) {
  if (*(volatile const unsigned*)err & 15u) return;  // needs valid offsets, ids in range and sorted rows
  unsigned long long lt = 0, gt = 0;
  bool bad = false;
  const int32_t floor = undirected ? 0 : *floor_deg;
  for_each_arc<1>(rp, ci, n, m, [&](const bool* ok, const int32_t* uu, const int64_t*, const int32_t* vv) {
    if (!ok[0]) return;
    const int32_t u = uu[0], v = vv[0];
    if (undirected && v < u) {
      ++gt;
      return;
    }
    ++lt;
    if (!row_has(rrp, rci, tree, v, u)) bad = true;
    if (!undirected) {
      const int64_t both = (int64_t)(__ldg(&rp[u + 1]) - __ldg(&rp[u])) + (__ldg(&rrp[u + 1]) - __ldg(&rrp[u]));
      if (both >= floor && row_has(rrp, rci, tree, u, v)) atomicAdd(&recip[u], 1u);
    }
  });
  if (__any_sync(FULL, bad) && lane_id() == 0) atomicOr(err, 16u);
  if (undirected) {
    lt = warp_sum_u64(lt);
    gt = warp_sum_u64(gt);
    if (lane_id() == 0) {
      atomicAdd(&lt_gt[0], lt);
      atomicAdd(&lt_gt[1], gt);
    }
  }
}

// the largest max(out, in) of any node (directed graphs; offsets already validated)
__global__ void k_floor_degree(const int32_t* rp, const int32_t* rrp, int32_t n, int32_t* floor_deg) {
  int32_t d = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    d = max(d, max(rp[v + 1] - rp[v], rrp[v + 1] - rrp[v]));
  d = __reduce_max_sync(FULL, d);
  if (lane_id() == 0) atomicMax(floor_deg, d);
}

// The root r of the VD bound: the lowest-id node of maximum degree in the
// underlying undirected graph, |out(v) U in(v)| = out + in - reciprocal arcs
// (directed; the nodes whose reciprocal arcs were not counted stay below the
// others), as a key degree << 32 | ~id under atomicMax.
// Also counts the nodes without out-arcs and those without in-arcs (idle).
__global__ void k_und_degree_key(const int32_t* rp, const int32_t* rrp, const uint32_t* recip, int32_t n,
                                 int directed, unsigned long long* best, uint32_t* idle) {
  unsigned long long mine = 0;
  uint32_t no_out = 0, no_in = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t d = rp[v + 1] - rp[v];
    no_out += d == 0;
    no_in += rrp[v + 1] == rrp[v];
    if (directed) d += (int64_t)(rrp[v + 1] - rrp[v]) - recip[v];
    const unsigned long long key = ((unsigned long long)d << 32) | (0xFFFFFFFFu - (uint32_t)v);
    mine = key > mine ? key : mine;
  }
  // one update per warp: one per thread queued on the address (Chung-Lu of 10^6
  // nodes, with its memsets: 0.12 -> 0.03 ms)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(FULL, mine, o);
    mine = x > mine ? x : mine;
  }
  no_out = __reduce_add_sync(FULL, no_out);
  no_in = __reduce_add_sync(FULL, no_in);
  if (lane_id() == 0) {
    atomicMax(best, mine);
    if (no_out) atomicAdd(&idle[0], no_out);
    if (no_in) atomicAdd(&idle[1], no_in);
  }
}

__device__ __forceinline__ int32_t key_root(unsigned long long key) {
  return (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));
}

// the root r from its key: level 0 = {r}
__global__ void k_bfs_root(const unsigned long long* best, int32_t* dist, int32_t* front) {
  const int32_t r = key_root(*best);
  dist[r] = 0;
  front[0] = r;
}

// One level of a BFS from r along the arcs of one CSR: out-arcs for the
// distances from r, in-arcs for the distances to r.  Top-down, a warp
// expands one frontier node's row (tr, tc) of up to BFS_CHUNK arcs; a longer
// row is cut into BFS_CHUNK-arc items for k_bfs_items, so that a hub's row
// is spread over many warps.
constexpr int BFS_CHUNK = 1024;

struct BfsItem {
  int32_t v, begin, end;
  int32_t look;  // bottom-up: 1, the arcs are searched for a node at the current level
};

// cuts arcs [a, b) of v's row, more than one chunk, into items (one warp);
// returns the first arc that found no room, or b
__device__ __forceinline__ int32_t bfs_cut(int32_t v, int32_t a, int32_t b, int32_t look, BfsItem* items,
                                           int32_t* nitems, int32_t items_cap) {
  const int lane = lane_id();
  const int32_t k = (b - a + BFS_CHUNK - 1) / BFS_CHUNK;  // items of this row
  int32_t at = 0;
  if (lane == 0) at = atomicAdd(nitems, k);
  at = __shfl_sync(FULL, at, 0);
  for (int32_t q = lane; q < k; q += 32) {
    if (at + q < items_cap) {
      const int32_t s = a + q * BFS_CHUNK;
      items[at + q] = BfsItem{v, s, b - s > BFS_CHUNK ? s + BFS_CHUNK : b, look};
    }
  }
  return at + k > items_cap ? a + (items_cap > at ? items_cap - at : 0) * BFS_CHUNK : b;
}

// one of arcs [a, b) of row c is a node at `level` (one warp)
__device__ __forceinline__ bool bfs_look(const int32_t* c, int64_t a, int32_t b, const int32_t* dist, int32_t level) {
  for (; a < b; a += 32)
    if (__any_sync(FULL, a + lane_id() < b && dist[c[a + lane_id()]] == level)) return true;
  return false;
}

// scans arcs [a, b) of row c and appends the newly reached heads to next;
// arcs: their rows' arcs, of this lane's heads
__device__ __forceinline__ void bfs_scan(const int32_t* tr, const int32_t* c, int32_t a, int32_t b, int32_t* next,
                                         int32_t* nnext, int32_t* dist, int32_t level, int32_t& arcs) {
  const int lane = lane_id();
  for (int64_t base = a; base < b; base += 32) {  // bounds uniform in the warp
    const int64_t e = base + lane;
    int32_t y = 0;
    bool mine = false;
    if (e < b) {
      y = c[e];
      mine = dist[y] < 0 && atomicCAS(&dist[y], -1, level + 1) == -1;
    }
    // one queue reservation per warp and window, not per node
    const unsigned got = __ballot_sync(FULL, mine);
    if (got) {
      int32_t at = 0;
      if (lane == 0) at = atomicAdd(nnext, __popc(got));
      at = __shfl_sync(FULL, at, 0);
      if (mine) next[at + __popc(got & ((1u << lane) - 1u))] = y;
      if (mine) arcs += tr[y + 1] - tr[y];
    }
  }
}

// a warp's part of the next frontier's arcs (nnext[2])
__device__ __forceinline__ void bfs_add_arcs(int32_t arcs, int32_t* nnext) {
  arcs = __reduce_add_sync(FULL, arcs);
  if (lane_id() == 0 && arcs) atomicAdd(nnext + 2, arcs);
}

// Passes over all nodes that fill a queue: a warp takes up to NODE_GROUPS
// groups of 32 nodes per reservation, since its counter takes one update at a
// time: a reservation and an arc count per 32 nodes were the time of a
// bottom-up level (both BFS of R-MAT scale 24 3.97 ms; 4, 16, 32 groups and
// one arc count per warp 1.21, 1.31, 1.36 ms).
constexpr int NODE_GROUPS = 4;

// appends this lane's nodes first + 32 * q + lane (bit q of bits, q < groups) to queue, size *count
__device__ __forceinline__ void warp_append_groups(uint32_t bits, int groups, int64_t first, int32_t* queue,
                                                   int32_t* count) {
  const int lane = lane_id();
  const int total = __reduce_add_sync(FULL, __popc(bits));
  if (!total) return;
  int32_t at = 0;
  if (lane == 0) at = atomicAdd(count, total);
  at = __shfl_sync(FULL, at, 0);
  for (int q = 0; q < groups; ++q) {
    const unsigned got = __ballot_sync(FULL, (bits >> q) & 1u);
    if ((bits >> q) & 1u) queue[at + __popc(got & ((1u << lane) - 1u))] = (int32_t)(first + 32 * q + lane);
    at += __popc(got);
  }
}

// The frontier's size is read on the device (*nfront_dev, or 1 for the root's
// level when it is null), so the host can queue several levels at once.
// A frontier of more than n / BFS_BOTTOM_UP nodes, or whose rows hold more
// than m / BFS_BOTTOM_UP_ARCS arcs, is expanded bottom-up (Beamer et al.'s
// direction-optimising BFS): every unvisited node looks in its row of the
// opposite CSR (br, bc) for a node at the current level and stops at the
// first, after m / (frontier arcs) looks or so.  A lane looks at BFS_LOOK arcs
// of its node's row; the rest of a longer row, one the level may not reach at
// all, goes to the whole warp, and beyond a chunk to k_bfs_items (an
// undirected graph of 4.4 M nodes with a hub of 100,000 arcs out of reach on
// two levels: load 18.98 -> 0.54 ms).  Either direction yields the same
// next level.  The arcs count for themselves: the neighbours of a
// power-law graph's largest hub are few, but hold most arcs (both BFS of
// R-MAT scale 24: 6.7 -> 4.0 ms).  Whole loads with m, m/16, m/32 and m/64:
// R-MAT scale 20 3.03, 2.17, 2.17, 2.17 ms, Chung-Lu of 10^6 nodes 0.82, 0.73,
// 0.74, 0.74 ms, BA of 300,000 nodes 0.58, 0.59, 0.51, 0.51 ms.
constexpr int BFS_BOTTOM_UP = 16;
constexpr int BFS_BOTTOM_UP_ARCS = 32;
constexpr int BFS_LOOK = 64;

__global__ void k_bfs_level(const int32_t* tr, const int32_t* tc, const int32_t* br, const int32_t* bc,
                            const int32_t* front, const int32_t* nfront_dev, int32_t* next, int32_t* nnext,
                            int32_t* dist, int32_t level, BfsItem* items, int32_t* nitems, int32_t items_cap,
                            int32_t n, int64_t m) {
  const int lane = lane_id();
  const int32_t nfront = nfront_dev ? *nfront_dev : 1;
  const int32_t arcs = nfront_dev ? nfront_dev[2] : 0;
  if (nfront > n / BFS_BOTTOM_UP || arcs > m / BFS_BOTTOM_UP_ARCS) {
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int groups = n >= NODE_GROUPS * nthreads ? NODE_GROUPS : 1;  // of 32 nodes per reservation
    int32_t own = 0;
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32 * groups; base < n;
         base += nthreads * groups) {
      uint32_t bits = 0;
      for (int q = 0; q < groups; ++q) {
        const int64_t v = base + 32 * q + lane;
        bool mine = false;
        int32_t a = 0, b = 0;  // what is left of the row
        if (v < n && dist[v] < 0) {
          a = br[v];
          b = br[v + 1];
          const int32_t stop = b - a > BFS_LOOK ? a + BFS_LOOK : b;
          for (; a < stop && !mine; ++a) mine = dist[bc[a]] == level;
        }
        for (unsigned rows = __ballot_sync(FULL, !mine && a < b); rows; rows &= rows - 1) {
          const int j = __ffs(rows) - 1;
          int32_t aj = __shfl_sync(FULL, a, j);
          const int32_t bj = __shfl_sync(FULL, b, j);
          if (bj - aj > BFS_CHUNK) aj = bfs_cut((int32_t)(v - lane + j), aj, bj, 1, items, nitems, items_cap);
          if (bfs_look(bc, aj, bj, dist, level) && lane == j) mine = true;
        }
        if (mine) {
          dist[v] = level + 1;  // only this thread writes v's entry in this launch
          own += tr[v + 1] - tr[v];
          bits |= 1u << q;
        }
      }
      warp_append_groups(bits, groups, base, next, nnext);
    }
    bfs_add_arcs(own, nnext);
    return;
  }
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int32_t own = 0;
  for (int64_t i = w0; i < nfront; i += nwarps) {
    const int32_t v = front[i];
    const int32_t a = tr[v], b = tr[v + 1];
    if (b - a <= BFS_CHUNK) {
      bfs_scan(tr, tc, a, b, next, nnext, dist, level, own);
      continue;
    }
    // items beyond the buffer: this warp scans them
    bfs_scan(tr, tc, bfs_cut(v, a, b, 0, items, nitems, items_cap), b, next, nnext, dist, level, own);
  }
  bfs_add_arcs(own, nnext);
}

__global__ void k_bfs_items(const int32_t* tr, const int32_t* tc, const int32_t* bc, const BfsItem* items,
                            const int32_t* nitems, int32_t items_cap, int32_t* next, int32_t* nnext, int32_t* dist,
                            int32_t level) {
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int32_t k = *nitems < items_cap ? *nitems : items_cap;
  int32_t own = 0;
  for (int64_t i = w0; i < k; i += nwarps) {
    const BfsItem it = items[i];
    if (!it.look) {
      bfs_scan(tr, tc, it.begin, it.end, next, nnext, dist, level, own);
    } else if (__shfl_sync(FULL, *(volatile const int32_t*)&dist[it.v], 0) < 0 &&
               bfs_look(bc, it.begin, it.end, dist, level) && lane_id() == 0 &&
               atomicCAS(&dist[it.v], -1, level + 1) == -1) {  // not found by another of the row's items
      next[atomicAdd(nnext, 1)] = it.v;
      own += tr[it.v + 1] - tr[it.v];
    }
  }
  bfs_add_arcs(own, nnext);
}

// ---- VD bound from the condensation into strongly connected components.
// A shortest path visits the components along a path of the condensation,
// each in a contiguous stretch that is a shortest path inside it: at most
// |C| nodes, or e_in + e_out + 1 inside the root's component C_r (e_out and
// e_in its largest distances from and to r).  The bound is the heaviest path
// of the condensation under these weights.  Components get a label, the id
// of one of their nodes: r for C_r (reached from r and reaching r), the node
// itself for one trimmed away (no successor or no predecessor left among the
// unlabelled nodes), the largest id of the component for the rest (colour
// propagation: a node's colour is the largest id that reaches it; the nodes
// of a root's colour that reach the root form its component).
struct VdCore {
  unsigned long long size;  // |C_r|
  int32_t e_out, e_in;
  uint32_t idle[2];         // nodes without out-arcs, without in-arcs
};

__global__ void k_vd_core(const int32_t* df, const int32_t* db, int32_t n, VdCore* out) {
  unsigned long long cnt = 0;
  int32_t eo = 0, ei = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = df[v], b = db[v];
    if (a >= 0 && b >= 0) {
      ++cnt;
      eo = a > eo ? a : eo;
      ei = b > ei ? b : ei;
    }
  }
  cnt = warp_sum_u64(cnt);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    eo = max(eo, __shfl_xor_sync(FULL, eo, o));
    ei = max(ei, __shfl_xor_sync(FULL, ei, o));
  }
  if (lane_id() == 0) {
    if (cnt) atomicAdd(&out->size, cnt);
    atomicMax(&out->e_out, eo);
    atomicMax(&out->e_in, ei);
  }
}

#define VD_FOR_NODES(v) \
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)

// On power-law graphs the nodes outside the root's component have short rows,
// and few of the arcs: passes that need only their arcs then go by node.  One
// longer row among them (*long_rows) and the passes go by arc instead, balanced
// whatever the rows' lengths.  R-MAT scale 24, by arc and by node: arcs
// entering the components 1.36 -> 0.22 ms, condensation levels 3.1 -> 0.95 ms.
constexpr int VD_LONG_ROW = 1024;

__global__ void k_vd_label_init(const int32_t* df, const int32_t* db, int32_t n, const unsigned long long* best,
                                int32_t* lab, const int32_t* rp, const int32_t* rrp, int32_t* long_rows) {
  const int32_t r = key_root(*best);
  bool any = false;
  VD_FOR_NODES(v) {
    const bool core = df[v] >= 0 && db[v] >= 0;
    lab[v] = core ? r : -1;
    any |= !core && max(rp[v + 1] - rp[v], rrp[v + 1] - rrp[v]) > VD_LONG_ROW;
  }
  if (any) *long_rows = 1;
}

// Each lane's row [a, b) of col (empty: none): how many of its entries x have
// p(x, key) > 0, and the largest p.  All lanes of the warp; rows beyond 16
// entries are read by the whole warp.
struct VdRow {
  int32_t count;
  long long most;
};
template <class P>
__device__ __forceinline__ VdRow vd_rows(const int32_t* col, int32_t a, int32_t b, int32_t key, P p) {
  VdRow r = {0, 0};
  const bool own = b - a <= 16;
  if (own)
    for (int32_t e = a; e < b; ++e) {
      const long long w = p(__ldg(&col[e]), key);
      r.count += w > 0;
      r.most = w > r.most ? w : r.most;
    }
  for (unsigned rows = __ballot_sync(FULL, !own); rows; rows &= rows - 1) {
    const int j = __ffs(rows) - 1;
    const int32_t bj = __shfl_sync(FULL, b, j), kj = __shfl_sync(FULL, key, j);
    int32_t c = 0;
    long long most = 0;
    for (int64_t e = (int64_t)__shfl_sync(FULL, a, j) + lane_id(); e < bj; e += 32) {
      const long long w = p(__ldg(&col[e]), kj);
      c += w > 0;
      most = w > most ? w : most;
    }
    c = __reduce_add_sync(FULL, c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long x = __shfl_xor_sync(FULL, most, o);
      most = x > most ? x : most;
    }
    if (lane_id() == j) r = VdRow{c, most};
  }
  return r;
}

// One trimming round.  A node of a component with two or more nodes keeps an
// unlabelled successor and predecessor inside it, so it is never trimmed;
// labels written by other threads in the same round may or may not be seen,
// and either reading is valid.
__global__ void k_vd_trim(const int32_t* rp, const int32_t* ci, const int32_t* rrp, const int32_t* rci, int32_t n,
                          int32_t* lab, int32_t* changed) {
  bool any = false;
  VD_FOR_NODES(v) {
    if (lab[v] >= 0) continue;
    bool out = false, in = false;
    for (int32_t e = rp[v]; e < rp[v + 1] && !out; ++e) out = lab[ci[e]] < 0;
    if (out)
      for (int32_t e = rrp[v]; e < rrp[v + 1] && !in; ++e) in = lab[rci[e]] < 0;
    if (!out || !in) {
      lab[v] = (int32_t)v;
      any = true;
    }
  }
  if (__any_sync(FULL, any) && lane_id() == 0) *changed = 1;
}

// unlabelled nodes: colour = own id, not yet known to reach their root
__global__ void k_vd_color_init(const int32_t* lab, int32_t n, int32_t* col, int32_t* reach, int32_t* left) {
  bool any = false;
  VD_FOR_NODES(v) if (lab[v] < 0) {
    col[v] = (int32_t)v;
    reach[v] = 0;
    any = true;
  }
  if (__any_sync(FULL, any) && lane_id() == 0) *left = 1;
}

// colour <- the largest colour among unlabelled predecessors (monotone; a
// round without a change is the fixed point)
__global__ void k_vd_color(const int32_t* rrp, const int32_t* rci, int32_t n, const int32_t* lab, int32_t* col,
                           int32_t* changed) {
  bool any = false;
  VD_FOR_NODES(v) {
    if (lab[v] >= 0) continue;
    int32_t c = col[v];
    for (int32_t e = rrp[v]; e < rrp[v + 1]; ++e) {
      const int32_t u = rci[e];
      if (lab[u] < 0) {
        const int32_t cu = col[u];
        c = cu > c ? cu : c;
      }
    }
    if (c > col[v]) {
      col[v] = c;
      any = true;
    }
  }
  if (__any_sync(FULL, any) && lane_id() == 0) *changed = 1;
}

__global__ void k_vd_reach_roots(const int32_t* lab, const int32_t* col, int32_t n, int32_t* reach) {
  VD_FOR_NODES(v) if (lab[v] < 0 && col[v] == (int32_t)v) reach[v] = 1;
}

// a node reaches its root if a successor of the same colour does
__global__ void k_vd_reach(const int32_t* rp, const int32_t* ci, int32_t n, const int32_t* lab, const int32_t* col,
                           int32_t* reach, int32_t* changed) {
  bool any = false;
  VD_FOR_NODES(v) {
    if (lab[v] >= 0 || reach[v]) continue;
    const int32_t c = col[v];
    for (int32_t e = rp[v]; e < rp[v + 1]; ++e) {
      const int32_t u = ci[e];
      if (lab[u] < 0 && col[u] == c && reach[u]) {
        reach[v] = 1;
        any = true;
        break;
      }
    }
  }
  if (__any_sync(FULL, any) && lane_id() == 0) *changed = 1;
}

__global__ void k_vd_assign(const int32_t* col, const int32_t* reach, int32_t n, int32_t* lab) {
  VD_FOR_NODES(v) if (lab[v] < 0 && reach[v]) lab[v] = col[v];
}

// component sizes (the root's is known), and the arcs entering each component
// from another.  The lanes of a warp that add to the same label add once.
__global__ void k_vd_sizes(const int32_t* lab, int32_t n, const unsigned long long* best, const VdCore* core,
                           int32_t* sz) {
  const int32_t root = key_root(*best);
  if (blockIdx.x == 0 && threadIdx.x == 0) sz[root] = (int32_t)core->size;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    const int32_t L = v < n ? lab[v] : root;
    if (__any_sync(FULL, L != root && L != v)) {
      const unsigned same = __match_any_sync(FULL, L);
      if (L != root && lane_id() == __ffs(same) - 1) atomicAdd(&sz[L], __popc(same));
    } else if (L != root) {
      atomicAdd(&sz[L], 1);
    }
  }
}

__global__ void k_vd_indeg(const int32_t* rp, const int32_t* ci, const int32_t* rrp, const int32_t* rci, int32_t n,
                           int64_t m, const int32_t* lab, const unsigned long long* best, const int32_t* long_rows,
                           int32_t* cnt) {
  const int32_t root = key_root(*best);
  // the arcs into the root's component, most of all, are counted per warp
  unsigned into_root = 0;
  if (!*long_rows) {  // every entering arc leaves or enters a node outside the root's component
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
      const int64_t v = base + threadIdx.x;
      const int32_t L = v < n ? lab[v] : root;
      if (!__any_sync(FULL, L != root)) continue;
      int32_t a = 0, b = 0, ra = 0, rb = 0;
      if (L != root) {
        a = rp[v];
        b = rp[v + 1];
        ra = rrp[v];
        rb = rrp[v + 1];
      }
      into_root += vd_rows(ci, a, b, root, [&](int32_t x, int32_t k) { return (long long)(__ldg(&lab[x]) == k); }).count;
      const int32_t c =
          vd_rows(rci, ra, rb, L, [&](int32_t x, int32_t k) { return (long long)(__ldg(&lab[x]) != k); }).count;
      if (c) atomicAdd(&cnt[L], c);
    }
  } else {
    for_each_arc<4>(rp, ci, n, m, [&](const bool* ok, const int32_t* u, const int64_t*, const int32_t* v) {
      int32_t lu[4], lv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        lu[k] = ok[k] ? __ldg(&lab[u[k]]) : 0;
        lv[k] = ok[k] ? __ldg(&lab[v[k]]) : 0;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (lu[k] == lv[k]) continue;
        if (lv[k] == root)
          ++into_root;
        else
          atomicAdd(&cnt[lv[k]], 1);
      }
    });
  }
  into_root = __reduce_add_sync(FULL, into_root);
  if (into_root && lane_id() == 0) atomicAdd(&cnt[root], (int32_t)into_root);
}

// The heaviest path of the condensation, level by level in topological order
// (Kahn): a component is ready once every arc entering it has been
// processed; its heaviest path ending in it weighs w + best[label].
// Single-node components join the node frontier; a larger component ready at
// level l is marked rdy[label] = l, and at that level a pass over the in-arcs
// (balanced, whatever the rows' lengths) takes the arcs that leave it.  slot[0] of
// level l: the next frontier's size; slot[1]: a larger component is ready at
// level l + 1.

struct VdKahn {
  const int32_t *rp, *ci, *rrp, *rci, *lab, *sz;
  int32_t* cnt;
  long long* best;
  int32_t* rdy;
  int32_t n;
  int32_t root_label;
  long long root_w;
  long long* vd;
  const int32_t* long_rows;
};

__device__ __forceinline__ long long vd_weight(const VdKahn& K, int32_t L) {
  return L == K.root_label ? K.root_w : (long long)K.sz[L];
}

// all nodes whose label has no entering arc: level 0 (slot prev of level 0)
__global__ void k_vd_kahn_init(VdKahn K, int32_t* front, int32_t* slot) {
  const int32_t n = K.n;
  const int lane = lane_id();
  const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
  const int groups = n >= NODE_GROUPS * nthreads ? NODE_GROUPS : 1;
  for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32 * groups; base < n;
       base += nthreads * groups) {
    uint32_t bits = 0;
    for (int q = 0; q < groups; ++q) {
      const int64_t v = base + 32 * q + lane;
      if (v >= n) continue;
      const int32_t L = K.lab[v];
      if (K.cnt[L] != 0) continue;
      if (K.sz[L] == 1) {
        bits |= 1u << q;
      } else if (L == (int32_t)v) {
        K.rdy[L] = 0;
        slot[1] = 1;
      }
    }
    warp_append_groups(bits, groups, base, front, &slot[0]);
  }
}

// What a warp has for the root's component and for the bound, added once at
// its end: millions of nodes enter that component, and every node's path
// weight is a candidate, so each adding for itself queued on one address
// (the levels of R-MAT scale 24: 10.1 -> 3.1 ms).
struct VdWarp {
  long long vd, root_w;  // the largest path weight; the largest of an arc into the root's component
  int32_t into_root;     // those arcs
};

// The arcs a .. b of one ready single-node component u (path weight w) into
// other components, by a warp.
__device__ __forceinline__ void vd_kahn_row(const VdKahn& K, int32_t u, long long w, int32_t a, int32_t b,
                                            int32_t level, int32_t* next, int32_t* slot, VdWarp& W) {
  const int lane = lane_id();
  for (int64_t base = a; base < b; base += 32) {
    const int64_t e = base + lane;
    bool push = false;
    int32_t Ly = u;  // this lane's arc enters no other component unless set below
    if (e < b) Ly = K.lab[K.ci[e]];
    const int32_t k0 = __popc(__ballot_sync(FULL, Ly != u && Ly == K.root_label));
    if (k0) {
      W.into_root += k0;
      W.root_w = w > W.root_w ? w : W.root_w;
    }
    // lanes whose arcs enter the same component update it once
    const bool on = Ly != u && Ly != K.root_label;
    if (__any_sync(FULL, on)) {
      const unsigned same = __match_any_sync(FULL, Ly);
      if (on && lane == __ffs(same) - 1) {
        atomicMax(&K.best[Ly], w);
        const int k = __popc(same);
        if (atomicSub(&K.cnt[Ly], k) == k) {
          if (K.sz[Ly] == 1) {
            push = true;  // a single-node component is its node
          } else {
            K.rdy[Ly] = level + 1;
            slot[1] = 1;
          }
        }
      }
    }
    const unsigned got = __ballot_sync(FULL, push);
    if (got) {
      int32_t at = 0;
      if (lane == 0) at = atomicAdd(&slot[0], __popc(got));
      at = __shfl_sync(FULL, at, 0);
      if (push) next[at + __popc(got & ((1u << lane) - 1u))] = Ly;
    }
  }
}

__global__ void k_vd_kahn_level(VdKahn K, int64_t m, const int32_t* front, const int32_t* prev, int32_t* next,
                                int32_t* slot, int32_t level) {
  const int64_t nfront = prev[0];
  VdWarp W = {0, 0, 0};
  // a warp takes 32 ready nodes at a time, and the rows of those that have one
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~31ll; i0 < nfront;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int lane = lane_id();
    int32_t u = 0, a = 0, b = 0;
    long long w = 0;
    if (i0 + lane < nfront) {
      u = front[i0 + lane];
      a = K.rp[u];
      b = K.rp[u + 1];
      w = vd_weight(K, u) + K.best[u];  // a single-node component's label is its node
    }
    W.vd = w > W.vd ? w : W.vd;
    for (unsigned rows = __ballot_sync(FULL, b > a); rows; rows &= rows - 1) {
      const int j = __ffs(rows) - 1;
      vd_kahn_row(K, __shfl_sync(FULL, u, j), __shfl_sync(FULL, w, j), __shfl_sync(FULL, a, j),
                  __shfl_sync(FULL, b, j), level, next, slot, W);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long x = __shfl_xor_sync(FULL, W.vd, o);
    W.vd = x > W.vd ? x : W.vd;
  }
  if (lane_id() == 0) {
    if (W.vd > 0) atomicMax(K.vd, W.vd);
    if (W.into_root) {
      atomicMax(&K.best[K.root_label], W.root_w);
      if (atomicSub(&K.cnt[K.root_label], W.into_root) == W.into_root) {
        if (K.sz[K.root_label] == 1) {
          next[atomicAdd(&slot[0], 1)] = K.root_label;
        } else {
          K.rdy[K.root_label] = level + 1;
          slot[1] = 1;
        }
      }
    }
  }
  if (!prev[1]) return;
  // larger components ready at this level: their representatives' path
  // weights, then every arc leaving one of their nodes
  const int32_t n = K.n;
  VD_FOR_NODES(v) {
    const int32_t L = K.lab[v];
    if (L == (int32_t)v && K.sz[L] > 1 && K.rdy[L] == level) atomicMax(K.vd, vd_weight(K, L) + K.best[L]);
  }
  // The root's component was ready at this level or before (a value that this
  // level's launch leaves as it is, or moves from -1 to level + 1): the nodes
  // still waiting are outside it, and all their rows are short.
  const int32_t root_rdy = *(volatile const int32_t*)&K.rdy[K.root_label];
  if (!*K.long_rows && root_rdy >= 0 && root_rdy <= level) {
    const int lane = lane_id();
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int groups = n >= NODE_GROUPS * nthreads ? NODE_GROUPS : 1;
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32 * groups; base < n;
         base += nthreads * groups) {
      uint32_t ready = 0;
      for (int q = 0; q < groups; ++q) {
        const int64_t y = base + 32 * q + lane;
        int32_t L = K.root_label, a = 0, b = 0;
        if (y < n) L = K.lab[y];
        const bool waits = *(volatile const int32_t*)&K.cnt[L] > 0;
        if (!__any_sync(FULL, waits)) continue;
        if (waits && y < n) {
          a = K.rrp[y];
          b = K.rrp[y + 1];
        }
        const VdRow r = vd_rows(K.rci, a, b, L, [&](int32_t u, int32_t ly) {
          const int32_t lu = K.lab[u];
          return lu != ly && K.sz[lu] > 1 && K.rdy[lu] == level ? vd_weight(K, lu) + K.best[lu] : 0ll;
        });
        if (r.count) {
          atomicMax(&K.best[L], r.most);
          if (atomicSub(&K.cnt[L], r.count) == r.count) {
            if (K.sz[L] == 1) {
              ready |= 1u << q;  // a single-node component is its node
            } else {
              K.rdy[L] = level + 1;
              slot[1] = 1;
            }
          }
        }
      }
      warp_append_groups(ready, groups, base, next, &slot[0]);
    }
    return;
  }
  // Pulled along the in-arcs of the components still waiting: those are few
  // on power-law graphs (the ready giant component holds most arcs), and a
  // row's arcs from ready components make one update, not one each.
  for_each_arc<4>(K.rrp, K.rci, n, m, [&](const bool* ok, const int32_t* y, const int64_t*, const int32_t* u) {
    int32_t Ly[4], Lu[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) Ly[k] = ok[k] ? K.lab[y[k]] : -1;
#pragma unroll
    for (int k = 0; k < 4; ++k) Lu[k] = Ly[k] >= 0 && *(volatile const int32_t*)&K.cnt[Ly[k]] > 0 ? K.lab[u[k]] : Ly[k];
    unsigned ready = 0;  // bit k: this lane's update made Ly[k], a single node, ready
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
      const int32_t ly = k == 0 ? Ly[0] : k == 1 ? Ly[1] : k == 2 ? Ly[2] : Ly[3];
      const int32_t lu = k == 0 ? Lu[0] : k == 1 ? Lu[1] : k == 2 ? Lu[2] : Lu[3];
      const bool on = lu != ly && K.sz[lu] > 1 && K.rdy[lu] == level;
      if (!__any_sync(FULL, on)) continue;
      // the lanes whose arcs go from one component into the same other one
      const unsigned long long pair = on ? ((unsigned long long)(uint32_t)lu << 32) | (uint32_t)ly : ~0ull;
      const unsigned same = __match_any_sync(FULL, pair);
      if (on && lane_id() == __ffs(same) - 1) {
        atomicMax(&K.best[ly], vd_weight(K, lu) + K.best[lu]);
        const int c = __popc(same);
        if (atomicSub(&K.cnt[ly], c) == c) {
          if (K.sz[ly] == 1) {
            ready |= 1u << k;
          } else {
            K.rdy[ly] = level + 1;
            slot[1] = 1;
          }
        }
      }
    }
    const int total = __reduce_add_sync(FULL, __popc(ready));
    if (!total) return;
    int32_t at = 0;
    if (lane_id() == 0) at = atomicAdd(&slot[0], total);
    at = __shfl_sync(FULL, at, 0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned got = __ballot_sync(FULL, (ready >> k) & 1u);
      if ((ready >> k) & 1u) next[at + __popc(got & ((1u << lane_id()) - 1u))] = Ly[k];  // its node
      at += __popc(got);
    }
  });
}

// ============================================================== host side
thread_local std::string g_last_error;

kadabra_status fail(kadabra_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

#define KCK(call)                                                                                   \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess)                                                                          \
      return fail(e_ == cudaErrorMemoryAllocation ? KADABRA_ERR_OOM : KADABRA_ERR_CUDA,             \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                              \
  } while (0)

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

int ceil_log2(uint64_t x) {
  int k = 0;
  while ((1ull << k) < x) ++k;
  return k;
}

}  // namespace

namespace {

// Sampler workspace: everything a sampler launch needs besides the graph and
// its outputs.  A standalone graph owns one; the graphs of a batch share the
// batch's, sized for its largest graph (their calls must not overlap).
// A device-driven main loop (CUDA graph) and its device state, rebuilt only
// when the launch parameters it was captured with change.
struct LoopCache {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaStream_t cap = nullptr;      // capture stream
  void* dev = nullptr;             // LoopState, G LoopGraph, G Job, G CheckTabJob
  size_t dev_bytes = 0;
  std::vector<unsigned char> sig;  // launch parameters the graph was built with
  void drop_graph() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    exec = nullptr;
    graph = nullptr;
    sig.clear();
  }
  ~LoopCache() {
    drop_graph();
    if (cap) cudaStreamDestroy(cap);
    if (dev) cudaFree(dev);
  }
};

struct Workspace {
  bool ready = false;
  int device = 0, num_sms = 0;
  int32_t max_n = 0;
  int64_t max_m = 0;
  int grid_fast = 0, grid_big = 0, grid_gm = 0, grid_compact = 0, grid_tiny = 0, grid_warp = 0;
  size_t smem_fast = 0, smem_big = 0, smem_compact = 0, smem_tiny = 0, smem_warp = 0;
  unsigned long long* ctr = nullptr;
  int32_t* status = nullptr;
  unsigned long long* qb = nullptr;  // queue for tier B
  unsigned long long* ql = nullptr;  // queue for tier L
  unsigned long long* qs = nullptr;  // queue for tier S (fed by tier W or k_screen)
  uint64_t deferred_cap = 0;
  PiEntry* pi_fast = nullptr;
  PiEntry* pi_gm = nullptr;
  int pcap_gm = 0;
  unsigned char* med_base = nullptr;
  size_t med_stride = 0;
  unsigned char* gm_base = nullptr;
  size_t gm_stride = 0;
  int gm_hlog = 0;
  int gm_lcap = 0;
  Job* d_jobs = nullptr;  // job array of multi-graph launches
  int jobs_cap = 0;
  void* d_checks = nullptr;  // stop-test descriptors and results of runs
  int checks_cap = 0;
  void* d_nz = nullptr;  // warm-up count compaction descriptors of runs
  int nz_cap = 0;
  LoopCache loop;  // device-driven loop of batched runs (one-graph runs keep theirs in the graph object)
  std::vector<void*> allocs;
  ~Workspace() {
    for (void* p : allocs)
      if (p) cudaFree(p);
  }
};

}  // namespace

// graph object (opaque in the ABI)
struct kadabra_graph {
  int32_t n = 0;
  int64_t m = 0;
  int directed = 0;
  int32_t *rp = nullptr, *ci = nullptr, *rrp = nullptr, *rci = nullptr;
  int64_t vd = 0;
  double idle = 0.0;           // share of the samples that end at a root without arcs
  bool csr_beyond_l2 = false;  // forward (+ reverse) CSR larger than the L2: long rows are searched
  int device = 0;
  int num_sms = 0;
  uint32_t flags = 0;
  Workspace* ws = nullptr;
  bool owns_ws = false;
  bool is_view = false;  // a batch's view: released with the batch
  // run buffers
  uint32_t *counts = nullptr, *count0 = nullptr;
  double* btilde = nullptr;
  long long* totals = nullptr;
  double* lntab = nullptr;  // computeDelta table, ln(1/delta) by warm-up count
  uint64_t lntab_cap = 0;
  // top-k mode (allocated on first use)
  uint32_t* count_pre = nullptr;     // preliminary-estimate hits (Sec. 5)
  double *lnLv = nullptr, *lnUv = nullptr;  // per-node ln(1/delta_L), ln(1/delta_U)
  unsigned long long* tk_cand = nullptr;    // first-stage selection survivors
  void* tk_dev = nullptr;            // TopkJob + TopkOut
  void* tk_stage = nullptr;          // scatter staging: ids, lnL, lnU values
  size_t tk_stage_cap = 0;           // entries
  struct TuneTable {  // autotuned setup by probe size class and allowed set (-1: not yet)
    int v[18][16];
    uint32_t flags = 0;  // the launch flags of its probes; another set starts it anew
    TuneTable() { std::memset(v, 0xFF, sizeof(v)); }
  } tier_choice, shared_choice;      // launches of its own; a batch's, tuned on this graph
  uint64_t fingerprint = 0;          // shape and sampled CSR entries (key of the autotuner's cache)
  // device-driven main loop of one-graph all-nodes runs (a CUDA graph), built on first use
  LoopCache loop;
  std::vector<void*> allocs;  // CSR copies and run buffers
};

namespace {
// internal launch flag: the graph's CSR exceeds the L2, so pass 1 searches
// its long rows (KADABRA_FLAG_ASYNC_SCAN asks for that explicitly)
constexpr uint32_t FLAG_VEC_AUTO = 1u << 31;
// internal launch flag: no graph of the launch has more than TINY_NODES nodes
constexpr uint32_t FLAG_TINY_AUTO = 1u << 29;
// the flags a launch shared by several graphs takes from any of them (they
// change no result; the tier-skipping flags stay per graph)
constexpr uint32_t SHARED_LAUNCH_FLAGS = KADABRA_FLAG_WARP_TIER | KADABRA_FLAG_ASYNC_SCAN | FLAG_VEC_AUTO;

uint32_t launch_flags(const kadabra_graph* g) {
  return g->flags | (g->csr_beyond_l2 ? FLAG_VEC_AUTO : 0u) | (g->n <= TINY_NODES ? FLAG_TINY_AUTO : 0u);
}

// k_screen before tier S, in launches of at least SCREEN_SAMPLES samples at
// least SCREEN_MIN of which are expected to end at a root without arcs (over
// all graphs of the launch).  It costs a launch (3 to 5 us) and a second draw
// of the others; without and with it, in us: 1,000 samples 109 and 114 (R-MAT
// scale 17); 8,192 445 and 436 (scale 20); 16,384 249 and 238 (scale 17);
// 65,536 1,092 and 996 (scale 20).  With a quarter of the samples idle, random
// directed graphs of mean degree 2, 8 and 16: 8,192 samples 773 and 766, 404
// and 408, 206 and 207; 65,536 4,738 and 4,697, 2,751 and 2,700, 1,369 and
// 1,325.
constexpr double SCREEN_MIN = 0.25;
constexpr uint64_t SCREEN_SAMPLES = 8192;
void choose_screen(SampleParams& P, uint64_t samples, double idle_samples) {
  if (samples >= SCREEN_SAMPLES && idle_samples >= SCREEN_MIN * (double)samples) P.tier_flags |= TF_SCREEN;
}
}  // namespace

// G graphs whose CSRs share one device arena
struct kadabra_batch {
  int32_t G = 0;
  std::vector<kadabra_graph*> views;
  Workspace ws;
  void* arena = nullptr;
};

namespace {

kadabra_status dev_alloc(std::vector<void*>& allocs, void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
  if (e != cudaSuccess)
    return fail(KADABRA_ERR_OOM, std::string("cudaMalloc(") + std::to_string(bytes) + "): " + cudaGetErrorString(e));
  allocs.push_back(*p);
  return KADABRA_OK;
}

#define KTRY(expr)                        \
  do {                                    \
    kadabra_status s_ = (expr);           \
    if (s_ != KADABRA_OK) return s_;      \
  } while (0)

void dev_free(std::vector<void*>& allocs, void* p) {
  if (!p) return;
  for (auto& a : allocs)
    if (a == p) a = nullptr;
  cudaFree(p);
}

// Allocations of graph objects and graph loads come from the device's
// default memory pool with no release threshold, so that memory freed by
// one load is handed to the next without cudaMalloc or cudaFree (graphs
// are loaded and freed once per end-to-end run).  Allocated in order on the
// legacy stream, which is synchronized before the memory is used elsewhere;
// freed after the device is idle.  kadabra_release_cached returns the
// pool's free memory to the device (cudaMemPoolTrimTo).
void pool_setup(int dev) {
  static std::mutex mu;
  static std::vector<int> done;
  std::lock_guard<std::mutex> lk(mu);
  for (int d : done)
    if (d == dev) return;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  done.push_back(dev);
}

kadabra_status pool_alloc(void** p, size_t bytes) {
  int dev = 0;
  KCK(cudaGetDevice(&dev));
  pool_setup(dev);
  cudaError_t e = cudaMallocAsync(p, bytes ? bytes : 16, 0);
  if (e == cudaSuccess) e = cudaStreamSynchronize(0);
  if (e != cudaSuccess)
    return fail(KADABRA_ERR_OOM, std::string("cudaMallocAsync(") + std::to_string(bytes) + "): " + cudaGetErrorString(e));
  return KADABRA_OK;
}

void pool_free(void* p) {
  if (p) cudaFreeAsync(p, 0);
}

kadabra_status gdev_alloc(std::vector<void*>& allocs, void** p, size_t bytes) {
  KTRY(pool_alloc(p, bytes));
  allocs.push_back(*p);
  return KADABRA_OK;
}

void gdev_free(std::vector<void*>& allocs, void* p) {
  if (!p) return;
  for (auto& a : allocs)
    if (a == p) a = nullptr;
  pool_free(p);
}

kadabra_status ensure_ws(Workspace* w, uint64_t deferred_need, int njobs) {
  if (!w->ready) {
    KCK(cudaSetDevice(w->device));
    w->smem_fast = fast_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w->smem_fast));
    KCK(cudaFuncSetAttribute(k_sample<0, SL_FAST, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)w->smem_fast));
    int per_sm = 0;
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<0>, 32 * NW_S, w->smem_fast));
    if (per_sm < 1) return fail(KADABRA_ERR_CAPACITY, "sampler does not fit on an SM");
    w->grid_fast = w->num_sms * per_sm;
    w->smem_compact = compact_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample<0, SL_COMPACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w->smem_compact));
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<0, SL_COMPACT>, 32 * NW_CMP, w->smem_compact));
    w->grid_compact = w->num_sms * std::max(per_sm, 1);
    w->smem_tiny = tiny_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample<0, SL_TINY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w->smem_tiny));
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<0, SL_TINY>, 32 * NW_TINY, w->smem_tiny));
    w->grid_tiny = w->num_sms * std::max(per_sm, 1);
    w->smem_warp = warp_tier_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w->smem_warp));
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample_warp, 32 * WT_WARPS, w->smem_warp));
    w->grid_warp = w->num_sms * std::max(per_sm, 1);
    w->smem_big = big_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w->smem_big));
    KCK(cudaFuncSetAttribute(k_sample<2, SL_FAST, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)w->smem_big));
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<2>, 32 * NW_BIG, w->smem_big));
    if (per_sm < 1) return fail(KADABRA_ERR_CAPACITY, "large-table sampler does not fit on an SM");
    w->grid_big = w->num_sms * per_sm;
    // n-sized tables for the rare samples beyond the others: hash of >= 2n slots, lists of n
    w->gm_hlog = std::max(12, ceil_log2(2ull * (uint64_t)w->max_n));
    w->gm_lcap = w->max_n;
    w->pcap_gm = (int)std::min<int64_t>(std::max<int64_t>(w->max_m, 1024), 1 << 18);
    {
      size_t a, b, c2, d;
      w->gm_stride = gm_layout(w->gm_hlog, w->gm_lcap, GM_MAXD, &a, &b, &c2, &d);
      w->med_stride = gm_layout(MED_HLOG, MED_LCAP, MED_MAXD, &a, &b, &c2, &d);
    }
    const size_t per_cta = w->gm_stride + sizeof(PiEntry) * PI_SEGS * (size_t)w->pcap_gm;
    // such samples are rare on small-world graphs; 1 GiB of tables keeps
    // at least a few CTAs busy on them
    const size_t budget = (size_t)1 << 30;
    w->grid_gm = (int)std::max<size_t>(1, std::min<size_t>((size_t)w->num_sms, budget / per_cta));
    void* p;
    KTRY(dev_alloc(w->allocs, &p, Q_COUNT * sizeof(unsigned long long)));
    w->ctr = (unsigned long long*)p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(int32_t)));
    w->status = (int32_t*)p;
    KCK(cudaMemset(w->status, 0, sizeof(int32_t)));
    KTRY(dev_alloc(w->allocs, &p, sizeof(PiEntry) * PI_SEGS * (size_t)FAST_PCAP * std::max(w->grid_fast, w->grid_compact)));
    w->pi_fast = (PiEntry*)p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(PiEntry) * PI_SEGS * (size_t)w->pcap_gm * w->grid_gm));
    w->pi_gm = (PiEntry*)p;
    KTRY(dev_alloc(w->allocs, &p, w->gm_stride * w->grid_gm));
    w->gm_base = (unsigned char*)p;
    KCK(cudaMemset(w->gm_base, 0, w->gm_stride * w->grid_gm));
    for (int b = 0; b < w->grid_gm; ++b)  // every key word EMPTY (sigma stays 0)
      KCK(cudaMemset(w->gm_base + (size_t)b * w->gm_stride, 0xFF, sizeof(unsigned long long) << w->gm_hlog));
    KTRY(dev_alloc(w->allocs, &p, w->med_stride * w->grid_big));
    w->med_base = (unsigned char*)p;
    KCK(cudaMemset(w->med_base, 0, w->med_stride * w->grid_big));
    for (int b = 0; b < w->grid_big; ++b)
      KCK(cudaMemset(w->med_base + (size_t)b * w->med_stride, 0xFF, sizeof(unsigned long long) << MED_HLOG));
    KCK(cudaDeviceSynchronize());
    w->ready = true;
  }
  if (deferred_need > w->deferred_cap) {
    KCK(cudaDeviceSynchronize());
    dev_free(w->allocs, w->qb);
    dev_free(w->allocs, w->ql);
    dev_free(w->allocs, w->qs);
    w->qb = w->ql = w->qs = nullptr;
    const uint64_t cap = std::max<uint64_t>(deferred_need, 1 << 16);
    void* p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(unsigned long long) * cap));
    w->qb = (unsigned long long*)p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(unsigned long long) * cap));
    w->ql = (unsigned long long*)p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(unsigned long long) * cap));
    w->qs = (unsigned long long*)p;
    w->deferred_cap = cap;
  }
  if (njobs > w->jobs_cap) {
    KCK(cudaDeviceSynchronize());
    dev_free(w->allocs, w->d_jobs);
    void* p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(Job) * (size_t)njobs));
    w->d_jobs = (Job*)p;
    w->jobs_cap = njobs;
  }
  return KADABRA_OK;
}

// per-graph run buffers (hit counters, b~, totals)
kadabra_status ensure_run_buffers(kadabra_graph* g) {
  if (g->counts) return KADABRA_OK;
  void* p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(uint32_t) * (size_t)g->n));
  g->counts = (uint32_t*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(uint32_t) * (size_t)g->n));
  g->count0 = (uint32_t*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(double) * (size_t)g->n));
  g->btilde = (double*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(long long) * KADABRA_NSTAT));
  g->totals = (long long*)p;
  return KADABRA_OK;
}

kadabra_status ensure_workspace(kadabra_graph* g, uint64_t deferred_need) {
  KTRY(ensure_ws(g->ws, deferred_need, 0));
  return ensure_run_buffers(g);
}

GraphDev graph_dev(const kadabra_graph* g) {
  GraphDev d;
  d.n = g->n;
  d.m = g->m;
  d.rp = g->rp;
  d.ci = g->ci;
  d.rrp = g->directed ? g->rrp : g->rp;
  d.rci = g->directed ? g->rci : g->ci;
  return d;
}

SampleParams ws_params(const Workspace* w, uint32_t flags) {
  SampleParams P;
  std::memset(&P, 0, sizeof(P));
  P.njobs = 1;
  P.ctr = w->ctr;
  P.qb = w->qb;
  P.ql = w->ql;
  P.deferred_cap = w->deferred_cap;
  P.status = w->status;
  P.med_base = w->med_base;
  P.med_stride = w->med_stride;
  P.med_hlog = MED_HLOG;
  P.med_lcap = MED_LCAP;
  P.gm_base = w->gm_base;
  P.gm_stride = w->gm_stride;
  P.gm_hlog = w->gm_hlog;
  P.gm_lcap = w->gm_lcap;
  P.tier_flags = 0;
  if (flags & KADABRA_FLAG_GLOBAL_TABLES) P.tier_flags |= TF_SKIP_S | TF_SKIP_B | TF_SKIP_M;
  if (flags & KADABRA_FLAG_MEDIUM_TABLES) P.tier_flags |= TF_SKIP_S | TF_SKIP_B;
  if (flags & KADABRA_FLAG_LARGE_SHARED_TABLES) P.tier_flags |= TF_SKIP_S;
  if (flags & KADABRA_FLAG_WARP_TIER) P.tier_flags |= TF_WARP;
  if (flags & (KADABRA_FLAG_ASYNC_SCAN | FLAG_VEC_AUTO)) P.tier_flags |= TF_VEC;
  if (flags & KADABRA_FLAG_FRONTIER_SEGMENTS) P.tier_flags |= TF_SEG64;
  if (flags & KADABRA_FLAG_COMPACT_TABLES) P.tier_flags |= TF_COMPACT;
  if (flags & FLAG_TINY_AUTO) P.tier_flags |= TF_TINY;
  return P;
}

SampleParams base_params(kadabra_graph* g) {
  SampleParams P = ws_params(g->ws, launch_flags(g));
  P.job0.g = graph_dev(g);
  return P;
}

// launches the main sampler grid, then the large-table pass and the
// n-sized-table pass for the samples queued by the launch before (each exits
// at once when its queue is empty)
// variant bit 0: the compact tier-S layout with one more CTA per SM, or on
// graphs of at most TINY_NODES nodes the small one
// variant bit 1: tier W (one warp per sample) first; tier S takes only the
// samples it queues
kadabra_status launch_sampler_kernels(Workspace* w, SampleParams P, cudaStream_t st, int variant = 0) {
  P.pi_base = w->pi_fast;
  P.pcap = FAST_PCAP;
  if (((variant & 2) || (P.tier_flags & TF_WARP)) && !(P.tier_flags & TF_SKIP_S)) {
    P.q0 = w->qs;  // tier W's overflow queue, tier S's input
    k_sample_warp<<<w->grid_warp, 32 * WT_WARPS, w->smem_warp, st>>>(P);
    KCK(cudaGetLastError());
  } else if ((P.tier_flags & TF_SCREEN) && !(P.tier_flags & TF_SKIP_S)) {
    P.q0 = w->qs;
    k_screen<<<2 * w->num_sms, 256, 0, st>>>(P);
    KCK(cudaGetLastError());
  }
  const bool rg = (P.tier_flags & TF_VEC) != 0;
  if ((variant & 1) && (P.tier_flags & TF_TINY) && !(P.tier_flags & TF_COMPACT)) {
    // more CTAs share the candidate buffers; a sample beyond its part goes on to tier B
    SampleParams T = P;
    T.pcap = (int)((int64_t)FAST_PCAP * std::max(w->grid_fast, w->grid_compact) / w->grid_tiny);
    k_sample<0, SL_TINY><<<w->grid_tiny, 32 * NW_TINY, w->smem_tiny, st>>>(T);
  } else if ((variant & 1) || ((P.tier_flags & TF_COMPACT) && !rg))  // the compact layout has no beyond-L2 variant
    k_sample<0, SL_COMPACT><<<w->grid_compact, 32 * NW_CMP, w->smem_compact, st>>>(P);
  else if (rg)
    k_sample<0, SL_FAST, true><<<w->grid_fast, 32 * NW_S, w->smem_fast, st>>>(P);
  else
    k_sample<0><<<w->grid_fast, 32 * NW_S, w->smem_fast, st>>>(P);
  KCK(cudaGetLastError());
  if (rg)  // tier B (and M): the scan kind of tier S
    k_sample<2, SL_FAST, true><<<w->grid_big, 32 * NW_BIG, w->smem_big, st>>>(P);
  else
    k_sample<2><<<w->grid_big, 32 * NW_BIG, w->smem_big, st>>>(P);
  KCK(cudaGetLastError());
  P.pi_base = w->pi_gm;
  P.pcap = w->pcap_gm;
  if (rg)
    k_sample<1, SL_FAST, true><<<w->grid_gm, 32 * NW_S, CTL_BYTES<NW_S> + sizeof(LongRows), st>>>(P);
  else
    k_sample<1><<<w->grid_gm, 32 * NW_S, CTL_BYTES<NW_S> + sizeof(LongRows), st>>>(P);
  KCK(cudaGetLastError());
  return KADABRA_OK;
}

kadabra_status launch_sampler(Workspace* w, SampleParams P, cudaStream_t st, int variant = 0) {
  KCK(cudaMemsetAsync(w->ctr, 0, Q_COUNT * sizeof(unsigned long long), st));
  return launch_sampler_kernels(w, P, st, variant);
}

kadabra_status read_status(Workspace* w, cudaStream_t st) {
  int32_t h = 0;
  KCK(cudaMemcpyAsync(&h, w->status, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  KCK(cudaStreamSynchronize(st));
  if (h != 0) {
    KCK(cudaMemsetAsync(w->status, 0, sizeof(int32_t), st));
    KCK(cudaStreamSynchronize(st));
    std::string what = h == KADABRA_ERR_SIGMA_OVERFLOW ? "a shortest-path count exceeded 2^64-1"
                       : h == KADABRA_ERR_CAPACITY     ? "a sampler capacity bound was exceeded"
                                                       : "the sampler reported an internal error";
#ifdef KADABRA_CHECKED
    unsigned long long ck = 0;
    if (cudaMemcpyFromSymbol(&ck, g_checked, sizeof(ck)) == cudaSuccess && ck)
      what += " (checked build: index check " + std::to_string(ck >> 40) + " failed at index " +
              std::to_string(ck & ((1ull << 40) - 1)) + ")";
#endif
    return fail((kadabra_status)h, what);
  }
  return KADABRA_OK;
}

// ---------------------------------------------------------------- omega
int64_t floor_log2_pos(int64_t x) {  // x >= 1
  int64_t k = -1;
  while (x > 0) {
    x >>= 1;
    ++k;
  }
  return k;
}

double omega_host(double lambda, double delta, int64_t vd) {
  const int64_t fl = vd - 2 >= 1 ? floor_log2_pos(vd - 2) : 0;
  return (0.5 / (lambda * lambda)) * ((double)(fl + 1) + std::log(2.0 / delta));
}

// Samples between stop tests when the caller leaves it to the library: about
// 32 tests up to the cap, at least 1024 samples each.  A function of omega
// only, so every path that uses it samples and stops identically.
uint64_t auto_check_interval(double omega) {
  const double k = std::ceil(omega / 32.0);
  return k < 1024.0 ? 1024 : (uint64_t)k;
}

// ---------------------------------------------------------------- computeDelta
// Alg. 2 with lambda_L = lambda_U = lambda.  In this mode delta(v) depends
// only on v's warm-up count k = count0(v) (at most alpha), so the result is a
// table lnT[k] = ln(1/delta) for k = 0..kmax.  nz holds the non-zero warm-up counts
// in increasing node order: the bisection's sum runs over them in that order
// (the other nodes add exact zeros), with the exponential of each distinct
// count evaluated once per step.
kadabra_status compute_delta_table(int64_t n, const uint32_t* nz, size_t nnz, uint64_t alpha, uint64_t kmax,
                                   double omega, double lambda, double delta, double eps, double* lnT,
                                   double* C_out) {
  std::unordered_map<uint32_t, size_t> idx_of;
  std::vector<uint32_t> distinct;
  std::vector<size_t> which(nnz);
  for (size_t i = 0; i < nnz; ++i) {
    auto it = idx_of.find(nz[i]);
    if (it == idx_of.end()) {
      it = idx_of.emplace(nz[i], distinct.size()).first;
      distinct.push_back(nz[i]);
    }
    which[i] = it->second;
  }
  for (uint32_t k : distinct)
    if (k > kmax) return fail(KADABRA_ERR_INTERNAL, "computeDelta: a warm-up count exceeds the table");
  std::vector<double> cval(distinct.size()), ex(distinct.size());
  for (size_t k = 0; k < distinct.size(); ++k) {
    const double b0 = (double)distinct[k] / (double)alpha;
    cval[k] = ((2.0 * b0) * omega) / (lambda * lambda);
  }
  const double target = (delta / 2.0) - (eps * delta);
  auto sum_at = [&](double C) {
    for (size_t k = 0; k < distinct.size(); ++k) ex[k] = std::exp(-C / cval[k]);
    double sum = 0.0;
    for (size_t i = 0; i < nnz; ++i) {
      const double e = ex[which[i]];
      sum += e + e;
    }
    return sum;
  };
  double C = 0.0;
  if (nnz) {
    double lo = 0.0, hi = 1.0;
    int guard = 0;
    while (!(sum_at(hi) <= target)) {
      lo = hi;
      hi = 2.0 * hi;
      if (++guard > 2100) return fail(KADABRA_ERR_INTERNAL, "computeDelta: no bracket for C");
    }
    for (guard = 0; guard < 4000; ++guard) {
      const double mid = 0.5 * (lo + hi);
      if (mid <= lo || mid >= hi) break;
      if (sum_at(mid) <= target)
        hi = mid;
      else
        lo = mid;
    }
    C = hi;
  }
  const double floor_term = (eps * delta) / (2.0 * (double)n);
  for (uint64_t k = 0; k <= kmax; ++k) lnT[k] = -std::log(0.0 + floor_term);
  for (size_t k = 0; k < distinct.size(); ++k) lnT[distinct[k]] = -std::log(std::exp(-C / cval[k]) + floor_term);
  *C_out = C;
  return KADABRA_OK;
}

// the same, with per-node outputs (ln(1/delta_L) = ln(1/delta_U) for every node)
kadabra_status compute_delta_host(int64_t n, const uint32_t* count0, uint64_t alpha, double omega, double lambda,
                                  double delta, double eps, double* lnL, double* lnU, double* C_out) {
  std::vector<uint32_t> nz;
  uint64_t top = 0;
  for (int64_t v = 0; v < n; ++v)
    if (count0[v]) {
      nz.push_back(count0[v]);
      top = std::max<uint64_t>(top, count0[v]);
    }
  const uint64_t kmax = std::max<uint64_t>(alpha, top);
  std::vector<double> lnT(kmax + 1);
  KTRY(compute_delta_table(n, nz.data(), nz.size(), alpha, kmax, omega, lambda, delta, eps, lnT.data(), C_out));
  for (int64_t v = 0; v < n; ++v) lnL[v] = lnU[v] = lnT[count0[v]];
  return KADABRA_OK;
}

// Phase timing of graph loads and top-k runs on stderr when the environment
// variable KADABRA_TRACE is set (each phase ends with a device
// synchronisation then, which also slows the traced call).
struct LoadTrace {
  bool on;
  const char* what;
  std::chrono::steady_clock::time_point t0;
  explicit LoadTrace(const char* w = "load")
      : on(std::getenv("KADABRA_TRACE") != nullptr), what(w), t0(std::chrono::steady_clock::now()) {}
  void mark(const char* phase) {
    if (!on) return;
    cudaDeviceSynchronize();
    const auto t1 = std::chrono::steady_clock::now();
    std::fprintf(stderr, "kadabra %s: %-34s %8.3f ms\n", what, phase,
                 std::chrono::duration<double, std::milli>(t1 - t0).count());
    t0 = t1;
  }
};

// Device scratch of one graph load, one allocation: the check results, the
// reciprocal-arc counts (directed graphs) and the BFS state.
struct LoadHead {  // the start of the scratch, read back at once
  unsigned err, pad;             // error bits
  unsigned long long lt_gt[2];   // the mirror test's two arc counts
  unsigned long long best;       // the VD root's key
  int32_t floor_deg, unused[7];  // the largest max(out, in) degree (directed graphs)
  int32_t fp[64];                // fingerprint entries
};
static_assert(offsetof(LoadHead, fp) == 64, "what load_scratch clears");

struct LoadScratch {
  unsigned* err;               // [0] error bits
  unsigned long long* lt_gt;   // the mirror test's two arc counts
  int32_t* fp;                 // 64 fingerprint entries
  unsigned long long* best;    // the VD root's key
  RowTree tree;                // of the searched column array (graphs beyond the L2)
  int32_t* floor_deg;          // the largest max(out, in) degree (directed graphs)
  int32_t* cnt;                // BFS level counters: slot l % 8 holds {next frontier's size, items, its arcs} of level l
  uint32_t* recip;             // n (directed graphs), else null
  VdCore* core;                // the root's component: size, e_out, e_in
  int32_t *dist, *qa, *qb;     // n each: distances from r, BFS queues
  int32_t* dist_b;             // n (directed graphs): distances to r, else null
  BfsItem* items;
  int32_t items_cap;
  void* base;
};

uint64_t l2_bytes(int device) {
  int l2 = 0;
  if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device) != cudaSuccess) l2 = 0;
  return l2 > 0 ? (uint64_t)l2 : ~0ull;
}
uint64_t csr_bytes(const kadabra_graph* g) {
  return (4ull * ((uint64_t)g->n + 1) + 4ull * (uint64_t)g->m) * (g->directed ? 2 : 1);
}

kadabra_status load_scratch(const kadabra_graph* g, LoadScratch* S) {
  const size_t n = (size_t)g->n;
  const int64_t cap = std::min<int64_t>((int64_t)1 << 24, 4 * g->m / BFS_CHUNK + 64);
  S->items_cap = (int32_t)cap;
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t o_head = 0, o_recip = up(1024), o_dist = o_recip + (g->directed ? up(4 * n) : 0);
  const size_t o_qa = o_dist + up(4 * n), o_qb = o_qa + up(4 * n), o_distb = o_qb + up(4 * n);
  const size_t o_items = o_distb + (g->directed ? up(4 * n) : 0);
  S->base = nullptr;
  S->tree.levels = 0;
  size_t total = up(o_items + sizeof(BfsItem) * (size_t)cap), o_lv[TREE_LEVELS];
  if (csr_bytes(g) > l2_bytes(g->device)) {
    for (int64_t c = (g->m + (1ll << TREE_SHIFT) - 1) >> TREE_SHIFT; S->tree.levels < TREE_LEVELS; c = (c + 7) / 8) {
      o_lv[S->tree.levels++] = total;
      total += up(4 * (size_t)c);
      if (c <= 1) break;
    }
  }
  if (S->tree.levels && pool_alloc(&S->base, total) != KADABRA_OK) {  // no room: binary searches
    cudaGetLastError();
    S->tree.levels = 0;
    total = o_lv[0];
    S->base = nullptr;
  }
  if (!S->base) KTRY(pool_alloc(&S->base, total));
  unsigned char* b = static_cast<unsigned char*>(S->base);
  LoadHead* head = reinterpret_cast<LoadHead*>(b + o_head);  // device addresses
  S->err = &head->err;
  S->lt_gt = head->lt_gt;
  S->best = &head->best;
  S->floor_deg = &head->floor_deg;
  S->cnt = reinterpret_cast<int32_t*>(b + o_head + 512);
  S->fp = head->fp;
  S->recip = g->directed ? reinterpret_cast<uint32_t*>(b + o_recip) : nullptr;
  S->core = reinterpret_cast<VdCore*>(b + o_head + 768);
  S->dist = reinterpret_cast<int32_t*>(b + o_dist);
  S->dist_b = g->directed ? reinterpret_cast<int32_t*>(b + o_distb) : nullptr;
  S->qa = reinterpret_cast<int32_t*>(b + o_qa);
  S->qb = reinterpret_cast<int32_t*>(b + o_qb);
  S->items = reinterpret_cast<BfsItem*>(b + o_items);
  for (int k = 0; k < S->tree.levels; ++k) S->tree.lv[k] = reinterpret_cast<int32_t*>(b + o_lv[k]);
  const int32_t* searched = g->directed ? g->rci : g->ci;
  S->tree.groups = (reinterpret_cast<uintptr_t>(searched) & 31) ? 0 : (int32_t)(g->m / 8);
  KCK(cudaMemset(S->base, 0, 64));
  if (S->recip) KCK(cudaMemset(S->recip, 0, 4 * n));
  return KADABRA_OK;
}

// Queues a BFS from the root along (tr, tc) into dist (bottom-up levels look
// in (br, bc)).  Levels are queued BFS_BATCH at a time and their sizes read
// back once per batch; levels past the end find an empty frontier and do
// nothing.
kadabra_status vd_bfs(kadabra_graph* g, const LoadScratch& S, const int32_t* tr, const int32_t* tc,
                      const int32_t* br, const int32_t* bc, int32_t* dist) {
  const int32_t n = g->n;
  constexpr int BFS_BATCH = 4, SLOTS = 8, SLOT = 4;  // slot: next frontier's nodes, long-row items, its arcs
  k_bfs_root<<<1, 1>>>(S.best, dist, S.qa);  // the root stays on the device
  KCK(cudaGetLastError());
  bool done = false;
  for (int32_t l0 = 0; !done && l0 <= n; l0 += BFS_BATCH) {
    for (int k = 0; k < BFS_BATCH; ++k)
      KCK(cudaMemsetAsync(S.cnt + SLOT * ((l0 + k) % SLOTS), 0, SLOT * sizeof(int32_t)));
    for (int k = 0; k < BFS_BATCH; ++k) {
      const int32_t l = l0 + k;
      int32_t* in_q = (l & 1) ? S.qb : S.qa;
      int32_t* out_q = (l & 1) ? S.qa : S.qb;
      int32_t* c = S.cnt + SLOT * (l % SLOTS);
      const int32_t* prev = l == 0 ? nullptr : S.cnt + SLOT * ((l + SLOTS - 1) % SLOTS);
      k_bfs_level<<<8 * g->num_sms, 256>>>(tr, tc, br, bc, in_q, prev, out_q, c, dist, l, S.items, c + 1,
                                           S.items_cap, n, g->m);
      k_bfs_items<<<8 * g->num_sms, 256>>>(tr, tc, bc, S.items, c + 1, S.items_cap, out_q, c, dist, l);
    }
    int32_t h[SLOT * SLOTS];
    if (cudaMemcpy(h, S.cnt, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(KADABRA_ERR_CUDA, std::string("vd bfs: ") + cudaGetErrorString(cudaGetLastError()));
    for (int k = 0; k < BFS_BATCH; ++k)
      if (h[SLOT * ((l0 + k) % SLOTS)] == 0) {
        done = true;
        break;
      }
  }
  return KADABRA_OK;
}

// The condensation's heaviest path when the root's component is not the
// whole graph (kernels k_vd_*): labels by trimming and colour propagation,
// then a level-by-level pass in topological order.
kadabra_status vd_condensation(kadabra_graph* g, LoadTrace& tr, const LoadScratch& S, const int32_t* db,
                               long long root_w, int64_t* vd_out) {
  const int32_t n = g->n;
  const int64_t m = g->m;
  const int32_t* rrp = g->directed ? g->rrp : g->rp;
  const int32_t* rci = g->directed ? g->rci : g->ci;
  const int bn = std::max(1, std::min(16 * g->num_sms, (n + 255) / 256));
  const int ba = (int)std::max<int64_t>(1, std::min<int64_t>(16 * g->num_sms, (m + 255) / 256));
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t N4 = up(4 * (size_t)n), N8 = up(8 * (size_t)n);
  void* base = nullptr;
  KTRY(pool_alloc(&base, 256 + 6 * N4 + N8));
  struct Free {
    void* p;
    ~Free() { pool_free(p); }
  } guard{base};
  unsigned char* b = static_cast<unsigned char*>(base);
  int32_t* flag = reinterpret_cast<int32_t*>(b);              // [0] a change, [1] an unlabelled node, [2] a long row
  int32_t* slots = reinterpret_cast<int32_t*>(b + 64);        // 8 level slots of 2
  long long* vd = reinterpret_cast<long long*>(b + 128);
  int32_t* lab = reinterpret_cast<int32_t*>(b + 256);
  int32_t* col = reinterpret_cast<int32_t*>(b + 256 + N4);
  int32_t* reach = reinterpret_cast<int32_t*>(b + 256 + 2 * N4);
  int32_t* sz = reinterpret_cast<int32_t*>(b + 256 + 3 * N4);
  int32_t* cnt = reinterpret_cast<int32_t*>(b + 256 + 4 * N4);
  int32_t* rdy = reinterpret_cast<int32_t*>(b + 256 + 5 * N4);
  long long* best = reinterpret_cast<long long*>(b + 256 + 6 * N4);
  KCK(cudaMemsetAsync(flag, 0, 3 * sizeof(int32_t)));
  k_vd_label_init<<<bn, 256>>>(S.dist, db, n, S.best, lab, g->rp, rrp, flag + 2);
  KCK(cudaGetLastError());
  // repeats a kernel (4 queued rounds per read-back) until a round changes
  // nothing: at most n rounds change something, then one read-back more
  auto until_stable = [&](auto&& round) -> kadabra_status {
    for (int64_t it = 0; it < (int64_t)n + 4; it += 4) {
      KCK(cudaMemsetAsync(flag, 0, sizeof(int32_t)));
      for (int k = 0; k < 4; ++k) round();
      int32_t h = 0;
      if (cudaMemcpy(&h, flag, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(KADABRA_ERR_CUDA, std::string("vd bound: ") + cudaGetErrorString(cudaGetLastError()));
      if (!h) return KADABRA_OK;
    }
    return fail(KADABRA_ERR_INTERNAL, "vd bound: no fixed point");
  };
  for (int64_t outer = 0;; ++outer) {
    if (outer > (int64_t)n) return fail(KADABRA_ERR_INTERNAL, "vd bound: components not all labelled");
    KTRY(until_stable([&] { k_vd_trim<<<bn, 256>>>(g->rp, g->ci, rrp, rci, n, lab, flag); }));
    KCK(cudaMemsetAsync(flag + 1, 0, sizeof(int32_t)));
    k_vd_color_init<<<bn, 256>>>(lab, n, col, reach, flag + 1);
    int32_t left = 0;
    if (cudaMemcpy(&left, flag + 1, sizeof(left), cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(KADABRA_ERR_CUDA, "vd bound");
    if (!left) break;
    KTRY(until_stable([&] { k_vd_color<<<bn, 256>>>(rrp, rci, n, lab, col, flag); }));
    k_vd_reach_roots<<<bn, 256>>>(lab, col, n, reach);
    KTRY(until_stable([&] { k_vd_reach<<<bn, 256>>>(g->rp, g->ci, n, lab, col, reach, flag); }));
    k_vd_assign<<<bn, 256>>>(col, reach, n, lab);
  }
  tr.mark("vd components");
  KCK(cudaMemsetAsync(sz, 0, 2 * N4));  // sz, cnt
  KCK(cudaMemsetAsync(rdy, 0xFF, N4));
  KCK(cudaMemsetAsync(best, 0, N8));
  KCK(cudaMemsetAsync(b + 64, 0, 192));  // slots, vd
  k_vd_sizes<<<bn, 256>>>(lab, n, S.best, S.core, sz);
  k_vd_indeg<<<ba, 256>>>(g->rp, g->ci, rrp, rci, n, m, lab, S.best, flag + 2, cnt);
  unsigned long long key = 0;
  if (cudaMemcpy(&key, S.best, sizeof(key), cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail(KADABRA_ERR_CUDA, "vd bound");
  VdKahn K{g->rp, g->ci, rrp, rci, lab, sz, cnt, best, rdy, n, (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull)),
           root_w, vd, flag + 2};
  constexpr int SLOTS = 8, BATCH = 4;
  k_vd_kahn_init<<<bn, 256>>>(K, S.qa, slots + 2 * (SLOTS - 1));  // the slot level 0 reads
  KCK(cudaGetLastError());
  bool done = false;
  for (int32_t l0 = 0; !done; l0 += BATCH) {
    if (l0 > n) return fail(KADABRA_ERR_INTERNAL, "vd bound: condensation levels");
    for (int k = 0; k < BATCH; ++k) KCK(cudaMemsetAsync(slots + 2 * ((l0 + k) % SLOTS), 0, 2 * sizeof(int32_t)));
    for (int k = 0; k < BATCH; ++k) {
      const int32_t l = l0 + k;
      k_vd_kahn_level<<<8 * g->num_sms, 256>>>(K, m, (l & 1) ? S.qb : S.qa, slots + 2 * ((l + SLOTS - 1) % SLOTS),
                                               (l & 1) ? S.qa : S.qb, slots + 2 * (l % SLOTS), l);
    }
    int32_t h[2 * SLOTS];
    if (cudaMemcpy(h, slots, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(KADABRA_ERR_CUDA, std::string("vd bound: ") + cudaGetErrorString(cudaGetLastError()));
    for (int k = 0; k < BATCH; ++k) {
      const int32_t* sl = h + 2 * ((l0 + k) % SLOTS);
      if (sl[0] == 0 && sl[1] == 0) {
        done = true;
        break;
      }
    }
  }
  long long hv = 0;
  if (cudaMemcpy(&hv, vd, sizeof(hv), cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail(KADABRA_ERR_CUDA, "vd bound");
  *vd_out = hv;
  tr.mark("vd condensation");
  return KADABRA_OK;
}

// VD bound (omega of Alg. 1; Sec. 2): BFS from the root r forward (and,
// for a directed graph, backward) gives the root's component C_r and its
// weight e_out + e_in + 1 (2 ecc(r) + 1 undirected).  When C_r is the whole
// graph that is the bound; otherwise the condensation decides it.
kadabra_status compute_vd(kadabra_graph* g, LoadTrace& tr, const LoadScratch& S) {
  const int32_t n = g->n;
  const int32_t* rrp = g->directed ? g->rrp : g->rp;
  const int32_t* rci = g->directed ? g->rci : g->ci;
  const int blocks = std::max(1, std::min(4 * g->num_sms, (n + 255) / 256));
  KCK(cudaMemsetAsync(S.dist, 0xFF, sizeof(int32_t) * (size_t)n));
  if (g->directed) KCK(cudaMemsetAsync(S.dist_b, 0xFF, sizeof(int32_t) * (size_t)n));
  KCK(cudaMemsetAsync(S.core, 0, sizeof(VdCore)));
  k_und_degree_key<<<blocks, 256>>>(g->rp, rrp, S.recip, n, g->directed, S.best, S.core->idle);
  KCK(cudaGetLastError());
  tr.mark("vd root");
  KTRY(vd_bfs(g, S, g->rp, g->ci, rrp, rci, S.dist));
  const int32_t* db = S.dist;
  if (g->directed) {
    KTRY(vd_bfs(g, S, rrp, rci, g->rp, g->ci, S.dist_b));
    db = S.dist_b;
  }
  k_vd_core<<<blocks, 256>>>(S.dist, db, n, S.core);
  VdCore core;
  if (cudaMemcpy(&core, S.core, sizeof(core), cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail(KADABRA_ERR_CUDA, std::string("vd: ") + cudaGetErrorString(cudaGetLastError()));
  tr.mark("vd bfs");
  g->idle = 1.0 - (1.0 - (double)core.idle[0] / n) * (1.0 - (double)core.idle[1] / n);
  const long long root_w = (long long)core.e_out + core.e_in + 1;
  if (core.size == (unsigned long long)n) {
    g->vd = root_w;
    return KADABRA_OK;
  }
  int64_t vd = 0;
  KTRY(vd_condensation(g, tr, S, db, root_w, &vd));
  g->vd = vd;
  return KADABRA_OK;
}

// Validates a device CSR (offsets, ids, order, self-loops, mirror/symmetry),
// takes its fingerprint and computes the VD bound.
kadabra_status finish_load(kadabra_graph* g) {
  LoadTrace tr;
  LoadScratch S;
  KTRY(load_scratch(g, &S));
  tr.mark("scratch");
  const int32_t n = g->n;
  const int64_t m = g->m;
  const int bn = std::max(1, std::min(16 * g->num_sms, (n + 255) / 256));
  const int ba = (int)std::max<int64_t>(1, std::min<int64_t>(16 * g->num_sms, (m + 255) / 256));
  const int32_t* rrp = g->directed ? g->rrp : g->rp;
  const int32_t* rci = g->directed ? g->rci : g->ci;
  unsigned h = 0;
  kadabra_status st = KADABRA_OK;
  do {
    // every check is queued at once; each looks on the device whether the ones
    // it relies on have passed, and the host reads all results back together
    k_validate_offsets<<<bn, 256>>>(g->rp, n, m, S.err);
    if (g->directed) k_validate_offsets<<<bn, 256>>>(g->rrp, n, m, S.err);
    k_validate_arcs<<<ba, 256>>>(g->rp, g->ci, n, m, S.err);
    if (g->directed) k_validate_arcs<<<ba, 256>>>(g->rrp, g->rci, n, m, S.err);
    tr.mark("validate rows");
    if (S.tree.levels) k_row_tree<<<ba, 256>>>(rci, m, S.tree);
    if (g->directed) k_floor_degree<<<bn, 256>>>(g->rp, rrp, n, S.floor_deg);
    k_validate_mirror<<<ba, 256>>>(g->rp, g->ci, rrp, rci, n, m, g->directed ? 0 : 1, S.err, S.lt_gt, S.recip,
                                   S.floor_deg, S.tree);
    k_fingerprint<<<1, 64>>>(g->rp, g->ci, n, m, S.fp);
    LoadHead head;
    if (cudaMemcpy(&head, S.base, sizeof(head), cudaMemcpyDeviceToHost) != cudaSuccess) {
      st = fail(KADABRA_ERR_CUDA, std::string("CSR check: ") + cudaGetErrorString(cudaGetLastError()));
      break;
    }
    h = head.err;
    if (!g->directed && !h && head.lt_gt[0] != head.lt_gt[1]) h |= 16u;
    tr.mark("validate mirror");
    if (h) break;
    // fingerprint: FNV-1a over the shape and 64 sampled entries
    const int32_t* fp = head.fp;
    uint64_t x = 1469598103934665603ull;
    auto mix = [&](uint64_t v) {
      for (int b = 0; b < 8; ++b) {
        x ^= (v >> (8 * b)) & 0xFF;
        x *= 1099511628211ull;
      }
    };
    mix((uint64_t)n);
    mix((uint64_t)m);
    mix((uint64_t)g->directed);
    for (int i = 0; i < 64; ++i) mix((uint64_t)(uint32_t)fp[i]);
    g->fingerprint = x;
    st = compute_vd(g, tr, S);
  } while (0);
  pool_free(S.base);
  tr.mark("scratch free");
  if (st != KADABRA_OK) return st;
  if (h) {
    std::string why;
    if (h & 1) why += " bad row offsets;";
    if (h & 2) why += " node id out of range;";
    if (h & 4) why += " row not strictly increasing;";
    if (h & 8) why += " self-loop;";
    if (h & 16) why += (g->directed ? " reverse CSR does not mirror the forward CSR;" : " adjacency not symmetric;");
    return fail(KADABRA_ERR_CSR, "invalid CSR:" + why);
  }
  g->csr_beyond_l2 = csr_bytes(g) > l2_bytes(g->device);
  return KADABRA_OK;
}

// Idle workspaces of freed graph objects, at most one per device.  The next
// graph object on that device takes it if it fits (its tables are sized for
// up to max_n nodes and max_m arcs), which spares the allocation and the
// table initialisation (about a millisecond for a 10^6-node graph) and the
// matching frees.  kadabra_release_cached frees them.
std::mutex g_ws_pool_mu;
std::vector<Workspace*> g_ws_pool;

Workspace* ws_acquire(int device, int num_sms, int32_t n, int64_t m) {
  Workspace* w = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_ws_pool_mu);
    for (size_t i = 0; i < g_ws_pool.size(); ++i)
      if (g_ws_pool[i]->device == device && g_ws_pool[i]->max_n >= n && g_ws_pool[i]->max_m >= m) {
        w = g_ws_pool[i];
        g_ws_pool.erase(g_ws_pool.begin() + (std::ptrdiff_t)i);
        break;
      }
  }
  if (w) {
    // a stale error of the previous owner must not reach the new one
    if (w->ready && cudaMemset(w->status, 0, sizeof(int32_t)) != cudaSuccess) {
      delete w;
      w = nullptr;
    } else {
      return w;
    }
  }
  w = new Workspace;
  w->device = device;
  w->num_sms = num_sms;
  w->max_n = n;
  w->max_m = m;
  return w;
}

// Takes back the workspace of a freed graph object (no work in flight on it).
void ws_release(Workspace* w) {
  Workspace* drop = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_ws_pool_mu);
    bool placed = false;
    for (Workspace*& p : g_ws_pool)
      if (p->device == w->device) {  // keep the one that fits more graphs
        if (w->max_n >= p->max_n && w->max_m >= p->max_m) {
          drop = p;
          p = w;
        } else {
          drop = w;
        }
        placed = true;
        break;
      }
    if (!placed) g_ws_pool.push_back(w);
  }
  delete drop;
}

kadabra_status new_graph(int32_t n, int64_t m, int directed, kadabra_graph** out, kadabra_graph** g_out) {
  if (!out) return fail(KADABRA_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (n < 2 || n > (1 << 24)) return fail(KADABRA_ERR_ARG, "n must be in [2, 2^24]");
  if (m < 0 || m >= ((int64_t)1 << 31)) return fail(KADABRA_ERR_ARG, "m must be in [0, 2^31)");
  kadabra_graph* g = new kadabra_graph;
  g->n = n;
  g->m = m;
  g->directed = directed ? 1 : 0;
  if (cudaGetDevice(&g->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&g->num_sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess) {
    delete g;
    return fail(KADABRA_ERR_CUDA, "no CUDA device");
  }
  g->ws = ws_acquire(g->device, g->num_sms, n, m);
  g->owns_ws = true;
  *g_out = g;
  return KADABRA_OK;
}

}  // namespace

namespace {




// ---------------------------------------------------------------- sampler autotuner
// Picks, per graph, the shared-memory sampler setup that samples it fastest,
// out of two independent choices: the tier-S table (2^FAST_HLOG slots at
// KD_MIN_BLOCKS CTAs per SM, or the compact layout with one more CTA per SM)
// and whether tier W (one warp per sample) runs first.  Small searches gain
// from more samples in flight, large ones lose to more escalations.  Every
// setup gives identical results, so the choice only changes speed.  It times
// a probe batch of samples in RNG domain 3 (results discarded) with each
// allowed setup, once per graph; cfg.ctas_per_sm and cfg.warp_tier fix either
// choice.  The probe batch is the run's own batch size K, capped at
// TUNE_PROBE: small batches are bound by the slowest sample, large ones by
// throughput, and the two can favour different setups.  A setup other than
// the default is taken only if it is at least 2% faster.  A probe of 4096
// samples saw the compact layout's 3.5 % gain on the Chung-Lu graph's
// 65,536-sample batches as a loss (tails of a few samples per CTA), and one
// of 16,384 picked either setup from run to run.
constexpr uint64_t TUNE_PROBE = 65536;
// process-wide: graphs with the same fingerprint, device and launch flags (a
// graph, or a batch, loaded again) reuse the probe's choice; a collision could
// only cost speed
std::mutex g_tune_mu;
std::unordered_map<uint64_t, int> g_tune_cache;

// flags, idle: the launches' flags and share of samples that end at a root
// without arcs; shared: the launches are a batch's, g its largest graph.
kadabra_status tier_variant(kadabra_graph* g, Workspace* w, cudaStream_t st, int32_t req_ctas, int32_t req_warp,
                            uint64_t batch, uint32_t flags, double idle, bool shared, int* variant) {
  const uint64_t probe = std::max<uint64_t>(1, std::min<uint64_t>(batch, TUNE_PROBE));
  const int size_class = probe >= TUNE_PROBE ? 0 : 1 + ceil_log2(probe);  // <= 17
  const int per_default = w->grid_fast / w->num_sms, per_compact = w->grid_compact / w->num_sms;
  unsigned s_ok, w_ok;  // allowed values of variant bit 0 and bit 1
  if (req_ctas == 0)
    s_ok = 3;
  else if (req_ctas == per_default)
    s_ok = 1;
  else if (req_ctas == per_compact)
    s_ok = 2;
  else
    return fail(KADABRA_ERR_ARG, "ctas_per_sm must be 0 (autotune), " + std::to_string(per_default) + " or " +
                                     std::to_string(per_compact));
  if (req_warp == 0)
    w_ok = 3;
  else if (req_warp == 1)
    w_ok = 2;
  else if (req_warp == -1)
    w_ok = 1;
  else
    return fail(KADABRA_ERR_ARG, "warp_tier must be 0 (autotune), 1 (on) or -1 (off)");
  unsigned allowed = 0;  // bit v: variant v may run
  for (int v = 0; v < 4; ++v)
    if ((s_ok >> (v & 1) & 1) && (w_ok >> (v >> 1) & 1)) allowed |= 1u << v;
  if ((allowed & (allowed - 1)) == 0) {  // one setup: nothing to tune
    *variant = __builtin_ctz(allowed);
    return KADABRA_OK;
  }
  kadabra_graph::TuneTable& table = shared ? g->shared_choice : g->tier_choice;
  if (table.flags != flags) table = kadabra_graph::TuneTable();
  table.flags = flags;
  int& choice = table.v[size_class][allowed];
  if (choice >= 0) {
    *variant = choice;
    return KADABRA_OK;
  }
  // what else the probes' launches depend on
  const bool screen = probe >= SCREEN_SAMPLES && idle >= SCREEN_MIN;
  const uint64_t how = (flags & 127u) | ((uint64_t)(flags >> 29) << 7) | ((uint64_t)shared << 10) | ((uint64_t)screen << 11);
  static_assert(KADABRA_FLAG_COMPACT_TABLES == 64 && FLAG_TINY_AUTO == 1u << 29, "the flags' bits in the key");
  const uint64_t key = g->fingerprint ^ ((uint64_t)g->device << 56) ^ (how << 44) ^ ((uint64_t)allowed << 40) ^
                       ((uint64_t)size_class << 32);
  const bool cached = g->fingerprint != 0;
  if (cached) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      choice = *variant = it->second;
      return KADABRA_OK;
    }
  }
  KTRY(ensure_ws(w, probe, 1));
  SampleParams P = ws_params(w, flags);
  P.total_work = probe;
  choose_screen(P, probe, idle * (double)probe);
  std::memset(&P.job0, 0, sizeof(Job));
  P.job0.g = graph_dev(g);
  P.job0.seed = 0x5EEDu;
  P.job0.domain = 3;
  P.job0.count = probe;  // counts and totals null: nothing is recorded
  cudaEvent_t e0, e1;
  KCK(cudaEventCreate(&e0));
  KCK(cudaEventCreate(&e1));
  float best[4] = {1e30f, 1e30f, 1e30f, 1e30f};
  kadabra_status stt = KADABRA_OK;
  // best of several rounds over the setups: two for large probes, up to
  // eight for small ones, whose times (tens of microseconds) vary more
  const int reps = (int)std::min<uint64_t>(8, std::max<uint64_t>(2, 16384 / probe));
  for (int rep = 0; rep < reps && stt == KADABRA_OK; ++rep)
    for (int v = 0; v < 4 && stt == KADABRA_OK; ++v) {
      if (!(allowed >> v & 1)) continue;
      cudaEventRecord(e0, st);
      stt = launch_sampler(w, P, st, v);
      cudaEventRecord(e1, st);
      if (cudaEventSynchronize(e1) != cudaSuccess) stt = fail(KADABRA_ERR_CUDA, "autotune probe");
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      best[v] = std::min(best[v], ms);
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  KTRY(stt);
  int32_t h = 0;  // a probe sample's error (the run reports its own) only ends the tuning
  KCK(cudaMemcpyAsync(&h, w->status, sizeof(h), cudaMemcpyDeviceToHost, st));
  KCK(cudaStreamSynchronize(st));
  const int first = __builtin_ctz(allowed);  // the default among the allowed setups
  int pick = first;
  if (h != 0) {
    KCK(cudaMemsetAsync(w->status, 0, sizeof(int32_t), st));
    KCK(cudaStreamSynchronize(st));
  } else {
    int fastest = first;
    for (int v = 0; v < 4; ++v)
      if ((allowed >> v & 1) && best[v] < best[fastest]) fastest = v;
    if (best[fastest] < 0.98f * best[first]) pick = fastest;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    if (cached) g_tune_cache[key] = pick;
  }
  choice = *variant = pick;
  return KADABRA_OK;
}

// The setup an autotuned run on g chose for batches of `batch` samples (every
// setup allowed), or the default if no run has tuned that size class; no probe.
int tuned_variant(const kadabra_graph* g, uint64_t batch) {
  const uint64_t probe = std::max<uint64_t>(1, std::min<uint64_t>(batch, TUNE_PROBE));
  const int size_class = probe >= TUNE_PROBE ? 0 : 1 + ceil_log2(probe);
  const int v = g->tier_choice.flags == launch_flags(g) ? g->tier_choice.v[size_class][15] : -1;
  return v >= 0 ? v : 0;
}

int variant_ctas_per_sm(const Workspace* w, int variant) {
  return ((variant & 1) ? w->grid_compact : w->grid_fast) / w->num_sms;
}

// ---------------------------------------------------------------- device-driven main loop
constexpr uint64_t LOOP_GRAPH_MIN_ROUNDS = 4;  // fewer possible rounds: host rounds cost as little

// The main loop of one all-nodes run as a CUDA graph: a while node whose body
// is {the sampler launches, k_loop_check}; the test's last block sets the
// while condition and the next round's range (k_loop_begin, before the
// graph, sets the first).  Built once per graph object and
// rebuilt only when the launch parameters it captured change (workspace
// buffers that grew, another table tier flag).
kadabra_status loop_graph_ready(LoopCache& L, Workspace* w, const SampleParams& P, int check_blocks, int G,
                                int variant) {
  std::vector<unsigned char> sig(sizeof(SampleParams) + 7 * sizeof(int64_t));
  std::memcpy(sig.data(), &P, sizeof(SampleParams));
  const int64_t more[7] = {w->grid_fast, w->grid_big, w->grid_gm, check_blocks, variant, G,
                           (int64_t)(uintptr_t)L.dev};
  std::memcpy(sig.data() + sizeof(SampleParams), more, sizeof(more));
  if (L.exec && sig == L.sig) return KADABRA_OK;
  L.drop_graph();
  if (!L.cap) KCK(cudaStreamCreateWithFlags(&L.cap, cudaStreamNonBlocking));
  LoopState* d_state = static_cast<LoopState*>(L.dev);
  KCK(cudaGraphCreate(&L.graph, 0));
  cudaGraphConditionalHandle h;
  KCK(cudaGraphConditionalHandleCreate(&h, L.graph, 1u, cudaGraphCondAssignDefault));
  cudaGraphNodeParams cp = {cudaGraphNodeTypeConditional};  // the rest zero
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  KCK(cudaGraphAddNode(&node, L.graph, nullptr, nullptr, 0, &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  KCK(cudaStreamBeginCaptureToGraph(L.cap, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  kadabra_status st = launch_sampler_kernels(w, P, L.cap, variant);
  k_loop_check<<<dim3(check_blocks, G), 256, 0, L.cap>>>(d_state, w->ctr, w->status, h);
  cudaGraph_t captured = nullptr;
  const cudaError_t ec = cudaStreamEndCapture(L.cap, &captured);
  if (st != KADABRA_OK) return st;
  KCK(ec);
  KCK(cudaGetLastError());
  KCK(cudaGraphInstantiate(&L.exec, L.graph, 0));
  L.sig = sig;
  return KADABRA_OK;
}

// One graph of a device-driven main loop: its state on entry (tau a
// multiple of K, or done), and on return its final tau, the number of tests
// the loop ran, whether one held, and the last test's result.
struct LoopRun {
  kadabra_graph* g;
  uint64_t seed, tau, cap, K, checks;
  double omega, lambda;
  bool done;
  int stopped;
  CheckOut co;
};

// Runs the main loops of several all-nodes runs on the device until each
// graph's test holds or it reaches ceil(omega).
kadabra_status run_loop_graph(LoopCache& L, Workspace* w, cudaStream_t st, std::vector<LoopRun>& R, uint32_t flags,
                              int variant) {
  const int G = (int)R.size();
  const size_t bytes = sizeof(LoopState) + (size_t)G * (sizeof(LoopGraph) + sizeof(Job) + sizeof(CheckTabJob));
  if (L.dev_bytes < bytes) {
    KCK(cudaStreamSynchronize(st));
    L.drop_graph();
    if (L.dev) cudaFree(L.dev);
    L.dev = nullptr;
    L.dev_bytes = 0;
    KCK(cudaMalloc(&L.dev, bytes));
    L.dev_bytes = bytes;
  }
  LoopState* d_state = static_cast<LoopState*>(L.dev);
  LoopGraph* d_lg = reinterpret_cast<LoopGraph*>(d_state + 1);
  Job* d_job = reinterpret_cast<Job*>(d_lg + G);
  SampleParams P = ws_params(w, flags);
  P.jobs = d_job;
  P.njobs = G;
  P.total_dev = &d_state->total_work;
  // The launches read total_dev; a round's samples only decide whether k_screen
  // runs.  No more than that decision goes into the parameters, so that a run
  // with another K (another lambda, if the library chooses K) finds the CUDA
  // graph as it is: building it anew took 65 to 70 us of a 1.0 ms run on 2,000
  // nodes.
  uint64_t round = 0;
  double idle = 0.0;
  for (const LoopRun& r : R) {
    if (r.done) continue;
    round += r.K;
    idle += r.g->idle * (double)r.K;
  }
  choose_screen(P, round, idle);
  int64_t max_n = 1;
  for (const LoopRun& r : R) max_n = std::max<int64_t>(max_n, r.g->n);
  const int64_t want = (4 * (int64_t)w->num_sms + G - 1) / G;
  const int check_blocks = (int)std::max<int64_t>(1, std::min<int64_t>(want, (max_n + 255) / 256));
  KTRY(loop_graph_ready(L, w, P, check_blocks, G, variant));
  std::vector<unsigned char> host(bytes, 0);
  LoopState* hs = reinterpret_cast<LoopState*>(host.data());
  LoopGraph* hl = reinterpret_cast<LoopGraph*>(hs + 1);
  Job* hj = reinterpret_cast<Job*>(hl + G);
  CheckTabJob* hc = reinterpret_cast<CheckTabJob*>(hj + G);
  hs->G = G;
  for (int i = 0; i < G; ++i) {
    const LoopRun& r = R[i];
    hl[i].tau = r.tau;
    hl[i].cap = r.cap;
    hl[i].K = r.K;
    hl[i].n = r.g->n;
    hl[i].done = r.done ? 1u : 0u;
    hj[i].g = graph_dev(r.g);
    hj[i].seed = r.seed;
    hj[i].domain = 0;
    hj[i].counts = r.g->counts;
    hj[i].totals = r.g->totals;
    hc[i].counts = r.g->counts;
    hc[i].count0 = r.g->count0;
    hc[i].fail_fast = 1;  // the loop reads only the decision; a test that holds finds no failure
    hc[i].lnT = r.g->lntab;
    hc[i].n = r.g->n;
    hc[i].omega = r.omega;
    hc[i].lambda = r.lambda;
    hc[i].out = &d_lg[i].co;
  }
  KCK(cudaMemcpyAsync(L.dev, host.data(), bytes, cudaMemcpyHostToDevice, st));
  k_loop_begin<<<1, 1, 0, st>>>(d_state, w->ctr);
  KCK(cudaGetLastError());
  KCK(cudaGraphLaunch(L.exec, st));
  KCK(cudaMemcpyAsync(hl, d_lg, sizeof(LoopGraph) * (size_t)G, cudaMemcpyDeviceToHost, st));
  KTRY(read_status(w, st));  // synchronises the stream, so hl (host memory that outlives the call) is filled
  for (int i = 0; i < G; ++i) {
    R[i].tau = hl[i].tau;
    R[i].checks = hl[i].checks;
    R[i].stopped = (int)hl[i].stopped;
    R[i].co = hl[i].co;
  }
  return KADABRA_OK;
}

// ---------------------------------------------------------------- Alg. 1 runner
constexpr int NZ_BLK = 128;  // compaction blocks per graph

// KADABRA on G graphs at once (kadabra_run is the case G = 1): warm-up of
// every graph in one sampler launch, computeDelta per graph on the host from
// its compacted warm-up counts, then rounds of one sampler launch over every
// unfinished graph's next batch and one stop-test launch over all of them.
kadabra_status run_graphs(Workspace* w, kadabra_graph* const* gs, int G, const double* lambda, const double* delta,
                          const uint64_t* seed, const int64_t* vd_override, const kadabra_config& cfg,
                          kadabra_result* out) {
  cudaStream_t st = as_stream(cfg.stream);
  LoadTrace tr(G == 1 ? "run" : "batch run");
  struct State {
    kadabra_graph* g;
    uint64_t cap, alpha, K, tau;
    uint64_t pre;  // main-loop samples already taken with the warm-up, not yet in tau
    bool done;
    bool have_max;  // max f, max g known: the test that held evaluated every node
  };
  std::vector<State> S(G);
  uint64_t sum_alpha = 0, sum_k = 0;
  for (int i = 0; i < G; ++i) {
    kadabra_result& r = out[i];
    State& s = S[i];
    s.g = gs[i];
    r.vd = (vd_override && vd_override[i] > 0) ? vd_override[i] : s.g->vd;
    r.omega = omega_host(lambda[i], delta[i], r.vd);
    const double cap_d = std::ceil(r.omega);
    if (!(cap_d >= 1.0 && cap_d < 1e15)) return fail(KADABRA_ERR_ARG, "omega out of range");
    s.cap = r.omega_cap = (uint64_t)cap_d;
    s.alpha = r.alpha = std::max<uint64_t>(1, (uint64_t)std::floor(r.omega / 100.0));
    s.K = r.check_interval = cfg.check_interval ? cfg.check_interval : auto_check_interval(r.omega);
    s.tau = 0;
    s.pre = 0;
    s.done = false;
    s.have_max = false;
    sum_alpha += s.alpha;
    sum_k += std::min(s.K, s.cap);
  }
  KTRY(ensure_ws(w, sum_alpha + sum_k, 2 * G));
  for (State& s : S) {
    KTRY(ensure_run_buffers(s.g));
    if (s.g->lntab_cap < s.alpha + 1) {
      KCK(cudaStreamSynchronize(st));
      gdev_free(s.g->allocs, s.g->lntab);
      void* p;
      KTRY(gdev_alloc(s.g->allocs, &p, sizeof(double) * (s.alpha + 1)));
      s.g->lntab = (double*)p;
      s.g->lntab_cap = s.alpha + 1;
    }
  }
  if (w->checks_cap < G) {
    KCK(cudaDeviceSynchronize());
    dev_free(w->allocs, w->d_checks);
    void* p;
    KTRY(dev_alloc(w->allocs, &p, (sizeof(CheckTabJob) + sizeof(CheckOut)) * (size_t)G));
    w->d_checks = p;
    w->checks_cap = G;
  }
  if (w->nz_cap < G) {
    KCK(cudaDeviceSynchronize());
    dev_free(w->allocs, w->d_nz);
    void* p;
    KTRY(dev_alloc(w->allocs, &p, (sizeof(NzJob) + sizeof(unsigned) * (NZ_BLK + 1)) * (size_t)G));
    w->d_nz = p;
    w->nz_cap = G;
  }
  CheckTabJob* d_cj = static_cast<CheckTabJob*>(w->d_checks);
  CheckOut* d_co = reinterpret_cast<CheckOut*>(d_cj + G);
  NzJob* d_nzj = static_cast<NzJob*>(w->d_nz);
  unsigned* d_blk = reinterpret_cast<unsigned*>(d_nzj + G);
  unsigned* d_nzt = d_blk + (size_t)NZ_BLK * G;
#define RCK(call)                                                                         \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) return fail(KADABRA_ERR_CUDA, cudaGetErrorString(e_));         \
  } while (0)
  // one graph: its flags.  Several share the launch: the small layout if every
  // graph allows it, and what SHARED_LAUNCH_FLAGS has of any graph.
  uint32_t fl = launch_flags(gs[0]);
  if (G > 1) {
    fl = FLAG_TINY_AUTO;
    for (int i = 0; i < G; ++i) fl &= launch_flags(gs[i]);
    for (int i = 0; i < G; ++i) fl |= launch_flags(gs[i]) & SHARED_LAUNCH_FLAGS;
  }
  // The tier-S setup of the launches: autotuned on the graph (one-graph
  // runs), or with the shared flags on the batch's largest graph, whose
  // samples take most of each shared launch (it changes no result).
  int variant = 0;
  {
    int big = 0;
    double idle_k = 0.0;
    for (int i = 0; i < G; ++i) {
      if (gs[i]->m > gs[big]->m) big = i;
      idle_k += gs[i]->idle * (double)std::min(S[i].K, S[i].cap);
    }
    KTRY(tier_variant(gs[big], w, st, cfg.ctas_per_sm, cfg.warp_tier, std::min(S[big].K, S[big].cap), fl,
                      idle_k / (double)sum_k, G > 1, &variant));
    for (int i = 0; i < G; ++i) {
      out[i].ctas_per_sm = variant_ctas_per_sm(w, variant);
      out[i].warp_tier = variant >> 1;
    }
  }
  for (State& s : S) {
    RCK(cudaMemsetAsync(s.g->totals, 0, sizeof(long long) * KADABRA_NSTAT, st));
    RCK(cudaMemsetAsync(s.g->count0, 0, sizeof(uint32_t) * s.g->n, st));
    RCK(cudaMemsetAsync(s.g->counts, 0, sizeof(uint32_t) * s.g->n, st));
  }
  std::vector<Job> jobs;
  double idle = 0.0;  // of the jobs' samples: expected to end at a root without arcs
  auto launch_jobs = [&]() -> kadabra_status {
    uint64_t work = 0;
    for (Job& j : jobs) {
      j.work_begin = work;
      work += j.count;
    }
    if (work == 0) return KADABRA_OK;
    SampleParams P = ws_params(w, fl);
    P.total_work = work;
    choose_screen(P, work, idle);
    idle = 0.0;
    if (jobs.size() == 1) {
      P.job0 = jobs[0];
    } else {
      RCK(cudaMemcpyAsync(w->d_jobs, jobs.data(), sizeof(Job) * jobs.size(), cudaMemcpyHostToDevice, st));
      P.jobs = w->d_jobs;
      P.njobs = (int)jobs.size();
    }
    return launch_sampler(w, P, st, variant);
  };
  auto make_job = [&](const State& s, uint32_t domain, uint64_t first, uint64_t count, uint32_t* counts,
                      uint64_t seed_i) {
    Job j;
    std::memset(&j, 0, sizeof(j));
    j.g = graph_dev(s.g);
    j.seed = seed_i;
    j.domain = domain;
    j.first_idx = first;
    j.count = count;
    j.counts = counts;
    j.totals = s.g->totals;
    idle += s.g->idle * (double)count;
    return j;
  };
  // Warm-up of every graph in one launch (Alg. 2 lines 1-5).  The same
  // launch also takes each graph's first main-loop batch: those samples
  // depend only on their indices, not on computeDelta, which only the first
  // stop test needs; so the warm-up's short launch does not run on its own.
  // The first round's test runs from the host; a device-driven loop takes
  // the later rounds.
  bool loop_on_device = false;
  for (const State& s : S) loop_on_device |= (s.cap + s.K - 1) / s.K > LOOP_GRAPH_MIN_ROUNDS;
  jobs.clear();
  for (int i = 0; i < G; ++i) jobs.push_back(make_job(S[i], 1, 0, S[i].alpha, S[i].g->count0, seed[i]));
  for (int i = 0; i < G; ++i) {
    S[i].pre = std::min<uint64_t>(S[i].K, S[i].cap);
    jobs.push_back(make_job(S[i], 0, 0, S[i].pre, S[i].g->counts, seed[i]));
  }
  tr.mark("setup, tuning");
  KTRY(launch_jobs());
  tr.mark("warm-up samples");
  // the non-zero warm-up counts of every graph, in node order, to the host
  {
    std::vector<NzJob> nzj(G);
    for (int i = 0; i < G; ++i) {
      nzj[i].count0 = S[i].g->count0;
      nzj[i].n = S[i].g->n;
      nzj[i].out = reinterpret_cast<uint32_t*>(S[i].g->btilde);  // scratch until b~ is computed
      nzj[i].blk = d_blk + (size_t)NZ_BLK * i;
      nzj[i].total = d_nzt + i;
    }
    RCK(cudaMemcpyAsync(d_nzj, nzj.data(), sizeof(NzJob) * G, cudaMemcpyHostToDevice, st));
    k_nz_count<<<dim3(NZ_BLK, G), 256, 0, st>>>(d_nzj);
    k_nz_offsets<<<G, 32, 0, st>>>(d_nzj, NZ_BLK);
    k_nz_scatter<<<dim3(NZ_BLK, G), 256, 0, st>>>(d_nzj);
    RCK(cudaGetLastError());
  }
  std::vector<unsigned> nnz(G);
  RCK(cudaMemcpyAsync(nnz.data(), d_nzt, sizeof(unsigned) * G, cudaMemcpyDeviceToHost, st));
  KTRY(read_status(w, st));
  std::vector<std::vector<uint32_t>> nzv(G);
  for (int i = 0; i < G; ++i) {
    nzv[i].resize(nnz[i]);
    if (nnz[i])
      RCK(cudaMemcpyAsync(nzv[i].data(), S[i].g->btilde, sizeof(uint32_t) * nnz[i], cudaMemcpyDeviceToHost, st));
  }
  RCK(cudaStreamSynchronize(st));
  // computeDelta per graph (Alg. 2 lines 6-14): a table by warm-up count
  std::vector<std::vector<double>> tab(G);
  for (int i = 0; i < G; ++i) {
    tab[i].resize(S[i].alpha + 1);
    KTRY(compute_delta_table(S[i].g->n, nzv[i].data(), nzv[i].size(), S[i].alpha, S[i].alpha, out[i].omega,
                             lambda[i], delta[i], cfg.eps, tab[i].data(), &out[i].C));
    RCK(cudaMemcpyAsync(S[i].g->lntab, tab[i].data(), sizeof(double) * tab[i].size(), cudaMemcpyHostToDevice, st));
  }
  tr.mark("compaction, Alg. 2");
  // stop tests of a set of graphs in one launch
  std::vector<CheckTabJob> cj;
  std::vector<CheckOut> co;
  // fail_fast: an intermediate test, whose maxima are read only if it holds
  auto check = [&](const std::vector<int>& which, bool fail_fast) -> kadabra_status {
    cj.clear();
    int64_t max_n = 1;
    for (int i : which) {
      CheckTabJob c;
      c.fail_fast = fail_fast ? 1 : 0;
      c.counts = S[i].g->counts;
      c.count0 = S[i].g->count0;
      c.lnT = S[i].g->lntab;
      c.n = S[i].g->n;
      c.tau = S[i].tau;
      c.omega = out[i].omega;
      c.lambda = lambda[i];
      c.out = d_co + cj.size();
      cj.push_back(c);
      max_n = std::max<int64_t>(max_n, c.n);
    }
    RCK(cudaMemcpyAsync(d_cj, cj.data(), sizeof(CheckTabJob) * cj.size(), cudaMemcpyHostToDevice, st));
    RCK(cudaMemsetAsync(d_co, 0, sizeof(CheckOut) * cj.size(), st));
    const int64_t want = (4 * (int64_t)w->num_sms + (int64_t)cj.size() - 1) / (int64_t)cj.size();
    const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(want, (max_n + 255) / 256));
    k_check_tab<<<dim3(bx, (unsigned)cj.size()), 256, 0, st>>>(d_cj);
    RCK(cudaGetLastError());
    co.resize(cj.size());
    RCK(cudaMemcpyAsync(co.data(), d_co, sizeof(CheckOut) * cj.size(), cudaMemcpyDeviceToHost, st));
    return read_status(w, st);
  };
  // main loop (Alg. 1): after the first round, on the device when some
  // graph has enough rounds left to repay building the CUDA graph, rounds
  // from the host otherwise (same results either way)
  for (bool first = true;; first = false) {
    bool left = false;
    for (const State& s : S) left |= !s.done;
    if (loop_on_device && !first && left) {  // rounds 2, 3, ... on the device
      std::vector<LoopRun> R(G);
      for (int i = 0; i < G; ++i) {
        R[i].g = S[i].g;
        R[i].seed = seed[i];
        R[i].tau = S[i].tau;
        R[i].cap = S[i].cap;
        R[i].K = S[i].K;
        R[i].omega = out[i].omega;
        R[i].lambda = lambda[i];
        R[i].done = S[i].done;
      }
      KTRY(run_loop_graph(G == 1 ? gs[0]->loop : w->loop, w, st, R, fl, variant));
      for (int i = 0; i < G; ++i) {
        if (S[i].done) continue;
        S[i].tau = R[i].tau;
        out[i].checks += R[i].checks;
        out[i].stopped_early = R[i].stopped;
        if (R[i].stopped) {  // the test that held found no failure, so its maxima are complete
          std::memcpy(&out[i].max_f, &R[i].co.max_f_bits, sizeof(double));
          std::memcpy(&out[i].max_g, &R[i].co.max_g_bits, sizeof(double));
          S[i].have_max = true;
        }
        S[i].done = true;
      }
      break;
    }
    jobs.clear();
    std::vector<int> sampled;
    std::vector<uint64_t> taken;
    for (int i = 0; i < G; ++i) {
      State& s = S[i];
      if (s.done) continue;
      if (s.pre) {  // the first batch, sampled with the warm-up
        taken.push_back(s.pre);
        s.pre = 0;
      } else {
        const uint64_t B = std::min<uint64_t>(s.K, s.cap - s.tau);
        jobs.push_back(make_job(s, 0, s.tau, B, s.g->counts, seed[i]));
        taken.push_back(B);
      }
      sampled.push_back(i);
    }
    if (sampled.empty()) break;
    if (!jobs.empty()) KTRY(launch_jobs());
    if (tr.on) {
      uint64_t ns = 0;
      for (const Job& j : jobs) ns += j.count;
      char what[64];
      std::snprintf(what, sizeof(what), "batch: %zu graphs, %llu samples", sampled.size(), (unsigned long long)ns);
      tr.mark(what);
    }
    std::vector<int> to_check;
    for (size_t q = 0; q < sampled.size(); ++q) {
      const int i = sampled[q];
      S[i].tau += taken[q];
      if (S[i].tau >= S[i].cap)
        S[i].done = true;
      else
        to_check.push_back(i);
    }
    if (to_check.empty()) {
      KTRY(read_status(w, st));
      continue;
    }
    KTRY(check(to_check, true));
    tr.mark("stop tests");
    for (size_t q = 0; q < to_check.size(); ++q) {
      const int i = to_check[q];
      out[i].checks++;
      if (!co[q].fail) {  // held: no failure cut it short, so its maxima are complete
        out[i].stopped_early = 1;
        S[i].done = true;
        std::memcpy(&out[i].max_f, &co[q].max_f_bits, sizeof(double));
        std::memcpy(&out[i].max_g, &co[q].max_g_bits, sizeof(double));
        S[i].have_max = true;
      }
    }
  }
  // f and g maxima at each final tau (a full test for the runs that reached
  // ceil(omega); the others keep those of the test that held); b~ = counts /
  // tau (Alg. 1 last line)
  std::vector<int> need;
  for (int i = 0; i < G; ++i)
    if (!S[i].have_max) need.push_back(i);
  if (!need.empty()) KTRY(check(need, false));
  for (size_t q = 0; q < need.size(); ++q) {
    std::memcpy(&out[need[q]].max_f, &co[q].max_f_bits, sizeof(double));
    std::memcpy(&out[need[q]].max_g, &co[q].max_g_bits, sizeof(double));
  }
  std::vector<long long> tot((size_t)G * KADABRA_NSTAT);
  for (int i = 0; i < G; ++i) {
    kadabra_result& r = out[i];
    kadabra_graph* g = S[i].g;
    r.tau = S[i].tau;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)w->num_sms, (g->n + 255) / 256));
    if (r.btilde || r.d_btilde) {
      k_btilde<<<blocks, 256, 0, st>>>(g->counts, g->n, r.tau, r.d_btilde ? r.d_btilde : g->btilde);
      RCK(cudaGetLastError());
    }
    if (r.d_counts)
      RCK(cudaMemcpyAsync(r.d_counts, g->counts, sizeof(uint32_t) * g->n, cudaMemcpyDeviceToDevice, st));
    if (r.counts) RCK(cudaMemcpyAsync(r.counts, g->counts, sizeof(uint32_t) * g->n, cudaMemcpyDeviceToHost, st));
    if (r.btilde)
      RCK(cudaMemcpyAsync(r.btilde, r.d_btilde ? r.d_btilde : g->btilde, sizeof(double) * g->n,
                          cudaMemcpyDeviceToHost, st));
    RCK(cudaMemcpyAsync(&tot[(size_t)i * KADABRA_NSTAT], g->totals, sizeof(long long) * KADABRA_NSTAT,
                        cudaMemcpyDeviceToHost, st));
  }
  KTRY(read_status(w, st));
  for (int i = 0; i < G; ++i)
    for (int q = 0; q < KADABRA_NSTAT; ++q) out[i].totals[q] = tot[(size_t)i * KADABRA_NSTAT + q];
#undef RCK
  return KADABRA_OK;
}


// ---------------------------------------------------------------- top-k runner
// Sec. 5 targets from the preliminary estimate, in the order the text gives
// them (the k first nodes, the others, then small gaps; every target below
// lambda raised to lambda).  top: the k1 first nodes' counts in ranking order.
struct TopkTargets {
  std::vector<double> L, U;  // for the k1 first nodes, in ranking order
  double lower_base;         // b~(v_k) - lambda_L(v_k) before the small-gap rule
  double a;                  // preliminary sample count
  double lambda;
  double others_U(uint32_t cnt) const {  // lambda_U of a node ranked below v_{k+1}
    const double u = lower_base - (double)cnt / a;
    return u >= lambda ? u : lambda;
  }
};

TopkTargets topk_targets(const std::vector<uint32_t>& top, int64_t n, int k, uint64_t alpha, double lambda) {
  TopkTargets T;
  const int k1 = (int)top.size();
  T.a = (double)alpha;
  T.lambda = lambda;
  T.L.assign(k1, 0.0);
  T.U.assign(k1, 0.0);
  auto bt = [&](int i) { return (double)top[i - 1] / T.a; };  // 1-based
  for (int i = 1; i <= k; ++i) {
    T.U[i - 1] = i == 1 ? 1.0 : (bt(i - 1) - bt(i)) / 2.0;
    T.L[i - 1] = i == n ? 1.0 : (bt(i) - bt(i + 1)) / 2.0;
  }
  T.lower_base = bt(k) - T.L[k - 1];
  for (int i = k + 1; i <= k1; ++i) {
    T.L[i - 1] = 1.0;
    T.U[i - 1] = bt(k) - T.L[k - 1] - bt(i);
  }
  for (int i = 1; i <= k && i + 1 <= n; ++i) {
    if (bt(i) - bt(i + 1) < 2.0 * lambda) T.L[i - 1] = T.U[i - 1] = T.L[i] = T.U[i] = lambda;
  }
  for (int i = 0; i < k1; ++i) {
    if (!(T.L[i] >= lambda)) T.L[i] = lambda;
    if (!(T.U[i] >= lambda)) T.U[i] = lambda;
  }
  return T;
}

// Alg. 2 with per-node targets over the nodes with a warm-up hit (node order);
// writes their ln(1/delta_L), ln(1/delta_U) and C; *l0 = the value of every
// node without a hit.
kadabra_status compute_delta_lv_host(int64_t n, const std::vector<double>& cL, const std::vector<double>& cU,
                                     double delta, double eps, std::vector<double>& lnL, std::vector<double>& lnU,
                                     double* C_out, double* l0) {
  const size_t m = cL.size();
  const double target = (delta / 2.0) - (eps * delta);
  // The c values repeat (they depend on a node's warm-up and preliminary
  // counts and, for the few top-k nodes, its rank): each bisection step
  // evaluates exp(-C / c) once per distinct c and then sums the nodes' terms
  // in node order, so every term and the order of the additions are those of
  // the plain per-node loop.
  std::vector<double> vals;                   // distinct positive c values
  std::vector<int32_t> iL(m, -1), iU(m, -1);  // each node's c_L, c_U in vals (-1: c <= 0)
  {
    size_t cap = 16;
    while (cap < 4 * m + 16) cap <<= 1;
    std::vector<uint64_t> keys(cap, 0);
    std::vector<int32_t> slot(cap, -1);
    auto intern = [&](double c) -> int32_t {
      if (!(c > 0.0)) return -1;
      uint64_t bits;
      std::memcpy(&bits, &c, sizeof(bits));
      size_t h = (size_t)((bits * 0x9E3779B97F4A7C15ull) >> 20) & (cap - 1);
      while (slot[h] >= 0 && keys[h] != bits) h = (h + 1) & (cap - 1);
      if (slot[h] < 0) {
        keys[h] = bits;
        slot[h] = (int32_t)vals.size();
        vals.push_back(c);
      }
      return slot[h];
    };
    for (size_t i = 0; i < m; ++i) {
      iL[i] = intern(cL[i]);
      iU[i] = intern(cU[i]);
    }
  }
  std::vector<double> ev(vals.size());
  auto sum_at = [&](double C) {
    for (size_t u = 0; u < vals.size(); ++u) ev[u] = std::exp(-C / vals[u]);
    double sum = 0.0;
    for (size_t i = 0; i < m; ++i) {
      const double eL = iL[i] >= 0 ? ev[iL[i]] : 0.0;
      const double eU = iU[i] >= 0 ? ev[iU[i]] : 0.0;
      sum += eL + eU;
    }
    return sum;
  };
  bool any = false;
  for (size_t i = 0; i < m; ++i) any = any || cL[i] > 0.0 || cU[i] > 0.0;
  double C = 0.0;
  if (any) {
    double lo = 0.0, hi = 1.0;
    int guard = 0;
    while (!(sum_at(hi) <= target)) {
      lo = hi;
      hi = 2.0 * hi;
      if (++guard > 2100) return fail(KADABRA_ERR_INTERNAL, "computeDelta: no bracket for C");
    }
    for (guard = 0; guard < 4000; ++guard) {
      const double mid = 0.5 * (lo + hi);
      if (mid <= lo || mid >= hi) break;
      if (sum_at(mid) <= target)
        hi = mid;
      else
        lo = mid;
    }
    C = hi;
  }
  const double floor_term = (eps * delta) / (2.0 * (double)n);
  lnL.resize(m);
  lnU.resize(m);
  for (size_t i = 0; i < m; ++i) {
    lnL[i] = -std::log((cL[i] > 0.0 ? std::exp(-C / cL[i]) : 0.0) + floor_term);
    lnU[i] = -std::log((cU[i] > 0.0 ? std::exp(-C / cU[i]) : 0.0) + floor_term);
  }
  *l0 = -std::log(0.0 + floor_term);
  *C_out = C;
  return KADABRA_OK;
}

kadabra_status ensure_topk_buffers(kadabra_graph* g, cudaStream_t st) {
  if (g->count_pre) return KADABRA_OK;
  KCK(cudaStreamSynchronize(st));
  void* p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(uint32_t) * (size_t)g->n));
  g->count_pre = (uint32_t*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(double) * (size_t)g->n));
  g->lnLv = (double*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(double) * (size_t)g->n));
  g->lnUv = (double*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(unsigned long long) * (size_t)TK_BLOCKS * (TOPK_MAX + 1)));
  g->tk_cand = (unsigned long long*)p;
  KTRY(gdev_alloc(g->allocs, &p, sizeof(TopkJob) + sizeof(TopkOut)));
  g->tk_dev = p;
  return KADABRA_OK;
}

// Alg. 1 in top-k mode on one graph: preliminary estimate (domain 2) and
// warm-up (domain 1) in one sampler launch, Sec. 5 targets, Alg. 2 with
// those targets, then batches of K samples with Alg. 3 after each.
kadabra_status run_topk(kadabra_graph* g, double lambda, double delta, int32_t k_in, uint64_t seed,
                        const kadabra_config& cfg, kadabra_result* out) {
  cudaStream_t st = as_stream(cfg.stream);
  Workspace* w = g->ws;
  const int64_t n = g->n;
  LoadTrace tr("top-k run");
  const int k = (int)std::min<int64_t>(k_in, n), k1 = (int)std::min<int64_t>((int64_t)k_in + 1, n);
  kadabra_result& r = *out;
  r.vd = cfg.vd > 0 ? cfg.vd : g->vd;
  r.omega = omega_host(lambda, delta, r.vd);
  const double cap_d = std::ceil(r.omega);
  if (!(cap_d >= 1.0 && cap_d < 1e15)) return fail(KADABRA_ERR_ARG, "omega out of range");
  const uint64_t cap = r.omega_cap = (uint64_t)cap_d;
  const uint64_t alpha = r.alpha = std::max<uint64_t>(1, (uint64_t)std::floor(r.omega / 100.0));
  const uint64_t K = r.check_interval = cfg.check_interval ? cfg.check_interval : auto_check_interval(r.omega);
  KTRY(ensure_ws(w, 2 * alpha + std::min(K, cap), 3));
  KTRY(ensure_run_buffers(g));
  KTRY(ensure_topk_buffers(g, st));
  if (w->nz_cap < 1) {
    KCK(cudaDeviceSynchronize());
    void* p;
    KTRY(dev_alloc(w->allocs, &p, sizeof(NzJob) + sizeof(unsigned) * (NZ_BLK + 1)));
    w->d_nz = p;
    w->nz_cap = 1;
  }
#define RCK(call)                                                                         \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) return fail(KADABRA_ERR_CUDA, cudaGetErrorString(e_));         \
  } while (0)
  TopkJob* d_job = static_cast<TopkJob*>(g->tk_dev);
  TopkOut* d_out = reinterpret_cast<TopkOut*>(d_job + 1);
  RCK(cudaMemsetAsync(g->totals, 0, sizeof(long long) * KADABRA_NSTAT, st));
  RCK(cudaMemsetAsync(g->count_pre, 0, sizeof(uint32_t) * n, st));
  RCK(cudaMemsetAsync(g->count0, 0, sizeof(uint32_t) * n, st));
  RCK(cudaMemsetAsync(g->counts, 0, sizeof(uint32_t) * n, st));
  int variant = 0;
  KTRY(tier_variant(g, w, st, cfg.ctas_per_sm, cfg.warp_tier, K, launch_flags(g), g->idle, false, &variant));
  r.ctas_per_sm = variant_ctas_per_sm(w, variant);
  r.warp_tier = variant >> 1;
  auto job = [&](uint32_t domain, uint64_t first, uint64_t count, uint32_t* counts) {
    Job j;
    std::memset(&j, 0, sizeof(j));
    j.g = graph_dev(g);
    j.seed = seed;
    j.domain = domain;
    j.first_idx = first;
    j.count = count;
    j.counts = counts;
    j.totals = g->totals;
    return j;
  };
  // preliminary estimate, warm-up and the first main-loop batch, one launch
  // (main-loop samples do not depend on the targets or computeDelta)
  const uint64_t B0 = std::min<uint64_t>(K, cap);
  {
    Job jobs[3] = {job(2, 0, alpha, g->count_pre), job(1, 0, alpha, g->count0), job(0, 0, B0, g->counts)};
    jobs[0].work_begin = 0;
    jobs[1].work_begin = alpha;
    jobs[2].work_begin = 2 * alpha;
    RCK(cudaMemcpyAsync(w->d_jobs, jobs, sizeof(jobs), cudaMemcpyHostToDevice, st));
    SampleParams P = ws_params(w, launch_flags(g));
    P.total_work = 2 * alpha + B0;
    choose_screen(P, P.total_work, g->idle * (double)P.total_work);
    P.jobs = w->d_jobs;
    P.njobs = 3;
    tr.mark("setup, tuning");
    KTRY(launch_sampler(w, P, st, variant));
    tr.mark("warm-up samples");
  }
  const int rest_blocks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)w->num_sms, (n + 255) / 256));
  // selection (select_only) or Alg. 3 over `counts` at `tau`
  TopkOut ho;
  auto topk_pass = [&](const uint32_t* counts, uint64_t tau, int select_only, int fail_fast = 0) -> kadabra_status {
    TopkJob J;
    std::memset(&J, 0, sizeof(J));
    J.counts = counts;
    J.lnL = g->lnLv;
    J.lnU = g->lnUv;
    J.n = n;
    J.tau = tau;
    J.omega = r.omega;
    J.lambda = lambda;
    J.k = k;
    J.k1 = k1;
    J.cand = g->tk_cand;
    J.select_only = select_only;
    J.fail_fast = fail_fast;
    J.out = d_out;
    RCK(cudaMemcpyAsync(d_job, &J, sizeof(J), cudaMemcpyHostToDevice, st));
    RCK(cudaMemsetAsync(d_out, 0, sizeof(TopkOut), st));
    k_topk_block<<<TK_BLOCKS, 256, 0, st>>>(counts, n, k1, g->tk_cand);
    k_topk_final<<<1, 256, 0, st>>>(d_job);
    if (!select_only) k_topk_rest<<<rest_blocks, 256, 0, st>>>(d_job);
    RCK(cudaGetLastError());
    RCK(cudaMemcpyAsync(&ho, d_out, sizeof(TopkOut), cudaMemcpyDeviceToHost, st));
    return read_status(w, st);
  };
  // the k1 first nodes of the preliminary estimate
  KTRY(topk_pass(g->count_pre, 1, 1));
  if (ho.nk != k1) return fail(KADABRA_ERR_INTERNAL, "top-k selection returned too few nodes");
  std::vector<uint32_t> top_cnt(k1), top_id(k1);
  for (int i = 0; i < k1; ++i) {
    top_cnt[i] = (uint32_t)(ho.keys[i] >> 32);
    top_id[i] = 0xFFFFFFFFu - (uint32_t)ho.keys[i];
  }
  const TopkTargets TT = topk_targets(top_cnt, n, k, alpha, lambda);
  std::unordered_map<uint32_t, int> rank_of;
  for (int i = 0; i < k1; ++i) rank_of[top_id[i]] = i;
  // nodes with a warm-up hit, in node order, with their preliminary hits
  NzJob* d_nzj = static_cast<NzJob*>(w->d_nz);
  unsigned* d_blk = reinterpret_cast<unsigned*>(d_nzj + 1);
  unsigned* d_nzt = d_blk + NZ_BLK;
  {
    NzJob z;
    std::memset(&z, 0, sizeof(z));
    z.count0 = g->count0;
    z.n = n;
    z.out = reinterpret_cast<uint32_t*>(g->btilde);  // scratch
    z.blk = d_blk;
    z.total = d_nzt;
    z.out_idx = reinterpret_cast<uint32_t*>(g->lnLv);  // scratch (filled below)
    z.aux = g->count_pre;
    z.out_aux = reinterpret_cast<uint32_t*>(g->lnUv);  // scratch
    RCK(cudaMemcpyAsync(d_nzj, &z, sizeof(z), cudaMemcpyHostToDevice, st));
    k_nz_count<<<dim3(NZ_BLK, 1), 256, 0, st>>>(d_nzj);
    k_nz_offsets<<<1, 32, 0, st>>>(d_nzj, NZ_BLK);
    k_nz_scatter<<<dim3(NZ_BLK, 1), 256, 0, st>>>(d_nzj);
    RCK(cudaGetLastError());
  }
  unsigned nnz = 0;
  RCK(cudaMemcpyAsync(&nnz, d_nzt, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  RCK(cudaStreamSynchronize(st));
  std::vector<uint32_t> nz_c0(nnz), nz_id(nnz), nz_pre(nnz);
  if (nnz) {
    RCK(cudaMemcpyAsync(nz_c0.data(), g->btilde, sizeof(uint32_t) * nnz, cudaMemcpyDeviceToHost, st));
    RCK(cudaMemcpyAsync(nz_id.data(), g->lnLv, sizeof(uint32_t) * nnz, cudaMemcpyDeviceToHost, st));
    RCK(cudaMemcpyAsync(nz_pre.data(), g->lnUv, sizeof(uint32_t) * nnz, cudaMemcpyDeviceToHost, st));
  }
  RCK(cudaStreamSynchronize(st));
  // c_L, c_U of those nodes (Alg. 2) with their Sec. 5 targets
  std::vector<double> cL(nnz), cU(nnz), vL, vU;
  for (unsigned i = 0; i < nnz; ++i) {
    double lamL = 1.0, lamU;
    auto it = rank_of.find(nz_id[i]);
    if (it != rank_of.end()) {
      lamL = TT.L[it->second];
      lamU = TT.U[it->second];
    } else {
      lamU = TT.others_U(nz_pre[i]);
    }
    const double b0 = (double)nz_c0[i] / (double)alpha;
    cL[i] = ((2.0 * b0) * r.omega) / (lamL * lamL);
    cU[i] = ((2.0 * b0) * r.omega) / (lamU * lamU);
  }
  double l0 = 0.0;
  tr.mark("selection, targets");
  KTRY(compute_delta_lv_host(n, cL, cU, delta, cfg.eps, vL, vU, &r.C, &l0));
  tr.mark("computeDelta");
  // per-node ln(1/delta) arrays: l0 everywhere, then the hit nodes' values
  if (g->tk_stage_cap < nnz) {
    KCK(cudaStreamSynchronize(st));
    gdev_free(g->allocs, g->tk_stage);
    void* p;
    KTRY(gdev_alloc(g->allocs, &p, (sizeof(uint32_t) + 2 * sizeof(double)) * (size_t)nnz));
    g->tk_stage = p;
    g->tk_stage_cap = nnz;
  }
  k_fill2<<<rest_blocks, 256, 0, st>>>(g->lnLv, g->lnUv, n, l0);
  RCK(cudaGetLastError());
  if (nnz) {
    double* sL = static_cast<double*>(g->tk_stage);
    double* sU = sL + nnz;
    uint32_t* sI = reinterpret_cast<uint32_t*>(sU + nnz);
    RCK(cudaMemcpyAsync(sI, nz_id.data(), sizeof(uint32_t) * nnz, cudaMemcpyHostToDevice, st));
    RCK(cudaMemcpyAsync(sL, vL.data(), sizeof(double) * nnz, cudaMemcpyHostToDevice, st));
    RCK(cudaMemcpyAsync(sU, vU.data(), sizeof(double) * nnz, cudaMemcpyHostToDevice, st));
    k_scatter2<<<rest_blocks, 256, 0, st>>>(g->lnLv, g->lnUv, sI, sL, sU, nnz);
    RCK(cudaGetLastError());
    RCK(cudaStreamSynchronize(st));  // host vectors stay alive until the copies are done
  }
  // main loop (Alg. 1) with Alg. 3 every K samples
  tr.mark("delta arrays");
  uint64_t tau = 0;
  for (;;) {
    const uint64_t B = std::min<uint64_t>(K, cap - tau);
    if (tau > 0) {  // the first batch came with the warm-up
      SampleParams P = ws_params(w, launch_flags(g));
      P.total_work = B;
      choose_screen(P, B, g->idle * (double)B);
      P.job0 = job(0, tau, B, g->counts);
      KTRY(launch_sampler(w, P, st, variant));
      tr.mark("main batch");
    }
    tau += B;
    if (tau >= cap) break;
    r.checks++;
    KTRY(topk_pass(g->counts, tau, 0, 1));  // the run's final pass below is a full one
    tr.mark("Alg. 3 test");
    if (!ho.fail) {
      r.stopped_early = 1;
      break;
    }
  }
  r.tau = tau;
  // a test that held found no failure, so its ranking and maxima are those of
  // a full pass at this tau; a run that reached ceil(omega) gets one
  if (!r.stopped_early) KTRY(topk_pass(g->counts, tau, 0));
  std::memcpy(&r.max_f, &ho.max_f_bits, sizeof(double));
  std::memcpy(&r.max_g, &ho.max_g_bits, sizeof(double));
  if (r.topk)
    for (int i = 0; i < k; ++i) r.topk[i] = (int32_t)(0xFFFFFFFFu - (uint32_t)ho.keys[i]);
  const int blocks = rest_blocks;
  if (r.btilde || r.d_btilde) {
    k_btilde<<<blocks, 256, 0, st>>>(g->counts, n, tau, r.d_btilde ? r.d_btilde : g->btilde);
    RCK(cudaGetLastError());
  }
  if (r.d_counts) RCK(cudaMemcpyAsync(r.d_counts, g->counts, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st));
  if (r.counts) RCK(cudaMemcpyAsync(r.counts, g->counts, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost, st));
  if (r.btilde)
    RCK(cudaMemcpyAsync(r.btilde, r.d_btilde ? r.d_btilde : g->btilde, sizeof(double) * n, cudaMemcpyDeviceToHost,
                        st));
  long long tot[KADABRA_NSTAT];
  RCK(cudaMemcpyAsync(tot, g->totals, sizeof(tot), cudaMemcpyDeviceToHost, st));
  KTRY(read_status(w, st));
  for (int q = 0; q < KADABRA_NSTAT; ++q) r.totals[q] = tot[q];
#undef RCK
  return KADABRA_OK;
}


// ================================================================ serving
// Continuous batching of KADABRA runs (Alg. 1, either mode) on one device.
// A worker thread admits submitted jobs in arrival order while the device
// memory their state needs fits the budget (and a slot is free), allocating
// that state stream-ordered; then, round after round, it samples the next
// batch of every active job in one sampler launch (the warm-up of a job just
// admitted, or its next K main-loop samples), runs each job's host step
// (computeDelta after its warm-up) and the stop tests of all jobs that
// sampled, and retires finished jobs.  A job's samples are keyed by its seed
// and sample index and its batches are the same K as alone, so its result
// does not depend on what runs beside it.
double mono_seconds() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

struct SrvJob {
  uint64_t id = 0;
  kadabra_graph* g = nullptr;
  double lambda = 0.0, delta = 0.0;
  int k = 0, k1 = 0;  // top-k mode when k > 0 (k, k1 clamped to n)
  uint64_t seed = 0;
  kadabra_config cfg;
  int64_t n = 0;
  uint64_t alpha = 0, cap = 0, K = 0, tau = 0, B = 0;
  uint64_t taken = 0, chunk = 0;  // samples of the current batch already taken, and in this round
  int phase = 0;  // 0 admitted, 1 warm-up next, 2 main loop, 3 finished
  bool final_due = false;
  void* block = nullptr;  // one stream-ordered allocation for all device state
  uint32_t *counts = nullptr, *count0 = nullptr, *count_pre = nullptr, *scratch = nullptr;
  double *lntab = nullptr, *lnLv = nullptr, *lnUv = nullptr;
  long long* totals = nullptr;
  unsigned long long* cand = nullptr;
  size_t footprint = 0;
  kadabra_result res;
  std::vector<uint32_t> h_counts;
  std::vector<int32_t> h_topk;
  kadabra_status status = KADABRA_OK;
  std::string err;
  bool finished = false;  // set under the server's lock
};

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// device bytes of a job's state (counters, compaction scratch, computeDelta
// table or per-node arrays, top-k selection survivors)
size_t srv_layout(SrvJob* J, bool carve) {
  const size_t n = (size_t)J->n;
  unsigned char* base = static_cast<unsigned char*>(J->block);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    void* p = carve ? base + off : nullptr;
    off += align256(bytes);
    return p;
  };
  J->counts = (uint32_t*)take(4 * n);
  J->count0 = (uint32_t*)take(4 * n);
  J->totals = (long long*)take(sizeof(long long) * KADABRA_NSTAT);
  if (J->k > 0) {
    J->count_pre = (uint32_t*)take(4 * n);
    J->lnLv = (double*)take(8 * n);
    J->lnUv = (double*)take(8 * n);
    J->scratch = (uint32_t*)take(20 * n);  // compaction (3 x 4n), then staging (20 per entry)
    J->cand = (unsigned long long*)take(sizeof(unsigned long long) * TK_BLOCKS * (TOPK_MAX + 1));
  } else {
    J->lntab = (double*)take(8 * (J->alpha + 1));
    J->scratch = (uint32_t*)take(4 * n);
  }
  return off;
}

} // namespace

struct kadabra_server {
  int device = 0, num_sms = 0;
  cudaStream_t st = nullptr;
  std::unique_ptr<Workspace> ws;
  size_t budget = 0, in_use = 0;
  int max_active = 0;
  std::mutex mu;
  std::condition_variable cv;
  std::deque<SrvJob*> pending;
  std::vector<SrvJob*> active;
  std::unordered_map<uint64_t, SrvJob*> jobs;
  bool stopping = false;
  std::thread th;
  // device descriptors of a round's batched kernels
  void* d_desc = nullptr;
  size_t desc_bytes = 0;
  TopkJob* d_tk = nullptr;
  TopkOut* d_tko = nullptr;
};

namespace {

std::atomic<uint64_t> g_next_job{1};
std::mutex g_srv_mu;
std::unordered_map<int, kadabra_server*> g_servers;
std::unordered_map<uint64_t, kadabra_server*> g_job_owner;
size_t g_srv_budget = 0;  // 0 = a quarter of the free device memory
int g_srv_max_active = 256;

#define SCK(call)                                                                         \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) return fail(KADABRA_ERR_CUDA, cudaGetErrorString(e_));         \
  } while (0)

kadabra_status srv_desc(kadabra_server* S, size_t bytes) {
  if (S->desc_bytes >= bytes) return KADABRA_OK;
  SCK(cudaStreamSynchronize(S->st));
  if (S->d_desc) cudaFree(S->d_desc);
  S->d_desc = nullptr;
  S->desc_bytes = 0;
  SCK(cudaMalloc(&S->d_desc, bytes));
  S->desc_bytes = bytes;
  return KADABRA_OK;
}

// the workspace must cover the largest graph of any job admitted
kadabra_status srv_workspace(kadabra_server* S, const kadabra_graph* g) {
  if (S->ws && S->ws->max_n >= g->n && S->ws->max_m >= g->m) return KADABRA_OK;
  SCK(cudaStreamSynchronize(S->st));
  auto w = std::make_unique<Workspace>();
  w->device = S->device;
  w->num_sms = S->num_sms;
  w->max_n = std::max<int32_t>(g->n, S->ws ? S->ws->max_n : 0);
  w->max_m = std::max<int64_t>(g->m, S->ws ? S->ws->max_m : 0);
  S->ws = std::move(w);
  return KADABRA_OK;
}

kadabra_status srv_start(kadabra_server* S, SrvJob* J) {
  KTRY(srv_workspace(S, J->g));
  SCK(cudaMallocAsync(&J->block, J->footprint, S->st));
  srv_layout(J, true);
  SCK(cudaMemsetAsync(J->counts, 0, 4 * (size_t)J->n, S->st));
  SCK(cudaMemsetAsync(J->count0, 0, 4 * (size_t)J->n, S->st));
  SCK(cudaMemsetAsync(J->totals, 0, sizeof(long long) * KADABRA_NSTAT, S->st));
  if (J->k > 0) SCK(cudaMemsetAsync(J->count_pre, 0, 4 * (size_t)J->n, S->st));
  J->phase = 1;
  return KADABRA_OK;
}

Job srv_job(const SrvJob* J, uint32_t domain, uint64_t first, uint64_t count, uint32_t* counts) {
  Job j;
  std::memset(&j, 0, sizeof(j));
  j.g = graph_dev(J->g);
  j.seed = J->seed;
  j.domain = domain;
  j.first_idx = first;
  j.count = count;
  j.counts = counts;
  j.totals = J->totals;
  return j;
}

// selection (select_only) or Alg. 3 of one top-k job over its counts at tau
kadabra_status srv_topk_pass(kadabra_server* S, SrvJob* J, const uint32_t* counts, int select_only, TopkOut* ho,
                             int fail_fast = 0) {
  TopkJob T;
  std::memset(&T, 0, sizeof(T));
  T.counts = counts;
  T.lnL = J->lnLv;
  T.lnU = J->lnUv;
  T.n = J->n;
  T.tau = J->tau;
  T.omega = J->res.omega;
  T.lambda = J->lambda;
  T.k = J->k;
  T.k1 = J->k1;
  T.cand = J->cand;
  T.select_only = select_only;
  T.fail_fast = fail_fast;
  T.out = S->d_tko;
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)S->num_sms, (J->n + 255) / 256));
  SCK(cudaMemcpyAsync(S->d_tk, &T, sizeof(T), cudaMemcpyHostToDevice, S->st));
  SCK(cudaMemsetAsync(S->d_tko, 0, sizeof(TopkOut), S->st));
  k_topk_block<<<TK_BLOCKS, 256, 0, S->st>>>(counts, J->n, J->k1, J->cand);
  k_topk_final<<<1, 256, 0, S->st>>>(S->d_tk);
  if (!select_only) k_topk_rest<<<blocks, 256, 0, S->st>>>(S->d_tk);
  SCK(cudaGetLastError());
  SCK(cudaMemcpyAsync(ho, S->d_tko, sizeof(TopkOut), cudaMemcpyDeviceToHost, S->st));
  SCK(cudaStreamSynchronize(S->st));
  return KADABRA_OK;
}

// computeDelta of jobs whose warm-up has just been sampled
kadabra_status srv_compute_delta(kadabra_server* S, const std::vector<SrvJob*>& W) {
  const int G = (int)W.size();
  if (G == 0) return KADABRA_OK;
  // top-k: the k1 first nodes of the preliminary estimate
  std::vector<TopkTargets> TT(G);
  std::vector<std::unordered_map<uint32_t, int>> rank_of(G);
  for (int i = 0; i < G; ++i) {
    SrvJob* J = W[i];
    if (J->k == 0) continue;
    TopkOut ho;
    KTRY(srv_topk_pass(S, J, J->count_pre, 1, &ho));
    if (ho.nk != J->k1) return fail(KADABRA_ERR_INTERNAL, "top-k selection returned too few nodes");
    std::vector<uint32_t> top(J->k1);
    for (int q = 0; q < J->k1; ++q) {
      top[q] = (uint32_t)(ho.keys[q] >> 32);
      rank_of[i][0xFFFFFFFFu - (uint32_t)ho.keys[q]] = q;
    }
    TT[i] = topk_targets(top, J->n, J->k, J->alpha, J->lambda);
  }
  // the warm-up hits of every job, compacted in node order (one launch set)
  KTRY(srv_desc(S, (sizeof(NzJob) + sizeof(unsigned) * (NZ_BLK + 1)) * (size_t)G));
  NzJob* d_nzj = static_cast<NzJob*>(S->d_desc);
  unsigned* d_blk = reinterpret_cast<unsigned*>(d_nzj + G);
  unsigned* d_nzt = d_blk + (size_t)NZ_BLK * G;
  std::vector<NzJob> nzj(G);
  for (int i = 0; i < G; ++i) {
    SrvJob* J = W[i];
    std::memset(&nzj[i], 0, sizeof(NzJob));
    nzj[i].count0 = J->count0;
    nzj[i].n = J->n;
    nzj[i].out = J->scratch;
    nzj[i].blk = d_blk + (size_t)NZ_BLK * i;
    nzj[i].total = d_nzt + i;
    if (J->k > 0) {
      nzj[i].out_idx = J->scratch + J->n;
      nzj[i].aux = J->count_pre;
      nzj[i].out_aux = J->scratch + 2 * J->n;
    }
  }
  SCK(cudaMemcpyAsync(d_nzj, nzj.data(), sizeof(NzJob) * G, cudaMemcpyHostToDevice, S->st));
  k_nz_count<<<dim3(NZ_BLK, G), 256, 0, S->st>>>(d_nzj);
  k_nz_offsets<<<G, 32, 0, S->st>>>(d_nzj, NZ_BLK);
  k_nz_scatter<<<dim3(NZ_BLK, G), 256, 0, S->st>>>(d_nzj);
  SCK(cudaGetLastError());
  std::vector<unsigned> nnz(G);
  SCK(cudaMemcpyAsync(nnz.data(), d_nzt, sizeof(unsigned) * G, cudaMemcpyDeviceToHost, S->st));
  SCK(cudaStreamSynchronize(S->st));
  std::vector<std::vector<uint32_t>> c0(G), ids(G), pre(G);
  for (int i = 0; i < G; ++i) {
    SrvJob* J = W[i];
    c0[i].resize(nnz[i]);
    if (!nnz[i]) continue;
    SCK(cudaMemcpyAsync(c0[i].data(), J->scratch, 4 * (size_t)nnz[i], cudaMemcpyDeviceToHost, S->st));
    if (J->k > 0) {
      ids[i].resize(nnz[i]);
      pre[i].resize(nnz[i]);
      SCK(cudaMemcpyAsync(ids[i].data(), J->scratch + J->n, 4 * (size_t)nnz[i], cudaMemcpyDeviceToHost, S->st));
      SCK(cudaMemcpyAsync(pre[i].data(), J->scratch + 2 * J->n, 4 * (size_t)nnz[i], cudaMemcpyDeviceToHost, S->st));
    }
  }
  SCK(cudaStreamSynchronize(S->st));
  std::vector<std::vector<double>> host_tab(G), hL(G), hU(G);
  for (int i = 0; i < G; ++i) {
    SrvJob* J = W[i];
    const double eps = J->cfg.eps;
    if (J->k == 0) {
      host_tab[i].resize(J->alpha + 1);
      KTRY(compute_delta_table(J->n, c0[i].data(), c0[i].size(), J->alpha, J->alpha, J->res.omega, J->lambda,
                               J->delta, eps, host_tab[i].data(), &J->res.C));
      SCK(cudaMemcpyAsync(J->lntab, host_tab[i].data(), sizeof(double) * host_tab[i].size(), cudaMemcpyHostToDevice,
                          S->st));
    } else {
      const unsigned m = nnz[i];
      std::vector<double> cL(m), cU(m);
      for (unsigned q = 0; q < m; ++q) {
        double lamL = 1.0, lamU;
        auto it = rank_of[i].find(ids[i][q]);
        if (it != rank_of[i].end()) {
          lamL = TT[i].L[it->second];
          lamU = TT[i].U[it->second];
        } else {
          lamU = TT[i].others_U(pre[i][q]);
        }
        const double b0 = (double)c0[i][q] / (double)J->alpha;
        cL[q] = ((2.0 * b0) * J->res.omega) / (lamL * lamL);
        cU[q] = ((2.0 * b0) * J->res.omega) / (lamU * lamU);
      }
      double l0 = 0.0;
      KTRY(compute_delta_lv_host(J->n, cL, cU, J->delta, eps, hL[i], hU[i], &J->res.C, &l0));
      const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)S->num_sms, (J->n + 255) / 256));
      k_fill2<<<blocks, 256, 0, S->st>>>(J->lnLv, J->lnUv, J->n, l0);
      SCK(cudaGetLastError());
      if (m) {
        // staging in the compaction scratch (20 bytes per entry)
        double* sL = reinterpret_cast<double*>(J->scratch);
        double* sU = sL + m;
        uint32_t* sI = reinterpret_cast<uint32_t*>(sU + m);
        SCK(cudaMemcpyAsync(sI, ids[i].data(), 4 * (size_t)m, cudaMemcpyHostToDevice, S->st));
        SCK(cudaMemcpyAsync(sL, hL[i].data(), 8 * (size_t)m, cudaMemcpyHostToDevice, S->st));
        SCK(cudaMemcpyAsync(sU, hU[i].data(), 8 * (size_t)m, cudaMemcpyHostToDevice, S->st));
        k_scatter2<<<blocks, 256, 0, S->st>>>(J->lnLv, J->lnUv, sI, sL, sU, m);
        SCK(cudaGetLastError());
      }
    }
    J->phase = 2;
    J->tau = 0;
  }
  SCK(cudaStreamSynchronize(S->st));  // host tables stay alive until copied
  return KADABRA_OK;
}

// stop tests (and final evaluations) of jobs that sampled this round
kadabra_status srv_checks(kadabra_server* S, const std::vector<SrvJob*>& C) {
  std::vector<SrvJob*> plain;
  for (SrvJob* J : C)
    if (J->k == 0) plain.push_back(J);
  if (!plain.empty()) {
    const int G = (int)plain.size();
    KTRY(srv_desc(S, (sizeof(CheckTabJob) + sizeof(CheckOut)) * (size_t)G));
    CheckTabJob* d_cj = static_cast<CheckTabJob*>(S->d_desc);
    CheckOut* d_co = reinterpret_cast<CheckOut*>(d_cj + G);
    std::vector<CheckTabJob> cj(G);
    int64_t max_n = 1;
    for (int i = 0; i < G; ++i) {
      SrvJob* J = plain[i];
      cj[i].counts = J->counts;
      cj[i].count0 = J->count0;
      cj[i].lnT = J->lntab;
      cj[i].n = J->n;
      cj[i].tau = J->tau;
      cj[i].omega = J->res.omega;
      cj[i].lambda = J->lambda;
      cj[i].out = d_co + i;
      cj[i].fail_fast = J->final_due ? 0 : 1;  // at ceil(omega) the maxima are the result
      max_n = std::max<int64_t>(max_n, J->n);
    }
    SCK(cudaMemcpyAsync(d_cj, cj.data(), sizeof(CheckTabJob) * G, cudaMemcpyHostToDevice, S->st));
    SCK(cudaMemsetAsync(d_co, 0, sizeof(CheckOut) * G, S->st));
    const int64_t want = (4 * (int64_t)S->num_sms + G - 1) / G;
    const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(want, (max_n + 255) / 256));
    k_check_tab<<<dim3(bx, (unsigned)G), 256, 0, S->st>>>(d_cj);
    SCK(cudaGetLastError());
    std::vector<CheckOut> co(G);
    SCK(cudaMemcpyAsync(co.data(), d_co, sizeof(CheckOut) * G, cudaMemcpyDeviceToHost, S->st));
    SCK(cudaStreamSynchronize(S->st));
    for (int i = 0; i < G; ++i) {
      SrvJob* J = plain[i];
      std::memcpy(&J->res.max_f, &co[i].max_f_bits, sizeof(double));
      std::memcpy(&J->res.max_g, &co[i].max_g_bits, sizeof(double));
      if (J->final_due) continue;  // reached ceil(omega): evaluation only
      J->res.checks++;
      if (!co[i].fail) {
        J->res.stopped_early = 1;
        J->final_due = true;
      }
    }
  }
  for (SrvJob* J : C) {
    if (J->k == 0) continue;
    TopkOut ho;
    KTRY(srv_topk_pass(S, J, J->counts, 0, &ho, J->final_due ? 0 : 1));
    std::memcpy(&J->res.max_f, &ho.max_f_bits, sizeof(double));
    std::memcpy(&J->res.max_g, &ho.max_g_bits, sizeof(double));
    J->h_topk.resize(J->k);
    for (int q = 0; q < J->k; ++q) J->h_topk[q] = (int32_t)(0xFFFFFFFFu - (uint32_t)ho.keys[q]);
    if (J->final_due) continue;
    J->res.checks++;
    if (!ho.fail) {
      J->res.stopped_early = 1;
      J->final_due = true;
    }
  }
  return KADABRA_OK;
}

kadabra_status srv_finish(kadabra_server* S, SrvJob* J) {
  J->res.tau = J->tau;
  J->h_counts.resize(J->n);
  long long tot[KADABRA_NSTAT];
  SCK(cudaMemcpyAsync(J->h_counts.data(), J->counts, 4 * (size_t)J->n, cudaMemcpyDeviceToHost, S->st));
  SCK(cudaMemcpyAsync(tot, J->totals, sizeof(tot), cudaMemcpyDeviceToHost, S->st));
  SCK(cudaStreamSynchronize(S->st));
  for (int q = 0; q < KADABRA_NSTAT; ++q) J->res.totals[q] = tot[q];
  return KADABRA_OK;
}

void srv_release(kadabra_server* S, SrvJob* J) {
  if (J->block) cudaFreeAsync(J->block, S->st);
  J->block = nullptr;
  J->phase = 3;
  J->res.t_done = mono_seconds();
}

// one round over the active jobs; returns the jobs that finished
// Samples one round takes in all, shared among the active jobs: a job's
// batch of K samples is taken in chunks of at least SRV_MIN_CHUNK over
// several rounds when many jobs are active, and its stop test runs once the
// K samples are in.  Sample indices and test points stay those of the job
// alone, so results do not change; a round no longer lasts as long as the
// largest job's batch, which would hold back the small jobs in it.
constexpr uint64_t SRV_ROUND_SAMPLES = 16384;
constexpr uint64_t SRV_MIN_CHUNK = 1024;

kadabra_status srv_round(kadabra_server* S, std::vector<SrvJob*>& act, std::vector<SrvJob*>& done) {
  std::vector<Job> jobs;
  std::vector<SrvJob*> warm, main_j;
  uint64_t nrun = 0;
  for (SrvJob* J : act) nrun += (J->phase == 1 || J->phase == 2) ? 1 : 0;
  const uint64_t quota = std::max<uint64_t>(SRV_MIN_CHUNK, SRV_ROUND_SAMPLES / std::max<uint64_t>(nrun, 1));
  std::vector<SrvJob*> first;  // new jobs whose first main-loop chunk rides with their warm-up
  double idle = 0.0;           // of the jobs' samples: expected to end at a root without arcs
  auto add = [&](SrvJob* J, const Job& j) {
    jobs.push_back(j);
    idle += J->g->idle * (double)j.count;
  };
  for (SrvJob* J : act) {
    if (J->phase == 1) {
      if (J->k > 0) add(J, srv_job(J, 2, 0, J->alpha, J->count_pre));
      add(J, srv_job(J, 1, 0, J->alpha, J->count0));
      warm.push_back(J);
      // main-loop samples do not depend on computeDelta: the first batch (or
      // its first chunk) goes into the same launch
      J->B = std::min<uint64_t>(J->K, J->cap - J->tau);
      J->taken = 0;
      J->chunk = std::min<uint64_t>(J->B, quota);
      add(J, srv_job(J, 0, J->tau, J->chunk, J->counts));
      first.push_back(J);
    } else if (J->phase == 2) {
      if (J->taken == 0) J->B = std::min<uint64_t>(J->K, J->cap - J->tau);  // the next batch
      J->chunk = std::min<uint64_t>(J->B - J->taken, quota);
      add(J, srv_job(J, 0, J->tau + J->taken, J->chunk, J->counts));
      main_j.push_back(J);
    }
  }
  if (jobs.empty()) return KADABRA_OK;
  uint64_t work = 0;
  for (Job& j : jobs) {
    j.work_begin = work;
    work += j.count;
  }
  Workspace* w = S->ws.get();
  KTRY(ensure_ws(w, work, (int)jobs.size()));
  uint32_t fl = 0;  // the warp tier and the row searches, if any job's graph takes them (they change no result)
  for (SrvJob* J : act) fl |= launch_flags(J->g) & SHARED_LAUNCH_FLAGS;
  SampleParams P = ws_params(w, fl);
  P.total_work = work;
  choose_screen(P, work, idle);
  if (jobs.size() == 1) {
    P.job0 = jobs[0];
  } else {
    SCK(cudaMemcpyAsync(w->d_jobs, jobs.data(), sizeof(Job) * jobs.size(), cudaMemcpyHostToDevice, S->st));
    P.jobs = w->d_jobs;
    P.njobs = (int)jobs.size();
  }
  KTRY(launch_sampler(w, P, S->st));
  KTRY(read_status(w, S->st));
  KTRY(srv_compute_delta(S, warm));
  main_j.insert(main_j.end(), first.begin(), first.end());  // now in the main loop, their chunk taken
  std::vector<SrvJob*> chk;
  for (SrvJob* J : main_j) {
    J->taken += J->chunk;
    if (J->taken < J->B) continue;  // the batch goes on next round
    J->taken = 0;
    J->tau += J->B;
    if (J->tau >= J->cap) J->final_due = true;
    chk.push_back(J);
  }
  KTRY(srv_checks(S, chk));
  for (SrvJob* J : chk)
    if (J->final_due) {
      KTRY(srv_finish(S, J));
      done.push_back(J);
    }
  return KADABRA_OK;
}

void srv_loop(kadabra_server* S) {
  cudaSetDevice(S->device);
  for (;;) {
    std::vector<SrvJob*> act, admitted;
    {
      std::unique_lock<std::mutex> lk(S->mu);
      S->cv.wait(lk, [&] { return S->stopping || !S->pending.empty() || !S->active.empty(); });
      if (S->stopping && S->pending.empty() && S->active.empty()) return;
      // admission in arrival order while memory and slots allow (a job larger
      // than the whole budget is admitted when nothing else is active)
      while (!S->pending.empty() && (int)S->active.size() < S->max_active) {
        SrvJob* J = S->pending.front();
        if (!S->active.empty() && S->in_use + J->footprint > S->budget) break;
        S->pending.pop_front();
        S->in_use += J->footprint;
        S->active.push_back(J);
        admitted.push_back(J);
      }
      act = S->active;
    }
    std::vector<SrvJob*> done;
    for (SrvJob* J : admitted) {
      J->res.t_start = mono_seconds();
      const kadabra_status st = srv_start(S, J);
      if (st != KADABRA_OK) {
        J->status = st;
        J->err = kadabra_last_error();
        done.push_back(J);
      }
    }
    std::vector<SrvJob*> live;
    for (SrvJob* J : act)
      if (std::find(done.begin(), done.end(), J) == done.end()) live.push_back(J);
    const kadabra_status st = srv_round(S, live, done);
    if (st != KADABRA_OK) {  // a device error of the round fails every job in it
      const std::string msg = kadabra_last_error();
      for (SrvJob* J : live)
        if (std::find(done.begin(), done.end(), J) == done.end()) {
          J->status = st;
          J->err = msg;
          done.push_back(J);
        }
    }
    for (SrvJob* J : done) srv_release(S, J);
    cudaStreamSynchronize(S->st);
    {
      std::lock_guard<std::mutex> lk(S->mu);
      for (SrvJob* J : done) {
        S->in_use -= J->footprint;
        S->active.erase(std::find(S->active.begin(), S->active.end(), J));
        J->finished = true;
      }
    }
    if (!done.empty()) S->cv.notify_all();
  }
}

kadabra_status srv_get(int device, kadabra_server** out) {
  std::lock_guard<std::mutex> lk(g_srv_mu);
  auto it = g_servers.find(device);
  if (it != g_servers.end()) {
    *out = it->second;
    return KADABRA_OK;
  }
  auto S = std::make_unique<kadabra_server>();
  S->device = device;
  SCK(cudaSetDevice(device));
  SCK(cudaDeviceGetAttribute(&S->num_sms, cudaDevAttrMultiProcessorCount, device));
  SCK(cudaStreamCreateWithFlags(&S->st, cudaStreamNonBlocking));
  size_t free_b = 0, total_b = 0;
  SCK(cudaMemGetInfo(&free_b, &total_b));
  S->budget = g_srv_budget ? g_srv_budget : free_b / 4;
  S->max_active = g_srv_max_active;
  SCK(cudaMalloc((void**)&S->d_tk, sizeof(TopkJob) + sizeof(TopkOut)));
  S->d_tko = reinterpret_cast<TopkOut*>(S->d_tk + 1);
  kadabra_server* raw = S.release();
  raw->th = std::thread(srv_loop, raw);
  g_servers[device] = raw;
  *out = raw;
  return KADABRA_OK;
}

// keeps the caller's buffer pointers, zeroes the rest of a result
void reset_result(kadabra_result* r) {
  uint32_t* ch = r->counts;
  double* bh = r->btilde;
  uint32_t* cd = r->d_counts;
  double* bd = r->d_btilde;
  int32_t* tk = r->topk;
  std::memset(r, 0, sizeof(*r));
  r->counts = ch;
  r->btilde = bh;
  r->d_counts = cd;
  r->d_btilde = bd;
  r->topk = tk;
}

// ================================================================ no-alloc sampler
// A variant of the sampler batch for callers that cannot allocate device
// memory.  Its scratch is one file-scope device array; see the ABI comment of
// kadabra_sample_batch_noalloc for the limits.
#ifndef KD_NA_MAX_CTAS
#define KD_NA_MAX_CTAS 304
#endif
#ifndef KD_NA_PCAP
#define KD_NA_PCAP 512
#endif
constexpr int NA_MAX_CTAS = KD_NA_MAX_CTAS;   // CTAs per launch at most (2 per SM on 152 SMs)
constexpr int NA_PCAP = KD_NA_PCAP;           // a sample has at most PI_SEGS * NA_PCAP candidate edges
constexpr int NA_MED_CTAS = 32;               // CTAs of the large-table launch (each with one tier-M table)
constexpr uint64_t NA_MAX_BATCH = 65536;      // samples per call
constexpr size_t NA_OFF_CTR = 0;              // Q_COUNT counters, then the status word
constexpr size_t NA_OFF_STATUS = sizeof(unsigned long long) * Q_COUNT;
constexpr size_t NA_HEADER = 256;             // cleared on every call
constexpr size_t NA_OFF_QB = NA_HEADER;
constexpr size_t NA_OFF_QL = NA_OFF_QB + sizeof(unsigned long long) * NA_MAX_BATCH;
constexpr size_t NA_OFF_PI = NA_OFF_QL + sizeof(unsigned long long) * NA_MAX_BATCH;
constexpr size_t NA_OFF_MED = NA_OFF_PI + sizeof(PiEntry) * (size_t)NA_MAX_CTAS * PI_SEGS * NA_PCAP;
constexpr int NA_MED_HLOG = 15;               // its tier-M tables: 32768 hash slots,
constexpr int NA_MED_LCAP = 16384;            //   lists of 16384 nodes
// one tier-M table (gm_layout of NA_MED_HLOG, NA_MED_LCAP, MED_MAXD), 256-byte aligned
constexpr size_t NA_MED_STRIDE =
    ((((2 * sizeof(unsigned long long)) << NA_MED_HLOG) + sizeof(int2) * ((size_t)NA_MED_LCAP + 1) +
      sizeof(int32_t) * (size_t)NA_MED_LCAP + sizeof(uint32_t) * (size_t)NA_MED_LCAP +
      sizeof(int) * 4 * (size_t)(MED_MAXD + 2)) +
     255) & ~size_t(255);
constexpr size_t NA_BYTES = NA_OFF_MED + NA_MED_STRIDE * NA_MED_CTAS;
static_assert(NA_OFF_STATUS + sizeof(int32_t) <= NA_HEADER, "no-alloc header");

// Shared by every call on a device; the host never names it directly except
// to ask for its device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

struct NoAllocDevice {
  bool ready = false;
  unsigned char* scratch = nullptr;  // device address of g_noalloc_scratch
  int grid_s = 0, grid_b = 0;
  size_t smem_s = 0, smem_b = 0;
};
constexpr int NA_MAX_DEVICES = 64;
NoAllocDevice g_na_dev[NA_MAX_DEVICES];
std::mutex g_na_mu;

// once per device, with that device current: kernel attributes, grid sizes
// and the device address of the scratch array
kadabra_status noalloc_setup(int dev, NoAllocDevice** out) {
  if (dev < 0 || dev >= NA_MAX_DEVICES) return fail(KADABRA_ERR_ARG, "device index out of range");
  std::lock_guard<std::mutex> lock(g_na_mu);
  NoAllocDevice& d = g_na_dev[dev];
  if (!d.ready) {
    int sms = 0, per_sm = 0;
    KCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    d.smem_s = fast_smem_bytes();
    d.smem_b = big_smem_bytes();
    KCK(cudaFuncSetAttribute(k_sample<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.smem_s));
    KCK(cudaFuncSetAttribute(k_sample<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.smem_b));
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<0>, 32 * NW_S, d.smem_s));
    if (per_sm < 1) return fail(KADABRA_ERR_CAPACITY, "sampler does not fit on an SM");
    d.grid_s = std::min(sms * per_sm, NA_MAX_CTAS);
    KCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample<2>, 32 * NW_BIG, d.smem_b));
    if (per_sm < 1) return fail(KADABRA_ERR_CAPACITY, "large-table sampler does not fit on an SM");
    d.grid_b = std::min(sms * per_sm, NA_MED_CTAS);
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || ptr == nullptr)
      return fail(KADABRA_ERR_CUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
    d.scratch = static_cast<unsigned char*>(ptr);
    {
      size_t a, b, c2, e2;
      if (gm_layout(NA_MED_HLOG, NA_MED_LCAP, MED_MAXD, &a, &b, &c2, &e2) != NA_MED_STRIDE)
        return fail(KADABRA_ERR_INTERNAL, "tier-M table layout");
    }
    // the tier-M tables start empty (every key word EMPTY, sigma 0); each
    // sample clears what it used, so they stay so from call to call
    KCK(cudaMemset(d.scratch + NA_OFF_MED, 0, NA_MED_STRIDE * NA_MED_CTAS));
    for (int b = 0; b < NA_MED_CTAS; ++b)
      KCK(cudaMemset(d.scratch + NA_OFF_MED + (size_t)b * NA_MED_STRIDE, 0xFF,
                     sizeof(unsigned long long) << NA_MED_HLOG));
    KCK(cudaDeviceSynchronize());
    d.ready = true;
  }
  *out = &d;
  return KADABRA_OK;
}

}  // namespace

// ================================================================ C ABI
extern "C" {


// ---------------------------------------------------------------- serving
kadabra_status kadabra_serve_configure(uint64_t budget_bytes, int32_t max_active) {
  if (max_active < 1) return fail(KADABRA_ERR_ARG, "max_active must be >= 1");
  std::lock_guard<std::mutex> lk(g_srv_mu);
  if (!g_servers.empty()) return fail(KADABRA_ERR_ARG, "the server is already running (configure before the first submit)");
  g_srv_budget = (size_t)budget_bytes;
  g_srv_max_active = max_active;
  return KADABRA_OK;
}

kadabra_status kadabra_submit(kadabra_graph* g, double lambda, double delta, int32_t k, uint64_t seed,
                              const kadabra_config* cfg_in, uint64_t* job) {
  if (!g || !job) return fail(KADABRA_ERR_ARG, "graph or job is NULL");
  if (g->is_view) return fail(KADABRA_ERR_ARG, "batch views cannot be submitted");
  kadabra_config cfg;
  kadabra_config_default(&cfg);
  if (cfg_in) cfg = *cfg_in;
  if (k < 0 || k > TOPK_MAX) return fail(KADABRA_ERR_ARG, "k must be in [0, 256]");
  if (!(lambda > 0.0 && lambda < 1.0) || !(delta > 0.0 && delta < 1.0) || !(cfg.eps >= 0.0 && cfg.eps < 0.5))
    return fail(KADABRA_ERR_ARG, "lambda and delta must be in (0,1), eps in [0,0.5)");
  auto J = std::make_unique<SrvJob>();
  std::memset(&J->res, 0, sizeof(J->res));
  J->g = g;
  J->lambda = lambda;
  J->delta = delta;
  J->seed = seed;
  J->cfg = cfg;
  J->n = g->n;
  J->k = (int)std::min<int64_t>(k, g->n);
  J->k1 = k > 0 ? (int)std::min<int64_t>((int64_t)k + 1, g->n) : 0;
  kadabra_result& r = J->res;
  r.vd = cfg.vd > 0 ? cfg.vd : g->vd;
  r.omega = omega_host(lambda, delta, r.vd);
  const double cap_d = std::ceil(r.omega);
  if (!(cap_d >= 1.0 && cap_d < 1e15)) return fail(KADABRA_ERR_ARG, "omega out of range");
  J->cap = r.omega_cap = (uint64_t)cap_d;
  J->alpha = r.alpha = std::max<uint64_t>(1, (uint64_t)std::floor(r.omega / 100.0));
  J->K = r.check_interval = cfg.check_interval ? cfg.check_interval : auto_check_interval(r.omega);
  J->footprint = srv_layout(J.get(), false);
  r.t_submit = mono_seconds();
  kadabra_server* S = nullptr;
  KTRY(srv_get(g->device, &S));
  J->id = g_next_job.fetch_add(1);
  *job = J->id;
  {
    std::lock_guard<std::mutex> lk(g_srv_mu);
    g_job_owner[J->id] = S;
  }
  {
    std::lock_guard<std::mutex> lk(S->mu);
    S->jobs[J->id] = J.get();
    S->pending.push_back(J.release());
  }
  S->cv.notify_all();
  return KADABRA_OK;
}

kadabra_status kadabra_poll(uint64_t job, int32_t wait, int32_t* done, kadabra_result* out) {
  if (!done) return fail(KADABRA_ERR_ARG, "done is NULL");
  *done = 0;
  kadabra_server* S = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_srv_mu);
    auto it = g_job_owner.find(job);
    if (it == g_job_owner.end()) return fail(KADABRA_ERR_ARG, "unknown job (never submitted, or already collected)");
    S = it->second;
  }
  SrvJob* J = nullptr;
  {
    std::unique_lock<std::mutex> lk(S->mu);
    J = S->jobs.at(job);
    if (!J->finished) {
      if (!wait) return KADABRA_OK;
      S->cv.wait(lk, [&] { return J->finished; });
    }
    S->jobs.erase(job);
  }
  {
    std::lock_guard<std::mutex> lk(g_srv_mu);
    g_job_owner.erase(job);
  }
  std::unique_ptr<SrvJob> own(J);
  *done = 1;
  if (!out) return J->status == KADABRA_OK ? KADABRA_OK : fail(J->status, J->err);
  kadabra_result keep = *out;
  *out = J->res;
  out->counts = keep.counts;
  out->btilde = keep.btilde;
  out->d_counts = keep.d_counts;
  out->d_btilde = keep.d_btilde;
  out->topk = keep.topk;
  out->status = J->status;
  if (J->status != KADABRA_OK) return fail(J->status, J->err);
  const int64_t n = J->n;
  const double t = (double)J->tau;
  if (out->counts) std::memcpy(out->counts, J->h_counts.data(), 4 * (size_t)n);
  if (out->btilde)
    for (int64_t v = 0; v < n; ++v) out->btilde[v] = (double)J->h_counts[v] / t;
  if (out->topk)
    for (int q = 0; q < J->k && q < (int)J->h_topk.size(); ++q) out->topk[q] = J->h_topk[q];
  if (out->d_counts || out->d_btilde) {
    KCK(cudaSetDevice(S->device));
    if (out->d_counts) KCK(cudaMemcpy(out->d_counts, J->h_counts.data(), 4 * (size_t)n, cudaMemcpyHostToDevice));
    if (out->d_btilde) {
      std::vector<double> b(n);
      for (int64_t v = 0; v < n; ++v) b[v] = (double)J->h_counts[v] / t;
      KCK(cudaMemcpy(out->d_btilde, b.data(), 8 * (size_t)n, cudaMemcpyHostToDevice));
    }
  }
  return KADABRA_OK;
}

void kadabra_serve_shutdown(void) {
  std::vector<kadabra_server*> all;
  {
    std::lock_guard<std::mutex> lk(g_srv_mu);
    for (auto& kv : g_servers) all.push_back(kv.second);
    g_servers.clear();
  }
  for (kadabra_server* S : all) {
    {
      std::lock_guard<std::mutex> lk(S->mu);
      S->stopping = true;
    }
    S->cv.notify_all();
    if (S->th.joinable()) S->th.join();
    cudaSetDevice(S->device);
    cudaStreamSynchronize(S->st);
    {
      std::lock_guard<std::mutex> lk(g_srv_mu);
      for (auto& kv : S->jobs) g_job_owner.erase(kv.first);
    }
    for (auto& kv : S->jobs) delete kv.second;
    if (S->d_desc) cudaFree(S->d_desc);
    if (S->d_tk) cudaFree(S->d_tk);
    S->ws.reset();
    cudaStreamDestroy(S->st);
    delete S;
  }
}


// ---------------------------------------------------------------- measurement helper
kadabra_status kadabra_l2_read_probe(uint64_t bytes, int32_t reps, double* gbs) {
  if (!gbs || bytes < 16 || reps < 1) return fail(KADABRA_ERR_ARG, "bad probe arguments");
  int dev = 0, sms = 0;
  KCK(cudaGetDevice(&dev));
  KCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const size_t n4 = (size_t)bytes / 16;
  float4* buf = nullptr;
  float* sink = nullptr;
  KCK(cudaMalloc(&buf, n4 * 16));
  if (cudaMalloc(&sink, sizeof(float)) != cudaSuccess) {
    cudaFree(buf);
    return fail(KADABRA_ERR_OOM, "probe sink");
  }
  cudaMemset(buf, 0, n4 * 16);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int grid = 8 * sms;
  k_l2_read<<<grid, 256>>>(buf, n4, 2, sink);  // brings the buffer into L2
  cudaEventRecord(e0);
  k_l2_read<<<grid, 256>>>(buf, n4, reps, sink);
  cudaEventRecord(e1);
  const cudaError_t e = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(buf);
  cudaFree(sink);
  if (e != cudaSuccess) return fail(KADABRA_ERR_CUDA, cudaGetErrorString(e));
  *gbs = (double)n4 * 16.0 * (double)reps / ((double)ms * 1e-3) / 1e9;
  return KADABRA_OK;
}

const char* kadabra_last_error(void) { return g_last_error.c_str(); }

void kadabra_config_default(kadabra_config* cfg) {
  if (!cfg) return;
  std::memset(cfg, 0, sizeof(*cfg));
  cfg->eps = 0.001;
  cfg->check_interval = 1000;
}

double kadabra_omega(double lambda, double delta, int64_t vd) { return omega_host(lambda, delta, vd); }

kadabra_status kadabra_load_csr(int32_t n, int64_t m, const int32_t* row_ptr, const int32_t* col, int directed,
                                const int32_t* rrow_ptr, const int32_t* rcol, kadabra_graph** out) {
  kadabra_graph* g = nullptr;
  KTRY(new_graph(n, m, directed, out, &g));
  if (!row_ptr || (m > 0 && !col) || (directed && (!rrow_ptr || (m > 0 && !rcol))) ||
      (!directed && (rrow_ptr || rcol))) {
    kadabra_free_graph(g);
    return fail(KADABRA_ERR_ARG, "missing or unexpected CSR arrays");
  }
  if (row_ptr[0] != 0 || row_ptr[n] != m || (directed && (rrow_ptr[0] != 0 || rrow_ptr[n] != m))) {
    kadabra_free_graph(g);
    return fail(KADABRA_ERR_CSR, "row_ptr[0] must be 0 and row_ptr[n] must equal m");
  }
  kadabra_status st = KADABRA_OK;
  void* p;
  const size_t rb = sizeof(int32_t) * ((size_t)n + 1), cb = sizeof(int32_t) * (size_t)m;
  if ((st = gdev_alloc(g->allocs, &p, rb)) != KADABRA_OK) goto bad;
  g->rp = (int32_t*)p;
  if ((st = gdev_alloc(g->allocs, &p, cb)) != KADABRA_OK) goto bad;
  g->ci = (int32_t*)p;
  if (cudaMemcpy(g->rp, row_ptr, rb, cudaMemcpyHostToDevice) != cudaSuccess ||
      (m > 0 && cudaMemcpy(g->ci, col, cb, cudaMemcpyHostToDevice) != cudaSuccess)) {
    st = fail(KADABRA_ERR_CUDA, "CSR upload failed");
    goto bad;
  }
  if (directed) {
    if ((st = gdev_alloc(g->allocs, &p, rb)) != KADABRA_OK) goto bad;
    g->rrp = (int32_t*)p;
    if ((st = gdev_alloc(g->allocs, &p, cb)) != KADABRA_OK) goto bad;
    g->rci = (int32_t*)p;
    if (cudaMemcpy(g->rrp, rrow_ptr, rb, cudaMemcpyHostToDevice) != cudaSuccess ||
        (m > 0 && cudaMemcpy(g->rci, rcol, cb, cudaMemcpyHostToDevice) != cudaSuccess)) {
      st = fail(KADABRA_ERR_CUDA, "reverse CSR upload failed");
      goto bad;
    }
  }
  if ((st = finish_load(g)) != KADABRA_OK) goto bad;
  *out = g;
  return KADABRA_OK;
bad:
  kadabra_free_graph(g);
  return st;
}

kadabra_status kadabra_load_csr_device(int32_t n, int64_t m, const int32_t* d_row_ptr, const int32_t* d_col,
                                       int directed, const int32_t* d_rrow_ptr, const int32_t* d_rcol,
                                       kadabra_graph** out) {
  kadabra_graph* g = nullptr;
  KTRY(new_graph(n, m, directed, out, &g));
  if (!d_row_ptr || (m > 0 && !d_col) || (directed && (!d_rrow_ptr || (m > 0 && !d_rcol))) ||
      (!directed && (d_rrow_ptr || d_rcol))) {
    kadabra_free_graph(g);
    return fail(KADABRA_ERR_ARG, "missing or unexpected CSR arrays");
  }
  int32_t ends[2];
  if (cudaMemcpy(&ends[0], d_row_ptr, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(&ends[1], d_row_ptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess) {
    kadabra_free_graph(g);
    return fail(KADABRA_ERR_ARG, "row_ptr is not readable device memory");
  }
  if (ends[0] != 0 || ends[1] != m) {
    kadabra_free_graph(g);
    return fail(KADABRA_ERR_CSR, "row_ptr[0] must be 0 and row_ptr[n] must equal m");
  }
  if (directed) {
    if (cudaMemcpy(&ends[0], d_rrow_ptr, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(&ends[1], d_rrow_ptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        ends[0] != 0 || ends[1] != m) {
      kadabra_free_graph(g);
      return fail(KADABRA_ERR_CSR, "reverse row_ptr[0] must be 0 and row_ptr[n] must equal m");
    }
  }
  g->rp = const_cast<int32_t*>(d_row_ptr);
  g->ci = const_cast<int32_t*>(d_col);
  g->rrp = const_cast<int32_t*>(d_rrow_ptr);
  g->rci = const_cast<int32_t*>(d_rcol);
  kadabra_status st = finish_load(g);
  if (st != KADABRA_OK) {
    kadabra_free_graph(g);
    return st;
  }
  *out = g;
  return KADABRA_OK;
}

void kadabra_free_graph(kadabra_graph* g) {
  if (!g || g->is_view) return;
  cudaDeviceSynchronize();
  for (void* p : g->allocs) pool_free(p);
  if (g->owns_ws) ws_release(g->ws);
  delete g;
}

void kadabra_release_cached(void) {
  std::vector<Workspace*> all;
  {
    std::lock_guard<std::mutex> lk(g_ws_pool_mu);
    all.swap(g_ws_pool);
  }
  for (Workspace* w : all) {
    cudaSetDevice(w->device);
    delete w;
  }
  // the free memory of the graph allocations' pool, on the current device
  int dev = 0;
  cudaMemPool_t pool;
  if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    cudaDeviceSynchronize();
    cudaMemPoolTrimTo(pool, 0);
  }
}

kadabra_status kadabra_graph_set_flags(kadabra_graph* g, uint32_t flags) {
  if (!g) return fail(KADABRA_ERR_ARG, "graph is NULL");
  if (flags & ~(uint32_t)(KADABRA_FLAG_GLOBAL_TABLES | KADABRA_FLAG_MEDIUM_TABLES | KADABRA_FLAG_LARGE_SHARED_TABLES |
                          KADABRA_FLAG_WARP_TIER | KADABRA_FLAG_ASYNC_SCAN | KADABRA_FLAG_FRONTIER_SEGMENTS |
                          KADABRA_FLAG_COMPACT_TABLES))
    return fail(KADABRA_ERR_ARG, "unknown flag");
  g->flags = flags;
  return KADABRA_OK;
}

kadabra_status kadabra_graph_info(const kadabra_graph* g, int32_t* n, int64_t* m, int* directed, int64_t* vd) {
  if (!g) return fail(KADABRA_ERR_ARG, "graph is NULL");
  if (n) *n = g->n;
  if (m) *m = g->m;
  if (directed) *directed = g->directed;
  if (vd) *vd = g->vd;
  return KADABRA_OK;
}

kadabra_status kadabra_sample_batch(kadabra_graph* g, uint64_t seed, uint32_t domain, uint64_t first_idx,
                                    uint64_t count, uint32_t* d_counts, int64_t* d_totals, void* stream) {
  if (!g) return fail(KADABRA_ERR_ARG, "graph is NULL");
  if (count == 0) return KADABRA_OK;
  KTRY(ensure_workspace(g, count));
  SampleParams P = base_params(g);
  P.job0.seed = seed;
  P.job0.domain = domain;
  P.job0.first_idx = first_idx;
  P.job0.count = count;
  P.job0.counts = d_counts;
  P.job0.totals = reinterpret_cast<long long*>(d_totals);
  P.total_work = count;
  choose_screen(P, count, g->idle * (double)count);
  return launch_sampler(g->ws, P, as_stream(stream), tuned_variant(g, count));
}

kadabra_status kadabra_sample_batch_noalloc(int32_t n, int64_t m, const int32_t* d_row_ptr, const int32_t* d_col,
                                            int directed, const int32_t* d_rrow_ptr, const int32_t* d_rcol,
                                            uint64_t seed, uint32_t domain, uint64_t first_idx, uint64_t count,
                                            uint32_t* d_counts, int64_t* d_totals, void* stream) {
  if (n < 2 || n > (1 << 24) || m < 0 || m >= ((int64_t)1 << 31) || !d_row_ptr || (m > 0 && !d_col) || !d_counts)
    return fail(KADABRA_ERR_ARG, "bad graph or output arguments");
  if (directed && (!d_rrow_ptr || (m > 0 && !d_rcol)))
    return fail(KADABRA_ERR_ARG, "a directed graph needs the reverse CSR");
  if (count > NA_MAX_BATCH)
    return fail(KADABRA_ERR_CAPACITY, "kadabra_sample_batch_noalloc takes at most " +
                                          std::to_string(NA_MAX_BATCH) + " samples per call");
  if (count == 0) return KADABRA_OK;
  int dev = 0;
  KCK(cudaGetDevice(&dev));
  NoAllocDevice* d = nullptr;
  KTRY(noalloc_setup(dev, &d));
  cudaStream_t st = as_stream(stream);
  SampleParams P;
  std::memset(&P, 0, sizeof(P));
  P.job0.g.n = n;
  P.job0.g.m = m;
  P.job0.g.rp = d_row_ptr;
  P.job0.g.ci = d_col;
  P.job0.g.rrp = directed ? d_rrow_ptr : d_row_ptr;
  P.job0.g.rci = directed ? d_rcol : d_col;
  P.job0.seed = seed;
  P.job0.domain = domain;
  P.job0.first_idx = first_idx;
  P.job0.count = count;
  P.job0.counts = d_counts;
  P.job0.totals = reinterpret_cast<long long*>(d_totals);
  P.njobs = 1;
  P.total_work = count;
  P.ctr = reinterpret_cast<unsigned long long*>(d->scratch + NA_OFF_CTR);
  P.status = reinterpret_cast<int32_t*>(d->scratch + NA_OFF_STATUS);
  P.qb = reinterpret_cast<unsigned long long*>(d->scratch + NA_OFF_QB);
  P.ql = reinterpret_cast<unsigned long long*>(d->scratch + NA_OFF_QL);
  P.deferred_cap = NA_MAX_BATCH;
  P.pi_base = reinterpret_cast<PiEntry*>(d->scratch + NA_OFF_PI);
  P.pcap = NA_PCAP;
  P.med_base = d->scratch + NA_OFF_MED;  // tier M for the large-table launch's CTAs
  P.med_stride = NA_MED_STRIDE;
  P.med_hlog = NA_MED_HLOG;
  P.med_lcap = NA_MED_LCAP;
  P.tier_flags = 0;  // tiers S, B and M; samples beyond tier M end the call with KADABRA_ERR_CAPACITY
  KCK(cudaMemsetAsync(d->scratch, 0, NA_HEADER, st));
  k_sample<0><<<d->grid_s, 32 * NW_S, d->smem_s, st>>>(P);
  KCK(cudaGetLastError());
  k_sample<2><<<d->grid_b, 32 * NW_BIG, d->smem_b, st>>>(P);
  KCK(cudaGetLastError());
  unsigned long long left = 0;
  int32_t status = 0;
  KCK(cudaMemcpyAsync(&left, P.ctr + Q_SIZE_L, sizeof(left), cudaMemcpyDeviceToHost, st));
  KCK(cudaMemcpyAsync(&status, P.status, sizeof(status), cudaMemcpyDeviceToHost, st));
  KCK(cudaStreamSynchronize(st));
  if (status != 0)
    return fail((kadabra_status)status, status == KADABRA_ERR_SIGMA_OVERFLOW
                                            ? "a shortest-path count exceeded 2^64-1"
                                            : "the sampler reported a capacity or internal error");
  if (left != 0)
    return fail(KADABRA_ERR_CAPACITY, std::to_string(left) +
                                          " samples outgrew the tables of this call and were not counted; "
                                          "use kadabra_sample_batch for this graph");
  return KADABRA_OK;
}

kadabra_status kadabra_sync_status(kadabra_graph* g, void* stream) {
  if (!g) return fail(KADABRA_ERR_ARG, "graph is NULL");
  if (!g->ws->ready) {
    KCK(cudaStreamSynchronize(as_stream(stream)));
    return KADABRA_OK;
  }
  return read_status(g->ws, as_stream(stream));
}

kadabra_status kadabra_sample_paths(kadabra_graph* g, uint64_t seed, uint32_t domain, uint64_t first_idx,
                                    uint32_t count, int32_t* st_out, int32_t* path_len, int32_t* paths,
                                    int32_t max_len, int64_t* stats, int32_t* status) {
  if (!g || !st_out || !path_len || !status || (paths && max_len <= 0))
    return fail(KADABRA_ERR_ARG, "bad sample_paths arguments");
  if (count == 0) return KADABRA_OK;
  KTRY(ensure_workspace(g, count));
  int32_t *d_st = nullptr, *d_pl = nullptr, *d_paths = nullptr, *d_ss = nullptr;
  long long* d_stats = nullptr;
  kadabra_status rc = KADABRA_OK;
  auto cleanup = [&]() {
    cudaFree(d_st);
    cudaFree(d_pl);
    cudaFree(d_paths);
    cudaFree(d_ss);
    cudaFree(d_stats);
  };
  if (cudaMalloc(&d_st, sizeof(int32_t) * 2 * count) != cudaSuccess ||
      cudaMalloc(&d_pl, sizeof(int32_t) * count) != cudaSuccess ||
      cudaMalloc(&d_ss, sizeof(int32_t) * count) != cudaSuccess ||
      cudaMalloc(&d_stats, sizeof(long long) * KADABRA_NSTAT * count) != cudaSuccess ||
      (paths && cudaMalloc(&d_paths, sizeof(int32_t) * (size_t)count * max_len) != cudaSuccess)) {
    cleanup();
    return fail(KADABRA_ERR_OOM, "sample_paths buffers");
  }
  SampleParams P = base_params(g);
  P.job0.seed = seed;
  P.job0.domain = domain;
  P.job0.first_idx = first_idx;
  P.job0.count = count;
  P.total_work = count;
  choose_screen(P, count, g->idle * (double)count);
  P.st_out = d_st;
  P.path_len = d_pl;
  P.paths = d_paths;
  P.max_len = max_len;
  P.stats = d_stats;
  P.sstatus = d_ss;
  rc = launch_sampler(g->ws, P, 0);
  if (rc == KADABRA_OK) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) rc = fail(KADABRA_ERR_CUDA, std::string("sampler: ") + cudaGetErrorString(e));
  }
  if (rc == KADABRA_OK) {
    std::vector<long long> hs((size_t)KADABRA_NSTAT * count);
    if (cudaMemcpy(st_out, d_st, sizeof(int32_t) * 2 * count, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(path_len, d_pl, sizeof(int32_t) * count, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(status, d_ss, sizeof(int32_t) * count, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(hs.data(), d_stats, sizeof(long long) * hs.size(), cudaMemcpyDeviceToHost) != cudaSuccess ||
        (paths && cudaMemcpy(paths, d_paths, sizeof(int32_t) * (size_t)count * max_len, cudaMemcpyDeviceToHost) !=
                      cudaSuccess))
      rc = fail(KADABRA_ERR_CUDA, "sample_paths copy-back");
    else if (stats)
      for (size_t i = 0; i < hs.size(); ++i) stats[i] = hs[i];
  }
  cleanup();
  if (rc == KADABRA_OK) rc = read_status(g->ws, 0);
  return rc;
}

kadabra_status kadabra_philox(uint64_t seed, uint32_t domain, uint32_t j, uint64_t first_idx, uint32_t count,
                              uint32_t* out) {
  if (!out) return fail(KADABRA_ERR_ARG, "out is NULL");
  if (count == 0) return KADABRA_OK;
  uint4* d = nullptr;
  KCK(cudaMalloc(&d, sizeof(uint4) * count));
  k_philox<<<(count + 255) / 256, 256>>>(seed, domain, j, first_idx, count, d);
  cudaError_t e = cudaMemcpy(out, d, sizeof(uint4) * count, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return fail(KADABRA_ERR_CUDA, cudaGetErrorString(e));
  return KADABRA_OK;
}

kadabra_status kadabra_check(int64_t n, const uint32_t* counts, uint64_t tau, double omega, const double* ln_inv_dl,
                             const double* ln_inv_du, double lambda, double* max_f, double* max_g, int* stop) {
  if (n < 1 || !counts || !ln_inv_dl || !ln_inv_du || !max_f || !max_g || !stop || tau == 0)
    return fail(KADABRA_ERR_ARG, "bad check arguments");
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t o_u = up(sizeof(double) * (size_t)n), o_c = 2 * o_u, o_out = o_c + up(sizeof(uint32_t) * (size_t)n);
  void* base = nullptr;
  if (pool_alloc(&base, o_out + sizeof(CheckOut)) != KADABRA_OK) return fail(KADABRA_ERR_OOM, "check buffers");
  unsigned char* b = static_cast<unsigned char*>(base);
  double* dl = reinterpret_cast<double*>(b);
  double* du = reinterpret_cast<double*>(b + o_u);
  uint32_t* dc = reinterpret_cast<uint32_t*>(b + o_c);
  CheckOut* dout = reinterpret_cast<CheckOut*>(b + o_out);
  kadabra_status rc = KADABRA_OK;
  CheckOut h;
  cudaMemcpy(dc, counts, sizeof(uint32_t) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(dl, ln_inv_dl, sizeof(double) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(du, ln_inv_du, sizeof(double) * n, cudaMemcpyHostToDevice);
  cudaMemset(dout, 0, sizeof(CheckOut));
  {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(4 * (int64_t)sms, (n + 255) / 256));
    k_check<<<blocks, 256>>>(dc, dl, du, n, tau, omega, lambda, dout);
  }
  if (cudaMemcpy(&h, dout, sizeof(CheckOut), cudaMemcpyDeviceToHost) != cudaSuccess) {
    rc = fail(KADABRA_ERR_CUDA, std::string("check: ") + cudaGetErrorString(cudaGetLastError()));
    goto done;
  }
  std::memcpy(max_f, &h.max_f_bits, sizeof(double));
  std::memcpy(max_g, &h.max_g_bits, sizeof(double));
  *stop = h.fail ? 0 : 1;
done:
  pool_free(base);
  return rc;
}

kadabra_status kadabra_compute_delta(int64_t n, const uint32_t* count0, uint64_t alpha, double omega, double lambda,
                                     double delta, double eps, double* ln_inv_dl, double* ln_inv_du, double* C) {
  if (n < 1 || !count0 || !ln_inv_dl || !ln_inv_du || !C || alpha == 0)
    return fail(KADABRA_ERR_ARG, "bad compute_delta arguments");
  return compute_delta_host(n, count0, alpha, omega, lambda, delta, eps, ln_inv_dl, ln_inv_du, C);
}

kadabra_status kadabra_run(kadabra_graph* g, double lambda, double delta, int32_t k, uint64_t seed,
                           const kadabra_config* cfg_in, kadabra_result* out) {
  if (!g || !out) return fail(KADABRA_ERR_ARG, "graph or result is NULL");
  reset_result(out);
  kadabra_config cfg;
  kadabra_config_default(&cfg);
  if (cfg_in) cfg = *cfg_in;
  auto finish = [&](kadabra_status s) {
    out->status = s;
    return s;
  };
  if (k < 0 || k > TOPK_MAX) return finish(fail(KADABRA_ERR_ARG, "k must be in [0, 256]"));
  if (!(lambda > 0.0 && lambda < 1.0) || !(delta > 0.0 && delta < 1.0) || !(cfg.eps >= 0.0 && cfg.eps < 0.5))
    return finish(fail(KADABRA_ERR_ARG, "lambda and delta must be in (0,1), eps in [0,0.5)"));
  if (k > 0) return finish(run_topk(g, lambda, delta, k, seed, cfg, out));
  const int64_t vd = cfg.vd;
  return finish(run_graphs(g->ws, &g, 1, &lambda, &delta, &seed, &vd, cfg, out));
}


kadabra_status kadabra_load_batch(int32_t G, const int32_t* n, const int64_t* m, const int32_t* const* row_ptr,
                                  const int32_t* const* col, const int* directed, const int32_t* const* rrow_ptr,
                                  const int32_t* const* rcol, kadabra_batch** out) {
  if (!out) return fail(KADABRA_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (G < 1 || !n || !m || !row_ptr || !col) return fail(KADABRA_ERR_ARG, "bad batch arguments");
  if (G > KADABRA_MAX_BATCH_GRAPHS) return fail(KADABRA_ERR_ARG, "too many graphs in one batch");
  kadabra_batch* b = new kadabra_batch;
  b->G = G;
  auto bail = [&](kadabra_status st) {
    kadabra_free_batch(b);
    return st;
  };
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return bail(fail(KADABRA_ERR_CUDA, "no CUDA device"));
  // arena layout: per graph row_ptr, col[, rrow_ptr, rcol], each 256-byte aligned
  std::vector<size_t> off;
  size_t total = 0;
  auto place = [&](size_t bytes) {
    off.push_back(total);
    total += (bytes + 255) & ~size_t(255);
  };
  for (int32_t i = 0; i < G; ++i) {
    const bool dir = directed && directed[i];
    if (n[i] < 2 || n[i] > (1 << 24) || m[i] < 0 || m[i] >= ((int64_t)1 << 31) || !row_ptr[i] ||
        (m[i] > 0 && !col[i]) || (dir && (!rrow_ptr || !rcol || !rrow_ptr[i] || (m[i] > 0 && !rcol[i]))))
      return bail(fail(KADABRA_ERR_ARG, "bad arrays or sizes for graph " + std::to_string(i)));
    if (row_ptr[i][0] != 0 || row_ptr[i][n[i]] != m[i] || (dir && (rrow_ptr[i][0] != 0 || rrow_ptr[i][n[i]] != m[i])))
      return bail(fail(KADABRA_ERR_CSR, "row_ptr[0] must be 0 and row_ptr[n] must equal m (graph " +
                                            std::to_string(i) + ")"));
    place(sizeof(int32_t) * ((size_t)n[i] + 1));
    place(sizeof(int32_t) * (size_t)m[i]);
    if (dir) {
      place(sizeof(int32_t) * ((size_t)n[i] + 1));
      place(sizeof(int32_t) * (size_t)m[i]);
    }
  }
  {
    const cudaError_t e = cudaMalloc(&b->arena, total ? total : 16);
    if (e != cudaSuccess) return bail(fail(KADABRA_ERR_OOM, std::string("batch arena: ") + cudaGetErrorString(e)));
  }
  unsigned char* base = static_cast<unsigned char*>(b->arena);
  size_t k = 0;
  int32_t max_n = 0;
  int64_t max_m = 0;
  for (int32_t i = 0; i < G; ++i) {
    const bool dir = directed && directed[i];
    kadabra_graph* g = new kadabra_graph;
    b->views.push_back(g);
    g->n = n[i];
    g->m = m[i];
    g->directed = dir ? 1 : 0;
    g->device = dev;
    g->num_sms = sms;
    g->ws = &b->ws;
    g->is_view = true;
    const size_t rb = sizeof(int32_t) * ((size_t)n[i] + 1), cb = sizeof(int32_t) * (size_t)m[i];
    g->rp = reinterpret_cast<int32_t*>(base + off[k++]);
    g->ci = reinterpret_cast<int32_t*>(base + off[k++]);
    if (cudaMemcpy(g->rp, row_ptr[i], rb, cudaMemcpyHostToDevice) != cudaSuccess ||
        (m[i] > 0 && cudaMemcpy(g->ci, col[i], cb, cudaMemcpyHostToDevice) != cudaSuccess))
      return bail(fail(KADABRA_ERR_CUDA, "batch CSR upload failed"));
    if (dir) {
      g->rrp = reinterpret_cast<int32_t*>(base + off[k++]);
      g->rci = reinterpret_cast<int32_t*>(base + off[k++]);
      if (cudaMemcpy(g->rrp, rrow_ptr[i], rb, cudaMemcpyHostToDevice) != cudaSuccess ||
          (m[i] > 0 && cudaMemcpy(g->rci, rcol[i], cb, cudaMemcpyHostToDevice) != cudaSuccess))
        return bail(fail(KADABRA_ERR_CUDA, "batch reverse CSR upload failed"));
    }
    const kadabra_status st = finish_load(g);
    if (st != KADABRA_OK) return bail(fail(st, std::string(kadabra_last_error()) + " (graph " + std::to_string(i) + ")"));
    max_n = std::max(max_n, n[i]);
    max_m = std::max(max_m, m[i]);
  }
  b->ws.device = dev;
  b->ws.num_sms = sms;
  b->ws.max_n = max_n;
  b->ws.max_m = max_m;
  *out = b;
  return KADABRA_OK;
}

void kadabra_free_batch(kadabra_batch* b) {
  if (!b) return;
  cudaDeviceSynchronize();
  for (kadabra_graph* g : b->views) {
    for (void* p : g->allocs) pool_free(p);
    delete g;  // also releases its loop graph
  }
  if (b->arena) cudaFree(b->arena);
  delete b;
}

kadabra_status kadabra_batch_graph(kadabra_batch* b, int32_t i, kadabra_graph** view) {
  if (!b || !view || i < 0 || i >= b->G) return fail(KADABRA_ERR_ARG, "bad batch graph index");
  *view = b->views[i];
  return KADABRA_OK;
}

kadabra_status kadabra_run_batch(kadabra_batch* b, const double* lambda, const double* delta, const uint64_t* seed,
                                 const kadabra_config* cfg_in, kadabra_result* out) {
  if (!b || !lambda || !delta || !seed || !out) return fail(KADABRA_ERR_ARG, "bad batch run arguments");
  kadabra_config cfg;
  kadabra_config_default(&cfg);
  if (cfg_in) cfg = *cfg_in;
  if (cfg.vd != 0) return fail(KADABRA_ERR_ARG, "a batch uses each graph's own VD bound (cfg->vd must be 0)");
  if (!(cfg.eps >= 0.0 && cfg.eps < 0.5)) return fail(KADABRA_ERR_ARG, "eps must be in [0, 0.5)");
  for (int i = 0; i < b->G; ++i) {
    reset_result(&out[i]);
    if (!(lambda[i] > 0.0 && lambda[i] < 1.0) || !(delta[i] > 0.0 && delta[i] < 1.0))
      return fail(KADABRA_ERR_ARG, "lambda and delta must be in (0,1) (graph " + std::to_string(i) + ")");
  }
  const kadabra_status s = run_graphs(&b->ws, b->views.data(), b->G, lambda, delta, seed, nullptr, cfg, out);
  for (int i = 0; i < b->G; ++i) out[i].status = s;
  return s;
}

}  // extern "C"
