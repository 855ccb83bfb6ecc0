// Standalone ranking of large live sets (the scan of Sec. IV-D, eqs. pipe and
// scan, generalised from one argmax to a top-k) and the TIDE fill of
// Sec. III-C (eqs. budget, promote, demote) over the same ranking.
//
// Every record gets a packed comparable key ck = score40 << 24 | ~index24:
// unsigned order on ck is the ranking order (larger score first, ties to
// the smaller index).  Three ordered selections are needed per live set:
//   V  victims: unpinned resident records, largest ck first (top-k);
//   D  fast-tier demotion candidates: unpinned fast-tier records, largest first;
//   P  HBM promotion candidates: unpinned HBM records, smallest ck first.
//
// One cooperative, persistent kernel does a whole call.  Each set owns a
// group of CTAs (in proportion to its records; with more sets than CTAs,
// each CTA takes whole sets in turn).  Per set, inside the group:
//   sample   up to 63 CTAs gather a jittered stratified sample and add it to a
//            4,096-bin histogram per list in global memory (bins monotone in
//            the list value).  Once every sampling CTA's counts are in, each
//            CTA of the group cuts the histograms at the lists'
//            sample ranks itself: per-list thresholds and per-turn thresholds
//            on the gap average (the score is monotone in the gap for a fixed
//            turn, so the streaming test needs no division).  Meanwhile every
//            CTA's producer warp already streams its first tiles into shared
//            memory.
//   filter   the group's CTAs take the set's tiles from a shared counter;
//            every record is read once (8 B: gap average, turn, flags, tier)
//            by TMA bulk copies and tested against the thresholds, and the
//            exact values of the records that pass are appended per list to
//            the CTA's own region, which moves into the set's list when the
//            CTA is done.
//            A set of at most 4,096 records streams nothing: three CTAs collect
//            one list's values each, from every eligible record.
//   finish   the last three CTAs of the group to finish streaming take one
//            list each: cuts into 256 buckets below the common prefix narrow the
//            candidates to few beyond the first M, which are sorted and the
//            first M kept; a list whose candidates overflowed or fell short is
//            re-selected exactly by streaming the set.  The last list's CTA runs the fill, 256
//            items at a time, and writes the outputs.
// The work words and sample histograms lie in one of two blocks: calls on a
// stream alternate between them, and each call zeroes what the one before it
// used.  (A captured call has memory of its own, cleared by a node before it.)
// Every wait on another CTA or on a copy is bounded: a wait that gives up
// records UNISON_ERR_TIMEOUT in the set's status word and the CTA carries on
// to the end of the kernel.  A cooperative launch keeps every CTA of the grid
// resident, so the waits on other CTAs end.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"
#include "profile.cuh"
#ifdef UNISON_DEBUG_HOOKS
#include "../../include/unison_debug.h"
#endif

using namespace unison;

namespace {

constexpr int kLists = 3;  // 0 = V, 1 = D, 2 = P
constexpr uint32_t kSample = 16384;      // largest set whose candidate lists have room for every record
constexpr uint32_t kCandCap = 65536;     // candidate slots per list and set
constexpr uint32_t kMaxGroup = 512;       // CTAs of one launch, at most (152 SMs x 3)
constexpr uint32_t kMaxSel = 4096;       // largest k and max_moves
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kSampleCtas = 63;     // sampling CTAs per set, at most
constexpr uint32_t kSampleQ = 4;         // samples per consumer thread
constexpr uint32_t kLaunchSamples = 131072;  // samples per launch, about,
constexpr uint32_t kSmallSample = 4096;  // the shortest lists, where this many samples give them
constexpr uint32_t kSetSamples = 16384;      // or this many a set
constexpr uint32_t kBins = 4096;         // histogram bins per list
constexpr uint32_t kEndTile = 0xFFFFFFFFu;

// CTA layout: 8 consumer warps and one producer warp.  A tile is 4,096
// records; two tiles are in flight per CTA.
constexpr int kStages = 2;
constexpr uint32_t kRec = 16;                          // records per consumer thread per tile
constexpr uint32_t kConsumers = 256;                   // consumer threads
constexpr uint32_t kBigTile = kConsumers * kRec;       // 4096 records per tile
constexpr uint32_t kGroups = kRec / 4;                 // groups of four records per thread
constexpr uint32_t kGroupStride = kConsumers * 4;      // records between a thread's groups
constexpr uint32_t kWarpBuf = 128;                     // flagged records a warp tests per pass
constexpr uint32_t kCtaThreads = kConsumers + 32;
constexpr uint32_t kPerCtaSamples = kConsumers * kSampleQ;
constexpr uint32_t kIpt = kMaxSel / kConsumers;        // fill items per consumer thread
static_assert(kConsumers >= kLutN * 5, "one consumer thread per bound-table entry");
static_assert(kMaxSel % kConsumers == 0 && kIpt % 4 == 0, "fill layout");
static_assert(kBins == 16 * kConsumers, "histogram cut layout");
constexpr uint32_t kMaxSample = kSampleCtas * kPerCtaSamples;
static_assert(kMaxSample < 65536, "16-bit counts");

struct __align__(128) FilterStage {
  uint32_t gap[kBigTile];
  uint16_t turn[kBigTile];
  uint8_t flags[kBigTile];
  uint8_t tier[kBigTile];
};
constexpr size_t kDynSmem = sizeof(FilterStage) * kStages;  // 64 KB, reused by the finish
// the merge kernel's area: values and sizes, and the bucket sort's copies of both
constexpr size_t kMergeSmem = 3 * kMaxSel * sizeof(uint64_t);  // 96 KB
constexpr uint32_t kDynWords = kDynSmem / 8;                // 8192 u64
constexpr uint32_t kSmemCand = kDynWords - kMaxSel;          // candidates copied to shared memory
static_assert(kSmemCand >= kMaxSel && kDynWords >= 2 * kMaxSel, "finish layout");

// Every wait is bounded in time (%globaltimer, ns).  A wait on another CTA
// (thresholds, the group's last arrival) gives up after kWaitNs; a wait on
// this CTA's own pipeline (a tile's copies, a stage's release, the finish's
// copy) after kPipeNs, longer, so that a producer never gives up while its
// consumers still wait on another CTA.
// a suspended waiter re-checks its bound at least this often
constexpr uint32_t kWaitHintNs = 20000;
#ifdef UNISON_DEBUG_HOOKS
constexpr uint64_t kWaitNs = 2000000ull;     // 2 ms: the tests make one run out
constexpr uint64_t kPipeNs = 50000000ull;    // 50 ms: well above any ordinary copy
__device__ int g_hook_flag_set = -1;   // set whose threshold wait first waits on a flag nothing sets
__device__ int g_hook_mbar_set = -1;   // set whose first tile wait first waits on a barrier nothing arrives at
#else
constexpr uint64_t kWaitNs = 2000000000ull;  // 2 s
constexpr uint64_t kPipeNs = 4000000000ull;  // 4 s
#endif

// Each group of words that many CTAs poll or update at once has a 128-byte
// line of its own: a flag polled by every CTA of a group and counters taken
// by atomics in the same line would serialise at one L2 slice.
struct alignas(128) RankWork {
  // the streaming counters (atomics while the tiles stream)
  unsigned int cand[kLists];    // candidates emitted per list
  unsigned int next_tile;       // the group's tile counter
  unsigned int pad0[28];
  // the sample's reads done (polled by the producers)
  unsigned int gathered;        // sampling CTAs whose sample has arrived
  unsigned int pad1[31];
  // the sample's counts in the histogram (polled by every CTA of the group)
  unsigned int sample_ticket;   // sampling CTAs whose counts have landed
  unsigned int pad2[31];
  // the finish
  unsigned int done_ctas;       // CTAs of the group done streaming
  unsigned int list_ticket;     // lists finished
  unsigned int got[kLists];     // selected entries per list
  unsigned int status;          // UNISON_ERR_TIMEOUT if a bounded wait gave up
  unsigned int dummy;           // never written: the debug hook waits on it
  unsigned int pad3[25];
};
static_assert(sizeof(RankWork) == 512, "four lines");

// Per-turn tables of one (sigma, P_Z) pair, shared by the sets that use it.
struct RankTab {
  uint64_t t2v[kLutN];   // eq. (t2) per turn index
  uint64_t mgv[kLutN];   // division magic of sigma per turn index
  uint32_t sigma[kLutN];
};

struct RankSet {
  const uint32_t *gap;
  const uint16_t *turn;
  const uint32_t *kv;
  const uint8_t *tier;
  const uint8_t *flags;
  uint32_t n, k, max_moves, kvb;
  uint64_t budget, free_s, free_h;
  uint32_t *victims, *promote, *demote, *counts;
  uint64_t *moved, *keys;
  const RankTab *tab;
  uint32_t ntiles;
  uint32_t cta0, nctas;          // the group: CTAs [cta0, cta0 + nctas)
  uint32_t ns, nruns;            // sample size, its runs of 8
  uint64_t sstep;                // stratum width n / nruns in 16.16 fixed point
  uint32_t sctas;                // sampling CTAs (the group's first sctas)
  uint32_t act;                  // active lists (bit L)
  uint32_t rL[kLists];           // sample rank of each list's threshold
  uint32_t ccap;                 // candidate slots per list (kCandCap, or n rounded up for a set too small to sample)
  uint32_t off;                  // index of record 0 in the whole set (a shard's slice), else 0
  uint32_t direct;               // small set, one CTA a list: each collects its list's values itself
  unsigned char *cands;          // a shard's candidate lists (unison_rank_shard), else null
  // scratch (per set)
  RankWork *work;
  uint64_t *cand;    // [3][ccap] the set's candidate lists (a global counter each)
  uint64_t *creg;    // [3][nctas][cr] each CTA's candidates while it streams
  uint32_t cr;       // region size
  uint64_t *sorted;  // [3][kMaxSel]
  uint32_t *ssz;     // [3][kMaxSel] KV tokens of the sorted entries (D and P)
  uint16_t *shist;      // [3][kBins] sample histogram (zero between calls)
};

// A shard's candidate lists (unison_rank_shard): a 64-byte header, then its
// V, D and P lists of (list value, KV tokens) in ranking order.
struct CandHeader {
  uint32_t count[kLists];
  uint32_t status;
  uint32_t n, off, k, max_moves;
  uint32_t pad[8];
};
static_assert(sizeof(CandHeader) == 64, "candidate header");
struct CandEntry {
  uint64_t v;
  uint32_t kv, pad;
};
constexpr uint32_t kMaxShards = 1024;
__host__ __device__ __forceinline__ size_t cand_bytes(uint32_t k, uint32_t m) {
  return sizeof(CandHeader) + sizeof(CandEntry) * ((size_t)k + 2ull * m);
}
__host__ __device__ __forceinline__ size_t cand_list_off(uint32_t k, uint32_t m, int L) {
  return sizeof(CandHeader) + sizeof(CandEntry) * (L == 0 ? 0ull : (L == 1 ? (size_t)k : (size_t)k + m));
}

// ---------------------------------------------------------------- keys ----
__device__ __forceinline__ uint64_t score_of(uint32_t g, uint32_t t, bool done, const uint64_t *t2,
                                             const uint64_t *magic) {
  if (done) return ~0ull;
  return __umul64hi((uint64_t)g * kLambda, magic[t]) + t2[t];
}

__device__ __forceinline__ uint64_t ck_of(uint64_t score, uint32_t idx) {
  const uint64_t k40 = score == ~0ull ? kKeyMax40 : score;
  return (k40 << 24) | ((~idx) & kIdMask);
}

__device__ __forceinline__ uint32_t elig_mask(uint8_t fl, uint8_t tr) {
  if (fl & 1) return 0;  // pinned: never ranked for eviction or migration
  uint32_t m = 0;
  if (tr == 1) m = 1u | 2u;
  if (tr == 2) m = 1u | 4u;
  return m;
}

// Smallest gap average whose score reaches K at turn index t.
__device__ __forceinline__ uint32_t g_at_least(uint64_t K, uint32_t sigma, uint64_t t2) {
  if (K <= t2) return 0;
  const uint64_t m = K - t2;
  const uint64_t g = (m * sigma + kLambda - 1) / kLambda;
  return g > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)g;
}

__device__ __forceinline__ uint64_t list_val(uint64_t ck, int L) { return L == 2 ? ~ck : ck; }

// ------------------------------------------------- barriers and copies ----
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same test, but a thread whose phase has not completed is suspended
// until it does or about hint_ns pass: a waiting thread then takes no issue
// slots from the warps that work.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t *bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait on an mbarrier phase; false when the bound ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, uint64_t limit_ns = kPipeNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = now_ns();
  while (now_ns() - t0 < limit_ns)
    if (mbar_try_wait_sleep(bar, parity, kWaitHintNs)) return true;
  return false;
}

// Barrier 1 over the consumer warps only (the producer warp never joins it).
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kConsumers) : "memory"); }
// Barrier 1 with an OR reduction of p over the consumer threads.
__device__ __forceinline__ bool consumers_sync_or(bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred pi, po;\n setp.ne.u32 pi, %1, 0;\n bar.red.or.pred po, 1, %2, pi;\n selp.u32 %0, 1, 0, po;\n}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(kConsumers)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void set_status(const RankSet &S, int code) { atomicExch(&S.work->status, (unsigned int)code); }

// Consumer thread 0 waits (bounded) until *word reaches target, then the
// consumers proceed with the other CTAs' writes visible.  False (for every
// consumer thread alike) on timeout.
__device__ bool wait_word(const RankSet &S, const unsigned int *word, unsigned int target) {
  __shared__ unsigned int ok;
  if (threadIdx.x == 0) {
    const uint64_t t0 = now_ns();
    uint32_t nap = 32;  // backoff: a word polled by many CTAs at once
    while (*(volatile const unsigned int *)word < target && now_ns() - t0 < kWaitNs) {
      __nanosleep(nap);
      nap = min(nap * 2, 256u);
    }
    ok = *(volatile const unsigned int *)word >= target;
    if (!ok) set_status(S, UNISON_ERR_TIMEOUT);
    __threadfence();
  }
  consumers_sync();
  return ok != 0;
}

// Consumer thread 0 waits (bounded) for an mbarrier phase; the others take
// its verdict, so every consumer thread takes the same path, then observe the
// completed phase themselves (one poll: it has completed) before they read
// what it guards.  False (for all) on timeout.
__device__ bool wait_phase_uniform(const RankSet &S, uint64_t *bar, uint32_t parity, uint64_t limit_ns = kPipeNs) {
  __shared__ unsigned int ok;
  if (threadIdx.x == 0) {
    ok = mbar_wait_bounded(bar, parity, limit_ns) ? 1u : 0u;
    if (!ok) set_status(S, UNISON_ERR_TIMEOUT);
  }
  consumers_sync();
  if (!ok) return false;
  mbar_try_wait(bar, parity);
  return true;
}

// ---------------------------------------------------- shared scratch ----
// The filter's bound table and flagged-record buffers, or the finish's
// radix-select scratch (never in use at the same time).
struct FilterScratch {
  uint2 ftab[kLutN * 5];
  uint16_t wbuf[kConsumers / 32][kWarpBuf];
};
struct SelectScratch {
  unsigned long long split[256];  // the splitter sort's splitters
  unsigned int hist[256];
  unsigned int off[256];  // the bucket sorts' bucket starts
  unsigned int pick[2];
  unsigned long long bcast[2];
  unsigned int cnt;
  unsigned int wtot[kConsumers / 32];
  unsigned long long wsq[kConsumers / 32];
};
union CtaScratch {
  FilterScratch f;
  SelectScratch s;
};

// ---------------------------------------------------- histogram bins ----
// 32-bit order-preserving summary of a list value v = key40 << 24 | low24:
// key40 >> 9 below the maximal key, and 2^31 | low24 on it (completed
// sessions all carry the maximal key, so only their index orders them).
// summary(a) <= summary(b) whenever a <= b; summary_floor(f) is the smallest
// list value whose summary is f.
__device__ __forceinline__ uint32_t summary_of(uint64_t v) {
  const uint64_t K = v >> 24;
  return K == kKeyMax40 ? (0x80000000u | (uint32_t)(v & kIdMask)) : (uint32_t)(K >> 9);
}
__device__ __forceinline__ uint64_t summary_floor(uint32_t f) {
  return (f & 0x80000000u) ? ((kKeyMax40 << 24) | (f & kIdMask)) : ((uint64_t)f << 33);
}
// Bin of a summary, monotone: summaries below 2^31 by octave (the position
// e of the leading one) and the 6 bits after it (bins 0..1983, a 1/64-octave
// resolution; below 64 one bin per value); summaries at or above 2^31 (the
// maximal key) by index, 8,192 indices a bin (bins 2048..4095).
// bin_floor(b) is the smallest summary in bin b.
__device__ __forceinline__ uint32_t bin_of(uint32_t f) {
  if (f & 0x80000000u) return 2048u + ((f & kIdMask) >> 13);
  if (f < 64u) return (f ? (uint32_t)(31 - __clz(f)) : 0u) * 64u + f;
  const uint32_t e = 31 - __clz(f);
  return e * 64u + ((f >> (e - 6)) & 63u);
}
__device__ __forceinline__ uint32_t bin_floor(uint32_t b) {
  if (b >= 2048u) return 0x80000000u | ((b - 2048u) << 13);
  const uint32_t e = b / 64u, m = b % 64u;
  return e < 6u ? m : (64u + m) << (e - 6u);
}
// The same per list.  P's values fall as keys rise, and its wanted ones are the
// smallest keys, which the octaves from the top would leave in one bin: its
// summaries are binned by their distance from the top, i.e. by octaves of the
// key.  (Key 0 has the flagged summaries, by index.)
__device__ __forceinline__ uint32_t list_bin(uint32_t f, int L) {
  return L != 2 || (f & 0x80000000u) ? bin_of(f) : 1983u - bin_of(0x7FFFFFFFu - f);
}
__device__ __forceinline__ uint32_t list_bin_floor(uint32_t b, int L) {
  return L != 2 || b >= 2048u ? bin_floor(b) : 0x7FFFFFFFu - (bin_floor(1984u - b) - 1u);
}

// Value with the given rank (1 = largest) among get(0..n-1), 64-bit values,
// MSB-first over the bytes where the values differ.  Consumer threads only;
// hist must be zero on entry and is zero on return.
template <typename Get>
__device__ uint64_t block_select_rank(Get get, uint32_t n, uint32_t rank, SelectScratch &ss) {
  unsigned long long a = ~0ull, o = 0ull;
  for (uint32_t i = threadIdx.x; i < n; i += kConsumers) {
    const uint64_t v = get(i);
    a &= v;
    o |= v;
  }
  for (int s = 16; s; s >>= 1) {
    a &= __shfl_xor_sync(kFull, a, s);
    o |= __shfl_xor_sync(kFull, o, s);
  }
  if (threadIdx.x == 0) {
    ss.bcast[0] = ~0ull;
    ss.bcast[1] = 0ull;
  }
  consumers_sync();
  if ((threadIdx.x & 31) == 0) {
    atomicAnd(&ss.bcast[0], a);
    atomicOr(&ss.bcast[1], o);
  }
  consumers_sync();
  const uint64_t same = ~(ss.bcast[0] ^ ss.bcast[1]);  // bits equal in every value
  const uint64_t common = ss.bcast[0] & same;
  int top = 7;
  while (top > 0 && ((same >> (8 * top)) & 0xFF) == 0xFF) top--;
  uint64_t mask = top < 7 ? (~0ull << (8 * (top + 1))) : 0ull;
  uint64_t prefix = common & mask;
  uint32_t need = rank;
  unsigned int *hist = ss.hist;
  for (int b = top; b >= 0; b--) {
    for (uint32_t base = 0; base < n; base += kConsumers) {
      const uint32_t i = base + threadIdx.x;
      bool in = false;
      uint32_t d = 0;
      if (i < n) {
        const uint64_t v = get(i);
        in = (v & mask) == prefix;
        d = (uint32_t)(v >> (8 * b)) & 0xFF;
      }
      const unsigned act = __ballot_sync(kFull, in);
      if (in) {
        const unsigned grp = __match_any_sync(act, d);
        if ((__ffs(grp) - 1) == (int)(threadIdx.x & 31)) atomicAdd(&hist[d], (unsigned)__popc(grp));
      }
    }
    consumers_sync();
    if (threadIdx.x < 32) {
      const int l = threadIdx.x;
      uint32_t c[8], tot = 0;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        c[q] = hist[255 - 8 * l - q];
        hist[255 - 8 * l - q] = 0;
        tot += c[q];
      }
      uint32_t incl = tot;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, s);
        if (l >= s) incl += y;
      }
      const uint32_t excl = incl - tot;
      const unsigned hit = __ballot_sync(kFull, excl < need && incl >= need);
      if (l == __ffs(hit) - 1) {
        uint32_t cum = excl;
#pragma unroll
        for (int q = 0; q < 8; q++) {
          if (cum + c[q] >= need) {
            ss.pick[0] = 255 - 8 * l - q;
            ss.pick[1] = need - cum;
            cum = 0xFFFFFFFFu;
            break;
          }
          cum += c[q];
        }
      }
    }
    consumers_sync();
    prefix |= (uint64_t)ss.pick[0] << (8 * b);
    mask |= 0xFFull << (8 * b);
    need = ss.pick[1];
  }
  consumers_sync();  // pick and bcast free for the caller
  return prefix;
}

// Cut of the kLists histograms hist[L * kBins ..] of 16-bit counts at once
// (their loads in flight together): the bin holding the need[L]-th value from
// the top, -1 for need[L] == 0 or too few values.  Every CTA of a group reads
// them, 24 KB from L2 (with 32-bit counts, 48 KB, one set of 2^20 records took
// 2 us more and 33 of them 4.5 us).
__device__ void hist_cut3(const uint16_t *hist, const uint32_t (&need)[kLists], int (&cut)[kLists]) {
  __shared__ unsigned int wtot[kLists][kConsumers / 32];
  __shared__ int scut[kLists];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lo = kBins - 16 * (tid + 1);
  uint32_t c[kLists][16], tot[kLists], ex[kLists];
#pragma unroll
  for (int L = 0; L < kLists; L++) {
    const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + L * kBins + lo);
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const uint4 x = __ldcg(h4 + q);
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int u = 0; u < 4; u++) {
        c[L][8 * q + 2 * u] = w[u] & 0xFFFFu;
        c[L][8 * q + 2 * u + 1] = w[u] >> 16;
      }
    }
  }
#pragma unroll
  for (int L = 0; L < kLists; L++) {
    tot[L] = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) tot[L] += c[L][q];
    uint32_t incl = tot[L];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if ((int)lane >= o) incl += y;
    }
    if (lane == 31) wtot[L][warp] = incl;
    ex[L] = incl - tot[L];
  }
  if (tid < kLists) scut[tid] = -1;
  consumers_sync();
#pragma unroll
  for (int L = 0; L < kLists; L++) {
    for (uint32_t w = 0; w < warp; w++) ex[L] += wtot[L][w];
    if (need[L] && ex[L] < need[L] && ex[L] + tot[L] >= need[L]) {
      uint32_t acc = ex[L];
      for (int q = 15; q >= 0; q--) {
        if (acc + c[L][q] >= need[L]) {
          scut[L] = (int)(lo + q);
          break;
        }
        acc += c[L][q];
      }
    }
  }
  consumers_sync();
#pragma unroll
  for (int L = 0; L < kLists; L++) cut[L] = scut[L];
}

static_assert(kConsumers == 256, "one bucket per consumer thread");  // the narrowing and the sorts below

// Values beyond the M wanted ones that a selection leaves to the sort: another
// step of narrow() costs about what sorting twice as many does.
__device__ __forceinline__ uint32_t slack(uint32_t M) { return max(M, 256u); }

// One step towards the rank-M value of a list of distinct values.  The values
// in [t, t + 2^sh) (all of them for sh == 64) hold it as their need-th
// largest: 256 buckets on the 8 bits below their common prefix, and [t, t +
// 2^sh) becomes the bucket that holds it.  Returns the values in that bucket;
// need becomes the rank in it.  each(fn) calls fn(v) once for every value,
// spread over the consumer threads in any order.  Bound by latency: two passes
// over the values and seven block barriers, about 2.5 us over 4,096 values in
// shared memory; over 13,000 in global memory 17 us with eight loads a thread
// in flight (26 us with one).
template <class Each>
__device__ uint32_t narrow(Each each, uint64_t &t, int &sh, uint32_t &need, SelectScratch &ss) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t lo = t;
  const int s0 = sh;
  auto in = [&](uint64_t v) { return s0 >= 64 || v >> s0 == lo >> s0; };
  uint64_t an = ~0ull, orv = 0ull;
  each([&](uint64_t v) {
    if (in(v)) {
      an &= v;
      orv |= v;
    }
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    an &= __shfl_xor_sync(kFull, an, o);
    orv |= __shfl_xor_sync(kFull, orv, o);
  }
  if (tid == 0) {
    ss.bcast[0] = ~0ull;
    ss.bcast[1] = 0ull;
  }
  ss.hist[tid] = 0;
  consumers_sync();
  if (lane == 0) {
    atomicAnd(&ss.bcast[0], an);
    atomicOr(&ss.bcast[1], orv);
  }
  consumers_sync();
  const uint64_t vary = ss.bcast[0] ^ ss.bcast[1], common = ss.bcast[0];
  const int top = vary ? 64 - __clzll((long long)vary) : 0;
  sh = top > 8 ? top - 8 : 0;
  const int s1 = sh;
  each([&](uint64_t v) {
    if (in(v)) atomicAdd(&ss.hist[(uint32_t)(v >> s1) & 255u], 1u);
  });
  consumers_sync();
  // thread i owns bucket 255 - i: counts from the top
  const uint32_t own = ss.hist[255 - tid];
  uint32_t incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31) ss.wtot[warp] = incl;
  consumers_sync();
  for (uint32_t w = 0; w < warp; w++) incl += ss.wtot[w];
  if (incl - own < need && incl >= need) {
    ss.pick[0] = 255 - tid;
    ss.pick[1] = incl - own;
    ss.cnt = own;
  }
  consumers_sync();
  // the common prefix above the 8 bits (none varies there), then the bucket
  const uint64_t pre = s1 >= 56 ? 0ull : common >> (s1 + 8) << (s1 + 8);
  t = pre | (uint64_t)ss.pick[0] << s1;
  need -= ss.pick[1];
  const uint32_t n = ss.cnt;
  consumers_sync();  // pick, hist and bcast free for the caller
  return n;
}

// Sort, descending, of the distinct values a[0..n) by bucket: the 8 bits
// below the values' common prefix name 256 buckets, a counting pass places
// each value in its bucket's range (buckets in descending order, in tmp),
// and each value's place within its bucket is the count of the bucket's
// values above it.  pay[] (when given) moves along, through tmp_pay.  Costs
// the sum over buckets of size^2 comparisons; declines (false, a and pay
// unchanged) when that sum is large, i.e. the values crowd into few buckets.
__device__ bool bucket_sort_desc(uint64_t *a, uint32_t n, uint64_t *tmp, SelectScratch &ss, uint32_t *pay = nullptr,
                                 uint32_t *tmp_pay = nullptr) {
  if (n <= 1) return true;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint64_t an = ~0ull, orv = 0ull;
  for (uint32_t i = tid; i < n; i += kConsumers) {
    const uint64_t v = a[i];
    an &= v;
    orv |= v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    an &= __shfl_xor_sync(kFull, an, o);
    orv |= __shfl_xor_sync(kFull, orv, o);
  }
  if (tid == 0) {
    ss.bcast[0] = ~0ull;
    ss.bcast[1] = 0ull;
  }
  ss.hist[tid] = 0;
  consumers_sync();
  if (lane == 0) {
    atomicAnd(&ss.bcast[0], an);
    atomicOr(&ss.bcast[1], orv);
  }
  consumers_sync();
  const uint64_t vary = ss.bcast[0] ^ ss.bcast[1];  // non-zero: the values are distinct
  const int top = 64 - __clzll((long long)vary);
  const int sh = top > 8 ? top - 8 : 0;
  for (uint32_t i = tid; i < n; i += kConsumers) atomicAdd(&ss.hist[(uint32_t)(a[i] >> sh) & 255u], 1u);
  consumers_sync();
  // thread t owns bucket 255 - t: exclusive offsets in descending bucket order
  const uint32_t c = ss.hist[255 - tid];
  uint32_t incl = c;
  uint64_t sq = (uint64_t)c * c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if ((int)lane >= o) incl += y;
    sq += __shfl_xor_sync(kFull, sq, o);
  }
  if (lane == 31) ss.wtot[warp] = incl;
  if (lane == 0) ss.wsq[warp] = sq;
  consumers_sync();
  uint32_t ex = incl - c;
  uint64_t sqt = 0;
  for (uint32_t w = 0; w < kConsumers / 32; w++) {
    if (w < warp) ex += ss.wtot[w];
    sqt += ss.wsq[w];
  }
  ss.off[255 - tid] = ex;
  consumers_sync();  // every count read before the cursors overwrite them
  if (sqt > 32ull * n + 8192ull) return false;  // the same verdict in every thread
  ss.hist[255 - tid] = ex;
  consumers_sync();
  for (uint32_t i = tid; i < n; i += kConsumers) {
    const uint64_t v = a[i];
    const uint32_t p = atomicAdd(&ss.hist[(uint32_t)(v >> sh) & 255u], 1u);
    tmp[p] = v;
    if (pay) tmp_pay[p] = pay[i];
  }
  consumers_sync();
  for (uint32_t p = tid; p < n; p += kConsumers) {
    const uint64_t v = tmp[p];
    const uint32_t b = (uint32_t)(v >> sh) & 255u, lo = ss.off[b], hi = ss.hist[b];
    uint32_t r = 0;
    for (uint32_t q = lo; q < hi; q++) r += tmp[q] > v ? 1u : 0u;
    a[lo + r] = v;
    if (pay) pay[lo + r] = tmp_pay[p];
  }
  consumers_sync();
  return true;
}

// Sort, descending, of n <= kCountSort distinct values: each value's place is
// the count of those above it.
constexpr uint32_t kCountSort = 2 * kConsumers;
__device__ void count_sort_desc(uint64_t *a, uint32_t n, uint32_t *pay) {
  const uint32_t tid = threadIdx.x, i1 = tid + kConsumers;
  const uint64_t v0 = tid < n ? a[tid] : 0ull, v1 = i1 < n ? a[i1] : 0ull;
  const uint32_t p0 = pay && tid < n ? pay[tid] : 0u, p1 = pay && i1 < n ? pay[i1] : 0u;
  uint32_t r0 = 0, r1 = 0;
#pragma unroll 8
  for (uint32_t q = 0; q < n; q++) {
    const uint64_t x = a[q];
    r0 += x > v0 ? 1u : 0u;
    r1 += x > v1 ? 1u : 0u;
  }
  consumers_sync();
  if (tid < n) {
    a[r0] = v0;
    if (pay) pay[r0] = p0;
  }
  if (i1 < n) {
    a[r1] = v1;
    if (pay) pay[r1] = p1;
  }
  consumers_sync();
}

// Sort, descending, of n > 256 distinct values whose bits crowd: 256 of the
// values, taken evenly over their (arbitrary) order and ranked by counting, split the
// rest into buckets of about n / 256 whatever their distribution; then as the
// bucket sort.
__device__ void splitter_sort_desc(uint64_t *a, uint32_t n, uint64_t *tmp, SelectScratch &ss, uint32_t *pay,
                                   uint32_t *tmp_pay) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t mine = a[(uint64_t)tid * n / kConsumers];
  tmp[tid] = mine;
  ss.hist[tid] = 0;
  consumers_sync();
  uint32_t r = 0;
#pragma unroll 8
  for (uint32_t q = 0; q < kConsumers; q++) r += tmp[q] > mine ? 1u : 0u;
  ss.split[r] = mine;
  consumers_sync();
  // the bucket of a value: the splitters above it, the last one left out
  auto bucket = [&](uint64_t v) {
    uint32_t lo = 0;
#pragma unroll
    for (uint32_t step = 128; step > 0; step >>= 1)
      if (ss.split[lo + step - 1] > v) lo += step;
    return lo;
  };
  for (uint32_t i = tid; i < n; i += kConsumers) atomicAdd(&ss.hist[bucket(a[i])], 1u);
  consumers_sync();
  const uint32_t c = ss.hist[tid];
  uint32_t incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31) ss.wtot[warp] = incl;
  consumers_sync();
  uint32_t ex = incl - c;
  for (uint32_t w = 0; w < warp; w++) ex += ss.wtot[w];
  ss.off[tid] = ex;
  ss.hist[tid] = ex;
  consumers_sync();
  for (uint32_t i = tid; i < n; i += kConsumers) {
    const uint64_t v = a[i];
    const uint32_t p = atomicAdd(&ss.hist[bucket(v)], 1u);
    tmp[p] = v;
    if (pay) tmp_pay[p] = pay[i];
  }
  consumers_sync();
  for (uint32_t p = tid; p < n; p += kConsumers) {
    const uint64_t v = tmp[p];
    const uint32_t b = bucket(v), lo = ss.off[b], hi = ss.hist[b];
    uint32_t k = 0;
    for (uint32_t q = lo; q < hi; q++) k += tmp[q] > v ? 1u : 0u;
    a[lo + k] = v;
    if (pay) pay[lo + k] = tmp_pay[p];
  }
  consumers_sync();
}

// Sort, descending, of distinct values by the cheapest of the three.  tmp:
// room for n values (and tmp_pay for n payloads when pay is given), apart from
// a and pay.
__device__ __forceinline__ void sort_desc(uint64_t *a, uint32_t n, uint64_t *tmp, SelectScratch &ss,
                                          uint32_t *pay = nullptr, uint32_t *tmp_pay = nullptr) {
  if (n <= kCountSort) count_sort_desc(a, n, pay);
  else if (!bucket_sort_desc(a, n, tmp, ss, pay, tmp_pay)) splitter_sort_desc(a, n, tmp, ss, pay, tmp_pay);
}

// ------------------------------------------------------------- sample ----
// Sample size and per-list ranks.  A list aims at target candidates: with a
// sample of ns of the n records, the threshold is the sample's rank r =
// ceil(target ns / n).  The candidates above the rank-r sample number about
// target / r Gamma(r), and fall short of the M wanted with probability
// P(Gamma(r) < r M / target) = P(Poisson(r M / target) >= r): r is large enough
// when that is below 1e-6 (sample_rank).  A shortfall costs time, never
// exactness (the finish re-selects the list).  A larger target needs a smaller
// rank, hence a smaller sample (28, 17, 13, 10 for M = 1,024 at the last four
// targets below: 0.9, 0.37, 0.21, 0.11 % of the records), but leaves more candidates to
// the streaming tests and the finish.  A set takes the smallest target whose
// sample is within its cap (plan_sample): 1,024 a sampling CTA, and the larger of its share
// of kLaunchSamples and kSetSamples, because a sample's runs are random rows of
// DRAM.  Measured, whole call: 33 sets of 2^20 records 118 us at 9,800 samples
// a set, 139 us at 4,096 (18,000 candidates a set in place of 13,000, and a
// longer last set); 7 sets of 2^24 199 us at 18,000 a set, 205 us at 35,000 (the
// calls took 8 to 12 us longer then than they do with 16-bit histograms).
// The threshold is the floor of the histogram bin holding the rank-r sample, so
// it admits a few more.
__host__ __forceinline__ uint64_t umin64(uint64_t a, uint64_t b) { return a < b ? a : b; }
__host__ __forceinline__ bool list_active(const RankSet &S, int L) {
  const uint32_t M = (L == 0) ? S.k : S.max_moves;
  return M > 0 && (L == 0 || S.budget > 0);
}
constexpr int kTargets = 6;
__host__ __forceinline__ uint64_t list_wanted(const RankSet &S, int L) { return (L == 0) ? S.k : S.max_moves; }
__host__ __forceinline__ uint64_t target_of(uint64_t M, int o) {
  const uint64_t mul[kTargets] = {2, 2, 2, 3, 4, 6}, add[kTargets] = {128, 256, 512, 512, 512, 512};
  return mul[o] * (M + add[o]);
}
// The smallest rank whose chance of a shortfall is below 1e-6, for a ratio M /
// target of at most q / 64 (q <= 32).
struct SampleRanks {
  uint32_t r[33];
  SampleRanks() {
    for (int q = 0; q <= 32; q++) {
      for (r[q] = 1; r[q] < 128; r[q]++) {
        // P(Poisson(x) >= r) <= x^r e^-x / r! / (1 - x / (r + 1))
        const double x = q / 64.0 * r[q];
        double p = std::exp(-x);
        for (uint32_t i = 1; i <= r[q]; i++) p *= x / i;
        if (p / (1.0 - x / (r[q] + 1)) < 1e-6) break;
      }
    }
  }
};
__host__ uint32_t sample_rank(uint64_t M, uint64_t target) {
  static const SampleRanks ranks;
  return ranks.r[std::min<uint64_t>((64 * M + target - 1) / target, 32)];
}
// Samples that target choice o of a list of M needs.
__host__ uint64_t sample_size(const RankSet &S, uint64_t M, int o) {
  const uint64_t t = target_of(M, o);
  return ((uint64_t)sample_rank(M, t) * S.n + t - 1) / t;
}

// CTAs a set can use: one a tile, and one a list for the finish (a set of
// 1,000 records whose one CTA finished its lists in turn took 58 us, with three
// 29 us, and 17 us when each collects its list's values itself).
__host__ __forceinline__ uint32_t most_ctas(const RankSet &S) { return std::max<uint32_t>(S.ntiles, kLists); }

// Groups of a launch of at most `ctas` sets: each set gets CTAs in proportion
// to its tiles (at least 1, at most most_ctas); CTAs left over go to the sets
// with the most tiles per CTA, and where the sets of less than a CTA's share
// took more than there are, the sets with the fewest tiles per CTA give theirs
// back.  Returns the CTAs of all groups: never more than `ctas`, which are
// resident at once (a cooperative launch of more is refused).
uint32_t share_ctas(std::vector<RankSet> &sets, uint32_t ctas, uint64_t tiles) {
  uint64_t used = 0;
  for (RankSet &s : sets) {
    s.nctas = (uint32_t)std::max<uint64_t>(1, (uint64_t)ctas * s.ntiles / tiles);
    s.nctas = std::min(s.nctas, most_ctas(s));
    used += s.nctas;
  }
  auto denser = [](const RankSet &a, const RankSet &b) {  // more tiles per CTA
    return (uint64_t)a.ntiles * b.nctas > (uint64_t)b.ntiles * a.nctas;
  };
  for (; used < ctas; used++) {
    RankSet *most = nullptr;
    for (RankSet &s : sets)
      if (s.nctas < most_ctas(s) && (!most || denser(s, *most))) most = &s;
    if (!most) break;
    most->nctas++;
  }
  for (; used > ctas; used--) {
    RankSet *least = nullptr;  // there is one: `ctas` sets or fewer hold more than `ctas`
    for (RankSet &s : sets)
      if (s.nctas > 1 && (!least || denser(*least, s))) least = &s;
    least->nctas--;
  }
  uint32_t cta = 0;
  for (RankSet &s : sets) {
    s.cta0 = cta;
    cta += s.nctas;
  }
  return cta;
}

// The sample plan of a set whose group (cta0, nctas) is fixed.  The longest
// list decides the sample; each other list takes the smallest target that this
// sample allows it (a short list needs more samples for a target of its size
// than a long one, and chosen for all lists together it put the long lists on
// larger targets: 9 sets of 2^22, k from 1 to 1,024, 100.3 us, 94.4 with a
// target a list and 16,384 samples a set in place of 12,288).
// The second target only where a set has few CTAs to share its candidates
// among: without it 16 sets of 2^18 (28 CTAs each) take 54.9 us in place of
// 52.7 and 8 of 2^20 (57 CTAs) 53.2 in place of 52.0; 33 and 7 sets of 2^20, 64
// of 2^18 and 8 of 2^22 the same within 0.5.  With it everywhere, 1 to 5 sets
// of 2^20 (91 CTAs and more) move between -1.0 and +0.2 us.
constexpr uint32_t kFewCtas = 64;
void plan_sample(RankSet &s, int n_sets) {
  const uint32_t most = std::min(s.nctas, kSampleCtas);
  const uint64_t share = std::max<uint64_t>(kLaunchSamples / n_sets, kSetSamples);
  const uint64_t cap = umin64((uint64_t)kPerCtaSamples * most, share);
  uint64_t longest = 0, ns = 0;
  for (int L = 0; L < kLists; L++)
    if (list_active(s, L)) longest = std::max(longest, list_wanted(s, L));
  // up to 4,096 records, the finish holds every record's value in shared
  // memory; a set of 16,000 takes 42 us with a sample, and about 75 us when
  // every record is a candidate
  if (s.n > kSmemCand && longest) {
    int o = 0;
    for (;; o++) {
      ns = sample_size(s, longest, o);
      const bool fits = ns <= (o == 0 ? umin64(cap, kSmallSample) : cap) && (o != 1 || s.nctas < kFewCtas);
      if (fits || o + 1 == kTargets) break;
    }
    if (s.n <= kSample && 2 * target_of(longest, o) > s.n) ns = 0;  // a sample would leave most records candidates
  }
  if (ns)
    for (int L = 0; L < kLists; L++)
      if (list_active(s, L)) ns = std::max(ns, sample_size(s, list_wanted(s, L), kTargets - 1));
  ns = umin64(ns, cap);
  // half a CTA's most a CTA where there are enough: the samples' latency is the
  // call's head
  s.direct = ns == 0 && s.n <= kSmemCand && s.nctas == kLists ? 1u : 0u;
  s.sctas = ns ? (uint32_t)umin64(most, (ns + kPerCtaSamples / 2 - 1) / (kPerCtaSamples / 2)) : 0u;
  if (ns) ns = (ns + 8ull * s.sctas - 1) / (8ull * s.sctas) * (8ull * s.sctas);  // whole runs, evenly split
  ns = umin64(ns, (uint64_t)kPerCtaSamples * s.sctas);
  s.ns = (uint32_t)ns;
  s.nruns = s.ns / 8;
  s.sstep = s.nruns ? ((uint64_t)s.n << 16) / s.nruns : 0;
  for (int L = 0; L < kLists; L++) {
    s.rL[L] = 0;
    if (!s.ns || !list_active(s, L)) continue;
    const uint64_t M = list_wanted(s, L);
    int o = 0;
    while (o + 1 < kTargets && sample_size(s, M, o) > s.ns) o++;
    s.rL[L] = (uint32_t)((target_of(M, o) * s.ns + s.n - 1) / s.n);
  }
}

// Sampling CTA r of set S (consumer threads): samples j = r * per + jt of
// the CTA's share, run j / 8 covering stratum j / 8 (records from about
// run n / nruns to (run+1) n / nruns), 8 consecutive records at a hashed
// offset in it.  Each eligible sample is added to its lists' histograms (the
// lanes of a warp that all hit one bin add to it once), and the CTA's ticket
// says its counts are in.
__device__ __noinline__ void sample_share(const RankSet &S, uint32_t r, const uint64_t *t2s, const uint64_t *mgs) {
  const uint32_t tid = threadIdx.x;
  const uint32_t nct = S.sctas, act = S.act;
  const uint32_t per = S.ns / nct;  // samples of this CTA (<= 1024, a multiple of 8)
  uint32_t rr[kSampleQ];
  bool ok[kSampleQ];
#pragma unroll
  for (int q = 0; q < (int)kSampleQ; q++) {
    const uint32_t jt = tid + kConsumers * q;
    ok[q] = jt < per;
    rr[q] = 0;
    if (ok[q]) {
      // stratum bounds about run n / nruns (16.16 fixed point: no division
      // on the sample's path; any stratification samples correctly)
      const uint32_t run = r * (per / 8) + jt / 8, o = jt % 8;
      const uint32_t lo = (uint32_t)((run * S.sstep) >> 16), hi = (uint32_t)(((run + 1) * S.sstep) >> 16);
      uint32_t h = run * 0x9E3779B1u;
      h ^= h >> 16;
      h *= 0x85EBCA6Bu;
      h ^= h >> 13;
      const uint32_t span = hi - lo >= 8 ? hi - lo - 8 : 0u;  // strata hold at least 8 records
      rr[q] = min(lo + __umulhi(h, span + 1) + o, S.n - 1);
    }
  }
  uint8_t fl[kSampleQ], tr[kSampleQ];
  uint16_t tu[kSampleQ];
  uint32_t gg[kSampleQ];
#pragma unroll
  for (int q = 0; q < (int)kSampleQ; q++) {  // index 0 for an unused slot: a valid record
    fl[q] = S.flags[rr[q]];
    tr[q] = S.tier[rr[q]];
    tu[q] = S.turn[rr[q]];
    gg[q] = S.gap[rr[q]];
  }
#pragma unroll
  for (int q = 0; q < (int)kSampleQ; q++) {
    const uint32_t t = min((uint32_t)tu[q], kTMax);
    const uint64_t ck = ck_of(score_of(gg[q], t, (fl[q] & 2) != 0, t2s, mgs), S.off + rr[q]);
    const uint32_t em = ok[q] ? elig_mask(fl[q], tr[q]) & act : 0u;
#pragma unroll
    for (int L = 0; L < kLists; L++) {
      const bool in = (em >> L) & 1;
      const uint32_t b = list_bin(summary_of(list_val(ck, L)), L);
      const unsigned who = __ballot_sync(kFull, in);
      const int first = who ? __ffs(who) - 1 : 0;
      const uint32_t b0 = __shfl_sync(kFull, b, first);
      const bool one = __ballot_sync(kFull, in && b == b0) == who;
      if (in && (!one || (int)(tid & 31) == first))
        // two counts a word: neither can pass 16 bits (kMaxSample)
        atomicAdd(reinterpret_cast<unsigned int *>(S.shist) + (L * kBins + b) / 2,
                  (one ? (unsigned)__popc(who) : 1u) << 16 * (b & 1));
    }
  }
  if (tid == 0) atomicAdd(&S.work->gathered, 1u);  // the group's copies may start now
  __threadfence();
  consumers_sync();
  if (tid == 0) atomicAdd(&S.work->sample_ticket, 1u);  // this CTA's counts are in the histogram
}

// ------------------------------------------------------------- filter ----
struct SetConst {
  uint64_t thr[kLists];        // threshold per list, in list-value space (0: every eligible record)
  uint32_t loV, loD, loP;      // index thresholds of the tie on the threshold key
  uint32_t dV, dD;             // completed records pass V / D iff lo >= dV / dD
  int32_t dP;                  // completed records pass P iff lo <= dP
  uint32_t act;                // active lists (bit L)
};

// Thresholds of one set into shared memory (consumer threads), computed by
// every CTA of the group alike once the sample's counts are all in the
// histogram: each list's histogram is cut at its sample rank r_L, the
// threshold is the smallest list value of the cut's bin (0, every eligible
// record, when the sample holds fewer than r_L), and per turn index t the
// bounds are the smallest gap whose key reaches the threshold's key (gA) or
// exceeds it (gB): vd = (gA_V, gB_V, gA_D, gB_D), pp = (gA_P, gB_P).  An
// inactive list gets bounds no gap passes.
__device__ void thresholds(const RankSet &S, const uint64_t *t2s, const uint32_t *sgs, uint4 *vd, uint2 *pp,
                           SetConst &c) {
  __shared__ uint64_t sthr[kLists];
  int cut[kLists] = {-1, -1, -1};
  if (S.ns) {
    const uint32_t need[kLists] = {S.rL[0], S.rL[1], S.rL[2]};
    hist_cut3(S.shist, need, cut);
  }
  if (threadIdx.x < kLists) sthr[threadIdx.x] = cut[threadIdx.x] >= 0 ? summary_floor(list_bin_floor((uint32_t)cut[threadIdx.x], (int)threadIdx.x)) : 0ull;
  consumers_sync();
  const bool aV = S.act & 1, aD = (S.act >> 1) & 1, aP = (S.act >> 2) & 1;
  if (threadIdx.x < kLutN) {
    const uint32_t t = threadIdx.x;
    uint2 g[kLists];
#pragma unroll
    for (int L = 0; L < kLists; L++) {
      const uint64_t thr_ck = (L == 2) ? ~sthr[L] : sthr[L];
      const uint64_t K = thr_ck >> 24;
      g[L] = make_uint2(g_at_least(K, sgs[t], t2s[t]), g_at_least(K + 1, sgs[t], t2s[t]));
    }
    vd[t] = make_uint4(aV ? g[0].x : kFull, aV ? g[0].y : kFull, aD ? g[1].x : kFull, aD ? g[1].y : kFull);
    pp[t] = aP ? g[2] : make_uint2(0u, 0u);
  }
  if (threadIdx.x == 32) {
    uint32_t lo[kLists], dok[kLists];
#pragma unroll
    for (int L = 0; L < kLists; L++) {
      const uint64_t thrv = sthr[L];
      c.thr[L] = thrv;
      const uint64_t thr_ck = (L == 2) ? ~thrv : thrv;
      const uint64_t K = thr_ck >> 24;
      lo[L] = (uint32_t)(thr_ck & kIdMask);
      // a completed record has the maximal key 2^40 - 1: 2 = always passes,
      // 1 = passes on the index part, 0 = never
      dok[L] = (L == 2) ? (kKeyMax40 == K ? 1u : 0u) : (kKeyMax40 > K ? 2u : (kKeyMax40 == K ? 1u : 0u));
    }
    c.loV = lo[0];
    c.loD = lo[1];
    c.loP = lo[2];
    c.dV = !aV ? 0x1000000u : (dok[0] == 2 ? 0u : (dok[0] == 1 ? lo[0] : 0x1000000u));
    c.dD = !aD ? 0x1000000u : (dok[1] == 2 ? 0u : (dok[1] == 1 ? lo[1] : 0x1000000u));
    c.dP = (aP && dok[2] == 1) ? (int32_t)lo[2] : -1;
    c.act = S.act;
  }
  consumers_sync();
}

// ------------------------------------------------------------- finish ----
// Exact top-M of list L over the whole set by one CTA, streaming records and
// keeping a pool of at most M + 4 * kConsumers values in pool[] (the
// fallback path).  The result is in pool[0..return).
__device__ __noinline__ uint32_t stream_topM(const RankSet &S, int L, uint32_t M, uint64_t *pool, const uint64_t *t2s,
                                const uint64_t *mgs, SelectScratch &ss) {
  if (threadIdx.x == 0) ss.cnt = 0;
  uint64_t floorv = 0;  // accept values strictly above (once a floor exists)
  bool have_floor = false;
  consumers_sync();
  for (uint32_t b = 0; b < S.n; b += 4 * kConsumers) {
    for (uint32_t q = 0; q < 4; q++) {
      const uint32_t r = b + q * kConsumers + threadIdx.x;
      if (r < S.n) {
        const uint32_t m = elig_mask(S.flags[r], S.tier[r]);
        if ((m >> L) & 1) {
          const uint32_t t = min((uint32_t)S.turn[r], kTMax);
          const uint64_t v = list_val(ck_of(score_of(S.gap[r], t, (S.flags[r] & 2) != 0, t2s, mgs), S.off + r), L);
          if (!have_floor || v > floorv) pool[atomicAdd(&ss.cnt, 1u)] = v;
        }
      }
    }
    consumers_sync();
    const uint32_t c = ss.cnt;
    if (c > M) {
      const uint64_t th = block_select_rank([&](uint32_t i) { return pool[i]; }, c, M, ss);
      // compact in place to the values >= th (exactly M: values are unique),
      // through registers so that no unread value is overwritten
      constexpr uint32_t kKeep = (kMaxSel + 4 * kConsumers) / kConsumers;  // entries a thread scans, at most
      uint64_t keep[kKeep];
      uint32_t nk = 0;
      for (uint32_t i = threadIdx.x; i < c; i += kConsumers) {
        const uint64_t v = pool[i];
        if (v >= th && nk < kKeep) keep[nk++] = v;
      }
      if (threadIdx.x == 0) ss.cnt = 0;
      consumers_sync();
      for (uint32_t i = 0; i < nk; i++) pool[atomicAdd(&ss.cnt, 1u)] = keep[i];
      consumers_sync();
      floorv = th;
      have_floor = true;
    }
    consumers_sync();
  }
  const uint32_t got = min(ss.cnt, M);
  consumers_sync();
  return got;
}

// Every eligible record's value of list L into buf (room for the set's
// records), and, for list 0, the keys when asked for.  Returns the count.
__device__ __noinline__ uint32_t collect_list(const RankSet &S, int L, uint64_t *buf, const uint64_t *t2s,
                                              const uint64_t *mgs, SelectScratch &ss) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, n = S.n;
  const bool active = (S.act >> L) & 1, keys = L == 0 && S.keys;
  if (tid == 0) ss.cnt = 0;
  consumers_sync();
  for (uint32_t b = 0; b < n; b += 4 * kConsumers) {
    const uint32_t i = b + 4 * tid;
    uint32_t g[4], t[4], fl[4], tr[4];
    if (i + 4 <= n) {
      const uint4 gq = *reinterpret_cast<const uint4 *>(S.gap + i);
      const uint2 tq = *reinterpret_cast<const uint2 *>(S.turn + i);
      const uint32_t fq = *reinterpret_cast<const uint32_t *>(S.flags + i);
      const uint32_t rq = *reinterpret_cast<const uint32_t *>(S.tier + i);
      g[0] = gq.x; g[1] = gq.y; g[2] = gq.z; g[3] = gq.w;
      t[0] = tq.x & 0xFFFFu; t[1] = tq.x >> 16; t[2] = tq.y & 0xFFFFu; t[3] = tq.y >> 16;
#pragma unroll
      for (int k = 0; k < 4; k++) {
        fl[k] = fq >> 8 * k & 0xFFu;
        tr[k] = rq >> 8 * k & 0xFFu;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const bool in = i + k < n;
        g[k] = in ? S.gap[i + k] : 0u;
        t[k] = in ? S.turn[i + k] : 0u;
        fl[k] = in ? S.flags[i + k] : 1u;  // padding reads as pinned: never eligible
        tr[k] = in ? S.tier[i + k] : 0u;
      }
    }
    uint64_t v[4];
    unsigned bal[4], at = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const uint64_t sc = score_of(g[k], min(t[k], kTMax), (fl[k] & 2) != 0, t2s, mgs);
      if (keys && i + k < n) S.keys[i + k] = sc;
      v[k] = list_val(ck_of(sc, S.off + i + k), L);
      bal[k] = __ballot_sync(kFull, active && ((elig_mask((uint8_t)fl[k], (uint8_t)tr[k]) >> L) & 1));
    }
    const uint32_t n0 = __popc(bal[0]), n1 = n0 + __popc(bal[1]), n2 = n1 + __popc(bal[2]);
    if (lane == 0) at = atomicAdd(&ss.cnt, n2 + __popc(bal[3]));
    at = __shfl_sync(kFull, at, 0);
    const uint32_t before[4] = {0u, n0, n1, n2};
#pragma unroll
    for (int k = 0; k < 4; k++)
      if (bal[k] >> lane & 1) buf[at + before[k] + __popc(bal[k] & ((1u << lane) - 1))] = v[k];
  }
  consumers_sync();
  return ss.cnt;
}

// List L of set S: the exact top-M of its candidates, sorted, with the moved
// records' sizes; victims are written out directly.  fin: the 64 KB dynamic
// area (the stages are idle).  Returns true when this was the set's last list.
// local >= 0: the area already holds that many candidates, every eligible
// record's (collect_list).
__device__ __noinline__ bool finish_list(const RankSet &S, int L, uint64_t *fin, const uint64_t *t2s, const uint64_t *mgs,
                                         SelectScratch &ss, const SetConst &cs, int local = -1) {
  __shared__ __align__(8) uint64_t cbar;
  __shared__ unsigned int last, sh_emitted, sh_flags, nsurv;
  const uint32_t Mw = (L == 0) ? S.k : S.max_moves;
  // the area holds what the sort takes (M and some slack, at most kMaxSel) and,
  // in the rest, the candidates (6,144 of them for lists of up to 1,024)
  const uint32_t selcap = min(Mw + slack(Mw), kMaxSel) + 1u & ~1u, bufcap = kDynWords - selcap;
  uint64_t *buf = fin;           // [bufcap] candidates
  uint64_t *sel = fin + bufcap;  // [selcap] the kept top-M
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  // one thread reads the other CTAs' results, so that every consumer thread
  // takes the same path through the barriers below
  if (tid == 0) {
    sh_emitted = local >= 0 ? (unsigned)local : __ldcg(&S.work->cand[L]);
    sh_flags = local >= 0 ? ((S.act >> L) & 1u) | 2u : ((cs.act >> L) & 1u) | (cs.thr[L] == 0 ? 2u : 0u);
  }
  consumers_sync();
  const bool active = sh_flags & 1;
  const uint32_t emitted = sh_emitted;
  // Candidates are every eligible record at or beyond the threshold.  They
  // certify the top Mw when there are at least Mw of them, or when the
  // threshold admitted every eligible record; otherwise (or when the list
  // overflowed) the list is re-selected exactly from the whole set.
  const bool all_admitted = (sh_flags & 2) != 0;
  const bool certified = emitted <= S.ccap && (emitted >= Mw || all_admitted);
  const uint32_t M = !active ? 0u : (certified ? min(Mw, emitted) : Mw);
  uint32_t got = 0;
  uint64_t *out = sel;
  if (M > 0) {
    const uint64_t *cand = S.cand + (size_t)L * S.ccap;
    if (certified) {
      const uint32_t c = emitted;
      const bool in_smem = c <= bufcap;
      if (in_smem && local < 0) {
        // one bulk copy (an even count: a 16-byte multiple; ccap is even, so
        // the list holds c + 1 entries when c is odd, and so does the area)
        const uint32_t bytes = ((c + 1) & ~1u) * 8u;
        fence_proxy_async();  // earlier generic accesses to the area before the async copy
        consumers_sync();
        if (tid == 0) {
          // the candidates are ordinary stores of every CTA of the group, seen
          // by this thread's wait; the copy reads them by another route
          fence_proxy_async_global();
          mbar_init(&cbar, 1);
          fence_mbar_init();
          mbar_expect_tx(&cbar, bytes);
          bulk_g2s(buf, cand, bytes, &cbar);
        }
        if (!wait_phase_uniform(S, &cbar, 0))
          wait_phase_uniform(S, &cbar, 0);  // let the copy land before the area is reused
      }
      const uint64_t *src = in_smem ? buf : cand;
      // every value of from[0..n), a block-wide pass, eight independent loads
      // a thread in flight (fn(v, ok): ok false past the end)
      auto each_w = [&](const uint64_t *from, uint32_t n, auto fn) {
        for (uint32_t base = 0; base < n; base += 8 * kConsumers) {
          uint64_t v[8];
#pragma unroll
          for (uint32_t u = 0; u < 8; u++) {
            const uint32_t i = base + u * kConsumers + tid;
            v[u] = i < n ? from[i] : 0ull;
          }
#pragma unroll
          for (uint32_t u = 0; u < 8; u++)
            if (base + u * kConsumers < n) fn(v[u], base + u * kConsumers + tid < n);
        }
      };
      // the values of from[0..n) at or above t, in any order
      auto keep_from = [&](const uint64_t *from, uint32_t n, uint64_t t, uint64_t *to) {
        if (tid == 0) nsurv = 0;
        consumers_sync();
        each_w(from, n, [&](uint64_t v, bool ok) {
          const bool keep = ok && v >= t;
          const unsigned bal = __ballot_sync(kFull, keep);
          unsigned wb = 0;
          if (lane == 0 && bal) wb = atomicAdd(&nsurv, (unsigned)__popc(bal));
          wb = __shfl_sync(kFull, wb, 0);
          const uint32_t pos = wb + __popc(bal & ((1u << lane) - 1));
          if (keep && pos < selcap) to[pos] = v;
        });
        consumers_sync();
      };
      if (c <= selcap) {
        // every candidate is kept (and the sort drops those beyond M)
        for (uint32_t i = tid; i < c; i += kConsumers) sel[i] = src[i];
        got = c;
      } else {
        // values at or above t hold the top M: t rises bucket by bucket until
        // few values beyond M are left.  Values that crowd (small keys, ties)
        // take a step more, where one cut would leave a bucket of thousands to
        // sort.  Once they fit, the values move to shared memory.
        const uint64_t *from = src;
        uint32_t n = c, need = M;
        uint64_t t = 0;
        int sh = 64;
        for (;;) {
          const uint32_t in = narrow(
              [&](auto fn) {
                each_w(from, n, [&](uint64_t v, bool ok) {
                  if (ok) fn(v);
                });
              },
              t, sh, need, ss);
          const uint32_t left = M - need + in;  // at or above t
          if (left <= selcap && (from != sel || left <= n / 2 || left <= M + slack(M) || sh == 0)) {
            if (from == sel) {  // (buf is free then)
              keep_from(sel, n, t, buf);
              for (uint32_t i = tid; i < left; i += kConsumers) sel[i] = buf[i];
              consumers_sync();
            } else {
              keep_from(from, n, t, sel);
            }
            from = sel;
            n = left;
          }
          if (sh == 0 || (from == sel && n <= M + slack(M))) break;
        }
        got = n;
      }
      consumers_sync();
      sort_desc(sel, got, buf, ss);
      got = min(got, M);
    } else {
      // candidates overflowed the buffer or fell short of M: exact re-selection
      ss.hist[threadIdx.x] = 0;
      consumers_sync();
      got = stream_topM(S, L, M, fin, t2s, mgs, ss);
      out = fin;
      sort_desc(fin, got, fin + kMaxSel, ss);
    }
    // store the list; the fill reads the moved records' sizes, gathered here
    // eight at a time (independent random reads)
    for (uint32_t base = 0; base < got; base += 8 * kConsumers) {
      uint64_t v[8];
      uint32_t kv[8];
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const uint32_t i = base + u * kConsumers + threadIdx.x;
        v[u] = i < got ? out[i] : 0ull;
        const uint32_t idx = (~(uint32_t)(L == 2 ? ~v[u] : v[u])) & kIdMask;
        kv[u] = (L != 0 && i < got) ? S.kv[idx - S.off] : 0u;
      }
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const uint32_t i = base + u * kConsumers + threadIdx.x;
        if (i < got) {
          if (S.cands) {  // a shard: the list goes out, keyed by the whole set's index
            CandEntry *e = reinterpret_cast<CandEntry *>(S.cands + cand_list_off(S.k, S.max_moves, L));
            e[i] = CandEntry{v[u], kv[u], 0u};
          } else {
            S.sorted[(size_t)L * kMaxSel + i] = v[u];
            if (L == 0) S.victims[i] = (~(uint32_t)v[u]) & kIdMask;
            else S.ssz[(size_t)L * kMaxSel + i] = kv[u];
          }
        }
      }
    }
  }
  if (threadIdx.x == 0) {
    S.work->got[L] = got;
    if (S.cands) reinterpret_cast<CandHeader *>(S.cands)->count[L] = got;
  }
  __threadfence();
  consumers_sync();
  if (threadIdx.x == 0) last = (atomicAdd(&S.work->list_ticket, 1u) == (unsigned)kLists - 1);
  consumers_sync();
  return last != 0;
}

// ------------------------------------------------------------- fill ----
// Inclusive prefix over the consumer threads of (a, b); the block's totals
// come back in (ta, tb).  Two barriers.
__device__ void block_incl_scan2(uint64_t &a, int64_t &b, uint64_t &ta, int64_t &tb) {
  __shared__ uint64_t wa[kConsumers / 32];
  __shared__ int64_t wb[kConsumers / 32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t ya = __shfl_up_sync(kFull, a, o);
    const int64_t yb = __shfl_up_sync(kFull, b, o);
    if ((int)lane >= o) {
      a += ya;
      b += yb;
    }
  }
  if (lane == 31) {
    wa[warp] = a;
    wb[warp] = b;
  }
  consumers_sync();
  uint64_t pa = 0, sa = 0;
  int64_t pb = 0, sb = 0;
#pragma unroll
  for (uint32_t w = 0; w < kConsumers / 32; w++) {
    if (w < warp) {
      pa += wa[w];
      pb += wb[w];
    }
    sa += wa[w];
    sb += wb[w];
  }
  a += pa;
  b += pb;
  ta = sa;
  tb = sb;
  consumers_sync();  // wa and wb free for the next call
}

// The TIDE fill of set S from its sorted lists (Sec. III-C): phase 1
// promotes the least evictable HBM records into free fast-tier space in order
// while the budget and the space last; phase 2 pairs the next HBM record with
// the j-th most evictable fast-tier record (demotions merged with the phase-1
// promotions) while the demoted one ranks above the promoted one and the
// budget and both tiers' capacities hold.  Each phase takes items in order
// and stops at the first that fails.  The state after j items is a prefix
// sum, so the consumer threads take a phase 256 items at a time, one item
// each: a block scan of the sizes, then the smallest failing item of the
// chunk; the fill stops at the first chunk that holds one (most fills end in
// the first).  Every size is in tokens and the budget test is on tokens: j
// items of s_1..s_j tokens cost (s_1 + ... + s_j) * kvb bytes, which is
// within the budget exactly when s_1 + ... + s_j <= floor(budget / kvb).
// The lists are staged in shared memory (P as ascending key, D descending,
// 12 bytes an entry) when they fit, else read in place.
__device__ __noinline__ void fill(const RankSet &S, uint64_t *fin) {
  __shared__ unsigned int sh_got[kLists], sh_act, sh_st, first_bad;
  __shared__ unsigned long long sh_tok;
  __threadfence();
  const uint32_t tid = threadIdx.x;
  if (tid == 0) {  // read once and shared: one path through the barriers
    for (int L = 0; L < kLists; L++) sh_got[L] = min(__ldcg(&S.work->got[L]), kMaxSel);
    sh_act = S.act & 6u;
    sh_st = *(volatile unsigned int *)&S.work->status;
  }
  consumers_sync();
  const uint32_t nv = sh_got[0], nd = sh_got[1], np = sh_got[2];
  const uint64_t *Pg = S.sorted + 2 * kMaxSel, *Dg = S.sorted + kMaxSel;
  const uint32_t *PSg = S.ssz + 2 * kMaxSel, *DSg = S.ssz + kMaxSel;
  const bool staged = 12ull * (np + nd) <= kDynSmem;
  uint64_t *pck = fin, *dck = fin + np;
  uint32_t *psz = reinterpret_cast<uint32_t *>(fin + np + nd), *dsz = psz + np;
  if (staged) {
    // both lists' loads in flight together, four entries of each a thread
    for (uint32_t base = tid; base < max(np, nd); base += 4 * kConsumers) {
      uint64_t pk[4], dk[4];
      uint32_t pz[4], dz[4];
#pragma unroll
      for (uint32_t u = 0; u < 4; u++) {
        const uint32_t i = base + u * kConsumers;
        pk[u] = i < np ? __ldcg(Pg + i) : 0ull;
        pz[u] = i < np ? __ldcg(PSg + i) : 0u;
        dk[u] = i < nd ? __ldcg(Dg + i) : 0ull;
        dz[u] = i < nd ? __ldcg(DSg + i) : 0u;
      }
#pragma unroll
      for (uint32_t u = 0; u < 4; u++) {
        const uint32_t i = base + u * kConsumers;
        if (i < np) {
          pck[i] = ~pk[u];
          psz[i] = pz[u];
        }
        if (i < nd) {
          dck[i] = dk[u];
          dsz[i] = dz[u];
        }
      }
    }
  }
  auto p_ck = [&](uint32_t i) -> uint64_t { return staged ? pck[i] : ~__ldcg(Pg + i); };
  auto p_sz = [&](uint32_t i) -> uint32_t { return staged ? psz[i] : __ldcg(PSg + i); };
  auto d_ck = [&](uint32_t i) -> uint64_t { return staged ? dck[i] : __ldcg(Dg + i); };
  auto d_sz = [&](uint32_t i) -> uint32_t { return staged ? dsz[i] : __ldcg(DSg + i); };
  if (tid == 0) first_bad = kFull;
  consumers_sync();
  const uint64_t kvb = S.kvb, cap_b = S.budget / kvb;  // tokens the budget pays for
  // phase 1: promotions into free fast-tier space, least evictable first
  const uint32_t lim1 = (sh_act & 4) ? min(np, S.max_moves) : 0u;
  const uint64_t cap1 = min(cap_b, S.free_s);
  uint32_t n1 = lim1;
  uint64_t tok1 = 0;  // tokens promoted so far
  for (uint32_t base = 0; base < lim1; base += kConsumers) {
    const uint32_t j = base + tid;
    uint64_t a = j < lim1 ? p_sz(j) : 0u, ta;
    int64_t b = 0, tb;
    block_incl_scan2(a, b, ta, tb);
    if (j < lim1 && tok1 + a > cap1) atomicMin(&first_bad, j);
    consumers_sync();
    const uint32_t fb = first_bad;
    if (fb != kFull) {
      if (j + 1 == fb) sh_tok = tok1 + a;
      consumers_sync();
      n1 = fb;
      if (fb > base) tok1 = sh_tok;
      if (tid == 0) first_bad = kFull;
      consumers_sync();
      break;
    }
    tok1 += ta;
  }
  // phase 2: pair P[n1 + j] with the j-th entry of the demotion order
  const uint64_t cap2b = cap_b - tok1, fs = S.free_s - tok1, fh = S.free_h + tok1;
  const uint32_t cap2 = S.max_moves > n1 ? S.max_moves - n1 : 0;
  const uint32_t nd2 = min(nd + n1, cap2);
  const uint32_t lim2 = ((sh_act & 6) == 6) ? min(np - n1, nd2) : 0u;
  // the j-th entry (descending) of D merged with P[n1-1], ..., P[0]
  auto demote_at = [&](uint32_t j, uint64_t &val, uint32_t &sz) {
    uint32_t lo = j + 1 > n1 ? j + 1 - n1 : 0u, hi = min(j + 1, nd);
    while (lo < hi) {  // D entries among the top j + 1
      const uint32_t mid = (lo + hi) >> 1;
      if (d_ck(mid) > p_ck(n1 - 1 - (j - mid))) lo = mid + 1; else hi = mid;
    }
    const uint32_t i = lo;
    if (i == 0 || (j + 1 - i > 0 && p_ck(n1 - 1 - (j - i)) < d_ck(i - 1))) {
      const uint32_t pj = n1 - 1 - (j - i);  // the smaller of the two last taken is from P
      val = p_ck(pj);
      sz = p_sz(pj);
    } else {
      val = d_ck(i - 1);
      sz = d_sz(i - 1);
    }
  };
  uint32_t pairs = lim2;
  uint64_t tok2 = 0;  // tokens moved by the pairs so far (both directions)
  int64_t bal = 0;    // net tokens into the fast tier so far
  for (uint32_t base = 0; base < lim2; base += kConsumers) {
    const uint32_t j = base + tid;
    uint64_t a = 0, ta;
    int64_t b = 0, tb;
    bool order_ok = false;
    if (j < lim2) {
      uint64_t dv;
      uint32_t sd;
      demote_at(j, dv, sd);
      const uint32_t sp = p_sz(n1 + j);
      order_ok = dv > p_ck(n1 + j);
      a = (uint64_t)sp + sd;
      b = (int64_t)sp - (int64_t)sd;
    }
    block_incl_scan2(a, b, ta, tb);
    const uint64_t A = tok2 + a;
    const int64_t Bv = bal + b;
    const bool ok = order_ok && A <= cap2b && (Bv <= 0 || (uint64_t)Bv <= fs) && (Bv >= 0 || (uint64_t)(-Bv) <= fh);
    if (j < lim2 && !ok) atomicMin(&first_bad, j);
    consumers_sync();
    const uint32_t fb = first_bad;
    if (fb != kFull) {
      if (j + 1 == fb) sh_tok = A;
      consumers_sync();
      pairs = fb;
      if (fb > base) tok2 = sh_tok;
      break;
    }
    tok2 += ta;
    bal += tb;
  }
  for (uint32_t i = tid; i < n1 + pairs; i += kConsumers) S.promote[i] = (~(uint32_t)p_ck(i)) & kIdMask;
  for (uint32_t i = tid; i < pairs; i += kConsumers) {
    uint64_t dv;
    uint32_t sd;
    demote_at(i, dv, sd);
    S.demote[i] = (~(uint32_t)dv) & kIdMask;
  }
  if (tid == 0) {
    S.counts[0] = nv;
    S.counts[1] = n1 + pairs;
    S.counts[2] = pairs;
    S.counts[3] = sh_st ? sh_st : (unsigned int)UNISON_OK;
    S.moved[0] = (tok1 + tok2) * kvb;  // at most floor(budget / kvb) tokens
  }
  consumers_sync();
}

// The set's last list is done: the fill, or a shard's header.
__device__ __forceinline__ void finish_set(const RankSet &S, uint64_t *fin) {
  if (!S.cands) {
    fill(S, fin);
  } else if (threadIdx.x == 0) {
    CandHeader *h = reinterpret_cast<CandHeader *>(S.cands);
    h->n = S.n;
    h->off = S.off;
    h->k = S.k;
    h->max_moves = S.max_moves;
    h->status = *(volatile unsigned int *)&S.work->status;
  }
}

// ------------------------------------------------------------- kernel ----
// Grouped (sequential == 0): CTA c serves the set whose group holds it.
// Sequential: CTA c serves sets c, c + G, c + 2G, ... one after another, each
// as a group of one.  The producer warp takes the group's tiles from the
// set's counter and announces each stage's tile in stile[]; a partial last
// tile (read directly from global memory by the consumers) and the end of
// the set (kEndTile) are announced with a plain arrival.
// zero (n_zero 16-byte words): the work words and sample histograms that the
// stream's previous call used, zeroed here for its next one.
// cmap (grouped launches): CTA b serves set cmap[b] & 0xFFFF, whose tables are
// tabs[cmap[b] >> 16]; null for a sequential launch.
// pack (d_sets null): the call's descriptors, tables and CTA map as a launch
// parameter, so that no upload precedes the kernel (it took 5 to 8 us of a
// call).  Calls of one set take a pack of one, up to 64 sets with at most two
// distinct tables a pack of 64 (about 20 KB of the 32 KB that a launch may
// bring); others upload theirs.
constexpr int kPackSets = 64, kPackTabs = 2;
template <int kSets>
struct RankPack {
  RankSet set[kSets];
  RankTab tab[kSets > 1 ? kPackTabs : 1];
  uint8_t of_cta[kSets > 1 ? kMaxGroup : 8];  // the set of each CTA
  uint8_t tab_of[kSets > 1 ? kSets : 8];
};
static_assert(sizeof(RankPack<kPackSets>) <= 30000, "a launch's parameters");
template <int kSets>
__global__ void __launch_bounds__(kCtaThreads, 3)
    rank_kernel(const RankSet *d_sets, int n_sets, int sequential, const uint32_t *cmap, const RankTab *tabs,
                uint4 *zero, uint32_t n_zero, const __grid_constant__ RankPack<kSets> pack) {
  extern __shared__ __align__(128) unsigned char dsm[];
  FilterStage *stage = reinterpret_cast<FilterStage *>(dsm);
  uint64_t *fin = reinterpret_cast<uint64_t *>(dsm);
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], sdone;
  __shared__ unsigned int stile[kStages];
  __shared__ uint4 vd[kLutN];
  __shared__ uint2 pp[kLutN];
  __shared__ uint64_t t2s[kLutN], mgs[kLutN];
  __shared__ SetConst cset;
  __shared__ RankSet rset;
  __shared__ unsigned int ccnt_s[kLists];  // candidates this CTA appended per list
  __shared__ unsigned int cbase_s[kLists];  // where its region goes in the set's list
  __shared__ uint32_t sgs[kLutN];
  __shared__ CtaScratch u;
  __shared__ unsigned int arrival;
#ifdef UNISON_DEBUG_HOOKS
  __shared__ __align__(8) uint64_t dummy_bar;
#endif

  {  // every CTA takes its share, before any returns
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x, gs = gridDim.x * blockDim.x;
    for (uint32_t w = g; w < n_zero; w += gs) zero[w] = make_uint4(0u, 0u, 0u, 0u);
  }
  const RankSet *const sets = d_sets ? d_sets : pack.set;
  int s0, sstep;
  const RankTab *tab0 = nullptr;  // the first set's tables, when the map names them
  if (sequential) {
    s0 = blockIdx.x;
    sstep = gridDim.x;
  } else if (!d_sets) {
    s0 = kSets > 1 ? pack.of_cta[blockIdx.x] : 0;
    tab0 = &pack.tab[kSets > 1 ? pack.tab_of[s0] : 0];
    sstep = n_sets;  // one set
  } else {
    const uint32_t e = __ldg(cmap + blockIdx.x);
    s0 = (int)(e & 0xFFFFu);
    tab0 = tabs + (e >> 16);
    sstep = n_sets;  // one set
  }
  if (s0 >= n_sets) return;
  if (threadIdx.x == 0) {
    for (int q = 0; q < kStages; q++) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], kConsumers / 32);
    }
    mbar_init(&sdone, 1);
#ifdef UNISON_DEBUG_HOOKS
    mbar_init(&dummy_bar, 1);
#endif
    fence_mbar_init();
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;

  if (threadIdx.x >= kConsumers) {
    // ---------------- producer warp (one lane issues)
    if (lane != 0) return;
    uint32_t lastph = 0;  // bit q: parity of the phase of stage q's last bulk copy
    uint32_t issued = 0;  // bit q: the last bulk copy into stage q may still be in flight
    uint32_t i = 0, nsets = 0;
    bool failed = false;
    int sfail = s0;
    for (int s = s0; s < n_sets && !failed; s += sstep) {
      const RankSet &T = sets[s];
      if (T.direct) return;  // (a grouped launch: this CTA's only set)
      const uint32_t r = sequential ? 0u : blockIdx.x - T.cta0, nct = sequential ? 1u : T.nctas;
      if (T.ns) {
        // The sample's random reads go first: the group's bulk copies would
        // otherwise queue ahead of them at the memory.  A short bounded wait;
        // if it runs out the copies simply start.
        const uint64_t t0 = now_ns();
        uint32_t nap = 64;
        while (*(volatile const unsigned int *)&T.work->gathered < T.sctas && now_ns() - t0 < 20000u) {
          __nanosleep(nap);
          nap = min(nap * 2, 512u);
        }
      }
      uint32_t claim = 0;  // the counter's answer for the next item, asked one item ahead
      for (uint32_t item = 0;; item++) {
        const int q = (int)(i % kStages);
        if (i >= (uint32_t)kStages) {
          // wait until the consumers released this stage's previous item
          if (!mbar_wait_bounded(&empty[q], ((i / kStages) - 1) & 1)) {
            failed = true;
            sfail = s;
            break;
          }
          issued &= ~(1u << q);
        }
        // the first kStages items of each CTA are dealt round-robin (every
        // CTA starts at once, and a set of few tiles spreads over the group);
        // the rest come from the group's counter, so that CTAs slowed by
        // candidate-heavy tiles take fewer
        const uint32_t t = item < (uint32_t)kStages ? r + item * nct : nct * kStages + claim;
        // ask for the next item's tile now: the answer's round trip overlaps
        // this item's copy and the wait for the next free stage
        if (item + 1 >= (uint32_t)kStages && t < T.ntiles) claim = atomicAdd(&T.work->next_tile, 1u);
        const uint32_t base = t < T.ntiles ? t * kBigTile : 0u;
        stile[q] = t < T.ntiles ? t : kEndTile;
        if (t >= T.ntiles || base + kBigTile > T.n) {
          mbar_arrive(&full[q]);  // the end of the set, or a partial tile read directly
          i++;
          if (t >= T.ntiles) break;
          continue;
        }
        FilterStage &d = stage[q];
        fence_proxy_async();
        mbar_expect_tx(&full[q], kBigTile * 8);
        bulk_g2s(d.gap, T.gap + base, kBigTile * 4, &full[q]);
        bulk_g2s(d.turn, T.turn + base, kBigTile * 2, &full[q]);
        bulk_g2s(d.flags, T.flags + base, kBigTile, &full[q]);
        bulk_g2s(d.tier, T.tier + base, kBigTile, &full[q]);
        issued |= 1u << q;
        lastph = (lastph & ~(1u << q)) | (((i / kStages) & 1) << q);
        i++;
      }
      // the consumers may use the stage memory for this set's finish: the next
      // set's copies wait until they are done with it
      if (!failed && s + sstep < n_sets) {
        if (!mbar_wait_bounded(&sdone, nsets & 1)) {
          failed = true;
          sfail = s;
        }
        nsets++;
      }
    }
    if (failed) {
      set_status(sets[sfail], UNISON_ERR_TIMEOUT);
      // consumers that still wait will time out too; let this CTA's copies land
      // before the CTA exits
      for (int q = 0; q < kStages; q++)
        if ((issued >> q) & 1) mbar_wait_bounded(&full[q], (lastph >> q) & 1);
    }
    return;
  }

  // ---------------- consumer warps
  const uint32_t ct = threadIdx.x;
  SetConst &c = cset;
  uint32_t i = 0;    // the CTA's running stage count (the producer's sequence)
  for (int s = s0; s < n_sets; s += sstep) {
    // the set's descriptor in shared memory: its fields are read throughout
    // the set's phases, each read from global memory a round trip.  The
    // tables come in the same round trip when the map names them.
    static_assert(sizeof(RankSet) % 8 == 0, "copied in 8-byte words");
    for (uint32_t w = ct; w < sizeof(RankSet) / 8; w += kConsumers)
      reinterpret_cast<uint64_t *>(&rset)[w] = reinterpret_cast<const uint64_t *>(sets + s)[w];
    if (tab0 && ct < kLutN) {
      t2s[ct] = tab0->t2v[ct];
      mgs[ct] = tab0->mgv[ct];
      sgs[ct] = tab0->sigma[ct];
    }
    consumers_sync();
    const RankSet &S = rset;
    const uint32_t r = sequential ? 0u : blockIdx.x - S.cta0;
    if (!tab0) {
      if (ct < kLutN) {
        t2s[ct] = S.tab->t2v[ct];
        mgs[ct] = S.tab->mgv[ct];
        sgs[ct] = S.tab->sigma[ct];
      }
      consumers_sync();
    }
    if (S.direct) {
      // no thresholds and no streaming: CTA r collects every eligible record's
      // value of list r and finishes the list
      const int local = (int)collect_list(S, (int)r, fin, t2s, mgs, u.s);
      const bool last = finish_list(S, (int)r, fin, t2s, mgs, u.s, c, local);
      if (last) finish_set(S, fin);
      return;
    }
    // 1. thresholds: the sampling CTAs sample; every CTA cuts the histograms
    if (r < S.sctas) sample_share(S, r, t2s, mgs);
#ifdef UNISON_DEBUG_HOOKS
    if (s == g_hook_flag_set) wait_word(S, &S.work->dummy, 1u);  // nothing sets it: runs out
#endif
    if (S.sctas) wait_word(S, &S.work->sample_ticket, S.sctas);
    if (ct < kLists) ccnt_s[ct] = 0;  // published by the barriers below
    thresholds(S, t2s, sgs, vd, pp, c);
    const uint32_t s_n = S.n;
    const bool s_keys = S.keys != nullptr;
    // Segment: a run of tiles over which every index condition of the set has
    // one class (all, none or mixed).  Within a set each condition changes
    // class at most twice (at the tile holding its boundary and the one
    // after), so a set has at most 13 segments.  A CTA's tiles come in
    // rising order.
    uint32_t seg_end = 0;  // first tile of the next segment
    bool seg_mixed = false, seg_none = false;
#ifdef UNISON_DEBUG_HOOKS
    bool first_tile = true;
#endif
    // 2. stream the tiles the group's counter hands this CTA: at most all of
    // the set's tiles and the end mark.  A wait that runs out ends the CTA's
    // streaming (its set's results are then undefined, and its status says so).
    for (uint32_t items = 0; items <= S.ntiles; items++, i++) {
      const int q = (int)(i % kStages);
#ifdef UNISON_DEBUG_HOOKS
      // a barrier nothing arrives at: the bounded wait runs out and reports
      if (first_tile && s == g_hook_mbar_set) wait_phase_uniform(S, &dummy_bar, 0, kWaitNs);
#endif
      if (!wait_phase_uniform(S, &full[q], (i / kStages) & 1)) {
        i++;
        break;
      }
      const uint32_t t = stile[q];
      if (t == kEndTile) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[q]);
        i++;
        break;
      }
      const uint32_t tb = t * kBigTile;
      if (t >= seg_end) {
        // Index conditions over this tile: record indices rise through the
        // tile, so lo = ~index falls from lo_hi to lo_lo and each tie condition
        // on lo holds for all, none or a part of the tile.
        const uint32_t tcount = min(kBigTile, s_n - tb);
        const uint32_t gtb = S.off + tb;  // the tile's first index in the whole set
        const uint32_t lo_hi = (~gtb) & kIdMask, lo_lo = (~(gtb + tcount - 1)) & kIdMask;
        // 0 none, 1 all, 2 mixed
        auto ge_class = [&](uint32_t x) { return lo_lo >= x ? 1u : (lo_hi < x ? 0u : 2u); };                   // lo >= x
        auto le_class = [&](int64_t x) { return (int64_t)lo_hi <= x ? 1u : ((int64_t)lo_lo > x ? 0u : 2u); };  // lo <= x
        const uint32_t iV = ge_class(c.loV), iD = ge_class(c.loD), iP = le_class((int64_t)c.loP);
        const uint32_t dV = ge_class(c.dV), dD = ge_class(c.dD), dP = le_class((int64_t)c.dP);
        seg_mixed = ((c.act & 1) && (iV == 2 || dV == 2)) || ((c.act & 2) && (iD == 2 || dD == 2)) ||
                    ((c.act & 4) && (iP == 2 || dP == 2));
        // next tile where a condition can change class: lo >= x holds for
        // indices up to kIdMask - x, lo <= x from kIdMask - x on; the change
        // points are the tile holding that index and the tile after it
        uint32_t nxt = S.ntiles;
        auto upd = [&](int64_t lo_bound) {
          const int64_t b = (int64_t)kIdMask - lo_bound - S.off;  // a local index
          if (b < 0 || b >= (int64_t)s_n) return;
          const uint32_t tbnd = (uint32_t)b / kBigTile;
          if (tbnd > t) nxt = min(nxt, tbnd);
          else if (tbnd + 1 > t) nxt = min(nxt, tbnd + 1);
        };
        upd(c.loV); upd(c.loD); upd(c.loP); upd(c.dV); upd(c.dD); upd(c.dP);
        seg_end = nxt;
        // Per-segment bound table over (turn index, record class): a record of
        // class cls at turn index t may be a candidate of some list iff
        // g >= x or g < y.  Classes: 0 not eligible, 1 live fast tier, 2 live
        // HBM tier, 3 completed fast tier, 4 completed HBM tier.
        consumers_sync();  // everyone is done with the previous table
        bool live = false;
        if (!seg_mixed && ct < kLutN * 5) {
          const uint32_t tt = ct / 5, cls = ct % 5;
          const uint4 a = vd[tt];
          const uint2 bb = pp[tt];
          const uint32_t bV = iV == 1 ? a.x : a.y, bD = iD == 1 ? a.z : a.w, bP = iP == 1 ? bb.y : bb.x;
          const bool pdV = (c.act & 1) && dV == 1, pdD = (c.act & 2) && dD == 1, pdP = (c.act & 4) && dP == 1;
          uint2 e = make_uint2(kFull, 0u);
          if (cls == 1) e = make_uint2(min(bV, bD), 0u);
          if (cls == 2) e = make_uint2(bV, bP);
          if (cls == 3) e = make_uint2(pdV || pdD ? 0u : kFull, 0u);
          if (cls == 4) e = make_uint2(pdV ? 0u : kFull, pdP ? kFull : 0u);
          u.f.ftab[ct] = e;
          // gaps are below 2^31: x >= 2^31 and y == 0 admit nothing
          live = e.x < 0x80000000u || e.y != 0u;
        }
        seg_none = !consumers_sync_or(live) && !seg_mixed;
      }
      const bool bulk = tb + kBigTile <= s_n;
      uint32_t g[kRec], tw[kRec / 2], fw[kGroups], rw[kGroups];
      if (bulk) {
        const FilterStage &d = stage[q];
#pragma unroll
        for (int gi = 0; gi < (int)kGroups; gi++) {
          const uint32_t o = gi * kGroupStride + 4 * ct;
          const uint4 gq = *reinterpret_cast<const uint4 *>(d.gap + o);
          g[4 * gi] = gq.x; g[4 * gi + 1] = gq.y; g[4 * gi + 2] = gq.z; g[4 * gi + 3] = gq.w;
          const uint2 tq = *reinterpret_cast<const uint2 *>(d.turn + o);
          tw[2 * gi] = tq.x; tw[2 * gi + 1] = tq.y;
          fw[gi] = *reinterpret_cast<const uint32_t *>(d.flags + o);
          rw[gi] = *reinterpret_cast<const uint32_t *>(d.tier + o);
        }
      } else {
#pragma unroll
        for (int gi = 0; gi < (int)kGroups; gi++) {
          tw[2 * gi] = tw[2 * gi + 1] = 0;
          fw[gi] = 0x01010101u;  // padding reads as pinned: never eligible
          rw[gi] = 0;
#pragma unroll
          for (uint32_t m = 0; m < 4; m++) {
            const uint32_t idx = tb + gi * kGroupStride + 4 * ct + m;
            g[4 * gi + m] = 0;
            if (idx < s_n) {
              g[4 * gi + m] = S.gap[idx];
              tw[2 * gi + (m >> 1)] |= (uint32_t)S.turn[idx] << (16 * (m & 1));
              const uint32_t sh = 8 * m;
              fw[gi] = (fw[gi] & ~(0xFFu << sh)) | ((uint32_t)S.flags[idx] << sh);
              rw[gi] = (rw[gi] & ~(0xFFu << sh)) | ((uint32_t)S.tier[idx] << sh);
            }
          }
        }
      }
#ifdef UNISON_DEBUG_HOOKS
      first_tile = false;
#endif
      auto turn_of = [&](uint32_t k) { return min((tw[k >> 1] >> (16 * (k & 1))) & 0xFFFF, kTMax); };
      auto index_of = [&](uint32_t k) { return tb + (k >> 2) * kGroupStride + 4 * ct + (k & 3); };
      // candidate bit per record (any list): one table lookup per record
      uint32_t cm = 0;
      if (seg_mixed) {
        // index conditions vary inside the tile: flag the records that pass
        // some list exactly
#pragma unroll
        for (uint32_t k = 0; k < kRec; k++) {
          const uint32_t sh = 8 * (k & 3);
          const uint32_t fl = (fw[k >> 2] >> sh) & 0xFF, tr = (rw[k >> 2] >> sh) & 0xFF;
          const uint32_t em = elig_mask((uint8_t)fl, (uint8_t)tr);
          const bool done = (fl & 2) != 0;
          const uint32_t gg = g[k], tt = turn_of(k), lo = (~(S.off + index_of(k))) & kIdMask;
          const uint4 a = vd[tt];
          const uint2 b = pp[tt];
          const bool pV = (em & 1) && (done ? lo >= c.dV : (gg >= a.y || (gg >= a.x && lo >= c.loV)));
          const bool pD = (em & 2) && (done ? lo >= c.dD : (gg >= a.w || (gg >= a.z && lo >= c.loD)));
          const bool pP = (em & 4) && (done ? (int32_t)lo <= c.dP : (gg < b.x || (gg < b.y && lo <= c.loP)));
          cm |= (uint32_t)(pV || pD || pP) << k;
        }
      } else if (!seg_none) {
        const unsigned char *tab = reinterpret_cast<const unsigned char *>(u.f.ftab);
#pragma unroll
        for (int gi = 0; gi < (int)kGroups; gi++) {
          // class * 8 per record, four records per word (SWAR)
          const uint32_t unp = __vcmpeq4(fw[gi] & 0x01010101u, 0u);
          const uint32_t isS = __vcmpeq4(rw[gi], 0x01010101u), isH = __vcmpeq4(rw[gi], 0x02020202u);
          const uint32_t dn = __vcmpne4(fw[gi] & 0x02020202u, 0u);
          const uint32_t c8 = (unp & ((isS & 0x08080808u) | (isH & 0x10101010u))) +
                              (unp & dn & (isS | isH) & 0x10101010u);
#pragma unroll
          for (uint32_t m = 0; m < 4; m++) {
            const uint32_t k = 4 * gi + m;
            const uint2 e = *reinterpret_cast<const uint2 *>(tab + turn_of(k) * 40 + ((c8 >> (8 * m)) & 0xFF));
            cm |= (uint32_t)(g[k] >= e.x || g[k] < e.y) << k;
          }
        }
      }
      // every record's key, when asked for (from registers)
      if (s_keys) {
#pragma unroll
        for (uint32_t k = 0; k < kRec; k++) {
          const uint32_t idx = index_of(k);
          if (idx < s_n) {
            const bool dn = (fw[k >> 2] >> (8 * (k & 3) + 1)) & 1;
            S.keys[idx] = score_of(g[k], turn_of(k), dn, t2s, mgs);
          }
        }
      }
      // The stage is handed back as soon as this warp no longer reads it: at
      // once when none of its records is flagged, else after the exact tests
      // below, which read the flagged records back from the stage.
      const bool flagged = __any_sync(kFull, cm != 0);
      if (!flagged) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[q]);
        continue;
      }
      // exact per-list tests of the flagged records: the warp lists their
      // offsets in the tile (kWarpBuf a pass), then each lane tests one and
      // appends its exact value to every list it passes (one atomic per warp
      // and list, the lists' atomics in flight together).  When the last
      // records tested are in registers the stage is handed back before the
      // appends, whose atomics then overlap the stage's next copy.
      uint16_t *wb = u.f.wbuf[ct >> 5];
      const FilterStage &d = stage[q];
      uint32_t rem = cm;
      bool released = false;
      while (__any_sync(kFull, rem != 0)) {
        const uint32_t mine = __popc(rem);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        const uint32_t nb = min(__shfl_sync(kFull, incl, 31), kWarpBuf);
        uint32_t pos = incl - mine, wrote = 0;
        for (uint32_t m = rem; m != 0 && pos < kWarpBuf; m &= m - 1, pos++) {
          const uint32_t k = __ffs(m) - 1;
          wb[pos] = (uint16_t)((k >> 2) * kGroupStride + 4 * ct + (k & 3));
          wrote |= 1u << k;
        }
        rem &= ~wrote;
        const bool more = __any_sync(kFull, rem != 0);  // another pass follows
        __syncwarp();
        for (uint32_t j0 = 0; j0 < nb; j0 += 32) {
          const uint32_t j = j0 + lane;
          bool pL[kLists] = {false, false, false};
          uint64_t ck = 0;
          if (j < nb) {
            const uint32_t o = wb[j], idx = tb + o;
            uint32_t gg, tt, fl, tr;
            if (bulk) {
              gg = d.gap[o];
              tt = d.turn[o];
              fl = d.flags[o];
              tr = d.tier[o];
            } else {  // the partial last tile: read from the set (padding is pinned)
              const bool in = idx < s_n;
              gg = in ? S.gap[idx] : 0u;
              tt = in ? S.turn[idx] : 0u;
              fl = in ? S.flags[idx] : 1u;
              tr = in ? S.tier[idx] : 0u;
            }
            tt = min(tt, kTMax);
            const uint32_t em = elig_mask((uint8_t)fl, (uint8_t)tr);
            const bool done = (fl & 2) != 0;
            const uint32_t lo = (~(S.off + idx)) & kIdMask;
            const uint4 a = vd[tt];
            const uint2 b = pp[tt];
            pL[0] = (em & 1) && (done ? lo >= c.dV : (gg >= a.y || (gg >= a.x && lo >= c.loV)));
            pL[1] = (em & 2) && (done ? lo >= c.dD : (gg >= a.w || (gg >= a.z && lo >= c.loD)));
            pL[2] = (em & 4) && (done ? (int32_t)lo <= c.dP : (gg < b.x || (gg < b.y && lo <= c.loP)));
            if (pL[0] || pL[1] || pL[2]) ck = ck_of(score_of(gg, tt, done, t2s, mgs), S.off + idx);
          }
          if (!more && j0 + 32 >= nb) {  // the warp's last reads of the stage are done
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[q]);
            released = true;
          }
          unsigned bal[kLists], base[kLists];
#pragma unroll
          for (int L = 0; L < kLists; L++) {
            bal[L] = __ballot_sync(kFull, pL[L]);
            base[L] = 0;
          }
          if (lane == 0) {
#pragma unroll
            for (int L = 0; L < kLists; L++)
              if (bal[L]) base[L] = atomicAdd(&ccnt_s[L], (unsigned)__popc(bal[L]));
          }
#pragma unroll
          for (int L = 0; L < kLists; L++) {
            if (!bal[L]) continue;
            const uint32_t lt = (1u << lane) - 1;
            const uint32_t at = __shfl_sync(kFull, base[L], 0) + __popc(bal[L] & lt);
            const uint64_t v = list_val(ck, L);
            if (pL[L] && at < S.cr) S.creg[((size_t)L * S.nctas + r) * S.cr + at] = v;
            // past the end of the CTA's region: straight into the set's list
            const unsigned ovf = __ballot_sync(kFull, pL[L] && at >= S.cr);
            if (ovf) {
              unsigned ob = 0;
              if (lane == 0) ob = atomicAdd(&S.work->cand[L], (unsigned)__popc(ovf));
              ob = __shfl_sync(kFull, ob, 0) + __popc(ovf & lt);
              if (pL[L] && at >= S.cr && ob < S.ccap) S.cand[(size_t)L * S.ccap + ob] = v;
            }
          }
        }
        __syncwarp();  // the buffer is rewritten by the next pass
      }
      if (!released && lane == 0) mbar_arrive(&empty[q]);
    }
    // 3. done streaming: the last three CTAs of the group take one list each
    // (a group of fewer CTAs: the last one takes the rest), once every CTA of
    // the group has emitted its candidates; the last list's CTA runs the fill
    // the CTA's region moves to the set's list: one range taken per list
    // (the three atomics in flight together), then copied
    consumers_sync();  // every warp's appends counted
    if (ct < kLists) {
      const uint32_t nr = min(ccnt_s[ct], S.cr);
      cbase_s[ct] = nr ? atomicAdd(&S.work->cand[ct], nr) : 0u;
    }
    consumers_sync();
#pragma unroll 1
    for (int L = 0; L < kLists; L++) {
      const uint32_t nr = min(ccnt_s[L], S.cr), b0 = cbase_s[L];
      const uint64_t *rg = S.creg + ((size_t)L * S.nctas + r) * S.cr;
      for (uint32_t j = ct; j < nr; j += kConsumers)
        if (b0 + j < S.ccap) S.cand[(size_t)L * S.ccap + b0 + j] = __ldcg(rg + j);
    }
    __threadfence();
    consumers_sync();
    if (ct == 0) {
      arrival = atomicAdd(&S.work->done_ctas, 1u);
      __threadfence();  // the earlier arrivals' candidates are visible after this
    }
    consumers_sync();
    const uint32_t nct = sequential ? 1u : S.nctas;
    const uint32_t qr = nct - 1 - arrival;
    uint32_t mine = 0;
#pragma unroll
    for (int L = 0; L < kLists; L++)
      if ((uint32_t)L == qr || (qr == 0 && (uint32_t)L >= nct)) mine |= 1u << L;
    if (mine) {
      if (qr > 0) wait_word(S, &S.work->done_ctas, nct);
      bool last = false;
#pragma unroll 1
      for (int L = 0; L < kLists; L++)
        if ((mine >> L) & 1) last = finish_list(S, L, fin, t2s, mgs, u.s, c);
      if (last) finish_set(S, fin);
    }
    // 4. the stage memory is free for the next set's copies
    consumers_sync();
    if (ct == 0) mbar_arrive(&sdone);
  }
}

// ------------------------------------------------------------- merge ----
// The shards' candidate lists, gathered (n_shards buffers of `stride` bytes
// each): CTA L selects list L's global top M (narrowed and sorted as in the
// finish, carrying the sizes), writes it as the finish does, and the last list's CTA runs the
// fill.  One CTA per list, consumer-sized (256 threads).
__global__ void __launch_bounds__(kConsumers) rank_merge_kernel(const __grid_constant__ RankSet desc,
                                                                const unsigned char *gathered, int n_shards,
                                                                uint64_t stride, uint4 *zero, uint32_t n_zero) {
  extern __shared__ __align__(128) unsigned char dsm[];
  uint64_t *fin = reinterpret_cast<uint64_t *>(dsm);
  __shared__ SelectScratch ss;
  __shared__ unsigned int pre[kMaxShards + 1];
  __shared__ unsigned int last;
  const RankSet &S = desc;
  for (uint32_t w = blockIdx.x * kConsumers + threadIdx.x; w < n_zero; w += kLists * kConsumers)
    zero[w] = make_uint4(0u, 0u, 0u, 0u);
  const int L = blockIdx.x;
  const uint32_t Mw = L == 0 ? S.k : S.max_moves;
  const bool active = (S.act >> L) & 1;
  const size_t loff = cand_list_off(S.k, S.max_moves, L);
  if (threadIdx.x == 0) {
    pre[0] = 0;
    for (int sh = 0; sh < n_shards; sh++) {
      const CandHeader *h = reinterpret_cast<const CandHeader *>(gathered + stride * sh);
      pre[sh + 1] = pre[sh] + min(h->count[L], Mw);
      if (h->status) set_status(S, (int)h->status);
    }
  }
  ss.hist[threadIdx.x] = 0;
  consumers_sync();
  const uint32_t c = pre[n_shards];
  const uint32_t M = active ? min(Mw, c) : 0u;
  auto entry = [&](uint32_t i) -> const CandEntry & {
    uint32_t lo = 0, hi = (uint32_t)n_shards - 1;  // the shard holding entry i: pre[sh] <= i < pre[sh + 1]
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (pre[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return reinterpret_cast<const CandEntry *>(gathered + stride * lo + loff)[i - pre[lo]];
  };
  uint64_t *val = fin;                                       // [kMaxSel]
  uint32_t *szs = reinterpret_cast<uint32_t *>(fin + kMaxSel);  // [kMaxSel]
  uint32_t got = 0;
  if (M > 0) {
    uint64_t *tval = fin + 3 * kMaxSel / 2;  // copies of both
    uint32_t *tszs = reinterpret_cast<uint32_t *>(fin + 5 * kMaxSel / 2);
    // fn(entry, ok) over every entry, eight independent reads a thread in flight
    auto each_entry = [&](auto fn) {
      for (uint32_t base = 0; base < c; base += 8 * kConsumers) {
        CandEntry e[8];
#pragma unroll
        for (uint32_t u = 0; u < 8; u++) {
          const uint32_t i = base + u * kConsumers + threadIdx.x;
          e[u] = i < c ? entry(i) : CandEntry{0ull, 0u, 0u};
        }
#pragma unroll
        for (uint32_t u = 0; u < 8; u++) fn(e[u], base + u * kConsumers + threadIdx.x < c);
      }
    };
    // as in finish_list: t rises until few entries beyond M are at or above it
    uint64_t t = 0;
    int sh = 64;
    uint32_t need = M, left = c;
    while (left > kMaxSel && sh > 0) {
      const uint32_t in = narrow(
          [&](auto fn) {
            each_entry([&](const CandEntry &e, bool ok) {
              if (ok) fn(e.v);
            });
          },
          t, sh, need, ss);
      left = M - need + in;
    }
    if (threadIdx.x == 0) ss.cnt = 0;
    consumers_sync();
    each_entry([&](const CandEntry &e, bool ok) {
      if (ok && e.v >= t) {
        const uint32_t pos = atomicAdd(&ss.cnt, 1u);
        if (pos < kMaxSel) {
          val[pos] = e.v;
          szs[pos] = e.kv;
        }
      }
    });
    consumers_sync();
    uint32_t keepn = min(ss.cnt, kMaxSel);
    consumers_sync();
    left = keepn;
    while (left > M + slack(M) && sh > 0) {
      const uint32_t in = narrow(
          [&](auto fn) {
            for (uint32_t i = threadIdx.x; i < keepn; i += kConsumers) fn(val[i]);
          },
          t, sh, need, ss);
      left = M - need + in;
    }
    if (left < keepn) {
      if (threadIdx.x == 0) ss.cnt = 0;
      consumers_sync();
      for (uint32_t i = threadIdx.x; i < keepn; i += kConsumers)
        if (val[i] >= t) {
          const uint32_t pos = atomicAdd(&ss.cnt, 1u);
          tval[pos] = val[i];
          tszs[pos] = szs[i];
        }
      consumers_sync();
      keepn = left;
      for (uint32_t i = threadIdx.x; i < keepn; i += kConsumers) {
        val[i] = tval[i];
        szs[i] = tszs[i];
      }
      consumers_sync();
    }
    sort_desc(val, keepn, tval, ss, szs, tszs);
    got = min(keepn, M);
    for (uint32_t i = threadIdx.x; i < got; i += kConsumers) {
      S.sorted[(size_t)L * kMaxSel + i] = val[i];
      if (L == 0) S.victims[i] = (~(uint32_t)val[i]) & kIdMask;
      else S.ssz[(size_t)L * kMaxSel + i] = szs[i];
    }
  }
  if (threadIdx.x == 0) S.work->got[L] = got;
  __threadfence();
  consumers_sync();
  if (threadIdx.x == 0) last = (atomicAdd(&S.work->list_ticket, 1u) == (unsigned)kLists - 1);
  consumers_sync();
  if (last) fill(S, fin);
}

// ------------------------------------------------------------ host side ----
size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Device scratch of the ranking calls, kept per (device, stream) and grown
// when a call needs more: calls on one stream run in order, so each reuses
// the buffers after the previous one is done with them (stream order), and
// calls on different streams get different buffers.  Held for the life of
// the process.  The stream handle is the key: a stream must outlive the
// ranking calls queued on it (a new stream that reuses a destroyed one's
// handle would otherwise share its scratch without being ordered after it).
// Per key: the calls' working scratch, and blocks for the state that a call
// must find zero (work words, then the sampled sets' histograms).  Calls
// alternate between two; each zeroes what the one before it used, so a
// block is all zero when its turn comes, whatever the calls' sizes, and no
// clearing precedes a launch (a memset and the upload of a single set's
// descriptor took about 10 of a call's 52 us at 2^20 records).
struct Scratch {
  char *p = nullptr;
  size_t bytes = 0;
};
// The stream's last call of several sets: one whose arguments are byte for
// byte the same finds its descriptors (once per block), tables and scratch
// layout already on the device and only launches.  Any other use of the
// working scratch drops it.
struct RankPlan {
  std::vector<unsigned char> key;
  size_t desc_b = 0, cmap_off = 0, tabs_off = 0;
  size_t zero_b = 0;  // bytes of a block that the call uses
  uint32_t grid = 0;
  int sequential = 0;
  bool packed = false;
  RankPack<kPackSets> pack[2];  // for each block
};
struct StreamState {
  int dev = 0;
  std::mutex mu;  // held from the choice of a block to the launch that uses it
  Scratch main, zero[2];
  size_t dirty[2] = {0, 0};  // bytes from a block's start that are not zero
  bool planned = false;
  RankPlan plan;
  // the last tables built, and what they were built from
  bool have_tab = false;
  uint16_t tab_sigma[kLutN];
  uint64_t tab_penalty = 0;
  RankTab tab;
};
std::mutex g_state_mu;
std::map<std::pair<int, cudaStream_t>, std::unique_ptr<StreamState>> g_state;

StreamState *stream_state(cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_state_mu);
  auto &e = g_state[std::make_pair(dev, stream)];
  if (!e) {
    e.reset(new StreamState());
    e->dev = dev;
  }
  return e.get();
}

int grow(Scratch &e, size_t bytes, bool zero, cudaStream_t stream) {
  if (e.bytes >= bytes) return UNISON_OK;
  if (e.p) cudaFreeAsync(e.p, stream);  // ordered after the calls that used it
  e.p = nullptr;
  e.bytes = 0;
  char *p = nullptr;
  if (unison_fault_alloc() || cudaMallocAsync(reinterpret_cast<void **>(&p), bytes, stream) != cudaSuccess) {
    cudaGetLastError();
    return UNISON_ERR_OOM;
  }
  if (zero && cudaMemsetAsync(p, 0, bytes, stream) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeAsync(p, stream);
    return UNISON_ERR_CUDA;
  }
  e.p = p;
  e.bytes = bytes;
  return UNISON_OK;
}

// The zero blocks at least `bytes` long (a new block is zero).
int grow_zero(StreamState &st, size_t bytes, cudaStream_t stream) {
  for (int i = 0; i < 2; i++) {
    if (st.zero[i].bytes >= bytes) continue;
    st.dirty[i] = 0;
    st.planned = false;  // the plan's descriptors name the old block
    const int rc = grow(st.zero[i], bytes, true, stream);
    if (rc != UNISON_OK) return rc;
  }
  return UNISON_OK;
}

// Memory of captured calls.  A call captured into a graph runs whenever the
// graph does, any number of times, on any stream and between any other calls,
// so it shares nothing with them: its scratch, its work words and histograms
// (cleared by a node of the graph) and the descriptors, tables and CTA map that
// do not go with the launch (written once, here: they never change) lie in
// memory of its own, which stays where it is.  The graph and every executable
// made from it hold that memory by a user object; when the last of them is gone
// its destructor, which may not call CUDA, leaves the memory on a list that the
// device's next ranking call frees.
struct GraphMem {
  char *p;
  int dev;
  GraphMem *next;
};
struct GraphPool {
  std::mutex mu;
  GraphMem *unused = nullptr;
  std::atomic<bool> any{false};  // something in the list
  cudaStream_t side[64] = {};    // for the memory's allocation and uploads
};
GraphPool &graph_pool() {
  static GraphPool *const g = new GraphPool;  // outlives the last graph
  return *g;
}
void CUDART_CB graph_gone(void *mem) {
  GraphPool &g = graph_pool();
  GraphMem *const m = static_cast<GraphMem *>(mem);
  std::lock_guard<std::mutex> lock(g.mu);
  m->next = g.unused;
  g.unused = m;
  g.any.store(true, std::memory_order_release);
}

// Frees, in `stream`'s order, the memory of the device's graphs that are gone.
void free_unused(int dev, cudaStream_t stream) {
  GraphPool &g = graph_pool();
  if (!g.any.load(std::memory_order_acquire)) return;
  GraphMem *mine = nullptr;
  {
    std::lock_guard<std::mutex> lock(g.mu);
    for (GraphMem **at = &g.unused; *at;) {
      GraphMem *const m = *at;
      if (m->dev != dev) {
        at = &m->next;
        continue;
      }
      *at = m->next;
      m->next = mine;
      mine = m;
    }
    g.any.store(g.unused != nullptr, std::memory_order_release);
  }
  while (mine) {
    GraphMem *const m = mine;
    mine = m->next;
    if (cudaFreeAsync(m->p, stream) != cudaSuccess) cudaGetLastError();
    delete m;
  }
}

// While a capture is under way its thread may allocate and wait only in this
// mode, on streams that are not captured.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Memory for one captured call, held by `graph`.
int graph_alloc(size_t bytes, cudaGraph_t graph, char **out) {
  GraphPool &g = graph_pool();
  RelaxedCapture relaxed;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return UNISON_ERR_CUDA;
  }
  cudaStream_t side = nullptr;
  {
    std::lock_guard<std::mutex> lock(g.mu);
    if (!g.side[dev] && cudaStreamCreateWithFlags(&g.side[dev], cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      g.side[dev] = nullptr;
      return UNISON_ERR_CUDA;
    }
    side = g.side[dev];
  }
  free_unused(dev, side);
  GraphMem *const m = new (std::nothrow) GraphMem{nullptr, dev, nullptr};
  if (!m) return UNISON_ERR_OOM;
  if (unison_fault_alloc() || cudaMallocAsync(reinterpret_cast<void **>(&m->p), bytes, side) != cudaSuccess) {
    cudaGetLastError();
    delete m;
    return UNISON_ERR_OOM;
  }
  cudaUserObject_t held = nullptr;
  if (cudaStreamSynchronize(side) != cudaSuccess ||
      cudaUserObjectCreate(&held, m, graph_gone, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeAsync(m->p, side);
    delete m;
    return UNISON_ERR_CUDA;
  }
  if (cudaGraphRetainUserObject(graph, held, 1, cudaGraphUserObjectMove) != cudaSuccess) {
    cudaGetLastError();
    cudaUserObjectRelease(held, 1);  // its destructor takes the memory
    return UNISON_ERR_CUDA;
  }
  *out = m->p;
  return UNISON_OK;
}

// Fills [dst, dst + bytes) of a captured call's memory from host memory, now.
int graph_write(char *dst, const void *src, size_t bytes) {
  RelaxedCapture relaxed;
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
    cudaStream_t side = nullptr;
    {
      std::lock_guard<std::mutex> lock(graph_pool().mu);
      side = graph_pool().side[dev];  // made by graph_alloc
    }
    if (side && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, side) == cudaSuccess &&
        cudaStreamSynchronize(side) == cudaSuccess)
      return UNISON_OK;
  }
  cudaGetLastError();
  return UNISON_ERR_CUDA;
}

// Whether `stream` is being captured, and into which graph.
int capture_of(cudaStream_t stream, bool *captured, cudaGraph_t *graph) {
  *captured = false;
  *graph = nullptr;
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &s) != cudaSuccess) {
    cudaGetLastError();  // (the legacy stream beside a capture: its launches are refused)
    return UNISON_OK;
  }
  if (s == cudaStreamCaptureStatusNone) return UNISON_OK;
  if (s != cudaStreamCaptureStatusActive ||
      cudaStreamGetCaptureInfo(stream, &s, nullptr, graph, nullptr, nullptr, nullptr) != cudaSuccess || !*graph) {
    cudaGetLastError();
    return UNISON_ERR_CUDA;  // a capture that failed already
  }
  *captured = true;
  return UNISON_OK;
}

// Pinned host staging for the per-call upload, a ring of buffers per device.
// A buffer is handed out only after the copy that last read it has finished
// (its event); staging_release() ends the caller's hold.
struct Staging {
  unsigned char *host = nullptr;
  size_t cap = 0;
  cudaEvent_t done = nullptr;
};
constexpr int kStagingRing = 8;
std::mutex g_staging_mu;
Staging g_staging[64][kStagingRing];
int g_staging_next[64] = {};

int staging_acquire(size_t bytes, unsigned char **host, cudaEvent_t *done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return UNISON_ERR_CUDA;
  }
  g_staging_mu.lock();
  Staging &b = g_staging[dev][g_staging_next[dev]];
  g_staging_next[dev] = (g_staging_next[dev] + 1) % kStagingRing;
  if (b.done && cudaEventSynchronize(b.done) != cudaSuccess) {
    cudaGetLastError();
    g_staging_mu.unlock();
    return UNISON_ERR_CUDA;
  }
  if (!b.done && cudaEventCreateWithFlags(&b.done, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    b.done = nullptr;
    g_staging_mu.unlock();
    return UNISON_ERR_CUDA;
  }
  if (b.cap < bytes) {
    if (b.host) cudaFreeHost(b.host);
    b.host = nullptr;
    b.cap = 0;
    const size_t cap = std::max<size_t>(bytes, 64 << 10);
    if (cudaMallocHost(reinterpret_cast<void **>(&b.host), cap) != cudaSuccess) {
      cudaGetLastError();
      b.host = nullptr;
      g_staging_mu.unlock();
      return UNISON_ERR_OOM;
    }
    b.cap = cap;
  }
  *host = b.host;
  *done = b.done;
  return UNISON_OK;  // the lock is held until staging_release()
}
void staging_release() { g_staging_mu.unlock(); }

// Kernel attributes and the grid (every CTA resident at once), set up once
// per device (the attributes belong to the device's context).
struct LaunchCfg {
  bool ok = false;
  uint32_t ctas = 0;
};
const LaunchCfg &launch_cfg() {
  static std::mutex mu;
  static LaunchCfg cfgs[64];
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    static LaunchCfg bad;
    return bad;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev]) {
    LaunchCfg c;
    int n_sm = 0, per_sm = 0, per_sm64 = 0, coop = 0;
    c.ok = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
           cudaFuncSetAttribute(rank_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynSmem) ==
               cudaSuccess &&
           cudaFuncSetAttribute(rank_kernel<kPackSets>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynSmem) ==
               cudaSuccess &&
           cudaFuncSetAttribute(rank_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMergeSmem) ==
               cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rank_kernel<1>, kCtaThreads, kDynSmem) ==
               cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm64, rank_kernel<kPackSets>, kCtaThreads, kDynSmem) ==
               cudaSuccess &&
           per_sm > 0 && per_sm64 >= per_sm;
    if (!c.ok) cudaGetLastError();
    c.ctas = (uint32_t)std::min(std::max(1, n_sm * per_sm), (int)kMaxGroup);
    cfgs[dev] = c;
    done[dev] = c.ok;
  }
  return cfgs[dev];
}

}  // namespace

#ifdef UNISON_DEBUG_HOOKS
// Test hooks of the debug build (absent from the default build): the next
// ranking calls' threshold wait of set flag_set first waits on a flag that
// nothing sets, and the first tile wait of set mbar_set first waits on a
// barrier nothing arrives at; both bounded waits run out and report
// UNISON_ERR_TIMEOUT in that set's counts[3].  -1 turns a hook off.
extern "C" int unison_debug_rank_wait_hooks(int flag_set, int mbar_set) {
  if (cudaMemcpyToSymbol(g_hook_flag_set, &flag_set, sizeof(int)) != cudaSuccess ||
      cudaMemcpyToSymbol(g_hook_mbar_set, &mbar_set, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return UNISON_ERR_CUDA;
  }
  return UNISON_OK;
}

// Leaves an error pending in the library's CUDA runtime, as a call that failed
// without clearing it would.  Nothing reaches the device.
extern "C" int unison_debug_leave_error(void) {
  return cudaSetDevice(-1) != cudaSuccess && cudaPeekAtLastError() != cudaSuccess ? UNISON_OK : UNISON_ERR_CUDA;
}
#endif

namespace {

// The call's arguments, byte for byte: what a plan is kept for.
void plan_key(std::vector<unsigned char> &k, const unison_records *sets, const unison_rank_params *params,
              const unison_rank_out *outs, int n_sets, uint32_t off, const unsigned char *cands) {
  k.clear();
  auto put = [&](const void *q, size_t b) {
    const unsigned char *c = static_cast<const unsigned char *>(q);
    k.insert(k.end(), c, c + b);
  };
  put(&n_sets, sizeof n_sets);
  put(&off, sizeof off);
  put(&cands, sizeof cands);
  put(sets, sizeof(unison_records) * n_sets);
  put(params, sizeof(unison_rank_params) * n_sets);
  if (!cands) put(outs, sizeof(unison_rank_out) * n_sets);
}

// Queues the kernel.  The verdict is the launch's own: cudaGetLastError() could
// name an older call's error although the kernel is queued and will leave its
// block dirty.
template <int kSets>
int queue_rank_kernel(uint32_t grid, const RankSet *d_sets, int n_sets, int sequential, const uint32_t *cmap,
                      const RankTab *tabs, const RankPack<kSets> &pack, char *other, size_t other_b,
                      cudaStream_t stream) {
  cudaError_t e;
  {
    ProfSpan span("rank", stream);
    cudaLaunchAttribute coop[1];
    coop[0].id = cudaLaunchAttributeCooperative;
    coop[0].val.cooperative = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(kCtaThreads);
    lc.dynamicSmemBytes = kDynSmem;
    lc.stream = stream;
    lc.attrs = coop;
    lc.numAttrs = 1;
    e = cudaLaunchKernelEx(&lc, rank_kernel<kSets>, d_sets, n_sets, sequential, cmap, tabs,
                           reinterpret_cast<uint4 *>(other), (uint32_t)(other_b / 16), pack);
  }
  count_launches(1);
  if (e == cudaSuccess) return UNISON_OK;
  cudaGetLastError();
  return UNISON_ERR_CUDA;  // nothing ran
}

// Launches a call on the zero block whose turn it is (zb: the bytes of it that
// the call uses), zeroing the other.  The caller holds st.mu and has passed
// that block (next_block) to the descriptors.
int next_block(const StreamState &st) { return st.dirty[0] == 0 ? 0 : 1; }
template <int kSets>
int launch_rank_kernel(StreamState &st, uint32_t grid, const RankSet *d_sets, int n_sets, int sequential,
                       const uint32_t *cmap, const RankTab *tabs, const RankPack<kSets> &pack, size_t zb,
                       cudaStream_t stream) {
  const int p = next_block(st);
  const int rc = queue_rank_kernel(grid, d_sets, n_sets, sequential, cmap, tabs, pack, st.zero[1 - p].p,
                                   st.dirty[1 - p], stream);
  if (rc != UNISON_OK) {
    st.planned = false;
    return rc;  // the blocks are as they were
  }
  st.dirty[p] = zb;
  st.dirty[1 - p] = 0;
  return UNISON_OK;
}

// A captured call: its own words are cleared by a node before the kernel's.
template <int kSets>
int capture_rank_kernel(uint32_t grid, const RankSet *d_sets, int n_sets, int sequential, const uint32_t *cmap,
                        const RankTab *tabs, const RankPack<kSets> &pack, char *words, size_t zb,
                        cudaStream_t stream) {
  if (cudaMemsetAsync(words, 0, zb, stream) != cudaSuccess) {
    cudaGetLastError();
    return UNISON_ERR_CUDA;
  }
  return queue_rank_kernel(grid, d_sets, n_sets, sequential, cmap, tabs, pack, nullptr, 0, stream);
}

// The ranking call: n_sets sets with their outputs, or (cands != null) one
// shard of a set whose record 0 has index `off` in the whole set, with its
// candidate lists going to cands instead of outputs.
int rank_launch(const unison_records *sets, const unison_rank_params *params, const unison_rank_out *outs,
                int n_sets, uint32_t off, unsigned char *cands, cudaStream_t stream) {
  StreamState *const state = stream_state(stream);
  if (!state) return UNISON_ERR_CUDA;
  StreamState &st = *state;
  bool captured = false;
  cudaGraph_t graph = nullptr;
  int rc = capture_of(stream, &captured, &graph);
  if (rc != UNISON_OK) return rc;
  std::lock_guard<std::mutex> lock(st.mu);
  if (!captured) free_unused(st.dev, stream);
  static const RankPack<1> none{};
  thread_local std::vector<unsigned char> key;
  if (n_sets > 1 && !captured) {
    plan_key(key, sets, params, outs, n_sets, off, cands);
    if (st.planned && st.plan.key == key) {
      const RankPlan &pl = st.plan;
      if (pl.packed)
        return launch_rank_kernel(st, pl.grid, nullptr, n_sets, 0, nullptr, nullptr, pl.pack[next_block(st)], pl.zero_b,
                                  stream);
      return launch_rank_kernel(
          st, pl.grid, reinterpret_cast<const RankSet *>(st.main.p + next_block(st) * pl.desc_b), n_sets, pl.sequential,
          pl.sequential ? nullptr : reinterpret_cast<const uint32_t *>(st.main.p + pl.cmap_off),
          reinterpret_cast<const RankTab *>(st.main.p + pl.tabs_off), none, pl.zero_b, stream);
    }
  }
  std::vector<RankSet> hs(n_sets);
  std::vector<RankTab> tabs;
  std::vector<int> tab_of(n_sets);
  std::vector<std::pair<const unison_rank_params *, int>> tab_keys;  // params whose tables are built
  uint64_t tiles = 0;
  for (int i = 0; i < n_sets; i++) {
    const unison_records &r = sets[i];
    const unison_rank_params &p = params[i];
    const unison_rank_out o = cands ? unison_rank_out{} : outs[i];
    if (r.n == 0 || r.n + off > (1ull << 24)) return UNISON_ERR_RANGE;
    if (!r.gap_q || !r.turn || !r.kv_tok || !r.tier || !r.flags) return UNISON_ERR_ARG;
    if (!aligned(r.gap_q, 16) || !aligned(r.turn, 16) || !aligned(r.tier, 16) || !aligned(r.flags, 16))
      return UNISON_ERR_ARG;
    if (p.k > kMaxSel || p.max_moves > kMaxSel) return UNISON_ERR_RANGE;
    if (p.penalty_q >= (1ull << 32) || p.kv_bytes_per_token == 0 || p.kv_bytes_per_token > (1u << 24))
      return UNISON_ERR_RANGE;
    if (!cands && (!o.counts || !o.moved_bytes || (p.k && !o.victims) || (p.max_moves && (!o.promote || !o.demote))))
      return UNISON_ERR_ARG;
    for (int t = 0; t < (int)kLutN; t++)
      if (p.sigma_q[t] < kEpsQ || p.sigma_q[t] > kLambda) return UNISON_ERR_RANGE;
    // per-turn tables, one per distinct (sigma, P_Z)
    int ti = -1;
    for (size_t j = 0; j < tab_keys.size() && ti < 0; j++) {
      const unison_rank_params &q = *tab_keys[j].first;
      if (q.penalty_q == p.penalty_q && std::memcmp(q.sigma_q, p.sigma_q, sizeof(p.sigma_q)) == 0)
        ti = tab_keys[j].second;
    }
    if (ti < 0) {
      if (!st.have_tab || st.tab_penalty != p.penalty_q || std::memcmp(st.tab_sigma, p.sigma_q, sizeof st.tab_sigma)) {
        for (int t = 0; t < (int)kLutN; t++) {
          st.tab.sigma[t] = p.sigma_q[t];
          st.tab.t2v[t] = ((uint64_t)(kLambda - p.sigma_q[t]) * p.penalty_q) / kLambda;  // eq. (t2)
          st.tab.mgv[t] = magic_for(p.sigma_q[t]);
        }
        std::memcpy(st.tab_sigma, p.sigma_q, sizeof st.tab_sigma);
        st.tab_penalty = p.penalty_q;
        st.have_tab = true;
      }
      ti = (int)tabs.size();
      tabs.push_back(st.tab);
      tab_keys.emplace_back(&p, ti);
    }
    tab_of[i] = ti;
    RankSet &s = hs[i];
    s.gap = r.gap_q;
    s.turn = r.turn;
    s.kv = r.kv_tok;
    s.tier = r.tier;
    s.flags = r.flags;
    s.n = (uint32_t)r.n;
    s.k = p.k;
    s.max_moves = p.max_moves;
    s.kvb = p.kv_bytes_per_token;
    s.budget = p.budget_bytes;
    s.free_s = p.free_fast_tok;
    s.free_h = p.free_hbm_tok;
    s.victims = o.victims;
    s.promote = o.promote;
    s.demote = o.demote;
    s.counts = o.counts;
    s.moved = o.moved_bytes;
    s.keys = o.keys;
    s.off = off;
    s.cands = cands;
    s.ntiles = (uint32_t)((r.n + kBigTile - 1) / kBigTile);
    tiles += s.ntiles;
    s.act = 0;
    for (int L = 0; L < kLists; L++) s.act |= list_active(s, L) ? 1u << L : 0u;
  }
  const LaunchCfg &cfg = launch_cfg();
  if (!cfg.ok) return UNISON_ERR_CUDA;
  // Groups; with more sets than CTAs, CTA c takes sets c, c + G, ...
  const int sequential = (uint64_t)n_sets > cfg.ctas ? 1 : 0;
  uint32_t grid = cfg.ctas;
  if (!sequential) {
    grid = share_ctas(hs, cfg.ctas, tiles);
  } else {
    for (int i = 0; i < n_sets; i++) {
      hs[i].cta0 = (uint32_t)(i % cfg.ctas);
      hs[i].nctas = 1;
    }
  }
  for (int i = 0; i < n_sets; i++) plan_sample(hs[i], n_sets);
  // scratch: the descriptors (for each zero block; a captured call has one),
  // CTA map and tables of a call whose launch does not bring them, then per
  // set: sorted lists and sizes, candidates.  In a zero block: every set's work
  // words, then the sampled sets' histograms
  const size_t fixed_set = align_up(sizeof(uint64_t) * kLists * kMaxSel, 256) +
                           align_up(sizeof(uint32_t) * kLists * kMaxSel, 256);
  const size_t hist_set = sizeof(uint16_t) * kLists * kBins;
  size_t sets_b = 0, hist_b = 0;  // hist_b: one block's histograms (sampled sets only)
  for (int i = 0; i < n_sets; i++) {
    RankSet &s = hs[i];
    // without a sample every eligible record is a candidate: at most n
    s.ccap = s.n > kSample ? kCandCap : (s.n + 31) & ~31u;
    // each CTA's region holds its share of ccap (at least 1,024 entries);
    // a CTA whose region fills appends the rest to the list directly
    s.cr = std::max<uint32_t>(s.ccap / s.nctas, std::min<uint32_t>(s.ccap, 1024u));
    sets_b += fixed_set + align_up(sizeof(uint64_t) * kLists * s.ccap, 256) +
              align_up(sizeof(uint64_t) * kLists * s.nctas * s.cr, 256);
    if (s.ns) hist_b += hist_set;
  }
  // descriptors go as a launch parameter where they fit
  const bool single = n_sets == 1;
  const bool packed = single || (!sequential && n_sets <= kPackSets && tabs.size() <= (size_t)kPackTabs);
  const size_t desc_b = packed ? 0 : align_up(sizeof(RankSet) * n_sets, 256);
  const size_t cmap_b = sequential || packed ? 0 : align_up(sizeof(uint32_t) * grid, 256);
  const size_t tab_b = packed ? 0 : align_up(sizeof(RankTab) * tabs.size(), 256);
  const size_t work_b = align_up(sizeof(RankWork) * n_sets, 256);
  const size_t zero_b = work_b + hist_b;
  const int images = captured ? 1 : 2;
  const size_t cmap_off = images * desc_b, tabs_off = cmap_off + cmap_b, up_b = tabs_off + tab_b;
  char *scratch = nullptr, *block[2] = {};
  if (captured) {
    rc = graph_alloc(up_b + sets_b + zero_b, graph, &scratch);
    if (rc != UNISON_OK) return rc;
    block[0] = scratch + up_b + sets_b;
  } else {
    st.planned = false;  // the scratch is rewritten below; the plan returns only if the launch succeeds
    rc = grow(st.main, up_b + sets_b, false, stream);
    if (rc == UNISON_OK) rc = grow_zero(st, zero_b, stream);
    if (rc != UNISON_OK) return rc;
    scratch = st.main.p;
    for (int b = 0; b < 2; b++) block[b] = st.zero[b].p;
  }
  RankTab *d_tabs = reinterpret_cast<RankTab *>(scratch + tabs_off);
  const uint32_t *d_cmap = sequential ? nullptr : reinterpret_cast<const uint32_t *>(scratch + cmap_off);
  char *p = scratch + up_b;
  for (int i = 0; i < n_sets; i++) {
    RankSet &s = hs[i];
    s.tab = d_tabs + tab_of[i];
    s.sorted = reinterpret_cast<uint64_t *>(p);
    p += align_up(sizeof(uint64_t) * kLists * kMaxSel, 256);
    s.ssz = reinterpret_cast<uint32_t *>(p);
    p += align_up(sizeof(uint32_t) * kLists * kMaxSel, 256);
    s.cand = reinterpret_cast<uint64_t *>(p);
    p += align_up(sizeof(uint64_t) * kLists * s.ccap, 256);
    s.creg = reinterpret_cast<uint64_t *>(p);
    p += align_up(sizeof(uint64_t) * kLists * s.nctas * s.cr, 256);
  }
  // the work words and histograms of the sets in block b
  auto in_block = [&](int b) {
    char *const z = block[b];
    size_t hoff = work_b;
    for (int i = 0; i < n_sets; i++) {
      RankSet &s = hs[i];
      s.work = reinterpret_cast<RankWork *>(z) + i;
      s.shist = s.ns ? reinterpret_cast<uint16_t *>(z + hoff) : nullptr;
      if (s.ns) hoff += hist_set;
    }
  };
  if (single) {
    in_block(captured ? 0 : next_block(st));
    RankPack<1> one;
    one.set[0] = hs[0];
    one.tab[0] = tabs[0];
    if (captured) return capture_rank_kernel(grid, nullptr, 1, 0, nullptr, nullptr, one, block[0], zero_b, stream);
    return launch_rank_kernel(st, grid, nullptr, 1, 0, nullptr, nullptr, one, zero_b, stream);
  }
  if (packed) {
    auto fill_pack = [&](RankPack<kPackSets> &pk) {
      std::memcpy(pk.set, hs.data(), sizeof(RankSet) * n_sets);
      std::memcpy(pk.tab, tabs.data(), sizeof(RankTab) * tabs.size());
      for (int i = 0; i < n_sets; i++) {
        pk.tab_of[i] = (uint8_t)tab_of[i];
        std::memset(pk.of_cta + hs[i].cta0, i, hs[i].nctas);
      }
    };
    if (captured) {
      RankPack<kPackSets> pk;
      in_block(0);
      fill_pack(pk);
      return capture_rank_kernel(grid, nullptr, n_sets, 0, nullptr, nullptr, pk, block[0], zero_b, stream);
    }
    RankPlan &pl = st.plan;
    for (int b = 0; b < 2; b++) {
      in_block(b);
      fill_pack(pl.pack[b]);
    }
    rc = launch_rank_kernel(st, grid, nullptr, n_sets, 0, nullptr, nullptr, pl.pack[next_block(st)], zero_b, stream);
    if (rc == UNISON_OK) {
      pl.key = key;
      pl.zero_b = zero_b;
      pl.grid = grid;
      pl.sequential = 0;
      pl.packed = true;
      st.planned = true;
    }
    return rc;
  }
  // the image of what the launch does not bring
  auto fill_image = [&](unsigned char *h) {
    for (int b = 0; b < images; b++) {
      in_block(b);
      std::memcpy(h + b * desc_b, hs.data(), sizeof(RankSet) * n_sets);
    }
    if (!sequential) {
      uint32_t *cm = reinterpret_cast<uint32_t *>(h + cmap_off);
      for (int i = 0; i < n_sets; i++)
        for (uint32_t b = hs[i].cta0; b < hs[i].cta0 + hs[i].nctas; b++) cm[b] = (uint32_t)i | ((uint32_t)tab_of[i] << 16);
    }
    std::memcpy(h + tabs_off, tabs.data(), sizeof(RankTab) * tabs.size());
  };
  if (captured) {
    std::vector<uint64_t> image((up_b + 7) / 8);
    fill_image(reinterpret_cast<unsigned char *>(image.data()));
    rc = graph_write(scratch, image.data(), up_b);
    if (rc != UNISON_OK) return rc;
    return capture_rank_kernel(grid, reinterpret_cast<const RankSet *>(scratch), n_sets, sequential, d_cmap, d_tabs,
                               none, block[0], zero_b, stream);
  }
  // one copy from pinned staging
  {
    unsigned char *h = nullptr;
    cudaEvent_t done = nullptr;
    const int sr = staging_acquire(up_b, &h, &done);
    if (sr != UNISON_OK) return sr;
    fill_image(h);
    if (cudaMemcpyAsync(scratch, h, up_b, cudaMemcpyHostToDevice, stream) != cudaSuccess) rc = UNISON_ERR_CUDA;
    if (cudaEventRecord(done, stream) != cudaSuccess) rc = UNISON_ERR_CUDA;  // the buffer is reused after this copy
    staging_release();
    if (rc != UNISON_OK) {
      cudaGetLastError();
      return rc;
    }
  }
  rc = launch_rank_kernel(st, grid, reinterpret_cast<const RankSet *>(scratch + next_block(st) * desc_b), n_sets,
                          sequential, d_cmap, d_tabs, none, zero_b, stream);
  if (rc == UNISON_OK) {
    RankPlan &pl = st.plan;
    pl.key = key;
    pl.desc_b = desc_b;
    pl.cmap_off = cmap_off;
    pl.tabs_off = tabs_off;
    pl.zero_b = zero_b;
    pl.grid = grid;
    pl.sequential = sequential;
    pl.packed = false;
    st.planned = true;
  }
  return rc;
}

}  // namespace

extern "C" int unison_rank_batch(const unison_records *sets, const unison_rank_params *params,
                                 const unison_rank_out *outs, int n_sets, void *cuda_stream) {
  if (n_sets < 0 || (n_sets > 0 && (!sets || !params || !outs))) return UNISON_ERR_ARG;
  if (n_sets == 0) return UNISON_OK;
  return rank_launch(sets, params, outs, n_sets, 0u, nullptr, static_cast<cudaStream_t>(cuda_stream));
}

extern "C" int unison_rank(const unison_records *records, const unison_rank_params *params,
                           const unison_rank_out *out, void *cuda_stream) {
  if (!records || !params || !out) return UNISON_ERR_ARG;
  return unison_rank_batch(records, params, out, 1, cuda_stream);
}

extern "C" uint64_t unison_rank_cands_bytes(uint32_t k, uint32_t max_moves) { return cand_bytes(k, max_moves); }

extern "C" int unison_rank_shard(const unison_records *slice, uint64_t index_offset, const unison_rank_params *params,
                                 void *cands_dev, void *cuda_stream) {
  if (!slice || !params || !cands_dev || !aligned(cands_dev, 256)) return UNISON_ERR_ARG;
  if (index_offset >= (1ull << 24)) return UNISON_ERR_RANGE;
  return rank_launch(slice, params, nullptr, 1, (uint32_t)index_offset, static_cast<unsigned char *>(cands_dev),
                     static_cast<cudaStream_t>(cuda_stream));
}

extern "C" int unison_rank_merge(const void *gathered_dev, int n_shards, const unison_rank_params *params,
                                 const unison_rank_out *out, void *cuda_stream) {
  if (!gathered_dev || !params || !out || n_shards < 1) return UNISON_ERR_ARG;
  if (n_shards > (int)kMaxShards) return UNISON_ERR_RANGE;
  const unison_rank_params &p = *params;
  const unison_rank_out &o = *out;
  if (p.k > kMaxSel || p.max_moves > kMaxSel) return UNISON_ERR_RANGE;
  if (p.kv_bytes_per_token == 0 || p.kv_bytes_per_token > (1u << 24)) return UNISON_ERR_RANGE;
  if (!o.counts || !o.moved_bytes || (p.k && !o.victims) || (p.max_moves && (!o.promote || !o.demote)))
    return UNISON_ERR_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  RankSet s{};
  s.k = p.k;
  s.max_moves = p.max_moves;
  s.kvb = p.kv_bytes_per_token;
  s.budget = p.budget_bytes;
  s.free_s = p.free_fast_tok;
  s.free_h = p.free_hbm_tok;
  s.victims = o.victims;
  s.promote = o.promote;
  s.demote = o.demote;
  s.counts = o.counts;
  s.moved = o.moved_bytes;
  for (int L = 0; L < kLists; L++) s.act |= list_active(s, L) ? 1u << L : 0u;
  // scratch: sorted lists; work words in the zero block whose turn it is
  const size_t work_b = align_up(sizeof(RankWork), 256);
  const size_t vals_b = align_up(sizeof(uint64_t) * kLists * kMaxSel, 256);
  const size_t lists_b = vals_b + align_up(sizeof(uint32_t) * kLists * kMaxSel, 256);
  const LaunchCfg &cfg = launch_cfg();
  if (!cfg.ok) return UNISON_ERR_CUDA;
  StreamState *const state = stream_state(stream);
  if (!state) return UNISON_ERR_CUDA;
  StreamState &st = *state;
  bool captured = false;
  cudaGraph_t graph = nullptr;
  int rc = capture_of(stream, &captured, &graph);
  if (rc != UNISON_OK) return rc;
  std::lock_guard<std::mutex> lock(st.mu);
  char *scratch = nullptr, *words = nullptr, *other = nullptr;
  size_t other_b = 0;
  const int b = next_block(st);
  if (captured) {  // (memory of its own, as in rank_launch)
    rc = graph_alloc(lists_b + work_b, graph, &scratch);
    if (rc != UNISON_OK) return rc;
    words = scratch + lists_b;
    if (cudaMemsetAsync(words, 0, work_b, stream) != cudaSuccess) {
      cudaGetLastError();
      return UNISON_ERR_CUDA;
    }
  } else {
    free_unused(st.dev, stream);
    st.planned = false;  // the scratch is rewritten below
    rc = grow(st.main, lists_b, false, stream);
    if (rc == UNISON_OK) rc = grow_zero(st, work_b, stream);
    if (rc != UNISON_OK) return rc;
    scratch = st.main.p;
    words = st.zero[b].p;
    other = st.zero[1 - b].p;
    other_b = st.dirty[1 - b];
  }
  s.work = reinterpret_cast<RankWork *>(words);
  s.sorted = reinterpret_cast<uint64_t *>(scratch);
  s.ssz = reinterpret_cast<uint32_t *>(scratch + vals_b);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(kLists);
  lc.blockDim = dim3(kConsumers);
  lc.dynamicSmemBytes = kMergeSmem;
  lc.stream = stream;
  const cudaError_t e = cudaLaunchKernelEx(
      &lc, rank_merge_kernel, s, static_cast<const unsigned char *>(gathered_dev), n_shards,
      (uint64_t)cand_bytes(p.k, p.max_moves), reinterpret_cast<uint4 *>(other), (uint32_t)(other_b / 16));
  count_launches(1);
  if (e != cudaSuccess) {  // (its own verdict, as in queue_rank_kernel)
    cudaGetLastError();
    return UNISON_ERR_CUDA;  // nothing ran: the blocks are as they were
  }
  if (captured) return UNISON_OK;
  st.dirty[b] = work_b;
  st.dirty[1 - b] = 0;
  return UNISON_OK;
}
