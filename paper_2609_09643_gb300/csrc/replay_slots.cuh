// The slot form of the replay's event loop (Algorithm 1): one warp per
// replay, residents in unordered slots of shared memory.
//
// Every resident keeps one slot from its placement to its eviction, whatever
// tier it is in and whether it is pinned or not.  An unpinned resident's slot
// holds one 32-bit word
//     fast tier << 31 | (rank + 1) << slot bits | slot
// and every other slot holds 0.  The rank orders the residents as their
// packed keys do (rank_keys_kernel below; recency and next-reference ranks
// come from event counts), so every choice of Algorithm 1 and of TIDE is one
// pass of the warp over the words and one reduction: the most evictable
// fast-tier session is the largest word, the least evictable HBM session the
// smallest non-zero one, the most evictable HBM session the largest once the
// tier bit is flipped, and the winner's low bits name its slot.  Ranking,
// placing, moving, pinning and dropping a session are single stores.
//
// What bounds it: the dependence chain of one warp.  The chain of a choice is
// a 16-byte shared load a lane for up to 128 slots, three maxima, one REDUX
// and the load of the winner's size.  An instruction costs about 2.7 cycles to
// issue and wait for, and a longer event loop runs slower.  So what follows from an arrival's
// class is left to account_arrivals, branches and rarely taken tests are kept
// few, and loops stay rolled.  The 1,024-replay sweep's launch, one GB300: 57.5
// ms with sorted lists of 64-bit keys in the warp's registers (375 instructions
// an event), 38.7 with slots (188), 32.1 with the accounting taken out (158),
// 26.8 with loops rolled, errors leaving by a jump, the bypass apart, each
// event's record found by a pointer and room in HBM for a demoted session tested
// in place.  Tried and not kept: the words' extremes
// found at the top of every event, beside the session's lookup (34.3 against
// 32.5 ms); 256 words loaded at once in every pass (34.0); HBM's making of room
// out of line for its second caller (48 against 31); the fast tier's payload
// loaded only when a swap is tried (31.6 against 31.2).
//
// Two variants keep a second array of words.  A stale-snapshot replay ranks by
// the snapshot's ranks and keeps the live ones beside them, so a choice is
// compared with the live one by a second pass and a sync rewrites the words of
// the sessions that changed, a lane each (16 replays over the four sync modes
// 148 -> 45 ms).  Under the online hazard table keys change while sessions are
// resident, so a word is the key itself in 64 bits, and a rebuilt table rewrites
// every word in place where sorted lists had to be sorted again (6 online, 6
// offline and 6 LRU replays with logs 111 -> 47 ms).
#pragma once

#include "common.cuh"

namespace unison_slots {

using namespace unison;

constexpr uint32_t kAll = 0xFFFFFFFFu;
constexpr uint32_t kFastBit = 0x80000000u;   // of a slot word
constexpr uint32_t kPromoted = 0x80000000u;  // of a payload's size word
constexpr uint32_t kSizeBits = 0x7FFFFFFFu;
constexpr uint32_t kMostSlots = 2048;  // 16 words a lane

// A resident's payload: size (and whether TIDE promoted it), session and tier
// (bit 31: fast).  Policies other than SPEAR+TIDE also keep the rank a Belady
// session will have once unpinned, and the time it was unpinned (Timeout).
template <bool kWide>
struct Payload;
template <>
struct Payload<false> {
  uint2 v;
};
template <>
struct Payload<true> {
  uint4 v;
};

// Events reach the warp through a ring of shared memory, 32 at a time, with
// the next batch landed and the one after it on its way.
struct SlotEvent {
  uint4 ev;   // time32, session | flags, in_tok, out_tok
  uint4 aux;  // rank, gap average (completions); next reference (arrivals)
};
constexpr uint32_t kRing = 128;
struct SlotBufs {
  SlotEvent e[kRing + 1];  // the last mirrors the first event's word, so that a batch's end reads on
};

// What one replay of the slot form reads besides its ReplayDesc.
struct SlotDesc {
  const uint32_t *rank;  // rank after each completion event (SPEAR policies), or null
  uint32_t cap_s, cap_h;  // tokens, at most the sum of every session's largest size (< 2^31)
  uint32_t nslots;        // slots the replay can need
  uint32_t sbits;         // slot bits of a word
  uint32_t form;          // kForm*
  uint32_t serial;        // 1: the prefill queue's times may pass 2^63 ns (account_arrivals)
};

// Forms of a launch: the session map's width, and how the words are passed over
// (see slot_maps in replay.cu).
constexpr int kFormPlain = 0, kFormDeep = 1, kFormMap8 = 2;

// What the event loop notes of each arrival, one byte in arrival order: the
// request class, whether TIDE had promoted the session, and where it was
// placed.  The bytes lie in the last eighth of the replay's TTFT area: arrival
// i's at byte 7 n_turns + i.
constexpr uint32_t kClassCold = 0, kClassFast = 1, kClassHbm = 2, kClassMiss = 3;  // the decision kinds
constexpr uint32_t kNotePromoted = 4, kNotePlaceShift = 3;  // bits 3-4: 0 fast tier, 1 HBM, 2 bypassed

// Bytes of shared memory of one replay: words, payloads, free slots, map.
__host__ __device__ inline size_t slot_words(uint32_t nslots) {
  return nslots <= 128 ? 128 : 128 + ((size_t)nslots - 128 + 255) / 256 * 256;
}
__host__ inline size_t slot_bytes(uint32_t nslots, uint32_t n_sessions, bool wide, bool map8) {
  const size_t pay = (size_t)nslots * (wide ? 16 : 8), fr = ((size_t)nslots * 2 + 15) / 16 * 16;
  const size_t map = ((size_t)n_sessions * (map8 ? 1 : 2) + 15) / 16 * 16;
  return slot_words(nslots) * 4 + (pay + 15) / 16 * 16 + fr + map;
}
// Beside those: a second array of words; a stale replay's live and snapshot
// ranks of every session and the sessions changed since the last sync; an
// online replay's arrivals of every session and its table.
constexpr uint32_t kDirtySlots = 64;
__host__ __device__ inline size_t round16(size_t b) { return (b + 15) / 16 * 16; }

// Where a replay's ranking comes from.
constexpr int kRanked = 0;  // ranks of the key stream, or recency
constexpr int kStale = 1;   // ranks of a register-file snapshot (eq. stale)
constexpr int kOnline = 2;  // keys under the online hazard table (Sec. V-F)

// The replay's state.  kLean: no decision log and no slot limit.
template <int kMode, bool kLean, bool kWide, bool kDeep>
struct Slots {
  uint32_t *W;
  uint32_t *L;            // kStale: the words by live ranks; kOnline: the words' low halves
  Payload<kWide> *P;
  uint16_t *F;            // freed slots, a stack
  uint32_t nfree, fresh;  // entries of F; slots handed out at least once
  uint32_t sbits, smask;
  // tokens: a tier's space beside all its residents, and beside its pinned ones
  uint32_t free_s, free_h, room_s, room_h;
  int status;
  // decision stream: event, hash (two halves), log
  uint32_t e, h_lo, h_hi;
  uint2 *log;         // the next entry
  uint64_t log_left;  // entries left (0 without a log)
  // counters (warp-uniform registers); those of arrivals come from the notes
  uint32_t n_evict, n_demote, n_promote, n_tide_demote, n_expire, n_tide_calls, n_res;
  uint32_t vict_n, vict_diff, prom_n, prom_diff;  // kStale: choices, and those unlike the live one
};

// h = (h ^ (event << 32 | kind << 24 | session)) * 0x100000001B3 mod 2^64.
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ void decide(Slots<kMode, kLean, kWide, kDeep> &st, uint32_t kind, uint32_t s, int lane) {
  static_assert(kFnvPrime == (1ull << 40 | 0x1B3u), "the multiplication below");
  const uint32_t lo = st.h_lo ^ (s | kind << 24), hi = st.h_hi ^ st.e;
  const uint64_t m = (uint64_t)lo * 0x1B3u;
  st.h_lo = (uint32_t)m;
  // (one multiply-add each; written as a shift, lo << 8 took an instruction more)
  uint32_t t = (uint32_t)(m >> 32) + hi * 0x1B3u;
  asm("mad.lo.u32 %0, %1, 256, %0;" : "+r"(t) : "r"(lo));
  st.h_hi = t;
  if constexpr (!kLean) {
    static_assert(sizeof(unison_decision) == sizeof(uint2), "a log entry: event, kind << 24 | session");
    if (st.log_left) {
      *st.log++ = make_uint2(st.e, kind << 24 | s);  // (every lane the same)
      st.log_left--;
    }
  }
}

// Extremes over the words of every slot handed out so far; the words past them
// are 0.  A pass takes 128 words, 4 a lane; past the first 128, kDeep takes 256
// at a time, two loads in flight.  Loops are kept rolled: unrolled by the
// compiler, which lengthens the event loop, 30 paper-scale replays took 31.6
// ms in place of 28.0.
__device__ __forceinline__ uint32_t max4(uint4 v) { return max(max(v.x, v.y), max(v.z, v.w)); }
__device__ __forceinline__ uint32_t max4(uint32_t m, uint4 v) { return max(max(m, max(v.x, v.y)), max(v.z, v.w)); }
__device__ __forceinline__ uint4 flip4(uint4 v) {
  return make_uint4(v.x ^ kFastBit, v.y ^ kFastBit, v.z ^ kFastBit, v.w ^ kFastBit);
}
__device__ __forceinline__ uint32_t min4_less1(uint4 v) {
  return min(min(v.x - 1u, v.y - 1u), min(v.z - 1u, v.w - 1u));
}
__device__ __forceinline__ uint32_t min4_less1(uint32_t m, uint4 v) {
  return min(min(m, min(v.x - 1u, v.y - 1u)), min(v.z - 1u, v.w - 1u));
}
template <bool kDeep>
__device__ __forceinline__ uint32_t max_of(const uint32_t *W, uint32_t fresh, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(W) + lane;
  uint4 v = w4[0];
  uint32_t m = max4(v);
#pragma unroll 1
  for (uint32_t q = 128; q < fresh; q += kDeep ? 256 : 128) {
    w4 += 32;
    v = *w4;
    if constexpr (kDeep) {
      w4 += 32;
      m = max4(m, *w4);
    }
    m = max4(m, v);
  }
  return __reduce_max_sync(kAll, m);
}
// The largest word with the tier bit flipped: > kFastBit if there is an HBM word.
template <bool kDeep>
__device__ __forceinline__ uint32_t max_hbm_of(const uint32_t *W, uint32_t fresh, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(W) + lane;
  uint4 v = w4[0];
  uint32_t m = max4(flip4(v));
#pragma unroll 1
  for (uint32_t q = 128; q < fresh; q += kDeep ? 256 : 128) {
    w4 += 32;
    v = *w4;
    if constexpr (kDeep) {
      w4 += 32;
      m = max4(m, flip4(*w4));
    }
    m = max4(m, flip4(v));
  }
  return __reduce_max_sync(kAll, m);
}
// The largest word, and the smallest word above 0 less 1 (below
// kFastBit - 1 if there is an HBM word).
template <bool kDeep>
__device__ __forceinline__ void extremes_of(const uint32_t *W, uint32_t fresh, uint32_t &mx, uint32_t &mn, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(W) + lane;
  uint4 v = w4[0];
  uint32_t a = max4(v), b = min4_less1(v);
#pragma unroll 1
  for (uint32_t q = 128; q < fresh; q += kDeep ? 256 : 128) {
    w4 += 32;
    v = *w4;
    if constexpr (kDeep) {
      w4 += 32;
      const uint4 u = *w4;
      a = max4(a, u);
      b = min4_less1(b, u);
    }
    a = max4(a, v);
    b = min4_less1(b, v);
  }
  mx = __reduce_max_sync(kAll, a);
  mn = __reduce_min_sync(kAll, b);
}

// The online table's keys change while sessions are resident, so a word holds
// the key itself: W a tier bit, a 1 and the key's upper 23 bits, L its lower
// 17 bits and the inverted session (15 bits, larger key and smaller id first).
// A completed session's maximal key is 2^39 here; live keys are below it.
constexpr uint32_t kOnlineLive = 0x40000000u;
constexpr uint32_t kOnlineIds = 0x7FFFu;
__device__ __forceinline__ uint64_t online_word(uint64_t key, uint32_t s) {
  return ((uint64_t)(kOnlineLive | (uint32_t)(key >> 17)) << 32) | ((uint32_t)key << 15) | (kOnlineIds - s);
}
// The most evictable word once W ^ flip (the wanted tier's words then have the
// top bit), as W ^ flip and L.  The least evictable HBM word comes as W ^
// kOnlineLive and L (the first below kOnlineLive if there is one).
__device__ __forceinline__ uint64_t online_max(const uint32_t *W, const uint32_t *L, uint32_t fresh, uint32_t flip,
                                               int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(W) + lane, *l4 = reinterpret_cast<const uint4 *>(L) + lane;
  auto of = [&](uint4 w, uint4 l) {
    return max(max((uint64_t)(w.x ^ flip) << 32 | l.x, (uint64_t)(w.y ^ flip) << 32 | l.y),
               max((uint64_t)(w.z ^ flip) << 32 | l.z, (uint64_t)(w.w ^ flip) << 32 | l.w));
  };
  uint64_t m = of(*w4, *l4);
#pragma unroll 1
  for (uint32_t q = 128; q < fresh; q += 128) m = max(m, of(*(w4 += 32), *(l4 += 32)));
  const uint32_t hi = __reduce_max_sync(kAll, (uint32_t)(m >> 32));
  return (uint64_t)hi << 32 | __reduce_max_sync(kAll, (uint32_t)(m >> 32) == hi ? (uint32_t)m : 0u);
}
// Both at once: the most evictable fast-tier word and the least evictable HBM one.
__device__ __forceinline__ void online_ends(const uint32_t *W, const uint32_t *L, uint32_t fresh, uint64_t &top,
                                            uint64_t &low, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(W) + lane, *l4 = reinterpret_cast<const uint4 *>(L) + lane;
  constexpr uint32_t x = kOnlineLive;
  auto most = [&](uint4 w, uint4 l) {
    return max(max((uint64_t)w.x << 32 | l.x, (uint64_t)w.y << 32 | l.y),
               max((uint64_t)w.z << 32 | l.z, (uint64_t)w.w << 32 | l.w));
  };
  auto least = [&](uint4 w, uint4 l) {
    return min(min((uint64_t)(w.x ^ x) << 32 | l.x, (uint64_t)(w.y ^ x) << 32 | l.y),
               min((uint64_t)(w.z ^ x) << 32 | l.z, (uint64_t)(w.w ^ x) << 32 | l.w));
  };
  uint64_t m = most(*w4, *l4), n = least(*w4, *l4);
#pragma unroll 1
  for (uint32_t q = 128; q < fresh; q += 128) {
    const uint4 w = *(w4 += 32), l = *(l4 += 32);
    m = max(m, most(w, l));
    n = min(n, least(w, l));
  }
  const uint32_t hi = __reduce_max_sync(kAll, (uint32_t)(m >> 32)), lo = __reduce_min_sync(kAll, (uint32_t)(n >> 32));
  top = (uint64_t)hi << 32 | __reduce_max_sync(kAll, (uint32_t)(m >> 32) == hi ? (uint32_t)m : 0u);
  low = (uint64_t)lo << 32 | __reduce_min_sync(kAll, (uint32_t)(n >> 32) == lo ? (uint32_t)n : kAll);
}

// The table of the sessions completed so far (eqs. (hazard), (hq), (survq),
// (t2) with bucket pooling), in shared memory.
struct OnlineTable {
  uint32_t n[kLutN], d[kLutN], sig[kLutN];
  unsigned long long t2[kLutN];
  unsigned long long mg[kLutN];  // magic_for(sig): eq. (t1)'s division by a multiply-high
};
__device__ __forceinline__ void online_init(OnlineTable &ot, int lane) {
  for (uint32_t t = lane; t < kLutN; t += 32) {
    ot.n[t] = ot.d[t] = 0u;
    ot.sig[t] = kLambda;  // no session completed: zero hazard
    ot.t2[t] = 0ull;
    ot.mg[t] = magic_for(kLambda);
  }
}
// A score under the table; g < 2^31 (gaps are clamped below 2^31 us), so g *
// Lambda < 2^43.
__device__ __forceinline__ uint64_t online_score(const OnlineTable &ot, uint32_t g, uint32_t t) {
  const uint32_t tt = t < kTMax ? t : kTMax;
  return __umul64hi((uint64_t)g * kLambda, ot.mg[tt]) + ot.t2[tt];
}
// A session of `turns` turns has completed: add it to the counts and rebuild
// sigma and T2 for every turn index.  With at most 32,768 sessions the pooled
// counts are below 2^15 (d) and 2^21 (n), so the quotient's terms fit 32 bits.
// True if an entry changed.
__device__ __noinline__ bool online_add(OnlineTable &ot, uint32_t turns, uint32_t bucket, uint64_t penalty, int lane) {
  for (uint32_t t = lane; t < kLutN; t += 32) {
    ot.n[t] += turns >= t + 1 ? 1u : 0u;
    ot.d[t] += turns == t + 1 ? 1u : 0u;
  }
  __syncwarp();
  bucket = min(bucket, kLutN);
  bool changed = false;
  uint32_t sg[2];
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const uint32_t t = lane + 32 * q;
    sg[q] = kLambda;
    if (t < kLutN) {
      const uint32_t u0 = t - t % bucket, u1 = min(u0 + bucket, kLutN);
      uint32_t nn = 0, dd = 0;
      for (uint32_t u = u0; u < u1; u++) {
        nn += ot.n[u];
        dd += ot.d[u];
      }
      const uint32_t hq = nn ? min((2u * dd * kLambda + nn) / (2u * nn), kLambda) : 0u;
      sg[q] = max(kLambda - hq, kEpsQ);
      changed |= ot.sig[t] != sg[q];
    }
  }
  changed = __any_sync(kAll, changed);  // T2 and the divisors follow from sigma
  if (!changed) return false;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const uint32_t t = lane + 32 * q;
    if (t < kLutN && ot.sig[t] != sg[q]) {
      ot.sig[t] = sg[q];
      ot.t2[t] = ((unsigned long long)(kLambda - sg[q]) * penalty) / kLambda;
      ot.mg[t] = magic_for(sg[q]);
    }
  }
  __syncwarp();
  return true;
}

// A choice among the residents: whether there is one, its slot, and a value
// that orders choices of either tier (larger: more evictable).
struct Choice {
  bool any;
  uint32_t slot;
  uint64_t order;
};
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ Choice most_evictable_fast(const Slots<kMode, kLean, kWide, kDeep> &st, const uint16_t *map,
                                                      int lane) {
  if constexpr (kMode == kOnline) {
    const uint64_t m = online_max(st.W, st.L, st.fresh, 0u, lane);
    const bool any = m >> 63 != 0;
    return {any, any ? map[kOnlineIds - ((uint32_t)m & kOnlineIds)] : 0u, m & ~(1ull << 63)};
  } else {
    const uint32_t w = max_of<kDeep>(st.W, st.fresh, lane);
    return {(w & kFastBit) != 0, w & st.smask, w & ~kFastBit};
  }
}
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ Choice most_evictable_hbm(const Slots<kMode, kLean, kWide, kDeep> &st, const uint16_t *map,
                                                     int lane) {
  if constexpr (kMode == kOnline) {
    const uint64_t m = online_max(st.W, st.L, st.fresh, kFastBit, lane);  // (an empty slot: kFastBit, 0)
    const bool any = m > (1ull << 63);
    return {any, any ? map[kOnlineIds - ((uint32_t)m & kOnlineIds)] : 0u, m & ~(1ull << 63)};
  } else {
    const uint32_t m = max_hbm_of<kDeep>(st.W, st.fresh, lane);
    return {m > kFastBit, m & st.smask, m & ~kFastBit};
  }
}
// The words of a choice in the other tier, or none.
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ void set_word(Slots<kMode, kLean, kWide, kDeep> &st, uint32_t slot, bool fast, uint64_t order) {
  const uint32_t bit = fast ? kFastBit : 0u;
  if constexpr (kMode == kOnline) {
    st.W[slot] = (uint32_t)(order >> 32) | bit;
    st.L[slot] = (uint32_t)order;
  } else {
    st.W[slot] = (uint32_t)order | bit;
    if constexpr (kMode == kStale) st.L[slot] = (st.L[slot] & ~kFastBit) | bit;
  }
}
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ void clear_word(Slots<kMode, kLean, kWide, kDeep> &st, uint32_t slot) {
  st.W[slot] = 0u;
  if constexpr (kMode != kRanked) st.L[slot] = 0u;
}

// kStale: a choice (slot) against the live ranks' over the same sessions.
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ void count_victim(Slots<kMode, kLean, kWide, kDeep> &st, uint32_t slot, uint32_t live_word) {
  if constexpr (kMode == kStale) {
    st.vict_n++;
    st.vict_diff += (live_word & st.smask) != slot;
  }
}

// Slot stores: every lane stores the same value to the same place, so each
// lane's later loads see it without a warp barrier; a __syncwarp separates a
// store from the loads of the old value before it.
template <class St>
__device__ __forceinline__ void release_slot(St &st, uint32_t slot) {
  clear_word(st, slot);
  st.P[slot].v.y = kIdMask;  // no session has this id
  st.F[st.nfree] = (uint16_t)slot;
  st.nfree++;
  st.n_res--;
}
template <class St>
__device__ __forceinline__ uint2 payload(const St &st, uint32_t slot) {
  const uint2 p = *reinterpret_cast<const uint2 *>(&st.P[slot]);
  __syncwarp();
  return p;
}

// Room in HBM for `size` tokens against its unpinned residents: evicts the
// most evictable ones, only those above `d` (a session demoted out of the fast
// tier; without one every resident is above).  False when the next one is not.
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ bool make_hbm_room(Slots<kMode, kLean, kWide, kDeep> &st, const uint16_t *map, uint32_t size,
                                              const Choice &d, int lane) {
  while (size > st.free_h) {
    const Choice v = most_evictable_hbm(st, map, lane);
    const bool drop = !v.any || (d.any && d.order > v.order);
    if constexpr (kMode == kStale) {
      // the live choice: among HBM's sessions and the demoted one
      uint32_t live = max_hbm_of<kDeep>(st.L, st.fresh, lane);
      live = live > kFastBit ? live & ~kFastBit : 0u;
      if (d.any) live = max(live, st.L[d.slot] & ~kFastBit);
      count_victim(st, drop ? d.slot : v.slot, live);
    }
    if (drop) return false;
    const uint2 p = payload(st, v.slot);
    st.free_h += p.x & kSizeBits;
    decide(st, UNISON_KIND_EVICT, p.y & kIdMask, lane);
    st.n_evict++;
    release_slot(st, v.slot);
  }
  return true;
}

__device__ __forceinline__ void async16(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory");
}

// Timeout: expire unpinned residents idle >= ttl, smallest session id first.
// `oldest` is a time no later than any unpinned resident's return, so most
// events need one comparison.  Past it, a pass over the words finds the two
// residents that returned first (ranks follow recency: the largest returned
// first, whatever its tier).  That settles an event on which none or one has
// expired; only where the second has expired too does a pass over the payloads
// look for the smallest id.  One replay of 2,000 sessions, up to 1,990 resident,
// 10 s to live: 77.3 ms with a pass over the payloads per expired session and
// one more, 34.4 so, 43.0 on sorted lists; with 1 s to live 71.8, 31.7, 35.4.
template <class St>
__device__ __forceinline__ void expire_slots(St &st, uint32_t now, uint32_t ttl, uint32_t &oldest, int lane) {
  if (now - oldest < ttl) return;
  for (;;) {
    uint32_t a = 0, b = 0;  // this lane's largest and second
    const uint4 *w4 = reinterpret_cast<const uint4 *>(st.W) + lane;
    auto take = [&](uint32_t w) {
      const uint32_t x = w & ~kFastBit;
      b = max(b, min(a, x));
      a = max(a, x);
    };
#pragma unroll 1
    for (uint32_t q = 0; q < st.fresh; q += 128, w4 += 32) {
      const uint4 v = *w4;
      take(v.x);
      take(v.y);
      take(v.z);
      take(v.w);
    }
    const uint32_t first = __reduce_max_sync(kAll, a);
    if (first == 0) {  // no unpinned resident
      oldest = now;
      return;
    }
    const uint32_t second = __reduce_max_sync(kAll, a == first ? b : a);
    uint32_t slot = first & st.smask;
    const uint32_t t1 = st.P[slot].v.w;
    if (now - t1 < ttl) {
      oldest = t1;
      return;
    }
    const uint32_t t2 = second ? st.P[second & st.smask].v.w : now;
    const bool more = second != 0 && now - t2 >= ttl;
    if (more) {
      uint32_t id = kAll, at = 0;
      for (uint32_t i = lane; i < st.fresh; i += 32) {
        if (st.W[i] == 0 || now - st.P[i].v.w < ttl) continue;
        const uint32_t s = st.P[i].v.y & kIdMask;
        if (s < id) {
          id = s;
          at = i;
        }
      }
      const uint32_t least = __reduce_min_sync(kAll, id);
      slot = __shfl_sync(kAll, at, __ffs(__ballot_sync(kAll, id == least)) - 1);
    }
    const uint32_t w = st.W[slot];
    const uint2 p = payload(st, slot);
    const uint32_t size = p.x & kSizeBits;
    st.free_s += w & kFastBit ? size : 0u;
    st.free_h += w & kFastBit ? 0u : size;
    decide(st, UNISON_KIND_EXPIRE, p.y & kIdMask, lane);
    st.n_expire++;
    release_slot(st, slot);
    __syncwarp();
    if (!more) {
      oldest = t2;
      return;
    }
  }
}

// TIDE at a gap_start with `budget` bytes, one move at a time as the pair loop
// of Algorithm 1 has it: phase 1 promotes the least evictable HBM sessions
// into free fast-tier space, phase 2 swaps the least evictable HBM session
// with the most evictable fast-tier one.  Returns the bytes moved.
template <int kMode, bool kLean, bool kWide, bool kDeep>
__device__ __forceinline__ uint64_t tide_slots(Slots<kMode, kLean, kWide, kDeep> &st, const uint16_t *map, uint64_t budget,
                                               uint32_t kvb, int lane) {
  uint64_t rem = budget;
  bool fill = true;  // phase 1
  for (;;) {
    Choice pc, dc;  // the least evictable HBM session, the most evictable fast-tier one
    if constexpr (kMode == kOnline) {
      uint64_t top, low;
      online_ends(st.W, st.L, st.fresh, top, low, lane);
      const bool any = low >> 32 < kOnlineLive, fast = top >> 63 != 0;
      pc = {any, any ? map[kOnlineIds - ((uint32_t)low & kOnlineIds)] : 0u, low | (uint64_t)kOnlineLive << 32};
      dc = {fast, fast ? map[kOnlineIds - ((uint32_t)top & kOnlineIds)] : 0u, top & ~(1ull << 63)};
    } else {
      uint32_t mx, mn;
      extremes_of<kDeep>(st.W, st.fresh, mx, mn, lane);
      pc = {mn < kFastBit - 1u, (mn + 1u) & st.smask, mn + 1u};
      dc = {(mx & kFastBit) != 0, mx & st.smask, mx & ~kFastBit};  // (a valid slot even when mx names none)
    }
    // (without an HBM session pc names a valid slot all the same)
    const uint2 p = *reinterpret_cast<const uint2 *>(&st.P[pc.slot]);
    const uint2 d = payload(st, dc.slot);
    const uint32_t sp = p.x & kSizeBits, pid = p.y & kIdMask;
    const uint32_t sd = d.x & kSizeBits, did = d.y & kIdMask;
    uint64_t by = (uint64_t)sp * kvb;
    fill = fill && pc.any && by <= rem && sp <= st.free_s;
    if (!fill) {
      // phase 2: the swap is legal and the demoted session the more evictable
      by += (uint64_t)sd * kvb;
      if (!(pc.any && dc.any && dc.order > pc.order && by <= rem && sp <= st.free_s + sd && sd <= st.free_h + sp)) break;
    }
    if constexpr (kMode == kStale) {
      uint32_t mx, mn;
      extremes_of<kDeep>(st.L, st.fresh, mx, mn, lane);
      st.prom_n++;
      st.prom_diff += ((mn + 1u) & st.smask) != pc.slot;
      if (!fill) count_victim(st, dc.slot, mx);
    }
    decide(st, UNISON_KIND_PROMOTE, pid, lane);
    if (!fill) {
      set_word(st, dc.slot, false, dc.order);
      st.P[dc.slot].v.y = did;
      st.free_s += sd;
      st.free_h -= sd;
      st.n_tide_demote++;
      decide(st, UNISON_KIND_TIDE_DEMOTE, did, lane);
    }
    rem -= by;
    st.free_s -= sp;
    st.free_h += sp;
    set_word(st, pc.slot, true, pc.order);
    *reinterpret_cast<uint2 *>(&st.P[pc.slot]) = make_uint2(p.x | kPromoted, pid | kFastBit);
    st.n_promote++;
  }
  return budget - rem;
}

// One replay.  kPol: its policy when the body is specialised for it, or -1
// for the body that reads the policy from the descriptor.  Branches are kept
// few (each costs an issue slot and a fetch, and one warp hides neither):
// classes and tiers are selected, and the loops that make room and migrate are
// the only ones an ordinary event passes.
template <int kMode, int kPol, bool kLean, int kForm, class Desc>
__device__ __forceinline__ void slot_replay(const Desc &D, const SlotDesc &Q, SlotBufs &bufs, unsigned char *smem,
                                            int lane) {
  constexpr bool kWide = kMode != kRanked || kPol != UNISON_SPEAR_TIDE, kMap8 = kForm == kFormMap8, kDeep = kForm != kFormPlain;
  const uint32_t policy = kPol >= 0 ? (uint32_t)kPol : D.policy;
  const bool spear = kMode != kRanked || policy == UNISON_SPEAR || policy == UNISON_SPEAR_TIDE;
  const bool tide_on = policy == UNISON_SPEAR_TIDE || policy == UNISON_LRU_TIDE;
  const bool belady = kMode == kRanked && policy == UNISON_BELADY;
  const bool timeout = kMode == kRanked && policy == UNISON_TIMEOUT && D.ttl != 0xFFFFFFFFu;

  Slots<kMode, kLean, kWide, kDeep> st;
  const uint32_t nslots = Q.nslots;
  st.sbits = Q.sbits;
  st.smask = (1u << Q.sbits) - 1u;
  unsigned char *p = smem;
  st.W = reinterpret_cast<uint32_t *>(p);
  p += slot_words(Q.nslots) * 4;
  st.P = reinterpret_cast<Payload<kWide> *>(p);
  p += ((size_t)Q.nslots * sizeof(Payload<kWide>) + 15) / 16 * 16;
  st.F = reinterpret_cast<uint16_t *>(p);
  p += ((size_t)Q.nslots * 2 + 15) / 16 * 16;
  uint8_t *const map8 = p;
  uint16_t *const map16 = reinterpret_cast<uint16_t *>(p);
  static_assert(kMode == kRanked || kForm == kFormPlain, "stale and online replays: SPEAR or SPEAR+TIDE, two-byte maps");
  // kStale: every session's live and snapshot rank, sessions changed since the
  // last sync; kOnline: every session's arrivals so far (saturating far above
  // the table's last row), the table
  uint32_t *live = nullptr, *snap = nullptr, *dirty = nullptr, n_dirty = 0, sync_arrivals = 0;
  uint16_t *turns = nullptr;
  OnlineTable *table = nullptr;
  if constexpr (kMode != kRanked) {
    unsigned char *q = p + round16((size_t)D.n_sessions * 2);
    st.L = reinterpret_cast<uint32_t *>(q);
    for (uint32_t i = lane; i < slot_words(Q.nslots); i += 32) st.L[i] = 0u;
    q += slot_words(Q.nslots) * 4;
    if constexpr (kMode == kStale) {
      live = reinterpret_cast<uint32_t *>(q);
      snap = live + D.n_sessions;
      dirty = snap + D.n_sessions;
      // a zero register row (gap average 0, turn 0, not done)
      for (uint32_t i = lane; i < D.n_sessions; i += 32) live[i] = snap[i] = Q.rank[D.n_events + i];
    } else {
      table = reinterpret_cast<OnlineTable *>(q);
      turns = reinterpret_cast<uint16_t *>(q + round16(sizeof(OnlineTable)));
      for (uint32_t i = lane; i < D.n_sessions; i += 32) turns[i] = 0;
      online_init(*table, lane);
    }
  }
  {
    uint4 *w4 = reinterpret_cast<uint4 *>(st.W);
#pragma unroll 1
    for (uint32_t i = lane; i < slot_words(Q.nslots) / 4; i += 32) w4[i] = make_uint4(0u, 0u, 0u, 0u);
    uint4 *m4 = reinterpret_cast<uint4 *>(p);
    const uint32_t mq = (D.n_sessions * (kMap8 ? 1u : 2u) + 15) / 16;
#pragma unroll 1
    for (uint32_t i = lane; i < mq; i += 32) m4[i] = make_uint4(0u, 0u, 0u, 0u);
    // the ring past the last event names session 0
#pragma unroll 1
    for (uint32_t i = lane; i <= kRing; i += 32) bufs.e[i].ev = make_uint4(0u, 0u, 0u, 0u);
    if (lane == 0) {
      st.P[0].v.y = kIdMask;  // a zero map entry finds no session
      st.F[0] = 0;
    }
    __syncwarp();
  }
  st.nfree = st.fresh = 0;
  st.free_s = st.room_s = Q.cap_s;
  st.free_h = st.room_h = Q.cap_h;
  st.status = UNISON_OK;
  st.h_lo = (uint32_t)kFnvOffset;
  st.h_hi = (uint32_t)(kFnvOffset >> 32);
  st.log = reinterpret_cast<uint2 *>(D.log);
  st.log_left = D.log ? D.log_cap : 0;
  st.n_evict = st.n_demote = st.n_promote = st.n_tide_demote = st.n_expire = st.n_tide_calls = 0;
  st.n_res = 0;
  st.vict_n = st.vict_diff = st.prom_n = st.prom_diff = 0;
  uint64_t dma_bytes = 0;
  uint32_t n_done = 0;
  const uint32_t n_turns = D.n_turns;
  uint8_t *note_out = reinterpret_cast<uint8_t *>(D.ttft) + 7ull * n_turns;
  // the DMA's last batch: its bytes (0: none in flight) and the time since it
  // began (saturating), advanced from completion to completion, which are less
  // than 2^32 us apart (the next event, and a turn, take less than 2^31)
  uint64_t busy_bytes = 0;
  uint32_t busy_us = 0;
  uint32_t oldest = 0;  // Timeout: see expire_slots
  const uint32_t kvb = D.kvb, max_sessions = D.max_sessions, dma = (uint32_t)D.dma;

  const uint32_t E = D.n_events;
  auto fetch = [&](uint32_t b) {
    const uint32_t i = b + lane;
    if (i < E) {
      SlotEvent &d = bufs.e[i & (kRing - 1)];
      async16(&d.ev, &D.ev[i]);
      if ((i & (kRing - 1)) == 0) async16(&bufs.e[kRing].ev, &D.ev[i]);
      if (spear && kMode != kOnline) async4(&d.aux.x, &Q.rank[i]);
      if (tide_on || kMode == kOnline) async4(&d.aux.y, &D.gq[i]);
      if (belady) async4(&d.aux.z, &D.nref[i]);
    }
    async_commit();
  };
  auto map_of = [&](uint32_t s) -> uint32_t { return kMap8 ? map8[s] : map16[s]; };
  fetch(0);
  fetch(32);
  async_wait<1>();
  __syncwarp();
  uint32_t last_done = bufs.e[0].ev.x;
  oldest = last_done;
  // the next event's session word and map entry are loaded while an event is
  // processed; a map entry changes only when its session is placed
  uint32_t nw = bufs.e[0].ev.y, nmap = map_of(nw & kIdMask), e = 0;

  while (e < E) {
    fetch(e + 64);
    async_wait<1>();  // the batch after this one has landed
    __syncwarp();
    const uint32_t end = min(E, e + 32);
    const SlotEvent *next = &bufs.e[e & (kRing - 1)];
    for (; e < end; e++) {
      const SlotEvent &rec = *next++;
      const uint32_t w1 = nw, s = w1 & kIdMask;
      uint32_t slot = nmap;
      nw = next->ev.y;
      const uint32_t ns = nw & kIdMask;
      st.e = e;
      if (timeout) {
        if constexpr (kWide) expire_slots(st, rec.ev.x, D.ttl, oldest, lane);
      }
      // the session's slot: the one its map entry names, if that slot is still
      // the session's own (an 8-bit entry names up to eight slots)
      if (kMap8) {
        const uint32_t c = slot + 256u * lane;
        const unsigned hit = __ballot_sync(kAll, c < st.fresh && (st.P[c].v.y & kIdMask) == s);
        slot += hit ? 256u * (__ffs(hit) - 1) : 0u;
      }
      const uint2 pl = *reinterpret_cast<const uint2 *>(&st.P[slot]);
      nmap = map_of(ns);
      __syncwarp();
      const bool found = (pl.y & kIdMask) == s, fast = (pl.y & kFastBit) != 0;
      const uint32_t size = pl.x & kSizeBits;

      if (w1 & kEvArrival) {
        const uint32_t n = rec.ev.w;
        const uint32_t cls = found ? (fast ? kClassFast : kClassHbm) : (w1 & kEvEdge ? kClassCold : kClassMiss);
        decide(st, cls, s, lane);
        uint32_t note = cls | (pl.x >> 31) * kNotePromoted;  // (the bit counts for fast-tier hits only)
        if (found) {
          clear_word(st, slot);
          const uint32_t in_s = size & (uint32_t)((int32_t)pl.y >> 31);
          st.free_s += in_s;
          st.free_h += size - in_s;
        }
        // placement; a session that was resident keeps its slot
        uint32_t tier = 0;  // 0 fast, 1 HBM, 2 bypassed
        if (!kLean && max_sessions && st.n_res - (found ? 1u : 0u) >= max_sessions && [&] {
              // as many pinned sessions as the limit allows: bypass
              uint32_t un = 0;
              for (uint32_t i = lane; i < st.fresh; i += 32) un += st.W[i] != 0u;
              return st.n_res - (found ? 1u : 0u) - __reduce_add_sync(kAll, un) >= max_sessions;
            }()) {
          tier = 2;
        } else if (n <= st.room_s) {
          while (n > st.free_s) {
            const Choice c = most_evictable_fast(st, map16, lane);
            if constexpr (kMode == kStale) count_victim(st, c.slot, max_of<kDeep>(st.L, st.fresh, lane));
            // it is demoted into HBM, displacing more evictable sessions
            // there, or dropped
            const uint2 d = payload(st, c.slot);
            const uint32_t sd = d.x & kSizeBits, did = d.y & kIdMask;
            st.free_s += sd;
            const bool keep =
                sd <= st.free_h || (c.any && sd <= st.room_h && make_hbm_room(st, map16, sd, c, lane));
            decide(st, keep ? (uint32_t)UNISON_KIND_DEMOTE : (uint32_t)UNISON_KIND_EVICT, did, lane);
            if (keep && c.any) {
              set_word(st, c.slot, false, c.order);
              st.P[c.slot].v.y = did;
              st.free_h -= sd;
              st.n_demote++;
            } else {
              if (!c.any) {  // no unpinned session although the tier is short of space
                st.status = UNISON_ERR_CAPACITY;
                goto out;
              }
              st.n_evict++;
              release_slot(st, c.slot);
            }
          }
          st.free_s -= n;
          st.room_s -= n;
        } else if (n <= st.room_h) {
          tier = 1;
          if (!make_hbm_room(st, map16, n, Choice{false, 0u, 0ull}, lane)) {
            st.status = UNISON_ERR_CAPACITY;
            goto out;
          }
          st.free_h -= n;
          st.room_h -= n;
        } else {
          tier = 2;
        }
        static_assert(UNISON_KIND_PLACE_H == UNISON_KIND_PLACE_S + 1 && UNISON_KIND_BYPASS == UNISON_KIND_PLACE_S + 2,
                      "placement kinds");
        if (tier == 2) {
          decide(st, UNISON_KIND_BYPASS, s, lane);
          if (found) release_slot(st, slot);
        } else {
          decide(st, UNISON_KIND_PLACE_S + tier, s, lane);
          if (!found) {
            // the last slot freed, else a new one
            const bool reuse = st.nfree != 0;
            const uint32_t f = st.F[reuse ? st.nfree - 1 : 0];
            slot = reuse ? f : st.fresh;
            st.nfree -= reuse ? 1u : 0u;
            st.fresh += reuse ? 0u : 1u;
            st.n_res++;
            if (slot >= nslots) {
              st.status = UNISON_ERR_CAPACITY;
              goto out;
            }
            __syncwarp();
            if (kMap8) map8[s] = (uint8_t)slot;
            else map16[s] = (uint16_t)slot;
            if (ns == s) nmap = kMap8 ? (slot & 255u) : slot;  // read before it was set
          }
          *reinterpret_cast<uint2 *>(&st.P[slot]) = make_uint2(n, s | (tier ? 0u : kFastBit));
          if constexpr (kWide) {
            // a session with no next arrival ranks above every event index,
            // the smaller id higher
            if (belady) {
              const uint32_t nr = rec.aux.z;
              st.P[slot].v.z = nr == kNoRef ? E + D.n_sessions - s : nr + 1u;
            }
          }
          if (!kLean && max_sessions) {
            while (st.n_res > max_sessions) {
              // the most evictable of both tiers
              const Choice f = most_evictable_fast(st, map16, lane), h = most_evictable_hbm(st, map16, lane);
              if (!f.any && !h.any) {
                st.status = UNISON_ERR_CAPACITY;
                goto out;
              }
              const uint32_t vs = f.any && (!h.any || f.order > h.order) ? f.slot : h.slot, vw = st.W[vs];
              if constexpr (kMode == kStale) {
                const uint32_t lh = max_hbm_of<kDeep>(st.L, st.fresh, lane), lf = max_of<kDeep>(st.L, st.fresh, lane);
                count_victim(st, vs, max(lh > kFastBit ? lh & ~kFastBit : 0u, lf & kFastBit ? lf & ~kFastBit : 0u));
              }
              const uint2 v = payload(st, vs);
              const uint32_t sv = v.x & kSizeBits;
              st.free_s += vw & kFastBit ? sv : 0u;
              st.free_h += vw & kFastBit ? 0u : sv;
              decide(st, UNISON_KIND_EVICT, v.y & kIdMask, lane);
              st.n_evict++;
              release_slot(st, vs);
              __syncwarp();
            }
          }
        }
        *note_out++ = (uint8_t)(note | tier << kNotePlaceShift);  // (every lane the same byte)
        if constexpr (kMode == kOnline) {
          const uint32_t k = turns[s];
          __syncwarp();
          turns[s] = (uint16_t)(k < 0xFFFFu ? k + 1 : k);
        }
      } else {
        // completion: the session is unpinned (if resident) with its new rank
        n_done++;
        const uint32_t now = rec.ev.x;
        const uint32_t el = busy_us + (now - last_done);
        busy_us = el < busy_us ? kAll : el;
        last_done = now;
        if (found) {
          if constexpr (kMode == kOnline) {
            const bool done = (w1 & kEvEdge) != 0;
            const uint32_t g = rec.aux.y, t = (uint32_t)turns[s] - 1u;
            st.P[slot].v.z = g;
            st.P[slot].v.w = done ? kAll : t;  // a completed session keeps the maximal key
            set_word(st, slot, fast, online_word(done ? 1ull << 39 : online_score(*table, g, t), s));
          } else {
            uint32_t rk;
            if (kMode == kStale) rk = snap[s];  // residents rank by their snapshot rows
            else if (spear) rk = rec.aux.x;
            else rk = n_turns - n_done + 1u;  // the later the touch, the less evictable
            if constexpr (kWide) {
              if (belady) rk = st.P[slot].v.z;
              if (timeout) st.P[slot].v.w = now;
            }
            st.W[slot] = rk << st.sbits | slot | (pl.y & kFastBit);
            if constexpr (kMode == kStale) st.L[slot] = rec.aux.x << st.sbits | slot | (pl.y & kFastBit);
          }
          const uint32_t in_s = size & (uint32_t)((int32_t)pl.y >> 31);
          st.room_s += in_s;
          st.room_h += size - in_s;
        }
        if constexpr (kMode == kOnline) {
          // Sec. V-F: the finished session's turn count joins the table, and
          // every resident is ranked under the rebuilt one
          if ((w1 & kEvEdge) && online_add(*table, turns[s], D.bucket, D.penalty, lane)) {
            for (uint32_t i = lane; i < st.fresh; i += 32) {
              const uint32_t w = st.W[i];
              const uint4 v = st.P[i].v;
              if (w == 0u || v.w == kAll) continue;
              const uint64_t o = online_word(online_score(*table, v.z, v.w), v.y & kIdMask);
              st.W[i] = (uint32_t)(o >> 32) | (w & kFastBit);
              st.L[i] = (uint32_t)o;
            }
            __syncwarp();
          }
        }
        if (tide_on) {
          // the DMA is free again from start + ceil(bytes / rate) us on, i.e.
          // once the elapsed us times the rate cover the bytes.  A batch's
          // bytes are at most 2^31 us of the rate, so the saturated time does.
          const bool busy = (uint64_t)busy_us * dma < busy_bytes;
          if (!busy && !(w1 & kEvEdge)) {
            st.n_tide_calls++;
            busy_bytes = tide_slots(st, map16, (uint64_t)rec.aux.y * dma, kvb, lane);  // (0 at rate 0: no budget)
            dma_bytes += busy_bytes;
            busy_us = 0;
          }
        }
      }
      if constexpr (kMode == kStale) {
        live[s] = rec.aux.x;
        __syncwarp();
        if (n_dirty < kDirtySlots) dirty[n_dirty] = s;
        n_dirty++;
        // a sync point copies every live row into the snapshot, after the
        // event's own decisions: the rows changed since the last one, a lane
        // each (a session noted twice is copied twice, alike), or all of them
        bool sync = D.stale_sync == UNISON_SYNC_EVENT;
        if ((w1 & kEvArrival) && D.stale_sync == UNISON_SYNC_ARRIVALS) sync = ++sync_arrivals % D.stale_m == 0;
        if (!(w1 & kEvArrival) && D.stale_sync == UNISON_SYNC_GAP_START) sync = !(w1 & kEvEdge);
        if (sync) {
          __syncwarp();
          if (n_dirty <= kDirtySlots) {
            for (uint32_t i = lane; i < n_dirty; i += 32) {
              const uint32_t d = dirty[i], r = live[d], at = map16[d];
              snap[d] = r;
              const uint32_t w = st.W[at];
              if ((st.P[at].v.y & kIdMask) == d && w != 0u) st.W[at] = r << st.sbits | at | (w & kFastBit);
            }
          } else {
            for (uint32_t i = lane; i < D.n_sessions; i += 32) snap[i] = live[i];
            for (uint32_t i = lane; i < st.fresh; i += 32) st.W[i] = st.L[i];
          }
          __syncwarp();
          n_dirty = 0;
        }
      }
    }
  }
out:
  async_wait<0>();
  if (lane == 0) {
    // the counters that follow from the arrivals' notes are account_arrivals'
    unison_replay_result r = {};
    r.events = min(e + (e < E ? 1u : 0u), E);
    r.evict = st.n_evict;
    r.demote = st.n_demote;
    r.promote = st.n_promote;
    r.tide_demote = st.n_tide_demote;
    r.expire = st.n_expire;
    r.dma_bytes = dma_bytes;
    r.tide_calls = st.n_tide_calls;
    r.ttft_n = (uint64_t)(note_out - (reinterpret_cast<uint8_t *>(D.ttft) + 7ull * n_turns));
    r.decision_hash = (uint64_t)st.h_hi << 32 | st.h_lo;
    r.vict_n = st.vict_n;
    r.vict_diff = st.vict_diff;
    r.prom_n = st.prom_n;
    r.prom_diff = st.prom_diff;
    if constexpr (!kLean) {
      const uint64_t made = r.ttft_n * 2 + r.evict + r.demote + r.promote + r.tide_demote + r.expire;
      if (D.log && made > D.log_cap && st.status == UNISON_OK) st.status = UNISON_ERR_LOG_FULL;
    }
    r.status = st.status;
    *D.result = r;
  }
}

// --------------------------------------------------------------------------
// Accounting of a replay's arrivals (Sec. V-A), from the event loop's notes:
// request and placement counters, token sums, and the TTFT of every request.
// The prefill queue is q' = max(q, a) + p with arrival a and prefill p; a run
// of requests is q' = max(q + P, M), and two runs compose to P1 + P2 and
// max(M1 + P2, M2), so the block scans 1,024 events at a time.  The event loop
// is a serial chain and the queue took about 22 of an arrival's instructions
// in it; here it takes about 0.85 of ttft_median_kernel's 1.22 ms over the
// 1,024-replay sweep, where leaving it out of the loop saved 6.6.  Not faster:
// 512 threads (1.44 ms), the next chunk's events loaded ahead (1.35 to 1.41),
// counters packed in 16 bits (1.24).  Times that
// could pass 2^63 ns (D.slot.serial) wrap as the recurrence does when one
// thread walks it.
// Values overwrite the notes in place: the 8-byte values of arrivals up to i
// end at or before the notes of arrivals past i (8 (i + 1) <= 7 n + i + 1), and
// a chunk's notes are read before its values are stored.
// --------------------------------------------------------------------------
constexpr int kAccThreads = 256, kAccItems = 4, kAccChunk = kAccThreads * kAccItems;

struct AccShared {
  unsigned long long us[8], p[8], m[8];
  uint32_t n[8];
  uint32_t cnt[8];
  unsigned long long tok[4], sum[2];
};

template <class Desc>
__device__ void account_arrivals(const Desc &D, AccShared &sh) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t E = D.n_events, load = D.load;
  const uint64_t n_arr = D.result->ttft_n;
  const uint64_t prefill_ns = D.prefill_ns;
  const uint64_t ns_per_us = (1000u % load == 0) ? 1000u / load : 0u;  // 0: divide exactly
  const uint8_t *const notes = reinterpret_cast<const uint8_t *>(D.ttft) + 7ull * D.n_turns;
  uint32_t cnt[8] = {};            // cold, fast, HBM, miss; promoted; placed fast, HBM, bypassed
  unsigned long long tok[4] = {};  // fast, HBM, miss; needed
  unsigned long long s_lo = 0, s_hi = 0;
  auto arrival_ns = [&](uint64_t us) { return ns_per_us ? us * ns_per_us : us * 1000ull / load; };
  auto note = [&](uint32_t c, uint32_t in, uint32_t prev) -> uint64_t {  // counts it; its prefill tokens
    const uint32_t cls = c & 3u;
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) cnt[k] += cls == k;
    cnt[4] += (c & (kNotePromoted | 3u)) == (kNotePromoted | kClassFast);
#pragma unroll
    for (uint32_t k = 0; k < 3; k++) cnt[5 + k] += c >> kNotePlaceShift == k;
#pragma unroll
    for (uint32_t k = 0; k < 3; k++) tok[k] += cls == k + 1 ? prev : 0u;
    tok[3] += cls != kClassCold ? in : 0u;
    return cls == kClassFast || cls == kClassHbm ? in - prev : in;
  };
  auto add = [&](uint64_t v) {
    const unsigned long long lo = s_lo + v;
    s_hi += lo < s_lo;
    s_lo = lo;
  };
  if (tid < 8) sh.cnt[tid] = 0;
  if (tid < 4) sh.tok[tid] = 0;
  if (tid < 2) sh.sum[tid] = 0;
  __syncthreads();
  if (D.slot.serial) {
    if (tid == 0) {
      uint64_t us = 0, q = 0, i = 0;
      for (uint32_t e = 0; e < E && i < n_arr; e++) {
        const uint4 ev = D.ev[e];
        if (e) us += (uint32_t)(ev.x - D.ev[e - 1].x);
        if (!(ev.y & kEvArrival)) continue;
        const uint64_t p = note(notes[i], ev.z, D.prev_out[e]), a = arrival_ns(us);
        if (q < a) q = a;
        q += p * prefill_ns;
        D.ttft[i++] = q - a;
        add(q - a);
      }
    }
  } else {
    unsigned long long us0 = 0, q0 = 0;  // before the chunk
    uint64_t i0 = 0;
    for (uint32_t base = 0; base < E && i0 < n_arr; base += kAccChunk) {
      const uint32_t e0 = base + kAccItems * tid;
      uint4 ev[kAccItems];
      uint32_t prev[kAccItems];
      uint32_t t = e0 > 0 && e0 < E ? D.ev[e0 - 1].x : 0u;
#pragma unroll
      for (int k = 0; k < kAccItems; k++) {
        const bool in = e0 + k < E;
        ev[k] = in ? D.ev[e0 + k] : make_uint4(0u, 0u, 0u, 0u);
        prev[k] = in ? D.prev_out[e0 + k] : 0u;
      }
      // time and arrivals up to each thread's first event
      if (e0 == 0) t = ev[0].x;
      unsigned long long us = 0, rel[kAccItems];
      uint32_t n = 0;
#pragma unroll
      for (int k = 0; k < kAccItems; k++) {
        if (e0 + k < E) us += (uint32_t)(ev[k].x - t);
        t = ev[k].x;
        rel[k] = us;
        n += ev[k].y >> 31;
      }
      static_assert(kEvArrival == 1u << 31, "arrival flag");
      unsigned long long us_in = us;
      uint32_t n_in = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kAll, us_in, o);
        const uint32_t z = __shfl_up_sync(kAll, n_in, o);
        if ((int)lane >= o) {
          us_in += y;
          n_in += z;
        }
      }
      if (lane == 31) {
        sh.us[warp] = us_in;
        sh.n[warp] = n_in;
      }
      __syncthreads();
      unsigned long long us_b = us0 + us_in - us;
      uint64_t i = i0 + n_in - n;
      uint32_t n_all = 0;
#pragma unroll
      for (uint32_t w = 0; w < 8; w++) {
        if (w < warp) {
          us_b += sh.us[w];
          i += sh.n[w];
        }
        us0 += sh.us[w];
        n_all += sh.n[w];
      }
      // each arrival's time and prefill, the thread's run of the queue
      unsigned long long P = 0, M = 0, a[kAccItems], p[kAccItems];
      uint64_t at = i;
#pragma unroll
      for (int k = 0; k < kAccItems; k++) {
        a[k] = p[k] = 0;
        if ((ev[k].y & kEvArrival) && at < n_arr) {
          p[k] = note(notes[at], ev[k].z, prev[k]) * prefill_ns;
          a[k] = arrival_ns(us_b + rel[k]);
          at++;
          M = max(M, a[k]) + p[k];  // max(M + p, a + p)
          P += p[k];
        }
      }
      unsigned long long Pi = P, Mi = M;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kAll, Pi, o), z = __shfl_up_sync(kAll, Mi, o);
        if ((int)lane >= o) {
          Mi = max(z + Pi, Mi);
          Pi += y;
        }
      }
      if (lane == 31) {
        sh.p[warp] = Pi;
        sh.m[warp] = Mi;
      }
      __syncthreads();  // and every note of the chunk has been read
      const unsigned long long Pe = __shfl_up_sync(kAll, Pi, 1), Me = __shfl_up_sync(kAll, Mi, 1);
      unsigned long long q = q0;
#pragma unroll
      for (uint32_t w = 0; w < 8; w++) {
        if (w < warp) q = max(q + sh.p[w], sh.m[w]);
        q0 = max(q0 + sh.p[w], sh.m[w]);
      }
      if (lane) q = max(q + Pe, Me);
#pragma unroll
      for (int k = 0; k < kAccItems; k++) {
        if ((ev[k].y & kEvArrival) && i < n_arr) {
          q = max(q, a[k]) + p[k];
          D.ttft[i++] = q - a[k];
          add(q - a[k]);
        }
      }
      i0 += n_all;
      __syncthreads();  // the next chunk rewrites the shared totals
    }
  }
#pragma unroll
  for (int k = 0; k < 8; k++) atomicAdd(&sh.cnt[k], cnt[k]);
#pragma unroll
  for (int k = 0; k < 4; k++) atomicAdd(&sh.tok[k], tok[k]);
  const unsigned long long before = atomicAdd(&sh.sum[0], s_lo);
  atomicAdd(&sh.sum[1], s_hi + (before + s_lo < before ? 1ull : 0ull));
  __syncthreads();
  if (tid == 0) {
    unison_replay_result &r = *D.result;
    r.cold = sh.cnt[0];
    r.hit_s = sh.cnt[1];
    r.hit_h = sh.cnt[2];
    r.miss = sh.cnt[3];
    r.req_warm = sh.cnt[1] + sh.cnt[2] + sh.cnt[3];
    r.promoted_then_hit_s = sh.cnt[4];
    r.place_s = sh.cnt[5];
    r.place_h = sh.cnt[6];
    r.bypass = sh.cnt[7];
    r.tok_hit_s = sh.tok[0];
    r.tok_hit_h = sh.tok[1];
    r.tok_miss = sh.tok[2];
    r.tok_needed = sh.tok[3];
    r.tok_computed = sh.tok[3] - sh.tok[0] - sh.tok[1];  // a hit computes in - prev
    r.ttft_sum_lo = sh.sum[0];
    r.ttft_sum_hi = sh.sum[1];
    // every decision has its counter
    r.log_len = n_arr * 2 + r.evict + r.demote + r.promote + r.tide_demote + r.expire;
  }
  __syncthreads();
}

// --------------------------------------------------------------------------
// Ranks of a key stream.  A session's key after a final completion is the
// maximal one, so those rank by descending id above all others
// (key_stream_kernel writes them).  The live completions' keys, given in
// order of descending session id, are sorted by key: least-significant-digit
// radix passes of 8 bits, each stable, so ties keep the larger id first --
// the packed key's order.  One block a key stream: each warp owns a run of
// the sequence, counts its digits, and after a scan over (digit, warp)
// places them in order (the lanes of 32 values with one digit find their
// places by a match).
// --------------------------------------------------------------------------
constexpr int kSortThreads = 1024;
constexpr int kSortWarps = kSortThreads / 32;
constexpr size_t kSortSmem = sizeof(uint32_t) * kSortWarps * 256;

struct RankDesc {
  unsigned long long *a, *b;  // [n] values key40 << 24 | entry of `rank`, and a second buffer
  uint32_t *rank;             // [E], or [E + S] with every event's rank and the zero rows'
  uint32_t n;
  uint32_t all;  // 1: ranks of every event's key and of the zero register rows (stale replays)
};

// Scratch of rank_keys_body beside the digit counts.
struct SortShared {
  unsigned long long all[kSortWarps], any[kSortWarps];
  uint32_t wtot[8], place[256];
};

__device__ void rank_keys_body(const RankDesc &d, uint32_t (*cnt)[256], SortShared &sh) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n = d.n;
  if (n == 0) return;
  unsigned long long *src = d.a, *dst = d.b;
  // digits on which every value agrees need no pass
  unsigned long long an = ~0ull, orv = 0ull;
  for (uint32_t i = tid; i < n; i += kSortThreads) {
    const unsigned long long v = src[i];
    an &= v;
    orv |= v;
  }
  for (int o = 16; o; o >>= 1) {
    an &= __shfl_xor_sync(kAll, an, o);
    orv |= __shfl_xor_sync(kAll, orv, o);
  }
  if (lane == 0) {
    sh.all[warp] = an;
    sh.any[warp] = orv;
  }
  __syncthreads();
  for (int w = 0; w < kSortWarps; w++) {
    an &= sh.all[w];
    orv |= sh.any[w];
  }
  const unsigned long long vary = an ^ orv;
  // warp w owns values [w * run, (w + 1) * run), a multiple of 32
  const uint32_t run = ((n + kSortThreads - 1) / kSortThreads) * 32;
  const uint32_t lo = min(n, warp * run), hi = min(n, lo + run);
  for (int bit = 24; bit < 64; bit += 8) {
    if (((vary >> bit) & 0xFFull) == 0) continue;
    for (uint32_t i = lane; i < 256; i += 32) cnt[warp][i] = 0;
    __syncwarp();
    for (uint32_t i0 = lo; i0 < hi; i0 += 128) {
      unsigned long long v[4];
#pragma unroll
      for (int q = 0; q < 4; q++) v[q] = i0 + 32 * q + lane < hi ? src[i0 + 32 * q + lane] : 0ull;
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (i0 + 32 * q + lane < hi) atomicAdd(&cnt[warp][(uint32_t)(v[q] >> bit) & 255u], 1u);
    }
    __syncthreads();
    // exclusive places: digit-major, then warp
    if (tid < 256) {
      uint32_t tot = 0;
      for (int w = 0; w < kSortWarps; w++) {
        const uint32_t c = cnt[w][tid];
        cnt[w][tid] = tot;
        tot += c;
      }
      uint32_t incl = tot;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, incl, o);
        if ((int)lane >= o) incl += y;
      }
      if (lane == 31) sh.wtot[warp] = incl;
      sh.place[tid] = incl - tot;
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t base = sh.place[tid];
      for (uint32_t w = 0; w < warp; w++) base += sh.wtot[w];
      for (int w = 0; w < kSortWarps; w++) cnt[w][tid] += base;
    }
    __syncthreads();
    for (uint32_t i0 = lo; i0 < hi; i0 += 128) {
      unsigned long long v[4];
#pragma unroll
      for (int q = 0; q < 4; q++) v[q] = i0 + 32 * q + lane < hi ? src[i0 + 32 * q + lane] : 0ull;
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const bool in = i0 + 32 * q + lane < hi;
        const uint32_t dg = in ? (uint32_t)(v[q] >> bit) & 255u : 256u + lane;
        const unsigned grp = __match_any_sync(kAll, dg);
        const uint32_t before = __popc(grp & ((1u << lane) - 1u));
        uint32_t at = 0;
        if (in) at = cnt[warp][dg] + before;
        __syncwarp();
        if (in && before == 0) cnt[warp][dg] += __popc(grp);
        __syncwarp();
        if (in) dst[at] = v[q];
      }
    }
    __syncthreads();
    unsigned long long *t = src;
    src = dst;
    dst = t;
  }
  for (uint32_t i = tid; i < n; i += kSortThreads) d.rank[(uint32_t)(src[i] & 0xFFFFFFull)] = i + 1;
}

}  // namespace unison_slots
