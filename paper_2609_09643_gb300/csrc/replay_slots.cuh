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
// and the load of the winner's size: 188 warp instructions and 1,010 cycles an
// event for the slowest of 152 sweep replays.  Sorted lists of 64-bit keys in
// the warp's registers, which this replaced, took 375 and 1,513 (49.2 -> 32.8 ms).
// One GB300, before and after: 1,024-replay sweep 65.0 -> 45.4 ms, 30 mixed
// paper-scale replays 76.3 -> 38.1 ms, 40,000-session pool 1,359 -> 760 ms, four
// tiny replays 1.68 -> 1.04 ms.
#pragma once

#include "common.cuh"

namespace unison_slots {

using namespace unison;

constexpr uint32_t kAll = 0xFFFFFFFFu;
constexpr uint32_t kFastBit = 0x80000000u;   // of a slot word
constexpr uint32_t kPromoted = 0x80000000u;  // of a payload's size word
constexpr uint32_t kSizeBits = 0x7FFFFFFFu;
constexpr uint32_t kInFast = 1, kInHbm = 2;
constexpr uint32_t kMostSlots = 2048;  // 16 words a lane

// A resident's payload: size (and whether TIDE promoted it), session and tier
// (bits 30-31).  Policies other than SPEAR+TIDE also keep the rank a Belady
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

struct SlotEvent {
  uint4 ev;   // time32, session | flags, in_tok, out_tok
  uint4 aux;  // previous turn's size (arrivals); rank and gap average (completions); next reference
};
struct SlotBufs {
  SlotEvent e[2][32];
};

// What one replay of the slot form reads besides its ReplayDesc.
struct SlotDesc {
  const uint32_t *rank;  // rank after each completion event (SPEAR policies), or null
  uint32_t cap_s, cap_h;  // tokens, at most the sum of every session's largest size (< 2^31)
  uint32_t nslots;        // slots the replay can need
  uint32_t sbits;         // slot bits of a word
  uint32_t map8;          // 1: the session map holds the slot's low byte only
};

// Bytes of shared memory of one replay: words, payloads, free slots, map.
__host__ __device__ inline size_t slot_words(uint32_t nslots) { return ((size_t)nslots + 127) / 128 * 128; }
__host__ inline size_t slot_bytes(uint32_t nslots, uint32_t n_sessions, bool wide, bool map8) {
  const size_t pay = (size_t)nslots * (wide ? 16 : 8), fr = ((size_t)nslots * 2 + 15) / 16 * 16;
  const size_t map = ((size_t)n_sessions * (map8 ? 1 : 2) + 15) / 16 * 16;
  return slot_words(nslots) * 4 + (pay + 15) / 16 * 16 + fr + map;
}

template <bool kWide>
struct Slots {
  uint32_t *W;
  Payload<kWide> *P;
  uint16_t *F;       // freed slots, a stack
  uint32_t nfree, fresh;  // entries of F; slots handed out at least once
  uint32_t nslots, sbits, smask;
  uint32_t used_s, used_h, pinned_s, pinned_h, cap_s, cap_h;  // tokens
  int status;
  // decision stream
  uint32_t e;
  uint64_t hash, log_len, log_cap;
  unison_decision *log;
  // counters (warp-uniform registers)
  uint32_t n_cold, n_hit_s, n_hit_h, n_miss, n_bypass, n_place_s, n_place_h;
  uint32_t n_evict, n_demote, n_promote, n_tide_demote, n_expire, n_tide_calls, n_pth, n_res;
};

// kLean: no decision log and no slot limit.
template <bool kLean, class St>
__device__ __forceinline__ void decide(St &st, uint32_t kind, uint32_t s, int lane) {
  const uint64_t w = ((uint64_t)st.e << 32) | (kind << 24 | s);
  st.hash = (st.hash ^ w) * kFnvPrime;
  if constexpr (!kLean) {
    if (st.log) {
      if (st.log_len < st.log_cap) {
        if (lane == 0) {
          unison_decision d;
          d.event = st.e;
          d.kind_session = (kind << 24) | s;
          st.log[st.log_len] = d;
        }
      } else if (st.status == UNISON_OK) {
        st.status = UNISON_ERR_LOG_FULL;
      }
    }
    st.log_len++;
  }
}

// Extremes over the words of every slot handed out so far (a multiple of 128
// words; the words past them are 0).
template <class St>
__device__ __forceinline__ uint32_t max_word(const St &st, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(st.W) + lane;
  uint4 v = w4[0];
  uint32_t m = max(max(v.x, v.y), max(v.z, v.w));
  for (uint32_t q = 128; q < st.fresh; q += 128) {
    w4 += 32;
    v = *w4;
    m = max(max(m, max(v.x, v.y)), max(v.z, v.w));
  }
  return __reduce_max_sync(kAll, m);
}
// The largest HBM word with its tier bit flipped: > kFastBit if there is one.
template <class St>
__device__ __forceinline__ uint32_t max_hbm(const St &st, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(st.W) + lane;
  uint32_t m = 0;
  for (uint32_t q = 0; q == 0 || q < st.fresh; q += 128, w4 += 32) {
    const uint4 v = *w4;
    m = max(max(m, max(v.x ^ kFastBit, v.y ^ kFastBit)), max(v.z ^ kFastBit, v.w ^ kFastBit));
  }
  return __reduce_max_sync(kAll, m);
}
// The largest word, and the smallest word above 0 less 1 (below
// kFastBit - 1 if there is an HBM word).
template <class St>
__device__ __forceinline__ void extremes(const St &st, uint32_t &mx, uint32_t &mn, int lane) {
  const uint4 *w4 = reinterpret_cast<const uint4 *>(st.W) + lane;
  uint4 v = w4[0];
  uint32_t a = max(max(v.x, v.y), max(v.z, v.w));
  uint32_t b = min(min(v.x - 1u, v.y - 1u), min(v.z - 1u, v.w - 1u));
  for (uint32_t q = 128; q < st.fresh; q += 128) {
    w4 += 32;
    v = *w4;
    a = max(max(a, max(v.x, v.y)), max(v.z, v.w));
    b = min(min(b, min(v.x - 1u, v.y - 1u)), min(v.z - 1u, v.w - 1u));
  }
  mx = __reduce_max_sync(kAll, a);
  mn = __reduce_min_sync(kAll, b);
}

// Slot stores: every lane stores the same value to the same place, so each
// lane's later loads see it without a warp barrier; a __syncwarp separates a
// store from the loads of the old value before it.
template <class St>
__device__ __forceinline__ void release_slot(St &st, uint32_t slot) {
  st.W[slot] = 0u;
  st.P[slot].v.y = kIdMask;  // no session has this id
  st.F[st.nfree] = (uint16_t)slot;
  st.nfree++;
}

template <bool kLean, class St>
__device__ __forceinline__ void evict_slot(St &st, uint32_t slot, uint32_t id, int lane) {
  decide<kLean>(st, UNISON_KIND_EVICT, id, lane);
  st.n_evict++;
  st.n_res--;
  release_slot(st, slot);
}

// Room in HBM for `size` tokens against its unpinned residents: evicts the
// most evictable ones, only those above `floor_word` (a word without the tier
// bit; 0 accepts every one).  False when the next one is not above it.
template <bool kLean, class St>
__device__ __forceinline__ bool make_hbm_room(St &st, uint32_t size, uint32_t floor_word, int lane) {
  while (st.used_h + size > st.cap_h) {
    const uint32_t m = max_hbm(st, lane);
    const uint32_t w = m ^ kFastBit;
    if (m <= kFastBit || w < floor_word) return false;
    const uint32_t slot = w & st.smask;
    const uint2 p = make_uint2(st.P[slot].v.x, st.P[slot].v.y);
    __syncwarp();
    st.used_h -= p.x & kSizeBits;
    evict_slot<kLean>(st, slot, p.y & kIdMask, lane);
  }
  return true;
}

// A session demoted out of the fast tier (its word w, payload p): into HBM,
// displacing more evictable sessions there, or dropped.
template <bool kLean, class St>
__device__ __forceinline__ void demote_slot(St &st, uint32_t w, uint32_t slot, uint32_t px, uint32_t py, int lane) {
  const uint32_t size = px & kSizeBits, id = py & kIdMask;
  const uint32_t hw = w & ~kFastBit;
  if (size > st.cap_h - st.pinned_h || !make_hbm_room<kLean>(st, size, hw, lane)) {
    evict_slot<kLean>(st, slot, id, lane);
    return;
  }
  st.W[slot] = hw;
  st.P[slot].v.y = id | (kInHbm << 30);
  st.used_h += size;
  decide<kLean>(st, UNISON_KIND_DEMOTE, id, lane);
  st.n_demote++;
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
// events need one comparison; a pass over the slots renews it.
template <class St>
__device__ __forceinline__ void expire_slots(St &st, uint32_t now, uint32_t ttl, uint32_t &oldest, int lane) {
  while (now - oldest >= ttl) {
    uint32_t id = kAll, at = 0, age = 0;
    for (uint32_t i = lane; i < st.fresh; i += 32) {
      if (st.W[i] == 0) continue;
      const uint32_t a = now - st.P[i].v.w;
      if (a >= ttl) {
        const uint32_t s = st.P[i].v.y & kIdMask;
        if (s < id) {
          id = s;
          at = i;
        }
      } else {
        age = max(age, a);
      }
    }
    const uint32_t first = __reduce_min_sync(kAll, id);
    if (first == kAll) {
      oldest = now - __reduce_max_sync(kAll, age);
      return;
    }
    const uint32_t slot = __shfl_sync(kAll, at, __ffs(__ballot_sync(kAll, id == first)) - 1);
    const uint32_t w = st.W[slot], size = st.P[slot].v.x & kSizeBits;
    __syncwarp();
    if (w & kFastBit) st.used_s -= size;
    else st.used_h -= size;
    decide<false>(st, UNISON_KIND_EXPIRE, first, lane);
    st.n_expire++;
    st.n_res--;
    release_slot(st, slot);
    __syncwarp();
  }
}

// TIDE at a gap_start with `budget` bytes, one move at a time as the pair loop
// of Algorithm 1 has it: phase 1 promotes the least evictable HBM sessions
// into free fast-tier space, phase 2 swaps the least evictable HBM session
// with the most evictable fast-tier one.  Returns the bytes moved.
template <bool kLean, class St>
__device__ __forceinline__ uint64_t tide_slots(St &st, uint64_t budget, uint32_t kvb, int lane) {
  uint64_t rem = budget;
  bool fill = true;  // phase 1
  for (;;) {
    uint32_t mx, mn;
    extremes(st, mx, mn, lane);
    if (mn >= kFastBit - 1u) break;  // HBM holds no unpinned session
    const uint32_t pw = mn + 1u, pslot = pw & st.smask;
    const uint32_t dslot = mx & st.smask;  // a valid slot even when mx names none
    const uint2 p = make_uint2(st.P[pslot].v.x, st.P[pslot].v.y);
    const uint2 d = make_uint2(st.P[dslot].v.x, st.P[dslot].v.y);
    const uint32_t sp = p.x & kSizeBits, pid = p.y & kIdMask;
    __syncwarp();
    if (fill) {
      const uint64_t by = (uint64_t)sp * kvb;
      if (by <= rem && st.used_s + sp <= st.cap_s) {
        rem -= by;
        st.used_s += sp;
        st.used_h -= sp;
        st.W[pslot] = pw | kFastBit;
        st.P[pslot].v.x = p.x | kPromoted;
        st.P[pslot].v.y = pid | (kInFast << 30);
        decide<kLean>(st, UNISON_KIND_PROMOTE, pid, lane);
        st.n_promote++;
        continue;
      }
      fill = false;
    }
    if (mx < kFastBit || (mx & ~kFastBit) <= pw) break;  // no fast-tier session, or none more evictable
    const uint32_t sd = d.x & kSizeBits, did = d.y & kIdMask;
    const uint64_t by = (uint64_t)(sp + sd) * kvb;
    if (by > rem || st.used_s - sd + sp > st.cap_s || st.used_h - sp + sd > st.cap_h) break;
    rem -= by;
    st.used_s = st.used_s - sd + sp;
    st.used_h = st.used_h - sp + sd;
    st.W[pslot] = pw | kFastBit;
    st.P[pslot].v.x = p.x | kPromoted;
    st.P[pslot].v.y = pid | (kInFast << 30);
    st.W[dslot] = mx & ~kFastBit;
    st.P[dslot].v.y = did | (kInHbm << 30);
    decide<kLean>(st, UNISON_KIND_PROMOTE, pid, lane);
    decide<kLean>(st, UNISON_KIND_TIDE_DEMOTE, did, lane);
    st.n_promote++;
    st.n_tide_demote++;
  }
  return budget - rem;
}

// One replay.  kPol: its policy when the body is specialised for it, or -1
// for the body that reads the policy from the descriptor.
template <int kPol, bool kLean, class Desc>
__device__ __forceinline__ void slot_replay(const Desc &D, const SlotDesc &Q, SlotBufs &bufs, unsigned char *smem,
                                            int lane) {
  constexpr bool kWide = kPol != UNISON_SPEAR_TIDE;
  const uint32_t policy = kPol >= 0 ? (uint32_t)kPol : D.policy;
  const bool spear = policy == UNISON_SPEAR || policy == UNISON_SPEAR_TIDE;
  const bool tide_on = policy == UNISON_SPEAR_TIDE || policy == UNISON_LRU_TIDE;
  const bool belady = policy == UNISON_BELADY;
  const bool timeout = policy == UNISON_TIMEOUT && D.ttl != 0xFFFFFFFFu;

  Slots<kWide> st;
  st.nslots = Q.nslots;
  st.sbits = Q.sbits;
  st.smask = (1u << Q.sbits) - 1u;
  unsigned char *p = smem;
  st.W = reinterpret_cast<uint32_t *>(p);
  p += slot_words(Q.nslots) * 4;
  st.P = reinterpret_cast<Payload<kWide> *>(p);
  p += ((size_t)Q.nslots * sizeof(Payload<kWide>) + 15) / 16 * 16;
  st.F = reinterpret_cast<uint16_t *>(p);
  p += ((size_t)Q.nslots * 2 + 15) / 16 * 16;
  uint8_t *const map8 = Q.map8 ? p : nullptr;
  uint16_t *const map16 = reinterpret_cast<uint16_t *>(p);
  {
    uint4 *w4 = reinterpret_cast<uint4 *>(st.W);
    for (uint32_t i = lane; i < slot_words(Q.nslots) / 4; i += 32) w4[i] = make_uint4(0u, 0u, 0u, 0u);
    uint4 *m4 = reinterpret_cast<uint4 *>(p);
    const uint32_t mq = (D.n_sessions * (Q.map8 ? 1u : 2u) + 15) / 16;
    for (uint32_t i = lane; i < mq; i += 32) m4[i] = make_uint4(0u, 0u, 0u, 0u);
    if (lane == 0) st.P[0].v.y = kIdMask;  // a zero map entry finds no session
    __syncwarp();
  }
  st.nfree = st.fresh = 0;
  st.used_s = st.used_h = st.pinned_s = st.pinned_h = 0;
  st.cap_s = Q.cap_s;
  st.cap_h = Q.cap_h;
  st.status = UNISON_OK;
  st.hash = kFnvOffset;
  st.log = D.log;
  st.log_cap = D.log_cap;
  st.log_len = 0;
  st.n_cold = st.n_hit_s = st.n_hit_h = st.n_miss = st.n_bypass = st.n_place_s = st.n_place_h = 0;
  st.n_evict = st.n_demote = st.n_promote = st.n_tide_demote = st.n_expire = st.n_tide_calls = st.n_pth = 0;
  st.n_res = 0;
  uint64_t tok_hit_s = 0, tok_hit_h = 0, tok_miss = 0, tok_needed = 0, dma_bytes = 0;

  // TTFT queue (Sec. V-A): arrivals compressed by the load factor.
  uint64_t rel_us = 0, q_free = 0;
  uint32_t n_arr = 0, n_ev = 0, n_done = 0;
  const uint32_t load = D.load;
  const uint64_t prefill_ns = D.prefill_ns;
  const uint32_t n_turns = D.n_turns;
  uint64_t *const ttft_out = D.ttft;
  const uint64_t ns_per_us = (1000u % load == 0) ? 1000u / load : 0u;  // 0: divide exactly
  unsigned long long s_lo = 0, s_hi = 0;
  bool dma_busy = false;
  uint64_t busy_from = 0, busy_bytes = 0;  // the DMA's last batch: start (rel_us) and bytes
  uint32_t oldest = 0;                     // Timeout: see expire_slots
  const uint32_t kvb = D.kvb, max_sessions = D.max_sessions;
  const uint64_t dma = D.dma;

  const uint32_t E = D.n_events;
  auto fetch = [&](uint32_t b, int bi) {
    const uint32_t i = b + lane;
    if (i < E) {
      SlotEvent &d = bufs.e[bi][lane];
      async16(&d.ev, &D.ev[i]);
      async4(&d.aux.x, &D.prev_out[i]);
      if (spear) async4(&d.aux.y, &Q.rank[i]);
      if (tide_on) async4(&d.aux.z, &D.gq[i]);
      if (belady) async4(&d.aux.w, &D.nref[i]);
    }
    async_commit();
  };
  auto map_of = [&](uint32_t s) -> uint32_t { return map8 ? map8[s] : map16[s]; };
  fetch(0, 0);
  async_wait<0>();
  __syncwarp();
  uint32_t prev_now = E ? bufs.e[0][0].ev.x : 0u;
  oldest = prev_now;

  int bi = 0;
  for (uint32_t b = 0; b < E && st.status != UNISON_ERR_CAPACITY; b += 32, bi ^= 1) {
    if (b + 32 < E) {
      fetch(b + 32, bi ^ 1);
      async_wait<1>();  // this batch's copies have landed
    } else {
      async_wait<0>();
    }
    __syncwarp();
    const uint32_t cnt = min(32u, E - b);
    // the next event's record and map entry are loaded while this one is
    // processed; a map entry changes only when its session is placed
    uint4 nev = bufs.e[bi][0].ev, naux = bufs.e[bi][0].aux;
    uint32_t nmap = map_of(nev.y & kIdMask);
    for (uint32_t j = 0; j < cnt; j++) {
      const uint4 ev = nev, aux = naux;
      uint32_t slot = nmap;
      const uint32_t jn = min(j + 1, cnt - 1);
      nev = bufs.e[bi][jn].ev;
      naux = bufs.e[bi][jn].aux;
      const uint32_t now = ev.x, s = ev.y & kIdMask;
      const bool arrival = (ev.y & kEvArrival) != 0, edge = (ev.y & kEvEdge) != 0;
      st.e = b + j;
      n_ev++;
      rel_us += (uint32_t)(now - prev_now);
      prev_now = now;
      if (kPol < 0 && timeout) {
        if constexpr (kWide) expire_slots(st, now, D.ttl, oldest, lane);
      }
      // the session's slot: the one its map entry names, if that slot is still
      // the session's own (an 8-bit entry names up to eight slots)
      bool found;
      if (map8) {
        const uint32_t c = slot + 256u * lane;
        const unsigned hit = __ballot_sync(kAll, c < st.fresh && (st.P[c].v.y & kIdMask) == s);
        found = hit != 0;
        slot += found ? 256u * (__ffs(hit) - 1) : 0u;
      }
      const uint2 pl = make_uint2(st.P[slot].v.x, st.P[slot].v.y);
      if (!map8) found = (pl.y & kIdMask) == s;
      nmap = map_of(nev.y & kIdMask);
      __syncwarp();

      if (arrival) {
        const uint32_t in = ev.z, n = ev.w, prev = aux.x;
        uint64_t prefill = in;
        if (edge) {
          decide<kLean>(st, UNISON_KIND_COLD, s, lane);
          st.n_cold++;
        } else {
          tok_needed += in;
          if (found) {
            const uint32_t size = pl.x & kSizeBits;
            prefill = in - prev;
            st.W[slot] = 0u;
            if (pl.y >> 30 == kInFast) {
              decide<kLean>(st, UNISON_KIND_HIT_S, s, lane);
              st.n_hit_s++;
              tok_hit_s += prev;
              if (pl.x & kPromoted) st.n_pth++;
              st.used_s -= size;
            } else {
              decide<kLean>(st, UNISON_KIND_HIT_H, s, lane);
              st.n_hit_h++;
              tok_hit_h += prev;
              st.used_h -= size;
            }
          } else {
            decide<kLean>(st, UNISON_KIND_MISS, s, lane);
            st.n_miss++;
            tok_miss += prev;
          }
        }
        {
          const uint64_t arr = ns_per_us ? rel_us * ns_per_us : rel_us * 1000ull / load;
          if (q_free < arr) q_free = arr;
          q_free += prefill * prefill_ns;
          const uint64_t v = q_free - arr;
          if (lane == 0 && n_arr < n_turns) ttft_out[n_arr] = v;
          n_arr++;
          const unsigned long long lo2 = s_lo + v;
          s_hi += (lo2 < s_lo);
          s_lo = lo2;
        }
        // placement; a session that was resident keeps its slot
        uint32_t tier = 0;
        if (!kLean && max_sessions && st.n_res - (found ? 1u : 0u) >= max_sessions && [&] {
              // as many pinned sessions as the limit allows: bypass
              uint32_t un = 0;
              for (uint32_t i = lane; i < st.fresh; i += 32) un += st.W[i] != 0u;
              return st.n_res - (found ? 1u : 0u) - __reduce_add_sync(kAll, un) >= max_sessions;
            }()) {
        } else if (n <= st.cap_s - st.pinned_s) {
          tier = kInFast;
          while (st.used_s + n > st.cap_s) {
            const uint32_t w = max_word(st, lane);  // the most evictable unpinned fast-tier session
            if (w < kFastBit) {
              st.status = UNISON_ERR_CAPACITY;
              break;
            }
            const uint32_t ds = w & st.smask;
            const uint2 d = make_uint2(st.P[ds].v.x, st.P[ds].v.y);
            __syncwarp();
            st.used_s -= d.x & kSizeBits;
            demote_slot<kLean>(st, w, ds, d.x, d.y, lane);
          }
        } else if (n <= st.cap_h - st.pinned_h) {
          tier = kInHbm;
          if (!make_hbm_room<kLean>(st, n, 0u, lane)) st.status = UNISON_ERR_CAPACITY;
        }
        if (st.status == UNISON_ERR_CAPACITY) break;
        if (tier) {
          if (!found) {
            if (st.nfree) {
              slot = st.F[--st.nfree];
            } else {
              slot = st.fresh++;
              if (slot >= st.nslots) {
                st.status = UNISON_ERR_CAPACITY;
                break;
              }
            }
            st.n_res++;
            __syncwarp();
            if (map8) map8[s] = (uint8_t)slot;
            else map16[s] = (uint16_t)slot;
          }
          st.P[slot].v.x = n;
          st.P[slot].v.y = s | (tier << 30);
          if constexpr (kWide) {
            // a session with no next arrival ranks above every event index,
            // the smaller id higher
            if (belady) st.P[slot].v.z = aux.w == kNoRef ? E + D.n_sessions - s : aux.w + 1u;
          }
          if (tier == kInFast) {
            st.used_s += n;
            st.pinned_s += n;
            decide<kLean>(st, UNISON_KIND_PLACE_S, s, lane);
            st.n_place_s++;
          } else {
            st.used_h += n;
            st.pinned_h += n;
            decide<kLean>(st, UNISON_KIND_PLACE_H, s, lane);
            st.n_place_h++;
          }
          if ((nev.y & kIdMask) == s) nmap = map8 ? (slot & 255u) : slot;  // read before it was set
          if (!kLean && max_sessions) {
            while (st.n_res > max_sessions) {
              // the most evictable of both tiers
              uint32_t m = 0;
              for (uint32_t i = lane; i < st.fresh; i += 32) m = max(m, st.W[i] & ~kFastBit);
              m = __reduce_max_sync(kAll, m);
              if (m == 0) {
                st.status = UNISON_ERR_CAPACITY;
                break;
              }
              const uint32_t vs = m & st.smask, vw = st.W[vs];
              const uint2 v = make_uint2(st.P[vs].v.x, st.P[vs].v.y);
              __syncwarp();
              if (vw & kFastBit) st.used_s -= v.x & kSizeBits;
              else st.used_h -= v.x & kSizeBits;
              evict_slot<kLean>(st, vs, v.y & kIdMask, lane);
              __syncwarp();
            }
            if (st.status == UNISON_ERR_CAPACITY) break;
          }
        } else {
          decide<kLean>(st, UNISON_KIND_BYPASS, s, lane);
          st.n_bypass++;
          if (found) {
            st.n_res--;
            release_slot(st, slot);
          }
        }
      } else {
        // completion: the session is unpinned (if resident) with its new rank
        n_done++;
        if (found) {
          uint32_t rk;
          if (spear) rk = aux.y + 1u;
          else rk = n_turns - n_done + 1u;  // the later the touch, the less evictable
          if constexpr (kWide) {
            if (belady) rk = st.P[slot].v.z;
            st.P[slot].v.w = now;
          }
          const uint32_t size = pl.x & kSizeBits;
          const bool fast = pl.y >> 30 == kInFast;
          st.W[slot] = rk << st.sbits | slot | (fast ? kFastBit : 0u);
          if (fast) st.pinned_s -= size;
          else st.pinned_h -= size;
        }
        if (!edge && tide_on) {
          // the DMA is free again from start + ceil(bytes / rate) us on, i.e.
          // once the elapsed us times the rate cover the bytes (the high word
          // of the product catches one past 2^64)
          if (dma_busy) {
            const uint64_t el = rel_us - busy_from;
            if (__umul64hi(el, dma) != 0 || el * dma >= busy_bytes) dma_busy = false;
          }
          if (!dma_busy) {
            st.n_tide_calls++;
            const uint64_t moved = tide_slots<kLean>(st, aux.z * dma, kvb, lane);
            if (moved) {
              dma_bytes += moved;
              if (dma) {
                dma_busy = true;
                busy_from = rel_us;
                busy_bytes = moved;
              }
            }
          }
        }
      }
    }
  }
  async_wait<0>();
  if (lane == 0) {
    const uint32_t warm = st.n_hit_s + st.n_hit_h + st.n_miss;
    unison_replay_result r = {};
    r.events = n_ev;
    r.req_warm = warm;
    r.cold = st.n_cold;
    r.hit_s = st.n_hit_s;
    r.hit_h = st.n_hit_h;
    r.miss = st.n_miss;
    r.bypass = st.n_bypass;
    r.place_s = st.n_place_s;
    r.place_h = st.n_place_h;
    r.evict = st.n_evict;
    r.demote = st.n_demote;
    r.promote = st.n_promote;
    r.tide_demote = st.n_tide_demote;
    r.expire = st.n_expire;
    r.tok_hit_s = tok_hit_s;
    r.tok_hit_h = tok_hit_h;
    r.tok_miss = tok_miss;
    r.tok_computed = tok_needed - tok_hit_s - tok_hit_h;  // a hit computes in - prev
    r.tok_needed = tok_needed;
    r.dma_bytes = dma_bytes;
    r.tide_calls = st.n_tide_calls;
    r.promoted_then_hit_s = st.n_pth;
    r.ttft_sum_lo = s_lo;
    r.ttft_sum_hi = s_hi;
    r.ttft_p50_ns = 0;
    r.ttft_n = n_arr;
    r.decision_hash = st.hash;
    // every decision has its counter
    r.log_len = (uint64_t)st.n_cold + warm + st.n_bypass + st.n_place_s + st.n_place_h + st.n_evict + st.n_demote +
                st.n_promote + st.n_tide_demote + st.n_expire;
    r.status = st.status;
    *D.result = r;
  }
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
  unsigned long long *a, *b;  // [n] values key40 << 24 | turn, and a second buffer
  const uint32_t *turn_ev;    // [2T]
  uint32_t *rank;             // [E]
  uint32_t n;
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
  for (uint32_t i = tid; i < n; i += kSortThreads) d.rank[d.turn_ev[2 * (uint32_t)(src[i] & 0xFFFFFFull) + 1]] = i;
}

}  // namespace unison_slots
