// Device side of the metric estimator (sm_103a).
//
//   enum_kernel   persistent, work-stealing CTAs.  Representative block (Sec. 4.2, 4.3):
//                 every (warp, access instruction) pair exactly -- per-instruction unique
//                 sectors (L1 request / write-through volumes) and half-warp bank cycles,
//                 once per access code where the block's footprints are made elsewhere
//                 (AccessCodes), else with the block bitmaps.  Wave / y / z sets of field
//                 groups that cannot take the row walk: per modelled warp, as sector
//                 intervals of row segments (segment walk) or address by address.
//   rows_kernel   wave, y set, z set and block footprints.  In closed form where a field's layout
//                 allows it (ws_footprint.h; nearly always): counted row by row in registers,
//                 without bitmaps.  Else as whole grid rows: each merged load run of a row is
//                 one sector range set with 64-bit red.or; per-warp store sectors by floor
//                 sums (Sec. 4.4, closed-form counting instead of implicit sets).
//   count_kernel  popcounts of the bitmaps: unique sectors, unique 128 B lines (nibble
//                 OR), y / z overlaps by AND / AND-NOT, reading only the pages the row
//                 walk flagged, one warp per page.  Leaves the bitmaps and flags zeroed for
//                 the next step (only non-zero positions are written).
//   model_kernel  fp64 capacity model and limiters (Sec. 2, 4.5), four lanes per candidate.
//   rank_count_kernel, rank_scatter_kernel   stable counting rank per segment (Sec. 5.8).
// The three persistent kernels take work items from an atomic counter and find each item's
// field group (or field) in an owner table the host lays out with the items.
#include <cuda_runtime.h>

#include <mutex>

#include "ws_footprint.h"
#include "ws_internal.h"
#include "ws_kernels.h"

namespace ws {

#define FULL 0xffffffffu

__device__ __forceinline__ int64_t floordiv_dev(int64_t a, int64_t b) {
  int64_t q = a / b;
  if ((a % b != 0) && ((a < 0) != (b < 0))) q -= 1;
  return q;
}

// Warp-cooperative insertion of one access instruction into a sector bitmap.
// rel: byte address relative to the bitmap origin.  Lanes whose word falls outside
// [0, nwords) are not inserted and are counted in *bad (the host compiler sizes every
// bitmap to hold all addresses, so this never happens unless a descriptor is wrong).
// Returns the number of distinct sectors the active lanes touched (warp-uniform).
__device__ __forceinline__ uint32_t bitmap_insert(uint32_t *__restrict__ bm, int64_t rel, bool act,
                                                  uint32_t lane, int64_t nwords, uint32_t &bad) {
  const bool inside = (uint64_t)(rel >> 10) < (uint64_t)nwords;
  bad += act && !inside;
  act = act && inside;
  uint32_t word = (uint32_t)(rel >> 10);
  uint32_t bit = 1u << ((uint32_t)(rel >> 5) & 31u);
  uint32_t pending = __ballot_sync(FULL, act);
  uint32_t cnt = 0;
  while (pending) {
    uint32_t leader = __ffs(pending) - 1;
    uint32_t lw = __shfl_sync(FULL, word, leader);
    bool mine = act && word == lw;
    uint32_t orv = __reduce_or_sync(FULL, mine ? bit : 0u);
    if (lane == leader) atomicOr(bm + lw, orv);
    cnt += __popc(orv);
    pending &= ~__ballot_sync(FULL, mine);
  }
  return cnt;
}

// Bank-conflict visitor for both half warps of one instruction (Sec. 4.2): unique
// bank words of each half warp, split greedily (ascending) into groups spanning less
// than the pairing distance, each group costs its most used bank.  The result is the
// sum over both halves, valid in every lane.
__device__ int bank_cycles_warp(int64_t addr, bool act, uint32_t lane, int banks, int bank_bytes,
                                int pair_dist) {
  int64_t word = floordiv_dev(addr, bank_bytes);
  int bank = (int)(((word % banks) + banks) % banks);
  uint32_t actm = __ballot_sync(FULL, act);
  uint32_t halfm = lane < 16 ? 0x0000ffffu : 0xffff0000u;
  uint32_t same = __match_any_sync(FULL, (unsigned long long)word) & actm & halfm;
  bool uniq = act && lane == (uint32_t)(__ffs(same) - 1);
  uint32_t todo = __ballot_sync(FULL, uniq);
  int cycles = 0;
  while (todo) {
    bool mine = (todo >> lane) & 1u;
    long long v = mine ? (long long)word : 0x7fffffffffffffffll;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
      long long o = __shfl_xor_sync(FULL, v, off);
      v = o < v ? o : v;
    }
    bool member = mine && (word - (int64_t)v) * (int64_t)bank_bytes < (int64_t)pair_dist;
    uint32_t mm = __ballot_sync(FULL, member);
    uint32_t sameb = __match_any_sync(FULL, bank) & mm & halfm;
    int c = member ? __popc(sameb) : 0;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) c = max(c, __shfl_xor_sync(FULL, c, off));
    if ((lane & 15u) == 0) cycles += c;
    todo &= ~mm;
  }
  return __reduce_add_sync(FULL, (uint32_t)cycles);
}

// The same visitor for power-of-two banks x bank width (their product dividing 1024)
// on 32-bit byte addresses relative to a 1024-byte aligned origin, which have the same
// banks and pairing distances as the absolute ones.
__device__ int bank_cycles_rel32(uint32_t rel, bool act, uint32_t lane, uint32_t bshift, uint32_t bmask,
                                 uint32_t pair_dist) {
  const uint32_t word = rel >> bshift, bank = word & bmask;
  const uint32_t actm = __ballot_sync(FULL, act);
  {
    // every lane active and each half warp's words ascending by 0 or 1 from lane to lane:
    // its unique words are the consecutive words first .. last, which fall in distinct
    // banks round-robin, so a group spanning less than the pairing distance costs
    // ceil(count / banks) cycles
    const uint32_t prev = __shfl_up_sync(FULL, word, 1);
    const bool step = (lane & 15u) == 0u || word - prev <= 1u;
    if (__all_sync(FULL, act && step)) {
      const uint32_t w0 = __shfl_sync(FULL, word, lane & 16u), w1 = __shfl_sync(FULL, word, (lane & 16u) | 15u);
      if (((w1 - w0) << bshift) < pair_dist) {
        const uint32_t nb = bmask + 1u, n = w1 - w0 + 1u;
        const uint32_t c = (n + nb - 1u) / nb;
        return (int)(__shfl_sync(FULL, c, 0) + __shfl_sync(FULL, c, 16));
      }
    }
  }
  const uint32_t halfm = lane < 16 ? 0x0000ffffu : 0xffff0000u;
  const uint32_t same = __match_any_sync(FULL, word) & actm & halfm;
  const bool uniq = act && lane == (uint32_t)(__ffs(same) - 1);
  uint32_t todo = __ballot_sync(FULL, uniq);
  int cycles = 0;
  while (todo) {
    const bool mine = (todo >> lane) & 1u;
    const uint32_t v = __reduce_min_sync(halfm, mine ? word : 0xffffffffu);
    const bool member = mine && ((word - v) << bshift) < pair_dist;
    const uint32_t mm = __ballot_sync(FULL, member);
    const uint32_t sameb = __match_any_sync(FULL, bank) & mm & halfm;
    const uint32_t c = __reduce_max_sync(halfm, member ? (uint32_t)__popc(sameb) : 0u);
    if ((lane & 15u) == 0) cycles += (int)c;
    todo &= ~mm;
  }
  return (int)__reduce_add_sync(FULL, (uint32_t)cycles);
}


__device__ __forceinline__ uint32_t fdiv(uint32_t n, const FastDiv &f) {
  return (__umulhi(n, f.m) + n) >> f.s;
}

// Run-head insertion of one access instruction (32-bit addresses).  Consecutive
// active lanes whose sectors step by 0 or 1 inside one bitmap word form a run; the
// first lane of each run sets the run's bit range [head sector, tail sector] with one
// red.or.  Every sector between head and tail is touched by some lane of the run, so
// the bitmap receives exactly the union of the lanes' sectors whatever the layout
// (a scattered layout just makes more, shorter runs).  r: byte address relative to
// the bitmap origin; lanes with r >= limit are skipped and counted in `bad`.
// With want_count the number of distinct sectors of the instruction is returned
// (warp-uniform): the sum of run lengths when runs increase strictly across the
// warp, else the exact per-word count.
__device__ __forceinline__ uint32_t runs_insert(uint32_t *__restrict__ bm, uint32_t r, bool act, uint32_t limit,
                                                uint32_t lane, uint32_t &bad, bool want_count) {
  const bool inside = r < limit;
  bad += act && !inside;
  act = act && inside;
  const uint32_t sec = r >> 5;
  const uint32_t prev = __shfl_up_sync(FULL, sec, 1);
  const uint32_t actm = __ballot_sync(FULL, act);
  const uint32_t below = actm & ((1u << lane) - 1u);
  const bool prev_act = ((actm << 1) >> lane) & 1u;
  const bool cont = prev_act && (sec - prev) <= 1u && ((sec ^ prev) >> 5) == 0u;
  const bool head = act && !cont;
  const uint32_t heads = __ballot_sync(FULL, head);
  const uint32_t ends = actm & ~((actm & ~heads) >> 1);
  const uint32_t t = __ffs(ends & (0xffffffffu << lane)) - 1u;
  const uint32_t tail = __shfl_sync(FULL, sec, t);
  if (head) {
    const uint32_t hb = sec & 31u, tb = tail & 31u;
    atomicOr(bm + (sec >> 5), (0xffffffffu >> (31u - tb)) & (0xffffffffu << hb));
  }
  if (!want_count) return 0;
  const uint32_t pl = below ? 31u - __clz(below) : 0u;
  const uint32_t psec = __shfl_sync(FULL, sec, pl);
  if (__all_sync(FULL, !head || below == 0u || sec > psec))
    return __reduce_add_sync(FULL, head ? tail - sec + 1u : 0u);
  uint32_t cnt = 0;   // overlapping runs: count distinct sectors word by word
  const uint32_t word = sec >> 5, bit = 1u << (sec & 31u);
  uint32_t pending = actm;
  while (pending) {
    const uint32_t lw = __shfl_sync(FULL, word, __ffs(pending) - 1);
    const bool mine = act && word == lw;
    cnt += __popc(__reduce_or_sync(FULL, mine ? bit : 0u));
    pending &= ~__ballot_sync(FULL, mine);
  }
  return cnt;
}

// Lane-per-access walk of the wave / y / z loads.  With P = the smallest power of two
// >= the field's folded loads (at most 32), the warp's lanes form 32/P groups of P
// lanes; lane (g, a) evaluates access a for the P threads g*P .. g*P+P-1 of the
// modelled warp, merging the sector bits of one bitmap word in a register and
// flushing it with one red.or when the word changes.  tbase: the slice's relative
// thread addresses; slice: which of them are valid.
template <int P, bool CHECK>
__device__ __forceinline__ void lpa_walk(const uint32_t *__restrict__ tbase, uint32_t slice, uint32_t b32,
                                         uint32_t limit, uint32_t *__restrict__ bm, uint32_t &cw, uint32_t &cb,
                                         uint32_t &bad) {
  auto step = [&](uint32_t tb) {
    const uint32_t r = tb + b32;
    if (CHECK && r >= limit) {
      ++bad;
      return;
    }
    const uint32_t w = r >> 10;
    const bool flush = w != cw;
    if (flush && cb) atomicOr(bm + cw, cb);
    cb = (flush ? 0u : cb) | __funnelshift_l(0u, 1u, r >> 5);
    cw = w;
  };
  constexpr uint32_t full = P == 32 ? 0xffffffffu : ((1u << P) - 1u);
  if (P >= 4) {
    const uint4 *t4 = reinterpret_cast<const uint4 *>(tbase);
    if (slice == full) {
#pragma unroll
      for (int q = 0; q < P / 4; ++q) {
        const uint4 v = t4[q];
        step(v.x);
        step(v.y);
        step(v.z);
        step(v.w);
      }
    } else {
#pragma unroll
      for (int q = 0; q < P / 4; ++q) {
        const uint4 v = t4[q];
        const uint32_t m = slice >> (4 * q);
        if (m & 1u) step(v.x);
        if (m & 2u) step(v.y);
        if (m & 4u) step(v.z);
        if (m & 8u) step(v.w);
      }
    }
  } else {
#pragma unroll
    for (int t = 0; t < P; ++t)
      if ((slice >> t) & 1u) step(tbase[t]);
  }
}

// The same walk over all 32 threads of a modelled warp, also counting the distinct
// sectors of the lane's access instruction: the number of sector changes along the
// walk, exact when the lane's sectors never decrease (`mono`).
__device__ __forceinline__ void lpa_walk_count(const uint32_t *__restrict__ tbase, uint32_t vmask, uint32_t b32,
                                               uint32_t *__restrict__ bm, uint32_t &cw, uint32_t &cb,
                                               uint32_t &nsec, bool &mono) {
  uint32_t last = 0xffffffffu;
  auto step = [&](uint32_t tb) {
    const uint32_t r = tb + b32;
    const uint32_t sec = r >> 5;
    nsec += sec != last;
    mono = mono && (last == 0xffffffffu || sec >= last);
    last = sec;
    const uint32_t w = r >> 10;
    const bool flush = w != cw;
    if (flush && cb) atomicOr(bm + cw, cb);
    cb = (flush ? 0u : cb) | __funnelshift_l(0u, 1u, sec);
    cw = w;
  };
  const uint4 *t4 = reinterpret_cast<const uint4 *>(tbase);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint4 v = t4[q];
    const uint32_t m = vmask >> (4 * q);
    if (m & 1u) step(v.x);
    if (m & 2u) step(v.y);
    if (m & 4u) step(v.z);
    if (m & 8u) step(v.w);
  }
}

// Exact distinct sectors of one instruction whose lanes hold relative addresses r.
__device__ __forceinline__ uint32_t warp_distinct_sectors(uint32_t r, bool act) {
  {
    // every lane active and sectors not decreasing from lane to lane: equal sectors are
    // neighbours, so the distinct ones are the lanes that start a new sector
    const uint32_t sec = r >> 5, prev = __shfl_up_sync(FULL, sec, 1);
    const uint32_t lane = threadIdx.x & 31u;
    if (__all_sync(FULL, act && (lane == 0u || sec >= prev)))
      return (uint32_t)__popc(__ballot_sync(FULL, lane == 0u || sec != prev));
  }
  const uint32_t word = r >> 10, bit = 1u << ((r >> 5) & 31u);
  uint32_t pending = __ballot_sync(FULL, act), cnt = 0;
  while (pending) {
    const uint32_t lw = __shfl_sync(FULL, word, __ffs(pending) - 1);
    const bool mine = act && word == lw;
    cnt += __popc(__reduce_or_sync(FULL, mine ? bit : 0u));
    pending &= ~__ballot_sync(FULL, mine);
  }
  return cnt;
}


// A uniform field group walks its loads (stores) lane per access when it has at least
// this many; with fewer, most lanes of such a walk would idle.
constexpr int kCombinedWalkMin = 8;

// Sets sectors [s0, s1] of a bitmap viewed as 64-bit units (one red.or per unit).
__device__ __forceinline__ void set_sector_range(unsigned long long *__restrict__ bm, uint32_t s0, uint32_t s1) {
  const uint32_t u0 = s0 >> 6, u1 = s1 >> 6;
  const unsigned long long m0 = ~0ull << (s0 & 63u);
  const unsigned long long m1 = ~0ull >> (63u - (s1 & 63u));
  if (u0 == u1) {
    atomicOr(bm + u0, m0 & m1);
    return;
  }
  atomicOr(bm + u0, m0);
  for (uint32_t u = u0 + 1; u < u1; ++u) atomicOr(bm + u, ~0ull);
  atomicOr(bm + u1, m1);
}

// Adds sectors [s0, s1] to a lane's pending 64-bit unit (cu, cb), flushing it with one
// red.or when the range leaves that unit; units the range covers entirely are written
// directly.  The caller flushes the last pending unit.  Returns the red.or issued.
__device__ __forceinline__ uint32_t put_range(unsigned long long *__restrict__ bm, uint32_t &cu,
                                              unsigned long long &cb, uint32_t s0, uint32_t s1) {
  const uint32_t u0 = s0 >> 6, u1 = s1 >> 6;
  const unsigned long long m0 = ~0ull << (s0 & 63u);
  const unsigned long long m1 = ~0ull >> (63u - (s1 & 63u));
  uint32_t n = 0;
  if (u0 == u1) {
    if (u0 == cu) {
      cb |= m0 & m1;
      return 0;
    }
    if (cb) {
      atomicOr(bm + cu, cb);
      n = 1;
    }
    cu = u0;
    cb = m0 & m1;
    return n;
  }
  if (u0 == cu) {
    atomicOr(bm + u0, cb | m0);
  } else {
    if (cb) {
      atomicOr(bm + cu, cb);
      n = 1;
    }
    atomicOr(bm + u0, m0);
  }
  for (uint32_t u = u0 + 1; u < u1; ++u) atomicOr(bm + u, ~0ull);
  cu = u1;
  cb = m1;
  return n + (u1 - u0);
}

// Flags the pages [p0, p1] of one bitmap as written.  The flag array starts zeroed and only
// ever receives ones until the counting kernel clears it, so plain byte stores suffice (the
// same value from any number of writers; reading a flag first to skip the store was slower).
__device__ __forceinline__ void flag_pages(uint8_t *__restrict__ fl, uint32_t p0, uint32_t p1) {
  for (uint32_t p = p0; p <= p1; ++p) fl[p] = 1;
}

// Byte range [lo, hi] (relative to the bitmap origin) of one row segment of a
// modelled warp under byte offset bo and extent ext.  Thread addresses are kept as
// their low 32 bits; `mn` is the warp's smallest full thread address, and every valid
// thread lies less than 2^32 bytes above it (the bitmap of a non-wide field spans
// less than that), so address - mn is exact in 32 bits.  Returns false when the range
// leaves [0, limit).
__device__ __forceinline__ bool segment_range(uint32_t th, uint32_t tt, int64_t mn, int64_t bo, uint32_t ext,
                                              uint32_t limit, uint32_t &lo, uint32_t &hi) {
  const uint32_t m32 = (uint32_t)mn;
  const uint32_t dh = th - m32, dt = tt - m32;
  const int64_t vlo = mn + (int64_t)min(dh, dt) + bo;
  const int64_t vhi = mn + (int64_t)max(dh, dt) + bo + (int64_t)ext;
  if (vlo < 0 || vhi >= (int64_t)limit) return false;
  lo = (uint32_t)vlo;
  hi = (uint32_t)vhi;
  return true;
}

// Sum_{i<n} floor((P*i + c) / 32) where every term's argument is >= 0 (P of any sign).
// The multiple-of-32 part of P and c comes out in closed form.  What is left, a, b < 32, is
// (a*i + b less its remainder) / 32 term by term; the remainders (a*i + b) mod 32 repeat after
// 32 / g terms, g the lowest bit of a, running through all values that agree with b modulo g,
// so only the terms of a last partial period (fewer than 8 for 4-byte elements, none at all
// for fp64 rows of four or more threads) are added one by one.
__device__ __forceinline__ int64_t sum_floor32(int64_t n, int64_t P, int64_t c) {
  if (n <= 0) return 0;
  if (P < 0) {
    c += P * (n - 1);
    P = -P;
  }
  int64_t res = (P >> 5) * (n * (n - 1) / 2) + (c >> 5) * n;
  const uint32_t a = (uint32_t)(P & 31), b = (uint32_t)(c & 31);
  if (a != 0) {
    const uint32_t g = a & (0u - a), lp = 5u - (31u - __clz(g)), per = 1u << lp;
    const uint32_t whole = per * (b & (g - 1u)) + g * (per * (per - 1u) / 2u);   // the remainders of one period
    uint32_t part = 0, v = b;
    for (uint32_t i = 0; i < ((uint32_t)n & (per - 1u)); ++i, v += a) part += v & 31u;
    res += ((int64_t)a * (n * (n - 1) / 2) + (int64_t)b * n - (n >> lp) * (int64_t)whole - (int64_t)part) >> 5;
  }
  return res;
}

// Distinct sectors of one store instruction summed over the warps of a row walk's grid
// row: the row's threads are split into warp segments (consecutive threads of one warp
// within one block; a warp's other segments lie in other rows and share no sector with
// this one), each counted as floor(last / 32) - floor(first / 32) + 1 bytes-to-sectors.
// Segments repeat from block to block with the address step B0 * step, so each segment
// position contributes two floor sums over the row's whole blocks; the block cut by N0
// is counted directly.  A0 + step * x is the relative address of point x of the row.
__device__ __forceinline__ int64_t row_store_sectors(int64_t A0, int64_t step, int32_t B0, int32_t N0, int32_t full_end,
                                                     uint32_t t, uint32_t bxa, uint32_t bxb) {
  auto direct = [&](int64_t x0, int64_t x1) -> int64_t {
    const int64_t p = A0 + step * x0, q = A0 + step * x1;
    return (max(p, q) >> 5) - (min(p, q) >> 5) + 1;
  };
  int64_t cnt = 0;
  const int64_t xa = (int64_t)bxa * B0, xb = min((int64_t)bxb * B0, (int64_t)N0);
  if ((B0 & 31) == 0) {
    // warps tile the row in aligned runs of 32 threads
    const int64_t nx = xb - xa, nq = nx >> 5;
    if (nq > 0) {
      const int64_t p0 = A0 + step * xa, p1 = A0 + step * (xa + 31);
      cnt += sum_floor32(nq, 32 * step, max(p0, p1)) - sum_floor32(nq, 32 * step, min(p0, p1)) + nq;
    }
    if (nx & 31) cnt += direct(xa + (nq << 5), xb - 1);
    return cnt;
  }
  const int32_t f1 = (int32_t)((32 - (((int64_t)t * B0) & 31)) & 31);
  const uint32_t bfe = min(bxb, (uint32_t)full_end);
  const int64_t nfull = bfe > bxa ? (int64_t)(bfe - bxa) : 0;
  const int64_t P = (int64_t)B0 * step;
  for (int32_t ta = 0; ta < B0;) {
    const int32_t tb = (ta == 0 && f1 > 0) ? min(f1, B0) : min(ta + 32, B0);
    if (nfull > 0) {
      const int64_t p0 = A0 + step * (xa + ta), p1 = A0 + step * (xa + tb - 1);
      cnt += sum_floor32(nfull, P, max(p0, p1)) - sum_floor32(nfull, P, min(p0, p1)) + nfull;
    }
    if (bxb > bfe) {
      const int64_t xs = (int64_t)full_end * B0 + ta, xe = min((int64_t)full_end * B0 + tb, (int64_t)N0);
      if (xe > xs) cnt += direct(xs, xe - 1);
    }
    ta = tb;
  }
  return cnt;
}

// The same out of line, for the closed form's kernel, whose code has to stay short.
__device__ __noinline__ int64_t row_store_sectors_call(int64_t A0, int64_t step, int32_t B0, int32_t N0, int32_t full_end,
                                                       uint32_t t, uint32_t bxa, uint32_t bxb) {
  return row_store_sectors(A0, step, B0, N0, full_end, t, bxa, bxb);
}

// Accesses of a group whose block is only counted (the row walk or the closed form makes its
// footprints), taken together by what an instruction's counts depend on: its lanes' addresses
// modulo a sector and the bank period, a multiple `period` of both, which for accesses of one
// layout is the place of any one address in the period, and the folded points that need it.
// The 25-point star has 9 such codes among its 26 accesses, the 84 accesses of a lattice Boltzmann
// step a handful.  The enumeration is bound by the latency of the warps' instruction chains and of
// a group's staging; its time (GB300), accesses one by one -> codes: 755 25-point candidates
// 61 -> 41 us, 755 lattice Boltzmann 173 -> 58, 4,000 mixed 517 -> 245, 40 served 100 -> 31.
// Groups of at most kFewPairs (class warp, access) pairs keep to the list: the codes' three barriers
// cost more than they save (one 7-point candidate 12.3 us with the list, 14.7 with codes).
constexpr int kFewPairs = 64;
struct AccessCodes {
  int n;              // codes; 0: this group's accesses are taken one by one
  uint32_t period;
  int64_t ref;        // byte offset of the group's first access
};

// Shared-memory images of one field group, staged by the enumeration and row kernels.
struct StageSmem {
  DCfg *c;
  DGroup *g;
  DField *fk;
  int32_t *loff, *soff, *ioff;   // first load / store / merged interval of field k
  uint8_t *af;                   // field of each staged access
  int64_t *boff;                 // byte offset of each staged access
  uint32_t *b32;                 // uniform groups: 32-bit offset from the shared thread address (may be null)
  uint8_t *kmin;                 // first folded point that needs each access
  int32_t (*gad)[17];            // issued accesses per thread by valid folded points, [0] levels 0-1, [1] 2-3
  int32_t *gwi;                  // access instructions, [0] levels 0-1, [1] 2-3
  int64_t *ibo;                  // merged load runs: offset relative to the field's bitmap origin
  uint32_t *iext;                //   extent
  uint8_t *iaf;                  //   field
  // row walk only (else null): the runs without a covering run of all fields first, then
  // those covered from another z row, then those covered within their z row; idst[j][k] =
  // first staged slot of field k's runs of kind j; cov = {runs without a covering run,
  // largest |ddy|, largest |ddz| of the covered runs, runs of the first two kinds, largest
  // |ddy| of the last kind}
  int32_t (*idst)[kMaxGroupFields];
  int32_t *cov;
  AccessCodes *codes;   // enumeration only (else null)
};

// Makes the codes of the staged group (b32: their counts, loads low and stores high; boff: the list
// of those that occur) or none; ends with a barrier.
__device__ __forceinline__ void stage_codes(const EnumArgs &a, const StageSmem &m) {
  const DGroup &G = *m.g;
  // one code per place in the period, and per first folded point where the block has threads with
  // fewer points than the fold; as many as the list of 32-bit offsets has entries
  const uint32_t period = (uint32_t)max(32, a.banks * a.bank_bytes);
  const DCfg &c = *m.c;
  const uint32_t bt = fdiv((uint32_t)c.rep, c.fd_gx), bz = fdiv(bt, c.fd_gy), by = bt - bz * (uint32_t)c.g[1];
  const bool whole = c.fold_axis == 0 || (c.fold_axis == 1 ? ((int)by + 1) * c.B[1] * c.fold <= c.N[1]
                                                           : ((int)bz + 1) * c.B[2] * c.fold <= c.N[2]);
  const uint32_t size = period * (whole ? 1u : (uint32_t)c.fold);
  if (size > (uint32_t)kMaxFoldedAccesses || m.fk[0].words[0] >= ((int64_t)1 << 22) - 4) {
    if (threadIdx.x == 0) m.codes->n = 0;
    __syncthreads();
    return;
  }
  for (uint32_t i = threadIdx.x; i < size; i += blockDim.x) m.b32[i] = 0u;
  if (threadIdx.x == 0) {
    m.codes->period = period;
    m.codes->ref = a.acc[m.fk[0].acc_begin].boff;
  }
  __syncthreads();
  for (int k = 0; k < G.f_count; ++k) {
    const DField &F = m.fk[k];
    for (int i = threadIdx.x; i < F.n_load + F.n_store; i += blockDim.x) {
      const DAcc d = a.acc[F.acc_begin + i];
      const uint32_t at = ((uint32_t)F.base + (uint32_t)d.boff) & (period - 1u);
      atomicAdd(m.b32 + at + (whole ? 0u : period * (uint32_t)d.kmin), i < F.n_load ? 1u : 0x10000u);
    }
  }
  __syncthreads();
  // in ascending order: the CTAs that share the group's items must number the codes alike
  uint2 *const list = reinterpret_cast<uint2 *>(m.boff);
  if (threadIdx.x < 32) {
    int have = 0;
    for (uint32_t i0 = 0; i0 < size; i0 += 32) {
      const uint32_t n = m.b32[i0 + threadIdx.x], some = __ballot_sync(FULL, n != 0u);
      if (n) list[have + __popc(some & ((1u << threadIdx.x) - 1u))] = make_uint2(i0 + threadIdx.x, n);
      have += __popc(some);
    }
    if (threadIdx.x == 0) m.codes->n = have;
  }
  __syncthreads();
}

// Stages group gi (and its candidate when it differs from cur_cfg); ends with a barrier.
// Returns true when the candidate changed.
__device__ bool stage_group(const EnumArgs &a, int gi, int cur_cfg, const StageSmem &m) {
  if (threadIdx.x == 0) *m.g = a.grp[gi];
  __syncthreads();
  const DGroup &G = *m.g;
  {
    // the group's fields, copied as 8-byte words by all threads
    static_assert(sizeof(DField) % 8 == 0, "DField is copied as 8-byte words");
    const int nw = G.f_count * (int)(sizeof(DField) / 8);
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(a.fld + G.f_begin);
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(m.fk);
    for (int i = threadIdx.x; i < nw; i += blockDim.x) dst[i] = src[i];
  }
  const bool new_cfg = G.cfg != cur_cfg;
  if (new_cfg && threadIdx.x == 0) *m.c = a.cfg[G.cfg];
  __syncthreads();
  if (threadIdx.x == 0) {
    // all loads of the group first (field by field), then all stores
    int o = 0;
    for (int k = 0; k < G.f_count; ++k) {
      m.loff[k] = o;
      o += m.fk[k].n_load;
    }
    m.loff[G.f_count] = o;
    for (int k = 0; k < G.f_count; ++k) {
      m.soff[k] = o;
      o += m.fk[k].n_store;
    }
    m.soff[G.f_count] = o;
    o = 0;
    for (int k = 0; k < G.f_count; ++k) {
      m.ioff[k] = o;
      o += G.iv ? m.fk[k].n_iv : 0;
    }
    m.ioff[G.f_count] = o;
    if (m.cov) {
      int u = 0, dy = 0, dz = 0, dyy = 0;
      for (int k = 0; k < G.f_count; ++k)
        if (G.iv) {
          m.idst[0][k] = u;
          u += m.fk[k].n_iv_unc;
          if (m.fk[k].n_iv_unc < m.fk[k].n_iv) {
            dy = max(dy, (int)m.fk[k].cov_dy);
            dz = max(dz, (int)m.fk[k].cov_dz);
            dyy = max(dyy, (int)m.fk[k].cov_dy_y);
          }
        }
      int c = u;
      for (int k = 0; k < G.f_count; ++k)
        if (G.iv) {
          m.idst[1][k] = c;
          c += m.fk[k].n_iv_zc;
        }
      const int uz = c;
      for (int k = 0; k < G.f_count; ++k)
        if (G.iv) {
          m.idst[2][k] = c;
          c += m.fk[k].n_iv - m.fk[k].n_iv_unc - m.fk[k].n_iv_zc;
        }
      m.cov[0] = u;
      m.cov[1] = dy;
      m.cov[2] = dz;
      m.cov[3] = uz;
      m.cov[4] = dyy;
    }
  }
  for (int t = threadIdx.x; t < 34; t += blockDim.x) {
    // issued accesses per thread (by valid folded points) and access instructions,
    // summed over the group's fields: [0] block and wave (loads and stores), [1] y / z
    const int lv = t / 17, kv = t % 17;
    int ad = 0, wi = 0;
    for (int k = 0; k < G.f_count; ++k) {
      ad += m.fk[k].cnt_load[kv] + (lv == 0 ? m.fk[k].cnt_store[kv] : 0);
      wi += m.fk[k].n_load + (lv == 0 ? m.fk[k].n_store : 0);
    }
    m.gad[lv][kv] = ad;
    if (kv == 0) m.gwi[lv] = wi;
  }
  __syncthreads();
  if (m.codes) {
    if (G.rows && a.bank_shift >= 0 && G.n_rep * G.acc_count > kFewPairs) {
      stage_codes(a, m);
      if (m.codes->n) return new_cfg;
    } else if (threadIdx.x == 0) {
      m.codes->n = 0;
    }
  }
  // merged load runs, offsets relative to each field's bitmap origin (the enumeration kernel
  // uses them only for groups without the row walk)
  const int n_runs = (m.cov != nullptr || !G.rows) ? m.ioff[G.f_count] : 0;
  for (int j = threadIdx.x; j < n_runs; j += blockDim.x) {
    int k = 0;
    while (m.ioff[k + 1] <= j) ++k;
    const DField &F = m.fk[k];
    const int jj = j - m.ioff[k];
    const DIv v = a.iv[F.iv_begin + jj];
    const int d = !m.cov                          ? j
                  : jj < F.n_iv_unc               ? m.idst[0][k] + jj
                  : jj < F.n_iv_unc + F.n_iv_zc   ? m.idst[1][k] + (jj - F.n_iv_unc)
                                                  : m.idst[2][k] + (jj - F.n_iv_unc - F.n_iv_zc);
    m.ibo[d] = v.boff + F.base - 32 * F.lo[1];
    m.iext[d] = v.ext;
    m.iaf[d] = (uint8_t)k;
  }
  // raw folded accesses; uniform groups fold each field's constant into the 32-bit
  // offsets, so that address = shared thread address + offset for every field
  for (int j = threadIdx.x; j < m.soff[G.f_count]; j += blockDim.x) {
    const bool st = j >= m.loff[G.f_count];
    int k = 0;
    if (!st) {
      while (m.loff[k + 1] <= j) ++k;
    } else {
      while (m.soff[k + 1] <= j) ++k;
    }
    const DField &F = m.fk[k];
    const int i = st ? F.n_load + (j - m.soff[k]) : j - m.loff[k];
    const DAcc d = a.acc[F.acc_begin + i];
    m.boff[j] = d.boff;
    if (m.b32) m.b32[j] = (uint32_t)d.boff + (G.uniform ? (uint32_t)(F.base - 32 * F.lo[1]) : 0u);
    m.kmin[j] = (uint8_t)d.kmin;
    m.af[j] = (uint8_t)k;
  }
  __syncthreads();
  return new_cfg;
}

struct BlockCounts {
  uint32_t lb, req, st, bank, addr, wi;
};

// Item kk of a group whose accesses come as codes: an instruction is a code with its loads and
// stores; the items share the (class warp, code) pairs evenly, the warps an item's.  tcs: the
// block's thread coordinates.
__device__ __forceinline__ BlockCounts block_codes(const EnumArgs &a, const StageSmem &m, const uint32_t *tcs, int64_t kk) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const DGroup &G = *m.g;
  const DCfg &c = *m.c;
  BlockCounts o = {0, 0, 0, 0, 0, 0};
  const uint2 *const codes = reinterpret_cast<const uint2 *>(m.boff);
  const uint32_t nc = (uint32_t)m.codes->n, np = (uint32_t)G.n_rep * nc, n0 = (uint32_t)G.n0_items;
  const uint32_t p0 = (uint32_t)((uint64_t)np * (uint32_t)kk / n0), p1 = (uint32_t)((uint64_t)np * (uint32_t)(kk + 1) / n0);
  const uint32_t per = (p1 - p0 + nwarps - 1) / nwarps;
  const uint32_t q0 = min(p0 + warp * per, p1), q1 = min(q0 + per, p1);
  const DField &F = m.fk[0];
  const uint32_t period = m.codes->period, pshift = 31u - __clz(period);
  const uint32_t from = ((uint32_t)F.base + (uint32_t)m.codes->ref) & (period - 1u);
  const uint32_t bt = fdiv((uint32_t)c.rep, c.fd_gx), bx = (uint32_t)c.rep - bt * (uint32_t)c.g[0];
  const uint32_t bz = fdiv(bt, c.fd_gy), by = bt - bz * (uint32_t)c.g[1];
  const int32_t faxis = c.fold_axis, fold = c.fold;
  uint32_t r = q0 / nc, j = q0 - r * nc, mult = 0, at = 0;
  int kv = 0;
  bool fresh = true;
  for (uint32_t pp = q0; pp < q1; ++pp) {
    if (fresh) {
      // a class warp's threads: the place of each one's first address
      fresh = false;
      mult = G.rep_mult[r];
      const uint32_t tid = (uint32_t)G.rep_warp[r] * 32u + lane;
      const uint32_t tc = tid < (uint32_t)c.T ? tcs[tid] : 0u;
      const int32_t x = (int32_t)bx * c.B[0] + (int32_t)(tc & 1023u);
      int32_t y = (int32_t)by * c.B[1] + (int32_t)((tc >> 10) & 1023u);
      int32_t z = (int32_t)bz * c.B[2] + (int32_t)(tc >> 20);
      if (faxis == 1) y *= fold;
      if (faxis == 2) z *= fold;
      kv = 0;
      if (tid < (uint32_t)c.T && x < c.N[0] && y < c.N[1] && z < c.N[2])
        kv = faxis == 1 ? min(fold, c.N[1] - y) : faxis == 2 ? min(fold, c.N[2] - z) : 1;
      if (j == 0u) {
        if (G.first_of_cfg) o.lb += mult * __reduce_add_sync(FULL, (uint32_t)kv);
        o.addr += mult * __reduce_add_sync(FULL, (uint32_t)m.gad[0][kv]);
        o.wi += mult * (uint32_t)m.gwi[0];
      }
      const int64_t lin = F.stride[0] * x + F.stride[1] * y + F.stride[2] * z;
      const int64_t r0 = F.base + (int64_t)F.esize * lin - 32 * F.lo[0] + m.codes->ref;
      if (r0 < 0 || r0 >= F.words[0] << 10) kv = 0;
      at = (uint32_t)r0 - from + period;   // (a period is added, so that none falls below the origin)
    }
    const uint2 cd = codes[j];
    const uint32_t rel = at + (cd.x & (period - 1u)), nl = cd.y & 0xffffu, ns = cd.y >> 16;
    const bool act = (int)(cd.x >> pshift) < kv;
    const uint32_t nsec = mult * warp_distinct_sectors(rel, act);
    o.req += nsec * nl;
    o.st += nsec * ns;
    o.bank += mult * (nl + ns) * (uint32_t)bank_cycles_rel32(rel, act, lane, (uint32_t)a.bank_shift,
                                                               (uint32_t)(a.banks - 1), (uint32_t)a.pair_dist);
    if (++j == nc) {
      j = 0;
      ++r;
      fresh = true;
    }
  }
  return o;
}

__global__ void __launch_bounds__(512, 2) enum_kernel(EnumArgs a) {
  __shared__ DCfg s_c;
  __shared__ DGroup s_g;
  __shared__ DField s_fk[kMaxGroupFields];
  __shared__ int32_t s_loff[kMaxGroupFields + 1];   // first load of field k in the staged lists
  __shared__ int32_t s_soff[kMaxGroupFields + 1];   // first store of field k (after all loads)
  __shared__ uint8_t s_af[kMaxFoldedAccesses];      // field of each staged access
  __shared__ int64_t s_boff[kMaxFoldedAccesses];
  __shared__ uint32_t s_b32[kMaxFoldedAccesses];
  __shared__ uint8_t s_kmin[kMaxFoldedAccesses];
  __shared__ uint32_t s_tc[1024];
  __shared__ __align__(16) uint32_t s_tbase[16][32];   // per warp: relative address of each thread's first point
  __shared__ uint8_t s_tkv[16][32];                    // per warp: valid folded points of each thread
  __shared__ uint32_t s_seg[16][32];                   // per warp: row segments (head lane, tail lane, kv)
  __shared__ int32_t s_ioff[kMaxGroupFields + 1];      // first merged interval of field k
  __shared__ uint16_t s_lg[2][32];                     // interval walk lanes: entry | segment phase << 8
  __shared__ uint32_t s_lgG[2];                        //   lanes per entry ([0] merged runs, [1] raw loads)
  __shared__ int32_t s_gad[2][17];                     // group's issued accesses per thread with kv points
  __shared__ int32_t s_gwi[2];                         // group's access instructions ([0] levels 0-1, [1] 2-3)
  __shared__ long long s_item;
  __shared__ AccessCodes s_codes;
  // merged load intervals of an interval-walk group (dynamic): offset, extent, field
  extern __shared__ __align__(16) unsigned char s_dyn[];
  const int iv_cap16 = (a.iv_cap + 15) & ~15;
  int64_t *const s_ibo = reinterpret_cast<int64_t *>(s_dyn);
  uint32_t *const s_iext = reinterpret_cast<uint32_t *>(s_dyn + 8 * iv_cap16);
  uint8_t *const s_iaf = s_dyn + 12 * iv_cap16;
  const StageSmem sm{&s_c, &s_g, s_fk, s_loff, s_soff, s_ioff, s_af, s_boff, s_b32, s_kmin, s_gad, s_gwi,
                     s_ibo, s_iext, s_iaf, nullptr, nullptr, &s_codes};

  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = threadIdx.x >> 5;
  const uint32_t nwarps = blockDim.x >> 5;
  int cur_g = -1, cur_cfg = -1;

  for (;;) {
    if (threadIdx.x == 0) s_item = a.item_lo + (long long)atomicAdd(a.grab, 1ull);
    __syncthreads();
    const int64_t item = s_item;
    if (item >= a.item_hi) break;
    const int gi = a.own_enum[item];
    if (gi != cur_g) {
      // stage the group, then the interval walk's lane layout and the thread table
      const bool new_cfg = stage_group(a, gi, cur_cfg, sm);
      // with M < 32 entries, G = 32 / M lanes share an entry and take every G-th row segment
      if (threadIdx.x < 64) {
        const int pi = threadIdx.x >> 5, l = threadIdx.x & 31;
        const int M = pi == 0 ? s_ioff[s_g.f_count] : s_loff[s_g.f_count];
        const int G = (M > 0 && M < 32) ? 32 / M : 1;
        const int e = G > 1 ? l % M : l, g = G > 1 ? l / M : 0;
        s_lg[pi][l] = (uint16_t)(e | (g << 8));
        if (l == 0) s_lgG[pi] = (uint32_t)G;
      }
      if (new_cfg) {
        for (int t = threadIdx.x; t < s_c.T; t += blockDim.x) {
          const uint32_t tx = t % s_c.B[0], ty = (t / s_c.B[0]) % s_c.B[1], tz = t / (s_c.B[0] * s_c.B[1]);
          s_tc[t] = tx | (ty << 10) | (tz << 20);
        }
      }
      __syncthreads();
      cur_g = gi;
      cur_cfg = s_g.cfg;
    }
    // the first n0_items items of a group cover the representative block as chunks of
    // (modelled warp, access instruction) pairs; the others chunks of the remaining
    // modelled warps (groups without the row walk)
    const int64_t kk = item - s_g.item_begin;
    const bool blk = kk < s_g.n0_items;
    const uint32_t mw0 = blk ? 0u : (uint32_t)(s_g.mw_block + (kk - s_g.n0_items) * (int64_t)a.chunk);
    const uint32_t mw1 = blk ? 0u : (uint32_t)min(s_g.mw_block + (kk - s_g.n0_items + 1) * (int64_t)a.chunk,
                                                   s_g.mw_end);
    uint32_t acc_lb = 0, acc_lw = 0, acc_req = 0, acc_st = 0, acc_bank = 0, acc_sreq = 0, acc_addr = 0, acc_wi = 0;
    uint32_t bad = 0;

    if (blk && s_codes.n) {
      const BlockCounts o = block_codes(a, sm, s_tc, kk);
      acc_lb = o.lb;
      acc_req = o.req;
      acc_st = o.st;
      acc_bank = o.bank;
      acc_addr = o.addr;
      acc_wi = o.wi;
    } else if (blk) {
      // ---- representative block (Sec. 4.2, 4.3): every (warp, instruction) exactly --
      // distinct sectors per instruction (L1 requests / write-through stores), the block
      // footprint bitmaps, and half-warp bank cycles.  Each warp takes a contiguous run of
      // the item's (class warp, instruction) pairs, instruction fastest, and keeps the class
      // warp's thread coordinates and the field's address base while they stay the same.
      const uint32_t LS = (uint32_t)s_soff[s_g.f_count], L = (uint32_t)s_loff[s_g.f_count];
      const uint32_t np = (uint32_t)s_g.n_rep * LS;
      const uint32_t p0 = (uint32_t)kk * (uint32_t)a.block_pairs, p1 = min(p0 + (uint32_t)a.block_pairs, np);
      const uint32_t per = (p1 - p0 + nwarps - 1) / nwarps;
      const uint32_t q0 = min(p0 + warp * per, p1), q1 = min(q0 + per, p1);
      const bool fast_banks = a.bank_shift >= 0;
      // with the row walk the block bitmaps are built there: count only, one warp per class
      const bool count_only = s_g.rows;
      const uint32_t b = (uint32_t)s_c.rep;
      const uint32_t bt = fdiv(b, s_c.fd_gx);
      const uint32_t bx = b - bt * (uint32_t)s_c.g[0];
      const uint32_t bz = fdiv(bt, s_c.fd_gy);
      const uint32_t by = bt - bz * (uint32_t)s_c.g[1];
      const int32_t faxis = s_c.fold_axis, fold = s_c.fold;
      uint32_t r = q0 / max(LS, 1u), j = q0 - r * LS;
      int cur_r = -1, cur_k = -1;
      uint32_t mult = 0;
      int32_t x = 0, y = 0, z = 0;
      int kv = 0;
      bool valid = false;
      int64_t rbase = 0, rlim = 0;
      for (uint32_t pp = q0; pp < q1; ++pp) {
        if ((int)r != cur_r) {
          cur_r = (int)r;
          cur_k = -1;
          const uint32_t mw = s_g.rep_warp[r];
          mult = s_g.rep_mult[r];
          const uint32_t tid = mw * 32u + lane;
          const bool exists = tid < (uint32_t)s_c.T;
          const uint32_t tc = exists ? s_tc[tid] : 0u;
          x = (int32_t)bx * s_c.B[0] + (int32_t)(tc & 1023u);
          y = (int32_t)by * s_c.B[1] + (int32_t)((tc >> 10) & 1023u);
          z = (int32_t)bz * s_c.B[2] + (int32_t)(tc >> 20);
          if (faxis == 1) y *= fold;
          if (faxis == 2) z *= fold;
          valid = exists && x < s_c.N[0] && y < s_c.N[1] && z < s_c.N[2];
          kv = 0;
          if (valid) kv = faxis == 1 ? min(fold, s_c.N[1] - y) : faxis == 2 ? min(fold, s_c.N[2] - z) : 1;
        }
        if (j == 0u) {
          if (s_g.first_of_cfg) acc_lb += mult * __reduce_add_sync(FULL, (uint32_t)kv);
          acc_addr += mult * __reduce_add_sync(FULL, (uint32_t)s_gad[0][kv]);
          acc_wi += mult * (uint32_t)s_gwi[0];
        }
        const int k = s_af[j];
        if (k != cur_k) {
          cur_k = k;
          const DField &F = s_fk[k];
          const int64_t lin = F.stride[0] * x + F.stride[1] * y + F.stride[2] * z;
          rbase = F.base + (int64_t)F.esize * lin - 32 * F.lo[0];
          rlim = F.words[0] << 10;
        }
        const DField &F = s_fk[k];
        const bool act = valid && (int)s_kmin[j] < kv;
        const int64_t rr = rbase + s_boff[j];
        const bool inside = rr >= 0 && rr < rlim;
        uint32_t nsec;
        if (count_only) nsec = warp_distinct_sectors((uint32_t)rr, act && inside);
        else nsec = bitmap_insert(a.scratch + F.bm[j < L ? BM_BL : BM_BS], rr, act, lane, F.words[0], bad);
        if (j < L) acc_req += mult * nsec;
        else acc_st += mult * nsec;
        if (fast_banks && !F.wide)
          acc_bank += mult * bank_cycles_rel32((uint32_t)rr, act && inside, lane, (uint32_t)a.bank_shift,
                                               (uint32_t)(a.banks - 1), (uint32_t)a.pair_dist);
        else
          acc_bank += mult * bank_cycles_warp(rr + 32 * F.lo[0], act, lane, a.banks, a.bank_bytes, a.pair_dist);
        if (++j == LS) {
          j = 0;
          ++r;
        }
      }
    }
    for (uint32_t mw = mw0 + warp; mw < mw1; mw += nwarps) {
      // ---- decode the modelled warp once for every field of the group
      uint32_t level, b, j;
      const FastDiv fwpb = s_c.fd_wpb;
      if (mw < (uint32_t)s_c.lev_end[0]) {
        level = 0; j = mw; b = (uint32_t)s_c.rep;
      } else if (mw < (uint32_t)s_c.lev_end[1]) {
        level = 1; j = mw - (uint32_t)s_c.lev_end[0]; b = (uint32_t)s_c.s + fdiv(j, fwpb);
      } else if (mw < (uint32_t)s_c.lev_end[2]) {
        level = 2; j = mw - (uint32_t)s_c.lev_end[1]; b = (uint32_t)s_c.y_lo + fdiv(j, fwpb);
      } else {
        level = 3; j = mw - (uint32_t)s_c.lev_end[2]; b = (uint32_t)s_c.z_lo + fdiv(j, fwpb);
      }
      const uint32_t gx = (uint32_t)s_c.g[0], gy = (uint32_t)s_c.g[1];
      const uint32_t w = j - fdiv(j, fwpb) * (uint32_t)s_c.wpb;
      const uint32_t bt = fdiv(b, s_c.fd_gx);
      const uint32_t bx = b - bt * gx;
      const uint32_t bz = fdiv(bt, s_c.fd_gy);
      const uint32_t by = bt - bz * gy;
      if (level == 2 && by == gy - 1) continue;
      if (level == 3 && b >= (uint32_t)s_c.y_lo && b < (uint32_t)s_c.y_hi && by != gy - 1) continue;

      const uint32_t tid = w * 32u + lane;
      const bool exists = tid < (uint32_t)s_c.T;
      const uint32_t tc = exists ? s_tc[tid] : 0u;
      const int32_t x = (int32_t)bx * s_c.B[0] + (int32_t)(tc & 1023u);
      int32_t y = (int32_t)by * s_c.B[1] + (int32_t)((tc >> 10) & 1023u);
      int32_t z = (int32_t)bz * s_c.B[2] + (int32_t)(tc >> 20);
      const int32_t faxis = s_c.fold_axis, fold = s_c.fold;
      if (faxis == 1) y *= fold;
      if (faxis == 2) z *= fold;
      const bool valid = exists && x < s_c.N[0] && y < s_c.N[1] && z < s_c.N[2];
      int kv = 0;
      if (valid) kv = faxis == 1 ? min(fold, s_c.N[1] - y) : faxis == 2 ? min(fold, s_c.N[2] - z) : 1;
      if (s_g.first_wave && level == 1) acc_lw += __reduce_add_sync(FULL, (uint32_t)kv);
      const uint32_t vmask = __ballot_sync(FULL, valid);
      // a thread with fewer valid folded points than the fold skips some accesses; such
      // warps (only at the domain edge) bound-check every address
      const bool partial = __any_sync(FULL, valid && kv < fold);
      uint32_t naddr = 0;

      bool fields_done = false;
      if (level >= 1 && s_g.iv) {
        // ---- interval walk (exact closed-form counting, Sec. 4.4): the warp's valid
        // threads form row segments of consecutive x, and a (segment, merged load run)
        // pair covers one contiguous sector range.  Partial warps (a thread with fewer
        // valid folded points than the fold) take the raw folded loads instead, each
        // checked against the segment's valid points.
        const DField &F0 = s_fk[0];
        const int64_t el = (int64_t)F0.esize * (F0.stride[0] * x + F0.stride[1] * y + F0.stride[2] * z);
        const uint32_t tme = (uint32_t)el;
        s_tbase[warp][lane] = tme;
        const int L = s_loff[s_g.f_count];
        const int S = level == 1 ? s_soff[s_g.f_count] - L : 0;
        if (vmask) {
          // the warp's address range: offsets from its first valid thread fit 32 bits
          // (every bitmap of an interval group spans less than 2^31 bytes); anything
          // else is a descriptor error and the warp is skipped
          const int64_t e0 = (int64_t)__shfl_sync(FULL, (long long)el, __ffs(vmask) - 1);
          const int64_t dd = el - e0;
          const bool fits = !valid || (dd >= -(int64_t)0x7fffffff && dd <= (int64_t)0x7fffffff);
          if (__all_sync(FULL, fits)) {
            const int32_t d = (int32_t)dd;
            const int64_t mn = e0 + __reduce_min_sync(FULL, valid ? d : 0x7fffffff);
            const int64_t mx = e0 + __reduce_max_sync(FULL, valid ? d : -0x7fffffff);
            const uint32_t tx = tc & 1023u;
            const uint32_t heads = __ballot_sync(FULL, valid && (lane == 0u || tx == 0u));
            const uint32_t ends = vmask & ~((vmask & ~heads) >> 1);
            const uint32_t nseg = __popc(heads);
            if ((heads >> lane) & 1u) {
              const uint32_t t = __ffs(ends & (0xffffffffu << lane)) - 1u;
              s_seg[warp][__popc(heads & ((1u << lane) - 1u))] = lane | (t << 8) | ((uint32_t)kv << 16);
            }
            __syncwarp();
            // loads: a lane takes one entry and every G-th segment (G lanes share an
            // entry when there are fewer than 32)
            const int pi = partial ? 1 : 0;
            const int M = partial ? L : s_ioff[s_g.f_count];
            const uint32_t G = s_lgG[pi], lg = s_lg[pi][lane];
            const uint32_t e_l = lg & 255u, g_l = lg >> 8;
            const int bsel = level == 1 ? BM_W : level == 2 ? BM_Y : BM_Z;
            for (int r0 = 0; r0 < M; r0 += 32) {
              const int e = r0 + (int)e_l;
              if (e >= M || g_l >= G) continue;
              int k;
              int64_t bo;
              uint32_t ext;
              if (!partial) {
                k = s_iaf[e];
                bo = s_ibo[e];
                ext = s_iext[e];
              } else {
                k = s_af[e];
                bo = s_boff[e] + s_fk[k].base - 32 * s_fk[k].lo[1];
                ext = 0u;
              }
              const DField &F = s_fk[k];
              const uint32_t limit = (uint32_t)(F.words[1] << 10);
              unsigned long long *const bm = reinterpret_cast<unsigned long long *>(a.scratch + F.bm[bsel]);
              uint32_t cu = 0xffffffffu;
              unsigned long long cb = 0ull;
              if (!partial) {
                // every segment issues the entry: one exact range check for the warp
                if (mn + bo < 0 || mx + bo + (int64_t)ext >= (int64_t)limit) {
                  ++bad;
                  continue;
                }
                const uint32_t b32 = (uint32_t)bo;
                for (uint32_t si = g_l; si < nseg; si += G) {
                  const uint32_t sg = s_seg[warp][si];
                  const uint32_t ra = s_tbase[warp][sg & 255u] + b32, rb = s_tbase[warp][(sg >> 8) & 255u] + b32;
                  put_range(bm, cu, cb, min(ra, rb) >> 5, (max(ra, rb) + ext) >> 5);
                }
              } else {
                const uint32_t kmin = s_kmin[e];
                for (uint32_t si = g_l; si < nseg; si += G) {
                  const uint32_t sg = s_seg[warp][si];
                  if (kmin >= (sg >> 16)) continue;
                  uint32_t lo, hi;
                  if (!segment_range(s_tbase[warp][sg & 255u], s_tbase[warp][(sg >> 8) & 255u], mn, bo, 0u, limit,
                                     lo, hi)) {
                    ++bad;
                    continue;
                  }
                  put_range(bm, cu, cb, lo >> 5, hi >> 5);
                }
              }
              if (cb) atomicOr(bm + cu, cb);
            }
            if (!partial) {
              // stores: lane per store instruction over all segments, counting the
              // instruction's distinct sectors (exact for non-decreasing segments)
              for (int a0 = 0; a0 < S; a0 += 32) {
                const int j = L + a0 + (int)lane;
                uint32_t nsec = 0u, plo = 0u, phi = 0u;
                bool mono = true, ok = false;
                if (j < L + S) {
                  const DField &F = s_fk[s_af[j]];
                  const int64_t bo = s_boff[j] + F.base - 32 * F.lo[1];
                  const uint32_t limit = (uint32_t)(F.words[1] << 10);
                  unsigned long long *const bm = reinterpret_cast<unsigned long long *>(a.scratch + F.bm[BM_WS]);
                  if (mn + bo < 0 || mx + bo >= (int64_t)limit) {
                    ++bad;
                  } else {
                    ok = true;
                    const uint32_t b32 = (uint32_t)bo;
                    uint32_t cu = 0xffffffffu;
                    unsigned long long cb = 0ull;
                    for (uint32_t si = 0; si < nseg; ++si) {
                      const uint32_t sg = s_seg[warp][si];
                      const uint32_t ra = s_tbase[warp][sg & 255u] + b32, rb = s_tbase[warp][(sg >> 8) & 255u] + b32;
                      const uint32_t s0 = min(ra, rb) >> 5, s1 = max(ra, rb) >> 5;
                      put_range(bm, cu, cb, s0, s1);
                      if (si == 0u) {
                        nsec = s1 - s0 + 1u;
                      } else {
                        mono = mono && s0 >= plo && s1 >= phi;
                        const uint32_t from = max(phi + 1u, s0);
                        nsec += s1 >= from ? s1 - from + 1u : 0u;
                      }
                      plo = s0;
                      phi = s1;
                    }
                    if (cb) atomicOr(bm + cu, cb);
                  }
                }
                acc_sreq += __reduce_add_sync(FULL, (ok && mono) ? nsec : 0u);
                uint32_t redo = __ballot_sync(FULL, ok && !mono);
                while (redo) {
                  const int src = __ffs(redo) - 1;
                  redo &= redo - 1;
                  acc_sreq += warp_distinct_sectors(tme + s_b32[L + a0 + src], valid);
                }
              }
            } else {
              for (int j = L; j < L + S; ++j) {
                const DField &F = s_fk[s_af[j]];
                const uint32_t limit = (uint32_t)(F.words[1] << 10);
                const bool act = valid && (int)s_kmin[j] < kv;
                acc_sreq += runs_insert(a.scratch + F.bm[BM_WS], tme + s_b32[j], act, limit, lane, bad, true);
              }
            }
          } else if (lane == 0u) {
            ++bad;
          }
        }
        __syncwarp();
        fields_done = true;
        naddr += (uint32_t)s_gad[level <= 1 ? 0 : 1][kv];
        acc_wi += (uint32_t)s_gwi[level <= 1 ? 0 : 1];
      } else if (level >= 1 && s_g.uniform && !partial) {
        // ---- uniform groups, wave / y / z levels: one walk over all the group's accesses
        const DField &F0 = s_fk[0];
        const int64_t el = (int64_t)F0.esize * (F0.stride[0] * x + F0.stride[1] * y + F0.stride[2] * z);
        s_tbase[warp][lane] = (uint32_t)el;
        int64_t mn = valid ? el : INT64_MAX, mx = valid ? el : INT64_MIN;
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
          mn = min(mn, (int64_t)__shfl_xor_sync(FULL, (long long)mn, off));
          mx = max(mx, (int64_t)__shfl_xor_sync(FULL, (long long)mx, off));
        }
        __syncwarp();
        const int L = s_loff[s_g.f_count];
        const int S = level == 1 ? s_soff[s_g.f_count] - L : 0;
        const uint32_t tme = s_tbase[warp][lane];
        if (L >= kCombinedWalkMin) {
          // lane per access over all 32 threads of the modelled warp
          for (int a0 = 0; a0 < L && vmask; a0 += 32) {
            const int j = a0 + (int)lane;
            uint32_t cw = 0xffffffffu, cb = 0u;
            uint32_t *bm = nullptr;
            if (j < L) {
              const DField &F = s_fk[s_af[j]];
              const int64_t bo = s_boff[j] + F.base - 32 * F.lo[1];
              const uint32_t limit = (uint32_t)(F.words[1] << 10);
              bm = a.scratch + F.bm[level == 1 ? BM_W : level == 2 ? BM_Y : BM_Z];
              if (mn + bo < 0 || mx + bo >= (int64_t)limit) bad += __popc(vmask);
              else lpa_walk<32, false>(&s_tbase[warp][0], vmask, s_b32[j], limit, bm, cw, cb, bad);
            }
            if (cb) atomicOr(bm + cw, cb);
          }
        } else {
          // few accesses: lane per thread, one run-head insertion per access
          for (int j = 0; j < L; ++j) {
            const DField &F = s_fk[s_af[j]];
            const uint32_t limit = (uint32_t)(F.words[1] << 10);
            uint32_t *const bm = a.scratch + F.bm[level == 1 ? BM_W : level == 2 ? BM_Y : BM_Z];
            runs_insert(bm, tme + s_b32[j], valid, limit, lane, bad, false);
          }
        }
        if (S >= kCombinedWalkMin) {
          for (int a0 = 0; a0 < S && vmask; a0 += 32) {
            const int j = L + a0 + (int)lane;
            uint32_t cw = 0xffffffffu, cb = 0u, nsec = 0u;
            bool mono = true, ok = false;
            uint32_t *bm = nullptr;
            if (j < L + S) {
              const DField &F = s_fk[s_af[j]];
              const int64_t bo = s_boff[j] + F.base - 32 * F.lo[1];
              const uint32_t limit = (uint32_t)(F.words[1] << 10);
              bm = a.scratch + F.bm[BM_WS];
              if (mn + bo < 0 || mx + bo >= (int64_t)limit) {
                bad += __popc(vmask);
              } else {
                lpa_walk_count(&s_tbase[warp][0], vmask, s_b32[j], bm, cw, cb, nsec, mono);
                ok = true;
              }
            }
            if (cb) atomicOr(bm + cw, cb);
            // per-instruction distinct sectors: the lane's count when its sectors never
            // decreased, else an exact recount by the whole warp
            acc_sreq += __reduce_add_sync(FULL, (ok && mono) ? nsec : 0u);
            uint32_t redo = __ballot_sync(FULL, ok && !mono);
            while (redo) {
              const int src = __ffs(redo) - 1;
              redo &= redo - 1;
              acc_sreq += warp_distinct_sectors(tme + s_b32[L + a0 + src], valid);
            }
          }
        } else {
          for (int j = L; j < L + S; ++j) {
            const DField &F = s_fk[s_af[j]];
            const uint32_t limit = (uint32_t)(F.words[1] << 10);
            acc_sreq += runs_insert(a.scratch + F.bm[BM_WS], tme + s_b32[j], valid, limit, lane, bad, true);
          }
        }
        __syncwarp();
        fields_done = true;
        naddr += (uint32_t)s_gad[level <= 1 ? 0 : 1][kv];
        acc_wi += (uint32_t)s_gwi[level <= 1 ? 0 : 1];
      }

      // ---- every field of the group
      for (int k = 0; k < s_g.f_count && !fields_done; ++k) {
        const DField &F = s_fk[k];
        const int n_load = F.n_load;
        const int nst = level <= 1 ? F.n_store : 0;
        if (n_load + (level <= 1 ? nst : 0) == 0 || (level >= 2 && n_load == 0)) continue;
        const int lo_ = s_loff[k], so_ = s_soff[k] - n_load;   // load i at lo_ + i, store i at so_ + i
        naddr += (uint32_t)(F.cnt_load[kv] + (level <= 1 ? F.cnt_store[kv] : 0));
        acc_wi += (uint32_t)(n_load + nst);
        const int64_t lin = F.stride[0] * x + F.stride[1] * y + F.stride[2] * z;

        if (!F.wide) {
          const int64_t rel = F.base + (int64_t)F.esize * lin - 32 * F.lo[1];
          // uniform groups staged the field constant into the 32-bit offsets already
          const uint32_t r0 = s_g.uniform ? (uint32_t)((int64_t)F.esize * lin) : (uint32_t)rel;
          const uint32_t limit = (uint32_t)(F.words[1] << 10);
          uint32_t *const bm = a.scratch + F.bm[level == 1 ? BM_W : level == 2 ? BM_Y : BM_Z];
          if (n_load > 0) {
            // lane per access over slices of P threads (P = 2^lp >= loads, <= 32)
            const int lp = F.lpa_log2p, P = 1 << lp;
            if (P > 1) {
              s_tbase[warp][lane] = r0;
              s_tkv[warp][lane] = (uint8_t)kv;
              __syncwarp();
            }
            // fields with a full warp per access check each lane's range once
            int64_t mn = 0, mx = 0;
            if (P == 32 && !partial) {
              mn = valid ? rel : INT64_MAX;
              mx = valid ? rel : INT64_MIN;
#pragma unroll
              for (int off = 16; off >= 1; off >>= 1) {
                mn = min(mn, (int64_t)__shfl_xor_sync(FULL, (long long)mn, off));
                mx = max(mx, (int64_t)__shfl_xor_sync(FULL, (long long)mx, off));
              }
            }
            const uint32_t al = lane & (uint32_t)(P - 1), g0 = (lane >> lp) << lp;
            const uint32_t slice = (P == 32 ? vmask : (vmask >> g0) & ((1u << P) - 1u));
            const uint32_t *tb = &s_tbase[warp][g0];
            for (int a0 = 0; a0 < n_load && vmask; a0 += P) {
              const int ai = a0 + (int)al;
              uint32_t cw = 0xffffffffu, cb = 0u;
              if (ai < n_load && slice) {
                const uint32_t b32 = s_b32[lo_ + ai];
                if (!partial) {
                  if (P == 32) {
                    const int64_t bo = s_boff[lo_ + ai];
                    if (mn + bo < 0 || mx + bo >= (int64_t)limit) bad += __popc(slice);
                    else lpa_walk<32, false>(tb, slice, b32, limit, bm, cw, cb, bad);
                  } else {
                    switch (lp) {
                      case 0: {  // one thread per lane: its own address, no staging
                        const uint32_t r = r0 + b32;
                        if (r >= limit) {
                          ++bad;
                        } else {
                          cw = r >> 10;
                          cb = __funnelshift_l(0u, 1u, r >> 5);
                        }
                        break;
                      }
                      case 1: lpa_walk<2, true>(tb, slice, b32, limit, bm, cw, cb, bad); break;
                      case 2: lpa_walk<4, true>(tb, slice, b32, limit, bm, cw, cb, bad); break;
                      case 3: lpa_walk<8, true>(tb, slice, b32, limit, bm, cw, cb, bad); break;
                      default: lpa_walk<16, true>(tb, slice, b32, limit, bm, cw, cb, bad); break;
                    }
                  }
                } else {
                  const int km = s_kmin[lo_ + ai];
                  for (int t = 0; t < P; ++t) {
                    if (!((slice >> t) & 1u) || km >= (P > 1 ? (int)s_tkv[warp][g0 + t] : kv)) continue;
                    const uint32_t r = (P > 1 ? tb[t] : r0) + b32;
                    if (r >= limit) {
                      ++bad;
                      continue;
                    }
                    const uint32_t wd = r >> 10;
                    if (wd != cw) {
                      if (cb) atomicOr(bm + cw, cb);
                      cw = wd;
                      cb = 0u;
                    }
                    cb |= 1u << ((r >> 5) & 31u);
                  }
                }
              }
              if (P == 32) {
                if (cb) atomicOr(bm + cw, cb);
              } else {
                // several slices per access: lanes whose last word coincides (other
                // slices, other accesses) merge it into one red.or
                const uint32_t key = cb ? cw : (0x80000000u | lane);
                const uint32_t m = __match_any_sync(FULL, key);
                const uint32_t orcb = __reduce_or_sync(m, cb);
                if (cb && lane == (uint32_t)(__ffs(m) - 1)) atomicOr(bm + cw, orcb);
              }
            }
            if (P > 1) __syncwarp();
          }
          // wave stores: per-instruction unique sectors (partial-store model)
          uint32_t *const ws_ = a.scratch + F.bm[BM_WS];
          for (int i = n_load; i < n_load + nst; ++i) {
            const bool act = valid && (int)s_kmin[so_ + i] < kv;
            acc_sreq += runs_insert(ws_, r0 + s_b32[so_ + i], act, limit, lane, bad, true);
          }
        } else {
          const int64_t rel = F.base + (int64_t)F.esize * lin - 32 * F.lo[1];
          uint32_t *const bm = a.scratch + F.bm[level == 1 ? BM_W : level == 2 ? BM_Y : BM_Z];
          for (int i = 0; i < n_load; ++i) {
            const bool act = valid && (int)s_kmin[lo_ + i] < kv;
            bitmap_insert(bm, rel + s_boff[lo_ + i], act, lane, F.words[1], bad);
          }
          uint32_t *const ws_ = a.scratch + F.bm[BM_WS];
          for (int i = n_load; i < n_load + nst; ++i) {
            const bool act = valid && (int)s_kmin[so_ + i] < kv;
            acc_sreq += bitmap_insert(ws_, rel + s_boff[so_ + i], act, lane, F.words[1], bad);
          }
        }
      }
      acc_addr += __reduce_add_sync(FULL, naddr);
    }
    bad = __reduce_add_sync(FULL, bad);
    if (lane == 0) {
      unsigned long long *c = (unsigned long long *)(a.counters + (int64_t)s_g.cfg * N_COUNTERS);
      typedef unsigned long long u64;
      if (bad) atomicAdd(c + C_OVERFLOW, (u64)bad);
      if (acc_lb) atomicAdd(c + C_LUPS_BLOCK, (u64)acc_lb);
      if (acc_lw) atomicAdd(c + C_LUPS_WAVE, (u64)acc_lw);
      if (acc_req) atomicAdd(c + C_L1_REQ, (u64)acc_req);
      if (acc_st) atomicAdd(c + C_L1_STORE, (u64)acc_st);
      if (acc_bank) atomicAdd(c + C_BANK, (u64)acc_bank);
      if (acc_sreq) atomicAdd(c + C_W_SREQ, (u64)acc_sreq);
      if (acc_addr) atomicAdd(c + C_ADDR, (u64)acc_addr);
      if (acc_addr && blk) atomicAdd(c + C_ADDR0, (u64)acc_addr);
      if (acc_wi) atomicAdd(c + C_WINSTR, (u64)acc_wi);
    }
    __syncthreads();
  }
}


// Row walk of the wave and the y / z layer sets (exact closed-form interval counting,
// Sec. 4.4).  The blocks of a level that share a block row are consecutive in x, so
// the threads of those blocks with one (ty, tz) form one grid row of consecutive x.
// Work item = (field group, chunk of row slots); one grid row per warp.  Each merged
// load run (raw loads when the row has fewer valid folded points than the fold) is one
// sector range of the row; wave stores also add their per-warp sector counts in closed
// form (row_store_sectors).
// Magic numbers of FastDiv for a divisor fixed per work item (once per thread and item).
__device__ __forceinline__ FastDiv make_fastdiv_dev(uint32_t d) {
  FastDiv f;
  f.d = d;
  f.s = d <= 1u ? 0u : 32u - __clz(d - 1u);
  f.m = (uint32_t)((((unsigned long long)1 << 32) * (((unsigned long long)1 << f.s) - d)) / d + 1ull);
  return f;
}

// One decoded row slot (a lane's): the byte range of its row (relative to the field
// base; the fields of a row-walk group share element size and strides), the start of the
// row, its thread row, block run, level and valid folded points.
struct RowSlot {
  int64_t lo, hi, el0;
  uint32_t t, bxa, bxb;
  int32_t y, z;           // grid row of the slot's first folded point
  uint8_t lv, kv, pad[2];
};

// True when every grid row displaced from row (y, z) of level lv by at most dy rows in y
// and dz in z (multiples of the fold along the folding axis) is a thread row of the same
// level whose block run contains [bxa, bxb) and whose folded points are all inside the
// domain.  The displaced rows' block rows lie between those of the two extreme corners
// (R = by + gy * bz grows with by and bz), so the level's block interval is checked at
// those two; the z set is checked against its tighter bound (before the y set) throughout.
// Then every run whose covering run lies within that displacement may be skipped at this
// row: the covering run sets a containing range from the displaced row, which the walk
// visits with a containing block run (and if it skips that run there in turn, a run even
// earlier in the covering order covers both).
__device__ __forceinline__ bool row_interior(const DCfg &c, int lv, int32_t y, int32_t z, uint32_t bxa, uint32_t bxb,
                                             int32_t dy, int32_t dz) {
  const int32_t fy = c.fold_axis == 1 ? c.fold : 1, fz = c.fold_axis == 2 ? c.fold : 1;
  if (y < dy || z < dz || y + dy + fy > c.N[1] || z + dz + fz > c.N[2]) return false;
  uint32_t y0 = (uint32_t)(y - dy), y1 = (uint32_t)(y + dy), z0 = (uint32_t)(z - dz), z1 = (uint32_t)(z + dz);
  if (c.fold_axis == 1) {
    y0 = fdiv(y0, c.fd_fold);
    y1 = fdiv(y1, c.fd_fold);
  } else if (c.fold_axis == 2) {
    z0 = fdiv(z0, c.fd_fold);
    z1 = fdiv(z1, c.fd_fold);
  }
  const uint32_t by0 = fdiv(y0, c.fd_b1), by1 = fdiv(y1, c.fd_b1);
  const uint32_t bz0 = fdiv(z0, c.fd_b2), bz1 = fdiv(z1, c.fd_b2);
  if (lv == 3) return by0 == by1 && bz0 == bz1;   // the representative block's own thread rows
  const int64_t gx = c.g[0], gy = c.g[1];
  const int64_t lo = ((int64_t)by0 + gy * (int64_t)bz0) * gx + bxa;
  const int64_t hi = ((int64_t)by1 + gy * (int64_t)bz1) * gx + bxb;
  if (lv == 0) return c.s <= lo && hi <= c.s + c.weff;
  if (lv == 1) return (int64_t)by1 != gy - 1 && c.y_lo <= lo && hi <= c.y_hi;
  const int64_t up = c.y_hi > c.y_lo ? min(c.z_hi, c.y_lo) : c.z_hi;
  return c.z_lo <= lo && hi <= up;
}


// ---- closed-form footprints (ws_footprint.h) -------------------------------------------
// A warp takes one part of one field's loads, stores and representative block.  It goes over a
// task's target rows in units: the rows of a plane, repeated over the planes in which the
// blocks' slabs let every state repeat (a block 64 planes deep has some 60 of them), whose
// addresses differ by whole planes.  Parts share out the units in turn.  Inside a unit the warp
// advances in windows of 32 rows, a lane per row.  First a lane per displacement looks up
// which run of each level lands in the window and up to which row that stays so; displacements
// constant over the window give their range to all rows with warp reductions, the others are
// looked up row by row.  When everything is constant, the stretch up to the next change is
// counted at once: its first 32 rows, then one period of the row addresses modulo a line (32
// rows when the pitch is a multiple of four bytes) with the number of times each position
// repeats.  Repeated planes likewise are counted once per position of the plane address modulo
// a line; a window of few rows counts several of those positions at a time.
constexpr int kFootRowCache = 64, kFootList = 48;

// A task of a field: the loads or stores of the wave or of the block.
struct FootTask {
  const int4 *dsp;     // displacements
  uint32_t base;       // address of x = 0 in row 0 (modulo 2^32; only its place in a line counts)
  int32_t nd;          // their number (0: no such task)
  int32_t P;           // pitch of a row
  int32_t hmin;        // lowest byte of a row's ranges
  int32_t pz, pzs;     // planes until their addresses repeat modulo a line (a power of two), log2
  int32_t ymin;        // smallest displacement within a plane
  int32_t rows;        // rows of a plane's unit that can hold anything
  int32_t single;      // planes around a slab's end that units take one by one
  int32_t zmove;       // wave loads: the z set's lines are the wave's, this many bytes on (-1: its own)
  int32_t tr[4];       // target rows (foot_targets)
};
struct FootSmem {
  FootGeo geo[2];      // wave, block: geometry of the warp's current field group
  FootTask task[4];    // of its current field: wave loads, wave stores, block loads, block stores
  // the row before a window: its ranges and levels (foot_join)
  int32_t vl[3], vh[3];
  uint32_t vm;
  int ld;                                   // the unit's displacements
  union {
    unsigned long long sreq[kFootRowCache];   // store sectors of rows by what they depend on (foot_stats)
    int4 list[kFootList];                     // the displacements left of a unit (foot_merge_list)
  };
};

// Displacements up to which the rows of a short unit look them all up (a lane per row); with
// more, and in long units, a lane per displacement first finds those that are constant over the
// window.
constexpr int kFootFew = 12;

__device__ __forceinline__ void foot_sum(FootCounts &a, const FootCounts &b) {
  a.sec += b.sec;
  a.lin += b.lin;
  a.ylin += b.ylin;
  a.zlin += b.zlin;
  a.ovy += b.ovy;
  a.ovz += b.ovz;
}

// Counts a lane's target row t, `rows` times, where a level's first and last block rows leave a
// gap between them (on this row or on another of the window): every displacement of the row and
// of the row before it, piece by piece.  reps: the row's repeated planes (of at most `planes`).
// Seldom taken and long: kept out of the walk's code, whose instructions have to stay in the SM's
// caches.
__device__ __noinline__ FootCounts foot_gaps(const FootGeo &g, const FootTask &k, const FootSmem &m, int nl, int32_t t,
                                             uint32_t rows, int32_t reps, int32_t planes) {
  FootCounts out = {0, 0, 0, 0, 0, 0};
  if (reps <= 0 || rows == 0) return out;
  const int nd = m.ld >= 0 ? m.ld : k.nd;
  const int4 *const dsp = m.ld >= 0 ? m.list : k.dsp;
  FootHull cur, prv;
  cur.clear();
  prv.clear();
#pragma unroll 1
  for (int e = 0; e < nd; ++e) {
    const int4 v = dsp[e];
    FootRow row;
    foot_row(g, nl, t - v.x, false, row);
    foot_add(row, nl, v.y, v.z, cur);
    foot_row(g, nl, t - 1 - v.x, false, row);
    foot_add(row, nl, v.y, v.z, prv);
  }
  const int32_t A = (int32_t)((k.base + (uint32_t)k.P * (uint32_t)t) & 127u), pzs = k.pzs;
  const int32_t plane = (int32_t)(((uint32_t)k.P * (uint32_t)g.q) & 127u);
  uint32_t zl = 0;
#pragma unroll 1
  for (int32_t i = 0; i < min(planes, k.pz); ++i) {
    const uint32_t mult = rows * ((uint32_t)(reps - i + k.pz - 1) >> pzs);
    if (mult) {
      foot_count_pieces(cur, prv, A + i * plane, k.P, k.hmin, mult, out);
      if (k.zmove > 0) {
        FootCounts moved = {0, 0, 0, 0, 0, 0};
        foot_count_pieces(cur, prv, A + i * plane + k.zmove, k.P, k.hmin, mult, moved);
        zl += moved.lin;
      }
    }
  }
  if (k.zmove > 0) out.zlin = zl;
  return out;
}

// Counts target rows [t_begin, t_end), each repeated over `reps` planes.  prime: the row before
// t_begin may hold something (else it is empty in every plane).  Where the rows of whole planes
// join (not every plane's stand alone), the first row's own predecessor lies before the repeated
// planes and may differ from theirs: that row, t_first, is counted once, and the row q further
// on, t_last, whose predecessor is the plane's last row, reps - 1 times in its place (kRowNone:
// no such row among these).
constexpr int32_t kRowNone = -kRowInf;
__device__ __forceinline__ void foot_walk(const FootGeo &g, const FootTask &k, FootSmem &m, int nl, int32_t t_begin,
                                          int32_t t_end, int32_t reps, bool prime, int32_t t_first, int32_t t_last,
                                          FootCounts &out) {
  const uint32_t lane = threadIdx.x & 31u;
  __syncwarp();
  if (lane == 0) {
    m.vm = 0;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      m.vl[l] = kHullLo;
      m.vh[l] = kHullHi;
    }
  }
  __syncwarp();
  const int32_t t_lim = t_last != kRowNone ? t_last : t_end;   // (t_last is the last row)
  const int32_t P = k.P, pzs = k.pzs, nres = min(reps, k.pz);
  const int nd = m.ld >= 0 ? m.ld : k.nd;
  const int4 *const dsp = m.ld >= 0 ? m.list : k.dsp;
  const int32_t plane = (int32_t)(((uint32_t)P * (uint32_t)g.q) & 127u);
  // the row before the first one is looked up too, but not counted
  int32_t t = t_begin - (prime ? 1 : 0);
#pragma unroll 1
  for (;;) {
  int gap = 0;   // rows of a window that takes foot_gaps (called outside the windows' loop)
#pragma unroll 1
  while (t < t_end) {
    FootHull U;
    U.clear();
    const int32_t left = t_end - t;
    bool varies = true;
    int32_t nb = kRowInf;   // first row at which a displacement constant over the window changes
    uint32_t todo = (1u << min(nd, kFootFew)) - 1u;   // displacements left to the rows (lane j: of the j-th 32)
    if (left > 32 || nd > kFootFew) {
      uint32_t some = 0;
#pragma unroll 1
      for (int e0 = 0; e0 < nd; e0 += 32) {
        bool part = false;
        if (e0 + (int)lane < nd) {
          const int4 v = dsp[e0 + (int)lane];
          FootRow row;
          const int32_t nx = foot_row(g, nl, t - v.x, true, row);
          const int32_t nt = nx == kRowInf ? kRowInf : nx + v.x;
          part = nt < t + min(32, left);
          if (!part) {
            nb = min(nb, nt);
            foot_add(row, nl, v.y, v.z, U);
          }
        }
        const uint32_t pm = __ballot_sync(FULL, part);
        if (lane == (uint32_t)e0 >> 5) todo = pm;
        some |= pm;
      }
      varies = some != 0u;
      // the constant displacements' ranges, for all rows
      nb = __reduce_min_sync(FULL, nb);
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        if (l > 0 && nl == 1) break;
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (__any_sync(FULL, U.lo[l][c] <= U.hi[l][c])) {
            U.lo[l][c] = __reduce_min_sync(FULL, U.lo[l][c]);
            U.hi[l][c] = __reduce_max_sync(FULL, U.hi[l][c]);
          }
      }
    }
    if (varies) {
#pragma unroll 1
      for (int e0 = 0; e0 < nd; e0 += 32) {
        uint32_t pm = __shfl_sync(FULL, todo, e0 >> 5);
#pragma unroll 1
        while (pm) {
          const int4 v = dsp[e0 + __ffs(pm) - 1];
          pm &= pm - 1;
          FootRow row;
          foot_row(g, nl, t + (int32_t)lane - v.x, false, row);
          foot_add(row, nl, v.y, v.z, U);
        }
      }
    }
    int32_t cl[3], ch[3], pl[3], ph[3];
    const uint32_t um = foot_join(U, nl, cl, ch);
    uint32_t um1 = __shfl_up_sync(FULL, um, 1);
    if (lane == 0) um1 = m.vm;
    const int32_t tl = t + (int32_t)lane;
    const bool act = (um | um1) != 0u && (int32_t)lane < left && tl >= t_begin;
    uint32_t levels = __reduce_or_sync(FULL, act ? um | um1 : 0u);
    int32_t n = min(32, left), rest = 0;
    if (!varies) {
      // constant up to row nb (row t_last, if among them, is left to the next window)
      n = max(n, min(nb, t_lim) - t);
      rest = n - 32;
    }
    if (levels & 8u) {
      gap = n;
    } else if (levels) {
      int32_t rl = !act ? 0 : tl == t_last ? reps - 1 : tl == t_first ? 1 : reps;
      {
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          pl[l] = __shfl_up_sync(FULL, cl[l], 1);
          ph[l] = __shfl_up_sync(FULL, ch[l], 1);
          if (lane == 0) {
            pl[l] = m.vl[l];
            ph[l] = m.vh[l];
          }
        }
        int32_t A = (int32_t)((k.base + (uint32_t)P * (uint32_t)tl) & 127u);
        const uint32_t am = __ballot_sync(FULL, act);
        const int first = __ffs(am) - 1, span = 32 - __clz(am) - first;
        __syncwarp();
        if ((int)lane == min(n, 32) - 1) {
#pragma unroll
          for (int l = 0; l < 3; ++l) {
            m.vl[l] = cl[l];
            m.vh[l] = ch[l];
          }
        }
        __syncwarp();
        int32_t i0 = 0, di = 1;
        if (nres > 1 && span <= 16) {
          // few rows: 32 / w plane positions at a time, w >= the rows
          const int ws = span <= 1 ? 0 : 32 - __clz(span - 1), j = (int)lane & ((1 << ws) - 1);
#pragma unroll
          for (int l = 0; l < 3; ++l) {
            if (l > 0 && nl == 1) break;
            cl[l] = __shfl_sync(FULL, cl[l], first + j);
            ch[l] = __shfl_sync(FULL, ch[l], first + j);
            pl[l] = __shfl_sync(FULL, pl[l], first + j);
            ph[l] = __shfl_sync(FULL, ph[l], first + j);
          }
          A = __shfl_sync(FULL, A, first + j);
          rl = __shfl_sync(FULL, rl, first + j);
          if (j >= span) rl = 0;
          i0 = (int32_t)lane >> ws;
          di = 32 >> ws;
        }
        if (k.zmove < 0) levels |= 16u;
        // the window's rows, then one period of the positions of the rows behind it
        uint32_t times = 1;
        const int32_t pers = 5 + (P & 1 ? 2 : P & 2 ? 1 : 0), per = 1 << pers;
        int32_t j0 = -32;
#pragma unroll 1
        for (;;) {
          if (rl > 0)
#pragma unroll 1
            for (int32_t i = i0; i < nres; i += di) {
              const uint32_t mult = times * ((uint32_t)(rl - i + k.pz - 1) >> pzs);
              if (mult) {
                foot_count(cl, ch, pl, ph, A + i * plane, P, k.hmin, mult, levels, out);
                if (k.zmove > 0 && (levels & 1u))
                  out.zlin += mult * foot_count_lines(cl[0], ch[0], pl[0], ph[0], A + i * plane + k.zmove, P, k.hmin);
              }
            }
          j0 += 32;
          if (j0 >= min(per, rest)) break;
          const int32_t j = j0 + (int32_t)lane;
          times = j < rest ? (uint32_t)(rest - j + per - 1) >> pers : 0u;
          rl = reps;
          A = (int32_t)((k.base + (uint32_t)P * (uint32_t)(t + 32 + j)) & 127u);
          i0 = 0;
          di = 1;
#pragma unroll
          for (int l = 0; l < 3; ++l) {
            cl[l] = pl[l] = m.vl[l];   // the state of the window's last row
            ch[l] = ph[l] = m.vh[l];
          }
        }
      }
    }
    // the state of the stretch's last row (a constant stretch: of any of its rows)
    __syncwarp();
    if ((int)lane == min(n, 32) - 1) {
      m.vm = um;
      if (!levels || (levels & 8u)) {
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          m.vl[l] = cl[l];
          m.vh[l] = ch[l];
        }
      }
    }
    __syncwarp();
    if (gap) break;
    t += n;
  }
  if (!gap) break;
  // the window's rows, then one period of the positions of the rows behind it
  {
    const int32_t tl = t + (int32_t)lane;
    const int32_t rl = (int32_t)lane >= gap || tl < t_begin ? 0
                       : tl == t_last                       ? reps - 1
                       : tl == t_first                      ? 1
                                                            : reps;
    foot_sum(out, foot_gaps(g, k, m, nl, tl, 1u, rl, reps));
    const int32_t pers = 5 + (P & 1 ? 2 : P & 2 ? 1 : 0), rest = gap - 32;
#pragma unroll 1
    for (int32_t j = (int32_t)lane; j < min(1 << pers, rest); j += 32)
      foot_sum(out, foot_gaps(g, k, m, nl, t + 32 + j, (uint32_t)(rest - j + (1 << pers) - 1) >> pers, reps, reps));
  }
  t += gap;
  }
}

// floor(a / q) and the remainder of any a > -2^30
__device__ __forceinline__ int32_t foot_rem(int32_t a, const FootGeo &g) {
  const int32_t z = a >= 0 ? (int32_t)foot_div((uint32_t)a, g.fq_m, g.fq_s)
                           : -(int32_t)foot_div((uint32_t)(g.q - 1 - a), g.fq_m, g.fq_s);
  return a - z * g.q;
}

// The displacements of a unit of n rows from t - 1 on: those whose source rows hold nothing are
// left out, those that look up the same states throughout (equal row in a plane of the same
// slab, as the out-of-plane arms of a star on deep blocks) become one with their common range of
// rests.  m.ld = -1: too many, the task's own list stands.
__device__ __forceinline__ void foot_merge_list(const FootGeo &g, const FootTask &k, FootSmem &m, int32_t t, int32_t n) {
  const uint32_t lane = threadIdx.x & 31u;
  int have = 0;
  __syncwarp();
#pragma unroll 1
  for (int e0 = 0; e0 < k.nd && have >= 0; e0 += 32) {
    const int e = e0 + (int)lane;
    int4 v = make_int4(0, 0, 0, 0);
    int32_t key[4] = {-1 - (int32_t)lane, -2, -2, -2};
    bool on = false;
    if (e < k.nd) {
      v = __ldg(k.dsp + e);
      on = foot_key(g, t - 1 - v.x, n, key);
    }
    uint32_t same = __match_any_sync(FULL, key[0]);
    if (__any_sync(FULL, on && (same & (same - 1u)))) {
      same &= __match_any_sync(FULL, key[1]) & __match_any_sync(FULL, key[2]) & __match_any_sync(FULL, key[3]);
      v.y = __reduce_min_sync(same, v.y);
      v.z = __reduce_max_sync(same, v.z);
    }
    const bool keep = on && (int)lane == __ffs(same) - 1;
    const uint32_t km = __ballot_sync(FULL, keep);
    const int at = have + __popc(km & ((1u << lane) - 1u));
    have += __popc(km);
    if (have > kFootList) have = -1;
    else if (keep) m.list[at] = v;
  }
  if (lane == 0) m.ld = have;
  __syncwarp();
}

// One task's share: planes in units, the ones around a slab's ends one by one and the others
// between them together; the parts take equal numbers of units in order.
__device__ __noinline__ FootCounts foot_task(FootSmem &m, int kind, int part, int parts) {
  const uint32_t lane = threadIdx.x & 31u;
  FootCounts out = {0, 0, 0, 0, 0, 0};
  const FootGeo &g = m.geo[kind >> 1];
  const FootTask &k = m.task[kind];
  const int nl = kind == 0 ? 3 : 1;
  // with an empty row to spare on both sides of its rows every plane's stand alone
  const int32_t rows = k.rows, q = g.q;
  const bool isolated = rows + 1 <= q;
#pragma unroll 1
  for (int s = 0; s < 4; s += 2) {
    const int32_t t0 = k.tr[s], t1 = k.tr[s + 1];
    if (t0 >= t1) continue;
    // planes begin where the first displaced plane begins, so that a plane's rows with points
    // are not cut in two
    const int32_t ph0 = foot_rem(t0 - k.ymin, g), np = (int32_t)foot_div((uint32_t)(t1 - t0 + ph0 + q - 1), g.fq_m, g.fq_s);
    int32_t a = 0, b = np;
    uint32_t cut = 1, piece = 0;
    if (parts > 1) {
      // planes before unit u: `single` units of one plane and one of the rest per slab, and
      // `single` at the end (any rising cut of the planes is correct); where the wave's loads have
      // more parts than units the units' rows are cut, too
      const uint32_t n = (uint32_t)np, one = min((uint32_t)k.single, n), n1 = n - one;
      const uint32_t per = (uint32_t)k.single + 1u, b2f = (uint32_t)g.b2f;
      const bool deep = b2f > per;
      const uint32_t full = deep ? foot_div(n1, g.fb2_m, g.fb2_s) : 0u;
      const uint32_t u1 = deep ? full * per + min(n1 - full * b2f, per) : n1, units = u1 + one;
      cut = kind == 0 ? max(1u, (uint32_t)parts / units) : 1u;
      const uint32_t pp = min((uint32_t)parts / cut, units), pu = (uint32_t)part / cut;
      piece = (uint32_t)part - pu * cut;
      if (pu >= pp) continue;
      // (units and pieces stay below 2^25, parts below 2^7)
#pragma unroll 1
      for (uint32_t i = 0; i < 2u; ++i) {
        const uint32_t u = units * (pu + i) / pp, sl = deep ? u / per : 0u;
        const int32_t pl = (int32_t)(u >= u1 ? n1 + (u - u1) : min(n1, deep ? sl * b2f + (u - sl * per) : u));
        if (i == 0u) a = pl;
        else b = pu + 1u == pp ? np : pl;
      }
    }
    int32_t t = max(t0, t0 - ph0 + a * q), ph = a == 0 ? ph0 : 0;
    const int32_t te = min(t1, t0 - ph0 + b * q);
#pragma unroll 1
    while (t < te) {
      if (isolated && ph >= rows) {   // the rest of the plane is empty
        t += q - ph;
        ph = 0;
        continue;
      }
      int32_t n = 1, end = min(te, t + (q - ph));
      if (ph == 0 && te - t >= 2 * q) {
        int32_t r = kRowInf;
#pragma unroll 1
        for (int e = (int)lane; e < k.nd; e += 32) r = min(r, foot_repeat(g, t - __ldg(&k.dsp[e].x)));
        r = __reduce_min_sync(FULL, r);
        n = min(r, (int32_t)foot_div((uint32_t)(te - t), g.fq_m, g.fq_s));
        end = t + n * q;
      }
      int32_t from = t, stop = isolated ? min(end, t + (rows - ph)) : n > 1 ? t + q : end;
      const bool wrap = n > 1 && !isolated;
      bool prime = !(isolated && ph == 0);
      if (cut > 1u) {
        const uint32_t len = (uint32_t)(stop - t);
        from = t + (int32_t)(len * piece / cut);
        stop = t + (int32_t)(len * (piece + 1u) / cut);
        prime = prime || from > t;
      }
      if (from < stop) {
        const int32_t first = wrap && from == t ? t : kRowNone, last = wrap && stop == t + q ? stop : kRowNone;
        if (last != kRowNone) stop = last + 1;
        foot_merge_list(g, k, m, from, stop - from + 1);
        if (m.ld != 0) foot_walk(g, k, m, nl, from, stop, n, prime, first, last, out);
      }
      ph = 0;
      t = end;
    }
  }
  return out;
}

// Counters of a task's sectors and lines (wave loads, wave stores, block loads, block stores), and
// of the wave's loads' y and z lines and overlaps.
__constant__ uint32_t kFootDst[4] = {C_W_LS | C_W_LL << 8, C_W_SS | C_W_SL << 8, C_BLK_LS | C_BLK_LL << 8,
                                     C_BLK_SS | C_BLK_SL << 8};
constexpr uint32_t kFootDst3 = C_Y_LINES | C_Z_LINES << 8 | C_OV_Y << 16 | (uint32_t)C_OV_Z << 24;

// What the walk does not count of a field group, once per group: the wave's lattice updates, the
// valid address evaluations (threads of each level with all folded points valid and with fewer,
// at the domain's end) and the per-warp store sectors of the wave (the partial-store request
// volume).  The latter take a lane per thread row, in closed form.  A row's count depends on
// the store's address only modulo 32 bytes and on the first valid folded point it needs, so the
// group's stores that agree on both are counted together; and on the row only through its start
// modulo 32 bytes, t * B0 modulo 32 and the block run (whole, or cut at the wave's first or last
// block), so the warp keeps the counts it has by those.
__device__ __noinline__ void foot_stats(const EnumArgs &a, const DGroup &G, unsigned long long *cache, int part, int parts) {
  const uint32_t lane = threadIdx.x & 31u;
  const DCfg &c = a.cfg[G.cfg];
  unsigned long long *const cnt = (unsigned long long *)(a.counters + (int64_t)G.cfg * N_COUNTERS);
  if (part == 0) {
    const int32_t rest = c.fold_axis ? c.N[c.fold_axis] % c.fold : 0;
    // a lane per term, then a lane per (level, all or only partly valid threads)
    __syncwarp();
    if (lane < 24u) cache[lane] = (unsigned long long)foot_thread_term(c, (int)(lane % 12u), lane >= 12u);
    __syncwarp();
    unsigned long long th = 0;
    if (lane < 6u) {
      const uint32_t l = lane >> 1;
      for (uint32_t j = l == 0 ? 0u : l == 1 ? 2u : 6u; j < (l == 0 ? 2u : l == 1 ? 6u : 12u); ++j)
        th += cache[j + ((lane & 1u) ? 12u : 0u)];
    }
    __syncwarp();
    int32_t lf = 0, lp = 0, sf = 0, sp = 0;
    if ((int)lane < G.f_count) {
      const DField &f = a.fld[G.f_begin + (int)lane];
      lf = f.cnt_load[c.fold];
      sf = f.cnt_store[c.fold];
      lp = f.cnt_load[rest];
      sp = f.cnt_store[rest];
    }
    lf = __reduce_add_sync(FULL, lf);
    lp = __reduce_add_sync(FULL, lp);
    sf = __reduce_add_sync(FULL, sf);
    sp = __reduce_add_sync(FULL, sp);
    unsigned long long ad = 0, lups = 0;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const unsigned long long all = __shfl_sync(FULL, th, 2 * l), few = __shfl_sync(FULL, th, 2 * l + 1);
      ad += (all - few) * (unsigned long long)(lf + (l == 0 ? sf : 0)) +
            few * (unsigned long long)(lp + (l == 0 ? sp : 0));
      if (l == 0) lups = (all - few) * (unsigned long long)c.fold + few * (unsigned long long)rest;
    }
    if (lane == 0) {
      if (ad) atomicAdd(cnt + C_ADDR, ad);
      if (G.first_wave && lups) atomicAdd(cnt + C_LUPS_WAVE, lups);
    }
  }
  unsigned long long sum = 0;
  const DField &F0 = a.fld[G.f_begin];
  const int64_t es = F0.esize, sxe = es * F0.stride[0];
  const int32_t slots = (int32_t)c.rows_slot_end[0];
  const uint32_t gx = (uint32_t)c.g[0], gy = (uint32_t)c.g[1];
  const uint32_t py = (uint32_t)(es * F0.stride[1]) & 31u, pz = (uint32_t)(es * F0.stride[2]) & 31u;
  const uint32_t w0 = (uint32_t)c.s, w1 = (uint32_t)(c.s + c.weff);
  __syncwarp();
  for (int i = (int)lane; i < kFootRowCache; i += 32) cache[i] = ~0ull;
  __syncwarp();
  // the group's distinct (address modulo 32, first needed point) codes, a lane each, and how many
  // stores have them; taken through the rows when 32 might not hold more, and at the end
  uint32_t code = 0, times = 0;
  int nu = 0, k = 0, j0 = 0;   // codes held; next field and its next store
#pragma unroll 1
  for (;;) {
    // up to 32 stores: of one field, or of several in a row
    uint32_t mine = 0xffffffffu;
    int have = 0;
#pragma unroll 1
    while (k < G.f_count && have < 32) {
      const DField &F = a.fld[G.f_begin + k];
      const int take = min(32 - have, F.n_store - j0), at = (int)lane - have;
      if (at >= 0 && at < take) {
        const DAcc x = a.acc[F.acc_begin + F.n_load + j0 + at];
        mine = (uint32_t)((x.boff + F.base) & 31) | ((uint32_t)x.kmin << 5);
      }
      have += take;
      j0 += take;
      if (j0 >= F.n_store) {
        ++k;
        j0 = 0;
      }
    }
    const uint32_t same = __match_any_sync(FULL, mine);
    uint32_t todo = __ballot_sync(FULL, (int)lane < have && (int)lane == __ffs(same) - 1);
    if (have == 0 || nu + __popc(todo) > 32) {
      const int64_t n0 = ((int64_t)slots + 31) / 32;   // this part's rows, 32 at a time
      for (int32_t r = (int32_t)(n0 * part / parts); r < (int32_t)(n0 * (part + 1) / parts) && nu > 0; ++r) {
        const int32_t slot = 32 * r + (int32_t)lane;
        const uint32_t pq = fdiv((uint32_t)slot, c.fd_rows);
        const uint32_t t = (uint32_t)slot - pq * (uint32_t)c.rows_per_blk;
        const uint32_t R = (uint32_t)c.rows_R_lo[0] + pq;
        const uint32_t bz = fdiv(R, c.fd_gy), by = R - bz * gy, rb0 = R * gx;
        const uint32_t bxa = w0 > rb0 ? w0 - rb0 : 0u, bxb = min(w1 - rb0, gx);   // (a row of the wave: not empty)
        const uint32_t tz = fdiv(t, c.fd_b1), ty = t - tz * (uint32_t)c.B[1];
        int32_t y = (int32_t)(by * (uint32_t)c.B[1] + ty), z = (int32_t)(bz * (uint32_t)c.B[2] + tz);
        if (c.fold_axis == 1) y *= c.fold;
        if (c.fold_axis == 2) z *= c.fold;
        int kv = c.fold_axis == 1   ? min(c.fold, c.N[1] - y)
                 : c.fold_axis == 2 ? min(c.fold, c.N[2] - z)
                                    : 1;
        if (slot >= slots || y >= c.N[1] || z >= c.N[2]) kv = 0;
        const uint32_t a0 = py * (uint32_t)y + pz * (uint32_t)z;
        // one block run starts inside a block row, one ends inside one
        const uint32_t tag0 = (((t * (uint32_t)c.B[0]) & 31u) << 5) | (bxa > 0u ? 1u << 10 : 0u) | (bxb < gx ? 1u << 11 : 0u);
#pragma unroll 1
        for (int u = 0; u < nu; ++u) {
          const uint32_t cd = __shfl_sync(FULL, code, u), ct = __shfl_sync(FULL, times, u);
          if ((int32_t)(cd >> 5) >= kv) continue;
          const uint32_t A0 = (a0 + cd) & 31u, tag = tag0 | A0, at = (tag * 0x9E3779B1u) >> 26;
          const unsigned long long hit = cache[at];
          uint32_t val = (uint32_t)hit;
          if ((uint32_t)(hit >> 32) != tag) {
            val = (uint32_t)row_store_sectors_call((int64_t)A0, sxe, c.B[0], c.N[0], c.full_end, t, bxa, bxb);
            cache[at] = ((unsigned long long)tag << 32) | val;
          }
          sum += (unsigned long long)val * ct;
        }
        __syncwarp();
      }
      nu = 0;
      if (have == 0) break;
    }
#pragma unroll 1
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const uint32_t cd = __shfl_sync(FULL, mine, src), n = (uint32_t)__popc(__shfl_sync(FULL, same, src));
      const bool held = (int)lane < nu && code == cd;
      if (__any_sync(FULL, held)) {
        if (held) times += n;
      } else {
        if ((int)lane == nu) {
          code = cd;
          times = n;
        }
        ++nu;
      }
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
  if (lane == 0 && sum) atomicAdd(cnt + C_W_SREQ, sum);
}

// Geometry of a field group: the wave and its y and z sets, and the representative block.
__device__ __noinline__ void foot_setup(FootSmem &m, const DCfg &c, const DField &F) {
  const uint32_t lane = threadIdx.x & 31u;
  __syncwarp();
  const int32_t esx = (int32_t)(F.esize * F.stride[0]);
  if (lane < 6) foot_level(m.geo[lane < 3 ? 0 : 1], c, F.q, esx, lane >= 3, (int)(lane < 3 ? lane : lane - 3));
  __syncwarp();
  if (lane < 2) {
    FootGeo &g = m.geo[lane];
    foot_finish(g, c, F.q, esx);
    g.fq_m = F.fq_m;
    g.fq_s = F.fq_s;
  }
  __syncwarp();
}

// The tasks of a field, a lane each.
__device__ __noinline__ void foot_field(const EnumArgs &a, FootSmem &m, const DField &F, uint32_t foot) {
  const uint32_t lane = threadIdx.x & 31u;
  __syncwarp();
  if (lane < 4) {
    FootTask &k = m.task[lane];
    const bool st = lane & 1u, blk = lane >= 2u;
    const FootGeo &g = m.geo[lane >> 1];
    const int nd = st ? F.n_dsp_s : F.n_dsp_l;
    const int32_t P = (int32_t)(F.esize * F.stride[1]);
    k.nd = (foot & (blk ? 2u : 1u)) && (st ? F.mult_s : F.mult_l) ? nd : 0;
    if (k.nd > 0) {
      // the list is sorted by d; its first entry also holds the smallest clo, its second the
      // smallest displacement within a plane
      const int4 *const dsp = reinterpret_cast<const int4 *>(a.iv + F.iv_begin + F.n_iv + (st ? F.n_dsp_l : 0));
      const int4 d0 = __ldg(dsp), d1 = __ldg(dsp + (nd > 1 ? 1 : 0));
      const uint32_t pb = ((uint32_t)P * (uint32_t)g.q) & 127u;
      k.dsp = dsp;
      k.base = (uint32_t)(F.base + (int64_t)F.esize * (F.stride[1] * g.y0 + F.stride[2] * g.z0));
      k.P = P;
      k.hmin = d0.w;
      k.pzs = pb ? 8 - __ffs(pb) : 0;
      k.pz = 1 << k.pzs;
      k.ymin = nd > 1 ? d1.w : d0.x;
      // the displaced rows with points and the cell behind them
      k.rows = g.y_act + (st ? F.y_span_s : F.y_span_l) + 1;
      k.single = (int32_t)foot_div((uint32_t)(__ldg(&dsp[nd - 1].x) - d0.x), g.fq_m, g.fq_s) + 1;
      k.zmove = lane == 0 ? (int32_t)F.zmove - 1 : -1;
      foot_targets(g, lane == 0 ? 3 : 1, d0.x, __ldg(&dsp[nd - 1].x), k.zmove < 0, k.tr);
    }
  }
  __syncwarp();
}

// The closed-form items of a pass: warps take fchunk consecutive ones at a time (one, in plans of fewer
// than some 34,000 mixed candidates) and make a field group's geometry anew unless the item before was of
// the same one; before them each group's s_parts items for what the walk does not count.
__device__ __forceinline__ void foot_items(const EnumArgs &a, FootSmem &m) {
  const uint32_t lane = threadIdx.x & 31u;
  int cur = -1;
#pragma unroll 1
  for (;;) {
    unsigned long long i0 = 0;
    if (lane == 0) i0 = atomicAdd(a.fgrab, (unsigned long long)a.fchunk);
    const int64_t it0 = a.fitem_lo + (int64_t)__shfl_sync(FULL, i0, 0);
    const int64_t ns = a.sitem_hi - a.sitem_lo;
    const int64_t it_end = a.fitem_hi + ns;
    if (it0 >= it_end) break;
    const int64_t it1 = min(it0 + a.fchunk, it_end);
#pragma unroll 1
    for (int64_t it = it0; it < it1; ++it) {
      if (it < a.fitem_lo + ns) {
        const int64_t s = a.sitem_lo + (it - a.fitem_lo);
        const DGroup &G = a.grp[a.own_stat[s]];
        foot_stats(a, G, m.sreq, (int)(s - G.sitem_begin), G.s_parts);
        continue;
      }
      const int64_t itf = it - ns;
      const int gi = a.own_foot[itf];
      const DGroup &G = a.grp[gi];
      const int parts = G.f_parts, o = (int)(itf - G.fitem_begin), nth = o / parts, p = o - nth * parts;
      // the nth counted field of the group
      const uint32_t ff = G.foot_fields;
      const int k = __ffs(__ballot_sync(FULL, ((ff >> lane) & 1u) && __popc(ff & ((1u << lane) - 1u)) == nth)) - 1;
      const DField &F = a.fld[G.f_begin + k];
      if (gi != cur) {
        cur = gi;
        foot_setup(m, a.cfg[G.cfg], F);
      }
      foot_field(a, m, F, G.foot);
      const bool zs = F.zmove == 1;   // the z set's lines are the wave's
      unsigned long long *const cnt = (unsigned long long *)(a.counters + (int64_t)G.cfg * N_COUNTERS);
      // a task's units are shared out among the parts
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        int kind = i;   // not a constant: the walk's code, made once, has to stay in the instruction cache
        asm volatile("" : "+r"(kind));
        const bool st = kind & 1;
        if (m.task[kind].nd == 0) continue;
        // (the kinds' first parts, often the longest, fall to different warps)
        const int at = kind == 0 ? p : kind == 1 ? parts - 1 - p : p >= parts / 2 ? p - parts / 2 : p + parts - parts / 2;
        const FootCounts n = foot_task(m, kind, at, parts);
        // lane i adds the i-th count; the counters of each kind, a byte each
        const uint32_t v0 = __reduce_add_sync(FULL, n.sec), v1 = __reduce_add_sync(FULL, n.lin);
        uint32_t v = lane == 0 ? v0 : v1, dst = lane < 2 ? (kFootDst[kind] >> (8 * lane)) & 255u : 255u;
        if (kind == 0) {
          const uint32_t v2 = __reduce_add_sync(FULL, n.ylin), v3 = zs ? v1 : __reduce_add_sync(FULL, n.zlin);
          const uint32_t v4 = __reduce_add_sync(FULL, n.ovy), v5 = __reduce_add_sync(FULL, n.ovz);
          v = lane < 2 ? v : lane == 2 ? v2 : lane == 3 ? v3 : lane == 4 ? v4 : v5;
          if (lane >= 2 && lane < 6) dst = (uint32_t)(kFootDst3 >> (8 * (lane - 2))) & 255u;
        }
        if (dst != 255u && v) atomicAdd(cnt + dst, (unsigned long long)v * (st ? F.mult_s : F.mult_l));
      }
    }
  }
}

// Row items first (CTAs), then the closed-form items (warps).  Bound by latency: with the four warps a
// scheduler that 128 registers allow (3.3 to 3.6 active), issue slots are 32 to 42 % busy; per issue 2.5 warps
// wait for the ALU result before, 1.3 to 3.3 for an instruction fetch (a unit runs a few thousand instructions
// once) and 0.6 to 2.2 for memory (ncu: 755 25-point, 189 lattice Boltzmann, 400 mixed candidates).  So
// there is one copy of the walk and rare paths are out of line, and two CTAs an SM with 128 registers
// beat three or four that spill (0.23 against 0.29 and 0.35 ms, 25-point sweep of 755).  Footprints of 755 25-point candidates at 640 x 512 x 512: 0.193 ms of
// red.or and 0.092 ms of counting 179 MB of bitmaps -> 0.221 and 0.023 ms; 755 lattice Boltzmann
// candidates: 1.163 and 0.984 -> 0.229 and 0.002 ms (3.66 GB of bitmaps not read, fields that are
// whole-line copies counted once); 4,000 mixed candidates: 2.66 and 1.32 -> 1.89 and 0.08 ms.
// Without closed-form items the row walk has an instance of its own, 64 registers and four CTAs an
// SM: 755 25-point candidates with descending rows 0.287 -> 0.196 ms, 755 lattice Boltzmann ones whose
// planes are no whole number of rows apart 1.84 -> 1.46 ms.
template <bool kFoot>
__global__ void __launch_bounds__(256, kFoot ? 2 : 4) rows_kernel(EnumArgs a) {
  __shared__ DCfg s_c;
  __shared__ DGroup s_g;
  __shared__ DField s_fk[kMaxGroupFields];
  __shared__ int32_t s_loff[kMaxGroupFields + 1];
  __shared__ int32_t s_soff[kMaxGroupFields + 1];
  __shared__ int32_t s_ioff[kMaxGroupFields + 1];
  __shared__ int32_t s_idst[3][kMaxGroupFields];
  __shared__ int32_t s_cov[5];
  __shared__ uint8_t s_af[kMaxFoldedAccesses];
  __shared__ __align__(16) int64_t s_boff[kMaxFoldedAccesses];
  __shared__ uint8_t s_kmin[kMaxFoldedAccesses];
  __shared__ int32_t s_gad[2][17];
  __shared__ int32_t s_gwi[2];
  __shared__ long long s_item;
  __shared__ unsigned long long s_memo_key[kRowsThreads];       // per thread: last store-sector count
  __shared__ uint32_t s_memo_val[kRowsThreads];
  // per field of the staged group: bitmap word offsets, page-flag byte offsets, bitmap byte
  // sizes (block, wave), wave minus block origin and the stores' origin adjustment (block, wave)
  __shared__ int64_t s_fbm[kMaxGroupFields][N_BITMAPS];
  __shared__ int64_t s_fpg[kMaxGroupFields][N_BITMAPS];
  __shared__ int64_t s_flim[kMaxGroupFields][2];
  __shared__ int64_t s_fblk[kMaxGroupFields];
  __shared__ int64_t s_forg[kMaxGroupFields][2];
  __shared__ uint32_t s_fzc[kMaxGroupFields][2];                 // z-set clip window (sectors)
  __shared__ unsigned long long s_acc[kRowsThreads / 32][5];     // per warp: the item's counts
  __shared__ int s_batch;                                         // next batch of 32 slots of the item
  extern __shared__ __align__(16) unsigned char s_dyn[];
  const int iv_cap16 = (a.iv_cap + 15) & ~15;
  int64_t *const s_ibo = reinterpret_cast<int64_t *>(s_dyn);
  uint32_t *const s_iext = reinterpret_cast<uint32_t *>(s_dyn + 8 * iv_cap16);
  uint8_t *const s_iaf = s_dyn + 12 * iv_cap16;
  const StageSmem sm{&s_c, &s_g, s_fk, s_loff, s_soff, s_ioff, s_af, s_boff, nullptr, s_kmin, s_gad, s_gwi,
                     s_ibo, s_iext, s_iaf, s_idst, s_cov, nullptr};

  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = threadIdx.x >> 5;
  int cur_g = -1, cur_cfg = -1;

  for (;;) {
    if (threadIdx.x == 0) {
      s_item = a.ritem_lo + (long long)atomicAdd(a.rgrab, 1ull);
      s_batch = 0;
    }
    __syncthreads();
    const int64_t item = s_item;
    if (item >= a.ritem_hi) break;
    const int gi = a.own_rows[item];
    if (gi != cur_g) {
      stage_group(a, gi, cur_cfg, sm);
      cur_g = gi;
      cur_cfg = s_g.cfg;
      s_memo_key[threadIdx.x] = ~0ull;   // store-sector counts hold for one candidate's geometry
      for (int i = threadIdx.x; i < s_g.f_count * N_BITMAPS; i += blockDim.x) {
        const int k = i / N_BITMAPS, b = i - k * N_BITMAPS;
        const DField &F = s_fk[k];
        s_fbm[k][b] = F.bm[b];
        s_fpg[k][b] = 4 * F.pg + page_flag_off(b, F.words[0], F.words[1]);
        if (b < 2) {
          s_flim[k][b] = F.words[b] << 10;
          s_forg[k][b] = F.base - 32 * F.lo[b];
        }
        if (b == 0) {
          s_fblk[k] = 32 * (F.lo[1] - F.lo[0]);
          s_fzc[k][0] = F.zshift ? (uint32_t)F.zc_lo : 0u;
          s_fzc[k][1] = F.zshift ? (uint32_t)F.zc_hi : 0xffffffffu;
        }
      }
      __syncthreads();
    }
    const int64_t kk = item - s_g.ritem_begin;
    // ---- row walk of levels 1-3 and the block: every slot is one grid row of a level
    // (block run x thread row); each merged load run (raw loads when the row has fewer
    // valid folded points than the fold) is one sector range of the row, and stores also
    // add their per-warp sector counts in closed form.  A warp takes 32 slots at once, one
    // per lane, and each lane walks the runs and stores of its own row.
    // levels counted in closed form have no slots here
    const int64_t q0 = ((s_g.foot & 1) || !(s_g.levels & 2) ? s_c.rows_slot_end[2] : 0) + kk * (int64_t)a.chunk_rows;
    const int64_t q1 = min(q0 + (int64_t)a.chunk_rows, s_c.rows_slot_end[(s_g.levels & 1) && !(s_g.foot & 2) ? 3 : 2]);
    const int L = s_loff[s_g.f_count];
    const int S = s_soff[s_g.f_count] - L;
    const int Mfull = s_ioff[s_g.f_count];
    // runs [0, Mu) have no covering run; at rows inside their level (row_interior) only those
    // are taken, when they are at most half of all runs (otherwise the test of each row costs
    // more than the runs it saves: all runs are taken everywhere).  Runs [Muz, Mfull) are
    // covered from their own z row: at rows whose rows displaced in y alone lie inside the
    // level (a wave is often thinner in z than the z displacements) [0, Muz) are taken.
    const int Mu = 2 * s_cov[0] <= Mfull ? s_cov[0] : Mfull;
    const int Muz = s_cov[3];
    const DField &F0 = s_fk[0];
    const int64_t es = F0.esize, sxe = es * F0.stride[0];
    const int32_t faxis = s_c.fold_axis, fold = s_c.fold;
    uint32_t bad = 0, nred = 0;
    unsigned long long lups = 0, naddr = 0, sreq = 0;
    // the warps take the item's batches of 32 slots as they finish the previous one
    for (;;) {
      int bi = 0;
      if (lane == 0) bi = atomicAdd(&s_batch, 1);
      const int64_t b0 = q0 + 32 * (int64_t)__shfl_sync(FULL, bi, 0);
      if (b0 >= q1) break;
      // ---- decode: lane l takes slot b0 + l
      const int64_t slot = b0 + lane;
      bool ok = false;
      RowSlot r;
      if (slot < q1) {
        int lv;
        int64_t loc;
        if (slot < s_c.rows_slot_end[0]) {
          lv = 0; loc = slot;
        } else if (slot < s_c.rows_slot_end[1]) {
          lv = 1; loc = slot - s_c.rows_slot_end[0];
        } else if (slot < s_c.rows_slot_end[2]) {
          lv = 2; loc = slot - s_c.rows_slot_end[1];
        } else {
          lv = 3; loc = slot - s_c.rows_slot_end[2];   // the representative block's rows
        }
        const uint32_t pq = fdiv((uint32_t)loc, s_c.fd_rows);
        const uint32_t t = (uint32_t)loc - pq * (uint32_t)s_c.rows_per_blk;
        const uint32_t R = (uint32_t)s_c.rows_R_lo[lv] + pq;
        const uint32_t gx = (uint32_t)s_c.g[0], gy = (uint32_t)s_c.g[1];
        const uint32_t bz = fdiv(R, s_c.fd_gy), by = R - bz * gy;
        const int64_t rb0 = (int64_t)R * gx, rb1 = rb0 + gx;
        int64_t ba, bb;
        bool in = true;
        if (lv == 0) {
          ba = max(s_c.s, rb0);
          bb = min(s_c.s + s_c.weff, rb1);
        } else if (lv == 3) {
          ba = s_c.rep;
          bb = s_c.rep + 1;
        } else if (lv == 1) {
          in = by != gy - 1;
          ba = max(s_c.y_lo, rb0);
          bb = min(s_c.y_hi, rb1);
        } else {
          // z set minus the y set: the y set takes [y_lo, y_hi) outside the last block row,
          // and z_hi <= y_hi (both are the wave shifted back, the z set by a whole slab), so
          // only the blocks before y_lo remain in the other rows
          ba = max(s_c.z_lo, rb0);
          bb = min(s_c.z_hi, rb1);
          if (by != gy - 1 && s_c.y_hi > s_c.y_lo) bb = min(bb, s_c.y_lo);
        }
        const uint32_t tz = fdiv(t, s_c.fd_b1), ty = t - tz * (uint32_t)s_c.B[1];
        int32_t y = (int32_t)(by * (uint32_t)s_c.B[1] + ty), z = (int32_t)(bz * (uint32_t)s_c.B[2] + tz);
        if (faxis == 1) y *= fold;
        if (faxis == 2) z *= fold;
        if (in && ba < bb && y < s_c.N[1] && z < s_c.N[2]) {
          ok = true;
          r.bxa = (uint32_t)(ba - rb0);
          r.bxb = (uint32_t)(bb - rb0);
          const int32_t xa = (int32_t)r.bxa * s_c.B[0], xb = min((int32_t)r.bxb * s_c.B[0], s_c.N[0]);
          const int kv = faxis == 1 ? min(fold, s_c.N[1] - y) : faxis == 2 ? min(fold, s_c.N[2] - z) : 1;
          const int64_t nx = xb - xa;
          // the block level only fills the block bitmaps: its counts come from enum_kernel
          if (lv != 3) {
            if (lv == 0 && s_g.first_wave) lups += (unsigned long long)(nx * kv);
            naddr += (unsigned long long)(nx * s_gad[lv == 0 ? 0 : 1][kv]);
          }
          r.el0 = es * (F0.stride[1] * y + F0.stride[2] * z);
          const int64_t ea = r.el0 + sxe * xa, eb = r.el0 + sxe * (xb - 1);
          r.lo = min(ea, eb);
          r.hi = max(ea, eb);
          r.t = t;
          r.y = y;
          r.z = z;
          r.lv = (uint8_t)lv;
          r.kv = (uint8_t)kv;
        }
      }
      const bool full = ok && r.kv == fold;
      const bool inner = full && Mu < Mfull && row_interior(s_c, r.lv, r.y, r.z, r.bxa, r.bxb, s_cov[1], s_cov[2]);
      const bool inner_y = full && !inner && Muz < Mfull && row_interior(s_c, r.lv, r.y, r.z, r.bxa, r.bxb, s_cov[4], 0);
      const bool blk = r.lv == 3;
      const int bsel = r.lv == 0 ? BM_W : r.lv == 1 ? BM_Y : r.lv == 2 ? BM_Z : BM_BL;
      // ---- loads of a full-fold row: its merged runs, [0, Mu) when it lies inside its level.
      // The lanes walk the same run at the same time (broadcast shared-memory reads); a lane
      // keeps its field's bitmap pointers, merges consecutive runs that end in one 64-bit
      // unit into one red.or, and stores a page flag only when the page range moves.  The
      // z-set ranges of a field whose z set is the wave moved by whole lines are clipped to
      // the wave's address range: the counts take only their sectors that meet the wave.
      if (__any_sync(FULL, full)) {
        const int me = !full ? 0 : inner ? Mu : inner_y ? Muz : Mfull;
        int kc = -1;
        unsigned long long *bm = nullptr;
        uint8_t *fl = nullptr;
        int64_t lim = 0, fb = 0;
        uint32_t cu = 0xffffffffu, pl0 = 1u, pl1 = 0u, zlo = 0u, zhi = 0xffffffffu;
        unsigned long long cb = 0ull;
        for (int e = 0; e < me; ++e) {
          const int k = s_iaf[e];
          if (k != kc) {
            if (cb) {
              atomicOr(bm + cu, cb);
              ++nred;
            }
            cu = 0xffffffffu;
            cb = 0ull;
            kc = k;
            bm = reinterpret_cast<unsigned long long *>(a.scratch + s_fbm[k][bsel]);
            fl = reinterpret_cast<uint8_t *>(a.scratch) + s_fpg[k][bsel];
            lim = s_flim[k][blk ? 0 : 1];
            fb = blk ? s_fblk[k] : 0;   // staged offsets are relative to the wave origin
            pl0 = 1u;
            pl1 = 0u;
            zlo = r.lv == 2 ? s_fzc[k][0] : 0u;
            zhi = r.lv == 2 ? s_fzc[k][1] : 0xffffffffu;
          }
          const int64_t bo = s_ibo[e] + fb;
          const int64_t a0 = r.lo + bo, a1 = r.hi + bo + (int64_t)s_iext[e];
          if (a0 < 0 || a1 >= lim) {
            ++bad;
            continue;
          }
          const uint32_t s0 = max((uint32_t)(a0 >> 5), zlo), s1 = min((uint32_t)(a1 >> 5), zhi);
          if (s0 > s1) continue;
          nred += put_range(bm, cu, cb, s0, s1);
          constexpr int kPageShiftSectors = kPageShiftBytes - 5;
          const uint32_t p0 = s0 >> kPageShiftSectors, p1 = s1 >> kPageShiftSectors;
          if (p0 < pl0 || p1 > pl1) {
            flag_pages(fl, p0, p1);
            pl0 = p0;
            pl1 = p1;
          }
        }
        if (cb) {
          atomicOr(bm + cu, cb);
          ++nred;
        }
      }
      // ---- loads of rows with fewer valid folded points than the fold (domain edge): the
      // raw folded loads, each issued iff a valid point needs it
      if (__any_sync(FULL, ok && !full)) {
        if (ok && !full) {
          for (int e = 0; e < L; ++e) {
            if ((int)s_kmin[e] >= r.kv) continue;
            const int k = s_af[e];
            const int64_t bo = s_boff[e] + s_forg[k][blk ? 0 : 1];
            const int64_t a0 = r.lo + bo, a1 = r.hi + bo;
            if (a0 < 0 || a1 >= s_flim[k][blk ? 0 : 1]) {
              ++bad;
              continue;
            }
            unsigned long long *const bm = reinterpret_cast<unsigned long long *>(a.scratch + s_fbm[k][bsel]);
            uint32_t cu = 0xffffffffu;
            unsigned long long cb = 0ull;
            nred += put_range(bm, cu, cb, (uint32_t)(a0 >> 5), (uint32_t)(a1 >> 5)) + (cb ? 1u : 0u);
            if (cb) atomicOr(bm + cu, cb);
            flag_pages(reinterpret_cast<uint8_t *>(a.scratch) + s_fpg[k][bsel], (uint32_t)(a0 >> kPageShiftBytes),
                       (uint32_t)(a1 >> kPageShiftBytes));
          }
        }
      }
      // ---- stores of wave and block rows; wave rows add their per-warp store sectors
      const bool st = ok && (r.lv == 0 || r.lv == 3) && S > 0;
      if (__any_sync(FULL, st)) {
        if (st) {
          const int sb = blk ? BM_BS : BM_WS;
          for (int j = L; j < L + S; ++j) {
            if ((int)s_kmin[j] >= r.kv) continue;
            const int k = s_af[j];
            const int64_t bo = s_boff[j] + s_forg[k][blk ? 0 : 1];
            const int64_t a0 = r.lo + bo, a1 = r.hi + bo;
            if (a0 < 0 || a1 >= s_flim[k][blk ? 0 : 1]) {
              ++bad;
              continue;
            }
            unsigned long long *const bm = reinterpret_cast<unsigned long long *>(a.scratch + s_fbm[k][sb]);
            uint32_t cu = 0xffffffffu;
            unsigned long long cb = 0ull;
            nred += put_range(bm, cu, cb, (uint32_t)(a0 >> 5), (uint32_t)(a1 >> 5)) + (cb ? 1u : 0u);
            if (cb) atomicOr(bm + cu, cb);
            flag_pages(reinterpret_cast<uint8_t *>(a.scratch) + s_fpg[k][sb], (uint32_t)(a0 >> kPageShiftBytes),
                       (uint32_t)(a1 >> kPageShiftBytes));
            if (!blk) {
              // the count depends on the row start only modulo 32 bytes, on t only through
              // t * B0 modulo 32 (where the row's first warp ends) and on the block run, so
              // rows that agree on those reuse this thread's previous count
              const int64_t A0 = r.el0 + bo;
              const unsigned long long key = (unsigned long long)(A0 & 31) |
                                             ((unsigned long long)((r.t * (uint32_t)s_c.B[0]) & 31u) << 5) |
                                             ((unsigned long long)r.bxa << 10) | ((unsigned long long)r.bxb << 37);
              if (s_memo_key[threadIdx.x] != key) {
                if constexpr (kFoot)
                  s_memo_val[threadIdx.x] =
                      (uint32_t)row_store_sectors_call(A0, sxe, s_c.B[0], s_c.N[0], s_c.full_end, r.t, r.bxa, r.bxb);
                else
                  s_memo_val[threadIdx.x] =
                      (uint32_t)row_store_sectors(A0, sxe, s_c.B[0], s_c.N[0], s_c.full_end, r.t, r.bxa, r.bxb);
                s_memo_key[threadIdx.x] = key;
              }
              sreq += s_memo_val[threadIdx.x];
            }
          }
        }
      }
    }

    // the item's counts: per warp, then once per CTA
    bad = __reduce_add_sync(FULL, bad);
    nred = __reduce_add_sync(FULL, nred);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      lups += __shfl_xor_sync(FULL, lups, o);
      naddr += __shfl_xor_sync(FULL, naddr, o);
      sreq += __shfl_xor_sync(FULL, sreq, o);
    }
    if (lane == 0) {
      s_acc[warp][0] = lups;
      s_acc[warp][1] = naddr;
      s_acc[warp][2] = sreq;
      s_acc[warp][3] = bad;
      s_acc[warp][4] = nred;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
      const int k = threadIdx.x;
      unsigned long long v = 0;
      for (int w = 0; w < kRowsThreads / 32; ++w) v += s_acc[w][k];
      unsigned long long *const c = (unsigned long long *)(a.counters + (int64_t)s_g.cfg * N_COUNTERS);
      const int dst = k == 0 ? C_LUPS_WAVE : k == 1 ? C_ADDR : k == 2 ? C_W_SREQ : k == 3 ? C_OVERFLOW : C_RED;
      if (v) atomicAdd(c + dst, v);
    }
  }
  // then the closed-form items, a warp each, their state in the room of the row walk's access
  // offsets (every warp has passed the last item's barriers)
  static_assert(sizeof(FootSmem) * (kRowsThreads / 32) <= sizeof(s_boff) && alignof(FootSmem) <= 16, "FootSmem in s_boff");
  if constexpr (kFoot) foot_items(a, reinterpret_cast<FootSmem *>(s_boff)[threadIdx.x >> 5]);
}

__constant__ int kCountDst[12] = {C_BLK_LS, C_BLK_LL, C_BLK_SS, C_BLK_SL, C_W_LS, C_W_LL,
                                  C_Y_LINES, C_Z_LINES, C_OV_Y, C_OV_Z, C_W_SS, C_W_SL};

// Lines of four consecutive bitmap words: bit i of a word <-> sector lo + i with lo a
// multiple of 32, so each nibble is one 128 B line; a word's nibbles are reduced to one bit
// each (bit 4k) and the four words' bits interleaved into one word for a single popcount.
__device__ __forceinline__ uint32_t line_bits(uint32_t x) {
  uint32_t t = x | (x >> 1);
  t |= t >> 2;
  return t & 0x11111111u;
}
__device__ __forceinline__ uint32_t lines4(const uint4 &v) {
  return __popc(line_bits(v.x) | (line_bits(v.y) << 1) | (line_bits(v.z) << 2) | (line_bits(v.w) << 3));
}

__device__ __forceinline__ bool nz(const uint4 &v) { return (v.x | v.y | v.z | v.w) != 0u; }

__device__ __forceinline__ void tally_sectors_lines(uint32_t &sec, uint32_t &lin, const uint4 &v) {
  sec += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
  lin += lines4(v);
}

// zs: the z set is the wave moved by whole lines (its bitmap holds only the sectors that can
// meet the wave), so its lines are the wave's
__device__ __forceinline__ void tally_wave(uint32_t acc[12], const uint4 &w, const uint4 &y, const uint4 &z, bool zs) {
  tally_sectors_lines(acc[4], acc[5], w);
  acc[6] += lines4(y);
  acc[7] += lines4(zs ? w : z);
  acc[8] += __popc(w.x & y.x) + __popc(w.y & y.y) + __popc(w.z & y.z) + __popc(w.w & y.w);
  acc[9] += __popc(w.x & z.x & ~y.x) + __popc(w.y & z.y & ~y.y) + __popc(w.z & z.z & ~y.z) + __popc(w.w & z.w & ~y.w);
}

// Read-and-clear counting of the bitmaps of one pass.  Counting unit = (field, chunk of the
// words of its block bitmaps or of its wave bitmaps); work item = consecutive units of one
// candidate (at most kCountMaxPages pages, kCountItemUnits units), so that a CTA places the
// many small block parts of a large batch together.  Chunks are cut into pages of
// kPageWords words; for a field the row walk filled, only the pages it flagged are read
// (and their flags cleared), otherwise every page.  One warp takes one page at a time: each
// lane loads two 16-byte positions of every bitmap of the part that has the page flagged
// (all loads in flight together), tallies sectors, lines and overlaps, and clears the
// non-zero positions, so the bitmaps are left zeroed for the next step.
__device__ __forceinline__ uint4 ld_v4(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

__global__ void __launch_bounds__(kCountThreads, 4) count_kernel(CountArgs a) {
  __shared__ long long s_item[2];   // this item and the next one (fetched while this one is counted)
  __shared__ uint32_t s_red[kCountThreads / 32][13];
  __shared__ uint32_t s_pl[kCountMaxPages];        // pages to read: bitmap mask | unit << 4 | page << 12
  __shared__ int s_npl;
  // the item's units: bitmap positions (16-byte units), their flags, first item page
  __shared__ uint4 *s_ubp[kCountItemUnits][4];
  __shared__ uint8_t *s_ufl[kCountItemUnits][4];
  __shared__ int64_t s_uq0[kCountItemUnits];       // first 16-byte position of the chunk
  __shared__ int64_t s_uq1[kCountItemUnits];       // end position of the chunk
  __shared__ int32_t s_uw[kCountItemUnits];        // words of the chunk
  __shared__ int32_t s_upg[kCountItemUnits + 1];   // first item page of each unit, then the end
  __shared__ uint8_t s_unb[kCountItemUnits];       // bitmaps of the part (2 block, 4 wave)
  __shared__ uint8_t s_uzs[kCountItemUnits];       // the field's z set is its wave moved by whole lines
  __shared__ int s_cfg;
  const uint32_t lane = threadIdx.x & 31u;
  const int warp = threadIdx.x >> 5;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) {
    s_item[0] = a.citem_lo + (long long)atomicAdd(a.grab, 1ull);
    s_npl = 0;
  }
  __syncthreads();
  for (int par = 0;; par ^= 1) {
    const int64_t item = s_item[par];
    if (item >= a.citem_hi) break;
    long long nxt = 0;
    if (threadIdx.x == 0) nxt = a.citem_lo + (long long)atomicAdd(a.grab, 1ull);
    const int u0 = a.item_unit[item], nu = a.item_unit[item + 1] - u0;
    // ---- a thread per unit: where its chunk's bitmaps and flags lie
    if (threadIdx.x < nu) {
      const int t = threadIdx.x;
      const int cf = a.units[2 * (u0 + t)];
      const int64_t k = a.units[2 * (u0 + t) + 1];
      const DField &F = a.fld[cf];
      const bool paged = F.pg >= 0;
      const int64_t cw = paged ? kPagedChunkWords : a.chunk_words;
      const int64_t kb = (F.words[0] + cw - 1) / cw;
      const bool blk = k < kb;
      const int64_t c0 = (blk ? k : k - kb) * cw;
      const int64_t c1 = min(c0 + cw, blk ? F.words[0] : F.words[1]);
      const int NB = blk ? 2 : 4;
      const int b0 = blk ? BM_BL : BM_W;   // BL, BS | W, Y, Z, WS are consecutive bitmap indices
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const bool has = b < NB && F.bm[b0 + b] >= 0;
        s_ubp[t][b] = has ? reinterpret_cast<uint4 *>(a.scratch + F.bm[b0 + b]) : nullptr;
        s_ufl[t][b] = has && paged ? reinterpret_cast<uint8_t *>(a.scratch + F.pg) +
                                         page_flag_off(b0 + b, F.words[0], F.words[1]) + c0 / kPageWords
                                   : nullptr;
      }
      s_uq0[t] = c0 / 4;
      s_uq1[t] = c1 / 4;
      s_uw[t] = (int32_t)(c1 - c0);
      s_upg[t + 1] = (int32_t)((c1 - c0 + kPageWords - 1) / kPageWords);
      s_unb[t] = (uint8_t)NB;
      s_uzs[t] = (uint8_t)(F.zshift != 0);
      if (t == 0) {
        s_cfg = F.cfg;
        s_upg[0] = 0;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int t = 0; t < nu; ++t) s_upg[t + 1] += s_upg[t];
    __syncthreads();
    const int npg = s_upg[nu];
    uint32_t rd = 0;   // bitmap bytes of the pages this thread lists
    // ---- a thread per page: which bitmaps to read (flags cleared in device memory as they
    // are taken); pages with none are dropped
    for (int j = threadIdx.x; j < npg; j += kCountThreads) {
      int lo = 0, hi = nu - 1;   // the unit holding page j: s_upg[u] <= j < s_upg[u + 1]
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_upg[mid] <= j) lo = mid;
        else hi = mid - 1;
      }
      const int u = lo, lp = j - s_upg[u];
      const uint32_t pbytes = 4u * (uint32_t)min(kPageWords, s_uw[u] - lp * kPageWords);
      uint32_t m = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if (s_ubp[u][b] == nullptr) continue;
        bool on = true;
        uint8_t *const fl = s_ufl[u][b];
        if (fl != nullptr) {
          const uint8_t v = fl[lp];
          if (v) fl[lp] = 0;
          on = v != 0;
        }
        if (on) {
          m |= 1u << b;
          rd += pbytes;
        }
      }
      if (m) s_pl[atomicAdd(&s_npl, 1)] = m | ((uint32_t)u << 4) | ((uint32_t)lp << 12);
    }
    __syncthreads();
    uint32_t acc[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    const int npl = s_npl;
    for (int i = warp; i < npl; i += kCountThreads / 32) {
      const uint32_t ent = s_pl[i];
      const uint32_t m = ent & 15u;
      const int u = (int)((ent >> 4) & 255u), lp = (int)(ent >> 12);
      const bool blk = s_unb[u] == 2, zs = s_uzs[u] != 0;
      uint4 *const *const bp = s_ubp[u];
      const int64_t q0 = s_uq0[u] + (int64_t)lp * (kPageWords / 4);           // first position of the page
      const int np = (int)min((int64_t)(kPageWords / 4), s_uq1[u] - q0);      // its positions (<= 64)
      uint4 v[4][2];
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = (int)lane + 32 * h;
          v[b][h] = ((m >> b) & 1u) && r < np ? ld_v4(bp[b] + q0 + r) : zero;
        }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t q = q0 + (int)lane + 32 * h;
        if (blk) {
          if (nz(v[0][h])) {
            tally_sectors_lines(acc[0], acc[1], v[0][h]);
            bp[0][q] = zero;
          }
          if (nz(v[1][h])) {
            tally_sectors_lines(acc[2], acc[3], v[1][h]);
            bp[1][q] = zero;
          }
        } else {
          if (nz(v[0][h]) | nz(v[1][h]) | nz(v[2][h])) {
            tally_wave(acc, v[0][h], v[1][h], v[2][h], zs);
#pragma unroll
            for (int b = 0; b < 3; ++b)
              if (nz(v[b][h])) bp[b][q] = zero;
          }
          if (nz(v[3][h])) {
            tally_sectors_lines(acc[10], acc[11], v[3][h]);
            bp[3][q] = zero;
          }
        }
      }
    }
#pragma unroll
    for (int kk = 0; kk < 12; ++kk) {
      uint32_t v = __reduce_add_sync(FULL, acc[kk]);
      if (lane == 0) s_red[warp][kk] = v;
    }
    {
      const uint32_t v = __reduce_add_sync(FULL, rd);
      if (lane == 0) s_red[warp][12] = v;
    }
    __syncthreads();
    if (threadIdx.x < 13) {
      unsigned long long t = 0;
      for (int wi = 0; wi < kCountThreads / 32; ++wi) t += s_red[wi][threadIdx.x];
      const int dst = threadIdx.x < 12 ? kCountDst[threadIdx.x] : C_CBYTES;
      if (t) atomicAdd((unsigned long long *)(a.counters + (int64_t)s_cfg * N_COUNTERS + dst), t);
    }
    if (threadIdx.x == 0) {
      s_item[par ^ 1] = nxt;
      s_npl = 0;
    }
    __syncthreads();
  }
}

// R(O) = a * exp(-b * exp(-c * O)), Sec. 4.5
__device__ __forceinline__ double rhat_dev(const double h[3], double O) {
  return __dmul_rn(h[0], exp(-__dmul_rn(h[1], exp(-__dmul_rn(h[2], O)))));
}

__device__ double rank_key_dev(double t) {
  if (!(t > 0.0) || isinf(t)) return t;
  int e = 0;
  double m = frexp(t, &e);
  return ldexp(rint(ldexp(m, 40)), e - 40);
}

// The capacity model and the four limiters.  Products and quotients use explicit
// round-to-nearest intrinsics so that no multiply-add is fused and the evaluation order is the
// one written here.  Four lanes per candidate: the model is bound by the latency of its fp64 chain (a division takes
// some 40 dependent operations, the unit one of a warp every 16 cycles), and most of its terms do
// not depend on one another.  Each division below is up to four, and each lane takes one of the
// four hit rates; every value is computed with the operations and in the order of the formula.
// One thread per candidate: 20.5 us for 755 candidates, four lanes 12.3 (GB300; 20,000 candidates,
// where the fp64 units are full, 27 -> 41 us of a step of some 10 ms).
__global__ void __launch_bounds__(32) model_kernel(ModelArgs a) {
  const uint32_t lane = threadIdx.x, q = lane & 3u;
  const int at = (int)(blockIdx.x * 8u + (lane >> 2)), i = min(at, a.n - 1);
  const DCfg &C = a.cfg[i];
  const int64_t *c = a.counters + (int64_t)i * N_COUNTERS;
  ws_result r;
  memset(&r, 0, sizeof(r));
  r.status = C.status;
  if (r.status == WS_OK && c[C_OVERFLOW] != 0) r.status = WS_EOVERFLOW;
  r.lups_block = c[C_LUPS_BLOCK];
  r.lups_wave = c[C_LUPS_WAVE];
  r.l1_req_sectors = c[C_L1_REQ];
  r.l1_bank_cycles = c[C_BANK];
  r.l1_store_sectors = c[C_L1_STORE];
  r.blk_load_sectors = c[C_BLK_LS];
  r.blk_load_lines = c[C_BLK_LL];
  r.blk_store_sectors = c[C_BLK_SS];
  r.blk_store_lines = c[C_BLK_SL];
  r.wave_load_sectors = c[C_W_LS];
  r.wave_load_lines = c[C_W_LL];
  r.wave_store_sectors = c[C_W_SS];
  r.wave_store_lines = c[C_W_SL];
  r.wave_store_req_sectors = c[C_W_SREQ];
  r.ov_y = c[C_OV_Y];
  r.ov_z = c[C_OV_Z];
  r.y_lines = c[C_Y_LINES];
  r.z_lines = c[C_Z_LINES];
  r.wave_blocks = C.weff;
  r.wave_first_block = C.s;
  r.y_dist_blocks = C.y_dist;
  r.z_dist_blocks = C.z_dist;
  r.blocks_per_sm = C.bpsm;

  const DHw &h = a.hw;
  const double lb = (double)r.lups_block, lw = (double)r.lups_wave;
  auto of_lane = [&](double v, uint32_t k) { return __shfl_sync(FULL, v, (int)((lane & ~3u) + k)); };
  auto mine = [&](double v0, double v1, double v2, double v3) { return q == 0 ? v0 : q == 1 ? v1 : q == 2 ? v2 : v3; };
  auto bytes = [](double unit, int64_t n) { return __dmul_rn(unit, (double)n); };
  // L1 <-> L2: requests per instruction are V_up (v_l1), the block footprint is V_comp.  [v_l1,
  // wave lines per block, the same, v_l2_store]
  const double d0 = __ddiv_rn(q == 0   ? bytes(32.0, r.l1_req_sectors)
                              : q == 3 ? bytes(32.0, r.l1_store_sectors)
                                       : bytes(128.0, r.wave_load_lines),
                              q == 1 || q == 2 ? (double)C.weff : lb);
  // oversubscription of L1 by the blocks, of L2 by the y and z layers and by the stores
  const double o = __ddiv_rn(q == 0   ? __dmul_rn(bytes(128.0, r.blk_load_lines), (double)C.bpsm)
                             : q == 3 ? bytes(128.0, r.wave_store_lines)
                                      : __dmul_rn((double)(q == 1 ? C.y_dist : C.z_dist), d0),
                             q == 0 ? h.l1_bytes : h.l2_bytes);
  const double rate = h.capacity_model != 0 ? rhat_dev(h.hit[q], o) : 1.0;
  // [v_comp, v_dcomp, v_red, v_dram_store]
  const double d1 = __ddiv_rn(bytes(32.0, q == 0   ? r.blk_load_sectors
                                          : q == 1 ? r.wave_load_sectors
                                          : q == 2 ? r.wave_store_req_sectors - r.wave_store_sectors
                                                   : r.wave_store_sectors),
                              q == 0 ? lb : lw);
  // DRAM <-> L2: wave footprint minus layer-condition reuse plus partial-store reads.  [bank cycles
  // per LUP, layer hits, t_fp]
  const double r_y = of_lane(rate, 1), r_z = of_lane(rate, 2);
  const bool fp = C.flops > 0.0 && h.fp_peak > 0.0;
  const double d2 = __ddiv_rn(mine((double)r.l1_bank_cycles,
                                   __dadd_rn(__dmul_rn(r_y, bytes(32.0, r.ov_y)), __dmul_rn(r_z, bytes(32.0, r.ov_z))),
                                   fp ? C.flops : 0.0, 0.0),
                              mine(lb, lw, fp ? h.fp_peak : 1.0, 1.0));
  const double r_l1 = of_lane(rate, 0), r_st = of_lane(rate, 3), v_comp = of_lane(d1, 0), v_dcomp = of_lane(d1, 1),
               v_red = of_lane(d1, 2);
  r.v_l1 = of_lane(d0, 0);
  r.v_l2_store = of_lane(d0, 3);
  r.o_l1 = of_lane(o, 0);
  r.o_y = of_lane(o, 1);
  r.o_z = of_lane(o, 2);
  r.o_st = of_lane(o, 3);
  r.v_dram_store = of_lane(d1, 3);
  r.v_l2_load = __dadd_rn(v_comp, __dmul_rn(__dsub_rn(1.0, r_l1), __dsub_rn(r.v_l1, v_comp)));
  r.v_dram_load = __dadd_rn(__dsub_rn(v_dcomp, of_lane(d2, 1)), __dmul_rn(__dsub_rn(1.0, r_st), v_red));
  // limiters: seconds per LUP for the whole GPU
  const double d3 = __ddiv_rn(mine(d2, __dadd_rn(r.v_l2_load, r.v_l2_store), __dadd_rn(r.v_dram_load, r.v_dram_store), 0.0),
                              mine(__dmul_rn(h.clock_hz, (double)h.sms), h.bw_l2, h.bw_dram, 1.0));
  r.t_l1 = of_lane(d3, 0);
  r.t_l2 = of_lane(d3, 1);
  r.t_dram = of_lane(d3, 2);
  r.t_fp = of_lane(d2, 2);
  if (q != 0 || at >= a.n) return;
  a.rank[i] = 0;
  if (r.status != WS_OK) {
    const int32_t status = r.status;
    memset(&r, 0, sizeof(r));
    r.status = status;
    r.t_pred = __longlong_as_double(0x7ff0000000000000ll);
    r.glups = 0.0;
    a.results[i] = r;
    a.keys[i] = r.t_pred;
    return;
  }
  double best = r.t_l1;
  int lim = WS_LIMITER_L1;
  if (r.t_l2 > best) { best = r.t_l2; lim = WS_LIMITER_L2; }
  if (r.t_dram > best) { best = r.t_dram; lim = WS_LIMITER_DRAM; }
  if (r.t_fp > best) { best = r.t_fp; lim = WS_LIMITER_FP; }
  r.t_pred = best;
  r.limiter = lim;
  r.glups = __ddiv_rn(1e-9, best);
  a.results[i] = r;
  a.keys[i] = rank_key_dev(best);
}

// Stable rank within segments: rank(i) = #{j in seg : key_j < key_i or
// (key_j == key_i and j < i)}; NaN counts as +inf.  order[seg_begin + rank(i)] = i.
// Block (x, y) compares its kRankTile candidates with the y-th tile of kRankTile keys of
// their segments and adds the partial counts to rank[i] (zeroed by the kernel that made the keys,
// which saves a memset between them: 11 -> 9 us of ranking); the scatter
// kernel then places every candidate.
constexpr int kRankTile = 256;

__device__ __forceinline__ int rank_seg_of(const RankArgs &a, int64_t x) {
  int lo = 0, hi = a.n_seg;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.seg[mid] <= x) lo = mid;
    else hi = mid;
  }
  return lo;
}

// The rank keys as integers in the same order as the doubles they stand for (NaN
// counts as +inf, -0 as +0): a sign-magnitude bit pattern maps monotonically to two's
// complement by flipping the magnitude bits of negative values.  Integer compares keep
// the ranking off the fp64 pipe.
__device__ __forceinline__ long long rank_ord_of(double v) {
  long long b = isnan(v) ? 0x7ff0000000000000ll : __double_as_longlong(v);
  if ((b << 1) == 0) b = 0;
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

__global__ void __launch_bounds__(kRankTile) rank_count_kernel(RankArgs a) {
  __shared__ long long s_key[kRankTile];
  const int64_t i_first = (int64_t)blockIdx.x * kRankTile;
  if (i_first >= a.n) return;
  const int64_t i = i_first + threadIdx.x;
  const int64_t i_last = min((int64_t)a.n, i_first + kRankTile) - 1;
  const int64_t j_lo = a.seg[rank_seg_of(a, i_first)], j_hi = a.seg[rank_seg_of(a, i_last) + 1];
  const int64_t t0 = j_lo + (int64_t)blockIdx.y * kRankTile;
  if (t0 >= j_hi) return;
  if (t0 + threadIdx.x < j_hi) s_key[threadIdx.x] = rank_ord_of(a.keys[t0 + threadIdx.x]);
  __syncthreads();
  if (i >= a.n) return;
  const int my_seg = rank_seg_of(a, i);
  const int64_t a0 = max(t0, (int64_t)a.seg[my_seg]), a1 = min(t0 + kRankTile, (int64_t)a.seg[my_seg + 1]);
  const long long ki = rank_ord_of(a.keys[i]);
  int cnt = 0;
  for (int64_t j = a0; j < a1; ++j) {
    const long long kj = s_key[j - t0];
    cnt += (kj < ki) || (kj == ki && j < i);
  }
  if (cnt) atomicAdd(a.rank + i, cnt);
}

__global__ void rank_scatter_kernel(RankArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  a.order[a.seg[rank_seg_of(a, i)] + a.rank[i]] = (int32_t)i;
}

// Rank keys of given results (used when ranking results that came from the host).
__global__ void keys_kernel(const ws_result *__restrict__ res, int n, double *__restrict__ keys,
                            int32_t *__restrict__ rank) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = rank_key_dev(res[i].t_pred);
  rank[i] = 0;
}

// ---- launchers ---------------------------------------------------------------------
size_t enum_dyn_smem(int iv_cap) { return (size_t)((iv_cap + 15) & ~15) * (8 + 4 + 1); }

// Raises the dynamic shared-memory limit of the enumeration and row kernels (once per
// device and size).
static cudaError_t enum_allow_smem(size_t dyn) {
  static std::mutex mu;
  static size_t allowed[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> g(mu);
  if (dyn <= allowed[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(enum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  for (auto *rows : {rows_kernel<false>, rows_kernel<true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  if (e == cudaSuccess) allowed[dev] = dyn;
  return e;
}

cudaError_t launch_enum(const EnumArgs &args, int grid, int threads, cudaStream_t st) {
  const size_t dyn = enum_dyn_smem(args.iv_cap);
  cudaError_t e = enum_allow_smem(dyn);
  if (e != cudaSuccess) return e;
  enum_kernel<<<grid, threads, dyn, st>>>(args);
  return cudaGetLastError();
}
cudaError_t launch_rows(const EnumArgs &args, int grid, cudaStream_t st) {
  const size_t dyn = enum_dyn_smem(args.iv_cap);
  cudaError_t e = enum_allow_smem(dyn);
  if (e != cudaSuccess) return e;
  if (args.fitem_hi > args.fitem_lo) rows_kernel<true><<<grid, kRowsThreads, dyn, st>>>(args);
  else rows_kernel<false><<<grid, kRowsThreads, dyn, st>>>(args);
  return cudaGetLastError();
}
cudaError_t launch_count(const CountArgs &args, int grid, cudaStream_t st) {
  count_kernel<<<grid, kCountThreads, 0, st>>>(args);
  return cudaGetLastError();
}
cudaError_t launch_model(const ModelArgs &args, cudaStream_t st) {
  if (args.n <= 0) return cudaSuccess;
  // one warp per CTA, eight candidates each: the model is fp64 (1/64 of the fp32 rate on this
  // part), so the candidates are spread over as many SMs' fp64 pipes as possible
  model_kernel<<<(args.n + 7) / 8, 32, 0, st>>>(args);
  return cudaGetLastError();
}
cudaError_t launch_rank(const RankArgs &args, cudaStream_t st) {
  if (args.n <= 0) return cudaSuccess;
  const unsigned tiles = (unsigned)((args.n + kRankTile - 1) / kRankTile);
  rank_count_kernel<<<dim3(tiles, tiles), kRankTile, 0, st>>>(args);
  rank_scatter_kernel<<<tiles, kRankTile, 0, st>>>(args);
  return cudaGetLastError();
}
cudaError_t launch_keys(const ws_result *res, int n, double *keys, int32_t *rank, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  keys_kernel<<<(n + 255) / 256, 256, 0, st>>>(res, n, keys, rank);
  return cudaGetLastError();
}
cudaError_t enum_occupancy(int threads, int iv_cap, int *blocks_per_sm) {
  const size_t dyn = enum_dyn_smem(iv_cap);
  cudaError_t e = enum_allow_smem(dyn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, enum_kernel, threads, dyn);
}
cudaError_t rows_occupancy(int iv_cap, bool foot, int *blocks_per_sm) {
  const size_t dyn = enum_dyn_smem(iv_cap);
  cudaError_t e = enum_allow_smem(dyn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, foot ? rows_kernel<true> : rows_kernel<false>,
                                                       kRowsThreads, dyn);
}
cudaError_t count_occupancy(int *blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, count_kernel, kCountThreads, 0);
}

}  // namespace ws
