// Tour construction by Eq. 1 (Section II; the integer roulette of reading R2),
// for every tiling, with the unvisited cities compacted twice along the walk
// where a chunk holds 36 cities or more (one or two warps, or one warp segment,
// per ant).
//
// A step that handles every city of the row, visited or not, pays for the
// visited ones too.  The walk therefore runs in up to three phases:
//   phase 0  (more unvisited cities than phase 1 has slots): lane t owns the
//            contiguous chunk [tC, tC + C) of the row and skips visited cities
//            by their tabu bits;
//   phase 1  the unvisited cities, in ascending order, are listed in shared
//            memory and dealt out C1 = 4*ceil(C/16) per lane (lane t takes
//            entries [t*C1, t*C1 + C1)); each step reads the entries and
//            then their weights from the staged row through them.  A visited
//            slot's entry is pointed at a float beside the row that stays 0,
//            so these phases keep no tabu bits and mask nothing (entries are
//            byte offsets for a single instance, city indices in pools);
//   phase 2  the same with C2 = 4*ceil(C/32) per lane (when smaller than C1).
// Phase p starts at the first step at which the unvisited cities fit in the
// segment's H*Cp slots.  Every phase keeps the cities of the segment in
// ascending order, lane after lane and slot after slot, so the first city
// whose inclusive prefix sum exceeds the target is the CPU oracle's choice.
// With several warps per ant the group's threads hold the slots in that
// order, warp 0 first; the warps combine their totals through shared memory,
// and the warp whose range holds the target publishes the city.  The row is
// still staged whole (bulk copy), so the L2 bytes do not change; the
// per-candidate work of the last quarter and eighth of the steps shrinks.
//
// Construct, GB300, ms, m = n unless given: quantised 64-bit sums -> this
// walk: n = 48 0.034 -> 0.029, n = 200 0.163 -> 0.116, n = 384 0.310 -> 0.222,
// n = 517 0.464 -> 0.313, n = 1002 1.118 -> 0.762, n = 1500 2.13 -> 1.37,
// n = 2392 5.05 -> 3.20, n = 4096 with m = 1024 9.02 -> 6.12.  Small instances
// are bound by the step's chain (about 1500 cycles at n = 1002: the row copy
// 500, the sums 200, the scan and the lane 280, the slot 150, the rest
// issue), large ones also by the rows: 54.7 GB at n = 2392 take 2.7 ms at the
// L2's read rate.
#pragma once

namespace aco {

// The weight bits a list entry points at: entry = city * kUnit (kUnit 1: a
// city index; 4: a byte offset into the staged row).
template <uint32_t kUnit>
__device__ __forceinline__ uint32_t entry_weight(const float* row, uint32_t e) {
  if constexpr (kUnit == 4u)
    return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(row) + e);
  else
    return __float_as_uint(row[e]);
}

struct WalkState {
  int cur;       // current city
  int s;         // next step (1 .. n-1)
  int live;      // unvisited cities listed for the current phase (gather phases)
  float u;       // this lane's uniform r / 2^64 for its step of the window
  uint32_t parity;          // mbarrier phase of the row copy
  // The thread's index in the group (0 issues the copies), or, after a wait that
  // gave up, -2 minus the parity it waited for.  (One value for both: a flag of
  // its own in the issue condition cost the walk 1 %.)
  int role;
};

// The city of one step: `next`, and in gather phases the thread and slot that
// hold it (chosen = -1: already marked).
struct Pick {
  int next, chosen, slot;
};

// The integer roulette of one step from the staged row (reading R2), slot by
// slot: taken when the float search below cannot tell which city the target
// falls on, or no open weight is positive (0.1-2 % of the steps).  Its loops
// stay rolled and read the row again, so that it costs the walk no registers;
// as a call of its own it cost 3 % (the values kept across the call).
// list = nullptr: slot i of thread tg is city tg*cp + i with tabu bits vis;
// otherwise the list entry tg*cp + i.
template <int G, int H, uint32_t kUnit, int NW>
__device__ __forceinline__ Pick exact_pick(const float* row, uint16_t* list, int cp,
                                           uint32_t zero_entry, const uint32_t (&vis)[NW], int tg,
                                           int bar_id, GroupSmem* gs, unsigned long long r) {
  constexpr int NT = G * H;
  const Seg<H> seg(threadIdx.x & 31);
  const int hl = seg.hl, wg = G > 1 ? tg >> 5 : 0;
  auto group_wait = [&]() {
    if constexpr (G > 1)
      group_sync(bar_id, NT);
    else
      seg.sync();
  };
  auto closed = [&](int i) {
    uint32_t word = vis[0];
#pragma unroll
    for (int w = 1; w < NW; ++w)
      if (i >= 32 * w) word = vis[w];
    return (word >> (i & 31)) & 1u;
  };
  auto weight = [&](int i) -> uint32_t {
    if (list) return entry_weight<kUnit>(row, list[tg * cp + i]);
    return closed(i) ? 0u : __float_as_uint(row[tg * cp + i]);
  };
  uint32_t mx = 0u;
#pragma unroll 1
  for (int i = 0; i < cp; ++i) mx = max(mx, weight(i));
  mx = seg.max_u32(mx);
  if constexpr (G > 1) {
    if (hl == 0) gs->wmax[wg] = mx;
    group_wait();
#pragma unroll
    for (int k = 0; k < G; ++k) mx = max(mx, gs->wmax[k]);
  }
  if (mx == 0u) {
    // Every open weight is zero: the lowest open city (a list's smallest
    // entry; zero_entry is above every city's).
    uint32_t cand = 0xffffffffu;
#pragma unroll 1
    for (int i = cp - 1; i >= 0; --i) {
      if (list) {
        cand = min(cand, (uint32_t)list[tg * cp + i]);
      } else {
        if (!closed(i)) cand = (uint32_t)(tg * cp + i);
      }
    }
    cand = seg.min_u32(cand);
    if constexpr (G > 1) {
      if (hl == 0) gs->wmin[wg] = (int)cand;
      group_wait();
#pragma unroll
      for (int k = 0; k < G; ++k) cand = min(cand, (uint32_t)gs->wmin[k]);
    }
    if (!list) return Pick{(int)cand, -1, 0};
    // no other thread reads these entries until the step's end
#pragma unroll 1
    for (int i = 0; i < cp; ++i)
      if (list[tg * cp + i] == cand) list[tg * cp + i] = (uint16_t)zero_entry;
    return Pick{(int)(cand / kUnit), -1, 0};
  }
  float f1, f1s, f2;
  quant_factors(kRouletteBits - 1 - exponent_of_bits(mx), f1, f1s, f2);
  unsigned long long mine = 0;
#pragma unroll 1
  for (int i = 0; i < cp; ++i) mine += quant_value(weight(i), f1, f1s, f2);
  const unsigned long long incl = seg.inclusive_scan(mine);
  const unsigned long long wtot = seg.shfl(incl, H - 1);
  unsigned long long woff = 0, Q = wtot;
  if constexpr (G > 1) {
    if (hl == 0) gs->wsum[wg] = wtot;
    group_wait();
    Q = 0;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const unsigned long long v = gs->wsum[k];
      if (k < wg) woff += v;
      Q += v;
    }
  }
  const unsigned long long T = __umul64hi(r, Q);
  Pick out{0, 0, 0};
  if (G == 1 || (T >= woff && T - woff < wtot)) {
    const int L = max(__ffs(seg.ballot(woff + incl > T)) - 1, 0);
    int slot = 0, city = 0;
    if (hl == L) {
      unsigned long long c = woff + incl - mine;
#pragma unroll 1
      for (; slot < cp - 1; ++slot) {
        c += quant_value(weight(slot), f1, f1s, f2);
        if (c > T) break;
      }
      city = list ? (int)(list[tg * cp + slot] / kUnit) : tg * cp + slot;
    }
    out.next = seg.shfl(city, L);
    out.chosen = wg * 32 + L;
    out.slot = seg.shfl(slot, L);
    if constexpr (G > 1) {
      if (hl == 0) {
        gs->xnext = out.next;
        gs->xchosen = out.chosen;
        gs->xslot = out.slot;
      }
    }
  }
  if constexpr (G > 1) {
    group_wait();
    out = Pick{gs->xnext, gs->xchosen, gs->xslot};
  }
  return out;
}

// Steps [w.s, s_end) of one phase.  CP: slots per thread.  kGather = false:
// slot i of thread t is city t*C + i (phase 0); true: slot i holds the entry
// ulist[t*CP + i] (its city's weight, or the zero slot once visited).  CPN > 0:
// afterwards, list the unvisited cities for a phase of CPN slots per thread.
//
// A step samples the integer roulette without its integers.  With S the sum
// of the open weights and u = r / 2^64, the roulette takes the city whose
// interval of the prefix sums holds u S, up to the floors of its quantiser:
// at most n 2^-45 S.  The step forms the prefix sums in single precision
// (per part of a thread's slots, a warp scan over the threads, a second scan
// over the chosen part) and takes the city only if u S lies inside its
// interval by more than eps S on both sides, eps = kRoundings 2^-24: every
// partial sum of non-negative terms is within (its roundings) 2^-24 S of the
// true one, so the integer roulette takes the same city.  Otherwise (the
// target within the error of a boundary; S zero, tiny, infinite or NaN) the
// step runs exact_pick().  This drops the max pass, the three FMAs of the
// quantiser and half of every shuffle (64-bit scans) from a step.
template <int C, int CP, int CPN, int G, int H, bool kGather, bool kPool, bool kLane>
__device__ __forceinline__ void eq1_phase(const Instance& I, const int ant, const int tg,
                                          const Seg<H> seg, GroupSmem* gs, const int bar_id,
                                          float* srow, uint16_t* ulist, const int start,
                                          const int s_end, WalkState& w) {
  static_assert(CP % 4 == 0 && CP >= 4 && CP <= 160, "CP must be a multiple of 4 in [4,160]");
  static_assert(kGather || CP == C, "the direct phase reads whole chunks");
  static_assert(G == 1 || H == 32, "several warps per ant use whole warps");
  constexpr int NT = G * H;  // threads per ant
  constexpr int NW = (CP + 31) / 32;  // tabu words per lane (direct phase)
  // The second-level search takes a part of kPart slots, whole in every lane.
  constexpr int kPart = CP < 8 ? CP : 8;
  constexpr int K = (CP + kPart - 1) / kPart;
  constexpr bool kHalfTail = CP % kPart != 0;  // the last part holds four slots
  constexpr int kScan = H == 32 ? 5 : (H == 16 ? 4 : 3);
  // roundings on the way to one side of the test: the prefix before the lane
  // and, inside the target, S (part sums of 4 + 1 additions, parts, scan,
  // warps each); the part's prefix inside the lane, the slot's prefix inside
  // the part; the target and the differences; two to spare for the
  // quantiser's floors and the second-order terms
  constexpr int kRoundings = 2 * (5 + K + kScan + G) + (5 + K) + kPart + 10;
  constexpr float kEps = (float)kRoundings * 0x1p-24f;
  constexpr int kListCap = StageLayout<C, G, H>::kListEntries;
  const int n = I.n, ld = I.ld;
  const int hl = seg.hl;          // lane within the segment
  const int wg = G > 1 ? tg >> 5 : 0;  // warp within the group
  const int base = tg * C;        // phase 0: the thread's chunk in the row
  auto group_wait = [&]() {
    if constexpr (G > 1)
      group_sync(bar_id, NT);
    else
      seg.sync();
  };
  const uint32_t iter = (uint32_t)I.st->iteration;
  const unsigned long long seed = I.seed;
  const uint32_t srow_a = smem_u32(srow);
  const uint32_t bar = srow_a + (uint32_t)StageLayout<C, G, H>::kRowFloats * 4u;
  const uint32_t row_bytes = (uint32_t)ld * 4u;
  int32_t* tour = I.tours + (size_t)ant * I.ldt;
  const float* const choice = I.choice;

  // Direct phase: tabu bits (1 = visited, or no city in the slot).  Gather
  // phases keep no tabu bits: a slot's list entry points at its city's
  // weight in the staged row while it is unvisited, and at kZeroSlot (a
  // float beside the row that stays 0) once it is visited or holds no city,
  // so a visited slot reads weight 0 and is never chosen.
  constexpr uint32_t kZeroSlot = StageLayout<C, G, H>::kZeroSlot;
  // A single instance lists byte offsets into the staged row (city * 4: no
  // address arithmetic per read), pools list city indices (measured faster
  // for the batched classes, slower for one instance).
  constexpr uint32_t kUnit = kPool ? 1u : 4u;
  constexpr uint32_t kZeroEntry = kZeroSlot * kUnit;
  static_assert(kZeroEntry <= 0xffffu, "list entries are 16-bit");
  uint32_t vis[kGather ? 1 : NW];
  if constexpr (!kGather) {
#pragma unroll
    for (int wd = 0; wd < NW; ++wd) {
      const int real = n - (base + 32 * wd);  // local cities of word wd below n
      uint32_t word = real <= 0 ? FULL : (real >= 32 ? 0u : (FULL << real));
      const int inchunk = C - 32 * wd;
      if (inchunk < 32) word |= FULL << inchunk;
      vis[wd] = word;
    }
    const int li = start - base;
    if (li >= 0 && li < C) {
#pragma unroll
      for (int wd = 0; wd < NW; ++wd)
        if (wd == (li >> 5)) vis[wd] |= 1u << (li & 31);
    }
  } else {
    // The thread's slots past the listed cities point at the zero weight.
#pragma unroll
    for (int i = 0; i < CP; ++i) {
      const int k = tg * CP + i;
      if (k >= w.live) ulist[k] = (uint16_t)kZeroEntry;
    }
    group_wait();  // other lanes read these entries in the rescan
  }

  for (; w.s < s_end; ++w.s) {
    const int s = w.s;
    const int cur = w.cur;
    // Everyone is done with the previous row (the group agreed on `cur`).
    // Its reads are complete and nothing but the copy engine writes it, so
    // the copy needs no proxy fence.
    if constexpr (kLane) {
      const float* src = choice + (size_t)cur * ld + 4 * tg;
#pragma unroll
      for (int i = 0; i < C / 4; ++i)
        cp_async16_if(4 * (tg + i * NT) < ld, srow_a + 16u * (uint32_t)(tg + i * NT),
                      src + 4 * i * NT);
      cp_async_wait_all();
    } else {
      bulk_load_if(w.role == 0, srow_a, choice + (size_t)cur * ld, row_bytes, bar);
    }
    const int off = (s - 1) % H;
    if (off == 0) {
      const Philox4 x = step_draw(seed, (uint32_t)(s + hl), (uint32_t)ant, iter);
      w.u = __fmul_rn(__uint2float_rn(x.x1), 0x1p-32f);
    }
    const float u = seg.shfl(w.u, off);
    if constexpr (kLane) {
      group_wait();
    } else {
      if (!mbar_try_wait(bar, w.parity) && w.role >= 0 && !mbar_wait_bounded(bar, w.parity)) {
        // stale data and no further copies from here on; the status word says so
        w.role = -2 - (int)w.parity;
        atomicOr(&I.st->status, kStatusTimeout);
      }
      w.parity ^= 1u;
    }
    const float* row = srow;

    // Inclusive sums of the open weights over the parts; the last is the
    // thread's.
    float pincl[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      float acc[2] = {0.0f, 0.0f};
#pragma unroll
      for (int g = k * (kPart / 4); g < (k + 1) * (kPart / 4) && g < CP / 4; ++g) {
        float v[4];
        if constexpr (!kGather) {
          // Chunk entries at or beyond ld hold stale data; their tabu bits are set.
          const float4 t = *reinterpret_cast<const float4*>(row + base + 4 * g);
          v[0] = t.x;
          v[1] = t.y;
          v[2] = t.z;
          v[3] = t.w;
        } else {
          const uint2 e = reinterpret_cast<const uint2*>(ulist + tg * CP)[g];
          v[0] = __uint_as_float(entry_weight<kUnit>(row, e.x & 0xffffu));
          v[1] = __uint_as_float(entry_weight<kUnit>(row, e.x >> 16));
          v[2] = __uint_as_float(entry_weight<kUnit>(row, e.y & 0xffffu));
          v[3] = __uint_as_float(entry_weight<kUnit>(row, e.y >> 16));
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          bool open = true;
          if constexpr (!kGather) open = !((vis[(4 * g + e) >> 5] >> ((4 * g + e) & 31)) & 1u);
          if (open) acc[e & 1] = __fadd_rn(acc[e & 1], v[e]);
        }
      }
      const float v = __fadd_rn(acc[0], acc[1]);
      pincl[k] = k ? __fadd_rn(pincl[k - 1], v) : v;
    }
    const float mine = pincl[K - 1];
    const float incl = seg.inclusive_scan_f(mine);
    const float wtot = seg.shfl(incl, H - 1);
    float woff = 0.0f, S = wtot;
    if constexpr (G > 1) {
      if (hl == 0) gs->wtot[wg] = wtot;
      group_wait();
      S = 0.0f;
#pragma unroll
      for (int k = 0; k < G; ++k) {
        if (k == wg) woff = S;
        S = __fadd_rn(S, gs->wtot[k]);
      }
    }
    // The target inside this thread's range, and the part of the thread's
    // slots that holds it if it lies there.  Every lane works this out while
    // the vote finds the lane.
    const float t1 = __fsub_rn(__fmul_rn(u, S), woff);
    const float err = S >= 0x1p-120f ? __fmul_rn(kEps, S) : __int_as_float(0x7f800000);
    const uint32_t passed = seg.ballot(!(incl > t1));
    const float t2 = __fsub_rn(t1, __fsub_rn(incl, mine));
    uint32_t part = 0u;
    float before = 0.0f;
#pragma unroll
    for (int k = 0; k < K - 1; ++k)
      if (pincl[k] <= t2) {
        part = (uint32_t)(k + 1);
        before = pincl[k];
      }
    if constexpr (!kGather) {
      // the part's tabu bits beside its number
      uint32_t word = vis[0];
#pragma unroll
      for (int wd = 1; wd < NW; ++wd)
        if (part * kPart >= 32u * wd) word = vis[wd];
      part |= (word >> ((part * kPart) & 31u)) << 8;
    }
    // the inclusive sums ascend: as many lanes are passed as lie before L
    const int L = min(__popc(passed), H - 1);
    const float t3 = seg.shfl(__fsub_rn(t2, before), L);
    part = seg.shfl(part, L);
    const uint32_t closed = part >> 8;  // direct phase
    if constexpr (!kGather) part &= 0xffu;
    // The slot inside the part: every lane reads the part and decides alike,
    // with no further exchange.
    const float hi_t = __fadd_rn(t3, err), lo_t = __fsub_rn(t3, err);
    const int tL = wg * 32 + L;  // thread of lane L within the group
    const int pstart = (int)part * kPart;
    float wv[kPart];
    uint32_t ent[kGather ? kPart : 1] = {};
    if constexpr (!kGather) {
      // (past the chunk's end: the tabu bits there are set, and the staged row
      // is followed by its mbarrier and the zero weight, 16 bytes)
      const float4* p4 = reinterpret_cast<const float4*>(row + tL * C + pstart);
#pragma unroll
      for (int g = 0; g < kPart / 4; ++g) {
        const float4 t = p4[g];
        wv[4 * g] = t.x;
        wv[4 * g + 1] = t.y;
        wv[4 * g + 2] = t.z;
        wv[4 * g + 3] = t.w;
      }
    } else {
      const uint2* lw = reinterpret_cast<const uint2*>(ulist + tL * CP + pstart);
      const bool half = kHalfTail && part == (uint32_t)(K - 1);
#pragma unroll
      for (int g = 0; g < kPart / 4; ++g) {
        uint2 e = lw[g > 0 && half ? 0 : g];
        if (g > 0 && half) e = make_uint2(kZeroEntry * 0x10001u, kZeroEntry * 0x10001u);
        ent[4 * g] = e.x & 0xffffu;
        ent[4 * g + 1] = e.x >> 16;
        ent[4 * g + 2] = e.y & 0xffffu;
        ent[4 * g + 3] = e.y >> 16;
      }
#pragma unroll
      for (int i = 0; i < kPart; ++i) wv[i] = __uint_as_float(entry_weight<kUnit>(row, ent[i]));
    }
    // The first slot whose inclusive sum passes the target by the error; sure
    // if the sum before it lies below the target by the error as well.
    int slot = 0;
    float c = 0.0f, below = 0.0f;
    uint32_t hit = kGather ? ent[0] : 0u;
#pragma unroll
    for (int i = 0; i < kPart; ++i) {
      if (kGather || !((closed >> i) & 1u)) c = __fadd_rn(c, wv[i]);
      if (!(c > hi_t)) {
        slot = i + 1;
        below = c;
        if (kGather && i + 1 < kPart) hit = ent[i + 1];
      }
    }
    bool found = slot < kPart && below < lo_t;
    Pick got{kGather ? (int)(hit / kUnit) : tL * C + pstart + slot, tL, pstart + slot};
    if constexpr (G > 1) {
      // One warp at most is sure.  fnext[s & 1] was reset between the two
      // barriers of the step before, after every read of step s - 2's.
      if (found && hl == 0) {
        gs->fnext[s & 1] = got.next;
        gs->chosen = got.chosen;
        gs->slot = got.slot;
      }
      if (tg == 0) gs->fnext[(s + 1) & 1] = -1;
      group_wait();
      got = Pick{gs->fnext[s & 1], gs->chosen, gs->slot};
      found = got.next >= 0;
    }
    if (!found) {
      const Philox4 x = step_draw(seed, (uint32_t)s, (uint32_t)ant, iter);
      const unsigned long long r = ((unsigned long long)x.x1 << 32) | x.x0;
      got = exact_pick<G, H, kUnit>(row, kGather ? ulist : nullptr, CP, kZeroEntry, vis, tg, bar_id,
                                    gs, r);
      // A city outside [0, n) can only come from a defect; record it and stay
      // in bounds instead of reading past the matrix.
      if ((unsigned)got.next >= (unsigned)n) {
        if (tg == 0) atomicOr(&I.st->status, kStatusBadTour);
        got.next = start;
        got.chosen = -1;
      }
    }
    const int next = got.next;
    if constexpr (!kGather) {
      const int li = next - base;
      if (li >= 0 && li < C) {
#pragma unroll
        for (int wd = 0; wd < NW; ++wd)
          if (wd == (li >> 5)) vis[wd] |= 1u << (li & 31);
      }
    } else {
      // Every lane of the chosen thread's warp (or segment) read this entry to
      // decide: they all have to be past those reads before it changes.  (With
      // several warps per ant the barrier that published the city says so.)
      if constexpr (G == 1) seg.sync();
      if (tg == got.chosen) ulist[tg * CP + got.slot] = (uint16_t)kZeroEntry;
    }
    if (tg == 0) tour[s] = next;
    w.cur = next;
    // G > 1: the barrier above (or exact_pick's last) already follows every
    // read of the row; the lanes of a warp still have to see the mark.
    if constexpr (G > 1 && !kLane)
      __syncwarp();
    else
      group_wait();
  }

  if constexpr (CPN > 0) {
    if constexpr (G > 1) group_wait();
    // List the unvisited cities for the next phase, ascending: lane after
    // lane, each lane's slots in order.
    uint32_t cnt = 0;
    uint32_t own[kGather ? CP : 1];  // gather phases: the thread's entries
    if constexpr (kGather) {
      const uint2* lw = reinterpret_cast<const uint2*>(ulist + tg * CP);
#pragma unroll
      for (int i = 0; i < CP; i += 4) {
        const uint2 e = lw[i >> 2];
        own[i] = e.x & 0xffffu;
        own[i + 1] = e.x >> 16;
        own[i + 2] = e.y & 0xffffu;
        own[i + 3] = e.y >> 16;
      }
#pragma unroll
      for (int i = 0; i < CP; ++i) cnt += own[i] != kZeroEntry ? 1u : 0u;
    } else {
#pragma unroll
      for (int wd = 0; wd < NW; ++wd) cnt += __popc(~vis[wd]);
    }
    const unsigned long long incl = seg.inclusive_scan((unsigned long long)cnt);
    int total = (int)seg.shfl(incl, H - 1);
    int k = (int)(incl - cnt);
    if constexpr (G > 1) {
      if (hl == 0) gs->wsum[wg] = (unsigned long long)total;
      group_wait();
      total = 0;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int v = (int)gs->wsum[q];
        if (q < wg) k += v;
        total += v;
      }
    }
    group_wait();  // the list of this phase is no longer read
#pragma unroll
    for (int i = 0; i < CP; ++i) {
      bool live;
      if constexpr (kGather)
        live = own[i] != kZeroEntry;
      else
        live = !((vis[i >> 5] >> (i & 31)) & 1u);
      if (live) {
        // a defect can leave more entries than the list holds: keep in bounds
        if (k < kListCap) ulist[k] = (uint16_t)(kGather ? own[i] : kUnit * (uint32_t)(base + i));
        ++k;
      }
    }
    w.live = total < NT * CPN ? total : NT * CPN;
    group_wait();
  }
}

// Phase J of the walk and the ones after it.  Phase J runs while the
// unvisited cities do not fit in the next phase's slots, then lists them for
// it; the last phase runs to the end of the tour.
template <int C, int G, int H, bool kPool, bool kLane, int J>
__device__ __forceinline__ void eq1_phases(const Instance& I, const int ant, const int tg,
                                           const Seg<H> seg, GroupSmem* gs, const int bar_id,
                                           float* srow, uint16_t* ulist, const int start,
                                           WalkState& w) {
  using Cm = Compaction<C, G>;
  constexpr int CP = Cm::slots(J);
  constexpr int CPN = Cm::slots(J + 1);
  const int s_end = CPN > 0 ? max(w.s, I.n - G * H * CPN) : I.n;
  eq1_phase<C, CP, CPN, G, H, (J > 0), kPool, kLane>(I, ant, tg, seg, gs, bar_id, srow, ulist,
                                                     start, s_end, w);
  if constexpr (CPN > 0)
    eq1_phases<C, G, H, kPool, kLane, J + 1>(I, ant, tg, seg, gs, bar_id, srow, ulist, start, w);
}

// The whole walk of one ant (G warps or one H-lane segment) and its length
// and neighbour buckets.  False where this thread's wait for a row gave up: the
// staging memory may still have a copy in flight, and no further bulk copy may
// use it.
template <int C, int G, int H, bool kPool>
__device__ __forceinline__ bool construct_ant_phased(const Instance& I, const int ant,
                                                     const int tg, const Seg<H> seg,
                                                     GroupSmem* gs, const int bar_id, float* srow,
                                                     const bool lane_copy) {
  constexpr int NT = G * H;
  uint16_t* ulist = reinterpret_cast<uint16_t*>(reinterpret_cast<char*>(srow) +
                                                StageLayout<C, G, H>::kListOffset);
  const int n = I.n;
  const int hl = seg.hl;
  const int wg = G > 1 ? tg >> 5 : 0;
  auto group_wait = [&]() {
    if constexpr (G > 1)
      group_sync(bar_id, NT);
    else
      seg.sync();
  };
  const uint32_t iter = (uint32_t)I.st->iteration;
  const Philox4 x0 = step_draw(I.seed, 0u, (uint32_t)ant, iter);
  const int start = (int)__umulhi(x0.x0, (uint32_t)n);
  int32_t* tour = I.tours + (size_t)ant * I.ldt;
  if (tg == 0) tour[0] = start;
  const uint32_t bar = smem_u32(srow) + (uint32_t)StageLayout<C, G, H>::kRowFloats * 4u;
  if (tg == 0) {
    if (!lane_copy) {
      mbar_init(bar, 1);
      fence_mbar_init();
    }
    srow[StageLayout<C, G, H>::kZeroSlot] = 0.0f;  // the weight of a visited list slot
    if (G > 1) gs->fnext[0] = gs->fnext[1] = -1;
  }
  // In a persistent launch the ant before may have staged its rows by lane
  // copies (generic proxy) in these bytes: each lane orders its own before the
  // bulk copies that follow the group's wait.
  fence_proxy_async_smem();
  group_wait();

  WalkState w{start, 1, 0, 0.0f, 0u, tg};
  if (lane_copy)
    eq1_phases<C, G, H, kPool, true, 0>(I, ant, tg, seg, gs, bar_id, srow, ulist, start, w);
  else
    eq1_phases<C, G, H, kPool, false, 0>(I, ant, tg, seg, gs, bar_id, srow, ulist, start, w);
  // the copy in flight, again with a limit
  if (w.role < 0) mbar_wait_bounded(bar, (uint32_t)w.role & 1u);
  if (tg == 0) tour[n] = start;
  group_wait();

  // C^k (Section II) and the per-city neighbour buckets.
  long long len = 0;
  for (int s = tg; s < n; s += NT) {
    const int a = tour[s], b = tour[s + 1];
    const int p = tour[s == 0 ? n - 1 : s - 1];
    len += I.dist[(size_t)a * I.ld + b];
    I.nbr[(size_t)a * I.ldm + ant] = ((uint32_t)p << 16) | (uint32_t)b;
  }
#pragma unroll
  for (int o = H / 2; o > 0; o >>= 1) len += seg.shfl_xor(len, o);
  if constexpr (G > 1) {
    if (hl == 0) gs->wlen[wg] = len;
    group_wait();
    len = 0;
#pragma unroll
    for (int k = 0; k < G; ++k) len += gs->wlen[k];
  }
  if (tg == 0) I.lens[ant] = len;
  // In a persistent launch the warp's next ant, of this class or another, uses
  // these bytes for its row or its own barrier.  (Initialised again while alive,
  // the barrier's first wait timed out there, beside classes with lane copies.)
  if (tg == 0 && !lane_copy && w.role >= 0) mbar_inval(bar);
  return w.role >= 0;
}

}  // namespace aco
