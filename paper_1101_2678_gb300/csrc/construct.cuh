// Tour construction (Section II, Eq. 1; data-parallel design of Section III-A):
// the pieces shared by the construction kernels, the per-candidate rules, and
// the kernels.  The Eq. 1 walk itself is in construct_phased.cuh.
//
// One group of threads builds one ant's tour: G whole warps (H = 32), or an
// H-lane segment of a warp (H = 8 or 16, G = 1), so that 32/H ants share
// every warp instruction.  Thread t of the group owns the contiguous cities
// [t*C, t*C + C) of every row, and keeps their tabu bits (the paper's "1 =
// unvisited" integer per city, here one bit per city in registers).  At each
// step one thread copies row choice[cur] into shared memory with the
// bulk-copy engine; the group waits on an mbarrier, reads its chunks (C
// floats per thread, conflict-free 16-byte loads) and selects.
// The selection is defined by exact maxima and exact integer sums (the integer
// roulette: M = max over unvisited; q_j = floor(w_j * 2^(45-ilogb M)); Q their
// sum; T = floor(r Q / 2^64) with r from Philox; the first j whose prefix sum
// exceeds T), so the chosen city is the same for every (C, G, H) tiling and
// equals the CPU oracle's choice.
// Every warp-level intrinsic names only the segment's lanes, so segments of
// one warp never wait on each other even when their control flow differs.
// After the last step the group computes C^k = sum of d over the tour and
// writes, for every city of the tour, its predecessor and successor into
// nbr[city][ant] (the bucketing used by the gather deposit).
#pragma once

#include "aco_device.cuh"

namespace aco {

struct GroupSmem {
  uint32_t wmax[4];
  unsigned long long wsum[4];
  long long wlen[4];
  int wmin[4];
  // the Eq. 1 walk
  float wtot[4];
  int fnext[2], chosen, slot;
  int xnext, xchosen, xslot;
};

constexpr int kMaxGroupsPerCta = 8;

__device__ __forceinline__ void group_sync(int bar_id, int nthreads) {
  if (nthreads == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(nthreads) : "memory");
  }
}

// Roulette weight bits: q_j = floor(w_j * 2^(kRouletteBits-1-ilogb M)).
constexpr int kRouletteBits = 46;
constexpr float kTwo23 = 8388608.0f;
constexpr uint32_t kTwo23Bits = 0x4b000000u;

// q = floor(w * 2^sc) < 2^46 as hi * 2^23 + lo, in three FP32 FMAs.
// With t = w * f1 (f1 = 2^(sc-23), so t < 2^23):
//   zh = fma.rz(w, f1, 2^23)           = 2^23 + floor(t)          (one rounding of w*f1 + 2^23)
//   c  = fma(zh, -2^23, 2^46 + 2^23)   = 2^23 - floor(t) * 2^23   (exact: representable)
//   zl = fma.rz(w, f1 * 2^23, c)       = 2^23 + floor(frac(t) * 2^23)
// zh and zl are floats in [2^23, 2^24) whose bit patterns are 0x4b000000 +
// hi and 0x4b000000 + lo.  Each rounding is of an exactly known value, so
// both floors are exact for every w >= 0 (subnormal products included: the
// fused multiply-add never rounds w * f1 on its own).
struct QuantParts {
  uint32_t hi_bits, lo_bits;
};

constexpr float kTwo46p23 = 70368752566272.0f;  // 2^46 + 2^23

__device__ __forceinline__ QuantParts quant_parts(uint32_t b, float f1, float f1s) {
  const float w = __uint_as_float(b);
  const float zh = __fmaf_rz(w, f1, kTwo23);
  const float c = __fmaf_rn(zh, -kTwo23, kTwo46p23);
  const float zl = __fmaf_rz(w, f1s, c);
  return QuantParts{__float_as_uint(zh), __float_as_uint(zl)};
}

// q of a weight that still needs the pre-scaling by f2 (see quant_factors).
__device__ __forceinline__ unsigned long long quant_value(uint32_t b, float f1, float f1s,
                                                          float f2) {
  if (f2 != 1.0f) b = __float_as_uint(__fmul_rn(__uint_as_float(b), f2));
  const QuantParts q = quant_parts(b, f1, f1s);
  return ((unsigned long long)(q.hi_bits - kTwo23Bits) << 23) + (q.lo_bits - kTwo23Bits);
}

// Factors for the step: f1 = 2^(sc-23) and f1s = f1 * 2^23 must both be
// normal floats, i.e. sc - 23 <= 104.  Beyond that (largest unvisited
// weight below 2^-82) the weights are first scaled up exactly by f2.
__device__ __forceinline__ void quant_factors(int sc, float& f1, float& f1s, float& f2) {
  const int e = sc - 23;
  if (e <= 104) {
    f1 = pow2f(e);
    f1s = pow2f(e + 23);
    f2 = 1.0f;
  } else {
    f1 = pow2f(104);
    f1s = pow2f(127);
    f2 = pow2f(e - 104);
  }
}

// The lanes of one warp segment (H = 32: the whole warp).
template <int H>
struct Seg {
  unsigned mask;
  int sub;  // segment index within the warp
  int hl;   // lane within the segment
  __device__ __forceinline__ explicit Seg(int lane)
      : mask(H == 32 ? FULL : (((1u << H) - 1u) << ((lane / H) * H))), sub(lane / H),
        hl(lane % H) {}
  template <typename T>
  __device__ __forceinline__ T shfl(T v, int src) const {
    return __shfl_sync(mask, v, src, H);
  }
  template <typename T>
  __device__ __forceinline__ T shfl_up(T v, int d) const {
    return __shfl_up_sync(mask, v, d, H);
  }
  template <typename T>
  __device__ __forceinline__ T shfl_xor(T v, int d) const {
    return __shfl_xor_sync(mask, v, d, H);
  }
  __device__ __forceinline__ uint32_t ballot(bool p) const {
    const uint32_t b = __ballot_sync(mask, p);
    return H == 32 ? b : (b >> (sub * H)) & ((1u << H) - 1u);
  }
  __device__ __forceinline__ uint32_t max_u32(uint32_t v) const {
    if constexpr (H == 32) {
      return __reduce_max_sync(FULL, v);
    } else {
#pragma unroll
      for (int o = H / 2; o > 0; o >>= 1) v = max(v, shfl_xor(v, o));
      return v;
    }
  }
  __device__ __forceinline__ uint32_t min_u32(uint32_t v) const {
    if constexpr (H == 32) {
      return __reduce_min_sync(FULL, v);
    } else {
#pragma unroll
      for (int o = H / 2; o > 0; o >>= 1) v = min(v, shfl_xor(v, o));
      return v;
    }
  }
  __device__ __forceinline__ unsigned long long inclusive_scan(unsigned long long x) const {
#pragma unroll
    for (int o = 1; o < H; o <<= 1) {
      const unsigned long long t = shfl_up(x, o);
      if (hl >= o) x += t;
    }
    return x;
  }
  // Inclusive sums in single precision; the shuffle's own predicate says
  // whether a lane d below exists in the segment.
  __device__ __forceinline__ float inclusive_scan_f(float x) const {
#pragma unroll
    for (int o = 1; o < H; o <<= 1)
      asm volatile(
          "{\n\t.reg .pred p;\n\t.reg .f32 t;\n\t"
          "shfl.sync.up.b32 t|p, %0, %1, %2, %3;\n\t"
          "@p add.rn.f32 %0, %0, t;\n\t}"
          : "+f"(x)
          : "r"(o), "n"((32 - H) << 8), "r"(mask));
    return x;
  }
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};

// Cities per thread before and after the compactions of the Eq. 1 walk (see
// construct_phased.cuh): C, then 4*ceil(C/16) and 4*ceil(C/32) (about C/4 and
// C/8 in whole 4-city groups), repeats dropped.  A listed city costs an index
// load and an indexed load more than a chunk's, a visited chunk city two
// instructions, so a first compaction at C/2 loses (n = 1002 0.801 ms with
// C/2, C/4 and C/8, 0.782 with C/4 and C/8, 0.796 with C/4 alone; n = 2392
// 3.35, 3.24, 3.26; a step of 256 instances 14.3, 12.3, 12.4), and chunks
// below 36 cities are not compacted at all (n = 517 0.317 ms against 0.335;
// n = 800 0.543 against 0.552).  One warp (or segment) or two warps per ant
// compact; four warps per ant never do.
constexpr int kCompactMinC = 36;
template <int C, int G>
struct Compaction {
  static constexpr bool kOn = (G == 1 || G == 2) && C >= kCompactMinC;
  static constexpr int kPhases = 3;
  // candidate count i: C * kSixteenths[i] / 16 rounded up to a multiple of 4
  __host__ __device__ static constexpr int raw(int i) {
    constexpr int kSixteenths[kPhases] = {16, 4, 2};
    return kSixteenths[i] == 16 ? C : 4 * ((kSixteenths[i] * C + 63) / 64);
  }
  // Slot count of phase j (0 = the direct phase, C), or 0 past the last.
  __host__ __device__ static constexpr int slots(int j) {
    if (!kOn) return j == 0 ? C : 0;
    int prev = 1 << 30, k = -1;
    for (int i = 0; i < kPhases; ++i) {
      const int v = raw(i);
      if (v > 0 && v < prev) {
        if (++k == j) return v;
        prev = v;
      }
    }
    return 0;
  }
};

// Shared memory of one ant group: the staged row (H*G*C floats, 16-byte
// aligned), its mbarrier, and (when the walk compacts) the list of unvisited
// cities, up to H*G * 4*ceil(C/16) 16-bit entries.  (Rows of ld floats would
// leave room for more ants, but a group stride known only at run time made the
// compacting walk 10-30 % slower: n = 2392 3.34 -> 4.31 ms.)
template <int C, int G, int H>
struct StageLayout {
  static constexpr int kRowFloats = H * G * C;
  static constexpr int kListOffset = kRowFloats * 4 + 16;
  // A float index beside the row (after the mbarrier, before the list) that
  // holds 0: the list entry of a visited slot of the walk with compaction.
  static constexpr int kZeroSlot = kRowFloats + 2;
  static constexpr int kListEntries = Compaction<C, G>::kOn ? H * G * Compaction<C, G>::slots(1) : 0;
  static constexpr int kBytes = ((kListOffset + 2 * kListEntries) + 15) / 16 * 16;
};

// Ant groups per CTA of `warps` warps.
template <int G, int H>
__host__ __device__ constexpr int groups_per_cta(int warps) {
  return H == 32 ? warps / G : warps * (32 / H);
}

// E = -ln(v 2^-24) for the candidate word x, v = floor(x / 2^8) + 1 in
// [1, 2^24], in single precision by the range-reduced inverse-hyperbolic-
// tangent series of the logarithm: v = 2^e f with f in [1, 2), halved when
// f > sqrt 2; s = (f - 1) / (f + 1); ln f = 2 s (1 + z/3 + z^2/5 + z^3/7 +
// z^4/9), z = s^2; E = (24 - e) ln 2 - ln f.  Every operation is rounded on
// its own (no contraction), so any IEEE implementation of the same sequence
// gives the same bits.  The constants are the floats nearest sqrt 2, ln 2,
// 1/3, 1/5, 1/7 and 1/9.
__device__ __forceinline__ float race_exponential(uint32_t x) {
  const uint32_t v = (x >> 8) + 1u;
  int e = 31 - __clz((int)v);
  // v 2^-e, exact: v < 2^25 is a float and 2^-e a normal power of two
  float f = __fmul_rn(__uint2float_rn(v), __uint_as_float((uint32_t)(127 - e) << 23));
  if (f > 0x1.6a09e6p+0f) {
    f = __fmul_rn(f, 0.5f);
    e += 1;
  }
  const float s = __fdiv_rn(__fsub_rn(f, 1.0f), __fadd_rn(f, 1.0f));
  const float z = __fmul_rn(s, s);
  float p = 0x1.c71c72p-4f;
  p = __fadd_rn(__fmul_rn(p, z), 0x1.24924ap-3f);
  p = __fadd_rn(__fmul_rn(p, z), 0x1.99999ap-3f);
  p = __fadd_rn(__fmul_rn(p, z), 0x1.555556p-2f);
  p = __fadd_rn(__fmul_rn(p, z), 1.0f);
  const float ln_f = __fmul_rn(__fadd_rn(s, s), p);
  return __fsub_rn(__fmul_rn(__int2float_rn(24 - e), 0x1.62e430p-1f), ln_f);
}

// The per-candidate rules.  R = 1: the paper's data-parallel rule: every
// unvisited city scores u_j * w_j with its own uniform u_j, the highest score
// wins (ties to the lower index; all scores 0: the lowest unvisited city).
// R = 2: the exponential race, which samples Eq. 1: every unvisited city gets
// the key E_j / w_j from its own exponential variate E_j, the smallest key
// wins (ties to the lower index; zero weights and overflowing keys are +inf,
// so with every weight 0 the lowest unvisited city wins).
template <int C, int G, int H, int R>
__device__ __forceinline__ void construct_ant_rule(const Instance& I, const int ant, const int tg,
                                              const Seg<H> seg, GroupSmem* gs, const int bar_id,
                                              float* srow, const bool lane_copy) {
  static_assert(C % 4 == 0 && C >= 4 && C <= 128, "C must be a multiple of 4 in [4,128]");
  static_assert((C / 4) % 2 == 1, "C/4 must be odd: lanes then read their chunks from shared "
                                  "memory without bank conflicts");
  static_assert(G == 1 || G == 2 || G == 4, "G must be 1, 2 or 4");
  static_assert(H == 8 || H == 16 || H == 32, "H must be 8, 16 or 32");
  static_assert(H == 32 || G == 1, "segments smaller than a warp serve one ant each");
  constexpr int NW = (C + 31) / 32;  // tabu words per thread
  constexpr int NT = H == 32 ? 32 * G : H;  // threads per ant
  const int n = I.n, ld = I.ld;
  const int hl = seg.hl;          // lane within the segment
  const int wg = H == 32 ? tg >> 5 : 0;  // warp within the group (G > 1)
  const int base = tg * C;
  const uint32_t iter = (uint32_t)I.st->iteration;
  const unsigned long long seed = I.seed;
  auto group_wait = [&]() {
    if (H == 32)
      group_sync(bar_id, NT);
    else
      seg.sync();
  };

  // Tabu bits: 1 = visited.  Padding cities (index >= n) and bits beyond C
  // start out visited.
  uint32_t vis[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const int real = n - (base + 32 * w);  // local cities of word w below n
    uint32_t word = real <= 0 ? FULL : (real >= 32 ? 0u : (FULL << real));
    const int inchunk = C - 32 * w;
    if (inchunk < 32) word |= FULL << inchunk;
    vis[w] = word;
  }

  const Philox4 x0 = step_draw(seed, 0u, (uint32_t)ant, iter);
  const int start = (int)__umulhi(x0.x0, (uint32_t)n);
  {
    const int li = start - base;
    if (li >= 0 && li < C) {
#pragma unroll
      for (int w = 0; w < NW; ++w)
        if (w == (li >> 5)) vis[w] |= 1u << (li & 31);
    }
  }
  int32_t* tour = I.tours + (size_t)ant * I.ldt;
  const float* const choice = I.choice;
  if (tg == 0) tour[0] = start;
  int cur = start;

  const uint32_t srow_a = smem_u32(srow);
  const uint32_t bar = srow_a + (uint32_t)StageLayout<C, G, H>::kRowFloats * 4u;
  const uint32_t row_bytes = (uint32_t)ld * 4u;
  uint32_t phase = 0;
  int role = tg;  // 0 issues the copies; -2 minus the parity of a wait that gave up
  if (tg == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  group_wait();

  for (int s = 1; s < n; ++s) {
    // Everyone is done with the previous row (the group agreed on `cur`).
    if (lane_copy) {
      // The group copies the row with coalesced 16-byte loads (through L1,
      // so a row another group of this SM read recently may hit there).
      const float4* src = reinterpret_cast<const float4*>(choice + (size_t)cur * ld);
      float4* dst = reinterpret_cast<float4*>(srow);
      for (int i = tg; i < (ld >> 2); i += NT) dst[i] = src[i];
      group_wait();
    } else {
      bulk_load_if(role == 0, srow_a, choice + (size_t)cur * ld, row_bytes, bar);
      if (!mbar_try_wait(bar, phase) && role >= 0 && !mbar_wait_bounded(bar, phase)) {
        // stale data and no further copies from here on; the status word says so
        role = -2 - (int)phase;
        atomicOr(&I.st->status, kStatusTimeout);
      }
      phase ^= 1u;
    }
    const float* row = srow;

    uint32_t mx;  // 0: no score or key decides
    int next;
    // A group of four consecutive cities (C and base are multiples of 4)
    // shares one Philox call.
    auto group_draw = [&](int g) {
      return philox4x32_10((uint32_t)s, (uint32_t)ant, iter, 1u + (uint32_t)((base >> 2) + g),
                           (uint32_t)seed, (uint32_t)(seed >> 32));
    };
    // its weight bits, 0 where visited (entries at or beyond ld hold stale
    // data; their tabu bits are set)
    auto group_weights = [&](int g, uint32_t (&wv)[4]) {
      const uint4 t = *reinterpret_cast<const uint4*>(row + base + 4 * g);
      uint32_t word = vis[0];
#pragma unroll
      for (int w = 1; w < NW; ++w)
        if (w == (g >> 3)) word = vis[w];
      word >>= (4 * g) & 31;
      wv[0] = word & 1u ? 0u : t.x;
      wv[1] = word & 2u ? 0u : t.y;
      wv[2] = word & 4u ? 0u : t.z;
      wv[3] = word & 8u ? 0u : t.w;
    };
    if constexpr (R == 1) {
      // Scores fl(u_j w_j), u_j <= 1: a score is at most its weight, so a
      // group whose largest open weight is below the best score so far needs
      // no random numbers.  Every lane starts with its heaviest group, the
      // warp's best score then leaves a few groups in a few lanes.  (Drawing
      // for every city took 788e6 warp-instructions at n = 1002 and 1.74 ms.)
      constexpr int NGC = C / 4;
      uint32_t gm[NGC];  // largest open weight of each group
      uint32_t top = 0u, rem = 0u;
      int g = 0;
#pragma unroll
      for (int i = 0; i < NGC; ++i) {
        uint32_t wv[4];
        group_weights(i, wv);
        gm[i] = max(max(wv[0], wv[1]), max(wv[2], wv[3]));
        if (gm[i] > top) {
          top = gm[i];
          g = i;
        }
        rem |= gm[i] ? 1u << i : 0u;
      }
      uint32_t bs = 0u, bj = 0xffffffffu, best = 0u;  // score bits order like scores
      bool mine = NGC == 1 || rem != 0u;
      do {
        if (mine) {
          const Philox4 x = group_draw(g);
          const uint32_t xs[4] = {x.x0, x.x1, x.x2, x.x3};
          uint32_t wv[4];
          group_weights(g, wv);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t sb =
                __float_as_uint(__fmul_rn(candidate_uniform_of(xs[e]), __uint_as_float(wv[e])));
            const uint32_t j = (uint32_t)(base + 4 * g + e);
            if (sb > bs || (sb == bs && sb != 0u && j < bj)) {
              bs = sb;
              bj = j;
            }
          }
          rem &= ~(1u << g);
        }
        best = seg.max_u32(bs);
#pragma unroll
        for (int i = 0; i < NGC; ++i)
          if (gm[i] < best) rem &= ~(1u << i);
        mine = rem != 0u;
        g = __ffs(rem) - 1;
      } while (NGC > 1 && seg.ballot(mine));
      bj = seg.min_u32(bs == best ? bj : 0xffffffffu);
      // (score bits << 32) | ~index: max = best score, lowest index
      uint64_t key = best ? ((uint64_t)best << 32) | (uint32_t)(0xffffffffu - bj) : 0ull;
      if (G > 1) {
        if (hl == 0) gs->wsum[wg] = key;
        group_sync(bar_id, NT);
#pragma unroll
        for (int w = 0; w < G; ++w) key = gs->wsum[w] > key ? gs->wsum[w] : key;
      }
      mx = key != 0 ? 1u : 0u;  // 0: every score is 0, the lowest unvisited city
      next = (int)(0xffffffffu - (uint32_t)key);
    }
    if constexpr (R == 2) {
      // Keys fl(E_j / w_j); non-negative floats order like their bits.  Since
      // E = -ln u >= 1 - u, a city's key can only be below the best so far if
      // 1 - u <= best w, a conversion and a multiply-add on the random word x
      // (u = (floor(x / 2^8) + 1) 2^-24, so 1 - u >= 1 - (x + 256) 2^-32; the
      // slack of 2048 in 2^32 and 2^-18 of best covers that, the roundings and
      // E's 2.5 ulp).  Only cities that pass get the logarithm and the
      // division.  Best keys below 2^-92 count as 2^-92: heavier weights than
      // 2^92 pass, whatever underflows.  (The logarithm and division for
      // every open city took 2.58e9 warp-instructions at n = 1002, 6.29 ms;
      // this 2.93 ms, with the loop unrolled three or nine times 3.01 and 3.50.)
      constexpr uint32_t kInf = 0x7f800000u;
      uint32_t bkey = kInf, bj = 0xffffffffu;  // the lane's smallest key and its city
      float reach = __uint_as_float(kInf);     // best 2^32 (1 + 2^-18) over the warp
#pragma unroll 1
      for (int g = 0; g < C / 4; ++g) {
        const Philox4 x = group_draw(g);
        const uint32_t xs[4] = {x.x0, x.x1, x.x2, x.x3};
        uint32_t wv[4];
        group_weights(g, wv);
        uint32_t pass = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (__uint2float_rn(xs[e]) >= __fmaf_rn(-reach, __uint_as_float(wv[e]), 4294965248.0f))
            pass |= 1u << e;
        if (seg.ballot(pass != 0u)) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float w = __uint_as_float(wv[e]);
            if (((pass >> e) & 1u) && w > 0.0f) {
              const uint32_t kb = __float_as_uint(__fdiv_rn(race_exponential(xs[e]), w));
              if (kb < bkey) {
                bkey = kb;
                bj = (uint32_t)(base + 4 * g + e);
              }
            }
          }
          reach = fmaxf(__fmul_rn(__uint_as_float(seg.min_u32(bkey)), 4294983680.0f), 0x1p-60f);
        }
      }
      const uint32_t best = seg.min_u32(bkey);
      bj = seg.min_u32(bkey == best ? bj : 0xffffffffu);
      uint64_t key = ((uint64_t)best << 32) | bj;
      if (G > 1) {
        if (hl == 0) gs->wsum[wg] = key;
        group_sync(bar_id, NT);
#pragma unroll
        for (int w = 0; w < G; ++w) key = gs->wsum[w] < key ? gs->wsum[w] : key;
      }
      // no finite key: zero weights and overflowing keys are all +inf
      mx = (uint32_t)(key >> 32) < kInf ? 1u : 0u;
      next = (int)(uint32_t)key;
    }
    if (mx == 0u) {
      // Every unvisited weight is zero: the lowest-index unvisited city.
      uint32_t cand = 0xffffffffu;
#pragma unroll
      for (int w = NW - 1; w >= 0; --w) {
        const uint32_t fr = ~vis[w];
        if (fr) cand = (uint32_t)(base + 32 * w + __ffs(fr) - 1);
      }
      cand = seg.min_u32(cand);
      if (G > 1) {
        if (hl == 0) gs->wmin[wg] = (int)cand;
        group_sync(bar_id, NT);
#pragma unroll
        for (int w = 0; w < G; ++w) cand = min(cand, (uint32_t)gs->wmin[w]);
      }
      next = (int)cand;
    }

    // A city outside [0, n) can only come from a defect; record it and stay
    // in bounds instead of reading past the matrix.
    if ((unsigned)next >= (unsigned)n) {
      if (tg == 0) atomicOr(&I.st->status, kStatusBadTour);
      next = start;
    }
    const int li = next - base;
    if (li >= 0 && li < C) {
#pragma unroll
      for (int w = 0; w < NW; ++w)
        if (w == (li >> 5)) vis[w] |= 1u << (li & 31);
    }
    if (tg == 0) tour[s] = next;
    cur = next;
    group_wait();
  }
  // the copy in flight, again with a limit
  if (role < 0) mbar_wait_bounded(bar, (uint32_t)role & 1u);
  if (tg == 0) tour[n] = start;
  group_wait();

  // C^k (Section II) and the per-city neighbour buckets.
  long long len = 0;
  for (int s = tg; s < n; s += NT) {
    const int a = tour[s], b = tour[s + 1];
    const int p = tour[s == 0 ? n - 1 : s - 1];
    len += I.dist[(size_t)a * ld + b];
    I.nbr[(size_t)a * I.ldm + ant] = ((uint32_t)p << 16) | (uint32_t)b;
  }
#pragma unroll
  for (int o = H / 2; o > 0; o >>= 1) len += seg.shfl_xor(len, o);
  if (G > 1) {
    if (hl == 0) gs->wlen[wg] = len;
    group_sync(bar_id, NT);
    len = 0;
#pragma unroll
    for (int w = 0; w < G; ++w) len += gs->wlen[w];
  }
  if (tg == 0) I.lens[ant] = len;
}

}  // namespace aco

#include "construct_phased.cuh"

namespace aco {

// Placement of one thread: its ant group within the CTA and its index tg
// within the group.
template <int G, int H>
__device__ __forceinline__ void group_of_thread(int& grp, int& tg) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (H == 32) {
    grp = threadIdx.x / (32 * G);
    tg = threadIdx.x % (32 * G);
  } else {
    grp = warp * (32 / H) + lane / H;
    tg = lane % H;
  }
}

// One CTA holds groups_per_cta<G, H>(blockDim.x / 32) ant groups; dynamic
// shared memory holds one StageLayout<C, G, H> per group.
template <int C, int G, int H, int R>
__global__ void __launch_bounds__(256) construct_rule_kernel(Instance I) {
  __shared__ GroupSmem gs[kMaxGroupsPerCta];
  extern __shared__ __align__(16) unsigned char stage[];
  int grp, tg;
  group_of_thread<G, H>(grp, tg);
  const int ant = blockIdx.x * groups_per_cta<G, H>(blockDim.x >> 5) + grp;
  if (ant >= I.m) return;
  float* srow = reinterpret_cast<float*>(stage + grp * StageLayout<C, G, H>::kBytes);
  construct_ant_rule<C, G, H, R>(I, ant, tg, Seg<H>(threadIdx.x & 31), &gs[H == 32 ? grp : 0], 1 + grp,
                            srow, I.stage != 0);
}

// The Eq. 1 walk with compaction (construct_phased.cuh), one group of H lanes
// (or two warps) per ant.  Its phases are inlined into one body; without a
// ceiling the register allocator hoists the row's loads.  The ceilings were
// chosen by measurement on the GB300: 64 up to C = 36, where the shared
// memory of a row leaves room for 32 ants an SM (with lists at C/2 still: n =
// 1002, m = 4864 1.58 ms against 1.98 at 72, a step of 256 instances 14.3 ms
// against 14.5; 48 and 56 are 1-2 % slower everywhere); above, the rows limit
// the ants and 128 costs nothing (n = 2392 3.30 ms; 96: 3.32, 72: 3.34).
// Two warps per ant (n > 2432) would hold 2 x 13 warps at C = 52 and 2 x 11 at
// C = 60 by their rows: ceilings that let them all reside (n = 3100 11.6 ms at
// 128, 9.73 at 72).
template <int C, int G>
struct PhasedRegs {
  static constexpr int v = C <= 36               ? 64
                           : G == 1              ? 128
                           : C <= 44             ? 64
                           : C <= 52             ? 72
                           : C <= 60             ? 80
                                                 : 96;
};

template <int C, int G, int H>
__global__ void __maxnreg__((PhasedRegs<C, G>::v)) construct_phased_kernel(Instance I) {
  __shared__ GroupSmem gs[kMaxGroupsPerCta];
  extern __shared__ __align__(16) unsigned char stage[];
  int grp, tg;
  group_of_thread<G, H>(grp, tg);
  const int ant = blockIdx.x * groups_per_cta<G, H>(blockDim.x >> 5) + grp;
  if (ant >= I.m) return;
  construct_ant_phased<C, G, H, false>(
      I, ant, tg, Seg<H>(threadIdx.x & 31), &gs[H == 32 ? grp : 0], 1 + grp,
      reinterpret_cast<float*>(stage + grp * StageLayout<C, G, H>::kBytes), I.stage != 0);
}

template <int C, int G, int H>
__global__ void __maxnreg__((PhasedRegs<C, G>::v))
    construct_phased_items_kernel(const Instance* __restrict__ insts,
                                  const int2* __restrict__ items, int count, int lane_copy) {
  __shared__ GroupSmem gs[kMaxGroupsPerCta];
  extern __shared__ __align__(16) unsigned char stage[];
  int grp, tg;
  group_of_thread<G, H>(grp, tg);
  const int idx = blockIdx.x * groups_per_cta<G, H>(blockDim.x >> 5) + grp;
  if (idx >= count) return;
  const int2 it = items[idx];
  construct_ant_phased<C, G, H, true>(
      insts[it.x], it.y, tg, Seg<H>(threadIdx.x & 31), &gs[H == 32 ? grp : 0], 1 + grp,
      reinterpret_cast<float*>(stage + grp * StageLayout<C, G, H>::kBytes), lane_copy != 0);
}

// Dynamic shared memory for a CTA of `warps` warps, with the opt-in above
// 48 KB set once per kernel and device.
template <int C, int G, int H, bool kItems, int R = 0>
inline size_t construct_smem_setup(int warps) {
  const size_t bytes = (size_t)groups_per_cta<G, H>(warps) * StageLayout<C, G, H>::kBytes;
  static std::atomic<unsigned long long> done{0};
  once_per_device(done, [] {
    const int most = groups_per_cta<G, H>(8) * StageLayout<C, G, H>::kBytes;
    if constexpr (kItems)
      return cudaFuncSetAttribute(construct_phased_items_kernel<C, G, H>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    else if constexpr (R == 0)
      return cudaFuncSetAttribute(construct_phased_kernel<C, G, H>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    else
      return cudaFuncSetAttribute(construct_rule_kernel<C, G, H, R>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  });
  return bytes;
}

}  // namespace aco
