// Ant Colony System (Dorigo and Gambardella, IEEE Trans. Evol. Comp. 1(1),
// 1997), the ACO variant the paper names as its next target (Section V), on
// the same data layout as the Ant System:
//  - the pseudo-random proportional rule: at step s ant k draws Philox
//    (s, k, iteration, 0); it exploits when word x2 < floor(q0 2^32), taking
//    the unvisited city of largest choice_info (ties to the lower index), and
//    otherwise samples Eq. 1 by the exact integer roulette;
//  - the local update: the ants move in lockstep, all choosing their s-th
//    city from the same state; then every edge crossed at that step gets
//    tau <- fl(fl((1-xi) tau) + fl(xi tau0)) once per ant that crossed it,
//    in both directions, with its choice_info; the closing edge is the n-th
//    such step;
//  - the global update: only the best-so-far tour's edges get
//    tau <- fl(fl((1-rho) tau) + fl(rho dtau)), dtau = 1/C_bs.
// The colony (m <= 32 ants, the variant's usual m = 10) runs in one CTA, one
// warp per ant, so the per-step lockstep is a CTA barrier; many colonies (a
// pool's Ant Colony System slots) run as one launch of one CTA per colony.
#include "aco_device.cuh"
#include "construct.cuh"
#include "construct_chunks.h"
#include "kernels.h"

namespace aco {

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

__device__ __forceinline__ unsigned long long warp_incl_scan_u64(unsigned long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long w = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += w;
  }
  return v;
}

// One local update of one cell.
__device__ __forceinline__ float acs_local(float tau, float keep, float add) {
  return __fadd_rn(__fmul_rn(keep, tau), add);
}

// Ant's next city from `cur` by its whole row: the heaviest unvisited city
// (exploit), or Eq. 1 by the integer roulette with the draw x.  One warp.
__device__ __forceinline__ int acs_dense_choice(const Instance& I, int cur, const uint32_t* seen,
                                                int lane, const Philox4& x, bool exploit) {
  const int n = I.n, ld = I.ld;
  const float* row = I.choice + (size_t)cur * ld;
  // Lane l reads cities 4l..4l+3 of every 128 with one 16-byte load (ld
  // is a multiple of 4, so the load stays inside the row); the three
  // passes read the same lines, the later two from L1.  Loads after the
  // CTA barrier see the local updates of the previous step.
  // Pass 1: the largest unvisited weight, ties to the lower index.  The
  // bits of non-negative floats order like their values; an unvisited
  // city's key is bits(w) + 1 and a visited one's 0, so a zero weight
  // still beats every visited city.  Each lane visits its cities in
  // ascending order and keeps the first of its largest keys; the warp
  // reduction breaks ties by index.
  uint32_t bkey = 0u;
  int bj = 0;
#pragma unroll 4
  for (int j0 = 4 * lane; j0 < n; j0 += 128) {
    const uint4 w4 = *reinterpret_cast<const uint4*>(row + j0);
    const uint32_t fr = ~seen[j0 >> 5] >> (j0 & 31);  // 4 free bits (j0 % 4 == 0)
    const uint32_t wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t kk = ((fr >> e) & 1u) && j0 + e < n ? wv[e] + 1u : 0u;
      if (kk > bkey) {
        bkey = kk;
        bj = j0 + e;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint32_t ok = __shfl_xor_sync(FULL, bkey, o);
    const int oj = __shfl_xor_sync(FULL, bj, o);
    if (ok > bkey || (ok == bkey && oj < bj)) {
      bkey = ok;
      bj = oj;
    }
  }
  const uint32_t mbits = bkey - 1u;  // bkey >= 1: a city is unvisited
  int next = bj;
  if (!exploit && mbits != 0u) {
    // Eq. 1 by the integer roulette: q_j = floor(w_j 2^(45 - ilogb M)),
    // T = floor(r Q / 2^64), the first j whose prefix sum exceeds T.
    // (the three-FMA quantiser of the construction kernel: exact, branch-free)
    float f1, f1s, f2;
    quant_factors(kRouletteBits - 1 - exponent_of_bits(mbits), f1, f1s, f2);
    unsigned long long part = 0ull;
#pragma unroll 4
    for (int j0 = 4 * lane; j0 < n; j0 += 128) {
      const uint4 w4 = *reinterpret_cast<const uint4*>(row + j0);
      const uint32_t fr = ~seen[j0 >> 5] >> (j0 & 31);
      const uint32_t wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        part += quant_value(((fr >> e) & 1u) && j0 + e < n ? wv[e] : 0u, f1, f1s, f2);
    }
    const unsigned long long Q = warp_sum_u64(part);
    const unsigned long long r = ((unsigned long long)x.x1 << 32) | x.x0;
    const unsigned long long T = __umul64hi(r, Q);
    // Pass 3: 256 cities at a time in ascending order, lane l holding
    // cities 8l..8l+7 of the chunk; a warp scan of the lanes' eight-city
    // sums finds the lane, the lane its city.
    unsigned long long running = 0ull;
    for (int c0 = 0; c0 < n; c0 += 256) {
      const int j0 = c0 + 8 * lane;
      unsigned long long q[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) q[e] = 0ull;
      if (j0 < n) {
        const uint32_t fr = ~seen[j0 >> 5] >> (j0 & 31);  // 8 free bits (j0 % 8 == 0)
        const uint4 wa = *reinterpret_cast<const uint4*>(row + j0);
        // the second half only if it starts inside the row (ld % 4 == 0)
        const uint4 wb = j0 + 4 < n ? *reinterpret_cast<const uint4*>(row + j0 + 4)
                                    : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
        for (int e = 0; e < 8; ++e)
          q[e] = quant_value(((fr >> e) & 1u) && j0 + e < n ? wv[e] : 0u, f1, f1s, f2);
      }
      unsigned long long mine = 0ull;
#pragma unroll
      for (int e = 0; e < 8; ++e) mine += q[e];
      const unsigned long long incl = warp_incl_scan_u64(mine, lane);
      const unsigned long long total = __shfl_sync(FULL, incl, 31);
      if (running + total > T) {
        const unsigned hit = __ballot_sync(FULL, running + incl > T);
        const int L = __ffs(hit) - 1;
        int pick = 0;
        if (lane == L) {
          // the first e whose inclusive prefix exceeds T: count the
          // prefixes that do not
          unsigned long long c = running + incl - mine;
#pragma unroll
          for (int e = 0; e < 7; ++e) {
            c += q[e];
            pick += c <= T ? 1 : 0;
          }
        }
        next = c0 + 8 * L + __shfl_sync(FULL, pick, L);
        break;
      }
      running += total;
    }
  }
  return next;
}

// One colony in one CTA.  Warp k < m builds ant k's tour; further warps (a
// launch over colonies with different m sizes the CTA for the largest) take
// part in the lockstep barriers only.  kNN: with the instance's
// nearest-neighbour lists (I.nn entries): lane l holds entry l of the
// current city's list and its current choice_info value.
template <bool kNN>
__device__ __forceinline__ void acs_construct_body(const Instance& I, uint32_t* acs_seen,
                                                   uint32_t* s_edge) {
  const int n = I.n, ld = I.ld, m = I.m;
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool active = k < m;
  const int words = (n + 31) >> 5;
  uint32_t* seen = acs_seen + (size_t)k * words;
  const uint32_t it = (uint32_t)I.st->iteration;
  const float tau0 = I.st->acs_tau0;
  const float keep = __fsub_rn(1.0f, I.acs_xi), add = __fmul_rn(I.acs_xi, tau0);
  int32_t* tour = I.tours + (size_t)k * I.ldt;

  int start = 0;
  if (active) {
    for (int w = lane; w < words; w += 32) seen[w] = 0u;
    __syncwarp();
    const Philox4 x0 = step_draw(I.seed, 0u, (uint32_t)k, it);
    start = (int)__umulhi(x0.x0, (uint32_t)n);
    if (lane == 0) {
      seen[start >> 5] |= 1u << (start & 31);
      tour[0] = start;
    }
    __syncwarp();
  }
  int cur = start;
  for (int s = 1; s <= n; ++s) {
    int next = start;
    bool listed = false;  // chosen among the list entries
    if constexpr (kNN) {
      if (active && s < n) {
        const Philox4 x = step_draw(I.seed, (uint32_t)s, (uint32_t)k, it);
        const float* row = I.choice + (size_t)cur * ld;
        int j = 0;
        uint32_t wb = 0u;
        bool unv = false;
        if (lane < I.nn) {
          j = I.nnlist[(size_t)cur * kNnStride + lane];
          wb = __float_as_uint(row[j]);  // after this colony's local updates
          unv = !((seen[j >> 5] >> (j & 31)) & 1u);
        }
        const unsigned any = __ballot_sync(FULL, unv);
        if (any) {
          listed = true;
          if ((unsigned long long)x.x2 < I.acs_threshold) {
            // the heaviest unvisited entry, ties to the earlier entry
            const uint32_t key = unv ? wb + 1u : 0u;
            const uint32_t top = __reduce_max_sync(FULL, key);
            next = __shfl_sync(FULL, j, __ffs(__ballot_sync(FULL, key == top)) - 1);
          } else {
            // Eq. 1 over the unvisited entries, in list order
            const uint32_t wm = unv ? wb : 0u;
            const uint32_t mx = __reduce_max_sync(FULL, wm);
            if (mx == 0u) {
              next = __shfl_sync(FULL, j, __ffs(any) - 1);
            } else {
              float f1, f1s, f2;
              quant_factors(kRouletteBits - 1 - exponent_of_bits(mx), f1, f1s, f2);
              const unsigned long long incl =
                  warp_incl_scan_u64(quant_value(wm, f1, f1s, f2), lane);
              const unsigned long long r = ((unsigned long long)x.x1 << 32) | x.x0;
              const unsigned long long T = __umul64hi(r, __shfl_sync(FULL, incl, 31));
              next = __shfl_sync(FULL, j, max(__ffs(__ballot_sync(FULL, incl > T)) - 1, 0));
            }
          }
        }
      }
    }
    if (active && s < n && !listed) {
      const Philox4 x = step_draw(I.seed, (uint32_t)s, (uint32_t)k, it);
      // with lists, every entry is visited here: the heaviest city, always
      next = acs_dense_choice(I, cur, seen, lane, x, kNN || (unsigned long long)x.x2 < I.acs_threshold);
      if ((unsigned)next >= (unsigned)n) {  // cannot happen while a city is unvisited
        if (lane == 0) atomicOr(&I.st->status, kStatusBadTour);
        next = start;
      }
      // The next step reads row `next`: start bringing it into L1 now (one
      // 128-byte line per lane and round), while this ant waits at the
      // barrier for the others.  Only this CTA writes the colony's matrices,
      // through the same L1, so the lines the local updates change stay
      // current; the prefetch is a hint and changes no result.
      if (s + 1 < n) {
        const float* nrow = I.choice + (size_t)next * ld;
        for (int f = 32 * lane; f < n; f += 32 * 32)
          asm volatile("prefetch.global.L1 [%0];" ::"l"(nrow + f));
      }
    }
    if constexpr (kNN) {
      if (active && s < n && (unsigned)next >= (unsigned)n) {  // cannot happen
        if (lane == 0) atomicOr(&I.st->status, kStatusBadTour);
        next = start;
      }
    }
    // lockstep: every ant has chosen from the same state; then the local
    // updates of this step, one writer per distinct edge applying it once
    // per ant that crossed the edge
    const uint32_t lo = (uint32_t)min(cur, next), hi = (uint32_t)max(cur, next);
    const size_t ab = (size_t)lo * ld + hi, ba = (size_t)hi * ld + lo;
    // The crossed cell's tau and eta^beta, read before the barrier: only this
    // step's writer of the edge stores to it, after the barrier, so the
    // values read here are the current ones and the load latency overlaps
    // the other ants' selection.
    float t = 0.0f, h = 0.0f;
    if (active && lane == 0) {
      s_edge[k] = (lo << 16) | hi;
      t = __ldcg(I.tau + ab);
      h = I.heta[ab];
    }
    __syncthreads();
    if (active) {
      const uint32_t e = s_edge[k];
      const unsigned same = __ballot_sync(FULL, lane < m && s_edge[lane < m ? lane : 0] == e);
      if (lane == 0 && __ffs(same) - 1 == k) {
        for (int c = __popc(same); c > 0; --c) t = acs_local(t, keep, add);
        const float ch = choice_of(t, h, I.alpha);
        I.tau[ab] = t;
        I.tau[ba] = t;
        I.choice[ab] = ch;
        I.choice[ba] = ch;
      }
      if (lane == 0 && s < n) {
        seen[next >> 5] |= 1u << (next & 31);
        tour[s] = next;
      }
    }
    __syncthreads();
    cur = next;
  }
  if (!active) return;
  if (lane == 0) tour[n] = start;
  __syncwarp();
  long long len = 0;
  for (int s = lane; s < n; s += 32) len += I.dist[(size_t)tour[s] * ld + tour[s + 1]];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(FULL, len, o);
  if (lane == 0) I.lens[k] = len;
}

// Cells that other warps of the CTA may be reading or storing to.
__device__ __forceinline__ float load_cell(const float* p) {
  float v;
  asm volatile("ld.relaxed.cta.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void store_cell(float* p, float v) {
  asm volatile("st.relaxed.cta.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

// Order this thread's global stores before later bulk copies of what they wrote.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// The same colony without lists, for n <= 128 B: each warp brings its ant's
// current row into shared memory with one bulk copy and its registers (lane l
// holds cities 128 j + 4 l + e), and keeps the tabu bits in one register per
// eight blocks.  One colony is a chain of n lockstep steps on one SM, so what
// counts is a step's latency:
//  - the next row and the crossed edge's tau and eta^beta are fetched together
//    as soon as the city is known, before the barriers; the few cells of the
//    row that this step's local updates change are put in afterwards (the
//    edges and their new choice_info are in shared memory by then);
//  - an exploiting step is one max pass and two REDUX (value, lowest index);
//  - an exploring step forms the prefix sums in single precision, one warp
//    scan per block of 128 cities side by side, and the lane whose city holds
//    the target with the rounding error to spare names it (see eq1_phase in
//    construct_phased.cuh for why that is the integer roulette's city);
//    otherwise the step runs the integer roulette (acs_dense_choice).
// m = 10, GB300, ms per construction, every pass over the row from L1 / rows
// loaded by the lanes / this kernel: n = 48 0.083 / 0.054 / 0.057, n = 200
// 0.374 / 0.200 / 0.221, n = 517 1.29 / 1.01 / 0.66, n = 1002 3.89 / 2.32 /
// 1.42, n = 2392 14.3 / 11.3 / 5.69, n = 4096 35.8 / 35.3 / 18.1 (loads by ten
// warps queue in the SM's load unit for 1400 cycles of a step at n = 1002); a
// step of 256 colonies 4.59 / 2.89 / 1.84.
template <int B>
__device__ __forceinline__ void acs_rows_body(const Instance& I, uint32_t* acs_seen,
                                              uint32_t* s_edge, float* s_choice,
                                              unsigned long long* s_bar, float* rows) {
  constexpr int NW = (B + 7) / 8;
  // roundings: the prefix before the lane's cities and, inside the target,
  // the whole sum (four cities, the scan, the blocks each); the lane's own
  // cities; the target and the differences, two to spare
  constexpr float kEps = (float)(2 * (2 + 5 + B) + 4 + 9) * 0x1p-24f;
  const int n = I.n, ld = I.ld, m = I.m;
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool active = k < m;
  const int words = (n + 31) >> 5;
  uint32_t* seen = acs_seen + (size_t)k * words;  // for the integer roulette
  const uint32_t it = (uint32_t)I.st->iteration;
  const float keep = __fsub_rn(1.0f, I.acs_xi), add = __fmul_rn(I.acs_xi, I.st->acs_tau0);
  int32_t* tour = I.tours + (size_t)k * I.ldt;

  float4 v[B];
  uint32_t vis[NW];  // bit 4 (j % 8) + e of word j / 8: city 128 j + 4 lane + e
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    vis[w] = 0u;
#pragma unroll
    for (int b = 0; b < 32; ++b)
      if (128 * (8 * w + b / 4) + 4 * lane + b % 4 >= n) vis[w] |= 1u << b;
  }
  auto mark = [&](int c) {
    if (lane == ((c >> 2) & 31)) {
#pragma unroll
      for (int w = 0; w < NW; ++w)
        if (w == (c >> 10)) vis[w] |= 1u << (4 * ((c >> 7) & 7) + (c & 3));
    }
    if (lane == 0) seen[c >> 5] |= 1u << (c & 31);
  };
  float* srow = rows + (size_t)k * ld;
  const uint32_t srow_a = smem_u32(srow), bar = smem_u32(s_bar + k);
  uint32_t parity = 0u;
  int role = lane;  // 0 issues the copies; -2 minus the parity of a wait that gave up
  auto load_row = [&](int c) {
    bulk_load_if(role == 0, srow_a, I.choice + (size_t)c * ld, (uint32_t)ld * 4u, bar);
  };
  // cells of the row that the last step's local updates changed: the ants
  // whose edges touch the current city, and their edges
  unsigned touch = 0u;
  uint32_t e = 0xffffffffu;

  int start = 0;
  if (active) {
    for (int w = lane; w < words; w += 32) seen[w] = 0u;
    __syncwarp();
    const Philox4 x0 = step_draw(I.seed, 0u, (uint32_t)k, it);
    start = (int)__umulhi(x0.x0, (uint32_t)n);
    if (lane == 0) {
      tour[0] = start;
      mbar_init(bar, 1);
      fence_mbar_init();
    }
    __syncwarp();
    mark(start);
    load_row(start);
  }
  int cur = start;
  uint32_t w1 = 0u, w2 = 0u;  // Philox words x1, x2 of this lane's step of the window
  for (int s = 1; s <= n; ++s) {
    int next = start;
    float t = 0.0f, h = 0.0f;
    if (active) {
      if (s < n) {
        const int off = (s - 1) & 31;
        if (off == 0) {
          const Philox4 x = step_draw(I.seed, (uint32_t)(s + lane), (uint32_t)k, it);
          w1 = x.x1;
          w2 = x.x2;
        }
        const uint32_t x1 = __shfl_sync(FULL, w1, off), x2 = __shfl_sync(FULL, w2, off);
        const bool exploit = (unsigned long long)x2 < I.acs_threshold;
        if (!mbar_try_wait(bar, parity) && role >= 0 && !mbar_wait_bounded(bar, parity)) {
          // stale data and no further copies from here on; the status word says so
          role = -2 - (int)parity;
          atomicOr(&I.st->status, kStatusTimeout);
        }
        parity ^= 1u;
        if (touch) {
          do {
            const int i = __ffs(touch) - 1;
            touch &= touch - 1;
            const uint32_t ei = __shfl_sync(FULL, e, i);
            if (lane == 0)
              srow[(ei >> 16) == (uint32_t)cur ? ei & 0xffffu : ei >> 16] = s_choice[i];
          } while (touch);
          if (lane == 0) fence_proxy_async_smem();  // before the next copy into the row
          __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < B; ++j)
          v[j] = 128 * j + 4 * lane < n
                     ? *reinterpret_cast<const float4*>(srow + 128 * j + 4 * lane)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
        // visited cities: below every weight, or nothing in a sum
        const float shut = exploit ? -1.0f : 0.0f;
#pragma unroll
        for (int j = 0; j < B; ++j) {
          const uint32_t b = vis[j / 8] >> (4 * (j % 8));
          if (b & 1u) v[j].x = shut;
          if (b & 2u) v[j].y = shut;
          if (b & 4u) v[j].z = shut;
          if (b & 8u) v[j].w = shut;
        }
        if (exploit) {
          float top = -1.0f;
#pragma unroll
          for (int j = 0; j < B; ++j)
            top = fmaxf(top, fmaxf(fmaxf(v[j].x, v[j].y), fmaxf(v[j].z, v[j].w)));
          // floats >= 0 order like their bits, and -1 is below them
          const int best = __reduce_max_sync(FULL, __float_as_int(top));
          uint32_t c = 0xffffffffu;
          if (__float_as_int(top) == best) {
#pragma unroll
            for (int j = B - 1; j >= 0; --j) {
              if (v[j].w == top) c = 128 * j + 3;
              if (v[j].z == top) c = 128 * j + 2;
              if (v[j].y == top) c = 128 * j + 1;
              if (v[j].x == top) c = 128 * j;
            }
            c += 4 * lane;
          }
          next = (int)__reduce_min_sync(FULL, c);
        } else {
          float in[B], base[B + 1];
#pragma unroll
          for (int j = 0; j < B; ++j)
            in[j] = __fadd_rn(__fadd_rn(v[j].x, v[j].y), __fadd_rn(v[j].z, v[j].w));
          const Seg<32> seg(lane);
#pragma unroll
          for (int j = 0; j < B; ++j) in[j] = seg.inclusive_scan_f(in[j]);
          base[0] = 0.0f;
#pragma unroll
          for (int j = 0; j < B; ++j) base[j + 1] = __fadd_rn(base[j], __shfl_sync(FULL, in[j], 31));
          const float S = base[B];
          const float target = __fmul_rn(__fmul_rn(__uint2float_rn(x1), 0x1p-32f), S);
          const float err = S >= 0x1p-120f ? __fmul_rn(kEps, S) : __int_as_float(0x7f800000);
          int pick = -1;
#pragma unroll
          for (int j = 0; j < B; ++j) {
            if (target >= base[j] && target < base[j + 1]) {
              const float in_j = __fsub_rn(target, base[j]);
              const float mine = __fadd_rn(__fadd_rn(v[j].x, v[j].y), __fadd_rn(v[j].z, v[j].w));
              const float x = __fsub_rn(in_j, __fsub_rn(in[j], mine));
              const float hi_t = __fadd_rn(x, err), lo_t = __fsub_rn(x, err);
              const float c1 = v[j].x, c2 = __fadd_rn(c1, v[j].y), c3 = __fadd_rn(c2, v[j].z),
                          c4 = __fadd_rn(c3, v[j].w);
              if (c1 > hi_t && 0.0f < lo_t) pick = 128 * j;
              if (c2 > hi_t && c1 < lo_t) pick = 128 * j + 1;
              if (c3 > hi_t && c2 < lo_t) pick = 128 * j + 2;
              if (c4 > hi_t && c3 < lo_t) pick = 128 * j + 3;
            }
          }
          const uint32_t sure = __ballot_sync(FULL, pick >= 0);
          if (sure) {
            const int L = __ffs(sure) - 1;
            next = __shfl_sync(FULL, pick, L) + 4 * L;
          } else {
            const Philox4 x = step_draw(I.seed, (uint32_t)s, (uint32_t)k, it);
            next = acs_dense_choice(I, cur, seen, lane, x, false);
          }
        }
        if ((unsigned)next >= (unsigned)n) {  // cannot happen while a city is unvisited
          if (lane == 0) atomicOr(&I.st->status, kStatusBadTour);
          next = start;
        }
        __syncwarp();  // every lane has read the row
        if (s + 1 < n) load_row(next);
        mark(next);
        if (lane == 0) tour[s] = next;
      }
      if (lane == 0) {
        const uint32_t lo = (uint32_t)min(cur, next), hi = (uint32_t)max(cur, next);
        s_edge[k] = (lo << 16) | hi;
        t = load_cell(I.tau + (size_t)lo * ld + hi);
        h = I.heta[(size_t)lo * ld + hi];
      }
    }
    // lockstep: every ant has chosen from the same state; then the local
    // updates, once per ant that crossed the edge, stored by the first of them
    __syncthreads();
    if (active) {
      const uint32_t mine = s_edge[k];
      e = 0xffffffffu;
      if (lane < m) e = s_edge[lane];
      const unsigned same = __ballot_sync(FULL, e == mine);
      if (lane == 0) {
        for (int c = __popc(same); c > 0; --c) t = acs_local(t, keep, add);
        const float ch = choice_of(t, h, I.alpha);
        s_choice[k] = ch;
        if (__ffs(same) - 1 == k) {
          const size_t lo = mine >> 16, hi = mine & 0xffffu;
          store_cell(I.tau + lo * ld + hi, t);
          store_cell(I.tau + hi * ld + lo, t);
          store_cell(I.choice + lo * ld + hi, ch);
          store_cell(I.choice + hi * ld + lo, ch);
          fence_proxy_async_global();
        }
      }
      // (the ant's own edge leads to a visited city)
      touch = __ballot_sync(FULL, lane < m && e != mine &&
                                      ((e >> 16) == (uint32_t)next || (e & 0xffffu) == (uint32_t)next));
    }
    __syncthreads();
    cur = next;
  }
  if (!active) return;
  // the copy in flight, again with a limit
  if (role < 0) mbar_wait_bounded(bar, (uint32_t)role & 1u);
  if (lane == 0) tour[n] = start;
  __syncwarp();
  long long len = 0;
  for (int s = lane; s < n; s += 32) len += I.dist[(size_t)tour[s] * ld + tour[s + 1]];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(FULL, len, o);
  if (lane == 0) I.lens[k] = len;
}

// Threads per colony that leave the registers for B blocks: the row, its
// sums and prefix sums.
template <int B>
constexpr int kAcsRowThreads = B <= 4 ? 1024 : (B <= 8 ? 512 : 320);

template <int B>
__global__ void __launch_bounds__(kAcsRowThreads<B>, 1) acs_rows_kernel(Instance I) {
  extern __shared__ __align__(16) float acs_rows[];  // a row per ant, then the tabu bitmaps
  __shared__ uint32_t s_edge[32];
  __shared__ float s_choice[32];
  __shared__ unsigned long long s_bar[32];
  acs_rows_body<B>(I, reinterpret_cast<uint32_t*>(acs_rows + (size_t)I.m * I.ld), s_edge, s_choice,
                   s_bar, acs_rows);
}

template <int B>
__global__ void __launch_bounds__(kAcsRowThreads<B>, 1)
    acs_rows_slots_kernel(const Instance* __restrict__ insts, const int* __restrict__ slots) {
  extern __shared__ __align__(16) float acs_rows[];  // a row per ant, then the tabu bitmaps
  __shared__ uint32_t s_edge[32];
  __shared__ float s_choice[32];
  __shared__ unsigned long long s_bar[32];
  const Instance& I = insts[slots[blockIdx.x]];
  acs_rows_body<B>(I, reinterpret_cast<uint32_t*>(acs_rows + (size_t)I.m * I.ld), s_edge, s_choice,
                   s_bar, acs_rows);
}

template <bool kNN>
__global__ void __launch_bounds__(1024, 1) acs_construct_kernel(Instance I) {
  extern __shared__ uint32_t acs_seen[];  // m tabu bitmaps of (n + 31) / 32 words
  __shared__ uint32_t s_edge[32];         // (min << 16 | max) crossed by ant k
  acs_construct_body<kNN>(I, acs_seen, s_edge);
}

// Many colonies per launch: CTA b runs the colony of slot slots[b] (all of
// them with lists, or all without).
template <bool kNN>
__global__ void __launch_bounds__(1024, 1)
    acs_construct_slots_kernel(const Instance* __restrict__ insts, const int* __restrict__ slots) {
  extern __shared__ uint32_t acs_seen[];
  __shared__ uint32_t s_edge[32];
  acs_construct_body<kNN>(insts[slots[blockIdx.x]], acs_seen, s_edge);
}

// Global update on the best-so-far tour: edge s of the tour per thread from
// `first` in steps of `stride` (each edge of a closed tour of n >= 3 cities
// occurs once).
__device__ __forceinline__ void acs_global_body(const Instance& I, int first, int stride,
                                                bool bump_iteration) {
  const int n = I.n, ld = I.ld;
  const float keep = __fsub_rn(1.0f, I.rho);
  const float dep = __fmul_rn(I.rho, (float)(1.0 / (double)I.st->best_len));
  for (int s = first; s < n; s += stride) {
    const int a = I.best_tour[s], b = I.best_tour[s + 1];
    const size_t ab = (size_t)a * ld + b, ba = (size_t)b * ld + a;
    const float t = __fadd_rn(__fmul_rn(keep, I.tau[ab]), dep);
    const float ch = choice_of(t, I.heta[ab], I.alpha);
    I.tau[ab] = t;
    I.tau[ba] = t;
    I.choice[ab] = ch;
    I.choice[ba] = ch;
  }
  if (bump_iteration) I.st->iteration += 1;
}

__global__ void acs_global_kernel(Instance I) {
  acs_global_body(I, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x,
                  blockIdx.x == 0 && threadIdx.x == 0);
}

__global__ void acs_global_slots_kernel(const Instance* __restrict__ insts,
                                        const int* __restrict__ slots) {
  acs_global_body(insts[slots[blockIdx.x]], threadIdx.x, blockDim.x, threadIdx.x == 0);
}

// Start: tau = tau0 = (float)(1 / (n C_nn)) off the diagonal, choice_info.
__global__ void acs_init_kernel(Instance I) {
  const float tau0 = (float)(1.0 / ((double)I.n * (double)I.st->nn_len));
  const int n = I.n, ld = I.ld;
  const size_t total = (size_t)n * ld;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / ld), j = (int)(e % ld);
    const float t = (j != i && j < n) ? tau0 : 0.0f;
    I.tau[e] = t;
    I.choice[e] = choice_of(t, I.heta[e], I.alpha);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) I.st->acs_tau0 = tau0;
}

cudaError_t launch_acs_init(const Instance& I, int sms, cudaStream_t st) {
  size_t blocks = ((size_t)I.n * I.ld + 255) / 256;
  if (blocks > (size_t)sms * 8) blocks = (size_t)sms * 8;
  acs_init_kernel<<<(int)blocks, 256, 0, st>>>(I);
  return cudaGetLastError();
}

// The row kernels by blocks of 128 cities; false: no kernel holds rows of n
// cities for m ants (n above 512 with more than 16 ants, above 1024 with more
// than 10), and the row is read again in every pass instead.
using AcsBlocks = ChunkList<1, 2, 4, 6, 8, 12, 16, 20, 24, 32>;

// Shared memory of a colony of up to m ants and n cities.
static size_t acs_rows_bytes(int n, int m) {
  return (size_t)m * (((size_t)n + 3) / 4 * 4 * sizeof(float) +
                      ((size_t)n + 31) / 32 * sizeof(uint32_t));
}

constexpr size_t kAcsRowsMost = 224 * 1024;

template <int B, bool kSlots>
static bool acs_rows_ready() {
  static std::atomic<unsigned long long> done{0};
  return once_per_device(done, [] {
           if constexpr (kSlots)
             return cudaFuncSetAttribute(acs_rows_slots_kernel<B>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kAcsRowsMost);
           else
             return cudaFuncSetAttribute(acs_rows_kernel<B>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kAcsRowsMost);
         }) == cudaSuccess;
}

template <int... Bs>
static bool launch_acs_rows(ChunkList<Bs...>, const Instance& I, cudaStream_t st) {
  const size_t smem = acs_rows_bytes(I.n, I.m);
  return smem <= kAcsRowsMost &&
         ((I.n <= 128 * Bs && 32 * I.m <= kAcsRowThreads<Bs> && acs_rows_ready<Bs, false>() &&
           (acs_rows_kernel<Bs><<<1, 32 * I.m, smem, st>>>(I), true)) ||
          ...);
}

// One block width for all colonies of the launch, that of the largest.  A step,
// ms, every pass over the rows from L1 -> this: 256 colonies of n = 100 0.65 ->
// 0.57, one of 1002 and 600 of 100 5.10 -> 2.48, one of 2392 and 1000 of 100
// 17.0 -> 7.6, one of 4096 and 800 of 200 39.7 -> 20.5, four of 600 and 1000 of
// 200 3.65 -> 3.65 (nowhere slower).
template <int... Bs>
static bool launch_acs_rows_slots(ChunkList<Bs...>, const Instance* insts, const int* slots,
                                  int count, int max_m, int max_n, cudaStream_t st) {
  const size_t smem = acs_rows_bytes(max_n, max_m);
  return smem <= kAcsRowsMost &&
         ((max_n <= 128 * Bs && 32 * max_m <= kAcsRowThreads<Bs> && acs_rows_ready<Bs, true>() &&
           (acs_rows_slots_kernel<Bs><<<count, 32 * max_m, smem, st>>>(insts, slots), true)) ||
          ...);
}

cudaError_t launch_acs_construct(const Instance& I, cudaStream_t st) {
  if (I.m < 1 || I.m > kAcsMaxAnts) return cudaErrorInvalidValue;
  const size_t smem = (size_t)I.m * ((I.n + 31) / 32) * sizeof(uint32_t);
  if (I.nn > 0)
    acs_construct_kernel<true><<<1, 32 * I.m, smem, st>>>(I);
  else if (!launch_acs_rows(AcsBlocks{}, I, st))
    acs_construct_kernel<false><<<1, 32 * I.m, smem, st>>>(I);
  return cudaGetLastError();
}

cudaError_t launch_acs_global(const Instance& I, cudaStream_t st) {
  acs_global_kernel<<<(I.n + 255) / 256, 256, 0, st>>>(I);
  return cudaGetLastError();
}

cudaError_t launch_acs_construct_slots(const Instance* insts, const int* slots, int count,
                                       int max_m, int max_n, bool lists, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  if (max_m < 1 || max_m > kAcsMaxAnts) return cudaErrorInvalidValue;
  const size_t smem = (size_t)max_m * ((max_n + 31) / 32) * sizeof(uint32_t);
  if (lists)
    acs_construct_slots_kernel<true><<<count, 32 * max_m, smem, st>>>(insts, slots);
  else if (!launch_acs_rows_slots(AcsBlocks{}, insts, slots, count, max_m, max_n, st))
    acs_construct_slots_kernel<false><<<count, 32 * max_m, smem, st>>>(insts, slots);
  return cudaGetLastError();
}

cudaError_t launch_acs_global_slots(const Instance* insts, const int* slots, int count,
                                    cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  acs_global_slots_kernel<<<count, 256, 0, st>>>(insts, slots);
  return cudaGetLastError();
}

}  // namespace aco
