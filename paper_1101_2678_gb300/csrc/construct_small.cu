// Tour construction by Eq. 1 for instances whose whole choice_info matrix fits
// in one CTA's shared memory (n <= 240, and few enough ants above n = 232).
//
// At these sizes a step is nothing but latency: the walk of
// construct_phased.cuh spends a third of its step waiting for the row's copy
// out of L2.  Here each CTA copies the matrix once (one bulk copy, a contiguous
// n * ld floats) and a step starts with a 16-byte shared-memory load.  One warp
// per ant, the ants dealt evenly over all SMs; lane l owns the cities [l*CH,
// l*CH + CH), CH = 4 up to n = 128, else 8.  Every lane works out which of its
// cities would hold the target; the votes that find the lane also carry the
// city's place in its chunk, so a step has one warp scan, one shuffle and a few
// votes.  The search is the single-precision one of eq1_phase() with its error
// bound, and exact_pick() decides where that cannot.
// Construct, GB300, ms, m = n unless given, the walk -> this kernel: n = 24
// 0.0176 -> 0.0118, n = 48 0.0286 -> 0.0172, n = 128 0.0708 -> 0.0373, n = 230
// 0.134 -> 0.070, with m = 4864 0.253 -> 0.201.  Which sizes take it is decided
// by small_warps().  A step takes about 520 cycles, the scan and the votes most
// of them.
#include "construct.cuh"
#include "kernels.h"

namespace aco {

namespace {

// Floats staged: the matrix, and a tail that the last row's lanes may read
// (their tabu bits are set there).
template <int CH>
__host__ __device__ constexpr size_t small_floats(int n, int ld) {
  return (size_t)n * ld + 32 * CH;
}

template <int CH>
size_t small_bytes(int n, int ld, int warps) {
  const size_t tour = ((size_t)n * 2 + 15) / 16 * 16;
  return 16 + small_floats<CH>(n, ld) * 4 + (size_t)warps * tour;
}

template <int CH>
__global__ void __launch_bounds__(1024) construct_small_kernel(Instance I) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  // roundings: see eq1_phase() (the lane's sum, the scan, the whole sum; the
  // cities of the lane; target and differences, two to spare)
  constexpr float kEps = (float)(2 * (CH + 5) + CH + 10) * 0x1p-24f;
  const int n = I.n, ld = I.ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* mat = reinterpret_cast<float*>(small_smem + 16);
  uint16_t* tour = reinterpret_cast<uint16_t*>(mat + small_floats<CH>(n, ld)) +
                   warp * ((n + 7) / 8 * 8);
  const uint32_t bar = smem_u32(small_smem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    bulk_load(smem_u32(mat), I.choice, (uint32_t)n * (uint32_t)ld * 4u, bar);
  }
  __syncthreads();
  const int ant = blockIdx.x * (blockDim.x >> 5) + warp;
  const uint32_t iter = (uint32_t)I.st->iteration;
  const unsigned long long seed = I.seed;
  // every warp waits for the copy, also those without an ant (the CTA's shared
  // memory must not go away under it)
  int start = 0;
  if (ant < I.m) {
    const Philox4 x0 = step_draw(seed, 0u, (uint32_t)ant, iter);
    start = (int)__umulhi(x0.x0, (uint32_t)n);
  }
  // (twice the limit: the CTA goes on to its end with the copy in flight if it
  // still has not come)
  if (!mbar_wait_bounded(bar, 0u, 2 * kWaitPolls) && lane == 0)
    atomicOr(&I.st->status, kStatusTimeout);
  if (ant >= I.m) return;

  const Seg<32> seg(lane);
  const int base = lane * CH;
  uint32_t vis[1];  // tabu bits, set past the row's end
  vis[0] = n - base <= 0 ? FULL : (n - base >= CH ? FULL << (CH - 1) << 1 : FULL << (n - base));
  auto mark = [&](int c) {
    if (c / CH == lane) vis[0] |= 1u << (c % CH);
  };
  mark(start);
  if (lane == 0) tour[0] = (uint16_t)start;
  int cur = start;
  for (int s0 = 1; s0 < n; s0 += 32) {
    // the draws of 32 steps, one per lane
    const Philox4 x = step_draw(seed, (uint32_t)(s0 + lane), (uint32_t)ant, iter);
    const float u = __fmul_rn(__uint2float_rn(x.x1), 0x1p-32f);
    const int s1 = min(n, s0 + 32);
    for (int s = s0; s < s1; ++s) {
      const float us = __shfl_sync(FULL, u, s - s0);
      const float* row = mat + (size_t)cur * ld;
      float v[CH];
#pragma unroll
      for (int g = 0; g < CH / 4; ++g) {
        const float4 t = *reinterpret_cast<const float4*>(row + base + 4 * g);
        v[4 * g] = t.x;
        v[4 * g + 1] = t.y;
        v[4 * g + 2] = t.z;
        v[4 * g + 3] = t.w;
      }
#pragma unroll
      for (int i = 0; i < CH; ++i)
        if ((vis[0] >> i) & 1u) v[i] = 0.0f;
      float mine = __fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3]));
      if constexpr (CH == 8)
        mine = __fadd_rn(mine, __fadd_rn(__fadd_rn(v[4], v[5]), __fadd_rn(v[6], v[7])));
      const float incl = seg.inclusive_scan_f(mine);
      const float S = __shfl_sync(FULL, incl, 31);
      const float err = S >= 0x1p-120f ? __fmul_rn(kEps, S) : __int_as_float(0x7f800000);
      // the target inside the lane, and the city that holds it for sure
      const float t = __fsub_rn(__fmul_rn(us, S), __fsub_rn(incl, mine));
      const float hi_t = __fadd_rn(t, err), lo_t = __fsub_rn(t, err);
      uint32_t slot = CH;
      float c = 0.0f;
#pragma unroll
      for (int i = 0; i < CH; ++i) {
        const float below = c;
        c = __fadd_rn(c, v[i]);
        if (c > hi_t && below < lo_t) slot = (uint32_t)i;
      }
      const uint32_t sure = __ballot_sync(FULL, slot < CH);
      int next = (__ffs(sure) - 1) * CH;
#pragma unroll
      for (int b = 1; b < CH; b <<= 1)
        if (__ballot_sync(FULL, slot < CH && (slot & b))) next += b;
      if (sure == 0u) {
        const Philox4 xr = step_draw(seed, (uint32_t)s, (uint32_t)ant, iter);
        const unsigned long long r = ((unsigned long long)xr.x1 << 32) | xr.x0;
        next = exact_pick<1, 32, 1>(row, nullptr, CH, 0u, vis, lane, 0, nullptr, r).next;
        if ((unsigned)next >= (unsigned)n) {  // only from a defect: record it, stay in bounds
          if (lane == 0) atomicOr(&I.st->status, kStatusBadTour);
          next = start;
        }
      }
      mark(next);
      if (lane == 0) tour[s] = (uint16_t)next;
      cur = next;
    }
  }
  __syncwarp();

  // The tour, C^k (Section II) and the per-city neighbour buckets.
  int32_t* out = I.tours + (size_t)ant * I.ldt;
  long long len = 0;
  for (int s = lane; s < n; s += 32) {
    const int a = tour[s], b = tour[s + 1 < n ? s + 1 : 0], p = tour[s == 0 ? n - 1 : s - 1];
    out[s] = a;
    len += I.dist[(size_t)a * ld + b];
    I.nbr[(size_t)a * I.ldm + ant] = ((uint32_t)p << 16) | (uint32_t)b;
  }
  if (lane == 0) out[n] = start;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) len += __shfl_xor_sync(FULL, len, o);
  if (lane == 0) I.lens[ant] = len;
}

constexpr size_t kSmallMost = 227 * 1024;

// Warps (ants) per CTA, one CTA on each SM at a time: the ants dealt evenly over
// as few rounds of CTAs as the shared memory allows; 0 where the walk is taken.
// From n = 233 on the matrix leaves room for fewer than 32 warps (233: 23,
// 237: 8, 240: 2), and a round costs what its longest step does, so many ants
// take many rounds.  Two rounds are still no slower than the walk, three are
// not: ms, as many rounds as it takes / the walk / this rule, n = 240 with m =
// 512 0.137 / 0.141 / 0.137, 1024 0.265 / 0.147 / 0.145, 4864 1.05 / 0.263 /
// 0.259; n = 238, m = 1024 0.155 / 0.147 / 0.137.  Even rounds: n = 200, m =
// 5000 (152 CTAs of 32 ants and 5 more) 0.337 / 0.245, of 17 ants 0.192.
template <int CH>
int small_warps(int n, int m, int sms) {
  const int ld = (n + 3) / 4 * 4;
  int most = 32;
  while (most > 0 && small_bytes<CH>(n, ld, most) > kSmallMost) --most;
  if (most == 0) return 0;
  const int rounds = (m + sms * most - 1) / (sms * most);
  if (most < 32 && rounds > 2) return 0;
  return (m + sms * rounds - 1) / (sms * rounds);
}

template <int CH>
cudaError_t launch_small(const Instance& I, int sms, cudaStream_t st) {
  const int warps = small_warps<CH>(I.n, I.m, sms);
  if (warps < 1) return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = once_per_device(done, [] {
    return cudaFuncSetAttribute(construct_small_kernel<CH>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallMost);
  });
  if (e != cudaSuccess) return e;
  construct_small_kernel<CH><<<(I.m + warps - 1) / warps, 32 * warps,
                               small_bytes<CH>(I.n, I.ld, warps), st>>>(I);
  return cudaGetLastError();
}

}  // namespace

bool construct_small_fits(int n, int m, int sms) {
  return n <= 256 && (n <= 128 ? small_warps<4>(n, m, sms) : small_warps<8>(n, m, sms)) > 0;
}

cudaError_t launch_construct_small(const Instance& I, int sms, cudaStream_t st) {
  return I.n <= 128 ? launch_small<4>(I, sms, st) : launch_small<8>(I, sms, st);
}

}  // namespace aco
