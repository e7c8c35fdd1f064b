// One persistent construction launch over every (instance, ant) item of a
// pool step (the batching pattern's single launch per phase), measured
// against one launch per tiling class.
//
// Each warp builds one ant at a time: it takes the next item from a global
// ticket (atomicAdd; no waiting on other warps), finds the item's class (the
// classes are listed largest chunk first, so the longest instances are taken
// first) and runs the Eq. 1 walk with that class's chunk width.  Every width
// is a separate code path of the one kernel, all under one register cap (64,
// 32 warps per SM).  A step of 256 instances takes 15.9 ms, against 12.4 ms
// with one launch per class.
#include "construct.cuh"
#include "kernels.h"

namespace aco {

namespace {

constexpr int kSingleWarps = 4;
constexpr int kSingleBytes = StageLayout<36, 1, 32>::kBytes;  // the widest chunk handled

template <int C>
struct Width {
  static constexpr int value = C;
};

__global__ void __maxnreg__(64)
    construct_single_kernel(const Instance* __restrict__ insts, const int2* __restrict__ items,
                            SingleClasses cls, int total, int* ticket) {
  __shared__ GroupSmem gs[kSingleWarps];
  extern __shared__ __align__(16) unsigned char stage[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* srow = reinterpret_cast<float*>(stage + warp * kSingleBytes);
  const Seg<32> seg(lane);
  bool ok = true;
  for (;;) {
    int t = 0;
    if (lane == 0) t = atomicAdd(ticket, 1);
    t = __shfl_sync(FULL, t, 0);
    if (t >= total) break;
    int k = 0, idx = t;
    while (k < cls.n - 1 && idx >= cls.count[k]) {
      idx -= cls.count[k];
      ++k;
    }
    const int2 it = items[cls.begin[k] + idx];
    const Instance& I = insts[it.x];
    // after a wait of this warp gave up: no more bulk copies, and every result
    // from its staging memory is marked
    const bool lc = cls.lane_copy[k] != 0 || !ok;
    if (!ok && lane == 0) atomicOr(&I.st->status, kStatusTimeout);
    bool waited = true;
    auto build = [&](auto width) {
      waited = construct_ant_phased<decltype(width)::value, 1, 32, true>(
          I, it.y, lane, seg, &gs[warp], 1 + warp, srow, lc);
    };
    switch (cls.C[k]) {
      case 4: build(Width<4>{}); break;
      case 12: build(Width<12>{}); break;
      case 20: build(Width<20>{}); break;
      case 28: build(Width<28>{}); break;
      case 36: build(Width<36>{}); break;
      default: break;
    }
    ok = __all_sync(FULL, waited) && ok;
  }
}

}  // namespace

bool single_launch_supports(int C) { return C == 4 || C == 12 || C == 20 || C == 28 || C == 36; }

cudaError_t launch_construct_single(const Instance* insts, const int2* items,
                                    const SingleClasses& cls, int total, int* ticket, int sms,
                                    cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  static std::atomic<unsigned long long> done{0};
  const int smem = kSingleWarps * kSingleBytes;
  cudaError_t e = once_per_device(done, [smem] {
    return cudaFuncSetAttribute(construct_single_kernel,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  });
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(ticket, 0, sizeof(int), st)) != cudaSuccess) return e;
  // 64 registers: 32 resident warps per SM, eight CTAs of four warps.
  construct_single_kernel<<<sms * 8, 32 * kSingleWarps, smem, st>>>(insts, items, cls, total,
                                                                     ticket);
  return cudaGetLastError();
}

}  // namespace aco
