// Pheromone update (evaporation + fixed-point atomic deposit + choice_info)
// on caller-owned device buffers, with its scratch in a file-scope device
// array instead of allocated memory (aco_update_pheromone_noalloc in aco.h).
//
// Some callers cannot call cudaMalloc at all: code running inside a region
// being captured into a CUDA graph by someone else, allocator-less embedded
// runtimes, or hosts that pre-plan every byte of device memory and forbid
// allocations after start-up.  For them this entry point needs no memory
// beyond the arrays they pass and one fixed static array that the module
// reserves on every GPU where the library is loaded.
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>

#include "../../include/aco.h"
#include "aco_device.cuh"
#include "runtime.h"

namespace aco {
namespace {

constexpr int kNoallocMaxN = ACO_NOALLOC_MAX_N;
constexpr int kNoallocMaxM = ACO_NOALLOC_MAX_M;
// [0, N*N): u64 accumulator, then one slot for S.
constexpr size_t kScratchWords = (size_t)kNoallocMaxN * kNoallocMaxN + 32;

static __device__ __align__(256) unsigned long long g_noalloc_scratch[kScratchWords];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned long long* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device, looked up once
// per device (with that device current) and cached.
int scratch_for_current_device(unsigned long long** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(ACO_EINVAL, "device %d beyond %d", dev, kMaxDevices);
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
    g_scratch_ptr[dev] = static_cast<unsigned long long*>(p);
  }
  *out = g_scratch_ptr[dev];
  return ACO_OK;
}

// The tour edge (a, b) is summed once, in acc[min(a,b)][max(a,b)]: half the
// atomics, clearing and reading of a full matrix (the caller's tau and eta^beta
// are still read and written cell by cell: nothing makes them symmetric).
// Calls back to back, GB300, four launches over the full accumulator -> these
// three: n = m = 1002 22.7 -> 18.6 us, n = 300, m = 2000 24.7 -> 14.5 us,
// n = 1024, m = 4096 59.6 -> 32.9 us.

// Clear the upper triangle (a warp per row); CTA 0 finds the deposit scale S
// meanwhile.
constexpr int kZeroThreads = 512;

__global__ void __launch_bounds__(kZeroThreads)
    noalloc_zero_prep_kernel(unsigned long long* acc, int n, const long long* __restrict__ lens,
                             int m, unsigned long long* shift_slot) {
  grid_release();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = kZeroThreads / 32;
  if (blockIdx.x > 0) {
    const int i = (blockIdx.x - 1) * warps + warp;
    if (i >= n) return;
    for (int j = i + lane; j < n; j += 32) acc[(size_t)i * n + j] = 0ull;
    return;
  }
  __shared__ long long red[kZeroThreads / 32];
  long long bl = LLONG_MAX;
  for (int k = threadIdx.x; k < m; k += blockDim.x) bl = min(bl, lens[k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bl = min(bl, __shfl_xor_sync(FULL, bl, o));
  if (lane == 0) red[warp] = bl;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < warps; ++w) bl = min(bl, red[w]);
    const float dmax = (float)(1.0 / (double)bl);
    *shift_slot = (unsigned long long)(62 - ceil_log2_u32((uint32_t)m) -
                                       exponent_of_bits(__float_as_uint(dmax)));
  }
}

// red.global.add.u64 of q_k on every tour edge, a run of ants per CTA; tours are
// m rows of n+1 cities.  Ants of a converging colony share most edges, and
// additions to one address follow each other at about 14 ns (m = 1002 on the
// edges of one tour: 14 us, whatever else the kernel does; m = 4096: 58 us), so
// the CTA adds up
// its ants first: each tour is turned into neighbours per city in shared
// memory, and the thread of a city keeps running sums of the edges to its
// higher neighbours, added to acc when another edge takes their place.
// A row that is not a closed tour of n different cities goes edge by edge:
// edges with an entry outside [0, n) are skipped, an edge from a city to
// itself counts for both of its directions.
constexpr int kDepositSums = 3;  // running sums per city
constexpr int kRunMost = 64;     // ants per CTA at most
constexpr uint32_t kNobody = 0xffffffffu;

// One thread per city (blockDim.x >= n).
__global__ void __launch_bounds__(kNoallocMaxN)
    noalloc_deposit_kernel(const int32_t* __restrict__ tours, int n, int m, int per_cta,
                           const long long* __restrict__ lens,
                           const unsigned long long* shift_slot, unsigned long long* acc) {
  __shared__ uint32_t nb[kNoallocMaxN];  // pred << 16 | succ of each city
  __shared__ unsigned long long s_q[kRunMost];
  grid_release();
  const int i = threadIdx.x;  // a place in the tours, then a city
  int to[kDepositSums];
  unsigned long long sum[kDepositSums];
#pragma unroll
  for (int c = 0; c < kDepositSums; ++c) {
    to[c] = -1;
    sum[c] = 0ull;
  }
  nb[i] = kNobody;
  const int k0 = blockIdx.x * per_cta, k1 = min(m, k0 + per_cta);
  // pred, city and succ at place i; the next tour's are loaded a tour ahead
  auto place = [&](int k, int& p, int& a, int& b) {
    p = a = b = 0;
    if (i < n && k < k1) {
      const int32_t* t = tours + (size_t)k * (n + 1);
      p = t[i == 0 ? n - 1 : i - 1];
      a = t[i];
      b = t[i + 1];
    }
  };
  grid_wait();
  int p, a, b;
  place(k0, p, a, b);
  // q_k = floor(dtau^k * 2^S), dtau^k = (float)(1/C^k), of the CTA's ants
  const int shift = (int)*shift_slot;
  if (k0 + i < k1) s_q[i] = fixed_of((float)(1.0 / (double)lens[k0 + i]), shift);
  if (blockDim.x < per_cta)  // fewer threads than ants
    for (int k = i + blockDim.x; k0 + k < k1; k += blockDim.x)
      s_q[k] = fixed_of((float)(1.0 / (double)lens[k0 + k]), shift);
  __syncthreads();
  for (int k = k0; k < k1; ++k) {
    const unsigned long long qk = s_q[k - k0];
    bool ok = true;
    if (i < n) {
      // the closing entry is the last place's succ and has to be the first city
      const int32_t* t = tours + (size_t)k * (n + 1);
      ok = (unsigned)a < (unsigned)n && (unsigned)b < (unsigned)n && (unsigned)p < (unsigned)n &&
           (i != n - 1 || b == t[0]);
      if (ok) nb[a] = (uint32_t)p << 16 | (uint32_t)b;
    }
    place(k + 1, p, a, b);
    __syncthreads();
    // n entries that reach all n cities are n different cities
    const uint32_t own = nb[i];
    nb[i] = kNobody;
    if (i < n && own == kNobody) ok = false;
    if (__syncthreads_and(ok)) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int j = (int)(half ? own & 0xffffu : own >> 16);
        if (i >= n || j <= i) continue;
        bool held = false;
#pragma unroll
        for (int c = 0; c < kDepositSums; ++c)
          if (to[c] == j) {
            sum[c] += qk;
            held = true;
          }
        if (!held) {
          if (to[0] >= 0) atomicAdd(acc + (size_t)i * n + to[0], sum[0]);
#pragma unroll
          for (int c = 0; c + 1 < kDepositSums; ++c) {
            to[c] = to[c + 1];
            sum[c] = sum[c + 1];
          }
          to[kDepositSums - 1] = j;
          sum[kDepositSums - 1] = qk;
        }
      }
    } else if (i < n) {
      const int32_t* t = tours + (size_t)k * (n + 1);
      const int x = t[i], y = t[i + 1];
      if ((unsigned)x < (unsigned)n && (unsigned)y < (unsigned)n)
        atomicAdd(acc + (size_t)min(x, y) * n + max(x, y), x == y ? 2 * qk : qk);
    }
  }
#pragma unroll
  for (int c = 0; c < kDepositSums; ++c)
    if (to[c] >= 0) atomicAdd(acc + (size_t)i * n + to[c], sum[c]);
}

// tau' = fl(fl((1-rho) tau) + fl(acc) * 2^-S), choice = tau'^alpha * eta^beta.
// A CTA of 32 x 8 threads per 32 x 32 tile (bi, bj), bi <= bj, of the upper
// triangle: its deposits go through shared memory to the mirrored tile, so
// that both are read and written row by row.
constexpr int kApplyTile = 32;

__global__ void __launch_bounds__(256)
    noalloc_apply_kernel(float* tau, const float* __restrict__ heta, float* choice,
                         const unsigned long long* acc, const unsigned long long* shift_slot,
                         int n, float alpha, float rho) {
  // (acc and shift_slot are still being written when this kernel starts: no
  // __restrict__, whose read-only promise would hold for its whole life)
  __shared__ float dep[kApplyTile][kApplyTile + 1];
  const int bi = blockIdx.y, bj = blockIdx.x;
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (bi > bj) return;
  grid_wait();
  const float keep = __fsub_rn(1.0f, rho);
  const float inv = pow2f(-(int)*shift_slot);
  auto cell = [&](int i, int j, float d) {
    const size_t e = (size_t)i * n + j;
    const float t = __fadd_rn(__fmul_rn(keep, tau[e]), d);
    tau[e] = t;
    choice[e] = choice_of(t, heta[e], alpha);
  };
  const int j = bj * kApplyTile + tx;
#pragma unroll
  for (int r = 0; r < kApplyTile; r += 8) {
    const int i = bi * kApplyTile + ty + r;
    if (i < n && j < n && j >= i) {
      const float d = __fmul_rn(__ull2float_rn(acc[(size_t)i * n + j]), inv);
      dep[ty + r][tx] = d;
      cell(i, j, d);
    }
  }
  __syncthreads();
  const int jt = bi * kApplyTile + tx;  // column of the mirrored tile
#pragma unroll
  for (int r = 0; r < kApplyTile; r += 8) {
    const int it = bj * kApplyTile + ty + r;  // row of the mirrored tile
    if (it < n && jt < n && jt < it) cell(it, jt, dep[tx][ty + r]);
  }
}

}  // namespace
}  // namespace aco

using namespace aco;

extern "C" int aco_update_pheromone_noalloc(int32_t n, int32_t m, const int32_t* tours,
                                            const int64_t* lens, const float* heta, float* tau,
                                            float* choice, float alpha, float rho,
                                            int64_t stream) {
  if (n < 3 || n > kNoallocMaxN)
    return fail(ACO_EINVAL, "n=%d outside [3, %d] (the static scratch holds %d x %d)", n,
                kNoallocMaxN, kNoallocMaxN, kNoallocMaxN);
  if (m < 1 || m > kNoallocMaxM)
    return fail(ACO_EINVAL, "m=%d outside [1, %d]", m, kNoallocMaxM);
  if (!tours || !lens || !heta || !tau || !choice) return fail(ACO_EINVAL, "NULL device pointer");
  if (!std::isfinite(alpha) || alpha < 0.0f) return fail(ACO_EINVAL, "alpha must be finite and >= 0");
  if (!(rho > 0.0f && rho <= 1.0f)) return fail(ACO_EINVAL, "rho must lie in (0, 1]");
  unsigned long long* scratch = nullptr;
  int rc = scratch_for_current_device(&scratch);
  if (rc) return rc;
  unsigned long long* acc = scratch;
  unsigned long long* shift_slot = scratch + (size_t)kNoallocMaxN * kNoallocMaxN;
  cudaStream_t st = (cudaStream_t)(intptr_t)stream;
  const int zero_rows = kZeroThreads / 32;
  // 1024 threads an SM: more ants to a CTA mean fewer additions to a shared
  // edge but a longer chain of tours
  const int threads = (n + 31) / 32 * 32;
  const int ctas = device_sms() * std::max(1, 1024 / threads);
  const int per_cta = std::min((m + ctas - 1) / ctas, kRunMost);
  noalloc_zero_prep_kernel<<<1 + (n + zero_rows - 1) / zero_rows, kZeroThreads, 0, st>>>(
      acc, n, reinterpret_cast<const long long*>(lens), m, shift_slot);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = launch_early(noalloc_deposit_kernel, (m + per_cta - 1) / per_cta, threads, 0, st,
                     tours, n, m, per_cta, reinterpret_cast<const long long*>(lens), shift_slot, acc);
  const int tiles = (n + kApplyTile - 1) / kApplyTile;
  if (e == cudaSuccess)
    e = launch_early(noalloc_apply_kernel, dim3(tiles, tiles), dim3(kApplyTile, 8), 0, st, tau,
                     heta, choice, acc, shift_slot, n, alpha, rho);
  if (e != cudaSuccess) return cuda_fail(e, "noalloc update launch");
  return ACO_OK;
}
