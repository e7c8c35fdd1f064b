// The Eq. 1 walk (construct_phased.cuh) on the host, every GPU thread a fibre of its own: a thread
// runs on until it meets a warp collective, a barrier or an unfinished copy, and the scheduler
// picks the next one at random.  The programming model promises no more than that between two
// synchronisations, so a result that needs the lanes of a warp to keep in step comes out wrong here.
//
// Also recorded: bulk copies (async proxy) into bytes that a thread wrote through the generic
// proxy without a proxy fence since (cp.async rows), and copies that follow one that never came.
#include <ucontext.h>

#include <bit>
#include <cfenv>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <tuple>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

namespace emu {

struct Group {  // lanes that meet at one collective or barrier
  int arrived = 0;
  unsigned long long gen = 0;
  int kind = 0;
  unsigned long long slot[2][32];
};
struct Fibre {
  ucontext_t ctx;
  std::vector<char> stack;
  bool done = false;
  Group* at = nullptr;  // blocked until at->gen != gen
  unsigned long long gen = 0;
};
struct Mbar {
  unsigned phase = 0;
  bool stuck = false;
};

static std::vector<Fibre> fibres;
static ucontext_t home;
static int self;
static uint3 tid;
static bool broken;  // lanes of one group met at different collectives, or none can go on
static int unfenced, late, reused, copies, stall;
static std::map<std::pair<int, unsigned>, Group> groups;
static std::map<uint32_t, Mbar> mbars;
alignas(16) static unsigned char smem[1 << 18];
static short writer[sizeof smem];  // 1 + thread that wrote the byte since its last proxy fence
static const char *src_lo, *src_hi;

static void yield() { swapcontext(&fibres[self].ctx, &home); }

static Group& meet(int key, unsigned mask, int count, int kind, unsigned long long v,
                   unsigned long long& gen) {
  Group& g = groups[{key, mask}];
  gen = g.gen;
  if (g.arrived == 0) g.kind = kind;
  if (g.kind != kind) broken = true;
  g.slot[gen & 1][self & 31] = v;
  if (++g.arrived == count) {
    g.arrived = 0;
    ++g.gen;
  } else {
    fibres[self].at = &g;
    fibres[self].gen = gen;
    yield();
  }
  return g;
}
// All lanes' values at a warp collective.
static const unsigned long long* trade(unsigned mask, int kind, unsigned long long v) {
  unsigned long long gen;
  Group& g = meet(self / 32, mask, std::popcount(mask), kind, v, gen);
  return g.slot[gen & 1];
}
template <class T>
unsigned long long raw(T v) {
  unsigned long long r = 0;
  memcpy(&r, &v, sizeof v);
  return r;
}
template <class T>
T as(unsigned long long r) {
  T v;
  memcpy(&v, &r, sizeof v);
  return v;
}
static void bar_sync(int id, int count) {
  unsigned long long gen;
  meet(1000 + id, 0u, count, 0, 0, gen);
}

}  // namespace emu

static uint3 blockIdx, blockDim;  // (the kernels around the walk are compiled, not run)
#define threadIdx emu::tid
#define __launch_bounds__(...)

template <class T>
T __shfl_sync(unsigned mask, T v, int src, int width = 32) {
  const auto* s = emu::trade(mask, 1, emu::raw(v));
  return emu::as<T>(s[(emu::self & 31 & ~(width - 1)) + (src & (width - 1))]);
}
template <class T>
T __shfl_up_sync(unsigned mask, T v, int d, int width = 32) {
  const auto* s = emu::trade(mask, 2, emu::raw(v));
  const int l = emu::self & 31;
  return l % width >= d ? emu::as<T>(s[l - d]) : v;
}
template <class T>
T __shfl_xor_sync(unsigned mask, T v, int d, int width = 32) {
  (void)width;
  const auto* s = emu::trade(mask, 3, emu::raw(v));
  return emu::as<T>(s[(emu::self & 31) ^ d]);
}
inline unsigned __ballot_sync(unsigned mask, bool p) {
  const auto* s = emu::trade(mask, 4, p);
  unsigned r = 0;
  for (int l = 0; l < 32; ++l)
    if ((mask >> l) & 1u) r |= (s[l] ? 1u : 0u) << l;
  return r;
}
inline void __syncwarp(unsigned mask = 0xffffffffu) { emu::trade(mask, 5, 0); }
inline unsigned __reduce_max_sync(unsigned mask, unsigned v) {
  const auto* s = emu::trade(mask, 6, v);
  unsigned r = 0;
  for (int l = 0; l < 32; ++l)
    if ((mask >> l) & 1u) r = s[l] > r ? (unsigned)s[l] : r;
  return r;
}
inline unsigned __reduce_min_sync(unsigned mask, unsigned v) {
  const auto* s = emu::trade(mask, 7, v);
  unsigned r = ~0u;
  for (int l = 0; l < 32; ++l)
    if ((mask >> l) & 1u) r = s[l] < r ? (unsigned)s[l] : r;
  return r;
}

inline float __int_as_float(int v) { return emu::as<float>((unsigned)v); }
inline float __uint_as_float(unsigned v) { return emu::as<float>(v); }
inline unsigned __float_as_uint(float v) { return (unsigned)emu::raw(v); }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdiv_rn(float a, float b) { return a / b; }
inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
inline float __fmaf_rz(float a, float b, float c) {
  // a b is exact in double and the sum's error has a sign: one step towards zero where it rounded up
  const double p = (double)a * b, s = p + c;
  const double t = s - p, err = (p - (s - t)) + (c - t);
  float r = (float)s;
  if ((double)r > s || ((double)r == s && err < 0.0)) r = nextafterf(r, 0.0f);  // (s > 0 here)
  return r;
}
inline float __uint2float_rn(unsigned v) { return (float)v; }
inline float __int2float_rn(int v) { return (float)v; }
inline float __ull2float_rn(unsigned long long v) { return (float)v; }
inline unsigned __umulhi(unsigned a, unsigned b) {
  return (unsigned)(((unsigned long long)a * b) >> 32);
}
inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
inline int __ffs(int v) { return __builtin_ffs(v); }
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline unsigned __cvta_generic_to_shared(const void* p) {
  return (unsigned)(static_cast<const unsigned char*>(p) - emu::smem);
}
template <class T, class U>
T max(T a, U b) { return a > (T)b ? a : (T)b; }
template <class T, class U>
T min(T a, U b) { return a < (T)b ? a : (T)b; }
inline int atomicOr(int* p, int v) {
  const int o = *p;
  *p |= v;
  return o;
}

// The PTX helpers: their names are taken from the header, and the host's stand in for them.
#define mbar_init ptx_mbar_init
#define mbar_inval ptx_mbar_inval
#define mbar_try_wait ptx_mbar_try_wait
#define mbar_wait_bounded ptx_mbar_wait_bounded
#define fence_mbar_init ptx_fence_mbar_init
#define fence_proxy_async_smem ptx_fence_proxy_async_smem
#define bulk_load_if ptx_bulk_load_if
#define cp_async16_if ptx_cp_async16_if
#define cp_async_wait_all ptx_cp_async_wait_all
#include "aco_device.cuh"
#undef mbar_init
#undef mbar_inval
#undef mbar_try_wait
#undef mbar_wait_bounded
#undef fence_mbar_init
#undef fence_proxy_async_smem
#undef bulk_load_if
#undef cp_async16_if
#undef cp_async_wait_all

namespace aco {
inline void mbar_init(uint32_t bar, uint32_t) {
  if (emu::mbars.count(bar)) ++emu::reused;
  emu::mbars[bar] = emu::Mbar{};
}
inline void mbar_inval(uint32_t bar) { emu::mbars.erase(bar); }
inline bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  if ((emu::mbars[bar].phase & 1u) != parity) return true;
  emu::yield();
  return false;
}
inline bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < (emu::mbars[bar].stuck ? 50 : 100000); ++i)
    if (mbar_try_wait(bar, parity)) return true;
  if (!emu::mbars[bar].stuck) emu::broken = true;
  return false;
}
inline void fence_mbar_init() {}
inline void fence_proxy_async_smem() {
  for (short& w : emu::writer)
    if (w == emu::self + 1) w = 0;
}
inline bool in_source(const void* src, uint32_t bytes) {
  const char* c = static_cast<const char*>(src);
  if (c >= emu::src_lo && c + bytes <= emu::src_hi) return true;
  emu::broken = true;
  return false;
}
inline void bulk_load_if(bool go, uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  if (!go) return;
  if (emu::mbars[bar].stuck) ++emu::late;
  if (emu::copies++ == emu::stall) emu::mbars[bar].stuck = true;
  if (emu::mbars[bar].stuck) return;
  for (uint32_t b = dst; b < dst + bytes; ++b)
    if (emu::writer[b]) {
      ++emu::unfenced;
      break;
    }
  if (in_source(src, bytes)) memcpy(emu::smem + dst, src, bytes);
  ++emu::mbars[bar].phase;
}
inline void cp_async16_if(bool go, uint32_t dst, const void* src) {
  if (!go || !in_source(src, 16)) return;
  memcpy(emu::smem + dst, src, 16);
  for (int b = 0; b < 16; ++b) emu::writer[dst + b] = (short)(emu::self + 1);
}
inline void cp_async_wait_all() {}
}  // namespace aco

#include "construct.cuh"

namespace {

struct Job {
  aco::Instance I;
  int ants;             // built one after another by each group, group g from ant g
  const int* lane_copy; // per round
};
Job job;
aco::GroupSmem gsm[4];

template <int C, int G, int H>
void thread_main() {
  constexpr int kGroups = H == 32 ? 1 : 32 / H;
  const int t = (int)threadIdx.x;
  const int grp = H == 32 ? 0 : (t & 31) / H, tg = H == 32 ? t : t % H;
  const aco::Seg<H> seg(t & 31);
  float* srow = reinterpret_cast<float*>(emu::smem + grp * aco::StageLayout<C, G, H>::kBytes);
  for (int r = 0; r * kGroups + grp < job.ants; ++r)
    aco::construct_ant_phased<C, G, H, false>(job.I, r * kGroups + grp, tg, seg, &gsm[grp],
                                              1 + grp, srow, job.lane_copy[r] != 0);
  emu::fibres[emu::self].done = true;
  for (;;) emu::yield();
}

void (*entry)();

}  // namespace

// Tours and lengths of `ants` ants; lane_copy[r]: row staging of the ants of round r, which share
// shared memory with the round before; stall: the bulk copy of that number never arrives (-1: all
// do).  Returns 0, or 1 where threads parted for good.  counts: bulk copies over generic-proxy
// writes without a fence; copies issued on a barrier after one that never came; status bits;
// barriers initialised again without having been invalidated.
extern "C" int emulate_walk(int C, int G, int H, int n, int ants, const int* lane_copy,
                            const float* choice, const int* dist, unsigned long long seed,
                            unsigned schedule, int stall, int* tours, long long* lens, int* counts) {
  using namespace emu;
  entry = C == 36 && G == 1 && H == 32   ? thread_main<36, 1, 32>
          : C == 36 && G == 1 && H == 16 ? thread_main<36, 1, 16>
          : C == 36 && G == 1 && H == 8  ? thread_main<36, 1, 8>
          : C == 36 && G == 2 && H == 32 ? thread_main<36, 2, 32>
          : C == 76 && G == 1 && H == 32 ? thread_main<76, 1, 32>
          : C == 12 && G == 1 && H == 32 ? thread_main<12, 1, 32>
                                         : nullptr;
  if (!entry || n > C * G * H) return 2;
  // (room for any index a wrong city can give)
  const int ld = (n + 3) / 4 * 4, cities = C * G * H + 8;
  std::vector<float> ch((size_t)n * ld);
  std::vector<int> d((size_t)cities * ld + cities);
  for (int i = 0; i < n; ++i) {
    memcpy(&ch[(size_t)i * ld], choice + (size_t)i * n, 4u * n);
    memcpy(&d[(size_t)i * ld], dist + (size_t)i * n, 4u * n);
  }
  aco::IterState st{};
  aco::Instance I{};
  I.n = n;
  I.m = ants;
  I.ld = ld;
  I.ldt = n + 1;
  I.ldm = (ants + 31) / 32 * 32;
  I.seed = seed;
  I.choice = ch.data();
  I.dist = d.data();
  I.tours = tours;
  I.lens = lens;
  std::vector<uint32_t> nbr((size_t)cities * I.ldm);
  I.nbr = nbr.data();
  I.st = &st;
  job = Job{I, ants, lane_copy};
  src_lo = reinterpret_cast<const char*>(ch.data());
  src_hi = src_lo + ch.size() * 4;
  memset(smem, 0xff, sizeof smem);
  memset(writer, 0, sizeof writer);
  groups.clear();
  mbars.clear();
  broken = false;
  unfenced = late = reused = copies = 0;
  emu::stall = stall;
  const int threads = G * 32;
  fibres = std::vector<Fibre>(threads);
  for (auto& f : fibres) {
    f.stack.resize(1 << 16);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = f.stack.size();
    f.ctx.uc_link = nullptr;
    makecontext(&f.ctx, entry, 0);
  }
  std::mt19937 rng(schedule);
  std::vector<int> ready;
  while (!broken) {
    ready.clear();
    bool all = true;
    for (int i = 0; i < threads; ++i) {
      const Fibre& f = fibres[i];
      if (f.done) continue;
      all = false;
      if (!f.at || f.at->gen != f.gen) ready.push_back(i);
    }
    if (all) break;
    if (ready.empty()) {
      broken = true;
      break;
    }
    self = ready[rng() % ready.size()];
    fibres[self].at = nullptr;
    tid = uint3{(unsigned)self, 0u, 0u};
    swapcontext(&home, &fibres[self].ctx);
  }
  counts[0] = unfenced;
  counts[1] = late;
  counts[2] = st.status;
  counts[3] = reused;
  return broken ? 1 : 0;
}
