// Batched LAP kernel (one warp per LAP) and the rlt2_lap_batched entry point.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "rlt2_internal.h"
#include "rlt2_lap.cuh"

namespace rlt2 {

int default_group(int m) { return m <= 8 ? 8 : (m <= 16 ? 16 : 32); }

// The fixed-point Z stage with prefetching (a.prefetch): each group's next tile
// and start duals are copied into shared memory by cp.async while the current
// LAP is solved, so the tile's HBM latency is off the warp's path.  The copy
// of tile k+1 is issued as soon as the column reduction of tile k has
// converted its raw entries (group_lap_fx's hook); the grid exponent of a tile is
// the largest exponent field of its raw entries, as in stage_tile.  Results
// are those of the staged form bit for bit.  With a.head set, warps claim
// their next step of 32/G LAPs from that counter (zero at launch) when they
// issue its copies, so that warps whose LAPs needed few searches take more of
// them and all warps end together; otherwise they take a fixed grid stride.
template <int PER>
__device__ __forceinline__ long long claim_step(const LapArgs& a, long long t, int lane) {
  if (a.head == nullptr || t < a.fixed_part) return t;
  unsigned long long b = 0;
  if (lane == 0) b = atomicAdd(a.head, (unsigned long long)PER);
  return a.fixed_part + (long long)__shfl_sync(kFull, b, 0);
}

// The same for LAPs whose two tile buffers would leave too few warps on an SM
// (launch_lap's rule): one tile per warp, converted onto the grid in place.
// The next tile is only prefetched into L2 while the current one is solved and
// copied into shared memory after it; the other warps cover that latency.
template <bool RR>
__device__ __forceinline__ void k_lap_one_tile(const LapArgs& a, unsigned char* base, int lane, bool warm,
                                               long long first, long long stride) {
  using T = long long;
  constexpr int G = 32;
  const int m = a.m, ld = tile_ld(m), mm = m * m;
  T* tile = reinterpret_cast<T*>(base);
  T* uv = tile + (size_t)m * ld;
  int* scr = reinterpret_cast<int*>(uv + 32);
  const double* raw = reinterpret_cast<const double*>(tile);
  unsigned long long aug_acc = 0, relax_acc = 0;
  auto slot = [&](long long tb) { return a.map ? (long long)a.map[tb] : tb; };
  // entries e = lane, lane + 32, ... of the tile, (r, c) advanced without a division per entry
  const int q32 = 32 / m, r32 = 32 - q32 * m, r_first = lane / m, c_first = lane - r_first * m;
  for (int r = lane; r < m; r += 32)
    if (ld > m) tile[r * ld + m] = 0;  // the padding column takes part in the exponent sweep
  long long t = claim_step<1>(a, first, lane);
  long long t_static = first;
  while (t < a.batch) {
    const long long ts = slot(t);
    const double* src = a.A + ts * mm;
    for (int e = lane, r = r_first, c = c_first; e < mm; e += 32) {
      cp_async8(tile + r * ld + c, src + e);
      r += q32;
      c += r32;
      if (c >= m) {
        c -= m;
        ++r;
      }
    }
    cp_async_commit();
    const double u0d = (warm && lane < m) ? __ldcs(a.u0 + ts * m + lane) : 0.0;
    cp_async_wait_all();
    __syncwarp();
    unsigned eb = 0;
    for (int e = lane; e < m * ld; e += 32) eb = max(eb, fx_expfield_hi(raw + e));
    eb = __reduce_max_sync(kFull, eb);
    const int L = fx_grid(eb);
    const T u0 = (warm && lane < m) ? start_dual<true>(u0d, L) : T(0);
    long long next = a.batch;
    auto advance = [&]() {
      t_static += stride;
      next = claim_step<1>(a, t_static, lane);
      if (next < a.batch) {
        const char* p = reinterpret_cast<const char*>(a.A + slot(next) * mm);
        for (int o = lane * 128; o < mm * 8; o += 32 * 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
      }
    };
    WarpLapResult<T> R;
    if (!warm && eb == 0 && group_all_zero<32>(raw, m * ld, lane, 1)) {
      zero_tile_result(R, lane, m);
      advance();
    } else {
      R = group_lap_fx<G, RR>(tile, ld, m, lane, warm, u0, scr, uv, raw, ld, L, advance);
    }
    if (lane < m) {
      if (a.u) a.u[ts * m + lane] = out_value<true>(R.u, L);
      if (a.v) a.v[ts * m + lane] = out_value<true>(R.v, L);
      if (a.r2c) a.r2c[ts * m + lane] = R.r2c;
    }
    if (lane == 0) {
      a.value[ts] = out_value<true>(R.value, L);
      if (a.naug) a.naug[ts] = R.naug;
      aug_acc += R.naug;
      relax_acc += R.nrelax;
    }
    __syncwarp();
    t = next;
  }
  if (a.stats && lane == 0 && (aug_acc | relax_acc)) {
    atomicAdd(a.stats + 0, aug_acc);
    atomicAdd(a.stats + 1, relax_acc);
  }
}

template <int G, bool RR>
__device__ __forceinline__ void k_lap_prefetching(const LapArgs& a, unsigned char* base, int lane, bool warm,
                                                  long long first, long long stride) {
  using T = long long;
  constexpr int per = 32 / G;
  const int grp = lane / G, gl = lane & (G - 1);
  const int m = a.m, ld = tile_ld(m), mm = m * m;
  T* tile = reinterpret_cast<T*>(base) + (size_t)grp * m * ld;
  T* uv = reinterpret_cast<T*>(base) + (size_t)per * m * ld;  // [0..31] u, [32..63] v
  int* scr = reinterpret_cast<int*>(uv + 64) + grp * G;
  double* raw = reinterpret_cast<double*>(base + warp_smem_bytes(m, G)) + (size_t)grp * raw_group_doubles(m);
  unsigned long long aug_acc = 0, relax_acc = 0;
  // copies of group grp's tile of the step starting at LAP t0 (nothing past the batch)
  auto issue = [&](long long t0) {
    const long long tb = t0 + grp;
    if (tb < a.batch) {
      const long long t = a.map ? (long long)a.map[tb] : tb;
      const double* src = a.A + t * mm;
      if (a.wide) {
#pragma unroll 2
        for (int e = 2 * gl; e < mm; e += 2 * G) cp_async16(raw + e, src + e);
      } else {
        for (int e = gl; e < mm; e += G) cp_async8(raw + e, src + e);
      }
      if (warm && gl < m) cp_async8(raw + mm + gl, a.u0 + t * m + gl);
    }
    cp_async_commit();
  };
  // the first LAP of this warp's next step (every lane of the warp); t = the
  // step's place in the fixed stride
  auto claim = [&](long long t) -> long long { return claim_step<per>(a, t, lane); };
  long long t0 = claim(first);
  long long t_static = first;
  issue(t0);
  while (t0 < a.batch) {
    const long long tb = t0 + grp;
    const bool have = tb < a.batch;
    const long long t = (have && a.map) ? (long long)a.map[tb] : tb;
    cp_async_wait_all();
    __syncwarp();
    unsigned eb = 0;
    if (have)
#pragma unroll 4
      for (int e = gl; e < mm; e += G) eb = max(eb, fx_expfield_hi(raw + e));
    if constexpr (G == 32) {
      eb = __reduce_max_sync(kFull, eb);
    } else {
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) eb = max(eb, __shfl_xor_sync(kFull, eb, off));
    }
    const int L = fx_grid(eb);
    T u0 = T(0);
    if (warm && have && gl < m) u0 = start_dual<true>(raw[mm + gl], L);
    long long next = a.batch;  // claimed in the hook, which group_lap_fx calls once (raw is set)
    auto advance = [&]() {
      t_static += stride;
      next = claim(t_static);
      issue(next);
    };
    bool zero = false;  // this group's tile, from a cold start
    if (!warm && __any_sync(kFull, have && eb == 0)) {
      const bool all = group_all_zero<G>(raw, have ? mm : 0, gl, 1);
      zero = have && all;
    }
    WarpLapResult<T> R;
    if (__any_sync(kFull, have && !zero)) {
      R = group_lap_fx<G, RR>(tile, ld, have && !zero ? m : 0, lane, warm, u0, scr, uv + grp * G, raw, m, L, advance);
    } else {
      __syncwarp();  // every lane's reads of raw are done
      advance();
    }
    if (zero) zero_tile_result(R, gl, m);
    if (have && gl < m) {
      if (a.u) a.u[t * m + gl] = out_value<true>(R.u, L);
      if (a.v) a.v[t * m + gl] = out_value<true>(R.v, L);
      if (a.r2c) a.r2c[t * m + gl] = R.r2c;
    }
    if (have && gl == 0) {
      a.value[t] = out_value<true>(R.value, L);
      if (a.naug) a.naug[t] = R.naug;
      aug_acc += R.naug;
      relax_acc += R.nrelax;
    }
    __syncwarp();
    t0 = next;
  }
  cp_async_wait_all();  // nothing may be in flight when the warp leaves
  if (a.stats && gl == 0 && (aug_acc | relax_acc)) {
    atomicAdd(a.stats + 0, aug_acc);
    atomicAdd(a.stats + 1, relax_acc);
  }
}

// Resident blocks that the registers are cut for.  G = 32: four (64 registers)
// against three (77): Z stage at n = 20 370 against 399 us, n = 30 3.38 against
// 3.65 ms; G = 16: three against four: n = 12 34.0 against 39.5 us.
template <int G>
constexpr int kLapBlocks = G == 16 ? 3 : 4;

// Grid-stride over LAPs, 32/G LAPs per warp per step.  FX selects the exact
// fixed-point arithmetic (canonical duals) with prefetching, else FP64; RR
// (fixed point, cold launches) reduces the rows of a cold start first.
template <int G, bool FX, bool RR = false>
__global__ void __launch_bounds__(kMaxWarpsPerBlock * 32, kLapBlocks<G>) k_lap(LapArgs a) {
  dependent_begin();
  if (a.skip && *a.skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const bool warm = a.u0 != nullptr && (a.warm_gate == nullptr || *a.warm_gate != 0);
  const long long nwarps = (long long)gridDim.x * wpb;
  constexpr int per = 32 / G;
  if constexpr (FX) {
    if constexpr (G == 32) {
      if (a.prefetch == 2) {
        k_lap_one_tile<RR>(a, smem_raw + (size_t)wib * warp_smem_bytes_one(a.m), lane, warm,
                           (long long)blockIdx.x * wpb + wib, nwarps);
        return;
      }
    }
    k_lap_prefetching<G, RR>(a, smem_raw + (size_t)wib * warp_smem_bytes_async(a.m, G), lane, warm,
                             ((long long)blockIdx.x * wpb + wib) * per, nwarps * per);
  } else {
    const int grp = lane / G, gl = lane & (G - 1);
    const int m = a.m, ld = tile_ld(m), mm = m * m;
    unsigned char* base = smem_raw + (size_t)wib * warp_smem_bytes(m, G);
    double* tile = reinterpret_cast<double*>(base) + (size_t)grp * m * ld;
    double* uv = reinterpret_cast<double*>(base) + (size_t)per * m * ld;  // [0..31] u, [32..63] v
    int* scr = reinterpret_cast<int*>(uv + 64) + grp * G;
    unsigned long long aug_acc = 0, relax_acc = 0;
    for (long long t0 = ((long long)blockIdx.x * wpb + wib) * per; t0 < a.batch; t0 += nwarps * per) {
      const long long tb = t0 + grp;
      const bool have = tb < a.batch;
      const long long t = (have && a.map) ? (long long)a.map[tb] : tb;
      stage_tile<G, false>(tile, ld, m, gl, have ? a.A + t * mm : nullptr, nullptr);
      const double u0 = (warm && have && gl < m) ? a.u0[t * m + gl] : 0.0;
      __syncwarp();
      bool zero = false;  // +0 throughout, cold: a glance at the first row's start, then all of the tile
      if (!warm && __all_sync(kFull, !have || gl >= m || __double_as_longlong(tile[gl]) == 0)) {
        bool all = true;  // rows are ld apart: one at a time
        for (int r = 0; r < m; ++r) all = group_all_zero<G>(tile + r * ld, have ? m : 0, gl, 0) && all;
        zero = have && all;
      }
      WarpLapResult<double> R;
      if (__any_sync(kFull, have && !zero))
        R = group_lap<G, true>(tile, ld, have && !zero ? m : 0, lane, warm, u0, a.dual_mode, scr, uv + grp * G);
      if (zero) zero_tile_result(R, gl, m);
      if (have && gl < m) {
        if (a.u) a.u[t * m + gl] = R.u;
        if (a.v) a.v[t * m + gl] = R.v;
        if (a.r2c) a.r2c[t * m + gl] = R.r2c;
      }
      if (have && gl == 0) {
        a.value[t] = R.value;
        if (a.naug) a.naug[t] = R.naug;
        aug_acc += R.naug;
        relax_acc += R.nrelax;
      }
      __syncwarp();
    }
    if (a.stats && gl == 0 && (aug_acc | relax_acc)) {
      atomicAdd(a.stats + 0, aug_acc);
      atomicAdd(a.stats + 1, relax_acc);
    }
  }
}

// The Y and X stages: few LAPs whose latency is the stage's time, costs A + Badd
// in, reduced costs out.  A block of four warps per LAP stages the tile (all of
// a thread's loads in flight at once, the grid from a block maximum, converted
// in registers) and writes the reduced costs; its first warp solves the LAP.
// One warp per LAP spent 6 us of the X stage's 19 (n = 20) on staging.  n = 20: Y
// 22.9 -> 17.9 us, X 19.1 -> 14.3; n = 12: 14.3 -> 12.7, 11.6 -> 9.7.
constexpr int kBlockThreads = 128;
template <bool FX, bool RR>
__global__ void __launch_bounds__(kBlockThreads) k_lap_block(LapArgs a) {
  dependent_begin();
  if (a.skip && *a.skip) return;
  using T = typename std::conditional<FX, long long, double>::type;
  constexpr int kPer = 32 * 32 / kBlockThreads;  // entries of a thread, m = 32
  __shared__ T tile[32 * 33];
  __shared__ T uv[64];  // [0..31] u, [32..63] v
  __shared__ int scr[32];
  __shared__ unsigned top[kBlockThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, m = a.m, ld = tile_ld(m), mm = m * m;
  const long long t = a.map ? (long long)a.map[blockIdx.x] : (long long)blockIdx.x;
  const bool warm = a.u0 != nullptr && (a.warm_gate == nullptr || *a.warm_gate != 0);
  const double* src = a.A + t * mm;
  const double* add = a.Badd ? a.Badd + t * mm : nullptr;
  double x[kPer], y[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int e = tid + k * kBlockThreads;
    x[k] = e < mm ? __ldcs(src + e) : 0.0;
    y[k] = (add && e < mm) ? __ldcs(add + e) : 0.0;
  }
  const double u0d = (warm && tid < m) ? a.u0[t * m + tid] : 0.0;
  unsigned eb = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (add) x[k] = __dadd_rn(x[k], y[k]);
    if constexpr (FX) eb = max(eb, fx_expfield(x[k]));  // entries past the tile are 0
  }
  int L = 0;
  if constexpr (FX) {
    eb = __reduce_max_sync(kFull, eb);
    if (lane == 0) top[tid >> 5] = eb;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kBlockThreads / 32; ++w) eb = max(eb, top[w]);
    L = fx_grid(eb);
  }
  // (r, c) of entry tid + k kBlockThreads, advanced without a division per entry
  const int rq = kBlockThreads / m, cq = kBlockThreads - rq * m, r0 = tid / m, c0 = tid - r0 * m;
  auto entries = [&](auto&& f) {
    int r = r0, c = c0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (tid + k * kBlockThreads < mm) f(k, r, c);
      r += rq;
      c += cq;
      if (c >= m) {
        c -= m;
        ++r;
      }
    }
  };
  entries([&](int k, int r, int c) {
    if constexpr (FX) tile[r * ld + c] = fx_floor(x[k], L, kFxEntryBits);
    else tile[r * ld + c] = x[k];
  });
  __syncthreads();
  if (tid < 32) {
    WarpLapResult<T> R;
    const T u0 = (warm && lane < m) ? start_dual<FX>(u0d, L) : T(0);
    if constexpr (FX) R = group_lap_fx<32, RR>(tile, ld, m, lane, warm, u0, scr, uv);
    else R = group_lap<32, false>(tile, ld, m, lane, warm, u0, a.dual_mode, scr, uv);
    uv[lane] = R.u;
    uv[32 + lane] = R.v;
    if (lane < m) {
      if (a.u) a.u[t * m + lane] = out_value<FX>(R.u, L);
      if (a.v) a.v[t * m + lane] = out_value<FX>(R.v, L);
      if (a.r2c) a.r2c[t * m + lane] = R.r2c;
    }
    if (lane == 0) {
      a.value[t] = out_value<FX>(R.value, L);
      if (a.naug) a.naug[t] = R.naug;
      if (a.stats) {
        atomicAdd(a.stats + 0, (unsigned long long)R.naug);
        atomicAdd(a.stats + 1, (unsigned long long)R.nrelax);
      }
    }
  }
  if (!a.pi) return;
  __syncthreads();
  double* dst = a.pi + t * mm;
  entries([&](int k, int r, int c) {
    dst[tid + k * kBlockThreads] = out_value<FX>(lap_sub(lap_sub(tile[r * ld + c], uv[r]), uv[32 + c]), L);
  });
}

using LapKernel = void (*)(LapArgs);

cudaError_t launch_lap_blocks(const LapArgs& a, cudaStream_t s) {
  if (a.batch <= 0) return cudaSuccess;
  if (a.m < 1 || a.m > 32 || a.batch > 0x7fffffffll) return cudaErrorInvalidValue;
  const int grid = (int)a.batch;
  const LapKernel kern =
      a.dual_mode != 1 ? k_lap_block<false, false> : (a.u0 ? k_lap_block<true, false> : k_lap_block<true, true>);
  return launch_dependent(kern, grid, kBlockThreads, 0, s, a);
}

static int gidx(int G) { return G == 8 ? 0 : (G == 16 ? 1 : 2); }

// The forms of k_lap: FP64, fixed point, fixed point with the row reduction of
// cold starts.
constexpr int kForms = 3;
template <int G>
static LapKernel lap_kernel(int form) {
  return form == 0 ? k_lap<G, false> : form == 1 ? k_lap<G, true> : k_lap<G, true, true>;
}
static LapKernel lap_kernel(int G, int form) {
  return G == 8 ? lap_kernel<8>(form) : (G == 16 ? lap_kernel<16>(form) : lap_kernel<32>(form));
}
static int lap_form(const LapArgs& a) { return a.dual_mode != 1 ? 0 : (a.u0 ? 1 : 2); }

// A launch of one form on the current device: its resident blocks and, for the
// fixed-point forms, a.prefetch (1 two tile buffers per warp, 2 the one-tile form).
struct LapPlan {
  int occ = 0;  // resident blocks per SM, 0 = not configured
  int prefetch = 0;
  size_t smem = 0;
};

// Launch configuration, kept per device and set once per (device, size; for nodes
// also lanes and warps) under g_cfg_mu: contexts may be created and used from different host
// threads and on different devices.  Like every per-device cache of the library
// it is not valid across a cudaDeviceReset.
static std::mutex g_cfg_mu;
constexpr int kMaxCfgDevices = 64;
struct LapDevCfg {
  int sms = 0;                        // multiprocessors of the device
  LapPlan plan[33][kForms];           // k_lap, for (m, form)
  int occ_nodes[33][3][2] = {};
  bool attr[3] = {};                  // dynamic shared-memory attribute set (k_lap, per G)
  bool attr_nodes[3] = {};            // the same for k_lap_nodes
};
static LapDevCfg g_devcfg[kMaxCfgDevices];

// The current device's entry, its SM count read on first use (g_cfg_mu held).
static cudaError_t current_cfg(LapDevCfg** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxCfgDevices) return cudaErrorInvalidDevice;
  LapDevCfg& c = g_devcfg[dev];
  if (!c.sms && (e = cudaDeviceGetAttribute(&c.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  *out = &c;
  return cudaSuccess;
}

// Every form of size m.  A fixed-point form takes two tile buffers per
// warp unless one tile alone lets more warps onto an SM: m = 28 (16 -> 32
// warps), not m = 18 (32 either way).
static cudaError_t prepare_one(LapDevCfg& cfg, int m) {
  const int G = default_group(m);
  constexpr int wpb = kMaxWarpsPerBlock;
  LapPlan* plan = cfg.plan[m];
  if (plan[kForms - 1].occ > 0) return cudaSuccess;
  cudaError_t e;
  const int cap = (int)(warp_smem_bytes_async(32, 32) * kMaxWarpsPerBlock);
  for (int k = 0; k < kForms; ++k) {
    const LapKernel kern = lap_kernel(G, k);
    if (!cfg.attr[gidx(G)] &&
        (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, cap)) != cudaSuccess)
      return e;
    auto occupancy = [&](size_t per_warp, int* o) {
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(o, kern, wpb * 32, per_warp * wpb);
    };
    LapPlan p;
    p.prefetch = k > 0 ? 1 : 0;
    p.smem = (p.prefetch ? warp_smem_bytes_async(m, G) : warp_smem_bytes(m, G)) * wpb;
    if ((e = occupancy(p.smem / wpb, &p.occ)) != cudaSuccess) return e;
    if (p.prefetch && G == 32) {
      int one = 0;
      if ((e = occupancy(warp_smem_bytes_one(m), &one)) != cudaSuccess) return e;
      if (one > p.occ) {
        p.occ = one;
        p.prefetch = 2;
        p.smem = warp_smem_bytes_one(m) * wpb;
      }
    }
    if (p.occ < 1) p.occ = 1;
    plan[k] = p;
  }
  cfg.attr[gidx(G)] = true;
  return cudaSuccess;
}

// The plan of an m-column LAP launch on the current device (configured on
// first use), *cap its resident block count.
static cudaError_t prepare_plan(int m, int form, LapPlan* plan, long long* cap) {
  if (m < 1 || m > 32) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(g_cfg_mu);
  LapDevCfg* cfg = nullptr;
  cudaError_t e = current_cfg(&cfg);
  if (e != cudaSuccess) return e;
  if ((e = prepare_one(*cfg, m)) != cudaSuccess) return e;
  *plan = cfg->plan[m][form];
  *cap = (long long)cfg->sms * plan->occ;
  return cudaSuccess;
}

cudaError_t prepare_lap(int m) {
  LapPlan plan;
  long long cap = 0;
  return prepare_plan(m, 0, &plan, &cap);
}

cudaError_t launch_lap(const LapArgs& a, cudaStream_t s) {
  if (a.batch <= 0) return cudaSuccess;
  const int G = default_group(a.m);
  constexpr int wpb = kMaxWarpsPerBlock;
  if (a.Badd || a.pi) return cudaErrorInvalidValue;  // launch_lap_blocks
  // a cold fixed-point launch reduces the rows first (the same canonical result)
  const int form = lap_form(a);
  LapPlan plan;
  long long cap = 0;
  cudaError_t e = prepare_plan(a.m, form, &plan, &cap);
  if (e != cudaSuccess) return e;
  LapArgs b = a;
  b.prefetch = plan.prefetch;
  b.wide = !(a.m & 1) && (reinterpret_cast<std::uintptr_t>(a.A) & 15) == 0;
  const long long per_block = (long long)wpb * (32 / G);
  const long long need = (a.batch + per_block - 1) / per_block;
  const int grid = (int)(need < cap ? need : cap);
  if (!b.prefetch || need <= cap) b.head = nullptr;  // one step per warp: nothing to share out
  if (b.head) {
    // half of the steps by fixed stride, the rest from the queue, so that the
    // warps still end together: the counter is one address, and at n = 20 the
    // 144,400 claims alone take 160 us (Z stage: none by stride 374 us, half 370,
    // three quarters 397)
    const long long round = (long long)grid * per_block;
    b.fixed_part = a.batch / round / 2 * round;
    if (!b.head_zeroed && (e = cudaMemsetAsync(b.head, 0, sizeof(unsigned long long), s)) != cudaSuccess) return e;
  }
  if (a.dependent) return launch_dependent(lap_kernel(G, form), grid, wpb * 32, plan.smem, s, b);
  lap_kernel(G, form)<<<grid, wpb * 32, plan.smem, s>>>(b);
  return cudaGetLastError();
}

bool lap_wants_queue(long long batch, int m) {
  LapPlan plan;
  long long cap = 0;
  if (prepare_plan(m, 1, &plan, &cap) != cudaSuccess) return false;
  return batch > cap * kMaxWarpsPerBlock * (32 / default_group(m));
}

// ---------------------------------------------------------------------------
// Batched branch-and-bound nodes: one persistent launch per stage over the LAPs
// of every node of a wave.  Warps pull 32/G LAPs at a time from a device queue
// (atomic head, no waiting), so nodes of uneven size share the GPU.
// The queue-fed node form of k_lap_prefetching (fixed point, Z stages): a
// warp claims its next queue slot before it solves the current one and copies
// that slot's tiles and start duals into shared memory by cp.async (issued by
// group_lap_fx's hook once the current raw tiles are converted).  The raw buffers
// are sized for the largest LAP of the stage.  Results are those of the staged
// form bit for bit (each LAP is independent of which warp solves it).
template <int G, bool RR>
__device__ __forceinline__ void k_lap_nodes_prefetching(const NodeLapArgs& a, const long long* s_prefix,
                                                        unsigned char* base, int lane) {
  using T = long long;
  constexpr int per = 32 / G;
  const int grp = lane / G, gl = lane & (G - 1);
  const int MM = a.max_m;
  T* tile = reinterpret_cast<T*>(base) + (size_t)grp * MM * tile_ld(MM);
  T* uv = reinterpret_cast<T*>(base) + (size_t)per * MM * tile_ld(MM);
  int* scr = reinterpret_cast<int*>(uv + 64) + grp * G;
  double* raw = reinterpret_cast<double*>(base + warp_smem_bytes(MM, G)) + (size_t)grp * raw_group_doubles(MM);
  unsigned long long aug_acc = 0, relax_acc = 0;
  // the queue slot's LAP of this group: node k, LAP li of that node (have = false past the end or for a
  // stopped node)
  struct Slot {
    bool have, warm;
    int k;
    long long li;
  };
  auto lookup = [&](unsigned long long b0) {
    Slot sl{false, false, 0, 0};
    const long long t = (long long)b0 + grp;
    if (b0 < (unsigned long long)a.total && t < a.total) {
      int lo = 0, hi = a.nnodes - 1;
      while (lo < hi) {  // largest k with prefix[k] <= t
        const int mid = (lo + hi + 1) >> 1;
        if (s_prefix[mid] <= t) lo = mid;
        else hi = mid - 1;
      }
      sl.k = lo;
      const NodeLapItem& it = a.items[lo];
      sl.li = RLT2_IDX(t - s_prefix[lo], it.count);
      sl.have = *it.skip == 0;
      sl.warm = sl.have && it.u0 != nullptr && (it.warm_gate == nullptr || *it.warm_gate != 0);
    }
    return sl;
  };
  auto grab = [&]() {
    unsigned long long b0 = 0;
    if (lane == 0) b0 = atomicAdd(a.head, (unsigned long long)per);
    return __shfl_sync(kFull, b0, 0);
  };
  auto issue = [&](const Slot& sl) {
    if (sl.have) {
      const NodeLapItem& it = a.items[sl.k];
      const int m = it.m, mm = m * m;
      const double* src = it.A + sl.li * mm;
      for (int e = gl; e < mm; e += G) cp_async8(raw + e, src + e);
      if (sl.warm && gl < m) cp_async8(raw + mm + gl, it.u0 + sl.li * m + gl);
    }
    cp_async_commit();
  };
  unsigned long long b0 = grab();
  Slot cur = lookup(b0);
  issue(cur);
  while (b0 < (unsigned long long)a.total) {
    const unsigned long long b1 = grab();
    const Slot nxt = lookup(b1);
    cp_async_wait_all();
    __syncwarp();
    const int m = cur.have ? a.items[cur.k].m : 0;
    const int mm = m * m;
    unsigned eb = 0;
    for (int e = gl; e < mm; e += G) eb = max(eb, fx_expfield_hi(raw + e));
    if constexpr (G == 32) {
      eb = __reduce_max_sync(kFull, eb);
    } else {
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) eb = max(eb, __shfl_xor_sync(kFull, eb, off));
    }
    const int L = fx_grid(eb);
    const T u0 = (cur.warm && gl < m) ? start_dual<true>(raw[mm + gl], L) : T(0);
    bool zero = false;  // this group's tile, from a cold start
    if (__any_sync(kFull, cur.have && !cur.warm && eb == 0)) {
      const bool all = group_all_zero<G>(raw, mm, gl, 1);
      zero = cur.have && !cur.warm && all;
    }
    WarpLapResult<T> R;
    if (__any_sync(kFull, cur.have && !zero)) {
      R = group_lap_fx<G, RR>(tile, tile_ld(m), zero ? 0 : m, lane, cur.warm, u0, scr, uv + grp * G, raw, m, L,
                              [&]() { issue(nxt); });
    } else {
      __syncwarp();  // every lane's reads of raw are done
      issue(nxt);
    }
    if (zero) zero_tile_result(R, gl, m);
    if (cur.have) {
      const NodeLapItem& it = a.items[cur.k];
      if (gl < m) {
        if (it.u) it.u[cur.li * m + gl] = out_value<true>(R.u, L);
        if (it.v) it.v[cur.li * m + gl] = out_value<true>(R.v, L);
        if (it.r2c) it.r2c[cur.li * m + gl] = R.r2c;
      }
      if (gl == 0) {
        it.value[cur.li] = out_value<true>(R.value, L);
        aug_acc += R.naug;
        relax_acc += R.nrelax;
      }
    }
    __syncwarp();
    b0 = b1;
    cur = nxt;
  }
  cp_async_wait_all();  // nothing may be in flight when the warp leaves
  if (a.stats && gl == 0 && (aug_acc | relax_acc)) {
    atomicAdd(a.stats + 0, aug_acc);
    atomicAdd(a.stats + 1, relax_acc);
  }
}

template <int G, bool PRE, bool FX, bool RR = false>
__global__ void __launch_bounds__(kMaxWarpsPerBlock * 32) k_lap_nodes(NodeLapArgs a) {
  using T = typename std::conditional<FX, long long, double>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int per = 32 / G;
  long long* s_prefix = reinterpret_cast<long long*>(smem_raw);
  for (int i = threadIdx.x; i <= a.nnodes; i += blockDim.x) s_prefix[i] = a.prefix[i];
  __syncthreads();
  if constexpr (PRE && FX) {
    if (a.prefetch) {
      const size_t pre = (((size_t)(a.nnodes + 1) * sizeof(long long)) + 255) & ~size_t(255);
      k_lap_nodes_prefetching<G, RR>(a, s_prefix,
                                 smem_raw + pre + (size_t)(threadIdx.x >> 5) * warp_smem_bytes_async(a.max_m, G),
                                 threadIdx.x & 31);
      return;
    }
  }
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int grp = lane / G, gl = lane & (G - 1);
  const size_t pre = (((size_t)(a.nnodes + 1) * sizeof(long long)) + 255) & ~size_t(255);
  const int MM = a.max_m;
  unsigned char* base = smem_raw + pre + (size_t)wib * warp_smem_bytes(MM, G);
  T* tile = reinterpret_cast<T*>(base) + (size_t)grp * MM * tile_ld(MM);
  T* uv = reinterpret_cast<T*>(base) + (size_t)per * MM * tile_ld(MM);
  int* scr = reinterpret_cast<int*>(uv + 64) + grp * G;
  unsigned long long aug_acc = 0, relax_acc = 0;
  for (;;) {
    unsigned long long b0 = 0;
    if (lane == 0) b0 = atomicAdd(a.head, (unsigned long long)per);
    b0 = __shfl_sync(kFull, b0, 0);
    if (b0 >= (unsigned long long)a.total) break;
    const long long t = (long long)b0 + grp;
    bool have = t < a.total;
    int k = 0;
    long long li = 0;
    NodeLapItem it{};
    if (have) {
      int lo = 0, hi = a.nnodes - 1;
      while (lo < hi) {  // largest k with prefix[k] <= t
        const int mid = (lo + hi + 1) >> 1;
        if (s_prefix[mid] <= t) lo = mid;
        else hi = mid - 1;
      }
      k = lo;
      it = a.items[k];
      li = RLT2_IDX(t - s_prefix[k], it.count);
      if (*it.skip) have = false;
    }
    const int m = have ? it.m : 0;
    const int ld = tile_ld(m);
    const int mm = m * m;
    const int L = stage_tile<G, FX>(tile, ld, m, gl, have ? it.A + li * mm : nullptr,
                                    (have && it.Badd) ? it.Badd + li * mm : nullptr);
    const bool warm = have && it.u0 != nullptr && (it.warm_gate == nullptr || *it.warm_gate != 0);
    const T u0 = (warm && gl < m) ? start_dual<FX>(it.u0[li * m + gl], L) : T(0);
    __syncwarp();
    WarpLapResult<T> R;
    if constexpr (FX) R = group_lap_fx<G, RR>(tile, ld, m, lane, warm, u0, scr, uv + grp * G);
    else R = group_lap<G, PRE>(tile, ld, m, lane, warm, u0, a.dual_mode, scr, uv + grp * G);
    if (have && gl < m) {
      if (it.u) it.u[li * m + gl] = out_value<FX>(R.u, L);
      if (it.v) it.v[li * m + gl] = out_value<FX>(R.v, L);
      if (it.r2c) it.r2c[li * m + gl] = R.r2c;
    }
    if (have && gl == 0) {
      it.value[li] = out_value<FX>(R.value, L);
      aug_acc += R.naug;
      relax_acc += R.nrelax;
    }
    uv[lane] = R.u;
    uv[32 + lane] = R.v;
    __syncwarp();
    if (have && it.pi) {
      double* dst = it.pi + li * mm;
      const T* ug = uv + grp * G;
      const T* vg = uv + 32 + grp * G;
      for (int e = gl; e < mm; e += G) {
        const int r = e / m, c = e - r * m;
        dst[e] = out_value<FX>(lap_sub(lap_sub(tile[r * ld + c], ug[r]), vg[c]), L);
      }
    }
    __syncwarp();
  }
  if (a.stats && gl == 0 && (aug_acc | relax_acc)) {
    atomicAdd(a.stats + 0, aug_acc);
    atomicAdd(a.stats + 1, relax_acc);
  }
}

using NodeLapKernel = void (*)(NodeLapArgs);

template <int G>
static NodeLapKernel node_lap_kernel(bool pre, bool fx, bool rr) {
  if (fx && rr) return pre ? k_lap_nodes<G, true, true, true> : k_lap_nodes<G, false, true, true>;
  if (pre) return fx ? k_lap_nodes<G, true, true> : k_lap_nodes<G, true, false>;
  return fx ? k_lap_nodes<G, false, true> : k_lap_nodes<G, false, false>;
}
static NodeLapKernel node_lap_kernel(int G, bool pre, bool fx, bool rr) {
  return G == 8 ? node_lap_kernel<8>(pre, fx, rr)
                : (G == 16 ? node_lap_kernel<16>(pre, fx, rr) : node_lap_kernel<32>(pre, fx, rr));
}

cudaError_t launch_lap_nodes(const NodeLapArgs& a, cudaStream_t s) {
  if (a.total <= 0) return cudaSuccess;
  if (a.max_m < 1 || a.max_m > 32 || a.nnodes < 1 || a.nnodes > kMaxWaveNodes) return cudaErrorInvalidValue;
  const int G = a.group ? a.group : default_group(a.max_m);
  const int wpb = a.warps_per_block ? a.warps_per_block : kMaxWarpsPerBlock;
  if (G < a.max_m || (wpb != 4 && wpb != 8)) return cudaErrorInvalidValue;
  const size_t pre = (((size_t)(a.nnodes + 1) * sizeof(long long)) + 255) & ~size_t(255);
  NodeLapArgs b = a;
  b.prefetch = (a.pre && a.dual_mode == 1) ? 1 : 0;
  const size_t per_warp = b.prefetch ? warp_smem_bytes_async(a.max_m, G) : warp_smem_bytes(a.max_m, G);
  const size_t smem = pre + per_warp * wpb;
  cudaError_t e;
  std::unique_lock<std::mutex> lock(g_cfg_mu);
  LapDevCfg* cfg = nullptr;
  if ((e = current_cfg(&cfg)) != cudaSuccess) return e;
  bool* attr_set = cfg->attr_nodes;
  const size_t cap_smem = (((size_t)(kMaxWaveNodes + 1) * sizeof(long long)) + 255) / 256 * 256 +
                          warp_smem_bytes_async(32, 32) * kMaxWarpsPerBlock;
  int& occ = cfg->occ_nodes[a.max_m][gidx(G)][wpb == 4 ? 0 : 1];
  // occupancy of the slowest of the six forms, computed once per size (the
  // prefix table's share of shared memory varies with the node count; a grid
  // above the resident count only queues blocks, which never wait on others)
  if (!occ) {
    int lo = 1 << 20;
    for (int k = 0; k < 6; ++k) {
      const bool kpre = (k & 1) != 0, kfx = (k & 2) != 0 || k >= 4;
      const NodeLapKernel kern = node_lap_kernel(G, kpre, kfx, k >= 4);
      if (!attr_set[gidx(G)]) {
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap_smem)) !=
            cudaSuccess)
          return e;
      }
      int o = 0;
      const size_t ksmem =
          pre + (kpre && kfx ? warp_smem_bytes_async(a.max_m, G) : warp_smem_bytes(a.max_m, G)) * wpb;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, wpb * 32, ksmem)) != cudaSuccess) return e;
      lo = o < lo ? o : lo;
    }
    attr_set[gidx(G)] = true;
    occ = lo < 1 ? 1 : lo;
  }
  const long long cap = (long long)cfg->sms * occ;
  lock.unlock();
  const long long per_block = (long long)wpb * (32 / G);
  const long long need = (a.total + per_block - 1) / per_block;
  const int grid = (int)(need < cap ? need : cap);
  const NodeLapKernel kern = node_lap_kernel(G, a.pre, a.dual_mode == 1, a.cold && a.dual_mode == 1);
  kern<<<grid, wpb * 32, smem, s>>>(b);
  return cudaGetLastError();
}

RLT2_DEFINE_OOB_QUERY(oob_lap)

}  // namespace rlt2

using namespace rlt2;

extern "C" rlt2_status rlt2_lap_batched(int batch, int m, const double* cost, const double* u0, double* value,
                                        double* u, double* v, int* row_to_col, int* n_aug, int dual_mode,
                                        void* stream) {
  if (batch < 0 || m < 1 || m > 32 || (batch > 0 && (!cost || !value)) || dual_mode < 0 || dual_mode > 2) {
    set_error("rlt2_lap_batched: invalid argument");
    return RLT2_EINVAL;
  }
  if (batch == 0) return RLT2_OK;
  LapArgs a{};
  a.batch = batch;
  a.m = m;
  a.A = cost;
  a.u0 = u0;
  a.value = value;
  a.u = u;
  a.v = v;
  a.r2c = row_to_col;
  a.naug = n_aug;
  a.dual_mode = dual_mode;
  const cudaStream_t s = (cudaStream_t)stream;
  // the fixed-point form's LAP queue: 8 stream-ordered bytes of the library's
  // pool, freed after the launch (without them the warps take a fixed stride;
  // the results are the same).  A batch that the resident warps hold at once
  // needs none
  unsigned long long* head = nullptr;
  if (dual_mode == 1 && lap_wants_queue(batch, m)) {
    // under stream capture the pool may not be created: the default one then
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaMemPool_t pool = nullptr;
    const bool own = cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone &&
                     library_pool(&pool) == cudaSuccess;
    const cudaError_t ea = own ? cudaMallocFromPoolAsync((void**)&head, sizeof(unsigned long long), pool, s)
                               : cudaMallocAsync((void**)&head, sizeof(unsigned long long), s);
    if (ea != cudaSuccess) head = nullptr;
    (void)cudaGetLastError();
  }
  a.head = head;
  a.dependent = 1;  // small batches back to back: 400 LAPs of size 7 14.7 -> 12.8 us a call
  cudaError_t e = launch_lap(a, s);
  if (head) {
    const cudaError_t ef = cudaFreeAsync(head, s);
    if (e == cudaSuccess) e = ef;
  }
  if (e != cudaSuccess) return cuda_fail(e, "rlt2_lap_batched");
  return RLT2_OK;
}
