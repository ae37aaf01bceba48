// Warp-level (group-per-LAP) Hungarian for sm_103a (GB300).
//
// Every LAP of the RLT2 dual ascent is small (Z: n-2, Y: n-1, X: n; n <= 32), so
// a group of G = 8, 16 or 32 lanes owns one LAP (32/G LAPs per warp, in
// lockstep): lane c holds column c (dual v_c, Dijkstra label d_c,
// predecessor row, "scanned" flag, matched row) and lane r holds row r (dual
// u_r, matched column).  The cost tile sits in shared memory with an odd row
// stride so that both row reads (lanes = columns) and column reads (lanes =
// rows) are bank-conflict free.  This replaces the paper's tiled alternating-
// tree Hungarian (Section 3.2, written for Kepler): no cross-LAP coupling, no
// host round trips, one launch per stage.
//
// GB300 runs FP64 at ~1/70 of its FP32 rate, and FP64 compares and min/max use
// the same slow pipe, so every comparison below is done on 64-bit integer
// keys that order exactly like the values (okey for doubles), and every argmin
// is a two-step warp integer min reduction (redux.sync) plus a ballot.  In the
// FP64 form the only FP64 instructions left are the additions the method
// needs; the fixed-point form has none outside the output conversions.
//
// Two arithmetic forms, chosen per launch:
//   FP64      IEEE double, round to nearest, in the CPU oracle's operation order
//             (raw duals match it bit for bit); used for raw duals and for the
//             FP64 canonical mode.
//   fixed     exact 64-bit integer arithmetic on a per-tile grid (canonical
//             duals, the default).  The tile is rounded down onto the grid
//             2^L with L = E - 48, where 2^E bounds every |entry|; the start
//             duals are rounded down and clamped to |u0| <= 2^(E+1).  Every
//             quantity the Hungarian and the canonical pass form then stays
//             below 2^59 grid steps for m <= 32 (labels are bounded by the
//             growth of the matching cost, duals by the labels), so no
//             addition can overflow, and the result is the exact optimum and
//             the exact canonical dual of the rounded tile (whose entries are
//             within 2^-47 of the tile's magnitude of the given ones): the
//             same for every start, so warm and cold solves agree bit for bit,
//             and dual feasible for the given tile too (rounding down only
//             lowers costs).  GB300 issues integer additions ~40x faster than
//             FP64 ones.
//             The bounds, in grid steps: |c| < 2^48 and |u0| <= 2^49 give start
//             column duals below 2^49.6; a search's sink label is the growth
//             of the matching's cost minus u_i + v_sink, so the sink labels of
//             all searches sum below 2^56 and every dual stays below 2^56.2;
//             reduced costs are below 2^57.1 and labels below 2^57.6; the
//             canonical pass's distances are u^c_r - (u_r - u_0) with
//             |u^c| < 31 * 2^49 < 2^54, below 2^57.3, candidates below 2^58.3.
//
// Order of the operations (the oracle's, by specification; exact in fixed point):
//   start     u = u0 or 0;  v_c = min_r (c_rc - u_r), ties to the lowest row
//   greedy    column c takes its argmin row if no lower column took that row
//   search    for every free row i (increasing): Dijkstra on reduced costs
//             pi(r,c) = (c_rc - u_r) - v_c; labels d_c = d_last + pi(r,c);
//             pick the unscanned column of least label (lowest index on ties);
//             relax only on strict '<'; stop at the first free column.
//   duals     v_c = v_c + (d_c - d_sink) on scanned columns, augment, then
//             u_r = c_{r,sigma(r)} - v_{sigma(r)} for every matched row
//   value     sum_r c_{r,sigma(r)} as a pairwise tree (lane i += lane i+h, h = P/2..1);
//             exact in fixed point, where one LAP per warp sums by warp reductions
//   canonical (dual_mode 1, 2) Dijkstra from row 0 over arcs r'->r with weight
//             pi(r, sigma(r')) (>= 0), u^c_r = dist_r + (u_r - u_0),
//             v^c_c = c_{sigma^-1(c),c} - u^c_{sigma^-1(c)}
#pragma once
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "rlt2_internal.h"

namespace rlt2 {

constexpr unsigned kFull = 0xffffffffu;

// Order-preserving 64-bit key of a double (non-NaN): a < b  <=>  okey(a) < okey(b),
// with -0 and +0 equal, exactly as the IEEE comparison.
__device__ __forceinline__ unsigned long long okey(double x) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  b = (b == 0x8000000000000000ull) ? 0ull : b;
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Lane holding the least key; lowest lane on ties.  The low words are compared
// only when several lanes share the least high word (a warp-uniform branch).
__device__ __forceinline__ int warp_argmin(unsigned long long key) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mhi = __reduce_min_sync(kFull, hi);
  unsigned ball = __ballot_sync(kFull, hi == mhi);
  if (ball & (ball - 1u)) {
    const unsigned mlo = __reduce_min_sync(kFull, hi == mhi ? lo : 0xffffffffu);
    ball = __ballot_sync(kFull, hi == mhi && lo == mlo);
  }
  return __ffs(ball) - 1;
}

__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }

// ---- fixed-point grid of a tile -------------------------------------------
// Biased exponent field of a double (0 for zeros and subnormals).
__device__ __forceinline__ unsigned fx_expfield(double x) {
  return (unsigned)(((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ffull);
}
// Grid exponent L of a tile whose largest exponent field is eb: every entry is
// below 2^E with E = max(eb, 1) - 1022, and L = E - 48.
__device__ __forceinline__ int fx_grid(unsigned eb) { return (int)(eb ? eb : 1u) - 1070; }

// floor(x / 2^L) for |x| < 2^(L + lim) (lim <= 53 + L - e_min keeps the shift
// positive); larger |x| clamp to +-2^lim.  Integer operations only: the signed
// mantissa shifted right arithmetically is the floor for either sign.
__device__ __forceinline__ long long fx_floor(double x, int L, int lim) {
  const long long b = __double_as_longlong(x);
  const int eb = (int)((b >> 52) & 0x7ff);
  const long long mant = (b & 0xFFFFFFFFFFFFFll) | (eb ? (1ll << 52) : 0ll);
  const int e = (eb ? eb : 1) - 1075;  // |x| = mant * 2^e
  if (e + 53 - L > lim) return b < 0 ? -(1ll << lim) : (1ll << lim);
  const int sh = min(L - e, 63);       // >= 53 - lim > 0
  return (b < 0 ? -mant : mant) >> sh;
}

// Biased exponent field from the high word of a double in shared memory.
__device__ __forceinline__ unsigned fx_expfield_hi(const double* p) {
  return (reinterpret_cast<const unsigned*>(p)[1] >> 20) & 0x7ffu;
}

// Asynchronous global -> shared copies of 8 bytes (cp.async, no registers held
// while in flight), committed as one group per call site and awaited with
// cp_async_wait_all (the copies of this thread; a __syncwarp then makes the
// group's copies visible to its lanes).
__device__ __forceinline__ void cp_async8(void* dst_smem, const void* src) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(src) : "memory");
}
// 16 bytes, both sides on a 16-byte boundary.
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// q * 2^L rounded to the nearest double (L >= -1069 by construction of fx_grid).
__device__ __forceinline__ double fx_to_double(long long q, int L) {
  const double p2 = L >= -1022 ? __longlong_as_double((long long)(L + 1023) << 52)
                               : __longlong_as_double(1ll << (L + 1074));
  return __dmul_rn(__ll2double_rn(q), p2);
}

constexpr int kFxEntryBits = 48;  // |entry| < 2^48 grid steps
constexpr int kFxStartBits = 49;  // |u0| <= 2^49 grid steps

template <typename T>
struct WarpLapResult {
  T u;           // row dual of row `gl` (group lane)
  T v;           // column dual of column `gl`
  int r2c;       // column matched to row `gl`
  int c2r;       // row matched to column `gl`
  T value;       // LAP optimum (all lanes of the group)
  int naug;      // augmenting searches
  int nrelax;    // label relaxations (instrumentation for the roofline)
};

// Lowest group lane holding the least key among the G lanes of this lane's
// group (aligned groups of G lanes).  Every lane of the warp must call it.
template <int G>
__device__ __forceinline__ int group_argmin(unsigned long long key, int gb) {
  if constexpr (G == 32) {
    return warp_argmin(key);
  } else if constexpr (G == 16) {
    // two full-warp reductions of the high words, each with the other half's
    // lanes at the maximum (no divergence, unlike a redux.sync on a half-warp
    // mask), the low words only where a half has a tie on the high word
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const bool g0 = gb == 0;
    const unsigned m0 = __reduce_min_sync(kFull, g0 ? hi : 0xffffffffu);
    const unsigned m1 = __reduce_min_sync(kFull, g0 ? 0xffffffffu : hi);
    const unsigned mhi = g0 ? m0 : m1;
    unsigned mine = (__ballot_sync(kFull, hi == mhi) >> gb) & 0xffffu;
    if (__any_sync(kFull, (mine & (mine - 1u)) != 0u)) {
      const bool cand = hi == mhi;
      const unsigned l0 = __reduce_min_sync(kFull, (g0 && cand) ? lo : 0xffffffffu);
      const unsigned l1 = __reduce_min_sync(kFull, (!g0 && cand) ? lo : 0xffffffffu);
      const unsigned mlo = g0 ? l0 : l1;
      mine = (__ballot_sync(kFull, cand && lo == mlo) >> gb) & 0xffffu;
    }
    return __ffs(mine) - 1;
  } else {
    // xor butterfly (a redux.sync on the group's own lane mask was slower
    // here: 0.121 against 0.104 ms per iteration at n = 12)
    unsigned long long k = key;
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_xor_sync(kFull, k, off);
      k = o < k ? o : k;
    }
    const unsigned ball = __ballot_sync(kFull, key == k);
    return __ffs((ball >> gb) & ((1u << G) - 1u)) - 1;
  }
}

template <int G>
__device__ __forceinline__ unsigned group_bits(unsigned ball, int gb) {
  if constexpr (G == 32) return ball;
  else return (ball >> gb) & ((1u << G) - 1u);
}

// Called by group_lap_fx once the column reduction has read the staged raw tile
// (all lanes, after a __syncwarp): the caller may then reuse the raw buffer.
struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};

// Solve one LAP per group of G lanes (32/G LAPs per warp) in lockstep, FP64 in
// the oracle's operation order: every intrinsic is executed by all 32 lanes
// with the full mask and all loops are warp-uniform (they run while any group
// still has work; idle groups only predicate their updates), so the LAPs of
// one warp share every instruction.  Group lane gl = lane % G holds row gl and
// column gl of its LAP.  `cs` is the group's m x m tile (row stride ld) in
// shared memory, `scr` G ints of group scratch, m the group's LAP size (0 = no
// LAP, 1 <= m <= G otherwise).  The arithmetic is identical for every G.
// PRE: the caller does not need the tile afterwards, so the canonical pass may
// replace it by its reduced costs first (uvs: 64 values of group staging).
template <int G, bool PRE>
__device__ __forceinline__ WarpLapResult<double> group_lap(double* __restrict__ cs, int ld, int m, int lane, bool warm,
                                                           double u0, int dual_mode, int* scr, double* uvs) {
  const int gl = lane & (G - 1);
  const int gb = lane - gl;
  const bool cv = gl < m;
  const int M = (G == 32) ? m : (int)__reduce_max_sync(kFull, (unsigned)m);
  WarpLapResult<double> R;
  double u = (cv && warm) ? u0 : 0.0;
  double v = 0.0;
  int naug = 0, nrelax = 0;

  // column reduction with the argmin row
  unsigned long long bestk = ~0ull;
  int arg = -1;
  for (int r = 0; r < M; ++r) {
    const double ur = __shfl_sync(kFull, u, gb + r);
    if (cv && r < m) {
      const double c = cs[r * ld + gl];
      const double x = warm ? dsub(c, ur) : c;  // c - 0 == c exactly
      if (arg < 0 || okey(x) < bestk) {
        bestk = okey(x);
        arg = r;
        v = x;
      }
    }
  }
  // greedy: the lowest column among those sharing an argmin row takes it
  const int marg = cv ? ((lane / G) << 6) + arg : (1 << 20) + lane;
  const unsigned same = __match_any_sync(kFull, marg);
  const bool win = cv && (__ffs(same) - 1) == lane;
  int c2r = win ? arg : -1;
  scr[gl] = -1;
  __syncwarp();
  if (win) scr[arg] = gl;
  __syncwarp();
  int r2c = cv ? scr[gl] : -1;
  __syncwarp();

  // at G = 32 the warp is one group, so every loop condition below is
  // warp-uniform and needs no vote
  unsigned freerows = group_bits<G>(__ballot_sync(kFull, cv && r2c < 0), gb);
  while (G == 32 ? freerows != 0 : __any_sync(kFull, freerows != 0)) {
    const bool act = freerows != 0;  // this group runs a search in this pass
    const int i = act ? __ffs(freerows) - 1 : 0;
    if (act) {
      freerows &= freerows - 1;
      ++naug;
      nrelax += m;
    }
    const double ui = __shfl_sync(kFull, u, gb + i);
    double d = (act && cv) ? dsub(dsub(cs[i * ld + gl], ui), v) : 0.0;
    unsigned long long dk = okey(d);  // cached key of d
    int pred = i;
    bool scanned = !(act && cv);
    bool searching = act;
    int sink = 0;
    double dlast = 0.0;
    while (G == 32 ? searching : __any_sync(kFull, searching)) {
      const int c = group_argmin<G>(scanned ? ~0ull : dk, gb);
      const double dm = __shfl_sync(kFull, d, gb + c);
      if (searching && gl == c) scanned = true;
      // the matching does not change during a search, so column c is free
      // exactly when it has no matched row
      const int r0 = __shfl_sync(kFull, c2r, gb + c);
      const bool found = searching && r0 < 0;
      if (found) {
        sink = c;
        dlast = dm;
      }
      const bool relaxing = searching && !found;
      const int r = r0 < 0 ? 0 : r0;
      const double ur = __shfl_sync(kFull, u, gb + r);
      if (relaxing && !scanned) {
        const double nd = dadd(dm, dsub(dsub(cs[RLT2_IDX(r, m) * ld + gl], ur), v));
        if (okey(nd) < dk) {
          d = nd;
          dk = okey(nd);
          pred = r;
        }
      }
      searching = relaxing;
    }
    // every step scanned one column, the last one the sink: the relaxing
    // steps are the scanned columns but one, and the k-th of them relaxed the
    // m - k columns still unscanned
    const int step = __popc(group_bits<G>(__ballot_sync(kFull, act && cv && scanned), gb)) - 1;
    if (act) nrelax += step * m - (step * (step + 1)) / 2;
    if (act && cv && scanned) v = dadd(v, dsub(d, dlast));
    // augment back to row i (groups walk their own chains in lockstep)
    bool walking = act;
    int col = sink;
    while (G == 32 ? walking : __any_sync(kFull, walking)) {
      const int r = __shfl_sync(kFull, pred, gb + col);
      const int nxt = __shfl_sync(kFull, r2c, gb + r);
      if (walking) {
        if (gl == col) c2r = r;
        if (gl == r) r2c = col;
        if (r == i) walking = false;
        else col = nxt;
      }
    }
    const int mc = (cv && r2c >= 0) ? r2c : 0;
    const double vm = __shfl_sync(kFull, v, gb + mc);
    if (act && cv && r2c >= 0) u = dsub(cs[gl * ld + RLT2_IDX(r2c, m)], vm);
  }

  // optimum: pairwise tree over P = next power of two >= m rows (empty rows add
  // nothing), lane i adding lane i + h for h = P/2, ..., 1
  const double xr = cv ? cs[gl * ld + RLT2_IDX(r2c, m)] : 0.0;
  int P = 1;
  while (P < m) P <<= 1;
  const int PM = (G == 32) ? P : (int)__reduce_max_sync(kFull, (unsigned)P);
  double val = xr;
  for (int h = PM >> 1; h >= 1; h >>= 1) {
    const double o = __shfl_xor_sync(kFull, val, h);
    if (h < P) val = dadd(val, o);
  }
  val = __shfl_sync(kFull, val, gb);

  if (dual_mode != 0) {
    // canonical duals: shortest paths from row 0 on reduced weights
    // pi(r, sigma(r')) = (c_{r,sigma(r')} - u_r) - v_{sigma(r')} >= 0
    const int s0 = __shfl_sync(kFull, r2c, gb);
    if constexpr (PRE) {
      // an FP64 instruction costs the same with few lanes active, so the group's
      // lanes take the m*m entries in row-major turns (every lane busy); (r, c)
      // of entry gl + k*G advance without a division per entry
      uvs[gl] = u;
      uvs[32 + gl] = v;
      __syncwarp();
      if (m > 0) {
        const int qg = G / m, rg = G - qg * m;
        int r = gl / m, c = gl - r * m;
        for (; r < m; r += qg) {
          cs[r * ld + c] = dsub(dsub(cs[r * ld + c], uvs[r]), uvs[32 + c]);
          c += rg;
          if (c >= m) {
            c -= m;
            ++r;
          }
        }
      }
      __syncwarp();
    }
    const double vs0 = __shfl_sync(kFull, v, gb + (s0 < 0 ? 0 : s0));
    double dist = 0.0;
    if (cv && gl != 0) {
      if constexpr (PRE) dist = cs[gl * ld + RLT2_IDX(s0, m)];
      else dist = dsub(dsub(cs[gl * ld + RLT2_IDX(s0, m)], u), vs0);
    }
    bool done = !cv || gl == 0;
    unsigned long long dk = okey(dist);  // cached key of dist
    for (int it = 0; it < M - 2; ++it) {
      const bool stepping = it < m - 2;
      const int rs = group_argmin<G>(done ? ~0ull : dk, gb);
      const double dr = __shfl_sync(kFull, dist, gb + rs);
      if (stepping && gl == rs) done = true;
      const int s = __shfl_sync(kFull, r2c, gb + rs);
      double vs = 0.0;
      if constexpr (!PRE) vs = __shfl_sync(kFull, v, gb + (s < 0 ? 0 : s));
      if (stepping && !done) {
        double w;
        if constexpr (PRE) w = cs[gl * ld + RLT2_IDX(s, m)];
        else w = dsub(dsub(cs[gl * ld + RLT2_IDX(s, m)], u), vs);
        const double nd = dadd(dr, w);
        if (okey(nd) < dk) {
          dist = nd;
          dk = okey(nd);
        }
      }
    }
    const double u0r = __shfl_sync(kFull, u, gb);
    const double ucan = cv ? (m > 1 ? dadd(dist, dsub(u, u0r)) : 0.0) : 0.0;
    // v_c = c_{sigma^-1(c), c} - u_{sigma^-1(c)}, from the matched row's own entry
    const double wrow = dsub(xr, ucan);
    const int rr = cv ? c2r : 0;
    const double vcan = __shfl_sync(kFull, wrow, gb + rr);
    u = ucan;
    v = cv ? vcan : 0.0;
  }
  R.u = u;
  R.v = v;
  R.r2c = r2c;
  R.c2r = c2r;
  R.value = val;
  R.naug = naug;
  R.nrelax = nrelax;
  return R;
}

// ---- exact form --------------------------------------------------------------
// Group lane of the least (kh, lo) pair, lowest lane on ties; a lane out of the
// race holds kh = ~0 (labels and distances are in [0, 2^58), so the high word of
// one in the race is smaller).  The low words are compared only where several
// lanes of a group share the least high word.  Every lane of the warp calls it.
template <int G>
__device__ __forceinline__ int fx_argmin(unsigned kh, unsigned lo, int gb) {
  if constexpr (G == 32) {
    const unsigned mh = __reduce_min_sync(kFull, kh);
    unsigned ball = __ballot_sync(kFull, kh == mh);
    if (ball & (ball - 1u)) {
      const unsigned ml = __reduce_min_sync(kFull, kh == mh ? lo : 0xffffffffu);
      ball = __ballot_sync(kFull, kh == mh && lo == ml);
    }
    return __ffs(ball) - 1;
  } else {
    constexpr unsigned mask = (1u << G) - 1u;
    auto group_min = [&](unsigned x) {
      if constexpr (G == 16) {
        // two full-warp reductions, each with the other half at the maximum (no
        // divergence, unlike a redux.sync on a half-warp mask)
        const unsigned a = __reduce_min_sync(kFull, gb ? 0xffffffffu : x);
        const unsigned b = __reduce_min_sync(kFull, gb ? x : 0xffffffffu);
        return gb ? b : a;
      } else {
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) x = min(x, __shfl_xor_sync(kFull, x, off));
        return x;
      }
    };
    const unsigned mh = group_min(kh);
    unsigned mine = (__ballot_sync(kFull, kh == mh) >> gb) & mask;
    if (__any_sync(kFull, (mine & (mine - 1u)) != 0u)) {
      const unsigned ml = group_min(kh == mh ? lo : 0xffffffffu);
      mine = (__ballot_sync(kFull, kh == mh && lo == ml) >> gb) & mask;
    }
    return __ffs(mine) - 1;
  }
}

// fx_floor_entry from the entry's words, kk = (L + 1075) << 20: sign, hidden bit
// (0 for exponent field 0) and shift without a branch.
__device__ __forceinline__ long long fx_floor_words(unsigned hi, unsigned lo, unsigned kk) {
  const unsigned ex = hi & 0x7ff00000u;
  const unsigned long long mant = ((unsigned long long)((hi & 0xfffffu) | min(ex, 0x100000u)) << 32) | lo;
  const long long neg = (long long)((int)hi >> 31);
  long long q;
  // 64-bit shifts by 64 and more leave the sign
  asm("shr.s64 %0, %1, %2;" : "=l"(q) : "l"(((long long)mant ^ neg) - neg), "r"((kk - max(ex, 0x100000u)) >> 20));
  return q;
}

// One LAP per group of G lanes in exact fixed point with canonical duals: the
// algorithm, tie rules and hence the results (assignment and counters too) are
// those of group_lap; exact sums may be taken in any order, so a step costs
// fewer instructions:
//   - column lane c keeps um = u of its matched row, and row duals exist in
//     shared memory only for free rows (uvs, the start duals): a step's
//     broadcast is d_c - um_c in one shuffle pair, its relaxation
//     (c_rc - v_c) + that, and the dual update touches the column lane alone
//     (a matched edge stays tight, so u falls by what v rises);
//   - the predecessor of a column is the column scanned before it, so the
//     augmenting path is a mask of columns and all its columns take their
//     new rows at once;
//   - lanes out of the race are marked in the word that the argmin compares;
//   - at one LAP per warp every loop condition is warp-uniform and needs no vote.
// raw (nullable): the tile as doubles with row stride rs, in shared memory and
// possibly the tile itself; the column reduction converts it into cs and then
// calls hook().  kk = (L + 1075) << 20 for the tile's grid 2^L.
// Bound by the ALU pipe (77 % busy) and issue (80 %).  Z stage, warm: n = 20 394
// -> 356 us (3,160 -> 2,700 warp instructions per LAP: 580 the column
// reduction, 900 the searches, 620 the canonical pass), n = 17 160 -> 139,
// n = 12 41.5 -> 34.
template <int G, bool RR = false, typename Hook = NoHook>
__device__ __forceinline__ WarpLapResult<long long> group_lap_fx(long long* cs, int ld, int m, int lane, bool warm,
                                                                 long long u0, int* scr, long long* uvs,
                                                                 const double* raw = nullptr, int rs = 0, int L = 0,
                                                                 const Hook& hook = Hook()) {
  using T = long long;
  constexpr unsigned kOut = 0xffffffffu;
  constexpr T kTop = 0x7fffffffffffffffll;
  const int gl = lane & (G - 1), gb = lane - gl;
  const bool cv = gl < m;
  const int gc = cv ? gl : 0;  // a lane past the LAP reads column 0
  const int M = (G == 32) ? m : (int)__reduce_max_sync(kFull, (unsigned)m);
  auto hi32 = [](T x) { return (unsigned)((unsigned long long)x >> 32); };
  const unsigned kk = (unsigned)(L + 1075) << 20;
  auto entry = [&](int r) {  // column gl's entry of row r, onto the grid
    const uint2 w = *reinterpret_cast<const uint2*>(raw + r * rs + gl);
    const T c = fx_floor_words(w.y, w.x, kk);
    cs[r * ld + gl] = c;
    return c;
  };
  T u = (cv && warm) ? u0 : T(0);
  if constexpr (RR) {
    if (!__any_sync(kFull, warm)) {  // warp-uniform: the launches with RR start every LAP cold
      if (raw) {
        if (cv)
          for (int r = 0; r < m; ++r) entry(r);
        __syncwarp();
        hook();
        raw = nullptr;
      }
      T mn = kTop;
      if (cv)
        for (int c = 0; c < m; ++c) {  // lane = row (odd row stride: no bank conflicts)
          const T x = cs[gl * ld + c];
          mn = x < mn ? x : mn;
        }
      u = cv ? mn : T(0);
    }
  }
  uvs[gl] = u;
  __syncwarp();
  // column reduction with the argmin row
  T v = kTop;
  int arg = 0;
  if (cv) {
    auto reduce = [&](int r, T c) {
      const T x = c - uvs[r];
      if (x < v) {
        v = x;
        arg = r;
      }
    };
    if (raw) {
#pragma unroll 3
      for (int r = 0; r < m; ++r) reduce(r, entry(r));
    } else {
#pragma unroll 3
      for (int r = 0; r < m; ++r) reduce(r, cs[r * ld + gl]);
    }
  } else {
    v = T(0);
  }
  if (raw) {
    __syncwarp();  // every lane's reads of raw are done
    hook();
  }
  // greedy: the lowest column among those sharing an argmin row takes it
  const unsigned same = __match_any_sync(kFull, cv ? (gb << 6) + arg : (1 << 20) + lane);
  const bool win = cv && (__ffs(same) - 1) == lane;
  int c2r = win ? arg : -1;
  T um = uvs[arg];  // used where the column is matched
  unsigned taken = __reduce_or_sync(kFull, win ? 1u << (gb + arg) : 0u);
  unsigned freerows = (m > 0 ? kFull >> (32 - m) : 0u) & ~(taken >> gb);
  int naug = 0, nrelax = 0;
  while (G == 32 ? freerows != 0 : __any_sync(kFull, freerows != 0)) {
    const bool act = freerows != 0;  // this group runs a search in this pass
    const int i = act ? __ffs(freerows) - 1 : 0;
    if (act) {
      freerows &= freerows - 1;
      ++naug;
      nrelax += m;
    }
    T d = (cs[i * ld + gc] - uvs[i]) - v;
    unsigned kh = (act && cv) ? hi32(d) : kOut;
    int from = -1;  // the column scanned before this one on its path (-1: reached from row i)
    int sink = 0;
    bool searching = act;
    // the free columns as a mask: at one LAP per warp the test is then on
    // uniform values
    const unsigned freecols = __ballot_sync(kFull, cv && c2r < 0) >> gb;
    while (G == 32 ? true : __any_sync(kFull, searching)) {
      const int c = fx_argmin<G>(kh, (unsigned)d, gb);
      if (G == 32 || searching) {
        if ((freecols >> c) & 1u) {
          sink = c;
          if constexpr (G == 32) break;
          searching = false;
        }
      }
      const int r0 = __shfl_sync(kFull, c2r, gb + c);
      const T es = __shfl_sync(kFull, d - um, gb + c);
      if (G == 32 || searching) {
        if (gl == c) kh = kOut;
        const T nd = (cs[RLT2_IDX(r0, m) * ld + gc] - v) + es;
        if (kh != kOut && nd < d) {
          d = nd;
          kh = hi32(nd);
          from = c;
        }
      }
    }
    if constexpr (G == 32) {
      if (__ballot_sync(kFull, cv && kh == kOut) == 0) {  // the nearest column was free: no dual changes
        if (gl == sink) {
          c2r = i;
          um = cs[i * ld + gl] - v;
        }
        continue;
      }
    }
    // the k-th scanned column relaxed the m - k columns still unscanned
    const bool scanned = act && cv && kh == kOut;
    const int step = __popc(group_bits<G>(__ballot_sync(kFull, scanned), gb));
    if (act) nrelax += step * m - (step * (step + 1)) / 2;
    const T dlast = __shfl_sync(kFull, d, gb + sink);
    if (scanned) {
      const T delta = d - dlast;
      v += delta;
      um -= delta;
    }
    // the path's columns, then their new rows at once
    const int row = __shfl_sync(kFull, c2r, gb + (from < 0 ? 0 : from));
    unsigned path = 0;
    int col = sink;
    bool walking = act;
    while (G == 32 ? true : __any_sync(kFull, walking)) {
      if (walking) path |= 1u << col;
      if constexpr (G == 32) {
        const int p = (int)__reduce_max_sync(kFull, lane == col ? (unsigned)(from + 1) : 0u);
        if (p == 0) break;
        col = p - 1;
      } else {
        const int p = __shfl_sync(kFull, from, gb + col);
        walking = walking && p >= 0;
        if (walking) col = p;
      }
    }
    if ((path >> gl) & 1u) {
      c2r = from < 0 ? i : row;
      um = cs[RLT2_IDX(c2r, m) * ld + gc] - v;
    }
  }
  // to row lanes: the matched column and the row dual
  __syncwarp();
  if (cv) {
    scr[c2r] = gl;
    uvs[c2r] = um;
  }
  __syncwarp();
  const int r2c = cv ? scr[gl] : 0;
  u = cv ? uvs[gl] : T(0);
  const T vown = __shfl_sync(kFull, v, gb + r2c);  // dual of the matched column
  const T xr = cv ? u + vown : T(0);               // the assigned entry
  T val;
  if constexpr (G == 32) {
    // the 64-bit entries as two non-negative 26-bit limbs and a signed top
    // part, each summed over the warp by one 32-bit reduction (no overflow)
    const unsigned long long ux = (unsigned long long)xr;
    const long long s0 = __reduce_add_sync(kFull, (int)(ux & 0x3ffffffull));
    const long long s1 = __reduce_add_sync(kFull, (int)((ux >> 26) & 0x3ffffffull));
    const long long s2 = __reduce_add_sync(kFull, (int)(xr >> 52));
    val = s2 * (1ll << 52) + s1 * (1ll << 26) + s0;
  } else {
    val = xr;
#pragma unroll
    for (int h = G / 2; h >= 1; h >>= 1) val += __shfl_xor_sync(kFull, val, h);
  }
  // canonical duals: Dijkstra from row 0 over arcs r' -> r of weight
  // (c_{r,sigma(r')} - u_r) - v_{sigma(r')}; row lanes broadcast dist - v_own
  T dist = 1ll << 61;  // above every distance
  unsigned kh = cv ? hi32(dist) : kOut;
  if (gl == 0) {
    dist = T(0);
    kh = kOut;
  }
  int rs0 = 0;
  for (int it = 0; it < M - 1; ++it) {
    if (it) rs0 = fx_argmin<G>(kh, (unsigned)dist, gb);
    const T es = __shfl_sync(kFull, dist - vown, gb + rs0);
    const int s = __shfl_sync(kFull, r2c, gb + rs0);
    if (G == 32 || it < m - 1) {
      if (gl == rs0) kh = kOut;
      const T nd = (cs[gc * ld + RLT2_IDX(s, m > 0 ? m : 1)] - u) + es;
      if (kh != kOut && nd < dist) {
        dist = nd;
        kh = hi32(nd);
      }
    }
  }
  const T u0r = __shfl_sync(kFull, u, gb);
  const T ucan = cv ? dist + (u - u0r) : T(0);
  const T vcan = __shfl_sync(kFull, xr - ucan, gb + (cv ? c2r : 0));
  __syncwarp();  // the reads of uvs and scr are done before a caller reuses them
  WarpLapResult<T> R;
  R.u = ucan;
  R.v = cv ? vcan : T(0);
  R.r2c = r2c;
  R.c2r = c2r;
  R.value = val;
  R.naug = naug;
  R.nrelax = nrelax;
  return R;
}

// ---- all-zero tiles ------------------------------------------------------------
// The first solve of every ascent has D^ = 0 (Algorithm 1, step 1): each tile is
// zero, every argmin a tie, and the searches walk through all matched columns
// (n = 30: 15.3 ms for that Z stage against 3.3 for a later one).  From a cold
// start the outcome is known: column 0 takes row 0; the search of row i scans
// columns 0 .. i-1 in lane order and takes column i; all duals stay 0.
template <int G>
__device__ __forceinline__ bool group_all_zero(const double* p, int count, int gl, unsigned ignore_sign) {
  unsigned nz = 0;
  for (int e = gl; e < count; e += G) {
    const unsigned* w = reinterpret_cast<const unsigned*>(p + e);
    nz |= w[0] | (w[1] << ignore_sign);
  }
  if constexpr (G == 32) {
    nz = __reduce_or_sync(kFull, nz);
  } else {
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) nz |= __shfl_xor_sync(kFull, nz, off);
  }
  return nz == 0;
}
template <typename T>
__device__ __forceinline__ void zero_tile_result(WarpLapResult<T>& R, int gl, int m) {
  R.u = R.v = R.value = T(0);
  R.r2c = R.c2r = gl;
  R.naug = m - 1;
  R.nrelax = m * (m - 1) + m * m * (m - 1) / 2 - (m - 1) * m * (m + 1) / 6;  // sum over i of m + i m - i (i+1) / 2
}

// ---- launch helpers shared by the LAP kernels ------------------------------
constexpr int kMaxWarpsPerBlock = 8;

__host__ __device__ inline int tile_ld(int m) { return m | 1; }  // odd stride: conflict-free rows and columns

// Shared memory per warp: 32/G tiles, u/v staging (64 doubles) and 32 ints.
__host__ __device__ inline size_t warp_smem_bytes(int m, int G) {
  return (size_t)(32 / G) * m * tile_ld(m) * sizeof(double) + 64 * sizeof(double) + 32 * sizeof(int);
}
// The prefetching form adds, per group, the next tile (m*m doubles, as stored)
// and its start duals (m doubles), rounded to 16 bytes.
__host__ __device__ inline size_t raw_group_doubles(int m) { return ((size_t)m * m + m + 1) & ~size_t(1); }
__host__ __device__ inline size_t warp_smem_bytes_async(int m, int G) {
  return warp_smem_bytes(m, G) + (size_t)(32 / G) * raw_group_doubles(m) * sizeof(double);
}

// The one-tile form (G = 32): the tile, 32 dual slots and 32 ints.
__host__ __device__ inline size_t warp_smem_bytes_one(int m) {
  return (size_t)m * tile_ld(m) * sizeof(double) + 32 * sizeof(double) + 32 * sizeof(int);
}

// The lane's entries e = gl, gl + G, ... < mm of src (+ add, rounded), each
// passed to f(e, x).  CG: load through L2 only (the tile was written by other SMs
// during the same launch, so a line in this SM's L1 may be stale).
template <int G, bool CG, typename F>
__device__ __forceinline__ void for_tile_entries(int mm, int gl, const double* src, const double* add, F&& f) {
  for (int e = gl; e < mm; e += G) {
    const double x = CG ? __ldcg(src + e) : __ldcs(src + e);
    if (add) f(e, __dadd_rn(x, CG ? __ldcg(add + e) : __ldcs(add + e)));
    else f(e, x);
  }
}

// Stages one group's tile (plus an optional addend) into shared memory, the
// group's G lanes reading a contiguous m*m run (coalesced).  FX: the tile is
// rounded down onto the group's fixed-point grid and the grid exponent L is
// returned (0 for FP64).  All 32 lanes call it; src == nullptr for a group
// without a LAP.
template <int G, bool FX, bool CG = false>
__device__ __forceinline__ int stage_tile(typename std::conditional<FX, long long, double>::type* tile, int ld,
                                          int m, int gl, const double* src, const double* add) {
  const int mm = m * m;
  if constexpr (!FX) {
    if (src)
      for_tile_entries<G, CG>(mm, gl, src, add, [&](int e, double x) {
        const int r = e / m, c = e - r * m;
        tile[r * ld + c] = x;
      });
    return 0;
  } else {
    unsigned eb = 0;
    if (src)
      for_tile_entries<G, CG>(mm, gl, src, add, [&](int e, double x) {
        const int r = e / m, c = e - r * m;
        tile[r * ld + c] = __double_as_longlong(x);  // bits; converted below once the grid is known
        eb = max(eb, fx_expfield(x));
      });
    if constexpr (G == 32) {
      eb = __reduce_max_sync(kFull, eb);
    } else {
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) eb = max(eb, __shfl_xor_sync(kFull, eb, off));
    }
    const int L = fx_grid(eb);
    if (src) {
      for (int e = gl; e < mm; e += G) {  // the entries this lane wrote
        const int r = e / m, c = e - r * m;
        tile[r * ld + c] = fx_floor(__longlong_as_double(tile[r * ld + c]), L, kFxEntryBits);
      }
    }
    return L;
  }
}

// Reduced costs: rounded in FP64, exact on the grid.
__device__ __forceinline__ double lap_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ long long lap_sub(long long a, long long b) { return a - b; }

template <bool FX, typename T>
__device__ __forceinline__ double out_value(T x, int L) {
  if constexpr (FX) return fx_to_double(x, L);
  else return x;
}

template <bool FX>
__device__ __forceinline__ typename std::conditional<FX, long long, double>::type start_dual(double u0, int L) {
  if constexpr (FX) return fx_floor(u0, L, kFxStartBits);
  else return u0;
}

}  // namespace rlt2
