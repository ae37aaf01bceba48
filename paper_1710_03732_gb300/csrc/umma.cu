// Learned-start inference on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// The warm-start network's two hidden layers for 128-row tiles in one
// persistent CTA of eight warps: the weights of both layers stay in shared
// memory for the whole launch (W1: 48 x 256, W2: 256 x 256, BF16), each
// 128 x 48 input tile is fetched into registers ahead of its turn (zeros past
// the last row), and one thread issues tcgen05.mma (kind::f16, BF16 x BF16 ->
// FP32, M = 128, N = 256) into 256 TMEM columns per layer, committed to an
// mbarrier.  The first MMA's epilogue reads the accumulator with tcgen05.ld
// (warp w owns TMEM lanes 32 (w mod 4) .. +31, the tile's rows, and half of the
// columns in turn) and writes relu(acc + b1) as BF16 straight into shared
// memory in the operand layout of the second MMA (over the input tile, which
// the first MMA has consumed); the second MMA's epilogue folds the output
// layer in, out = sum_c bf16(relu(acc_c + b2_c)) w3_c + b3 (the two column
// halves added through shared memory).  The hidden activations never leave
// the SM.
//
// Operand layout in shared memory: K-major, no swizzle, 8 x 16-byte core
// matrices; core matrix (r8, k8) of an R-row operand sits at byte
// (k8 * R/8 + r8) * 128, so the descriptor's stride between row groups (SBO)
// is 128 B and between K groups (LBO) is 16 R bytes.  Every wait on the
// mbarrier is bounded; a timeout sets *err and the CTA stops, releasing its
// TMEM.
#include <cuda_bf16.h>

#include <cstdint>
#include <mutex>

#include "rlt2_internal.h"

namespace rlt2 {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kN = 256;          // layer width (TMEM columns)
constexpr int kRowsPerTile = 128;  // M of the MMA = TMEM lanes
constexpr int kThreads = 256;
constexpr long long kWaitLimit = 1ll << 22;  // non-blocking mbarrier polls before giving up (~0.1 s)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// tcgen05 shared-memory matrix descriptor: start >> 4 (bits 0-13), LBO >> 4
// (16-29), SBO >> 4 (32-45), descriptor version 1 (46-47), no swizzle (61-63 = 0).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// (7-9 = 1) and B (10-12 = 1), both K-major (15, 16 = 0), N >> 3 (17-22),
// M >> 4 (24-28).
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) |
                            ((uint32_t)(kRowsPerTile >> 4) << 24);

__device__ __forceinline__ uint32_t core_off(int r, int k8, int R) {
  return (uint32_t)((k8 * (R / 8) + (r >> 3)) * 128 + (r & 7) * 16);
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t phase) {
  for (long long it = 0; it < kWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

struct UmmaMlpArgs {
  long long rows;
  const bf16* X;  // [rows][64]
  const bf16* W1;  // [64][256]
  const float* b1;
  const bf16* W2;  // [256][256]
  const float* b2;
  const float* w3;
  const float* b3;
  float* out;
  int* err;
  int withhold_commit;  // diagnostics: issue no MMA and no commit, so the first wait runs out
};

// W (row-major [rows][256], rows >= K) into the K-major operand layout: a thread
// turns 8 x 8 blocks in registers, so that both sides move 16 bytes at a time.
__device__ __forceinline__ void load_weights(unsigned char* Bs, const bf16* W, int K, int tid) {
  for (int e = tid; e < K * kN / 64; e += kThreads) {
    const int n8 = e % (kN / 8), k8 = e / (kN / 8);
    uint4 in[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) in[k] = *reinterpret_cast<const uint4*>(W + (size_t)(k8 * 8 + k) * kN + n8 * 8);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t w[4];
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) {
        const uint32_t lo = reinterpret_cast<const uint32_t*>(&in[2 * k2])[q >> 1];
        const uint32_t hi = reinterpret_cast<const uint32_t*>(&in[2 * k2 + 1])[q >> 1];
        w[k2] = __byte_perm(lo, hi, (q & 1) ? 0x7632 : 0x5410);
      }
      *reinterpret_cast<uint4*>(Bs + core_off(n8 * 8 + q, k8, kN)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// K steps of 16 [k0, k1) of a tile's product; step 0 overwrites the accumulator.
__device__ __forceinline__ void issue_mma(uint32_t tmem, uint32_t a_base, uint32_t b_base, int k0, int k1) {
#pragma unroll 1
  for (int kk = k0; kk < k1; ++kk) {
    const uint64_t ad = sdesc(a_base + kk * 2 * (16 * kRowsPerTile), 16 * kRowsPerTile, 128);
    const uint64_t bd = sdesc(b_base + kk * 2 * (16 * kN), 16 * kN, 128);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(kIdesc), "r"(kk)
        : "memory");
  }
}
__device__ __forceinline__ void commit_mma(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Two FP32 values through the BF16 rounding and max(x, 0), first one in the low
// half (a NaN becomes 0, as with fmaxf).
__device__ __forceinline__ uint32_t relu_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("{\n\tcvt.rn.bf16x2.f32 %0, %1, %2;\n\tmax.bf16x2 %0, %0, %3;\n\t}" : "=r"(r) : "f"(hi), "f"(lo), "r"(0));
  return r;
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// K of the first MMA: the 34 features in whole steps of 16 (the rest of a row
// is zero padding).
constexpr int kIn = 48;

// What bounds a tile is the chain MMA 1 -> epilogue 1 -> MMA 2 -> epilogue 2, so
// what can leave the chain does:
//   - the biases and the output weights sit in shared memory (as scalar global
//     loads per column they were most of the two epilogues);
//   - the next tile's input rows are fetched into registers during MMA 2, and
//     its MMA 1 (own accumulator) runs under this tile's epilogue 2;
//   - epilogue 1 goes through the columns in two halves of 128, MMA 2's first
//     eight K steps running under the second half.
// 262,144 rows: 138 -> 64 us (bit-identical); the whole of 144,400 tiles of size
// 18 with the features and starts 2.22 -> 1.41 ms.
__global__ void __launch_bounds__(kThreads, 1) k_umma_mlp(UmmaMlpArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* B1 = smem;                        // 256 x 48
  unsigned char* B2 = B1 + (size_t)kN * kIn * 2;   // 256 x 256
  unsigned char* Act = B2 + (size_t)kN * kN * 2;   // input tile (128 x 48), then hidden tile (128 x 256)
  float* vec = reinterpret_cast<float*>(Act + (size_t)kRowsPerTile * kN * 2);  // b1 | b2 | w3
  float* half = vec + 3 * kN;
  uint64_t* bar = reinterpret_cast<uint64_t*>(half + kRowsPerTile);
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar_a = smem_u32(bar);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(2 * kN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
  load_weights(B1, a.W1, kIn, tid);
  load_weights(B2, a.W2, kN, tid);
  for (int c = tid; c < kN; c += kThreads) {
    vec[c] = a.b1[c];
    vec[kN + c] = a.b2[c];
    vec[2 * kN + c] = a.w3[c];
  }
  const float b3 = *a.b3;
  const uint32_t act = smem_u32(Act), b1a = smem_u32(B1), b2a = smem_u32(B2);
  const int quarter = warp & 3, colh = warp >> 2;
  const int trow = quarter * 32 + lane;
  const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
  const long long ntiles = (a.rows + kRowsPerTile - 1) / kRowsPerTile;
  // the input tile in 16-byte pieces: row tid >> 1 of the tile, pieces
  // 3 (tid & 1) .. + 2 of its six
  const int xr = tid >> 1, xk = 3 * (tid & 1);
  uint4 x[3];
  auto fetch = [&](long long tile) {
    const long long r = tile * kRowsPerTile + xr;
    const bool in = r < a.rows;
    const uint4* src = reinterpret_cast<const uint4*>(a.X + (in ? r : 0) * 64) + xk;
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = in ? __ldg(src + k) : make_uint4(0, 0, 0, 0);
  };
  auto put = [&]() {
#pragma unroll
    for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(Act + core_off(xr, xk + k, kRowsPerTile)) = x[k];
  };
  // what the threads wrote into shared memory is visible to the MMAs that follow
  auto publish = [&]() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  uint32_t phase = 0;
  bool ok = true;
  // the MMAs committed last are done (every thread; false on a timeout)
  auto done = [&]() {
    const bool arrived = mbar_wait(bar_a, phase);
    if (__syncthreads_or(arrived ? 0 : 1)) {
      if (tid == 0) atomicExch(a.err, 1);
      return false;
    }
    phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return true;
  };
  fetch(blockIdx.x);  // the grid has no more blocks than tiles
  put();
  publish();
  const uint32_t acc1 = *slot, acc2 = acc1 + kN;
  if (tid == 0 && !a.withhold_commit) {
    issue_mma(acc1, act, b1a, 0, kIn / 16);
    commit_mma(bar_a);
  }
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long row = tile * kRowsPerTile + trow;
    const bool more = tile + gridDim.x < ntiles;
    if (!(ok = done())) break;  // MMA 1
    // hidden layer 1 -> BF16 operand of the second MMA, in shared memory (over
    // the input tile, which the first MMA has consumed)
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
#pragma unroll 1
      for (int c0 = 128 * h + 64 * colh; c0 < 128 * h + 64 * colh + 64; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(acc1 + lane_off + (uint32_t)c0, v);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const float4 ba = *reinterpret_cast<const float4*>(vec + c0 + 8 * g);
          const float4 bb = *reinterpret_cast<const float4*>(vec + c0 + 8 * g + 4);
          const uint32_t* w = v + 8 * g;
          uint4 p;
          p.x = relu_bf16x2(__uint_as_float(w[0]) + ba.x, __uint_as_float(w[1]) + ba.y);
          p.y = relu_bf16x2(__uint_as_float(w[2]) + ba.z, __uint_as_float(w[3]) + ba.w);
          p.z = relu_bf16x2(__uint_as_float(w[4]) + bb.x, __uint_as_float(w[5]) + bb.y);
          p.w = relu_bf16x2(__uint_as_float(w[6]) + bb.z, __uint_as_float(w[7]) + bb.w);
          *reinterpret_cast<uint4*>(Act + core_off(trow, (c0 >> 3) + g, kRowsPerTile)) = p;
        }
      }
      publish();
      if (tid == 0) {
        issue_mma(acc2, act, b2a, 8 * h, 8 * h + 8);
        if (h == 1) commit_mma(bar_a);
      }
    }
    if (more) fetch(tile + gridDim.x);
    if (!(ok = done())) break;  // MMA 2
    if (more) {
      put();
      publish();
      if (tid == 0) {
        issue_mma(acc1, act, b1a, 0, kIn / 16);
        commit_mma(bar_a);
      }
    }
    // hidden layer 2 and the output layer, columns in order within each half
    float acc_out = 0.0f;
#pragma unroll 1
    for (int c0 = colh * (kN / 2); c0 < (colh + 1) * (kN / 2); c0 += 32) {
      uint32_t v[32];
      tmem_ld32(acc2 + lane_off + (uint32_t)c0, v);
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        const float4 b = *reinterpret_cast<const float4*>(vec + kN + c0 + 4 * g);
        const float4 w = *reinterpret_cast<const float4*>(vec + 2 * kN + c0 + 4 * g);
        const uint32_t p0 = relu_bf16x2(__uint_as_float(v[4 * g]) + b.x, __uint_as_float(v[4 * g + 1]) + b.y);
        const uint32_t p1 = relu_bf16x2(__uint_as_float(v[4 * g + 2]) + b.z, __uint_as_float(v[4 * g + 3]) + b.w);
        acc_out = fmaf(__uint_as_float(p0 << 16), w.x, acc_out);
        acc_out = fmaf(__uint_as_float(p0 & 0xffff0000u), w.y, acc_out);
        acc_out = fmaf(__uint_as_float(p1 << 16), w.z, acc_out);
        acc_out = fmaf(__uint_as_float(p1 & 0xffff0000u), w.w, acc_out);
      }
    }
    if (colh == 1) half[trow] = acc_out;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (colh == 0 && row < a.rows) a.out[row] = (acc_out + half[trow]) + b3;
    // the next write of `half`, and of the second accumulator, comes after the
    // next tile's synchronisations
  }
  if (!ok && !a.withhold_commit) mbar_wait(bar_a, phase);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(acc1), "r"(2 * kN) : "memory");
}

constexpr size_t kMlpSmem = (size_t)kN * kIn * 2 + (size_t)kN * kN * 2 + (size_t)kRowsPerTile * kN * 2 + 3 * kN * 4 +
                            kRowsPerTile * 4 + 64;

}  // namespace

// out[r] = w3 . relu(W2^T relu(W1^T x_r + b1) + b2) + b3 for `rows` feature rows
// (X: [rows][64] BF16); err: device flag set on a timed-out wait.
cudaError_t umma_mlp_forward(const bf16* X, long long rows, const bf16* W1, const float* b1, const bf16* W2,
                             const float* b2, const float* w3, const float* b3, float* out, int* err,
                             cudaStream_t s, bool withhold_commit) {
  if (rows <= 0) return cudaSuccess;
  // launch configuration, once per device, from any host thread (not valid
  // across a cudaDeviceReset, like every per-device cache of the library)
  static std::mutex mu;
  constexpr int kDevs = 64;
  static int sms_of[kDevs];
  static bool attr_of[kDevs];
  cudaError_t e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= kDevs) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!sms_of[dev] &&
        (e = cudaDeviceGetAttribute(&sms_of[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
    if (!attr_of[dev]) {
      if ((e = cudaFuncSetAttribute(k_umma_mlp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem)) !=
          cudaSuccess)
        return e;
      attr_of[dev] = true;
    }
    sms = sms_of[dev];
  }
  const long long tiles = (rows + kRowsPerTile - 1) / kRowsPerTile;
  const int grid = (int)(tiles < sms ? tiles : sms);
  UmmaMlpArgs a{rows, X, W1, b1, W2, b2, w3, b3, out, err, withhold_commit ? 1 : 0};
  k_umma_mlp<<<grid, kThreads, kMlpSmem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace rlt2
