// The surrogate's forward and backward passes on packed activations (sm_103a): every layer's
// output is stored once, as the bfloat16 values the next product rounds its operand to, in the
// core-matrix layout that tcgen05 reads, so staging an operand is a few bulk copies and no thread
// converts or rearranges anything between layers. The float32 pre-activations are stored only
// where the backward pass needs them. The forward products, their K order, bias, activation and
// contraction are those of the general tcgen05 kernels (surrogate_kernels.cu), and so are its
// results, bit for bit; gradients differ from theirs in the order of float32 sums.
//
// The same layout is K-major for the forward products and the data gradients (rows = times,
// K = channels) and MN-major for the weight gradients (K = times), where a tap's shift along
// time is a row offset too, so one window serves the three taps there as well.
//
// Packed rows: 16 bytes = 8 consecutive channels (or features) of one row, rows of a channel
// group consecutive. Dense layers: [features/8][batch rows][8]. Convolutions: [sample][C/8]
// [packed_rows(L)][8], row 1 + t holding time t, the rows around the samples zero (the 'same'
// padding and the tail of the last tile), so a window of 130 rows is one copy per group. A
// gradient at an upsampled layer's output keeps its even and odd times apart, [sample][C/8][2]
// [packed_rows(L / 2)][8], so that both products over it see plain rows.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "surrogate_internal.h"
#include "surrogate_tc.cuh"

namespace sgk {
namespace {

constexpr int kRows = 128;              // MMA M: rows (times, or samples) of a tile
constexpr int kWinRows = kRows + 2;     // rows of a convolution's input window
constexpr uint32_t kWinGroup = kWinRows * 16;  // bytes of one channel group of a window
constexpr int kMaxStages = 4;
constexpr int kSmemLimit = 227 * 1024 - 1024;  // a CTA's dynamic part beside its static and reserved bytes

// Core-matrix descriptor (no swizzle, K-major): lbo = bytes to the next 8 K elements, rows 16
// bytes apart, 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t packed_desc(uint32_t addr, uint32_t lbo) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>(128u >> 4) << 32) | (1ull << 46);
}
// kind::f16, float32 D, bfloat16 K-major operands, M = 128
__device__ __forceinline__ uint32_t packed_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(kRows >> 4) << 24);
}
__device__ __forceinline__ void packed_mma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
// 16 columns of the warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  return static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(a))) |
         (static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(b))) << 16);
}
__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}

// ---- weights ------------------------------------------------------------------------------
// Row r of a dense layer's packed weights is feature f(r): r itself, or (z: the layer feeds the
// first convolution) channel 8 (r / 8 / l0) + r % 8 at time (r / 8) % l0, so that eight
// consecutive accumulator columns are the eight channels of one packed row.
__device__ __forceinline__ int dense_feature(int r, int l0) {
  if (l0 == 0) return r;
  const int q = r >> 3, cg = q / l0;
  return (8 * cg + (r & 7)) * l0 + (q - cg * l0);
}
// [N/64][Kp/8][64][8], zero for k >= K
__global__ void pack_dense_kernel(int N, int K, int Kp, int l0, const bf16* __restrict__ W, bf16* __restrict__ Wp) {
  const size_t total = static_cast<size_t>(N) * Kp;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int e = static_cast<int>(i & 7), n = static_cast<int>(i >> 3) & 63;
    const size_t blk = i >> 9;
    const int g = static_cast<int>(blk % (Kp / 8)), tile = static_cast<int>(blk / (Kp / 8));
    const int k = 8 * g + e;
    Wp[i] = k < K ? W[static_cast<size_t>(dense_feature(64 * tile + n, l0)) * K + k] : __float2bfloat16_rn(0.f);
  }
}
// [blocks][3][Ci/8][N][8]; with contract > 0 row n of block nb is output channel (n / 32) outC +
// 32 nb + n % 32 (all contracted copies of 32 channels), else n
__global__ void pack_conv_rows_kernel(int Ci, int N, int blocks, int outC, const bf16* __restrict__ W,
                                      bf16* __restrict__ Wp) {
  const size_t total = static_cast<size_t>(blocks) * 3 * Ci * N;
  const int G = Ci / 8;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int e = static_cast<int>(i & 7);
    size_t r = i >> 3;
    const int n = static_cast<int>(r % N);
    r /= N;
    const int g = static_cast<int>(r % G);
    r /= G;
    const int d = static_cast<int>(r % 3), nb = static_cast<int>(r / 3);
    const int o = outC ? (n >> 5) * outC + 32 * nb + (n & 31) : n;
    Wp[i] = W[(static_cast<size_t>(o) * Ci + 8 * g + e) * 3 + d];
  }
}

// ---- dense layers -------------------------------------------------------------------------
// out = gelu(W in + b) for 128 samples x 64 features per CTA. The whole K of both operands is
// staged at once (64 KB of weights, 128 KB of activations at K = 512, in four parts with a
// barrier each, so the MMAs of a part run under the copies of the next): the layers are bound
// by the latency of reading their weights, not by the products, so all copies fly together
// (256 samples of the default network's three layers: 124 us with tc_gemm_kernel, 22 us here).
struct DenseArgs {
  int B, Bp, K, Kp, N;
  const float* x;     // FROM_X: [B][K]
  const bf16* in;     // else packed [K/8][Bp][8]
  const bf16* W;      // packed
  const float* bias;
  bf16* out;          // packed [N/8][Bp][8], or (TO_Z) [B][c0/8][Lp][8]
  float* pre;         // null, or [B][N]
  float* act;         // null, or gelu(pre) [B][N]
  int l0, Lp;         // TO_Z
  int* err;
  int stall_test;
};

template <bool FROM_X, bool TO_Z>
__global__ void __launch_bounds__(256) dense_kernel(const DenseArgs a) {
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.Kp / 8;
  const uint32_t base = smem_addr(sm);
  const uint32_t sW = base, sA = base + G * 1024u;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + G * 3072);
  const uint32_t bar = smem_addr(bars);  // parts 0 .. 3, 4: products done, 5: never completed
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 6);
  float* sbias = reinterpret_cast<float*>(bars + 7);
  const int n0 = blockIdx.x * 64, m0 = blockIdx.y * kRows;
  const int parts = G % 8 == 0 ? 4 : 1, gp = G / parts;
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) bar_init(bar + 8 * i, 1);
    bar_init(bar + 32, 1);
    bar_init(bar + 40, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(smem_addr(slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid < 64) sbias[tid] = a.bias[dense_feature(n0 + tid, TO_Z ? a.l0 : 0)];
  if constexpr (FROM_X) {
    for (int i = tid; i < kRows * a.Kp; i += 256) {
      const int m = i & (kRows - 1), k = i >> 7;
      const float v = (m0 + m < a.B && k < a.K) ? a.x[static_cast<size_t>(m0 + m) * a.K + k] : 0.f;
      *reinterpret_cast<bf16*>(sm + G * 1024 + (k >> 3) * 2048 + m * 16 + (k & 7) * 2) = __float2bfloat16_rn(v);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool late = false;
  if (a.stall_test) late = !mbar_wait(bar + 40, 0, 20000000ull);
  if (!late && tid == 0) {
    const uint8_t* w = reinterpret_cast<const uint8_t*>(a.W) + static_cast<size_t>(blockIdx.x) * G * 1024;
    for (int p = 0; p < parts; ++p) {
      expect_tx(bar + 8 * p, gp * (FROM_X ? 1024u : 3072u));
      bulk_load(sW + p * gp * 1024u, w + static_cast<size_t>(p) * gp * 1024, gp * 1024u, bar + 8 * p);
      if constexpr (!FROM_X)
        for (int g = p * gp; g < (p + 1) * gp; ++g)
          bulk_load(sA + g * 2048u, a.in + (static_cast<size_t>(g) * a.Bp + m0) * 8, 2048u, bar + 8 * p);
    }
    const uint32_t idesc = packed_idesc(64);
    for (int p = 0; p < parts; ++p) {
      if (!mbar_wait(bar + 8 * p, 0)) late = true;  // (the other parts are still waited for)
      if (late) continue;
      tc_fence_after();
      for (int g = p * gp; g < (p + 1) * gp; g += 2)
        packed_mma(tmem, packed_desc(sA + g * 2048u, 2048u), packed_desc(sW + g * 1024u, 1024u), idesc, g != 0);
    }
    tc_commit(bars + 4);
    if (!mbar_wait(bar + 32, 0)) late = true;
  }
  const bool failed = __syncthreads_or(late) != 0;
  tc_fence_after();
  if (!failed) {
    const int q = warp & 3, h = warp >> 2, b = m0 + q * 32 + lane;
#pragma unroll
    for (int c = 0; c < 32; c += 16) {
      float v[16];
      const int col = 32 * h + c;
      tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + col, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] += sbias[col + i];
      if (b < a.B && a.pre) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          a.pre[static_cast<size_t>(b) * a.N + dense_feature(n0 + col + i, TO_Z ? a.l0 : 0)] = v[i];
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = gelu(v[i]);
      if (b < a.B && a.act) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          a.act[static_cast<size_t>(b) * a.N + dense_feature(n0 + col + i, TO_Z ? a.l0 : 0)] = v[i];
      }
      if (b < a.B) {
#pragma unroll
        for (int i = 0; i < 16; i += 8) {
          const int r = (n0 + col + i) >> 3;
          size_t row = static_cast<size_t>(r) * a.Bp + b;
          if constexpr (TO_Z) {
            const int cg = r / a.l0;
            row = (static_cast<size_t>(b) * (a.N / a.l0 / 8) + cg) * a.Lp + 1 + (r - cg * a.l0);
          }
          reinterpret_cast<uint4*>(a.out)[row] = pack8(v + i);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem) : "memory");
  if (failed && tid == 0) atomicExch(a.err, 1);
}

// ---- convolutions -------------------------------------------------------------------------
// A persistent CTA keeps the weights of its N accumulator columns in shared memory (36 KB a tap
// at 96 x 192) and walks tiles of 128 input times of one sample: warp 0 copies windows (one
// bulk copy per channel group) into a ring, warp 1 issues the MMAs (rows = times, columns =
// output channels), warps 2 .. 9 read the accumulators, two of which alternate in tensor
// memory, so copies, products and epilogues of neighbouring tiles overlap. Taps are row offsets
// of the same window. UP 2: output time 2 s + p reads input rows s + floor((p + d - 1) / 2), so
// the even and the odd output times are two accumulators over one window of the input that
// is not upsampled. K order per accumulator: 32-channel chunk, tap, 16 channels.
// Last convolution: the columns are K contracted copies of 32 output channels; the epilogue forms y = sum_k
// x_k (D_k + bias_k) in registers, so D (K times the output) never reaches memory (the general
// kernel wrote 1.2 GB of it per 256 samples of the default network and a second kernel read it
// back). The default network's forward pass of 4096 samples in chunks of 256, GB300: 16.6 ms
// with the general kernels (tc_conv_kernel 12.2, contraction 4.4, dense 2.0), 3.6 ms now, 880
// TFLOP/s of products; one sample 69 against 27 us, bound by the latency of seven launches.
// Training: the epilogue goes on to the error against the target, its square (SquareSum), dy = 2
// (y - t) / n, and the packed bfloat16 gradient x_k dy of every contracted copy; y and dy
// themselves are not stored (258 us for 256 samples, where the convolution, contraction, loss and
// expansion kernels took 1.7 ms).
struct ConvArgs {
  int B, Ci, Lin, Lpi, N, stages, blocks;
  const bf16* in;   // packed [B][Ci/8][Lpi][8]
  const bf16* W;    // packed rows
  const float* bias;
  bf16* out;        // packed [B][N/8][Lpo][8]
  int Lpo;
  float* pre;       // null, or [B][N][UP Lin]
  const float* x;   // LAST: [B][in_dim], contraction weights from k0 on
  int in_dim, k0, K, outC;
  float* y;         // inference: [B][outC][Lin]
  const float* target;  // training: [B][outC][Lin]
  float scale;      // 2 / outputs
  bf16* dD;         // packed gradient of the K outC channels
  float* row_sums;  // [B][4 tiles][outC] sums of dy over 32 times
  double* loss;     // per CTA, the sum of squared errors
  int* err;
  int stall_test;
};

// Sum of the lanes' v[i], in lanes 2 i and 2 i + 1 (a halving butterfly: 16 exchanges for the
// 16 sums).
__device__ __forceinline__ float warp_sums16(float (&v)[16], int lane) {
#pragma unroll
  for (int n = 8, off = 16; n >= 1; n >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, off);
    }
  }
  return v[0] + __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
}
// index i whose sum warp_sums16 leaves in this lane: its bits, most significant first, are the
// lane's bits 4 .. 1
__device__ __forceinline__ int warp_sums16_index(int lane) { return lane >> 1; }

// A sum of squared errors. A float32 pair takes the squares of 16 errors (each square exact as a
// pair, the sum to about 2^-46) where its range holds them: their sum from 2^-78, below which the
// low halves of the squares that count would underflow, to 2^100, which leaves room for every
// thread's share. Other groups (also all zeros, and NaN) are summed in float64, whose units are too
// few to take every group (with only the sums over the groups in float64 a training step of the
// default network took 1448 us, 1435 like this).
struct SquareSum {
  float hi = 0.f, lo = 0.f;
  double wide = 0.0;
  __device__ __forceinline__ static void two_sum(float& hi, float& lo, float s, float l) {
    const float t = hi + s, z = t - hi;
    lo += ((hi - (t - z)) + (s - z)) + l;
    hi = t;
  }
  __device__ __forceinline__ void add16(const float (&e)[16]) {
    float s = 0.f, l = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float sq = e[i] * e[i];
      two_sum(s, l, sq, fmaf(e[i], e[i], -sq));
    }
    if (s >= 0x1p-78f && s <= 0x1p100f)
      two_sum(hi, lo, s, l);
    else
      for (int i = 0; i < 16; ++i) wide += static_cast<double>(e[i]) * e[i];
  }
  __device__ __forceinline__ double value() const { return wide + (static_cast<double>(hi) + static_cast<double>(lo)); }
};

enum { kHidden = 0, kAnswer = 1, kTrain = 2 };

template <int UP, int KIND>
__global__ void __launch_bounds__(320, 1) packed_conv_kernel(const ConvArgs a) {
  constexpr bool LAST = KIND != kHidden;
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.Ci / 8;
  const uint32_t wbytes = 3u * a.Ci * a.N * 2, sbytes = G * kWinGroup;
  const uint32_t base = smem_addr(sm), sA = base + wbytes;
  float* sbias = reinterpret_cast<float*>(sm + wbytes + a.stages * sbytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sbias + a.N);
  const uint32_t full = smem_addr(bars), empty = full + 8 * kMaxStages, tfull = empty + 8 * kMaxStages,
                 tempty = tfull + 16, wfull = tempty + 16, never = wfull + 8;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 6);
  volatile int* dead = reinterpret_cast<volatile int*>(slot + 1);
  __shared__ double sloss[8];
  const int nb = blockIdx.x % a.blocks;
  const int ntt = (a.Lin + kRows - 1) / kRows, ntiles = a.B * ntt;
  const int first = blockIdx.x / a.blocks, step = gridDim.x / a.blocks;
  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      bar_init(full + 8 * i, 1);
      bar_init(empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(tfull + 8 * i, 1);
      bar_init(tempty + 8 * i, 8);
    }
    bar_init(wfull, 1);
    bar_init(never, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *dead = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int n = tid; n < a.N; n += 320) sbias[n] = a.bias[LAST ? (n >> 5) * a.outC + 32 * nb + (n & 31) : n];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool stalled = false;
  if (a.stall_test) {
    if (tid == 0) *dead = !mbar_wait(never, 0, 20000000ull);
    __syncthreads();
    stalled = *dead != 0;
  }
  int issued = 0;  // tiles this role has started
  if (stalled) {
    // nothing is issued
  } else if (warp == 0) {
    if (lane == 0) {
      const uint8_t* w = reinterpret_cast<const uint8_t*>(a.W) + static_cast<size_t>(nb) * wbytes;
      expect_tx(wfull, wbytes);
      for (int d = 0; d < 3; ++d) bulk_load(base + d * (wbytes / 3), w + d * (wbytes / 3), wbytes / 3, wfull);
      for (int tile = first; tile < ntiles && !*dead; tile += step, ++issued) {
        const int st = issued % a.stages;
        if (issued >= a.stages && !mbar_wait(empty + 8 * st, (issued / a.stages - 1) & 1)) {
          *dead = 1;
          break;
        }
        const int b = tile / ntt, t0 = (tile - b * ntt) * kRows;
        expect_tx(full + 8 * st, sbytes);
        const bf16* src = a.in + (static_cast<size_t>(b) * G * a.Lpi + t0) * 8;
        for (int g = 0; g < G; ++g)
          bulk_load(sA + st * sbytes + g * kWinGroup, src + static_cast<size_t>(g) * a.Lpi * 8, kWinGroup, full + 8 * st);
      }
      // the copies in flight land before the CTA may leave
      if (!mbar_wait(wfull, 0)) *dead = 1;
      for (int i = issued > a.stages ? issued - a.stages : 0; i < issued; ++i)
        if (!mbar_wait(full + 8 * (i % a.stages), (i / a.stages) & 1)) *dead = 1;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      if (!mbar_wait(wfull, 0)) *dead = 1;
      const uint32_t idesc = packed_idesc(a.N), lbo = a.N * 16u;
      for (int tile = first; tile < ntiles && !*dead; tile += step, ++issued) {
        const int st = issued % a.stages, buf = issued & 1;
        if ((issued >= 2 && !mbar_wait(tempty + 8 * buf, ((issued >> 1) - 1) & 1)) ||
            !mbar_wait(full + 8 * st, (issued / a.stages) & 1)) {
          *dead = 1;
          break;
        }
        tc_fence_after();
        const uint32_t win = sA + st * sbytes, acc = tmem + buf * 256u;
        bool start = true;
        for (int g0 = 0; g0 < G; g0 += 4)  // chunks of 32 channels
#pragma unroll
          for (int d = 0; d < 3; ++d)
            for (int g = g0; g < G && g < g0 + 4; g += 2) {
              const uint64_t dw = packed_desc(base + d * (wbytes / 3) + g * lbo, lbo);
#pragma unroll
              for (int p = 0; p < UP; ++p) {
                const int off = UP == 1 ? d : 1 + ((p + d - 1) >> 1);
                packed_mma(acc + p * a.N, packed_desc(win + g * kWinGroup + off * 16u, kWinGroup), dw, idesc,
                           !(start && g == 0 && d == 0));
              }
              start = false;
            }
        tc_commit(bars + kMaxStages + st);
        tc_commit(bars + 2 * kMaxStages + buf);
      }
      // the products in flight end before the CTA may free its tensor memory
      if (issued > 0 && !mbar_wait(tfull + 8 * ((issued - 1) & 1), ((issued - 1) >> 1) & 1)) *dead = 1;
    }
  } else {
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    SquareSum squares;
    for (int tile = first; tile < ntiles; tile += step, ++issued) {
      const int buf = issued & 1;
      const int b = tile / ntt, s = (tile - b * ntt) * kRows + q * 32 + lane;
      const size_t at = (static_cast<size_t>(b) * a.outC + 32 * nb + 16 * h) * a.Lin + s;  // last convolution
      float t[16];
      if constexpr (KIND == kTrain) {  // under the wait for the products
#pragma unroll
        for (int i = 0; i < 16; ++i) t[i] = s < a.Lin ? __ldg(a.target + at + static_cast<size_t>(i) * a.Lin) : 0.f;
      }
      if (__any_sync(0xFFFFFFFFu, *dead || !mbar_wait(tfull + 8 * buf, (issued >> 1) & 1))) {
        *dead = 1;
        break;
      }
      tc_fence_after();
      const uint32_t acc = tmem + lanes + buf * 256u;
      if constexpr (LAST) {
        float sum[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) sum[i] = 0.f;
        const float* xb = a.x + static_cast<size_t>(b) * a.in_dim + a.k0;
        for (int k = 0; k < a.K; ++k) {
          float v[16];
          const int col = 32 * k + 16 * h;
          tmem_ld16(acc + col, v);
          const float xk = __ldg(xb + k);
#pragma unroll
          for (int i = 0; i < 16; ++i) sum[i] = fmaf(xk, v[i] + sbias[col + i], sum[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(tempty + 8 * buf);
        if constexpr (KIND == kAnswer) {
          if (s < a.Lin) {
#pragma unroll
            for (int i = 0; i < 16; ++i) a.y[at + static_cast<size_t>(i) * a.Lin] = sum[i];
          }
        } else {
          if (s < a.Lin) {
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] -= t[i];
            squares.add16(sum);
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] *= a.scale;
            const int row = 1 + s, g0 = (32 * nb + 16 * h) / 8, gs = a.outC / 8;
            for (int k = 0; k < a.K; ++k) {
              const float xk = __ldg(xb + k);
              float v[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) v[i] = xk * sum[i];
              uint4* o = reinterpret_cast<uint4*>(a.dD) +
                         (static_cast<size_t>(b) * a.K * gs + k * gs + g0) * a.Lpi + row;
              o[0] = pack8(v);
              o[a.Lpi] = pack8(v + 8);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] = 0.f;
          }
          const float total = warp_sums16(sum, lane);
          if (!(lane & 1))
            a.row_sums[(static_cast<size_t>(b) * ntt * 4 + (tile - b * ntt) * 4 + q) * a.outC + 32 * nb + 16 * h +
                       warp_sums16_index(lane)] = total;
        }
      } else {
        const int half = a.N / 2, L = UP * a.Lin;
        uint4* out = reinterpret_cast<uint4*>(a.out) + static_cast<size_t>(b) * (a.N / 8) * a.Lpo + 1 + UP * s;
        for (int c = h * half; c < (h + 1) * half; c += 16) {
          float v[UP][16];
#pragma unroll
          for (int p = 0; p < UP; ++p) {
            tmem_ld16(acc + p * a.N + c, v[p]);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[p][i] += sbias[c + i];
          }
          if (s < a.Lin && a.pre) {
            float* pre = a.pre + (static_cast<size_t>(b) * a.N + c) * L + UP * s;
#pragma unroll
            for (int i = 0; i < 16; ++i)
#pragma unroll
              for (int p = 0; p < UP; ++p) pre[static_cast<size_t>(i) * L + p] = v[p][i];
          }
#pragma unroll
          for (int p = 0; p < UP; ++p)
#pragma unroll
            for (int i = 0; i < 16; ++i) v[p][i] = gelu(v[p][i]);
          if (s < a.Lin) {
#pragma unroll
            for (int i = 0; i < 16; i += 8)
#pragma unroll
              for (int p = 0; p < UP; ++p) out[static_cast<size_t>((c + i) >> 3) * a.Lpo + p] = pack8(v[p] + i);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(tempty + 8 * buf);
      }
    }
    if constexpr (KIND == kTrain) {
      double loss = squares.value();
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, off);
      if (lane == 0) reinterpret_cast<volatile double*>(sloss)[warp - 2] = loss;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  if (KIND == kTrain && tid == 0) {
    double sum = 0.0;
    for (int i = 0; i < 8; ++i) sum += stalled ? 0.0 : sloss[i];
    a.loss[blockIdx.x] = sum;
  }
  if (tid == 0 && *dead) atomicExch(a.err, 1);
}

// ---- weight gradients ---------------------------------------------------------------------
// dW[o][c][d] = sum_{b,t} dZ[b][o][t] X[b][c][(t + d - 1) / UP]: a CTA owns 128 output channels,
// every input channel and the three taps (3 Ci accumulator columns), over the samples of one of
// `splits` ranges. K runs along time: both operands are MN-major, groups of 8 channels apart by
// the group's rows, 8 times 128 bytes apart, and a tap (and, UP 2, the parity of t) is a row
// offset of the input window, so dZ and X are staged once for all taps. Warp 0 copies windows of
// 128 rows, a lane per group; warp 1 issues the MMAs; all warps store the result. Bound by L2:
// 448 bytes a time step for 37 k multiply-adds. Default network, 256 samples: the four layers
// 3.96 ms with the general kernel (a CTA per tap, threads rounding and storing every operand),
// 0.25 ms here, the last one 0.19 (0.91 PFLOP/s).
struct WgradArgs {
  int B, Ci, Co, Lin, Lp, stages, splits;
  const bf16* dZ;  // packed [B][Co/8][UP][Lp][8]
  const bf16* X;   // packed [B][Ci/8][Lp][8]
  float* dst;      // [splits][Co][Ci][3]
  int* err;
  int stall_test;
};
constexpr uint32_t kGradGroup = kRows * 16;  // bytes of a channel group of 128 rows of dZ

// kind::f16 descriptor of MN-major operands: mn = bytes to the next 8 channels
__device__ __forceinline__ uint64_t mn_desc(uint32_t addr, uint32_t mn) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) | (static_cast<uint64_t>(128u >> 4) << 16) |
         (static_cast<uint64_t>((mn >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

template <int UP>
__global__ void __launch_bounds__(256, 1) packed_wgrad_kernel(const WgradArgs a) {
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int GI = a.Ci / 8, GO = a.Co / 8;
  const uint32_t abytes = UP * 16 * kGradGroup, sbytes = abytes + GI * kWinGroup;
  const uint32_t base = smem_addr(sm);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + a.stages * sbytes);
  const uint32_t full = smem_addr(bars), empty = full + 8 * kMaxStages, done = empty + 8 * kMaxStages, never = done + 8;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 2);
  volatile int* dead = reinterpret_cast<volatile int*>(slot + 1);
  const int ntiles_o = (GO + 15) / 16, ot = blockIdx.x % ntiles_o, z = blockIdx.x / ntiles_o;
  const int go0 = ot * 16, go = min(16, GO - go0);
  const int b0 = static_cast<int>(static_cast<long long>(z) * a.B / a.splits);
  const int b1 = static_cast<int>(static_cast<long long>(z + 1) * a.B / a.splits);
  const int nt = (a.Lin + kRows - 1) / kRows, total = (b1 - b0) * nt;
  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      bar_init(full + 8 * i, 1);
      bar_init(empty + 8 * i, 1);
    }
    bar_init(done, 1);
    bar_init(never, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *dead = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool stalled = false;
  if (a.stall_test) {
    if (tid == 0) *dead = !mbar_wait(never, 0, 20000000ull);
    __syncthreads();
    stalled = *dead != 0;
  }
  if (!stalled && warp == 0) {
    int i = 0;
    for (; i < total; ++i) {
      const int st = i % a.stages;
      bool ok = true;
      if (lane == 0) {
        ok = !*dead && (i < a.stages || mbar_wait(empty + 8 * st, (i / a.stages - 1) & 1));
        if (ok) expect_tx(full + 8 * st, UP * go * kGradGroup + GI * kWinGroup);
      }
      if (!__shfl_sync(0xFFFFFFFFu, ok, 0)) {
        *dead = 1;
        break;
      }
      const int b = b0 + i / nt, t0 = (i % nt) * kRows;
      const uint32_t sa = base + st * sbytes;
      for (int g = lane; g < UP * go + GI; g += 32) {
        if (g < UP * go) {
          const int p = g / go, gg = g - p * go;
          bulk_load(sa + (p * 16 + gg) * kGradGroup,
                    a.dZ + (((static_cast<size_t>(b) * GO + go0 + gg) * UP + p) * a.Lp + 1 + t0) * 8, kGradGroup,
                    full + 8 * st);
        } else {
          const int gg = g - UP * go;
          bulk_load(sa + abytes + gg * kWinGroup, a.X + ((static_cast<size_t>(b) * GI + gg) * a.Lp + t0) * 8, kWinGroup,
                    full + 8 * st);
        }
      }
    }
    if (lane == 0)  // the copies in flight land before the CTA may leave
      for (int k = i > a.stages ? i - a.stages : 0; k < i; ++k)
        if (!mbar_wait(full + 8 * (k % a.stages), (k / a.stages) & 1)) *dead = 1;
  } else if (!stalled && warp == 1 && lane == 0) {
    const uint32_t idesc = packed_idesc(a.Ci) | (1u << 15) | (1u << 16);  // both operands MN-major
    for (int i = 0; i < total && !*dead; ++i) {
      const int st = i % a.stages;
      if (!mbar_wait(full + 8 * st, (i / a.stages) & 1)) {
        *dead = 1;
        break;
      }
      tc_fence_after();
      const uint32_t sa = base + st * sbytes, sx = sa + abytes;
      for (int k = 0; k < kRows; k += 16)
#pragma unroll
        for (int p = 0; p < UP; ++p)
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const int off = UP == 1 ? d : 1 + ((p + d - 1) >> 1);
            packed_mma(tmem + d * a.Ci, mn_desc(sa + p * 16 * kGradGroup + k * 16u, kGradGroup),
                       mn_desc(sx + (k + off) * 16u, kWinGroup), idesc, (i | k | p) != 0);
          }
      tc_commit(bars + kMaxStages + st);
    }
    tc_commit(bars + 2 * kMaxStages);
    if (!mbar_wait(done, 0)) *dead = 1;
  }
  __syncwarp();
  __syncthreads();
  tc_fence_after();
  const bool failed = *dead != 0;
  if (!failed) {
    const int q = warp & 3, o = ot * kRows + q * 32 + lane;
    float* dst = a.dst + (static_cast<size_t>(z) * a.Co + o) * a.Ci * 3;
    for (int cb = warp >> 2; cb < a.Ci / 16; cb += 2) {
      float v[3][16];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + d * a.Ci + 16 * cb, v[d]);
        if (total == 0)
#pragma unroll
          for (int i = 0; i < 16; ++i) v[d][i] = 0.f;
      }
      if (o < a.Co) {
        float4* w = reinterpret_cast<float4*>(dst + 48 * cb);
#pragma unroll
        for (int j = 0; j < 12; ++j)
          w[j] = make_float4(v[(4 * j) % 3][(4 * j) / 3], v[(4 * j + 1) % 3][(4 * j + 1) / 3],
                             v[(4 * j + 2) % 3][(4 * j + 2) / 3], v[(4 * j + 3) % 3][(4 * j + 3) / 3]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  if (tid == 0 && failed) atomicExch(a.err, 1);
}

// dW = the splits' sums in split order
__global__ void sum_splits_kernel(size_t n4, int splits, const float4* __restrict__ ws, float4* __restrict__ dW) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n4;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    float4 s = ws[i];
    for (int z = 1; z < splits; ++z) {
      const float4 v = ws[z * n4 + i];
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    dW[i] = s;
  }
}

// ---- data gradients -----------------------------------------------------------------------
// dX[b][c][t'] = sum_{o,d,r<UP} W[o][c][d] dZ[b][o][UP t' + r - d + 1], then dz = dX gelu'(pre)
// of the layer below, its bias sums and its packed bfloat16 copy, all in the epilogue, so dX
// stays in registers. Persistent CTAs walk items of 256 times of one sample: two row tiles that
// share each chunk of 32 output channels' weights, streamed with the windows (the last layer's
// 663 KB do not fit), two items' accumulators alternating. Term (r, d) reads the window of parity
// (r - d + 1) mod UP at a fixed row offset. K order: chunk, r, d, 16 channels. Bias sums are kept
// per thread over all of a CTA's tiles, and the pre-activations are loaded a block ahead of the
// activation's derivative (without that the three hidden layers took 78 us each, now 28). Last
// layer of the default network, 256 samples: 506 us with the general kernel, 189 here (0.90
// PFLOP/s; bound by L2: 35 KB a chunk for 660 cycles of products).
struct DgradArgs {
  int B, Ci, Co, Lin, Lp, stages;
  const bf16* dZ;    // packed [B][Co/8][UP][Lp][8]
  const bf16* Wt;    // packed [Co/32][3][4][Ci][8]
  const float* pre;  // [B][Ci][Lin]
  bf16* out;         // packed [B][Ci/8][out_up][Lpo][8], or null
  int out_up, Lpo;
  float* out_f32;    // [B][Ci][Lin], or null
  float* sums;       // [CTAs][Ci], or null
  int* err;
  int stall_test;
};

template <int UP>
__global__ void __launch_bounds__(320, 1) packed_dgrad_kernel(const DgradArgs a) {
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int GO = a.Co / 8, nq = a.Co / 32;
  const uint32_t tap = 4u * a.Ci * 16, wbytes = 3 * tap, abytes = 2 * UP * 4 * kWinGroup, sbytes = abytes + wbytes;
  const uint32_t base = smem_addr(sm);
  float* ssum = reinterpret_cast<float*>(sm + a.stages * sbytes);  // [4][Ci]
  uint64_t* bars = reinterpret_cast<uint64_t*>(ssum + 4 * a.Ci);
  const uint32_t full = smem_addr(bars), empty = full + 8 * kMaxStages, tfull = empty + 8 * kMaxStages,
                 tempty = tfull + 16, never = tempty + 16;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 5);
  volatile int* dead = reinterpret_cast<volatile int*>(slot + 1);
  const int ntt = (a.Lin + kRows - 1) / kRows, per = (ntt + 1) / 2, nitems = a.B * per;
  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      bar_init(full + 8 * i, 1);
      bar_init(empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(tfull + 8 * i, 1);
      bar_init(tempty + 8 * i, 8);
    }
    bar_init(never, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *dead = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  bool stalled = false;
  if (a.stall_test) {
    if (tid == 0) *dead = !mbar_wait(never, 0, 20000000ull);
    __syncthreads();
    stalled = *dead != 0;
  }
  if (stalled) {
    // nothing is issued
  } else if (warp == 0) {
    int i = 0;
    bool go_on = true;
    for (int item = blockIdx.x; item < nitems && go_on; item += gridDim.x) {
      const int b = item / per, tt = 2 * (item - b * per), mt = min(2, ntt - tt);
      for (int q = 0; q < nq; ++q, ++i) {
        const int st = i % a.stages;
        bool ok = true;
        if (lane == 0) {
          ok = !*dead && (i < a.stages || mbar_wait(empty + 8 * st, (i / a.stages - 1) & 1));
          if (ok) expect_tx(full + 8 * st, wbytes + mt * UP * 4 * kWinGroup);
        }
        if (!__shfl_sync(0xFFFFFFFFu, ok, 0)) {
          *dead = 1;
          go_on = false;
          break;
        }
        const uint32_t sa = base + st * sbytes;
        if (lane < mt * UP * 4) {  // (row tile, parity, group)
          const int g = lane & 3, p = UP == 2 ? (lane >> 2) & 1 : 0, m = lane / (UP * 4);
          bulk_load(sa + ((m * UP + p) * 4 + g) * kWinGroup,
                    a.dZ + (((static_cast<size_t>(b) * GO + 4 * q + g) * UP + p) * a.Lp + (tt + m) * kRows) * 8,
                    kWinGroup, full + 8 * st);
        } else if (lane == 31) {
          bulk_load(sa + abytes, a.Wt + static_cast<size_t>(q) * (wbytes / 2), wbytes, full + 8 * st);
        }
      }
    }
    if (lane == 0)  // the copies in flight land before the CTA may leave
      for (int k = i > a.stages ? i - a.stages : 0; k < i; ++k)
        if (!mbar_wait(full + 8 * (k % a.stages), (k / a.stages) & 1)) *dead = 1;
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = packed_idesc(a.Ci), lbo = a.Ci * 16u;
      int i = 0, n = 0;
      for (int item = blockIdx.x; item < nitems && !*dead; item += gridDim.x, ++n) {
        const int b = item / per, mt = min(2, ntt - 2 * (item - b * per)), buf = n & 1;
        if (n >= 2 && !mbar_wait(tempty + 8 * buf, ((n >> 1) - 1) & 1)) {
          *dead = 1;
          break;
        }
        bool ok = true;
        for (int q = 0; q < nq && ok; ++q, ++i) {
          const int st = i % a.stages;
          if (!mbar_wait(full + 8 * st, (i / a.stages) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = base + st * sbytes, sw = sa + abytes;
          for (int m = 0; m < mt; ++m)
#pragma unroll
            for (int r = 0; r < UP; ++r)
#pragma unroll
              for (int d = 0; d < 3; ++d) {
                const int e = r - d + 1, p = UP == 2 ? (e & 1) : 0, off = 1 + (UP == 2 ? (e - p) / 2 : e);
                const uint32_t win = sa + (m * UP + p) * 4 * kWinGroup + off * 16u;
#pragma unroll
                for (int g = 0; g < 4; g += 2)
                  packed_mma(tmem + (2 * buf + m) * a.Ci, packed_desc(win + g * kWinGroup, kWinGroup),
                             packed_desc(sw + d * tap + g * lbo, lbo), idesc, (q | r | d | g) != 0);
              }
          tc_commit(bars + kMaxStages + st);
        }
        if (!ok) {
          *dead = 1;
          break;
        }
        tc_commit(bars + 2 * kMaxStages + buf);
      }
      // the products in flight end before the CTA may free its tensor memory
      if (n > 0 && !mbar_wait(tfull + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1)) *dead = 1;
    }
  } else {
    const int q = warp & 3, h = (warp - 2) >> 2, nblk = a.Ci / 16;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    float bs[4][16];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 16; ++i) bs[j][i] = 0.f;
    int n = 0;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x, ++n) {
      const int b = item / per, tt = 2 * (item - b * per), mt = min(2, ntt - tt), buf = n & 1;
      // pre-activations a block ahead, the first under the wait for the products
      float pz[16], pn[16];
      auto fetch = [&](int m, int cb, float(&to)[16]) {
        const int t = (tt + m) * kRows + q * 32 + lane;
        const float* from = a.pre + (static_cast<size_t>(b) * a.Ci + 16 * cb) * a.Lin + t;
        if (m < mt && cb < nblk && t < a.Lin) {
#pragma unroll
          for (int i = 0; i < 16; ++i) to[i] = __ldg(from + static_cast<size_t>(i) * a.Lin);
        }
      };
      fetch(0, h, pn);
      if (__any_sync(0xFFFFFFFFu, *dead || !mbar_wait(tfull + 8 * buf, (n >> 1) & 1))) {
        *dead = 1;
        break;
      }
      tc_fence_after();
      for (int m = 0; m < mt; ++m) {
        const int t = (tt + m) * kRows + q * 32 + lane;
        const bool in = t < a.Lin;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int cb = 2 * j + h;
          if (cb >= nblk) continue;
#pragma unroll
          for (int i = 0; i < 16; ++i) pz[i] = pn[i];
          if (cb + 2 < nblk)
            fetch(m, cb + 2, pn);
          else
            fetch(m + 1, h, pn);
          float v[16];
          tmem_ld16(tmem + lanes + (2 * buf + m) * a.Ci + 16 * cb, v);
          const size_t at = (static_cast<size_t>(b) * a.Ci + 16 * cb) * a.Lin + t;
          if (in) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              v[i] *= gelu_grad(pz[i]);
              bs[j][i] += v[i];
            }
            if (a.out) {
              const int par = a.out_up == 2 ? t & 1 : 0, row = 1 + (a.out_up == 2 ? t >> 1 : t);
              uint4* o = reinterpret_cast<uint4*>(a.out) +
                         ((static_cast<size_t>(b) * (a.Ci / 8) + 2 * cb) * a.out_up + par) * a.Lpo + row;
              o[0] = pack8(v);
              o[static_cast<size_t>(a.out_up) * a.Lpo] = pack8(v + 8);
            }
            if (a.out_f32) {
#pragma unroll
              for (int i = 0; i < 16; ++i) a.out_f32[at + static_cast<size_t>(i) * a.Lin] = v[i];
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive(tempty + 8 * buf);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float total = warp_sums16(bs[j], lane);
      if (2 * j + h < nblk && !(lane & 1)) ssum[q * a.Ci + 16 * (2 * j + h) + warp_sums16_index(lane)] = total;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  if (a.sums && !stalled && tid < a.Ci)
    a.sums[static_cast<size_t>(blockIdx.x) * a.Ci + tid] =
        ((ssum[tid] + ssum[a.Ci + tid]) + ssum[2 * a.Ci + tid]) + ssum[3 * a.Ci + tid];
  if (tid == 0 && *dead) atomicExch(a.err, 1);
}

// db[c] = sum over the rows (CTAs) in order
__global__ void sum_rows_kernel(int rows, int C, const float* __restrict__ sums, float* __restrict__ db) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  float s = 0.f;
#pragma unroll 8
  for (int r = 0; r < rows; ++r) s += sums[static_cast<size_t>(r) * C + c];
  db[c] = s;
}

// sums[b][c] = sum over the parts of row_sums[b][part][c], in order, over the first part
__global__ void part_sums_kernel(int parts, int C, float* __restrict__ row_sums) {
  float* r = row_sums + static_cast<size_t>(blockIdx.x) * parts * C;
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int p = 0; p < parts; ++p) s += r[static_cast<size_t>(p) * C + c];
    r[c] = s;
  }
}
// db[k outC + c] = sum_b x[b][k0 + k] sums[b][c]: 32 channels a block, eight interleaved ranges of
// samples added in order.
__global__ void __launch_bounds__(256) contracted_bias_kernel(int B, size_t stride, int outC, int in_dim, int k0,
                                                              const float* __restrict__ x,
                                                              const float* __restrict__ sums, float* __restrict__ db) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane, k = blockIdx.y;
  float s = 0.f;
#pragma unroll 8
  for (int b = w; b < B; b += 8) s = fmaf(x[static_cast<size_t>(b) * in_dim + k0 + k], sums[b * stride + c], s);
  red[w][lane] = s;
  __syncthreads();
  if (w == 0) {
    for (int i = 1; i < 8; ++i) s += red[i][lane];
    db[static_cast<size_t>(k) * outC + c] = s;
  }
}

// Transposed weights of the data gradient, [Co/32][3][4][Ci][8]: element i of row c of group g of
// chunk q at tap d is W[32 q + 8 g + i][c][d].
__global__ void pack_conv_t_kernel(int Ci, int Co, const bf16* __restrict__ W, bf16* __restrict__ Wt) {
  const size_t total = static_cast<size_t>(3) * Ci * Co;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int e = static_cast<int>(i & 7);
    size_t r = i >> 3;
    const int c = static_cast<int>(r % Ci);
    r /= Ci;
    const int g = static_cast<int>(r & 3);
    r >>= 2;
    const int d = static_cast<int>(r % 3), q = static_cast<int>(r / 3);
    Wt[i] = W[(static_cast<size_t>(32 * q + 8 * g + e) * Ci + c) * 3 + d];
  }
}

int wgrad_smem(int Ci, int up, int stages) {
  return stages * (up * 16 * static_cast<int>(kGradGroup) + Ci / 8 * static_cast<int>(kWinGroup)) + (2 * kMaxStages + 4) * 8;
}
int wgrad_stages(int Ci, int up) {
  int st = kMaxStages;
  while (st > 1 && wgrad_smem(Ci, up, st) > kSmemLimit) --st;
  return st;
}
int dgrad_smem(int Ci, int up, int stages) {
  return stages * (8 * up * static_cast<int>(kWinGroup) + 12 * Ci * 16) + 16 * Ci + (2 * kMaxStages + 7) * 8;
}
int dgrad_stages(int Ci, int up) {
  int st = kMaxStages;
  while (st > 1 && dgrad_smem(Ci, up, st) > kSmemLimit) --st;
  return st;
}

int dense_smem(int Kp) { return Kp / 8 * 3072 + 7 * 8 + 64 * 4; }
int conv_smem(int Ci, int N, int stages) {
  return 3 * Ci * N * 2 + stages * (Ci / 8) * static_cast<int>(kWinGroup) + N * 4 + (2 * kMaxStages + 8) * 8;
}
int conv_stages(int Ci, int N) {
  int st = kMaxStages;
  while (st >= 2 && conv_smem(Ci, N, st) > kSmemLimit) --st;
  return st;
}
// one CTA per SM, the same number for every column block
int conv_grid(int B, int blocks, int Lin) {
  const long long tiles = static_cast<long long>(B) * ((Lin + kRows - 1) / kRows);
  return blocks * static_cast<int>(std::max<long long>(1, std::min<long long>(kSms / blocks, tiles)));
}
int grid1(size_t n) { return static_cast<int>(std::min<size_t>((n + 255) / 256, 65535)); }

// The attribute is the process's, not the launch's: every model sets the same value, so that a
// model in another thread, of other sizes, cannot lower it between this call and the launch.
template <class K>
cudaError_t raise_smem(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
}

}  // namespace

int packed_rows(int L) { return 2 + (L + kRows - 1) / kRows * kRows; }

bool packed_dense_ok(int K, int N) { return N % 64 == 0 && K > 0 && dense_smem((K + 31) / 32 * 32) <= kSmemLimit; }
bool packed_conv_ok(int Ci, int N, int up) {
  return Ci % 16 == 0 && N % 32 == 0 && N * up <= 256 && conv_stages(Ci, N) >= 2;
}
size_t packed_dense_elems(int K, int N) { return static_cast<size_t>(N) * ((K + 31) / 32 * 32); }

int pack_dense(int K, int N, int l0, const bf16* W, bf16* Wp, cudaStream_t s) {
  const int Kp = (K + 31) / 32 * 32;
  pack_dense_kernel<<<grid1(packed_dense_elems(K, N)), 256, 0, s>>>(N, K, Kp, l0, W, Wp);
  return static_cast<int>(cudaGetLastError());
}
int pack_conv(int Ci, int N, int blocks, int outC, const bf16* W, bf16* Wp, cudaStream_t s) {
  pack_conv_rows_kernel<<<grid1(static_cast<size_t>(blocks) * 3 * Ci * N), 256, 0, s>>>(Ci, N, blocks, outC, W, Wp);
  return static_cast<int>(cudaGetLastError());
}

template <bool FROM_X, bool TO_Z>
static int launch_dense(const DenseArgs& a, cudaStream_t s) {
  const int smem = dense_smem(a.Kp);
  const cudaError_t e = raise_smem(dense_kernel<FROM_X, TO_Z>);
  if (e != cudaSuccess) return static_cast<int>(e);
  dense_kernel<FROM_X, TO_Z><<<dim3(a.N / 64, (a.B + kRows - 1) / kRows), 256, smem, s>>>(a);
  return static_cast<int>(cudaGetLastError());
}

int packed_dense(int B, int Bp, int K, int N, const float* x, const bf16* in, const bf16* Wp, const float* bias,
                 bf16* out, float* pre, float* act, int l0, const Products& pr, cudaStream_t s) {
  DenseArgs a{};
  a.act = act;
  a.B = B;
  a.Bp = Bp;
  a.K = K;
  a.Kp = (K + 31) / 32 * 32;
  a.N = N;
  a.x = x;
  a.in = in;
  a.W = Wp;
  a.bias = bias;
  a.out = out;
  a.pre = pre;
  a.l0 = l0;
  a.Lp = l0 ? packed_rows(l0) : 0;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  if (x) return l0 ? launch_dense<true, true>(a, s) : launch_dense<true, false>(a, s);
  return l0 ? launch_dense<false, true>(a, s) : launch_dense<false, false>(a, s);
}

template <int UP, int KIND>
static int launch_conv(const ConvArgs& a, cudaStream_t s) {
  const int smem = conv_smem(a.Ci, a.N, a.stages);
  const cudaError_t e = raise_smem(packed_conv_kernel<UP, KIND>);
  if (e != cudaSuccess) return static_cast<int>(e);
  packed_conv_kernel<UP, KIND><<<conv_grid(a.B, a.blocks, a.Lin), 320, smem, s>>>(a);
  return static_cast<int>(cudaGetLastError());
}

int packed_conv(int B, int Ci, int N, int Lin, int up, const bf16* in, const bf16* Wp, const float* bias, bf16* out,
                float* pre, const Products& pr, cudaStream_t s) {
  ConvArgs a{};
  a.B = B;
  a.Ci = Ci;
  a.Lin = Lin;
  a.Lpi = packed_rows(Lin);
  a.N = N;
  a.stages = conv_stages(Ci, N);
  a.blocks = 1;
  a.in = in;
  a.W = Wp;
  a.bias = bias;
  a.out = out;
  a.Lpo = packed_rows(up * Lin);
  a.pre = pre;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  return up == 2 ? launch_conv<2, kHidden>(a, s) : launch_conv<1, kHidden>(a, s);
}

static ConvArgs contract_args(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp,
                              const float* bias, const float* x, const Products& pr) {
  ConvArgs a{};
  a.B = B;
  a.Ci = Ci;
  a.Lin = Lin;
  a.Lpi = packed_rows(Lin);
  a.N = 32 * K;
  a.stages = conv_stages(Ci, a.N);
  a.blocks = outC / 32;
  a.in = in;
  a.W = Wp;
  a.bias = bias;
  a.x = x;
  a.in_dim = in_dim;
  a.k0 = in_dim - K;
  a.K = K;
  a.outC = outC;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  return a;
}

int packed_conv_contract(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp,
                         const float* bias, const float* x, float* y, const Products& pr, cudaStream_t s) {
  ConvArgs a = contract_args(B, Ci, K, outC, Lin, in_dim, in, Wp, bias, x, pr);
  a.y = y;
  return launch_conv<1, kAnswer>(a, s);
}

int packed_loss(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp, const float* bias,
                const float* x, const float* target, bf16* dD, float* row_sums, float* db, double* loss,
                const Products& pr, cudaStream_t s) {
  ConvArgs a = contract_args(B, Ci, K, outC, Lin, in_dim, in, Wp, bias, x, pr);
  a.target = target;
  a.scale = 2.f / static_cast<float>(static_cast<size_t>(B) * outC * Lin);
  a.dD = dD;
  a.row_sums = row_sums;
  a.loss = loss;
  const int r = launch_conv<1, kTrain>(a, s);
  if (r) return r;
  const int parts = (Lin + kRows - 1) / kRows * 4;
  part_sums_kernel<<<B, std::min(256, outC), 0, s>>>(parts, outC, row_sums);
  contracted_bias_kernel<<<dim3(outC / 32, K), 256, 0, s>>>(B, static_cast<size_t>(parts) * outC, outC, in_dim,
                                                            in_dim - K, x, row_sums, db);
  return static_cast<int>(cudaGetLastError());
}

int packed_loss_blocks(int B, int outC, int Lin) {
  return conv_grid(B, outC / 32, Lin);
}

int loss_values(int B, int outC, int Lin) {
  return outC < 32 ? kLossBlocks : std::max(kLossBlocks, packed_loss_blocks(B, outC, Lin));
}

bool packed_backward_ok(int Ci, int Co, int up) {
  return Ci % 16 == 0 && Ci <= 128 && Co % 32 == 0 && (up == 1 || up == 2);
}

size_t packed_grad_elems(int Co, int Lin, int up) { return static_cast<size_t>(Co) * up * packed_rows(Lin); }

int pack_conv_t(int Ci, int Co, const bf16* W, bf16* Wt, cudaStream_t s) {
  pack_conv_t_kernel<<<grid1(static_cast<size_t>(3) * Ci * Co), 256, 0, s>>>(Ci, Co, W, Wt);
  return static_cast<int>(cudaGetLastError());
}

int packed_conv_wgrad(int B, int Ci, int Co, int Lin, int up, const bf16* dZ, const bf16* X, float* dW, float* ws,
                      const Products& pr, cudaStream_t s) {
  WgradArgs a{};
  a.B = B;
  a.Ci = Ci;
  a.Co = Co;
  a.Lin = Lin;
  a.Lp = packed_rows(Lin);
  a.dZ = dZ;
  a.X = X;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  const int ot = (Co + kRows - 1) / kRows;
  const size_t mn = static_cast<size_t>(Co) * Ci * 3;
  a.splits = std::max(1, std::min({B, kSms / ot, static_cast<int>(ws ? pr.ws_floats / mn : 1)}));
  a.dst = a.splits > 1 ? ws : dW;
  const int smem = wgrad_smem(Ci, up, wgrad_stages(Ci, up));
  a.stages = wgrad_stages(Ci, up);
  cudaError_t e = up == 2 ? raise_smem(packed_wgrad_kernel<2>) : raise_smem(packed_wgrad_kernel<1>);
  if (e != cudaSuccess) return static_cast<int>(e);
  if (up == 2)
    packed_wgrad_kernel<2><<<ot * a.splits, 256, smem, s>>>(a);
  else
    packed_wgrad_kernel<1><<<ot * a.splits, 256, smem, s>>>(a);
  if (a.splits > 1) sum_splits_kernel<<<grid1(mn / 4), 256, 0, s>>>(mn / 4, a.splits, reinterpret_cast<const float4*>(ws),
                                                                   reinterpret_cast<float4*>(dW));
  return static_cast<int>(cudaGetLastError());
}

int packed_conv_dgrad(int B, int Ci, int Co, int Lin, int up, const bf16* dZ, const bf16* Wt, const float* pre,
                      bf16* out, int out_up, float* out_f32, float* sums, float* db, const Products& pr,
                      cudaStream_t s) {
  DgradArgs a{};
  a.B = B;
  a.Ci = Ci;
  a.Co = Co;
  a.Lin = Lin;
  a.Lp = packed_rows(Lin);
  a.dZ = dZ;
  a.Wt = Wt;
  a.pre = pre;
  a.out = out;
  a.out_up = out_up;
  a.Lpo = out_up == 2 ? packed_rows(Lin / 2) : packed_rows(Lin);
  a.out_f32 = out_f32;
  a.sums = sums;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  a.stages = dgrad_stages(Ci, up);
  const int smem = dgrad_smem(Ci, up, a.stages);
  const int items = B * ((Lin + 2 * kRows - 1) / (2 * kRows)), grid = std::min(kSms, items);
  const cudaError_t e = up == 2 ? raise_smem(packed_dgrad_kernel<2>) : raise_smem(packed_dgrad_kernel<1>);
  if (e != cudaSuccess) return static_cast<int>(e);
  if (up == 2)
    packed_dgrad_kernel<2><<<grid, 320, smem, s>>>(a);
  else
    packed_dgrad_kernel<1><<<grid, 320, smem, s>>>(a);
  if (db) sum_rows_kernel<<<(Ci + 31) / 32, 32, 0, s>>>(grid, Ci, sums, db);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace sgk
