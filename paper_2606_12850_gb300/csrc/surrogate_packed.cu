// The surrogate's forward pass on packed activations (sm_103a): every layer's output is stored
// once, as the bfloat16 values the next product rounds its operand to, in the core-matrix
// layout that tcgen05 reads, so staging an operand is a few bulk copies and no thread converts
// or rearranges anything between layers. The float32 pre-activations are stored only where the
// backward pass needs them. Products, their K order, bias, activation and contraction are those
// of the general kernels (surrogate_kernels.cu), so results are the same bit for bit.
//
// Packed rows: 16 bytes = 8 consecutive channels (or features) of one row, rows of a channel
// group consecutive. Dense layers: [features/8][batch rows][8]. Convolutions: [sample][C/8]
// [packed_rows(L)][8], row 1 + t holding time t, the rows around the samples zero (the 'same'
// padding and the tail of the last tile), so a window of 130 rows is one copy per group.
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
constexpr int kSmemLimit = 227 * 1024;

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
// LAST: the columns are K contracted copies of 32 output channels; the epilogue forms y = sum_k
// x_k (D_k + bias_k) in registers, so D (K times the output) never reaches memory (the general
// kernel wrote 1.2 GB of it per 256 samples of the default network and a second kernel read it
// back). The default network's forward pass of 4096 samples in chunks of 256, GB300: 16.6 ms
// with the general kernels (tc_conv_kernel 12.2, contraction 4.4, dense 2.0), 3.6 ms now, 880
// TFLOP/s of products; one sample 69 against 27 us, bound by the latency of seven launches.
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
  float* y;         // LAST: [B][outC][Lin]
  int* err;
  int stall_test;
};

template <int UP, bool LAST>
__global__ void __launch_bounds__(320, 1) packed_conv_kernel(const ConvArgs a) {
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
    for (int tile = first; tile < ntiles; tile += step, ++issued) {
      const int buf = issued & 1;
      const int b = tile / ntt, s = (tile - b * ntt) * kRows + q * 32 + lane;
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
        if (s < a.Lin) {
          float* y = a.y + (static_cast<size_t>(b) * a.outC + 32 * nb + 16 * h) * a.Lin + s;
#pragma unroll
          for (int i = 0; i < 16; ++i) y[static_cast<size_t>(i) * a.Lin] = sum[i];
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
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  if (tid == 0 && *dead) atomicExch(a.err, 1);
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
int grid1(size_t n) { return static_cast<int>(std::min<size_t>((n + 255) / 256, 65535)); }

template <class K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
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
  const cudaError_t e = set_smem(dense_kernel<FROM_X, TO_Z>, smem);
  if (e != cudaSuccess) return static_cast<int>(e);
  dense_kernel<FROM_X, TO_Z><<<dim3(a.N / 64, (a.B + kRows - 1) / kRows), 256, smem, s>>>(a);
  return static_cast<int>(cudaGetLastError());
}

int packed_dense(int B, int Bp, int K, int N, const float* x, const bf16* in, const bf16* Wp, const float* bias,
                 bf16* out, float* pre, int l0, const Products& pr, cudaStream_t s) {
  DenseArgs a{};
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

template <int UP, bool LAST>
static int launch_conv(const ConvArgs& a, cudaStream_t s) {
  const int smem = conv_smem(a.Ci, a.N, a.stages);
  const cudaError_t e = set_smem(packed_conv_kernel<UP, LAST>, smem);
  if (e != cudaSuccess) return static_cast<int>(e);
  // one CTA per SM (152), the same number for every column block
  const long long tiles = static_cast<long long>(a.B) * ((a.Lin + kRows - 1) / kRows);
  const int per = static_cast<int>(std::max<long long>(1, std::min<long long>(152 / a.blocks, tiles)));
  packed_conv_kernel<UP, LAST><<<per * a.blocks, 320, smem, s>>>(a);
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
  return up == 2 ? launch_conv<2, false>(a, s) : launch_conv<1, false>(a, s);
}

int packed_conv_contract(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp,
                         const float* bias, const float* x, float* y, const Products& pr, cudaStream_t s) {
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
  a.y = y;
  a.err = pr.err;
  a.stall_test = pr.stall_test;
  return launch_conv<1, true>(a, s);
}

}  // namespace sgk
