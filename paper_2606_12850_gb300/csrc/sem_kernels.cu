// CUDA kernels of libsemgb (sm_103a) other than the force kernel (sem_forces.cuh): order
// dispatch, the Newmark corrector pass, sources/receivers, energy partials.
#include <cuda_runtime.h>

#include <cmath>

#include "sem_internal.h"
#include "sem_newmark.cuh"

namespace semgb {

// ---------------------------------------------------------------------------------------
// Dispatch to the per-order translation units (sem_forces_<N>.cu).
// ---------------------------------------------------------------------------------------
#define SEM_DECLARE_ORDER(n)                                                                                \
  int upload_basis_##n(const double* w, const double* h, void* stream, int ngll);                         \
  int launch_forces_##n(const ForceLaunch& L, void* stream);                                              \
  int forces_smem_bytes_##n();                                                                            \
  int launch_patch_forces_##n(const PatchLaunch& L, void* stream);                                        \
  int launch_group_sweep_##n(const GroupLaunch& L, void* stream);                                         \
  void patch_shape_##n(PatchShape* out);                                                                  \
  void patch_layout_##n(PatchLayout* out);                                                                \
  int launch_sensitivity_##n(const float* rec, const int* perm, const float* lam, const float* u_lo,       \
                             const float* u_mid, const float* u_hi, float* g_rho, float* g_kappa,       \
                             float* g_mu, int nspec, double c_m, double c_k, void* stream,              \
                             const DevCtl* idx, int back);
SEM_DECLARE_ORDER(2)
SEM_DECLARE_ORDER(3)
SEM_DECLARE_ORDER(4)
SEM_DECLARE_ORDER(5)
SEM_DECLARE_ORDER(6)
SEM_DECLARE_ORDER(7)
SEM_DECLARE_ORDER(8)
SEM_DECLARE_ORDER(9)
SEM_DECLARE_ORDER(10)

#define SEM_ORDER_SWITCH(n, call) \
  switch (n) {                    \
    case 2: return call(2);       \
    case 3: return call(3);       \
    case 4: return call(4);       \
    case 5: return call(5);       \
    case 6: return call(6);       \
    case 7: return call(7);       \
    case 8: return call(8);       \
    case 9: return call(9);       \
    case 10: return call(10);     \
    default: break;               \
  }

int upload_basis(int n, const double* w, const double* h, void* stream) {
#define SEM_CALL(k) upload_basis_##k(w, h, stream, n)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return static_cast<int>(cudaErrorInvalidValue);
}

int launch_group_sweep(int n, const GroupLaunch& L, void* stream) {
#define SEM_CALL(k) launch_group_sweep_##k(L, stream)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return static_cast<int>(cudaErrorInvalidValue);
}

int launch_forces(int n, const ForceLaunch& L, void* stream) {
#define SEM_CALL(k) launch_forces_##k(L, stream)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return static_cast<int>(cudaErrorInvalidValue);
}

int launch_sensitivity(int n, const float* rec, const int* perm, const float* lam, const float* u_lo,
                       const float* u_mid, const float* u_hi, float* g_rho, float* g_kappa, float* g_mu, int nspec,
                       double c_m, double c_k, void* stream, const DevCtl* idx, int back) {
#define SEM_CALL(k) \
  launch_sensitivity_##k(rec, perm, lam, u_lo, u_mid, u_hi, g_rho, g_kappa, g_mu, nspec, c_m, c_k, stream, idx, back)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return static_cast<int>(cudaErrorInvalidValue);
}

int launch_patch_forces(int n, const PatchLaunch& L, void* stream) {
#define SEM_CALL(k) launch_patch_forces_##k(L, stream)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return static_cast<int>(cudaErrorInvalidValue);
}

static int order_shape(int n, PatchShape* out) {
#define SEM_CALL(k) (patch_shape_##k(out), 0)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return -1;
}

// The order's brick. At NGLL 5, meshes from 4000 elements on take the cube of eight instead, which
// has 386 rim nodes of 729 rather than 450 of 765: there the rim's traffic counts, most with
// several shots and where the records no longer fit the 129 MB L2 (GB300, us a step, 2 x 2 x 2
// against 1 x 4 x 2: 40 x 36 x 44 170.1 / 174.2, 28^3 65.6 / 66.6, 24^3 44.5 / 44.9, 20^3 with 32
// shots 593 / 604). Below, and with one shot on meshes whose sides four divides, neither is the
// faster throughout: 20^3 26.4 / 25.1, 18^3 19.0 / 21.2, 16^3 16.9 / 16.9, 14^3 14.2 / 15.4, 12^3
// 12.7 / 12.5, 10^3 9.9 / 10.4, 8^3 8.69 / 8.63. The line is drawn where the cube is the safer of
// the two on average; SEM_OPT_PATCH_SHAPE sets either.
int patch_shape(int n, int nspec, PatchShape* out) {
  const int r = order_shape(n, out);
  if (r == 0 && n == 5 && nspec >= 4000) *out = PatchShape{2, 2, 2};
  return r;
}

int patch_layout(int n, PatchLayout* out) {
#define SEM_CALL(k) (patch_layout_##k(out), 0)
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return -1;
}

int forces_kernel_smem_bytes(int n) {
#define SEM_CALL(k) forces_smem_bytes_##k()
  SEM_ORDER_SWITCH(n, SEM_CALL)
#undef SEM_CALL
  return 0;
}

int forces_elements_per_cta(int n) {
  if (n < 2 || n > 10) return 0;
  return n * n <= 32 ? 4 * (32 / (n * n)) : 256 / (n * n);
}

// ---------------------------------------------------------------------------------------
// Newmark streaming passes (Sec. I / V-C explicit second-order Newmark, diagonal mass).
// One thread per (node, shot) reads one float4 of each field (the 4th lane stays zero) and the
// node's inverse mass; with several shots a block works on one shot pair, whose slots are
// consecutive, two a node (half 1, else 0).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ long long block_pair() { return static_cast<long long>(blockIdx.z) * gridDim.y + blockIdx.y; }

__device__ __forceinline__ float4 axpy3(float4 y, float s, float4 x) {
  return make_float4(y.x + s * x.x, y.y + s * x.y, y.z + s * x.z, 0.f);
}

// Predictor from a complete state (first step): u += dt v + dt^2/2 a ; v += dt/2 a.
__global__ void predictor_kernel(float4* __restrict__ u, float4* __restrict__ v, const float4* __restrict__ a,
                                 long long n, float dt, float hdt, float hdt2) {
  for (long long g = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; g < n;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float4 ag = a[g], vg = v[g], ug = u[g];
    u[g] = axpy3(axpy3(ug, dt, vg), hdt2, ag);
    v[g] = axpy3(vg, hdt, ag);
  }
}

// Corrector of step n-1 fused with the predictor of step n:
//   a = M^-1 a_raw ; v = v_half + dt/2 a ; u += dt v + dt^2/2 a ; v_half = v + dt/2 a
// a_raw stays in place: the next force sweep overwrites it at each node's first touch.
__global__ void fused_newmark_kernel(float4* __restrict__ u, float4* __restrict__ v,
                                     const float4* __restrict__ a, const float* __restrict__ minv, long long n,
                                     int pairs, int half, float dt, float hdt, float hdt2) {
  if (block_pair() >= pairs) return;
  u += block_pair() * n;
  v += block_pair() * n;
  a += block_pair() * n;
  for (long long g = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; g < n;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float m = minv[g >> half];
    const float4 ar = a[g], vh = v[g], ug = u[g];
    const float4 acc = make_float4(ar.x * m, ar.y * m, ar.z * m, 0.f);
    const float4 vf = axpy3(vh, hdt, acc);
    u[g] = axpy3(axpy3(ug, dt, vf), hdt2, acc);
    v[g] = axpy3(vf, hdt, acc);
  }
}

// Corrector alone (completes the state): a = M^-1 a_raw ; v = v_half + dt/2 a
__global__ void corrector_kernel(float4* __restrict__ v, float4* __restrict__ a, const float* __restrict__ minv,
                                 long long n, int pairs, int half, float hdt) {
  if (block_pair() >= pairs) return;
  v += block_pair() * n;
  a += block_pair() * n;
  for (long long g = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; g < n;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float m = minv[g >> half];
    const float4 ar = a[g];
    const float4 acc = make_float4(ar.x * m, ar.y * m, ar.z * m, 0.f);
    a[g] = acc;
    v[g] = axpy3(v[g], hdt, acc);
  }
}

// Blocks over the slots of a single shot or a shot pair, and the pairs.
static int stream_grid(long long n);
static long long pair_slots(int nglob, int shots) { return static_cast<long long>(nglob) * (shots > 1 ? 2 : 1); }
static dim3 pair_grid(int nglob, int shots) {
  const unsigned pairs = static_cast<unsigned>((shots + 1) / 2), y = pairs < 32768u ? pairs : 32768u;
  return dim3(stream_grid(pair_slots(nglob, shots)), y, (pairs + y - 1) / y);
}

static int stream_grid(long long n) {
  const long long g = (n + 255) / 256;
  return g < 1 ? 1 : static_cast<int>(g < (1ll << 30) ? g : (1ll << 30));
}

int launch_predictor(const DevProblem& p, void* stream) {
  const long long n = static_cast<long long>(p.nglob) * padded_shots(p.shots);
  predictor_kernel<<<stream_grid(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<float4*>(p.u), reinterpret_cast<float4*>(p.v), reinterpret_cast<const float4*>(p.a), n,
      static_cast<float>(p.dt), static_cast<float>(0.5 * p.dt), static_cast<float>(0.5 * p.dt * p.dt));
  return static_cast<int>(cudaGetLastError());
}

int launch_fused_newmark(const DevProblem& p, void* stream) {
  fused_newmark_kernel<<<pair_grid(p.nglob, p.shots), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<float4*>(p.u), reinterpret_cast<float4*>(p.v), reinterpret_cast<const float4*>(p.a), p.minv,
      pair_slots(p.nglob, p.shots), (p.shots + 1) / 2, p.shots > 1, static_cast<float>(p.dt), static_cast<float>(0.5 * p.dt), static_cast<float>(0.5 * p.dt * p.dt));
  return static_cast<int>(cudaGetLastError());
}

int launch_corrector(const DevProblem& p, void* stream) {
  corrector_kernel<<<pair_grid(p.nglob, p.shots), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<float4*>(p.v), reinterpret_cast<float4*>(p.a), p.minv, pair_slots(p.nglob, p.shots),
      (p.shots + 1) / 2, p.shots > 1, static_cast<float>(0.5 * p.dt));
  return static_cast<int>(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------
// The rim pass (Sec. IV-C assembly without colours or atomics): one thread per (rim node,
// shot) adds the partial sums the node's patches left, in sweep order, and does with the
// force what the sweep did at the inner nodes. The node's entry names up to four partials, so
// a face or edge node needs one dependent load before its partials; rim nodes are the last
// internal ids, so the fields stream, and neighbouring nodes of a face have neighbouring
// partials. The entry and the node's state, which no sweep writes at the rim, are loaded
// while the sweep drains. Bound by DRAM: 119 bytes a rim node (entry, partials, u, v, 1/M read,
// u, v written), 40 us for the 2.28 M rim nodes of a 48^3 mesh at NGLL 5, 6.0 TB/s.
// ---------------------------------------------------------------------------------------
template <bool MS, int NM>
__global__ void __launch_bounds__(256) rim_combine_kernel(const RimLaunch R) {
  const long long idx = blockIdx.x * 256ll + threadIdx.x;
  const int t = static_cast<int>(MS ? idx >> 1 : idx);
  const int shot = MS ? 2 * static_cast<int>(block_pair()) + static_cast<int>(idx & 1) : 0;
  const bool in = t < R.nrim && (!MS || shot < R.shots);
  SweepNewmark nm = R.nm;
  float4* f = reinterpret_cast<float4*>(R.f);
  const float4* __restrict__ part = reinterpret_cast<const float4*>(R.partials);
  if constexpr (MS) {
    const size_t slot = field_slot(nm.nglob, 2, 0, shot);
    move_fields(nm, slot);
    f += slot;
    part += field_slot(nm.nsums, 2, 0, shot);
  }
  const uint32_t node = static_cast<uint32_t>(R.ninner + (in ? t : 0));
  int4 q = make_int4(-1, -1, -1, -1);
  NodeState st;
  RimBlock blk{0, 0, 0, 0};
  if (in) {
    q = __ldg(reinterpret_cast<const int4*>(R.rim) + t);
    if constexpr (NM == 1 || NM == 2 || NM == 3) {
      load_node_state<MS, NM>(nm, node, st);
      blk = R.blocks[t / kRimBlock];
    }
  }
  wait_prerequisite_grid();
  allow_dependent_grid();
  if (!in) return;
  constexpr int S = MS ? 2 : 1;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 p0 = __ldcg(part + static_cast<size_t>(q.x) * S);
  const float4 p1 = __ldcg(part + static_cast<size_t>(q.y) * S);
  const float4 p2 = q.z >= 0 ? __ldcg(part + static_cast<size_t>(q.z) * S) : zero;
  const float4 p3 = q.w >= 0 ? __ldcg(part + static_cast<size_t>(q.w) * S) : zero;
  float fx = p0.x + p1.x, fy = p0.y + p1.y, fz = p0.z + p1.z;
  if (q.z >= 0) {
    fx += p2.x;
    fy += p2.y;
    fz += p2.z;
  }
  if (q.w >= 0) {
    fx += p3.x;
    fy += p3.y;
    fz += p3.z;
  } else if (q.w <= -2) {
    const int* __restrict__ o = R.over + (-2 - q.w);
    const int n = __ldg(o);
    for (int k = 1; k <= n; ++k) {
      const float4 p = __ldcg(part + static_cast<size_t>(__ldg(o + k)) * S);
      fx += p.x;
      fy += p.y;
      fz += p.z;
    }
  }
  complete_node<MS, NM>(nm, f, node, shot, st, nm.rim_src + blk.src_off, blk.nsrc, nm.rim_recv + blk.rec_off, blk.nrec,
                        fx, fy, fz);
}

template <bool MS, int NM>
static int launch_rim(const RimLaunch& R, cudaStream_t s) {
  const long long n = static_cast<long long>(R.nrim) * (MS ? 2 : 1);
  cudaLaunchConfig_t cfg = {};
  const unsigned pairs = MS ? (R.shots + 1) / 2 : 1, y = pairs < 32768u ? pairs : 32768u;
  cfg.gridDim = dim3(static_cast<unsigned>((n + 255) / 256), y, (pairs + y - 1) / y);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return static_cast<int>(cudaLaunchKernelEx(&cfg, rim_combine_kernel<MS, NM>, R));
}

int launch_rim_combine(const RimLaunch& R, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (R.nrim <= 0) return 0;
  if (R.shots > 1) {
    if (R.nm.mode > 2) return static_cast<int>(cudaErrorInvalidValue);
    return R.nm.mode ? launch_rim<true, 1>(R, s) : launch_rim<true, 0>(R, s);
  }
  switch (R.nm.mode) {
    case 0: return launch_rim<false, 0>(R, s);
    case 3: return launch_rim<false, 2>(R, s);
    case 4: return launch_rim<false, 4>(R, s);
    default: return R.nm.snap ? launch_rim<false, 3>(R, s) : launch_rim<false, 1>(R, s);
  }
}

// ---------------------------------------------------------------------------------------
// Adjoint leapfrog (the discrete adjoint of the scheme above, run backward in time):
//   lam_new = 2 lam - lam_old + dt^2 M^-1 F,  F = -K lam + R^T G / dt^2
// written over lam_old. Receiver residuals are added to F by one thread per receiver node,
// its receivers in ascending order (receivers may share a node).
// ---------------------------------------------------------------------------------------
__global__ void adjoint_inject_kernel(float* __restrict__ F, const float* __restrict__ G,
                                      const int* __restrict__ rnode, const int* __restrict__ roff,
                                      const int* __restrict__ rlist, int nnodes, float inv_dt2,
                                      const DevCtl* __restrict__ idx, int back) {
  if (idx) G = idx->adj_G + static_cast<long long>(idx->adj_j - back - 1) * idx->adj_gstep;
  // one thread per distinct receiver node; its receivers in ascending order (the order a
  // single thread walking the receivers would add them in)
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nnodes; t += gridDim.x * blockDim.x) {
    float* Fn = F + kNodeStride * static_cast<size_t>(rnode[t]);
    for (int q = roff[t]; q < roff[t + 1]; ++q) {
      const int r = rlist[q];
      for (int c = 0; c < 3; ++c) Fn[c] += G[3 * r + c] * inv_dt2;
    }
  }
}

__global__ void adjoint_leapfrog_kernel(const float4* __restrict__ lam, float4* __restrict__ lam_old,
                                        const float4* __restrict__ F, const float* __restrict__ minv, int nglob,
                                        float dt2) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < nglob; g += gridDim.x * blockDim.x) {
    const float s = dt2 * minv[g];
    const float4 l = lam[g], o = lam_old[g], f = F[g];
    lam_old[g] = make_float4(2.f * l.x - o.x + s * f.x, 2.f * l.y - o.y + s * f.y, 2.f * l.z - o.z + s * f.z, 0.f);
  }
}

__global__ void adjoint_index_kernel(DevCtl* ctl, const float* G, const float* u, long long n3, int gstep, int j) {
  ctl->adj_G = G;
  ctl->adj_u = u;
  ctl->adj_n3 = n3;
  ctl->adj_gstep = gstep;
  ctl->adj_j = j;
}

__global__ void adjoint_next_kernel(DevCtl* ctl, int steps) { ctl->adj_j -= steps; }

int launch_adjoint_index(DevCtl* ctl, const float* G, const float* u, long long n3, int gstep, int j, void* stream) {
  adjoint_index_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ctl, G, u, n3, gstep, j);
  return static_cast<int>(cudaGetLastError());
}

int launch_adjoint_next(DevCtl* ctl, int steps, void* stream) {
  adjoint_next_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ctl, steps);
  return static_cast<int>(cudaGetLastError());
}

__global__ void flush_partials_kernel(float* __restrict__ part, double* __restrict__ acc, long long n) {
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    acc[t] += static_cast<double>(part[t]);
    part[t] = 0.f;
  }
}

int launch_flush_partials(float* part, double* acc, long long n, void* stream) {
  if (n <= 0) return 0;
  flush_partials_kernel<<<stream_grid(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(part, acc, n);
  return static_cast<int>(cudaGetLastError());
}

// One thread per local point, in caller order within its element, so the stores stream; the reads
// of an element's accumulators are 1 KB at NGLL 5, one L1 line set. (The reordering ran on the
// host over a pageable copy: 7.2 ms of a 16 ms gradient of 20^3 elements at NGLL 5.)
template <class T>
__global__ void gradient_order_kernel(const double* __restrict__ acc, const int* __restrict__ order,
                                      T* __restrict__ out, int n, long long total) {
  const int np = n * n * n;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < total;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long s = t / np;
    const int p = static_cast<int>(t - s * np), i = p % n;
    out[static_cast<size_t>(order[s]) * np + p] = static_cast<T>(acc[s * np + i * n * n + p / n]);
  }
}
template <class T>
int launch_gradient_order(const double* acc, const int* order, T* out, int ngll, int nspec, void* stream) {
  const long long total = static_cast<long long>(nspec) * ngll * ngll * ngll;
  gradient_order_kernel<T><<<stream_grid(total), 256, 0, static_cast<cudaStream_t>(stream)>>>(acc, order, out, ngll, total);
  return static_cast<int>(cudaGetLastError());
}
template int launch_gradient_order<float>(const double*, const int*, float*, int, int, void*);
template int launch_gradient_order<double>(const double*, const int*, double*, int, int, void*);

int launch_adjoint_update(float* F, const float* G_dev, const int* rnode, const int* roff, const int* rlist,
                          int nnodes, const float* lam, float* lam_old, const float* minv, int nglob, double dt,
                          void* stream, const DevCtl* idx, int back) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (G_dev && nnodes > 0) {
    adjoint_inject_kernel<<<(nnodes + 127) / 128, 128, 0, s>>>(F, G_dev, rnode, roff, rlist, nnodes,
                                                             static_cast<float>(1.0 / (dt * dt)), idx, back);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return static_cast<int>(e);
  }
  adjoint_leapfrog_kernel<<<stream_grid(nglob), 256, 0, s>>>(
      reinterpret_cast<const float4*>(lam), reinterpret_cast<float4*>(lam_old), reinterpret_cast<const float4*>(F),
      minv, nglob, static_cast<float>(dt * dt));
  return static_cast<int>(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------
// Material (Sec. II-B: isotropic moduli; Sec. I: the diagonal mass M_I = sum rho J w w w
// over the local points that share node I). One thread per local point of a record slot.
// ---------------------------------------------------------------------------------------
__device__ inline void point_moduli(const MaterialLaunch& m, size_t q, double* rho, double* kappa, double* mu,
                                    double* vp) {
  const double rh = m.rho[q], a = m.p1[q], b = m.p2[q];
  *rho = rh;
  if (m.moduli) {
    *kappa = a;
    *mu = b;
    *vp = sqrt((a + 4.0 * b / 3.0) / rh);
  } else {
    *mu = rh * b * b;
    *kappa = rh * (a * a - 2.0 * b * b) + 2.0 * *mu / 3.0;
    *vp = a;
  }
}

__global__ void material_check_kernel(MaterialLaunch m, unsigned long long* first_bad) {
  const long long n = static_cast<long long>(m.nspec) * m.ngll * m.ngll * m.ngll;
  for (long long q = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; q < n;
       q += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float rh = m.rho[q], a = m.p1[q], b = m.p2[q];
    const bool finite = isfinite(rh) && isfinite(a) && isfinite(b);
    const bool ok = finite && (m.moduli ? (rh > 0.f && b >= 0.f && a > 0.f) : (rh > 0.f && b >= 0.f && a > b));
    if (!ok) atomicMin(first_bad, static_cast<unsigned long long>(q));
  }
}

__global__ void material_records_kernel(MaterialLaunch m) {
  const int n = m.ngll, np = n * n * n;
  const long long total = static_cast<long long>(m.nspec) * np;
  const size_t RW = (static_cast<size_t>(kRecFields) * np + 3) / 4 * 4;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < total;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long s = t / np;
    const int p = static_cast<int>(t - s * np);
    const int i = p % n, j = (p / n) % n, k = p / (n * n);
    const size_t q = static_cast<size_t>(m.order[s]) * np + p;
    double rh, kappa, mu, vp;
    point_moduli(m, q, &rh, &kappa, &mu, &vp);
    float* r = m.rec + s * RW;
    const int qq = i * n * n + j + n * k;
    const double J = r[kJac * np + qq];
    r[rec_at(np, 9, qq)] = static_cast<float>(J * kappa);
    r[rec_at(np, 10, qq)] = static_cast<float>(J * mu);
  }
}

__global__ void mass_color_kernel(MaterialLaunch m, int e0, int e1, double* mass) {
  const int n = m.ngll, np = n * n * n;
  const long long total = static_cast<long long>(e1 - e0) * np;
  const size_t RW = (static_cast<size_t>(kRecFields) * np + 3) / 4 * 4;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < total;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long it = t / np;
    const long long s = m.elist[e0 + it];  // record slot
    const int p = static_cast<int>(t - it * np);
    const int i = p % n, j = (p / n) % n, k = p / (n * n);
    const float* r = m.rec + s * RW;
    const uint32_t g = __float_as_uint(r[kIbool * np + p]) & kNodeMask;
    const double J = r[kJac * np + i * n * n + j + n * k];
    const double rh = m.rho[static_cast<size_t>(m.order[s]) * np + p];
    mass[g] += rh * J * m.w[i] * m.w[j] * m.w[k];  // elements of one colour share no node
  }
}

__global__ void inverse_mass_kernel(const double* __restrict__ mass, float* __restrict__ minv, int nglob) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < nglob; g += gridDim.x * blockDim.x)
    minv[g] = static_cast<float>(1.0 / mass[g]);
}

// One warp per element, its lanes over the points (a thread per element read its points one
// after another: 265 us for 8000 elements at NGLL 5).
__global__ void vpmax_kernel(MaterialLaunch m, double* vpmax) {
  const int np = m.ngll * m.ngll * m.ngll, lane = threadIdx.x & 31;
  const int warps = gridDim.x * (blockDim.x >> 5);
  for (int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); e < m.nspec; e += warps) {
    double best = 0.0;
    for (int p = lane; p < np; p += 32) {
      double rh, kappa, mu, vp;
      point_moduli(m, static_cast<size_t>(e) * np + p, &rh, &kappa, &mu, &vp);
      best = fmax(best, vp);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) best = fmax(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
    if (lane == 0) vpmax[e] = best;
  }
}

int launch_material_check(const MaterialLaunch& m, unsigned long long* first_bad, void* stream) {
  const long long n = static_cast<long long>(m.nspec) * m.ngll * m.ngll * m.ngll;
  material_check_kernel<<<stream_grid(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(m, first_bad);
  return static_cast<int>(cudaGetLastError());
}

int launch_material_apply(const MaterialLaunch& m, const int* sweep_off, int nranges, double* mass, float* minv,
                          double* vpmax, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int np = m.ngll * m.ngll * m.ngll;
  material_records_kernel<<<stream_grid(static_cast<long long>(m.nspec) * np), 256, 0, s>>>(m);
  cudaError_t e = cudaMemsetAsync(mass, 0, static_cast<size_t>(m.nglob) * sizeof(double), s);
  if (e != cudaSuccess) return static_cast<int>(e);
  for (int c = 0; c < nranges; ++c) {  // each range holds elements of one colour
    const int e0 = sweep_off[c], e1 = sweep_off[c + 1];
    if (e1 > e0) mass_color_kernel<<<stream_grid(static_cast<long long>(e1 - e0) * np), 256, 0, s>>>(m, e0, e1, mass);
  }
  inverse_mass_kernel<<<stream_grid(m.nglob), 256, 0, s>>>(mass, minv, m.nglob);
  vpmax_kernel<<<stream_grid(32ll * m.nspec), 256, 0, s>>>(m, vpmax);
  return static_cast<int>(cudaGetLastError());
}

// Layout changes between the solver's fields (internal node order) and the caller's arrays [shots][nglob][3] (caller node order through perm, or internal order when
// perm is null): state copies, displacement snapshots. One thread per (node, shot).
// Node and shot of slot t of the calling block's shot (pair); false for the slot past an odd
// last shot.
__device__ __forceinline__ bool slot_of(long long t, int shots, long long* node, long long* shot) {
  *node = shots > 1 ? t >> 1 : t;
  *shot = shots > 1 ? 2 * block_pair() + (t & 1) : 0;
  return *shot < shots;
}

__device__ __forceinline__ void pack_slots(const float4* __restrict__ u, float* __restrict__ out,
                                           const int* __restrict__ perm, long long nglob, int shots) {
  const long long n = nglob * (shots > 1 ? 2 : 1);
  u += block_pair() * n;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    long long g, sh;
    if (!slot_of(t, shots, &g, &sh)) continue;
    const float4 v = u[t];
    float* o = out + 3 * (sh * nglob + (perm ? perm[g] : g));
    o[0] = v.x;
    o[1] = v.y;
    o[2] = v.z;
  }
}

__global__ void pack_kernel(const float4* __restrict__ u, float* __restrict__ out, const int* __restrict__ perm,
                            long long nglob, int shots) {
  pack_slots(u, out, perm, nglob, shots);
}

__global__ void unpack_kernel(const float* __restrict__ in, float4* __restrict__ u, const int* __restrict__ perm,
                              long long nglob, int shots) {
  const long long n = nglob * (shots > 1 ? 2 : 1);
  u += block_pair() * n;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    long long g, sh;
    if (!slot_of(t, shots, &g, &sh)) continue;
    const float* i = in + 3 * (sh * nglob + (perm ? perm[g] : g));
    u[t] = make_float4(i[0], i[1], i[2], 0.f);
  }
}

int launch_pack(const float* u, float* out, const int* perm, int nglob, int shots, void* stream) {
  if (nglob <= 0) return 0;
  pack_kernel<<<pair_grid(nglob, shots), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<const float4*>(u), out, perm, nglob, shots);
  return static_cast<int>(cudaGetLastError());
}

int launch_unpack(const float* in, float* u, const int* perm, int nglob, int shots, void* stream) {
  if (nglob <= 0) return 0;
  unpack_kernel<<<pair_grid(nglob, shots), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      in, reinterpret_cast<float4*>(u), perm, nglob, shots);
  return static_cast<int>(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------
// Sources and receivers (Sec. V-C): Ricker point forces added to a_raw at t_{n+1} (the first
// block), then the displacement u^{n+1} sampled at the receiver nodes, one thread per receiver
// and shot; n is the device step counter plus the steps enqueued since it was written. Source
// nodes are distinct (the host merges duplicates), so the adds do not race.
// ---------------------------------------------------------------------------------------
__global__ void sources_record_kernel(float* __restrict__ a, const float4* __restrict__ u,
                                      const DevCtl* __restrict__ ctl, int ahead, int nglob, int shots, int nsrc,
                                      const int* __restrict__ src_node, const int* __restrict__ src_shot,
                                      const double* __restrict__ src_force, double f0, double t0, double dt, int nrec,
                                      const int* __restrict__ rec_node) {
  if (blockIdx.x == 0 && nsrc > 0) {
    const double tau = static_cast<double>(ctl->step + ahead + 1) * dt - t0;
    const double x = M_PI * f0 * tau;
    const double aa = x * x;
    const double R = (1.0 - 2.0 * aa) * exp(-aa);
    for (int s = threadIdx.x; s < nsrc; s += blockDim.x) {
      const size_t g = kNodeStride * field_slot(nglob, shots, src_node[s], src_shot[s]);
      a[g] += static_cast<float>(src_force[3 * s] * R);
      a[g + 1] += static_cast<float>(src_force[3 * s + 1] * R);
      a[g + 2] += static_cast<float>(src_force[3 * s + 2] * R);
    }
  }
  const int col = ctl->col + ahead, ncols = ctl->ncols;
  float* seis = ctl->seis;
  if (seis == nullptr || col >= ncols) return;  // seis [shots][nrec][3][ncols]
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nrec * shots; q += gridDim.x * blockDim.x) {
    const int r = q / shots, sh = q - r * shots;
    const float4 x = u[field_slot(nglob, shots, rec_node[r], sh)];
    float* o = seis + (static_cast<size_t>(sh) * nrec + r) * 3 * ncols + col;
    o[0] = x.x;
    o[ncols] = x.y;
    o[2 * static_cast<size_t>(ncols)] = x.z;
  }
}

// pack_kernel into the snapshot slot the step counter names (graph-replayable)
__global__ void snapshot_kernel(const float4* __restrict__ u, const DevCtl* __restrict__ ctl, int ahead,
                                const int* __restrict__ perm, long long nglob, int shots) {
  float* base = ctl->snap;
  if (!base) return;
  pack_slots(u, base + static_cast<long long>(ctl->col + ahead) * ctl->snap_per, perm, nglob, shots);
}

int launch_snapshot(const float* u, const DevCtl* ctl, int ahead, const int* perm, int nglob, int shots, void* stream) {
  if (nglob <= 0) return 0;
  snapshot_kernel<<<pair_grid(nglob, shots), 256, 0, static_cast<cudaStream_t>(stream)>>>(reinterpret_cast<const float4*>(u),
                                                                                 ctl, ahead, perm, nglob, shots);
  return static_cast<int>(cudaGetLastError());
}

__global__ void set_ctl_kernel(DevCtl* ctl, long long step, int ncols, float* seis, float* snap, long long snap_per) {
  ctl->step = step;
  ctl->col = 0;
  ctl->ncols = ncols;
  ctl->seis = seis;
  ctl->err = 0;
  ctl->snap = snap;
  ctl->snap_per = snap_per;
}

__global__ void advance_ctl_kernel(DevCtl* ctl, int steps) {
  ctl->step += steps;
  ctl->col += steps;
}

int launch_advance_ctl(DevCtl* ctl, int steps, void* stream) {
  advance_ctl_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ctl, steps);
  return static_cast<int>(cudaGetLastError());
}

int launch_set_ctl(DevCtl* ctl, long long step, int ncols, float* seis, void* stream, float* snap,
                   long long snap_per) {
  set_ctl_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ctl, step, ncols, seis, snap, snap_per);
  return static_cast<int>(cudaGetLastError());
}

int launch_sources_record(const DevProblem& p, int ahead, void* stream) {
  const long long n = static_cast<long long>(p.nrec) * p.shots;
  const int grid = static_cast<int>(n < 256 ? 1 : (n + 255) / 256 > 608 ? 608 : (n + 255) / 256);
  sources_record_kernel<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      p.a, reinterpret_cast<const float4*>(p.u), p.ctl, ahead, p.nglob, p.shots, p.nsrc, p.src_node, p.src_shot, p.src_force,
      p.f0, p.t0, p.dt, p.nrec, p.rec_node);
  return static_cast<int>(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------
// Divergence watchdog: flags any non-finite value of u, v or a ([nglob][kNodeStride]).
// Threads that find one write 1 into the flag word; the host clears it first.
// ---------------------------------------------------------------------------------------
__global__ void nonfinite_kernel(const float4* __restrict__ u, const float4* __restrict__ v,
                                 const float4* __restrict__ a, long long n, int* flag) {
  bool bad = false;
  for (long long t = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; t < n;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float4 x = u[t], y = v[t], z = a[t];
    bad |= !(isfinite(x.x) && isfinite(x.y) && isfinite(x.z) && isfinite(x.w));
    bad |= !(isfinite(y.x) && isfinite(y.y) && isfinite(y.z) && isfinite(y.w));
    bad |= !(isfinite(z.x) && isfinite(z.y) && isfinite(z.z) && isfinite(z.w));
  }
  if (bad) *flag = 1;
}

int launch_nonfinite_check(const DevProblem& p, int* flag, void* stream) {
  const long long n = static_cast<long long>(p.nglob) * padded_shots(p.shots);
  nonfinite_kernel<<<kEnergyBlocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<const float4*>(p.u), reinterpret_cast<const float4*>(p.v),
      reinterpret_cast<const float4*>(p.a), n, flag);
  return static_cast<int>(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------
// Energy partial sums: per block, sum_I |v_I|^2 / minv_I and sum_I u_I . f_I in float64.
// ---------------------------------------------------------------------------------------
__global__ void energy_partials_kernel(const float4* __restrict__ u, const float4* __restrict__ v,
                                       const float4* __restrict__ f, const float* __restrict__ minv, int nglob,
                                       int shots, double* __restrict__ partials) {
  __shared__ double sk[256], sp[256];
  double kin = 0.0, pot = 0.0;
  const long long n = static_cast<long long>(nglob) * padded_shots(shots);
  for (long long g = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; g < n;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const float m = minv[shots == 1 ? g : (g >> 1) % nglob];
    const float4 vg = v[g], ug = u[g], fg = f[g];
    const double vx = vg.x, vy = vg.y, vz = vg.z;
    kin += (vx * vx + vy * vy + vz * vz) / static_cast<double>(m);
    pot += static_cast<double>(ug.x) * fg.x + static_cast<double>(ug.y) * fg.y + static_cast<double>(ug.z) * fg.z;
  }
  sk[threadIdx.x] = kin;
  sp[threadIdx.x] = pot;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sk[threadIdx.x] += sk[threadIdx.x + w];
      sp[threadIdx.x] += sp[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = sk[0];
    partials[2 * blockIdx.x + 1] = sp[0];
  }
}

int launch_energy_partials(const float* u, const float* v, const float* f, const float* minv, int nglob,
                           int shots, double* partials, int nblocks, void* stream) {
  energy_partials_kernel<<<nblocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<const float4*>(u), reinterpret_cast<const float4*>(v), reinterpret_cast<const float4*>(f),
      minv, nglob, shots, partials);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace semgb
