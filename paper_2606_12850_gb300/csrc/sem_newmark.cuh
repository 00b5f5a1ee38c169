// What happens at a node whose force is complete (Sec. I, V-C): point sources, the explicit
// Newmark update, the adjoint leapfrog, displacement snapshots. Shared by the patch sweep
// (inner nodes, sem_forces.cuh) and the rim pass (sem_kernels.cu), so both run the same float
// operations in the same order.
#pragma once
#include <cuda_runtime.h>

#include "sem_internal.h"

namespace semgb {
namespace {

// Programmatic dependent launch (the kernels of a step overlap): a kernel's CTAs may be
// scheduled while the previous launch drains, and wait for it to complete, with its memory
// visible, before they read any wavefield. Both instructions are no-ops for a kernel launched
// without the programmatic attribute.
__device__ __forceinline__ void wait_prerequisite_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_dependent_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A wavefield the previous launch may have written is read only after that wait and never through
// the read-only path (__ldg), which is for data no one writes while the kernel runs, its start
// before the wait included: float4 nodes by __ldcg in the patch kernels, by plain loads (volatile,
// so that they stay behind the wait) in the element kernel; so too the nodes of caller arrays
// [nglob][3], whose three words share L1 lines (f = -K u on 44 x 36 x 40 elements at NGLL 5: 167
// us, with __ldcg 180).
__device__ __forceinline__ float4 load_node4(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 load_node3(const float* p) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v.x) : "l"(p) : "memory");
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v.y) : "l"(p + 1) : "memory");
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v.z) : "l"(p + 2) : "memory");
  return v;
}

// Index of a node's 16-byte slot in its shot's part of a field (see field_slot).
template <bool MS>
__device__ __forceinline__ size_t node_slot(uint32_t w) {
  return static_cast<size_t>(w & kNodeMask) * (MS ? 2 : 1);
}
// The update's fields, moved to the slots of a shot that start at `slot` (MS).
__device__ __forceinline__ void move_fields(SweepNewmark& nm, size_t slot) {
  nm.u += 4 * slot;
  nm.v += 4 * slot;
  nm.a += 4 * slot;
}

// The point sources src[0 .. nsrc) at a node: the Ricker wavelet at t_{n+1} times each force,
// added to the node's complete force in the order the entries are listed.
__device__ __forceinline__ void add_point_sources(const PatchSrc* __restrict__ src, int nsrc, const SweepNewmark& nm,
                                                  uint32_t node, int shot, float& fx, float& fy, float& fz) {
  for (int i = 0; i < nsrc; ++i) {
    const PatchSrc& s = src[i];
    if (s.node != static_cast<int>(node) || s.shot != shot) continue;
    const long long n = __ldcg(&nm.ctl->step) + nm.ahead + 1;
    const double tau = static_cast<double>(n) * nm.dtd - nm.t0;
    const double x = M_PI * nm.f0 * tau;
    const double aa = x * x;
    const double R = (1.0 - 2.0 * aa) * exp(-aa);
    fx += static_cast<float>(s.f[0] * R);
    fy += static_cast<float>(s.f[1] * R);
    fz += static_cast<float>(s.f[2] * R);
  }
}

// The inputs of a node's update: 1/M, and for Newmark the half-step velocity and (mode 1, or
// a snapshot) the displacement, for the adjoint lam^m and lam^{m+1}.
struct NodeState {
  float m;
  float4 v, u;
};
// NM: 1 Newmark (mode 1 or 2), 3 Newmark with a snapshot, 2 the adjoint leapfrog.
template <bool MS, int NM>
__device__ __forceinline__ void load_node_state(const SweepNewmark& nm, uint32_t w, NodeState& st) {
  const size_t g = node_slot<MS>(w);
  st.m = __ldg(nm.minv + (w & kNodeMask));
  st.v = __ldcg(reinterpret_cast<const float4*>(NM == 2 ? nm.lam_old : nm.v) + g);
  if (NM != 1 || nm.mode == 1) st.u = __ldcg(reinterpret_cast<const float4*>(nm.u) + g);
}

// Newmark update of a node whose complete force (fx, fy, fz) is known (mode 1 or 2):
//   a = M^-1 f ; v = v_half + dt/2 a ; mode 1: u <- u + dt v + dt^2/2 a, v_half <- v + dt/2 a ;
//   mode 2: v and a stored.
template <bool MS>
__device__ __forceinline__ void newmark_node(const SweepNewmark& nm, uint32_t w, const NodeState& st, float fx,
                                             float fy, float fz) {
  const size_t g = node_slot<MS>(w);
  const float ax = fx * st.m, ay = fy * st.m, az = fz * st.m;
  const float vx = st.v.x + nm.hdt * ax, vy = st.v.y + nm.hdt * ay, vz = st.v.z + nm.hdt * az;
  if (nm.mode == 1) {
    reinterpret_cast<float4*>(nm.u)[g] = make_float4((st.u.x + nm.dt * vx) + nm.hdt2 * ax,
                                                     (st.u.y + nm.dt * vy) + nm.hdt2 * ay,
                                                     (st.u.z + nm.dt * vz) + nm.hdt2 * az, 0.f);
    reinterpret_cast<float4*>(nm.v)[g] = make_float4(vx + nm.hdt * ax, vy + nm.hdt * ay, vz + nm.hdt * az, 0.f);
  } else {
    reinterpret_cast<float4*>(nm.v)[g] = make_float4(vx, vy, vz, 0.f);
    reinterpret_cast<float4*>(nm.a)[g] = make_float4(ax, ay, az, 0.f);
  }
}

// The snapshot of the node's displacement u^{n+1} (a Newmark sweep of a snapshot run).
__device__ __forceinline__ void snapshot_node(const SweepNewmark& nm, uint32_t w, const NodeState& st) {
  const DevCtl* ctl = nm.ctl;
  const uint32_t g = w & kNodeMask;
  float* o = ctl->snap + static_cast<long long>(ctl->col + nm.ahead) * ctl->snap_per +
             3 * static_cast<size_t>(nm.snap_perm ? __ldg(nm.snap_perm + g) : static_cast<int>(g));
  o[0] = st.u.x;
  o[1] = st.u.y;
  o[2] = st.u.z;
}

// The residuals of the step at the receivers recv[0 .. nrec) of a node, added to its force
// f = -K lam in ascending receiver order (G / dt^2).
__device__ __forceinline__ void adjoint_receivers(const SweepNewmark& nm, const PatchRecv* __restrict__ recv, int nrec,
                                                  uint32_t node, float& fx, float& fy, float& fz) {
  const float* G = nm.idx ? nm.idx->adj_G + static_cast<long long>(nm.idx->adj_j - nm.back - 1) * nm.idx->adj_gstep : nm.G;
  if (!G) return;
  for (int i = 0; i < nrec; ++i) {
    const PatchRecv e = recv[i];
    if (e.node != static_cast<int>(node)) continue;
    fx += G[3 * e.r] * nm.inv_dt2;
    fy += G[3 * e.r + 1] * nm.inv_dt2;
    fz += G[3 * e.r + 2] * nm.inv_dt2;
  }
}
// lam_old <- 2 lam - lam_old + dt^2 M^-1 f
__device__ __forceinline__ void adjoint_node(const SweepNewmark& nm, uint32_t w, const NodeState& st, float fx,
                                             float fy, float fz) {
  const size_t g = w & kNodeMask;
  const float s = nm.dt2 * st.m;
  const float4 l = st.u, o = st.v;
  reinterpret_cast<float4*>(nm.lam_old)[g] =
      make_float4(2.f * l.x - o.x + s * fx, 2.f * l.y - o.y + s * fy, 2.f * l.z - o.z + s * fz, 0.f);
}

// The complete force (fx, fy, fz) of a node, used: NM 0 stored in f, 4 stored in a caller array
// [nglob][3], 1 / 3 the sources and the Newmark update (3: and the snapshot), 2 the residuals
// and the leapfrog.
template <bool MS, int NM>
__device__ __forceinline__ void complete_node(const SweepNewmark& nm, float4* __restrict__ f, uint32_t w, int shot,
                                              const NodeState& st, const PatchSrc* __restrict__ src,
                                              int nsrc, const PatchRecv* __restrict__ recv, int nrec, float fx,
                                              float fy, float fz) {
  if constexpr (NM == 0) {
    f[node_slot<MS>(w)] = make_float4(fx, fy, fz, 0.f);
  } else if constexpr (NM == 4) {
    float* o = reinterpret_cast<float*>(f) + 3 * static_cast<size_t>(__ldg(nm.perm + (w & kNodeMask)));
    o[0] = fx;
    o[1] = fy;
    o[2] = fz;
  } else if constexpr (NM == 2) {
    if (nrec) adjoint_receivers(nm, recv, nrec, w & kNodeMask, fx, fy, fz);
    adjoint_node(nm, w, st, fx, fy, fz);
  } else {
    if constexpr (NM == 3) snapshot_node(nm, w, st);
    if (nsrc) add_point_sources(src, nsrc, nm, w & kNodeMask, shot, fx, fy, fz);
    newmark_node<MS>(nm, w, st, fx, fy, fz);
  }
}

}  // namespace
}  // namespace semgb
