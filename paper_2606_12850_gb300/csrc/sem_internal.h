// Internal declarations shared by the host set-up (sem_setup.cpp), the C ABI
// (sem_capi.cpp) and the CUDA kernels (sem_kernels.cu) of libsemgb.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

struct sem_ctx;

namespace semgb {

using sem_ctx_fwd = ::sem_ctx;

#ifdef __CUDACC__
#define SEM_HD __host__ __device__
#else
#define SEM_HD
#endif

constexpr int kMaxNgll = 10;
constexpr int kMinNgll = 2;

// Element record: per local point nine inverse-Jacobian terms dxi_r/dx_d (r-major: xix xiy xiz
// etax etay etaz gammax gammay gammaz), J kappa, J mu, the ibool word and J. Laid out for wide
// loads, the points of a field group in rec_pos order: [np][4] G0..G3, [np][4] G4..G7, [np][2]
// G8 and J kappa, [np] J mu, then [np] ibool words (natural point order) and [np] J, so the
// eleven values a force kernel needs at a point are two 16-byte, one 8-byte and one 4-byte load
// (eleven 4-byte loads of 500-byte fields, which straddle 128-byte lines, measured 1.8 L1
// wavefronts each at NGLL 5). The force kernels read the first kForceFields words per point
// (J sigma from J kappa and J mu needs no separate J); J serves the mass and the sensitivities.
constexpr int kRecFields = 13;
constexpr int kForceFields = 12;
constexpr int kIbool = 11, kJac = 12;  // words per point before the ibool words and before J
// Word of inverse-Jacobian term c (0 .. 8), J kappa (9) or J mu (10) at point position q.
SEM_HD constexpr int rec_at(int np, int c, int q) {
  return c < 4 ? 4 * q + c : c < 8 ? 4 * np + 4 * q + c - 4 : c < 10 ? 8 * np + 2 * q + c - 8 : 10 * np + q;
}

// The context's own wavefields u, v, a are float32 [nglob][kNodeStride]: x, y, z and a zero
// pad, so that every node is one aligned 16-byte access in the gather, the scatter and the
// Newmark passes. Caller-facing arrays stay [nglob][3]; copies at the boundary are strided.
constexpr int kNodeStride = 4;
// With several shots a field is [ceil(shots / 2)][nglob][2][kNodeStride]: the shots in pairs, a
// pair's two slots one 32-byte sector, the nodes of a pair as for a single shot. The gather of
// a shot pair reads a row of nodes as one run (with the shots of a node together, 512 bytes
// apart at 32 shots, every node was an L1 wavefront of its own). An odd last shot leaves a slot
// that stays zero.
SEM_HD constexpr int padded_shots(int shots) { return shots > 1 ? (shots + 1) / 2 * 2 : 1; }
SEM_HD inline size_t field_slot(size_t nglob, int shots, size_t node, int shot) {
  return shots > 1 ? (static_cast<size_t>(shot >> 1) * nglob + node) * 2 + (shot & 1) : node;
}

// Bit 31 of a record's ibool word marks the first contribution to that node in the
// colour-by-colour processing order: the force kernel stores instead of adding there,
// so the assembled array needs no zeroing pass.
constexpr uint32_t kFirstTouchBit = 0x80000000u;
// Bit 30 marks the same for the patch kernel's order (patch colour by patch colour), on the
// word of the first local point (in patch-table order) of each patch node. Bit 29 marks a
// local point that is the only one of its patch at its node (its element's team writes it
// alone). All three serve the forms that write nodes in place (element kernel, persistent
// sweeps). Node ids are below 2^28.
constexpr uint32_t kPatchFirstBit = 0x40000000u;
constexpr uint32_t kAloneBit = 0x20000000u;
constexpr uint32_t kNodeMask = 0x0FFFFFFFu;
constexpr int kMaxNodes = 1 << 28;

inline int rec_words(int ngll) {
  const int np = ngll * ngll * ngll;
  return (kRecFields * np + 3) / 4 * 4;  // 16-byte aligned element records
}

// Position of local point (i, j, k) inside a geometry or material field of an element
// record: points are stored i-major so that the NGLL^2 threads owning the xi-lines (j, k)
// of an element read consecutive words for a fixed i. The ibool field keeps the natural
// order p = i + NGLL*j + NGLL^2*k, which the gather and scatter threads walk.
inline int rec_pos(int ngll, int i, int j, int k) { return i * ngll * ngll + j + ngll * k; }

// ---- host set-up (sem_setup.cpp) -------------------------------------------------------
int gll_basis(int ngll, double* xi, double* w, double* hprime, std::string* err);

// Positions, inverse Jacobian and determinant at every GLL point of one trilinear element;
// xyz[np][3], G[np][9] (dxi_r/dx_d at 3r+d), J[np]; returns false if some J <= 0.
bool element_geometry(int ngll, const double* xi, const double* hprime, const double* ctrl,
                      double* xyz, double* G, double* J);
// The same from the positions xyz[np][3] of the element's GLL points (any geometry).
bool geometry_from_positions(int ngll, const double* hprime, const double* xyz, double* G, double* J);

int color_elements(int nspec, int ngll, int nglob, const int32_t* ibool,
                   std::vector<int32_t>* color, int* ncolors, std::string* err);

int locate_nodes(int nglob, const double* node_xyz, int npts, const double* xyz,
                 const double* surface_z, int32_t* out);

// Patches for the force sweep (sem_patches.cpp): bricks of bx x by x bz elements of the
// mesh's lattice coordinates, coloured so that no two patches of a colour share a node.
struct PatchShape {
  int bx = 1, by = 1, bz = 1;
};
struct PatchPlan {
  int ngll = 0;
  int npatch = 0;
  int ncolors = 0;
  int max_nodes = 0;              // largest patch node count
  int max_elems = 0;              // largest patch element count
  std::vector<int> elem;          // caller elements in sweep order, patch after patch
  std::vector<int> patch_off;     // [npatch + 1] into elem (sweep order)
  std::vector<int> color_off;     // [ncolors + 1] patch ranges of the sweep order
  std::vector<int> node_off;      // [npatch + 1] into nodes
  std::vector<uint32_t> nodes;    // patch node lists: caller node | kFirstTouchBit
  std::vector<int> table_of;      // per patch: its table
  std::vector<int> tab_nelem, tab_nnode, tab_nshared, tab_lid_off, tab_csr_off, tab_excl_off, tab_first_off;
  std::vector<uint16_t> lid;      // per table: [nelem][np] patch-local node of each local point
  std::vector<int> node_new;      // [nglob] internal id of every caller node
  int ninner = 0;                 // internal ids below this: nodes of one patch only
  std::vector<uint16_t> csr;      // per table: per shared patch node (one met by several local
                                  // points) kPatchSlots slots holding those local points
                                  // (le*np + p, ascending)
  std::vector<uint32_t> excl;     // per table: bit le*np + p set when that local point is the
                                  // only one at its patch node
  std::vector<uint16_t> first_q;  // per table: per patch node, its first local point
};
// Contribution slots per patch node: 8 (the elements meeting at a vertex of a structured
// hexahedral mesh), read as one 16-byte word. An unused slot holds kPatchNoSlot; a node met
// by more local points continues in another group of slots, named by its last slot as
// kPatchChain | group.
constexpr int kPatchSlots = 8;
constexpr uint16_t kPatchNoSlot = 0xFFFFu;
constexpr uint16_t kPatchChain = 0x8000u;
int build_patches(int nspec, int ngll, int nglob, const int32_t* ibool, const PatchShape& shape, PatchPlan* plan,
                  std::string* err);

// ---- device side (sem_kernels.cu) ------------------------------------------------------
struct DevCtl {
  long long step;  // steps taken since the state was set
  int col;         // next seismogram column
  int ncols;       // columns in the seismogram buffer (0: no recording)
  float* seis;     // [nrec][3][ncols] or null
  int err;
  int pad;
  float* snap;          // displacement snapshots [col][shots][nglob][3], or null
  long long snap_per;   // floats per snapshot
  // adjoint steps replayed from a graph: step j reads residual adj_G + (j - 1) adj_gstep and
  // snapshots adj_u + (j - 1 .. j + 1) adj_n3; j counts down
  const float* adj_G;
  const float* adj_u;
  long long adj_n3;
  int adj_gstep;
  int adj_j;   // the step the captured steps begin at (they count back from it)
};

struct DevProblem {
  int ngll;
  int nspec;
  int nglob;
  int shots;  // wavefields are (fields, kNodeStride)
  const float* rec;
  float* u;
  float* v;
  float* a;
  const float* minv;
  DevCtl* ctl;
  int nsrc;
  const int* src_node;   // per source: global node
  const int* src_shot;   // per source: shot it acts in
  const double* src_force;
  double f0, t0;
  int nrec;
  const int* rec_node;
  double dt;
};

// Copies hprime, hprime*w and w for this ngll into the kernels' constant banks.
int upload_basis(int ngll, const double* w, const double* hprime, void* stream);

// One colour's worth of elements [e0, e1) of the colour-sorted order: f (=|+=) -K u; a node
// is stored at its first touch in colour order and accumulated afterwards.
struct ForceLaunch {
  const float* rec;
  const int* elist;  // record slots in colour order; e0, e1 index this list
  const int* perm;   // internal -> caller node (caller arrays, node_stride 3)
  const float* u;
  float* f;
  int e0, e1;
  int node_stride;  // floats per node in u and f: kNodeStride (internal order), or 3 for caller
                    // arrays in caller order
  int shots;        // > 1: u and f are fields of several shots, items (element, shot)
  int nglob;
  int variant;      // contraction form: 0 the order's default, 1 line owners, 2 per point
  int atomic;       // colouring ablation: float atomic adds into a zeroed f, any element order
};
int launch_forces(int ngll, const ForceLaunch& launch, void* stream);

// A patch of the sweep. Its nodes are inner (of this patch only) or rim (shared with other
// patches); the sweep completes the inner ones and leaves one partial force sum per rim node
// in the partials buffer, which the rim pass (launch_rim_combine) sums per node.
struct alignas(16) PatchDesc {
  int slot0;     // record slot of the patch's first element (its elements are consecutive)
  int nelem;
  int nshared;   // patch nodes met by several of its local points
  int slot_off;  // its table: per shared node, kPatchSlots slots (shared-memory offsets of the
                 // forces of the local points meeting there)
  int word_off;  // its table: per shared node, the shared-memory offset of its first local
                 // point's ibool word
  int src_off;   // its point sources (PatchSrc entries [src_off, src_off + nsrc)): the ones at
  int nsrc;      // its inner nodes, added there to the complete force
  int inner0;    // its inner nodes: ids inner0 .. + nalone (one local point each, the shared-
  int nalone;    // memory offsets of their forces at alone_off), then nin met by several
  int alone_off; // (slot groups from in_slots on)
  int nin;
  int in_slots;
  int nrim;      // rim nodes, ascending internal id
  int rim_slots; // their slot groups (index of the first)
  int rim0;      // partial of rim node k: field_slot(partials a shot, shots, rim0 + k, shot)
  int rec_off;   // its receivers (PatchRecv entries [rec_off, rec_off + nrec)): the ones at its
  int nrec;      // inner nodes, then at rim nodes it touches last
  int nrec_in;   // how many of them are at inner nodes
  int pad[2];
};
static_assert(sizeof(PatchDesc) == 80, "PatchDesc is five 16-byte words");
// A receiver in the sweep: internal node, receiver index (residual G[3 r + c]).
struct PatchRecv {
  int node;
  int r;
};
struct DevCtl;
// A point source in the patch sweep: internal node, shot, force vector (Sec. V-C).
struct PatchSrc {
  int node;
  int shot;
  double f[3];
};
// The point sources and receivers at kRimBlock consecutive rim nodes (by block of rim nodes).
constexpr int kRimBlock = 256;
struct alignas(16) RimBlock {
  int src_off, nsrc;
  int rec_off, nrec;
};
// The partials that meet at a rim node, in sweep order of their patches: up to four indices
// (-1: none); with more, w = -2 - o names the list over[o] = count, over[o + 1 ..] = indices.
struct alignas(16) RimNode {
  int x, y, z, w;
};
// The explicit Newmark update (Sec. I) run by the sweep at every node whose force is complete:
// mode 1 corrector of step n fused with the predictor of step n+1
//   a = M^-1 f ; v = v_half + dt/2 a ; u <- u + dt v + dt^2/2 a ; v_half <- v + dt/2 a
// (f is then not stored), mode 2 the corrector alone (v <- v_half + dt/2 a, a stored), mode 0
// none (f stored), mode 4 none (f stored into a caller array [nglob][3] through perm). The
// point sources of the step, at t = (ctl->step + ahead + 1) dt, are added to f first.
struct SweepNewmark {
  int mode;           // 3: the adjoint leapfrog (u = lam^m; lam_old: lam^{m+1} in, lam^{m-1} out)
  int nglob, nsums;   // field and partials strides of a shot pair
  float* u;           // field, written where the force is complete (mode 1)
  float* v;           // field, half-step velocity in, out as above
  float* a;           // field, acceleration out (mode 2)
  const float* minv;  // [nglob]
  const PatchSrc* src;
  const PatchSrc* rim_src;  // the sources at rim nodes, by rim block
  const DevCtl* ctl;        // step counter, seismogram and snapshot buffers
  int ahead;                // steps enqueued since the counter was last set or advanced
  double f0, t0, dtd;       // Ricker centre frequency and delay, step (double)
  float dt, hdt, hdt2;
  // the receivers by patch: sampled (u^{n+1}, modes 1 and 2) into ctl->seis column ctl->col +
  // ahead before the patch's nodes are updated; adjoint (mode 3): their residuals G [nrec][3]
  // (or, with idx, those the device's adjoint counter names) added at inner nodes, and by rim
  // block at rim nodes, ascending receiver
  const PatchRecv* recv;
  const PatchRecv* rim_recv;
  int nrec;            // receivers of the model
  // snapshot run (modes 1, 2): u^{n+1} also stored where it is updated into ctl->snap +
  // (ctl->col + ahead) ctl->snap_per, [nglob][3] in the order snap_perm maps to
  int snap;
  const int* snap_perm;
  float* lam_old;
  const float* G;
  const DevCtl* idx;
  int back;   // steps since idx->adj_j was written
  float inv_dt2, dt2;
  const int* perm;  // mode 4: internal -> caller node
};
// Counters of a persistent sweep (all patch colours in one launch): patches taken, CTAs
// that have left, a wait that gave up, patches finished per colour. Zero between sweeps.
constexpr int kMaxSweepColors = 64;
struct SweepSync {
  unsigned int next;
  unsigned int exited;
  int err;
  int pad;
  unsigned int done[kMaxSweepColors];
};
// One persistent sweep over the patches of several models of one order (a group step):
// items are the patches of every model, colour-major (colour 0 of every model, then colour
// 1, ...); a patch of colour c writes once every patch of colour c - 1 of its own model has
// finished. Models and runs of items live in device memory.
constexpr int kMaxGroupModels = 64;
struct GroupModel {
  const float* rec;
  const PatchDesc* desc;
  const uint16_t* slots;
  const uint16_t* words;
  const float* u;        // [nglob][4]
  float* f;              // [nglob][4]
  const int* color_end;  // per colour, the end of its patch range (model-local patches)
  int ncolors;
  int pad;
};
struct GroupSeg {  // a run of consecutive items: patches [p0, p0 + count) of one (model, colour)
  int item0;
  int model;
  int color;
  int p0;
};
struct GroupSync {
  unsigned int next;
  unsigned int exited;
  int err;
  int pad;
  unsigned int done[kMaxGroupModels * kMaxSweepColors];  // [model][colour] finished patches
};
struct GroupLaunch {
  const GroupModel* models;
  const GroupSeg* segs;
  int nseg;
  int nitems;
  int nmodels;
  int variant;       // contraction form as in ForceLaunch
  unsigned int stall;  // a count that never arrives (tests)
  GroupSync* sync;
};
int launch_group_sweep(int ngll, const GroupLaunch& launch, void* stream);

// One patch sweep on (fields, kNodeStride) fields: f = -K u at the inner nodes (or their
// update, nm.mode), partial sums at the rim.
struct PatchLaunch {
  const float* rec;
  const PatchDesc* desc;
  const uint16_t* slots;
  const uint16_t* words;
  SweepSync* sync;        // non-null: one persistent launch over all colours (assembles all of f)
  const int* color_end;   // per colour, the end of its patch range (persistent launch)
  int ncolors;            // (persistent launch)
  int stall;              // (persistent launch) wait for a count that never arrives (tests)
  int npatch;
  const float* u;
  float* f;
  float* partials;  // laid out like a field over the rim partials
  int variant;  // contraction form as in ForceLaunch
  int shots;    // > 1: fields (fields, kNodeStride)
  int pairs;    // with shots > 1: one CTA per (patch, shot pair) (else one per (patch, shot))
  SweepNewmark nm;  // mode 0: forces only
};
int launch_patch_forces(int ngll, const PatchLaunch& launch, void* stream);
// Shared-memory layout of the patch kernels for this order: a local point (i, j, k) of an
// element workspace at float 3 (i + sy j + sz k); floats per element and per team of the sweep
// (es, ts) and of the persistent sweeps, which also keep the ibool words (from float words on;
// esw, tsw); elements per team.
struct PatchLayout {
  int sy, sz, es, ts, esw, tsw, words, e;
};
int patch_layout(int ngll, PatchLayout* out);
// the brick each order's patch kernel is compiled for
// (nspec: the elements of the mesh it is for)
int patch_shape(int ngll, int nspec, PatchShape* out);
int forces_kernel_smem_bytes(int ngll);
int forces_elements_per_cta(int ngll);

// The rim pass after a sweep: per rim node the sum of its partials in sweep order, then what
// the sweep did at the inner nodes (nm.mode).
struct RimLaunch {
  const RimNode* rim;   // [nrim]
  const int* over;
  const RimBlock* blocks;  // [ceil(nrim / kRimBlock)]
  const float* partials;
  float* f;
  int ninner;           // internal id of rim node 0
  int nrim;
  int shots;
  SweepNewmark nm;
};
int launch_rim_combine(const RimLaunch& launch, void* stream);
// step and column of the counter += steps
int launch_advance_ctl(DevCtl* ctl, int steps, void* stream);
int launch_set_ctl(DevCtl* ctl, long long step, int ncols, float* seis, void* stream, float* snap = nullptr,
                   long long snap_per = 0);
// the displacement into snapshot ctl->col + ahead
int launch_snapshot(const float* u, const DevCtl* ctl, int ahead, const int* perm, int nglob, int shots, void* stream);
int launch_predictor(const DevProblem& p, void* stream);
int launch_fused_newmark(const DevProblem& p, void* stream);
int launch_corrector(const DevProblem& p, void* stream);
int launch_sources_record(const DevProblem& p, int ahead, void* stream);
// u_lo, u_mid, u_hi: [nglob][3] in caller order (perm: internal -> caller node) or in
// internal order (perm null); the terms are added to float32 partials g_* [nlocal]
// (idx non-null: the snapshots are idx->adj_u + (j - 1 .. j + 1) idx->adj_n3, j = idx->adj_j - back)
int launch_sensitivity(int ngll, const float* rec, const int* perm, const float* lam, const float* u_lo,
                       const float* u_mid, const float* u_hi, float* g_rho, float* g_kappa, float* g_mu, int nspec,
                       double c_m, double c_k, void* stream, const DevCtl* idx = nullptr, int back = 0);
// fields in internal node order <-> caller layout
// [shots][nglob][3] in caller node order (perm: internal -> caller node)
int launch_pack(const float* u, float* out, const int* perm, int nglob, int shots, void* stream);
int launch_unpack(const float* in, float* u, const int* perm, int nglob, int shots, void* stream);
// rnode[nnodes]: distinct receiver nodes; rlist[roff[t] .. roff[t+1]): their receivers
// (idx non-null: G_dev is taken from idx->adj_G at step idx->adj_j - back; G_dev then only says
// whether there is one)
int launch_adjoint_update(float* F, const float* G_dev, const int* rnode, const int* roff, const int* rlist,
                          int nnodes, const float* lam, float* lam_old, const float* minv, int nglob, double dt,
                          void* stream, const DevCtl* idx = nullptr, int back = 0);
int launch_adjoint_index(DevCtl* ctl, const float* G, const float* u, long long n3, int gstep, int j, void* stream);
int launch_adjoint_next(DevCtl* ctl, int steps, void* stream);  // adj_j -= steps
// the accumulators (record order) in caller order [nspec][ngll^3], rounded to T
template <class T>
int launch_gradient_order(const double* acc, const int* order, T* out, int ngll, int nspec, void* stream);
// acc[t] += part[t] (float64), part[t] = 0, for t < n
int launch_flush_partials(float* part, double* acc, long long n, void* stream);
// Material on the device (Sec. II-B moduli, Sec. I diagonal mass). rho, p1, p2: per local
// point in caller order [nspec][ngll^3]; moduli: (p1, p2) = (kappa, mu), else (vp, vs).
struct MaterialLaunch {
  float* rec;          // colour-sorted element records
  const int* order;    // record slot -> caller element
  const int* elist;    // record slots in element colour order (the ranges below index it)
  const float* rho;
  const float* p1;
  const float* p2;
  int moduli;
  int ngll;
  int nspec;
  int nglob;
  double w[kMaxNgll];  // GLL weights
};
// index of the first local point that breaks rho > 0, mu (vs) >= 0, kappa > 0 (vp > vs) or
// is not finite, as an atomic minimum into *first_bad (caller presets it to ~0ull)
int launch_material_check(const MaterialLaunch& m, unsigned long long* first_bad, void* stream);
// kappa and mu into the records, the mass range by range of the sweep order (one colour per
// range, so no races), 1/mass,
// and the largest vp of every caller element (for the CFL suggestion)
int launch_material_apply(const MaterialLaunch& m, const int* sweep_off, int nranges, double* mass, float* minv,
                          double* vpmax, void* stream);
int launch_nonfinite_check(const DevProblem& p, int* flag, void* stream);
int launch_energy_partials(const float* u, const float* v, const float* f, const float* minv,
                           int nglob, int shots, double* partials, int nblocks, void* stream);
constexpr int kEnergyBlocks = 608;  // 4 CTAs per SM on 152 SMs

// ---- context access for entry points defined outside sem_capi.cpp ----------------------
struct CtxView {
  int device;
  void* stream;
  int nglob;
  const float* minv;     // internal node order
  const int* node_new;   // caller node -> internal node
};
// SEM_OK and the view when the material is set; otherwise an error code (message set).
int ctx_view(sem_ctx_fwd* c, CtxView* out);
int ctx_fail(sem_ctx_fwd* c, int code, const char* message);

}  // namespace semgb
