// Asynchronous concurrent insertion: one persistent launch per wave, no rounds.
//
// The paper's threads (Section 3.2) each own a Moore-curve partition of the points and insert
// them one after the other; a thread that would touch a tetrahedron another thread holds aborts
// the insertion and retries it later. Here every warp is such a thread: warp w takes the w-th
// contiguous segment of the wave's Moore order and inserts its points in that order, each walk
// starting from the warp's previous ball (Algorithm 1). Ownership is a 32-bit word per
// tetrahedron slot (0 = free, kExclusive = held by one warp, else the number of its sharers). One
// insertion:
//   1. walk (Section 2.1) from the previous ball, reading the mesh without locks;
//   2. cavity search (Section 2.1, Eq. 1) on those unlocked reads: the cavity C, its outside
//      neighbours A and the boundary facets, with every record kept in shared memory;
//   3. lock C, A (shared) and the slots the ball needs beyond C (Section 2.5 reuses C's slots
//      first), one atomic each; a slot held against it by another warp aborts the insertion (rule
//      (1) of Section 3.2: a thread touches only tetrahedra it owns);
//   4. re-read C (whole records) and A (vertices) under the locks: a difference means another
//      warp changed them between steps 2 and 3, and the insertion starts over from the walk;
//      also read which facet of each tetrahedron of A faces the cavity (neighbour slots hold
//      plain tetrahedron ids: it is the facet whose neighbour is the cavity tetrahedron);
//   5. write the ball (Section 2.5: one tetrahedron per boundary facet, adjacency through the
//      edge table), the back-pointers of A, then release every lock after a fence.
// Aborted points wait in a small per-warp list and are retried after later insertions; what is
// still left when the segment ends goes to the next launch. A cavity larger than the per-warp
// shared-memory workspace is inserted again in a global-memory workspace borrowed from a pool,
// else by a separate large-cavity launch; a predicate the FP32 stage cannot decide hands the
// point to a launch of the kernels with the exact stages (kExact). No warp ever waits on another,
// so every loop here is bounded by the segment length and fixed retry counts.
//
// The triangulation does not depend on the order of insertions (exact predicates and one
// symbolic perturbation, Section 2.4), so this engine gives the same tetrahedra as the
// round-based one.
//
// The file that includes this one sets kADefer, the aborted points a warp keeps for a retry (the
// borrowed workspaces of all of them have one layout: the same number in each).
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"
#include "predicates.cuh"

namespace dtg {
namespace {

constexpr int kAW = 4;            // warps per block of the shared-memory kernel
constexpr int kARetry = 3;        // immediate restarts after a failed re-read
constexpr int kATail = 48;        // further tries at its deferred points by a warp that has no others left
constexpr uint32_t kAChunk = 32;  // slots taken from the allocator at a time

enum AStatus : int {
  kAInserted = 0, kALost = 1, kARestart = 2, kABig = 3, kAWalkLimit = 4, kADup = 5, kAExact = 6, kANoSeed = 7
};

// Ball adjacency (Section 2.5): the n x n edge table for balls of at most 32 boundary vertices
// (the shared-memory workspaces), an edge hash for larger ones (the global-memory workspaces).
template <int kHashN, int kFMaxN, int kEdgeSlots>
struct AWSTail {
  static constexpr uint32_t kEdgeN = kEdgeSlots;
  uint32_t hkey[kHashN];
  uint8_t hval[kHashN];
  unsigned long long ekey[kEdgeN];
  uint32_t eval[kEdgeN];
  uint32_t hslot[3 * kFMaxN];
  uint32_t hold[3 * kFMaxN];
};
template <int kHashN, int kFMaxN>
struct AWSTail<kHashN, kFMaxN, 0> {
  // the visited set is needed only while the cavity is searched, the edge table only while the
  // ball is built: they share their bytes
  union {
    struct {
      uint32_t hkey[kHashN];
      uint8_t hval[kHashN];
    };
    uint16_t tab[32 * 32];
  };
};
// Working storage of one warp: the cavity's tetrahedra with their records as read, the outside
// tetrahedra with their vertices as read, the boundary facets, the ball's slots, a private pool
// of free slots, deferred points, and the warp's state (uniform across its lanes, written by
// lane 0). kEdgeSlots: slots of the edge hash, 0 for the edge table.
// kLocalB: the launch is one block, and the mesh is read and written through its SM's L1.
template <int kHashN, int kCMaxN, int kAMaxN, int kFMaxN, int kEdgeSlots, bool kCacheB, bool kLocalB = false>
struct AWS : AWSTail<kHashN, kFMaxN, kEdgeSlots> {
  static constexpr int kHash = kHashN, kCMax = kCMaxN, kAMax = kAMaxN, kFMax = kFMaxN;
  static constexpr bool kCache = kCacheB;  // conflict tests through the sub-determinant cache
  static constexpr int kPool = kFMaxN + 36;  // a refill of 32 slots always fits below kFMax
  static constexpr bool kTable = kEdgeSlots == 0;
  static constexpr bool kLocal = kLocalB;
  using CI = typename std::conditional<(kCMaxN > 255), uint16_t, uint8_t>::type;
  static_assert(!kTable || kCMaxN + kAMaxN + kFMaxN <= 32 * 32, "a lane's lock mask holds its entries");
  uint32_t cl[kCMaxN];       // cavity slots
  Tet cr[kCMaxN];            // their records as read
  uint32_t al[kAMaxN];       // outside slots
  uint4 av[kAMaxN];          // their vertex ids as read
  uint32_t slot[kFMaxN];     // slots of the new tetrahedra
  uint32_t ex[kFMaxN];       // slots beyond the cavity's, taken from the pool
  uint32_t vkey[32];
  uint32_t pool[kPool];
  uint32_t defer[kADefer];
  CI bl_ci[kFMaxN];          // boundary facet: cavity index
  uint8_t bl_f[kFMaxN];      // boundary facet: facet | 4 * the outside tetrahedron's facet
  unsigned long long fa, bump;  // allocator snapshot of the launch
  unsigned int cnt[8];          // inserted, lost, attempts, sum |C|, sum |B|, walk steps, restarts
  uint32_t hint;                // the warp's last ball
  int bn;                       // tetrahedra of the warp's last ball (0: none); slots in slot[]
  int np;                       // slots in the pool
  int nc, na, nb;               // cavity, outside and boundary-facet counts of the last search
  uint32_t emask;               // the edge hash's slots in use for this ball, less one
  // the segment's place: here and not in registers, which an insertion needs for itself
  uint32_t i, e0, k0, k1;       // next and end of the list's points, of the carried ones
  int nd, dhead, since;         // deferred points, the first of them, insertions since a retry
  int tail;                     // tries at them after the last of the segment's points
};

// Shared-memory workspace of the main kernel (cavities of up to 64 tetrahedra and 60 boundary
// facets), the global-memory one a warp borrows for a larger cavity (135 KB), and that of the
// large-cavity kernel (1.14 MB: the sphere's empty interior, a surface's first inner points).
template <bool kCache, bool kLocal = false>
using SmallWST = AWS<256, 64, 64, 60, 0, kCache, kLocal>;
template <bool kCache, bool kLocal = false>
using LargeWST = AWS<4096, 640, 704, 704, 4096, kCache, kLocal>;
using LargeWS = LargeWST<false>;  // the same layout with and without the cache
template <bool kCache>
using HugeWST = AWS<32768, 6144, 6144, 6144, 32768, kCache>;

// Reads and writes of the mesh by warps that run beside its writers: through L2, or, when all of
// them are in one block, through that block's L1, whose latency is a fraction (the first few
// hundred insertions of a mesh are one chain of such reads).
template <bool kLocal>
__device__ __forceinline__ uint4 ld_mesh(const uint4* p) {
  if constexpr (kLocal) {
    uint4 r;
    asm volatile("ld.relaxed.cta.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p)
                 : "memory");
    return r;
  } else {
    return __ldcg(p);
  }
}
template <bool kLocal>
__device__ __forceinline__ void st_mesh(uint4* p, const uint4& v) {
  if constexpr (kLocal)
    asm volatile("st.relaxed.cta.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
  else
    __stcg(p, v);
}
template <bool kLocal>
__device__ __forceinline__ void st_mesh(uint32_t* p, uint32_t v) {
  if constexpr (kLocal) asm volatile("st.relaxed.cta.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
  else __stcg(p, v);
}
template <bool kLocal>
__device__ __forceinline__ void fence_mesh() {
  if constexpr (kLocal) __threadfence_block();
  else __threadfence();
}

template <bool kLocal>
__device__ __forceinline__ Tet ld_tet(const Tet* T, uint32_t t) {
  Tet r;
  const uint4* p = reinterpret_cast<const uint4*>(T + t);
  r.v = ld_mesh<kLocal>(p);
  r.n = ld_mesh<kLocal>(p + 1);
  return r;
}

__device__ __forceinline__ bool same_tet(const Tet& a, const Tet& b) {
  return a.v.x == b.v.x && a.v.y == b.v.y && a.v.z == b.v.z && a.v.w == b.v.w && a.n.x == b.n.x &&
         a.n.y == b.n.y && a.n.z == b.n.z && a.n.w == b.n.w;
}

__device__ __forceinline__ bool same_v(const uint4& a, const uint4& b) {
  return a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w;
}

// A record that references only allocated vertices and slots (a record being rewritten may be
// read half old, half new; such a read is never followed).
__device__ __forceinline__ bool rec_ok(const Tet& T, uint32_t ntets, uint32_t npts) {
  // v + 1 wraps the ghost vertex to 0
  return max(max(T.v.x + 1u, T.v.y + 1u), max(T.v.z + 1u, T.v.w + 1u)) <= npts &&
         max(max(T.n.x, T.n.y), max(T.n.z, T.n.w)) < ntets;
}

// The predicates' FP32 stage on the double-float point copy (predicates.cuh: rigorous error
// bounds, Section 2.4's filters moved to FP32). When it cannot decide, the insertion is handed to
// the kernels built with kExact, which run the whole cascade (FP64 filter, exact arithmetic,
// symbolic perturbation): keeping the exact stages out of the common kernel keeps its registers
// free of the save and restore traffic their calls would cost. A return of 0 means "undecided".

__device__ __forceinline__ PtF pick(bool c, const PtF& x, const PtF& y) {
  PtF r;
  r.hx = c ? x.hx : y.hx; r.hy = c ? x.hy : y.hy; r.hz = c ? x.hz : y.hz; r.hw = 0.f;
  r.lx = c ? x.lx : y.lx; r.ly = c ? x.ly : y.ly; r.lz = c ? x.lz : y.lz; r.lw = 0.f;
  return r;
}

// orient3d of (v0, v1, v2, v3) with vertex i replaced by p. Moving p to the last place is an
// odd permutation for i = 0, 2 and an even one for i = 1, 3, so one FP32 evaluation on the other
// three vertices in their order serves every i (one copy of the code: the kernel's instruction
// footprint decides how often its warps wait for instructions).
__device__ __forceinline__ int orient_with_p(const Ctx& c, int i, const PtF& FP, const PtF& F0, const PtF& F1,
                                             const PtF& F2, const PtF& F3) {
  const PtF A = pick(i == 0, F1, F0), B = pick(i <= 1, F2, F1), C = pick(i <= 2, F3, F2);
  const int o = orient3d_f(A, B, C, FP, c.eta);
  return (i & 1) ? o : -o;
}

// Insphere of a finite tetrahedron v and p: -1 inside, 1 outside, 0 undecided.
__device__ __forceinline__ int inside_async(const Ctx& c, const uint4& v, const PtF& FP) {
  PtF A = load_ptf(c.ptf, v.x), B = load_ptf(c.ptf, v.y), C = load_ptf(c.ptf, v.z), D = load_ptf(c.ptf, v.w);
  return insphere_f(A, B, C, D, FP, c.eta);
}

// Sub-determinant cache (Section 2.4; an ablation, off unless the handle allocates it). With
// b, c, d, e the differences of the tetrahedron's other vertices and of p from its first vertex
// a, the insphere determinant expanded along e's row is ex Ax + ey Ay + ez Az + |e|^2 AL, and
// the cofactors A depend on the tetrahedron alone. Two float4 per slot: q0 = (Ax, Ay, Az, AL);
// q1 = (the permanents of Ax and Ay, then of Az and AL, each pair as two bfloat16 rounded up;
// the largest |coordinate| of b, c, d; 1 when the entry is valid). The same monomials as
// insphere_f's with fewer roundings on each (12 against 16), so insphere_f's bound holds;
// rounding the permanents up widens it by at most 2^-7 of itself.
__device__ __forceinline__ uint32_t bf16_up(float x) {  // x >= 0: the bfloat16 at or above x
  return (__float_as_uint(x) + 0xFFFFu) >> 16;
}
__device__ __forceinline__ float bf16_lo(float packed) { return __uint_as_float(__float_as_uint(packed) << 16); }
__device__ __forceinline__ float bf16_hi(float packed) {
  return __uint_as_float(__float_as_uint(packed) & 0xFFFF0000u);
}

__device__ __forceinline__ void subdet_make(const PtF& A, const PtF& B, const PtF& C, const PtF& D, float4& q0,
                                            float4& q1) {
  float bx, by, bz, cx, cy, cz, dx, dy, dz;
  diff_f(B, A, bx, by, bz);
  diff_f(C, A, cx, cy, cz);
  diff_f(D, A, dx, dy, dz);
  const float Lb = bx * bx + by * by + bz * bz, Lc = cx * cx + cy * cy + cz * cz, Ld = dx * dx + dy * dy + dz * dz;
  const float cd0 = cy * dz - cz * dy, cd1 = cx * dz - cz * dx, cd2 = cx * dy - cy * dx;
  const float bd0 = by * dz - bz * dy, bd1 = bx * dz - bz * dx, bd2 = bx * dy - by * dx;
  const float bc0 = by * cz - bz * cy, bc1 = bx * cz - bz * cx, bc2 = bx * cy - by * cx;
  const float pcd0 = fabsf(cy * dz) + fabsf(cz * dy), pcd1 = fabsf(cx * dz) + fabsf(cz * dx),
              pcd2 = fabsf(cx * dy) + fabsf(cy * dx);
  const float pbd0 = fabsf(by * dz) + fabsf(bz * dy), pbd1 = fabsf(bx * dz) + fabsf(bz * dx),
              pbd2 = fabsf(bx * dy) + fabsf(by * dx);
  const float pbc0 = fabsf(by * cz) + fabsf(bz * cy), pbc1 = fabsf(bx * cz) + fabsf(bz * cx),
              pbc2 = fabsf(bx * cy) + fabsf(by * cx);
  q0.x = Lc * bd0 - Lb * cd0 - Ld * bc0;
  q0.y = Lb * cd1 + Ld * bc1 - Lc * bd1;
  q0.z = Lc * bd2 - Lb * cd2 - Ld * bc2;
  q0.w = bx * cd0 - by * cd1 + bz * cd2;
  const float px = Lc * pbd0 + Lb * pcd0 + Ld * pbc0, py = Lc * pbd1 + Lb * pcd1 + Ld * pbc1,
              pz = Lc * pbd2 + Lb * pcd2 + Ld * pbc2;
  const float pl = fabsf(bx) * pcd0 + fabsf(by) * pcd1 + fabsf(bz) * pcd2;
  q1.x = __uint_as_float(bf16_up(px) | (bf16_up(py) << 16));
  q1.y = __uint_as_float(bf16_up(pz) | (bf16_up(pl) << 16));
  q1.z = fmaxf(fmaxf(fmaxf(fabsf(bx), fabsf(by)), fmaxf(fabsf(bz), fabsf(cx))),
               fmaxf(fmaxf(fabsf(cy), fabsf(cz)), fmaxf(fmaxf(fabsf(dx), fabsf(dy)), fabsf(dz))));
  q1.w = 1.f;
}

// insphere_f of the cached tetrahedron (first vertex A) and p: -1 inside, 1 outside, 0 undecided.
__device__ __forceinline__ int insphere_cached(const float4& q0, const float4& q1, const PtF& A, const PtF& FP,
                                               float eta) {
  float ex, ey, ez;
  diff_f(FP, A, ex, ey, ez);
  const float Le = ex * ex + ey * ey + ez * ez;
  const float det = (ex * q0.x + ey * q0.y) + (ez * q0.z + Le * q0.w);
  const float perm = (fabsf(ex) * bf16_lo(q1.x) + fabsf(ey) * bf16_hi(q1.x)) +
                     (fabsf(ez) * bf16_lo(q1.y) + Le * bf16_hi(q1.y));
  const float mm = fmaxf(q1.z, fmaxf(fabsf(ex), fmaxf(fabsf(ey), fabsf(ez)))) + eta, mm2 = mm * mm;
  const float eb = kInsphereCf * perm + 400.0f * eta * (mm2 * mm2);
  if (!(perm > 1e-30f && perm < 1e30f)) return 0;
  return det > eb ? 1 : (det < -eb ? -1 : 0);
}

// The conflict test of a finite tetrahedron u (vertices v) through the cache when its entry
// is valid, else from the coordinates.
__device__ __forceinline__ int inside_maybe_cached(const Ctx& c, uint32_t u, const uint4& v, const PtF& FP) {
  const float4 q1 = __ldcg(c.subdet + 2 * (size_t)u + 1);
  if (q1.w == 0.f) return inside_async(c, v, FP);
  const float4 q0 = __ldcg(c.subdet + 2 * (size_t)u);
  return insphere_cached(q0, q1, load_ptf(c.ptf, v.x), FP, c.eta);
}

// The exact signs behind the FP32 stage, for the kernels built with kExact (inputs the FP32 stage
// often cannot decide: lattices, co-spherical and coplanar sets). Out of line: their code and
// registers stay out of the common path.

// orient3d of the finite tetrahedron v with vertex i replaced by p.
static __device__ __noinline__ int orient_exact_at(const Pt* pts, DevState* st, uint4 v, int i, uint32_t p) {
  const Pt a = load_pt(pts, i == 0 ? p : v.x), b = load_pt(pts, i == 1 ? p : v.y), d = load_pt(pts, i == 2 ? p : v.z),
           e = load_pt(pts, i == 3 ? p : v.w);
  return orient3d(a, b, d, e, st);
}

// Whether p lies inside the perturbed sphere of the finite tetrahedron v.
static __device__ __noinline__ bool inside_exact_at(const Pt* pts, DevState* st, uint4 v, uint32_t p) {
  return insphere_sos(load_pt(pts, v.x), load_pt(pts, v.y), load_pt(pts, v.z), load_pt(pts, v.w), load_pt(pts, p),
                      st) < 0;
}

// Conflict of the ghost v (ghost vertex at position g, finite neighbour r) with p: p strictly
// beyond the hull facet, or on its plane and inside the finite neighbour's sphere (Section 2.6).
// The neighbour is read without a lock and need not be verified later: p on the facet's plane is
// inside the sphere of whatever tetrahedron is built on the facet from inside exactly when it is
// inside the facet's circle, and on the circle the perturbation decides by orient3d's with the
// apex among their four points, whose signs depend on the apex's side alone (the one without it
// is zero). So any live tetrahedron that holds the three vertices gives the same answer. Returns
// 1, 0, or -1 when r does not hold them (a record read mid-change).
static __device__ __noinline__ int ghost_exact_at(const Pt* pts, DevState* st, const Tet* tets, uint32_t npts, uint4 v,
                                                  int g, uint32_t r, uint32_t p) {
  const int o = orient_exact_at(pts, st, v, g, p);
  if (o != 0) return o > 0 ? 1 : 0;
  const uint4 R = __ldcg(reinterpret_cast<const uint4*>(tets + r));
  bool ok = !tet_dead(R) && R.x < npts && R.y < npts && R.z < npts && R.w < npts;
  for (int k = 0; k < 4; ++k) {
    const uint32_t q = get4(v, k);
    ok = ok && (k == g || R.x == q || R.y == q || R.z == q || R.w == q);
  }
  if (!ok) return -1;
  return inside_exact_at(pts, st, R, p) ? 1 : 0;
}

// Visibility walk (Section 2.1, ghost rules of Section 2.6) on unlocked reads. Lanes 0-3 test
// the four facets of the current tetrahedron at once (lane i: p against the facet opposite
// vertex i), and the walk leaves through the first facet p sees, in an order that turns with
// the steps. A record that is being rewritten may be read half old, half new: such reads end
// the walk with kARestart (or it runs into its step bound); nothing is trusted before step 4
// re-reads it under a lock. Called by the whole warp; the result is uniform: every lane reads the
// record, and while another warp rewrites it the lanes of one load may see it before and after, so
// each decision is a vote or one lane's. (Branching on each lane's own copy let a warp fall apart,
// once in some hundred calls on small clouds: a lost point, or an allocator in disorder.) *n_out: the
// neighbours of the tetrahedron reached.
template <bool kExact, bool kLocal>
__device__ __forceinline__ int walk_async(const Ctx& c, uint32_t p, const PtF& FP, uint32_t start, uint32_t salt,
                                          uint32_t max_steps, uint32_t* t_out, uint4* n_out, uint32_t* steps_out) {
  const int lane = threadIdx.x & 31;
  uint32_t t = start;
  Tet T;
  *steps_out = 0;
  *t_out = kNone;
  int hops = 0;
#pragma unroll 1
  for (;;) {
    if (t < c.tbase || t >= c.ntets) t = __ldcg(&c.st->anchor);
    t = __shfl_sync(kFull, t, 0);
    if (t >= c.ntets) return kARestart;
    T = ld_tet<kLocal>(c.tets, t);
    if (__all_sync(kFull, !tet_dead(T.v))) break;
    t = __shfl_sync(kFull, T.n.x, 0);  // dead slot: follow its redirect
    if (++hops > 64) return kARestart;
  }
  if (!__all_sync(kFull, rec_ok(T, c.ntets, c.npts))) return kARestart;
  const int g = ghost_pos(T.v);
  if (__any_sync(kFull, g >= 0)) {
    t = __shfl_sync(kFull, get4(T.n, g), 0);
    T = ld_tet<kLocal>(c.tets, t);
    if (!__all_sync(kFull, !tet_dead(T.v) && rec_ok(T, c.ntets, c.npts))) return kARestart;
  }
  uint32_t prev = kNone, steps = 0;
#pragma unroll 1
  for (;;) {
    if (__any_sync(kFull, ghost_pos(T.v) >= 0)) break;
    // lane i < 4: orientation of p against the facet opposite vertex i (0: undecided)
    int o = 1;
    const uint32_t nb = lane < 4 ? get4(T.n, lane) : prev;
    const bool mine = nb != prev;  // p is on this side of the facet just crossed
    if (mine) {

      const PtF F0 = load_ptf(c.ptf, T.v.x), F1 = load_ptf(c.ptf, T.v.y), F2 = load_ptf(c.ptf, T.v.z),
                F3 = load_ptf(c.ptf, T.v.w);
      o = orient_with_p(c, lane, FP, F0, F1, F2, F3);
    }
    unsigned sees = __ballot_sync(kFull, o < 0);
    // a facet the FP32 stage cannot decide matters only when no other facet is certainly seen:
    // any facet p sees is a valid exit of the visibility walk
    if (sees == 0 && __any_sync(kFull, o == 0)) {
      if constexpr (!kExact) return kAExact;
      if (o == 0) o = orient_exact_at(c.pts, c.st, T.v, lane, p);
      sees = __ballot_sync(kFull, o < 0);
    }
    if (sees == 0) {
      // p is inside (or on) this tetrahedron: a vertex equal to p would be a duplicate
      bool dup = false;
      if (lane < 4) {
        const PtF V = load_ptf(c.ptf, get4(T.v, lane));
        if (same_f(V, FP)) {
          const Pt P = load_pt(c.pts, p), Q = load_pt(c.pts, get4(T.v, lane));
          dup = Q.x == P.x && Q.y == P.y && Q.z == P.z;
        }
      }
      *t_out = t;
      *n_out = T.n;
      *steps_out = steps;
      return __any_sync(kFull, dup) ? kADup : kAInserted;
    }
    if (steps >= max_steps) {
      *t_out = t;
      *steps_out = steps;
      return kAWalkLimit;
    }
    // the first facet p sees, starting from a position that turns with the steps
    const unsigned rot = ((sees | (sees << 4)) >> ((salt + steps) & 3)) & 0xFu;
    const int exit = (__ffs(rot) - 1 + (int)((salt + steps) & 3)) & 3;
    prev = t;
    t = __shfl_sync(kFull, get4(T.n, exit), exit);
    T = ld_tet<kLocal>(c.tets, t);
    ++steps;
    if (!__all_sync(kFull, !tet_dead(T.v) && rec_ok(T, c.ntets, c.npts))) {
      *t_out = t;
      *steps_out = steps;
      return kARestart;
    }
  }
  *t_out = t;
  *n_out = T.n;
  *steps_out = steps;
  return kAInserted;
}

// Conflict of a record U (already read) with p: 1 in the cavity, 2 outside, 4 undecided by the
// FP32 stage, 8 not a consistent live record.
template <bool kCache, bool kExact>
__device__ __forceinline__ int conflict_async(const Ctx& c, uint32_t u, const Tet& U, uint32_t p, const PtF& FP) {
  const uint32_t vm = max(max(U.v.x, U.v.y), max(U.v.z, U.v.w)), nm = max(max(U.n.x, U.n.y), max(U.n.z, U.n.w));
  if (tet_dead(U.v) || nm >= c.ntets) return 8;
  if (vm < c.npts) {
    const int s = kCache ? inside_maybe_cached(c, u, U.v, FP) : inside_async(c, U.v, FP);
    if (s != 0) return s < 0 ? 1 : 2;
    if constexpr (!kExact) return 4;
    else return inside_exact_at(c.pts, c.st, U.v, p) ? 1 : 2;
  }
  const int g = ghost_pos(U.v);
  // the hull facet's three vertices
  const uint32_t a = g == 0 ? U.v.y : U.v.x, b = g <= 1 ? U.v.z : U.v.y, d = g <= 2 ? U.v.w : U.v.z;
  if (g < 0 || a >= c.npts || b >= c.npts || d >= c.npts) return 8;
  // orientation of the hull facet and p in the ghost's place
  int o = orient3d_f(load_ptf(c.ptf, a), load_ptf(c.ptf, b), load_ptf(c.ptf, d), FP, c.eta);
  o = (g & 1) ? o : -o;
  if (o != 0) return o > 0 ? 1 : 2;
  // p on the facet's plane as far as the FP32 stage can tell
  if constexpr (!kExact) return 4;
  const int s = ghost_exact_at(c.pts, c.st, c.tets, c.npts, U.v, g, get4(U.n, g), p);
  return s < 0 ? 8 : (s ? 1 : 2);
}

// The visited set's entry of key (its index), claimed for the caller when *mine comes back true.
// The table is never full: it has more entries than the lists have room for, plus one per lane.
template <class W>
__device__ __forceinline__ uint32_t hclaim(W& w, uint32_t key, bool* mine) {
  static_assert(W::kHash > W::kCMax + W::kAMax + 32, "room for every visited tetrahedron");
  uint32_t h = (hash32(key) >> 8) & (W::kHash - 1);
  *mine = false;
#pragma unroll 1
  for (int probe = 0; probe < W::kHash; ++probe) {
    const uint32_t old = atomicCAS(&w.hkey[h], kNone, key);
    if (old == kNone) *mine = true;
    if (old == kNone || old == key) break;
    h = (h + 1) & (W::kHash - 1);
  }
  return h;
}

// Step 2: the cavity of p on unlocked reads. The search starts from every tetrahedron of the
// first pass that is in conflict with p: with ball > 0 the ball last inserted by this warp
// (w.slot[0, ball)), else the walk's end t0 (which has to be in conflict) and its neighbours
// tn. The conflict region is connected, so the cavity found does not depend on where the search
// starts; starting from all of them at once takes the breadth-first levels from about seven to
// four (each level is a chain of dependent loads: record, points, test), and the test's code
// exists once. Returns kAInserted (lists filled), kANoSeed (no tetrahedron of the ball is in
// conflict), kARestart (an inconsistent read), kABig (the workspace is too small) or kAExact.
template <bool kExact, class W>
__device__ __forceinline__ int cavity_async(const Ctx& c, W& w, int ball, uint32_t t0, const uint4& tn, uint32_t p,
                                            const PtF& FP) {
  const int lane = threadIdx.x & 31;
  static_assert(W::kHash % 128 == 0, "cleared by 16 bytes a lane");
#pragma unroll 1
  for (int i = lane; i < W::kHash / 4; i += 32)
    reinterpret_cast<uint4*>(w.hkey)[i] = make_uint4(kNone, kNone, kNone, kNone);
  __syncwarp();
  int nc = 0, na = 0, nb = 0;
  {
    uint32_t u = kNone;
    if (ball > 0) {
      if (lane < ball) u = w.slot[lane];
    } else if (lane < 5) {
      u = lane == 0 ? t0 : get4(tn, lane - 1);
    }
    int res = 0;
    Tet U;
    if (u < c.ntets) {
      U = ld_tet<W::kLocal>(c.tets, u);
      res = conflict_async<W::kCache, kExact>(c, u, U, p, FP);
    }
    const unsigned m = __ballot_sync(kFull, res == 1);
    if (ball > 0) {
      if (m == 0) return kANoSeed;
    } else if (!(m & 1u)) {  // the walk's tetrahedron: undecided, or read mid-rewrite
      return __shfl_sync(kFull, res, 0) == 4 ? kAExact : kARestart;
    }
    if (res == 1) {
      bool mine;
      w.hval[hclaim(w, u, &mine)] = 1;
      const int pos = __popc(m & lanemask_lt());
      w.cl[pos] = u;
      w.cr[pos] = U;
    }
    nc = __popc(m);
    __syncwarp();
  }
  int flag = 0, head = 0;
#pragma unroll 1
  while (head < nc) {
    const int k = lane >> 2, f = lane & 3, ci = head + k;
    const bool active = ci < nc;
    head = min(head + 8, nc);
    uint32_t u = 0, h = 0;
    bool first = false;  // this lane is the first to reach u
    if (active) {
      u = reinterpret_cast<const uint32_t*>(&w.cr[ci].n)[f];
      h = hclaim(w, u, &first);
    }
    int res = 0;
    Tet U;
    if (first) {
      U = ld_tet<W::kLocal>(c.tets, u);  // u < ntets: the record that names it was checked
      res = conflict_async<W::kCache, kExact>(c, u, U, p, FP);
      w.hval[h] = (uint8_t)res;
    }
    __syncwarp();
    if (active && !first) res = vld(&w.hval[h]);
    const unsigned mX = __ballot_sync(kFull, res >= 4);
    const unsigned mC = __ballot_sync(kFull, first && res == 1);
    const unsigned mA = __ballot_sync(kFull, first && res == 2);
    const unsigned mB = __ballot_sync(kFull, res == 2);
    if (mX) {
      flag = __any_sync(kFull, res == 4) ? 4 : 1;
      break;
    }
    if (first) {
      if (res == 1) {
        const int pos = nc + __popc(mC & lanemask_lt());
        if (pos < W::kCMax) {
          w.cl[pos] = u;
          w.cr[pos] = U;
        }
      } else {  // outside tetrahedra (locked and verified)
        const int pos = na + __popc(mA & lanemask_lt());
        if (pos < W::kAMax) {
          w.al[pos] = u;
          w.av[pos] = U.v;
        }
      }
    }
    if (res == 2) {
      const int pos = nb + __popc(mB & lanemask_lt());
      if (pos < W::kFMax) {
        w.bl_ci[pos] = (typename W::CI)ci;
        w.bl_f[pos] = (uint8_t)f;
      }
    }
    nc += __popc(mC);
    na += __popc(mA);
    nb += __popc(mB);
    __syncwarp();
    if (nc > W::kCMax || na > W::kAMax || nb > W::kFMax) {
      flag = 2;
      break;
    }
  }
  if (lane == 0) {
    w.nc = nc;
    w.na = na;
    w.nb = nb;
  }
  __syncwarp();
  return flag == 0 ? kAInserted : flag == 4 ? kAExact : flag == 2 ? kABig : kARestart;
}

// Slot of lock-list entry i: cavity slots, then the outside slots, then the ball's extra slots.
template <class W>
__device__ __forceinline__ uint32_t lock_entry(const W& w, int i, int nc, int na, int nx) {
  if (i < nc) return w.cl[i];
  i -= nc;
  if (i < na) return w.al[i];
  i -= na;
  return i < nx ? w.ex[i] : kNone;
}

// Ownership words. A slot whose record is replaced (the cavity's, the ball's extra slots) is taken
// exclusively; an outside tetrahedron, which only gets a back-pointer in a facet slot of its own,
// is shared: two insertions whose cavities do not touch may hold the same one, each rewriting
// another facet (the one that faces its cavity). The word is the number of sharers, plus
// kExclusive while a warp holds it alone; a release subtracts what was added, so that an attempt
// to share in between is not lost.
constexpr uint32_t kExclusive = 0x80000000u;

// Takes the locks of the lists' entries. With the edge table (few entries a lane) bit k of *held
// stands for entry lane + 32 k, and every entry is tried, so that the atomics overlap; larger
// workspaces count: the entries are taken in order up to the first that is held against them.
template <class W>
__device__ __forceinline__ bool take_locks(const W& w, uint32_t* lock, int nc, int na, int nx, uint32_t* held) {
  const int lane = threadIdx.x & 31, nl = nc + na + nx;
  bool ok = true;
  uint32_t h = 0;
#pragma unroll 1
  for (int k = 0; lane + 32 * k < nl && (W::kTable || ok); ++k) {
    const int i = lane + 32 * k;
    uint32_t* word = &lock[lock_entry(w, i, nc, na, nx)];
    const bool shared = i >= nc && i < nc + na;
    const uint32_t old = shared ? atomicAdd(word, 1u) : atomicCAS(word, 0u, kExclusive);
    if (shared ? old >= kExclusive : old != 0u) {
      ok = false;
      if (shared) atomicSub(word, 1u);
    } else {
      h = W::kTable ? h | (1u << k) : h + 1;
    }
  }
  *held = h;
  return __all_sync(kFull, ok);
}

// Releases the locks of the entries this lane took.
template <class W>
__device__ __forceinline__ void release_held(const W& w, uint32_t* lock, uint32_t held, int nc, int na, int nx) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int k = 0; W::kTable ? (held >> k) != 0 : k < (int)held; ++k) {
    const int i = lane + 32 * k;
    if (!W::kTable || ((held >> k) & 1u))
      atomicSub(&lock[lock_entry(w, i, nc, na, nx)], i >= nc && i < nc + na ? 1u : kExclusive);
  }
}

// The same, and the first `heldx` of this lane's extra slots of a large workspace.
template <class W>
__device__ __forceinline__ void release_all(const W& w, uint32_t* lock, uint32_t held, uint32_t heldx, int nc, int na,
                                            int nx) {
  release_held(w, lock, held, nc, na, nx);
  if constexpr (!W::kTable) {
#pragma unroll 1
    for (uint32_t k = 0; k < heldx; ++k) atomicSub(&lock[w.ex[(threadIdx.x & 31) + 32 * k]], kExclusive);
  }
}

// Takes n slots from the warp's pool into w.ex, refilling it from the allocator (free list,
// then the bump pointer, as in the round-based engine). False when the store is full.
template <class W>
__device__ __forceinline__ bool pool_take(const Ctx& c, W& w, int n) {
  const int lane = threadIdx.x & 31;
  int np = w.np;
#pragma unroll 1
  while (np < n) {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&c.st->alloc_cursor, (unsigned long long)kAChunk);
    base = __shfl_sync(kFull, base, 0);
    bool fail = false;
    const uint32_t s = virtual_slot(c, base + lane, w.fa, w.bump, c.st->capacity, fail);
    if (__any_sync(kFull, fail)) {
      if (lane == 0) raise_error(c.st, kErrCapacity, 0xA5u);
      return false;
    }
    w.pool[np + lane] = s;  // np < n <= kFMax, so np + 32 <= kPool
    np += 32;
    __syncwarp();
  }
#pragma unroll 1
  for (int i = lane; i < n; i += 32) w.ex[i] = w.pool[np - 1 - i];
  __syncwarp();
  if (lane == 0) w.np = np - n;
  __syncwarp();
  return true;
}

// Puts n slots s[0, n) back into the pool; what does not fit goes to the pending list.
template <class W>
__device__ __forceinline__ void pool_give(const Ctx& c, W& w, const uint32_t* s, int n) {
  const int lane = threadIdx.x & 31;
  const int np = w.np;
  const int keep = min(n, W::kPool - np);
#pragma unroll 1
  for (int i = lane; i < keep; i += 32) w.pool[np + i] = s[i];
  if (n > keep) {
    unsigned long long pb = 0;
    if (lane == 0) pb = atomicAdd(&c.st->pending, (unsigned long long)(n - keep));
    pb = __shfl_sync(kFull, pb, 0);
#pragma unroll 1
    for (int i = keep + lane; i < n; i += 32) {
      if (pb + (i - keep) < c.st->free_capacity) c.pending[pb + (i - keep)] = s[i];
      else raise_error(c.st, kErrFreeList, 0xA7u);
    }
  }
  __syncwarp();
  if (lane == 0) w.np = np + keep;
  __syncwarp();
}

// One attempt at inserting p (steps 1-5). start: where a walk begins (kNone: where p was last
// located, else the grid's hints). w.hint is the warp's last ball, updated on success.
template <bool kExact, class W>
__device__ __forceinline__ int try_insert(const Ctx& c, W& w, uint32_t* lock, uint32_t p,
                                          const InsertLog& lg, bool ball_start, uint32_t start) {
  const int lane = threadIdx.x & 31;
  const PtF FP = load_ptf(c.ptf, p);
  // 1. a start in conflict with p. Consecutive points of a segment are close, so p is often
  //    inside the circumsphere of a tetrahedron of the previous ball (it will be joined to the
  //    previous point): the search's first pass tests them all, without a walk. Otherwise walk.
  int ball = ball_start ? w.bn : 0;
  __syncwarp();
  if (lane == 0) w.bn = 0;  // used once
#pragma unroll 1
  for (int attempt = 0; attempt <= kARetry;) {
    uint32_t t0 = kNone;
    uint4 tn = make_uint4(kNone, kNone, kNone, kNone);
    if (ball == 0) {
      if (start == kNone) start = c.point_hint[p];
      if (start == kNone) {
        uint32_t f, g;
        cells_of(c, FP, &f, &g);
        start = c.cell_hint[f];
        if (start == kNone) start = c.cell_hint2[g];
      }
      start = __shfl_sync(kFull, start, 0);
      uint32_t steps = 0;
      const int ws = walk_async<kExact, W::kLocal>(c, p, FP, start, p * 0x9E3779B1u >> 30, c.max_walk, &t0, &tn, &steps);
      if (lane == 0) {
        if (t0 != kNone && t0 < c.ntets) c.point_hint[p] = t0;
        w.cnt[5] += steps;
      }
      if (ws == kADup || ws == kAWalkLimit || ws == kAExact) return ws;
      if (ws == kARestart) {
        // the next attempt starts from the grid, the last one from the anchor (a hint may lead
        // into a chain of dead slots that is longer than a walk follows)
        if (lane == 0) {
          w.cnt[6] += 1;
          c.point_hint[p] = kNone;
        }
        __syncwarp();
        ++attempt;
        start = attempt == kARetry ? __ldcg(&c.st->anchor) : kNone;
        continue;
      }
    }
    // 2. cavity on unlocked reads
    const int r = cavity_async<kExact>(c, w, ball, t0, tn, p, FP);
    ball = 0;
    if (r == kANoSeed) continue;  // walk from the warp's last ball
    if (r == kABig && lane == 0) c.point_hint[p] = w.cl[0];
    if (r == kABig || r == kAExact) return r;
    start = kNone;  // a further attempt starts from the grid
    ++attempt;
    if (r == kARestart) {
      if (lane == 0) w.cnt[6] += 1;
      continue;
    }
    const int nc = w.nc, na = w.na, nb = w.nb;
    const int reuse = min(nc, nb);
    int nx = nb - reuse;
    // a large ball's extra slots are taken once its cavity is held: slots that come back from a
    // lost attempt would wait, beyond what the pool holds, for the launch's end
    const int nx0 = W::kTable ? nx : 0;
    if (nx0 > 0 && !pool_take(c, w, nx0)) return kALost;
    // 3. lock C, A and the extra slots
    uint32_t held, heldx = 0;
    bool locked = take_locks(w, lock, nc, na, nx0, &held);
    if constexpr (!W::kTable) {
      if (locked && nx > 0) {
        if (!pool_take(c, w, nx)) {
          release_held(w, lock, held, nc, na, 0);
          return kALost;
        }
        bool ok = true;
#pragma unroll 1
        for (int i = lane; i < nx && ok; i += 32) {
          ok = atomicCAS(&lock[w.ex[i]], 0u, kExclusive) == 0u;
          if (ok) ++heldx;
        }
        locked = __all_sync(kFull, ok);
      } else if (!locked) {
        nx = 0;
      }
    }
    if (!locked) {
      if (lane == 0) c.point_hint[p] = w.cl[0];  // a retry starts in the cavity
      release_all(w, lock, held, heldx, nc, na, nx0);
      if (nx > 0) pool_give(c, w, w.ex, nx);
      return kALost;
    }
    // a lane re-reads slots that other lanes locked: the warp first, then each lane's fence
    __syncwarp();
    fence_mesh<W::kLocal>();
    // 4. re-read under the locks
    bool same = true;
#pragma unroll 1
    for (int i = lane; i < nc; i += 32) same = same && same_tet(ld_tet<W::kLocal>(c.tets, w.cl[i]), w.cr[i]);
#pragma unroll 1
    for (int i = lane; i < na; i += 32) {
      const uint32_t a = w.al[i];
      same = same && same_v(ld_mesh<W::kLocal>(reinterpret_cast<const uint4*>(c.tets + a)), w.av[i]);
    }
    // which facet of each outside tetrahedron faces the cavity (it is locked: this stays true)
#pragma unroll 1
    for (int i = lane; i < nb; i += 32) {
      const int ci = w.bl_ci[i], f = w.bl_f[i] & 3;
      const uint32_t u = get4(w.cr[ci].n, f);
      const int back = back_facet(ld_mesh<W::kLocal>(reinterpret_cast<const uint4*>(&c.tets[u].n)), w.cl[ci]);
      same = same && back >= 0;
      w.bl_f[i] = (uint8_t)(f | ((back & 3) << 2));
    }
    if constexpr (W::kCache) {
      // the cache's decisions were taken on entries read without locks: each is taken again on
      // the entry as it stands under the locks (an entry changes only with its record)
#pragma unroll 1
      for (int i = lane; i < nc; i += 32) {
        const uint4 v = w.cr[i].v;
        if (ghost_pos(v) < 0) same = same && inside_maybe_cached(c, w.cl[i], v, FP) < 0;
      }
#pragma unroll 1
      for (int i = lane; i < na; i += 32) {
        const uint4 v = w.av[i];
        if (ghost_pos(v) < 0) same = same && inside_maybe_cached(c, w.al[i], v, FP) > 0;
      }
    }
    if (!__all_sync(kFull, same)) {
      release_all(w, lock, held, heldx, nc, na, nx0);
      if (nx > 0) pool_give(c, w, w.ex, nx);
      if (lane == 0) w.cnt[6] += 1;
      continue;
    }
    // 5. the ball: cavity slots first, then the extra slots
#pragma unroll 1
    for (int i = lane; i < nb; i += 32) w.slot[i] = i < reuse ? w.cl[i] : w.ex[i - reuse];
    w.vkey[lane] = kNoVertex;
    if constexpr (!W::kTable) {
      uint32_t en = 512;  // a power of two, at least 2.7 slots per edge (1.5 nb edges)
      while (en < W::kEdgeN && en < 4u * (uint32_t)nb) en <<= 1;
      if (lane == 0) w.emask = en - 1;
#pragma unroll 1
      for (uint32_t i = lane; i < en; i += 32) {
        w.ekey[i] = ~0ull;
        w.eval[i] = kNone;
      }
    }
    __syncwarp();
    // record every internal facet: facet a of new tetrahedron i holds the boundary edge b -> c
    bool vfail = false;
    // the table path's vertex slots of this lane's facets (lane and lane + 32; nb <= 60), kept
    // for the partner lookups below
    uint32_t vs[2] = {0, 0};
#pragma unroll 1
    for (int i = lane; i < nb; i += 32) {
      const int ci = w.bl_ci[i], f = w.bl_f[i] & 3;
      uint4 v = w.cr[ci].v;
      set4(v, f, p);
      int pos[3];
      after_pos(f, pos[0], pos[1], pos[2]);
      if constexpr (W::kTable) {
        const int la = vslot(w.vkey, get4(v, pos[0])), lb = vslot(w.vkey, get4(v, pos[1])),
                  lc = vslot(w.vkey, get4(v, pos[2]));
        if (la < 0 || lb < 0 || lc < 0) {
          vfail = true;
          continue;
        }
        vs[i >> 5] = (uint32_t)la | ((uint32_t)lb << 8) | ((uint32_t)lc << 16);
        w.tab[lb * 32 + lc] = (uint16_t)((i << 2) | pos[0]);
        w.tab[lc * 32 + la] = (uint16_t)((i << 2) | pos[1]);
        w.tab[la * 32 + lb] = (uint16_t)((i << 2) | pos[2]);
      } else {
        for (int k = 0; k < 3; ++k) {
          const uint32_t x = get4(v, pos[(k + 1) % 3]), y = get4(v, pos[(k + 2) % 3]);
          const unsigned long long key = ((unsigned long long)min(x, y) << 32) | max(x, y);
          const uint32_t em = w.emask;
          uint32_t h = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 40) & em, sl = kNone;
#pragma unroll 1
          for (uint32_t probe = 0; probe <= em; ++probe) {
            const unsigned long long old = atomicCAS(&w.ekey[h], ~0ull, key);
            if (old == ~0ull || old == key) {
              sl = h;
              break;
            }
            h = (h + 1) & em;
          }
          if (sl == kNone) {
            vfail = true;
            break;
          }
          w.hslot[3 * i + k] = sl;
          w.hold[3 * i + k] = atomicExch(&w.eval[sl], (uint32_t)((i << 2) | pos[k]));
        }
      }
    }
    __syncwarp();
    // every internal facet was recorded by its two sides (the cavity was verified under the
    // locks, so its boundary is a closed surface); a lookup that finds no partner is a bug
    bool bad = __any_sync(kFull, vfail);
#pragma unroll 1
    for (int i = lane; i < nb && !bad; i += 32) {
      const int ci = w.bl_ci[i], f = w.bl_f[i] & 3, back = w.bl_f[i] >> 2;
      uint4 v = w.cr[ci].v;
      const uint32_t out = get4(w.cr[ci].n, f);
      set4(v, f, p);
      int a, b, cc;
      after_pos(f, a, b, cc);
      uint32_t ea, eb, ec;
      if constexpr (W::kTable) {
        const uint32_t sl = vs[i >> 5];
        const int la = (int)(sl & 0xFFu), lb = (int)((sl >> 8) & 0xFFu), lc = (int)(sl >> 16);
        ea = vld(&w.tab[lc * 32 + lb]);
        eb = vld(&w.tab[la * 32 + lc]);
        ec = vld(&w.tab[lb * 32 + la]);
      } else {
        uint32_t e3[3];
        for (int k = 0; k < 3; ++k) {
          const uint32_t old = w.hold[3 * i + k];
          e3[k] = old != kNone ? old : vld(&w.eval[w.hslot[3 * i + k]]);
        }
        ea = e3[0];
        eb = e3[1];
        ec = e3[2];
      }
      if ((ea >> 2) >= (uint32_t)nb || (eb >> 2) >= (uint32_t)nb || (ec >> 2) >= (uint32_t)nb ||
          (ea >> 2) == (uint32_t)i || (eb >> 2) == (uint32_t)i || (ec >> 2) == (uint32_t)i) {
        bad = true;
        break;
      }
      uint4 n4;
      set4(n4, f, out);
      set4(n4, a, w.slot[ea >> 2]);
      set4(n4, b, w.slot[eb >> 2]);
      set4(n4, cc, w.slot[ec >> 2]);
      const uint32_t s = w.slot[i];
      uint4* dst = reinterpret_cast<uint4*>(c.tets + s);
      st_mesh<W::kLocal>(dst, v);
      st_mesh<W::kLocal>(dst + 1, n4);
      if constexpr (W::kCache) {
        float4 q0 = make_float4(0.f, 0.f, 0.f, 0.f), q1 = q0;  // a ghost's entry stays invalid
        if (ghost_pos(v) < 0)
          subdet_make(load_ptf(c.ptf, v.x), load_ptf(c.ptf, v.y), load_ptf(c.ptf, v.z), load_ptf(c.ptf, v.w), q0, q1);
        __stcg(c.subdet + 2 * (size_t)s, q0);
        __stcg(c.subdet + 2 * (size_t)s + 1, q1);
      }
      if constexpr (!W::kCache && (kExact || !W::kTable)) {  // no cache kept here: the entry it replaces is void
        if (c.subdet) __stcg(c.subdet + 2 * (size_t)s + 1, make_float4(0.f, 0.f, 0.f, 0.f));
      }
      st_mesh<W::kLocal>(reinterpret_cast<uint32_t*>(&c.tets[out].n) + back, s);
    }
    if (__any_sync(kFull, bad)) {
      if (lane == 0) raise_error(c.st, kErrInternal, 0xA8u);
      release_all(w, lock, held, heldx, nc, na, nx0);
      return kALost;
    }
    // cavity slots left over (|C| > |B|) die, keep a redirect into the ball, and join the pool
    const int freed = nc - nb;
    if (freed > 0) {
      const uint32_t redirect = w.slot[0];
#pragma unroll 1
      for (int i = lane; i < freed; i += 32) {
        uint4* dst = reinterpret_cast<uint4*>(c.tets + w.cl[nb + i]);
        st_mesh<W::kLocal>(dst, make_uint4(kDeadMark, kDeadMark, kDeadMark, kDeadMark));
        st_mesh<W::kLocal>(dst + 1, make_uint4(redirect, kNone, kNone, kNone));
      }
    }
    // a slot's lock is not always released by the lane that wrote its record (dead slots, extra
    // slots, back-pointers): every lane's writes come before every lane's fence, a vote orders none
    __syncwarp();
    fence_mesh<W::kLocal>();
    release_all(w, lock, held, heldx, nc, na, nx0);
    if (freed > 0) pool_give(c, w, w.cl + nb, freed);
    if (lane == 0) {
      const uint32_t s0 = w.slot[0];
      uint32_t f, g;
      cells_of(c, FP, &f, &g);
      c.cell_hint[f] = s0;
      c.cell_hint2[g] = s0;
      c.point_hint[p] = s0;
      // the handle's state shares one cache line with the allocator's atomics: every warp
      // writing it per insertion serialised the whole launch, so it is refreshed now and then
      if ((w.cnt[0] & 63u) == 0) c.st->anchor = s0;
      log_outcome(lg, p, kCandInserted, nc);
      w.hint = s0;
      w.bn = W::kTable ? (nb < 32 ? nb : 32) : 0;
    }
    if (lane == 0) w.cnt[0] += 1;
    if (lane == 3) w.cnt[3] += nc;
    if (lane == 4) w.cnt[4] += nb;
    return kAInserted;  // the caller's next __syncwarp orders these
  }
  return kALost;
}

// Hands point p to a queue of the host's next step (0: next pass, 1: large cavities, 2: the
// kernels with the exact predicates). Lane 0.
__device__ __forceinline__ void to_queue(const AsyncIO& io, const Ctx& c, int q, uint32_t p) {
  uint32_t* out = q == 0 ? io.lose_out : (q == 1 ? io.big_out : io.exact_out);
  const int qi = q == 0 ? io.lose_q : (q == 1 ? io.big_q : io.exact_q);
  const unsigned long long b = atomicAdd(&c.st->q[qi], 1ull);
  out[b] = p;
}

// A cavity too large for the warp's shared-memory workspace: the same insertion again in a
// global-memory workspace (of type L) borrowed from the launch's pool (tried at a few places,
// never waited for). Returns kABig when the cavity exceeds it too, kALost when none is free. The
// borrowed workspace's counters, spare slots and ball hint come back to the warp's own. Out of
// line: it runs for about one point in 1500, and inlined it would double the kernel's instruction
// footprint.
template <bool kExact, class L, class W>
__device__ __noinline__ int try_insert_large(const Ctx& c, L* pool, unsigned int* busy, uint32_t n, W& w, uint32_t* lock,
                                             uint32_t me, uint32_t p, const InsertLog& lg) {
  if (!pool || n == 0) return kABig;
  const int lane = threadIdx.x & 31;
  int k = -1;
  if (lane == 0)
#pragma unroll 1
    for (int t = 0; t < 8 && k < 0; ++t) {
      const uint32_t cand = (me * 0x9E3779B1u + (uint32_t)t * 0x85EBCA6Bu) % n;
      if (atomicCAS(&busy[cand], 0u, 1u) == 0u) k = (int)cand;
    }
  if (k >= 0) __threadfence();  // after the workspace's last borrower (it fences before its release)
  k = __shfl_sync(kFull, k, 0);
  if (k < 0) return kALost;
  L& b = pool[k];
  if (lane == 0) {
    b.fa = w.fa;
    b.bump = w.bump;
    b.np = 0;
    b.bn = 0;
    b.hint = w.hint;
    for (int q = 0; q < 8; ++q) b.cnt[q] = 0;
  }
  __syncwarp();
  const int r = try_insert<kExact>(c, b, lock, p, lg, false, kNone);
  pool_give(c, w, b.pool, b.np);
  if (lane == 0) {
    w.cnt[0] += b.cnt[0];
    w.cnt[3] += b.cnt[3];
    w.cnt[4] += b.cnt[4];
    w.cnt[5] += b.cnt[5];
    w.cnt[6] += b.cnt[6];
    if (r == kAInserted) {
      w.hint = b.hint;
      atomicAdd(&c.st->n_big, 1ull);
    }
    w.bn = 0;
    __threadfence();
    atomicExch(&busy[k], 0u);
  }
  __syncwarp();
  return r;
}

// One warp's work: its share [k0, k1) of the points carried over from earlier launches, each
// started where it was last located, then segment [b0, e0) of io's list in order; deferred points
// are retried after later insertions. At the end what is left is handed on, unused slots return
// and counters are flushed.
template <bool kExact, class W>
__device__ __forceinline__ void run_segment(const Ctx& c, const AsyncIO& io, W& w, uint32_t* lock, uint32_t me,
                                            uint32_t b0, uint32_t e0, uint32_t k0, uint32_t k1, const InsertLog& lg) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    w.fa = __ldcg(&c.st->free_avail);
    w.bump = __ldcg(&c.st->bump);
    w.np = 0;
    w.bn = 0;
    for (int k = 0; k < 8; ++k) w.cnt[k] = 0;
    w.hint = kNone;
    w.i = b0;
    w.e0 = e0;
    w.k0 = k0;
    w.k1 = k1;
    w.nd = w.dhead = w.since = w.tail = 0;
  }
#pragma unroll 1
  for (;;) {
    __syncwarp();  // lane 0's writes are seen by every lane below
    const uint32_t i = w.i;
    uint32_t p, start = kNone;
    bool retried = false, follows = false;  // follows: the point after the last inserted one
    if (w.nd > 0 && ((i >= w.e0 && w.k0 >= w.k1) || w.since >= 4)) {
      p = w.defer[w.dhead];
      retried = true;
    } else if (w.k0 < w.k1) {
      p = io.carry[w.k0];
    } else if (i < w.e0) {
      p = io.q ? io.q[i] : (io.vflag[i] ? kNone : i);
      follows = i > b0;
      if (follows) start = w.hint;
    } else {
      break;
    }
    __syncwarp();
    if (lane == 0) {
      if (retried) {
        w.dhead = (w.dhead + 1) % kADefer;
        w.nd -= 1;
        w.since = 0;
      } else if (w.k0 < w.k1) {
        w.k0 += 1;
      } else {
        w.i = i + 1;
      }
    }
    if (p == kNone) continue;  // a duplicate or one of the first four
    if (lane == 0) w.cnt[2] += 1;
    int r = try_insert<kExact>(c, w, lock, p, lg, follows && io.ball_start != 0, start);
    if constexpr (W::kTable) {
      if (r == kABig)
        r = try_insert_large<kExact>(c, static_cast<LargeWST<W::kCache, W::kLocal>*>(io.big_ws), io.big_busy, io.big_n, w, lock, me, p,
                                     lg);
    }
    // a raised error stops the launch; read every 16 points for the same reason as the anchor
    unsigned err = 0;
    if (lane == 0 && (w.cnt[2] & 15u) == 0) err = __ldcg(&c.st->error);
    if (__shfl_sync(kFull, err, 0) != 0u) break;
    if (r == kAInserted) {
      if (lane == 0) w.since += 1;
      continue;
    }
    // every lane holds the same r and `retried` and reads the same nd: uniform decisions
    if (r == kALost && lane == 0) {
      w.cnt[1] += 1;
      log_outcome(lg, p, kCandLost, 0);
    }
    if (r == kADup) {
      if (lane == 0) atomicAdd(&c.st->n_dups, 1ull);
    } else if (r == kABig) {
      if (lane == 0) to_queue(io, c, 1, p);
    } else if (r == kAExact) {
      if (lane == 0) to_queue(io, c, 2, p);
    } else if (r == kALost && w.nd < kADefer && (!retried || w.nd < kADefer / 2) && w.tail < kATail) {
      // lost: again after a few other insertions; at the segment's end, where the warps that it
      // loses to are about done too, again and again (a bounded number of times)
      const bool end = i >= w.e0 && w.k0 >= w.k1;
      __syncwarp();
      if (lane == 0) {
        w.defer[(w.dhead + w.nd) % kADefer] = p;
        w.nd += 1;
        w.tail += end ? 1 : 0;
      }
      if (end) __nanosleep(2000);
    } else {  // a walk over its step bound, or a point that lost again: the next pass
      if (lane == 0) to_queue(io, c, 0, p);
    }
  }
  __syncwarp();
  // what is left: deferred points to the next pass, unused slots back to the allocator
  if (lane == 0)
#pragma unroll 1
    for (int k = 0; k < w.nd; ++k) to_queue(io, c, 0, w.defer[(w.dhead + k) % kADefer]);
  const int np = w.np;
  if (np > 0) {
    unsigned long long pb = 0;
    if (lane == 0) pb = atomicAdd(&c.st->pending, (unsigned long long)np);
    pb = __shfl_sync(kFull, pb, 0);
#pragma unroll 1
    for (int k = lane; k < np; k += 32) {
      if (pb + k < c.st->free_capacity) c.pending[pb + k] = w.pool[k];
      else raise_error(c.st, kErrFreeList, 0xA9u);
    }
  }
  if (lane == 0) {
    unsigned long long* dst[8] = {&c.st->n_inserted, &c.st->n_conflicts, &c.st->n_attempts, &c.st->sum_cavity,
                                  &c.st->sum_ball, &c.st->sum_walk, &c.st->n_restart, &c.st->n_inserted_async};
    w.cnt[7] = w.cnt[0];
    if (!W::kTable && w.cnt[0]) atomicAdd(&c.st->n_big, (unsigned long long)w.cnt[0]);
#pragma unroll 1
    for (int k = 0; k < 8; ++k)
      if (w.cnt[k]) atomicAdd(dst[k], (unsigned long long)w.cnt[k]);
  }
}

}  // namespace
}  // namespace dtg
