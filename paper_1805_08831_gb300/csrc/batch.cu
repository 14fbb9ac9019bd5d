// Batches of independent clouds on the asynchronous engine.
//
// Every cloud is a mesh of its own in its own range of the tetrahedron store, with its own
// allocator, queues and hint grid, and all clouds grow together: launch k inserts the k-th wave of
// every cloud that has one (the waves of Section 2.3's rounds, contiguous ranges of the (cloud,
// round, wave, key) order), each warp a Moore segment of one cloud after its share of the points
// that cloud carries over. The segments follow from the cloud sizes alone, so the whole batch is
// one fixed sequence of launches without a host in between, captured into a graph. A warp that
// meets another holds nothing up, so clouds of all sizes share the chip: the one-block-per-cloud
// kernel before this ran each cloud in rounds between block barriers and waited for its largest
// cloud (512 clouds of 50 to 50000 points: 271 ms).
#include <cuda_runtime.h>

#include <algorithm>

namespace dtg {
constexpr int kADefer = 16;  // aborted points waiting for a retry
}

#include "async.cuh"

namespace dtg {

namespace {

// Hint grid of a cloud: 8 x 8 x 8 fine cells, 2 x 2 x 2 coarse cells.
constexpr int kBatchCb = 3;
constexpr uint32_t kBatchFine = 1u << (3 * kBatchCb);
constexpr uint32_t kBatchCoarse = 8;

// Queue indexes of a cloud's state (DevState::q).
__device__ __forceinline__ int list_queue(int k) { return k == 0 ? 0 : 6; }
constexpr int kQLarge = 1, kQBeyond = 3;

using BatchBigWS = AWS<65536, 16384, 16384, 16384, 65536, false>;

// The engine's context of one cloud.
__device__ __forceinline__ Ctx cloud_ctx(const Ctx& c0, const BatchMem& b, uint32_t ci) {
  const BatchCloud* cl = b.clouds + ci;
  Ctx c = c0;
  c.eta = *b.eta;
  c.st = b.states + ci;
  c.freelist = c0.freelist + cl->tb;
  c.pending = c0.pending + cl->tb;
  c.cell_hint = b.hint_fine + (size_t)ci * kBatchFine;
  c.cell_hint2 = b.hint_coarse + (size_t)ci * kBatchCoarse;
  for (int d = 0; d < 3; ++d) {
    c.lo[d] = cl->lo[d];
    c.sc[d] = cl->sc[d];
  }
  c.cb = kBatchCb;
  c.tbase = cl->tb;
  c.ntets = cl->tb + cl->tcap;
  c.npts = cl->ve;
  return c;
}

// A fresh state for every cloud (one block each), then its first tetrahedra.
__global__ void k_batch_init(Ctx c0, BatchMem b) {
  const uint32_t ci = blockIdx.x;
  BatchCloud* cl = b.clouds + ci;
  DevState* st = b.states + ci;
  for (uint32_t i = threadIdx.x; i < sizeof(DevState) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(st)[i] = 0;
  for (uint32_t i = threadIdx.x; i < kBatchFine; i += blockDim.x) b.hint_fine[(size_t)ci * kBatchFine + i] = kNone;
  if (threadIdx.x < kBatchCoarse) b.hint_coarse[(size_t)ci * kBatchCoarse + threadIdx.x] = kNone;
  // (the vertex records' kernel wrote the same values; without this loop and its pointer k_batch is
  // compiled to more spills, and 512 clouds take 73.0 ms instead of 70.2)
  for (uint32_t v = cl->vb + threadIdx.x; v < cl->ve; v += blockDim.x) {
    b.vflag[v] = b.dup[v];
    c0.point_hint[v] = kNone;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  st->bump = cl->tb;
  st->capacity = (unsigned long long)cl->tb + cl->tcap;
  st->free_capacity = cl->tcap;
  st->anchor = cl->tb;
  __threadfence();
  if (*b.bad) {
    cl->status = (uint32_t)kErrDegenerate;
    return;
  }
  const Ctx c = cloud_ctx(c0, b, ci);
  cl->status = init_mesh(c, cl->vb, cl->ve, b.vflag, cl->tb) ? 0u : (uint32_t)kErrDegenerate;
}

__device__ __forceinline__ AsyncIO cloud_io(const Ctx& c, const BatchMem& b, const BatchCloud* cl, int src) {
  AsyncIO io{};
  io.vflag = b.vflag;
  io.max_walk = c.max_walk;
  io.carry = b.list[src] + cl->vb;
  io.carry_n = __ldcg(&c.st->q[list_queue(src)]);
  io.lose_out = b.list[1 - src] + cl->vb;
  io.lose_q = list_queue(1 - src);
  io.big_out = b.list_big + cl->vb;
  io.big_q = kQLarge;
  io.big_ws = b.big_ws;
  io.big_busy = b.big_busy;
  io.big_n = b.big_n;
  io.ball_start = 1;
  return io;
}

// One warp per segment. All predicate stages: a cloud of any kind stays in the one sequence.
template <int kThreads, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_batch(Ctx c0, BatchMem b, const uint4* __restrict__ segs,
                                                                uint32_t n, int src) {
  extern __shared__ __align__(16) char s_mem[];
  const uint32_t wid = threadIdx.x >> 5, seg = blockIdx.x * (blockDim.x >> 5) + wid;
  if (seg >= n) return;
  const uint4 sg = segs[seg];
  const BatchCloud* cl = b.clouds + sg.x;
  if (cl->status != 0) return;
  const Ctx c = cloud_ctx(c0, b, sg.x);
  const AsyncIO io = cloud_io(c, b, cl, src);
  const uint32_t idx = sg.w & 0xFFFFu, W = sg.w >> 16;
  run_segment<true>(c, io, reinterpret_cast<SmallWST<false>*>(s_mem)[wid], b.lock, seg + 1, sg.y, sg.z,
                    (uint32_t)(io.carry_n * idx / W), (uint32_t)(io.carry_n * (idx + 1) / W), InsertLog{nullptr, nullptr});
}

// Large cavities waiting: warp w takes the clouds w, w + n, ... one after the other.
__global__ void __launch_bounds__(32) k_batch_big(Ctx c0, BatchMem b, BatchBigWS* ws, int src) {
  for (uint32_t ci = blockIdx.x; ci < b.n_clouds; ci += gridDim.x) {
    const BatchCloud* cl = b.clouds + ci;
    if (cl->status != 0) continue;
    const Ctx c = cloud_ctx(c0, b, ci);
    const uint64_t n = __ldcg(&c.st->q[kQLarge]);
    if (n == 0) continue;
    AsyncIO io = cloud_io(c, b, cl, src);
    io.carry = b.list_big + cl->vb;
    io.lose_out = b.list[src] + cl->vb;  // with the points that wait there
    io.lose_q = list_queue(src);
    io.big_out = b.list[1 - src] + cl->vb;
    io.big_q = kQBeyond;
    run_segment<true>(c, io, ws[blockIdx.x], b.lock, blockIdx.x + 1, 0, 0, 0, (uint32_t)n, InsertLog{nullptr, nullptr});
    __syncwarp();
    if (threadIdx.x == 0) {
      c.st->q[kQLarge] = 0;
      if (__ldcg(&c.st->q[kQBeyond])) raise_error(c.st, kErrBigCavity, (unsigned)n);
    }
  }
}

// Closes a launch: every cloud's allocator, and its consumed list.
__global__ void k_batch_close(Ctx c0, BatchMem b, int consumed) {
  const uint32_t ci = blockIdx.x;
  if (b.clouds[ci].status != 0) return;
  const Ctx c = cloud_ctx(c0, b, ci);
  finish_round_block(c);
  if (threadIdx.x == 0 && consumed >= 0) c.st->q[list_queue(consumed)] = 0;
}

__global__ void k_batch_finish(BatchMem b, int src) {
  for (uint32_t ci = blockIdx.x * blockDim.x + threadIdx.x; ci < b.n_clouds; ci += gridDim.x * blockDim.x) {
    BatchCloud* cl = b.clouds + ci;
    const DevState* st = b.states + ci;
    if (cl->status != kErrDegenerate) cl->status = st->error;
    cl->info = st->error_info;
    const bool ok = cl->status == 0;
    cl->used = ok ? (uint32_t)(st->bump - cl->tb) : 0u;
    cl->inserted = ok ? (uint32_t)st->n_inserted : 0u;
    const unsigned long long v[kBatchTotals] = {ok ? st->n_inserted : 0ull, st->n_conflicts, st->n_attempts,
                                                st->sum_cavity, st->sum_ball, st->sum_walk, ok ? st->q[kQLarge] : 0ull,
                                                ok ? st->q[list_queue(src)] : 0ull, st->n_dups, st->n_exact, st->n_sos,
                                                st->n_big};
    for (int k = 0; k < kBatchTotals; ++k)
      if (v[k]) atomicAdd(&b.totals[k], v[k]);
  }
}

// Finite tetrahedra of every cloud, vertex ids local to the cloud. Pass 0 counts per cloud;
// pass 1 writes from out_off[cloud] (one block per cloud, order inside a cloud unspecified).
__global__ void k_batch_collect(const BatchCloud* clouds, uint32_t n_clouds, const Tet* __restrict__ tets,
                                const Pt* __restrict__ pts, const uint64_t* __restrict__ in_off, int pass,
                                unsigned long long* counts, const unsigned long long* out_off, uint32_t* out,
                                int canonical) {
  for (uint32_t ci = blockIdx.x; ci < n_clouds; ci += gridDim.x) {
    const BatchCloud cl = clouds[ci];
    if (cl.status != 0) continue;
    unsigned long long pos = 0;
    for (uint64_t t0 = 0; t0 < cl.used; t0 += blockDim.x) {
      uint64_t t = t0 + threadIdx.x;
      bool keep = false;
      uint32_t r[4] = {0, 0, 0, 0};
      if (t < cl.used) {
        uint4 v = tets[cl.tb + t].v;
        keep = !tet_dead(v) && ghost_pos(v) < 0;
        if (keep) {
          r[0] = (uint32_t)((uint64_t)pts[v.x].w - in_off[ci]);
          r[1] = (uint32_t)((uint64_t)pts[v.y].w - in_off[ci]);
          r[2] = (uint32_t)((uint64_t)pts[v.z].w - in_off[ci]);
          r[3] = (uint32_t)((uint64_t)pts[v.w].w - in_off[ci]);
          if (canonical) canonical_rotation(r);
        }
      }
      unsigned bal = __ballot_sync(kFull, keep);
      __shared__ unsigned s_w[32];
      __shared__ unsigned long long s_base;
      const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
      if (lane == 0) s_w[wid] = __popc(bal);
      __syncthreads();
      if (threadIdx.x == 0) {
        unsigned long long acc = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
          unsigned x = s_w[w];
          s_w[w] = (unsigned)acc;
          acc += x;
        }
        s_base = pos;
        pos += acc;
      }
      __syncthreads();
      if (pass == 1 && keep) {
        unsigned long long at = out_off[ci] + s_base + s_w[wid] + __popc(bal & ((1u << lane) - 1u));
        reinterpret_cast<uint4*>(out)[at] = make_uint4(r[0], r[1], r[2], r[3]);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0 && pass == 0) counts[ci] = pos;
  }
}


// Hint grid of every cloud (8 cells per axis over its box) and the batch's FP32 error term
// eta = 2^-44 max|x| (+ the spacing of FP32 subnormals), as the single-cloud engine sets it.
__global__ void k_batch_prepare(BatchCloud* clouds, const double* __restrict__ cbox, uint32_t n_clouds,
                                float* eta) {
  __shared__ double s_max[256];
  double m = 0.0;
  for (uint32_t c = threadIdx.x; c < n_clouds; c += blockDim.x) {
    if (clouds[c].vb == clouds[c].ve) continue;  // its box is (inf, -inf)
    const double* B = cbox + 6ull * c;
    for (int k = 0; k < 6; ++k) m = fmax(m, fabs(B[k]));
    for (int k = 0; k < 3; ++k) {
      double ext = B[3 + k] - B[k];
      clouds[c].lo[k] = (float)B[k];
      clouds[c].sc[k] = ext > 0 ? (float)((double)(1u << kBatchCb) / ext) : 0.f;
    }
  }
  s_max[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) s_max[threadIdx.x] = fmax(s_max[threadIdx.x], s_max[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *eta = (float)(ldexp(s_max[0], -44) * 1.0001 + 1e-38);
}

}  // namespace

uint32_t batch_hint_fine() { return kBatchFine; }
uint32_t batch_hint_coarse() { return kBatchCoarse; }
size_t batch_big_ws_bytes() { return sizeof(BatchBigWS); }

bool batch_ready() {
  return cudaFuncSetAttribute(k_batch<1024, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              32 * (int)sizeof(SmallWST<false>)) == cudaSuccess;
}

void batch_init(const Ctx& c, const BatchMem& b, cudaStream_t s) {
  k_batch_init<<<b.n_clouds, 128, 0, s>>>(c, b);
  ++g_kernel_launches;
}

// Blocks of 4 warps unless more are asked for: with 128 registers (4 resident blocks per SM) for a
// launch that fits the chip so, where the length of one insertion counts (64 small clouds: 4.8 ms
// against 5.3), else with 80 (6 blocks; 512 clouds: 70.6 ms against 74.0).
int batch_min_blocks(int warps, uint64_t n) {
  return warps > 4 ? 1 : (n + warps - 1) / warps <= 152u * 4 ? 4 : 6;
}

int batch_launch(int warps, const Ctx& c, const BatchMem& b, const uint4* segs, uint32_t n, int src, cudaStream_t s) {
  const size_t smem = (size_t)warps * sizeof(SmallWST<false>);
  if (warps < 1 || warps > 32) return DT_EINVAL;
  const unsigned blocks = (n + warps - 1) / warps;
  switch (batch_min_blocks(warps, n)) {
    case 4: k_batch<128, 4><<<blocks, warps * 32, smem, s>>>(c, b, segs, n, src); break;
    case 6: k_batch<128, 6><<<blocks, warps * 32, smem, s>>>(c, b, segs, n, src); break;
    default: k_batch<1024, 1><<<blocks, warps * 32, smem, s>>>(c, b, segs, n, src);
  }
  k_batch_close<<<b.n_clouds, 128, 0, s>>>(c, b, src);
  g_kernel_launches += 2;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

int batch_launch_big(const Ctx& c, const BatchMem& b, void* ws, uint32_t n, int src, cudaStream_t s) {
  k_batch_big<<<std::min(n, b.n_clouds), 32, 0, s>>>(c, b, static_cast<BatchBigWS*>(ws), src);
  k_batch_close<<<b.n_clouds, 128, 0, s>>>(c, b, -1);
  g_kernel_launches += 2;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

void batch_finish(const Ctx&, const BatchMem& b, int src, cudaStream_t s) {
  cudaMemsetAsync(b.totals, 0, kBatchTotals * sizeof(unsigned long long), s);
  k_batch_finish<<<(b.n_clouds + 127) / 128, 128, 0, s>>>(b, src);
  ++g_kernel_launches;
}

void batch_prepare(BatchCloud* clouds, const double* cbox, uint32_t n_clouds, float* eta, cudaStream_t s) {
  k_batch_prepare<<<1, 256, 0, s>>>(clouds, cbox, n_clouds, eta);
  ++g_kernel_launches;
}

void batch_collect(const BatchCloud* clouds, uint32_t n_clouds, const Tet* tets, const Pt* pts, const uint64_t* in_off,
                   int pass, unsigned long long* counts, const unsigned long long* out_off, uint32_t* out,
                   int canonical, cudaStream_t s) {
  k_batch_collect<<<std::min<uint32_t>(n_clouds, 152u * 8), 256, 0, s>>>(clouds, n_clouds, tets, pts, in_off, pass,
                                                                        counts, out_off, out, canonical);
  ++g_kernel_launches;
}

}  // namespace dtg
