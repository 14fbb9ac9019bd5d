// Launches of the asynchronous insertion engine (async.cuh) on one mesh.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

namespace dtg {
constexpr int kADefer = 16;  // aborted points waiting for a retry
}

#include "async.cuh"
#include "per_device.h"

namespace dtg {
namespace {

template <int kMinBlocks, bool kCache = false, bool kExact = false>
__global__ void __launch_bounds__(kAW * 32, kMinBlocks) k_async(Ctx c, AsyncIO io, uint32_t* lock, InsertLog lg) {
  __shared__ SmallWST<kCache> s_ws[kAW];
  const int wid = threadIdx.x >> 5;
  const uint32_t seg = blockIdx.x * kAW + wid;
  if (seg >= io.W) return;
  uint64_t b0, e0;
  if (io.bounds && io.m) {  // segments of equal predicted work (the learned schedule)
    b0 = io.bounds[seg];
    e0 = io.bounds[seg + 1];
  } else {
    b0 = (uint64_t)seg * io.L;
    e0 = b0 + io.L < io.m ? b0 + io.L : io.m;
    if (b0 > e0) b0 = e0;
  }
  run_segment<kExact>(c, io, s_ws[wid], lock, seg + 1, (uint32_t)b0, (uint32_t)e0, (uint32_t)(io.carry_n * seg / io.W),
                      (uint32_t)(io.carry_n * (seg + 1) / io.W), lg);
}

// A launch of at most kLocalWarps warps on a mesh of at most a few hundred vertices: one block, the
// mesh read and written through its SM's L1 (async.cuh, ld_mesh). An insertion that runs alone is a
// chain of some thirty dependent reads, 13.5 us of them through L2.
constexpr uint32_t kLocalWarps = 16;

template <bool kExact>
__global__ void __launch_bounds__(kLocalWarps * 32, 1) k_async_local(Ctx c, AsyncIO io, uint32_t* lock, InsertLog lg) {
  extern __shared__ __align__(16) char s_mem[];
  const uint32_t seg = threadIdx.x >> 5;
  const uint64_t b0 = std::min<uint64_t>(seg * io.L, io.m), e0 = std::min<uint64_t>(b0 + io.L, io.m);
  run_segment<kExact>(c, io, reinterpret_cast<SmallWST<false, true>*>(s_mem)[seg], lock, seg + 1, (uint32_t)b0,
                      (uint32_t)e0, (uint32_t)(io.carry_n * seg / io.W), (uint32_t)(io.carry_n * (seg + 1) / io.W), lg);
}

// Large cavities (beyond the shared-memory workspaces): the same insertion with each warp's
// workspace in global memory.
template <bool kCache, bool kExact>
__global__ void __launch_bounds__(128) k_async_big(Ctx c, AsyncIO io, uint32_t* lock, InsertLog lg,
                                                  HugeWST<kCache>* ws) {
  const uint32_t seg = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (seg >= io.W) return;
  run_segment<kExact>(c, io, ws[seg], lock, seg + 1, 0, 0, (uint32_t)(io.carry_n * seg / io.W),
                      (uint32_t)(io.carry_n * (seg + 1) / io.W), lg);
}

// Folds the allocator of the launch into the free list, as a round close does
// (finish_round_block): the slots freed during the launch (pending) follow the free-list
// entries it did not consume. Copy on the whole grid, then the state on one thread.
__global__ void k_async_close_copy(Ctx c) {
  const DevState* st = c.st;
  const unsigned long long used = __ldcg(&st->alloc_cursor), fa = __ldcg(&st->free_avail);
  const unsigned long long consumed = used < fa ? used : fa, nfa = fa - consumed;
  unsigned long long np = __ldcg(&st->pending);
  if (nfa + np > st->free_capacity) np = st->free_capacity - nfa;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < np;
       i += (unsigned long long)gridDim.x * blockDim.x)
    c.freelist[nfa + i] = __ldcg(&c.pending[i]);
}

__global__ void k_async_close_state(Ctx c, int consumed_q) {
  DevState* st = c.st;
  if (consumed_q >= 0) st->q[consumed_q] = 0;  // the launch took the whole list
  const unsigned long long used = st->alloc_cursor, fa = st->free_avail;
  const unsigned long long consumed = used < fa ? used : fa, nfa = fa - consumed;
  unsigned long long np = st->pending;
  if (nfa + np > st->free_capacity) {
    raise_error(st, kErrFreeList, 0xAAu);
    np = st->free_capacity - nfa;
  }
  st->bump += used - consumed;
  st->free_avail = nfa + np;
  st->alloc_cursor = 0;
  st->pending = 0;
  st->stamp += 1;
  st->blocks_done = 0;
}

// Resident blocks per SM the kernels are built for. The FP32 kernel: 8 (32 warps per SM at 64
// registers) for launches that fill the chip, where it measured fastest (255 ms per 1e7 uniform step
// when first built against 265 at 6, 276 at 5 and 301 at 4), 4 (128 registers, no spills) for
// launches that fit the chip with that, where the latency of one insertion is what counts. The
// kernel with the exact stages: 4, its calls save and restore fewer registers.
constexpr int kFullBlocks = 8, kFewBlocks = 4, kExactBlocks = 4;

int current_device() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess ? dev : 0;
}

// Warps of the kernel that are resident on the current device at once.
template <int kMinBlocks, bool kCache = false, bool kExact = false>
int resident_warps() {
  static PerDevice kept;
  const int dev = current_device();
  return (int)kept.get(dev, [dev] {
    int sms = 0, per = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_async<kMinBlocks, kCache, kExact>, kAW * 32, 0) !=
        cudaSuccess)
      per = kMinBlocks;
    return std::max(1, sms * std::max(per, 1) * kAW);
  });
}

}  // namespace

int async_launch(const Ctx& c, const AsyncIO& io, uint32_t* lock, const InsertLog& lg, cudaStream_t s) {
  if (io.W == 0 || (io.m == 0 && io.carry_n == 0)) return DT_OK;
  Ctx cc = c;
  cc.coherent = 1;
  cc.max_walk = io.max_walk;
  const unsigned blocks = (io.W + kAW - 1) / kAW;
  const size_t local = io.W * sizeof(SmallWST<false, true>);
  if (io.local && io.exact) k_async_local<true><<<1, io.W * 32, local, s>>>(cc, io, lock, lg);
  else if (io.local) k_async_local<false><<<1, io.W * 32, local, s>>>(cc, io, lock, lg);
  else if (io.exact) k_async<kExactBlocks, false, true><<<blocks, kAW * 32, 0, s>>>(cc, io, lock, lg);
  else if (c.subdet) k_async<kFullBlocks, true><<<blocks, kAW * 32, 0, s>>>(cc, io, lock, lg);
  else if (io.W <= (uint32_t)resident_warps<kFewBlocks>()) k_async<kFewBlocks><<<blocks, kAW * 32, 0, s>>>(cc, io, lock, lg);
  else k_async<kFullBlocks><<<blocks, kAW * 32, 0, s>>>(cc, io, lock, lg);
  k_async_close_copy<<<152, 256, 0, s>>>(cc);
  k_async_close_state<<<1, 1, 0, s>>>(cc, io.carry_n ? io.carry_q : -1);
  g_kernel_launches += 3;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

size_t async_borrow_ws_bytes() { return sizeof(LargeWS); }
size_t async_big_ws_bytes() { return sizeof(HugeWST<false>); }

int async_launch_big(const Ctx& c, const AsyncIO& io, uint32_t* lock, const InsertLog& lg, void* ws, cudaStream_t s) {
  if (io.W == 0 || io.carry_n == 0) return DT_OK;
  Ctx cc = c;
  cc.coherent = 1;
  cc.max_walk = io.max_walk;
  HugeWST<false>* w = static_cast<HugeWST<false>*>(ws);
  if (io.exact) k_async_big<false, true><<<(io.W + 3) / 4, 128, 0, s>>>(cc, io, lock, lg, w);
  else k_async_big<false, false><<<(io.W + 3) / 4, 128, 0, s>>>(cc, io, lock, lg, w);
  k_async_close_copy<<<152, 256, 0, s>>>(cc);
  k_async_close_state<<<1, 1, 0, s>>>(cc, io.carry_q);
  g_kernel_launches += 3;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

// Most warps of a launch that runs as one block (AsyncIO::local) on the current device, 0 if it cannot.
uint32_t async_local_warps() {
  static PerDevice kept;
  return (uint32_t)kept.get(current_device(), [] {
    const int bytes = (int)(kLocalWarps * sizeof(SmallWST<false, true>));
    const auto opt_in = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_async_local<false>, opt_in, bytes) == cudaSuccess &&
                   cudaFuncSetAttribute(k_async_local<true>, opt_in, bytes) == cudaSuccess
               ? kLocalWarps
               : 0u;
  });
}

int async_max_warps() { return resident_warps<kFullBlocks>(); }

int async_max_warps_exact() { return std::min(resident_warps<kExactBlocks, false, true>(), async_max_warps()); }

}  // namespace dtg
