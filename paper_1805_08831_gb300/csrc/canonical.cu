// The canonical tetrahedron list: live finite tetrahedra with input vertex ids, each in its
// canonical rotation (smallest id first), the rows in lexicographic order.
//
// The rows are sorted as a bucket sort on the first id and a comparison sort inside the buckets:
// a tetrahedron's first id is its smallest, and the rows that share it are few (6.8 on average,
// 16 as a row meets them, in a uniform cloud). One pass over the slots writes the rotated rows
// and takes each row's place in its bucket from the atomic that counts it; a prefix sum of the
// counts says where the buckets start; one scattered write per row puts it into its bucket; and
// a block then orders the buckets of a run of rows in shared memory, each row's rank being the
// number of smaller rows in its bucket. That is 5 passes over the rows where an LSD radix sort
// of the four ids makes 16 of 24 bytes per row.
//
// A bucket of more than kBucketMax rows (a vertex with a huge star: the centre of a sphere of
// points) would cost its square: the rows of such buckets alone go through the radix sort.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "engine.cuh"
#include "internal.h"

namespace dtg {
namespace {

constexpr int kCollectThreads = 256, kCollectItems = 4;  // slots per block: 1024
constexpr uint32_t kTileRows = 1024;   // rows whose buckets a block orders
constexpr uint32_t kBucketMax = 1024;  // rows of the largest bucket ordered in shared memory
constexpr int kOrderThreads = 256;
constexpr int kOrderItems = (int)((kTileRows + kBucketMax) / kOrderThreads);

unsigned grid_of(uint64_t n, int per_block, unsigned most) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + per_block - 1) / per_block, most));
}

// Input index of every vertex: 4 bytes each, so the gathers below stay in L2 (40 MB at 1e7
// points) where the 32-byte point records would not.
__global__ void k_input_ids(const Pt* __restrict__ pts, uint64_t n, uint32_t* ids) {
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
    ids[v] = (uint32_t)pts[v].w;
}

// Whether a slot of a batch holds a tetrahedron of a triangulated cloud. The clouds' slot ranges
// ascend, so a thread's cloud only moves forward: *ci is where its last slot was.
__device__ __forceinline__ bool batch_slot(const BatchCloud* __restrict__ clouds, uint32_t n_clouds, uint64_t t,
                                           uint32_t* ci) {
  uint32_t lo = *ci, step = 1;
  while (lo + step < n_clouds && clouds[lo + step].tb <= t) {  // gallop, then halve
    lo += step;
    step <<= 1;
  }
  for (; step > 0; step >>= 1)
    if (lo + step < n_clouds && clouds[lo + step].tb <= t) lo += step;
  *ci = lo;
  return clouds[lo].status == 0 && t - clouds[lo].tb < clouds[lo].used;
}

// Live finite tetrahedra of slots [0, nslots): counted into count[0]; with rows != null also
// written as canonical rows of input ids, in any order, each with its place in the bucket of
// its first id (the buckets' sizes into cnt). count[1] becomes 1 when a bucket outgrows
// kBucketMax. One update of the row counter per block of 1024 slots.
template <bool kBatch>
__global__ void __launch_bounds__(kCollectThreads) k_canon_collect(
    const Tet* __restrict__ tets, uint64_t nslots, const uint32_t* __restrict__ ids, uint64_t npts,
    const BatchCloud* __restrict__ clouds, uint32_t n_clouds, uint4* rows, uint32_t* place, uint32_t* cnt,
    unsigned long long* count) {
  __shared__ unsigned s_warp[kCollectThreads / 32];
  __shared__ unsigned long long s_base;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  uint32_t ci = 0;
  const uint64_t tile = (uint64_t)kCollectThreads * kCollectItems;
  for (uint64_t t0 = blockIdx.x * tile; t0 < nslots; t0 += gridDim.x * tile) {
    uint4 v[kCollectItems];
    bool keep[kCollectItems];
    unsigned mine[kCollectItems], total = 0;  // this lane's rank among the warp's rows, per item
#pragma unroll
    for (int k = 0; k < kCollectItems; ++k) {
      const uint64_t t = t0 + (uint64_t)k * kCollectThreads + tid;
      keep[k] = t < nslots && (!kBatch || batch_slot(clouds, n_clouds, t, &ci));
      if (keep[k]) {
        v[k] = tets[t].v;
        keep[k] = !tet_dead(v[k]) && ghost_pos(v[k]) < 0 && v[k].x < npts && v[k].y < npts && v[k].z < npts &&
                  v[k].w < npts;
      }
    }
#pragma unroll
    for (int k = 0; k < kCollectItems; ++k) {
      const unsigned m = __ballot_sync(kFull, keep[k]);
      mine[k] = total + __popc(m & lanemask_lt());
      total += __popc(m);
    }
    if (lane == 0) s_warp[wid] = total;
    __syncthreads();
    if (tid == 0) {
      unsigned all = 0;
      for (int w = 0; w < kCollectThreads / 32; ++w) {
        const unsigned x = s_warp[w];
        s_warp[w] = all;
        all += x;
      }
      s_base = all ? atomicAdd(&count[0], (unsigned long long)all) : 0ull;
    }
    __syncthreads();
    if (rows) {
      const unsigned long long base = s_base + s_warp[wid];
#pragma unroll
      for (int k = 0; k < kCollectItems; ++k) {
        if (!keep[k]) continue;
        uint32_t r[4] = {ids[v[k].x], ids[v[k].y], ids[v[k].z], ids[v[k].w]};
        canonical_rotation(r);
        const uint32_t at = atomicAdd(&cnt[r[0]], 1u);
        if (at == kBucketMax) count[1] = 1ull;
        rows[base + mine[k]] = make_uint4(r[0], r[1], r[2], r[3]);
        place[base + mine[k]] = at;
      }
    }
    __syncthreads();  // s_warp and s_base are written again by the next tile
  }
}

__global__ void k_canon_scatter(const uint4* __restrict__ rows, const uint32_t* __restrict__ place, uint64_t T,
                                const uint32_t* __restrict__ first, uint4* out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < T; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 r = rows[i];
    out[(uint64_t)first[r.x] + place[i]] = r;
  }
}

// The rows [x, y) that tile b of kTileRows rows orders: the buckets that start in it, without
// one that is larger than kBucketMax (it can only be the last).
__global__ void k_canon_bounds(const uint4* __restrict__ in, uint64_t T, const uint32_t* __restrict__ first, uint64_t nt,
                               uint2* bounds) {
  for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < nt; b += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t i0 = b * kTileRows, i1 = i0 + kTileRows;
    uint32_t a = in[i0].x;
    const uint32_t lo = first[a] == i0 ? (uint32_t)i0 : first[a + 1];
    uint32_t hi = (uint32_t)T;
    if (i1 < T) {
      a = in[i1].x;
      const uint32_t s = first[a], e = first[a + 1];
      hi = (s == i1 || e - s > kBucketMax) ? s : e;
    }
    bounds[b] = make_uint2(lo, hi);
  }
}

__device__ __forceinline__ bool row_less(const uint4& p, const uint4& q) {  // rows of one bucket
  return p.y < q.y || (p.y == q.y && (p.z < q.z || (p.z == q.z && p.w < q.w)));
}

// Orders the buckets of one tile (in and out may be the same rows: a tile's rows are its own).
// cid and in_off (a batch): the cloud of every input index and the clouds' first input indices,
// subtracted so that a cloud's ids are its own.
__global__ void __launch_bounds__(kOrderThreads) k_canon_order(const uint4* in, uint4* out,
                                                               const uint2* __restrict__ bounds,
                                                               const uint32_t* __restrict__ first,
                                                               const uint32_t* __restrict__ cid,
                                                               const uint64_t* __restrict__ in_off) {
  __shared__ uint4 tile[kTileRows + kBucketMax];
  const uint2 b = bounds[blockIdx.x];
  if (b.x >= b.y) return;
  const int n = (int)(b.y - b.x);
  for (int i = threadIdx.x; i < n; i += kOrderThreads) tile[i] = in[(uint64_t)b.x + i];
  __syncthreads();
  uint4 r[kOrderItems];
  int at[kOrderItems];
#pragma unroll
  for (int k = 0; k < kOrderItems; ++k) {
    const int i = threadIdx.x + k * kOrderThreads;
    at[k] = -1;
    if (i < n) {
      r[k] = tile[i];
      const int s = (int)(first[r[k].x] - b.x), e = (int)(first[r[k].x + 1] - b.x);
      int rank = s;
      for (int j = s; j < e; ++j) rank += row_less(tile[j], r[k]) ? 1 : 0;
      at[k] = rank;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kOrderItems; ++k)
    if (at[k] >= 0) {
      if (in_off) {
        const uint32_t o = (uint32_t)in_off[cid[r[k].x]];
        r[k] = make_uint4(r[k].x - o, r[k].y - o, r[k].z - o, r[k].w - o);
      }
      tile[at[k]] = r[k];
    }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kOrderThreads) out[(uint64_t)b.x + i] = tile[i];
}

// ------------------------------------------------------------------ buckets beyond kBucketMax
// Their rows, in any order: counted with big == null, else written to big.
__global__ void k_canon_big(const uint4* __restrict__ rows, uint64_t T, const uint32_t* __restrict__ first,
                            unsigned long long* count, uint4* big) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < T; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 r = rows[i];
    if (first[r.x + 1] - first[r.x] <= kBucketMax) continue;
    const unsigned long long at = atomicAdd(count, 1ull);
    if (big) big[at] = r;
  }
}

__global__ void k_split_keys(const uint4* rows, uint64_t T, uint64_t* khi, uint64_t* klo, uint32_t* idx) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < T; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 t = rows[i];
    khi[i] = ((uint64_t)t.x << 32) | t.y;
    klo[i] = ((uint64_t)t.z << 32) | t.w;
    idx[i] = (uint32_t)i;
  }
}

__global__ void k_gather_keys(const uint64_t* src, const uint32_t* idx, uint64_t T, uint64_t* dst) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < T; i += (uint64_t)gridDim.x * blockDim.x)
    dst[i] = src[idx[i]];
}

// Row j of the sorted order belongs to bucket a = its first id, whose rows start at the first
// sorted row with that id (a binary search on the sorted keys).
__global__ void k_place_big(const uint4* __restrict__ big, const uint64_t* __restrict__ keys,
                            const uint32_t* __restrict__ idx, uint64_t m, const uint32_t* __restrict__ first,
                            const uint32_t* __restrict__ cid, const uint64_t* __restrict__ in_off, uint4* out) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < m; j += (uint64_t)gridDim.x * blockDim.x) {
    uint4 r = big[idx[j]];
    uint64_t lo = 0, hi = j;  // the first row of j's bucket lies in [lo, hi]
    while (lo < hi) {
      const uint64_t mid = (lo + hi) / 2;
      if ((uint32_t)(keys[mid] >> 32) < r.x) lo = mid + 1;
      else hi = mid;
    }
    const uint64_t at = (uint64_t)first[r.x] + (j - lo);
    if (in_off) {
      const uint32_t o = (uint32_t)in_off[cid[r.x]];
      r = make_uint4(r.x - o, r.y - o, r.z - o, r.w - o);
    }
    out[at] = r;
  }
}

// Where every cloud's rows start: its first input index's bucket.
__global__ void k_cloud_starts(const uint32_t* __restrict__ first, const uint64_t* __restrict__ in_off,
                               uint32_t n_clouds, unsigned long long* starts) {
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c <= n_clouds; c += gridDim.x * blockDim.x)
    starts[c] = first[in_off[c]];
}

int order_big(const uint4* rows, uint64_t T, const CanonWS& w, const uint32_t* cid, const uint64_t* in_off, uint4* out,
              cudaStream_t s) {
  unsigned long long m = 0;
  cudaMemsetAsync(w.count, 0, 8, s);
  k_canon_big<<<grid_of(T, 256, 152u * 16), 256, 0, s>>>(rows, T, w.first, w.count, nullptr);
  cudaMemcpyAsync(&m, w.count, 8, cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return DT_ECUDA;
  uint4* big = nullptr;
  uint64_t *khi = nullptr, *klo = nullptr, *ka = nullptr;
  uint32_t *idx = nullptr, *ia = nullptr, *hist = nullptr;
  const bool ok = cudaMalloc(&big, m * 16) == cudaSuccess && cudaMalloc(&khi, m * 8) == cudaSuccess &&
                  cudaMalloc(&klo, m * 8) == cudaSuccess && cudaMalloc(&ka, m * 8) == cudaSuccess &&
                  cudaMalloc(&idx, m * 4) == cudaSuccess && cudaMalloc(&ia, m * 4) == cudaSuccess &&
                  cudaMalloc(&hist, radix_hist_entries(m) * 4) == cudaSuccess;
  int rc = DT_OK;
  if (ok) {
    const unsigned g = grid_of(m, 256, 152u * 16);
    cudaMemsetAsync(w.count, 0, 8, s);
    k_canon_big<<<grid_of(T, 256, 152u * 16), 256, 0, s>>>(rows, T, w.first, w.count, big);
    // stable LSD passes on (c, d), then (a, b)
    k_split_keys<<<g, 256, 0, s>>>(big, m, khi, klo, idx);
    const bool alt = radix_sort_pairs(klo, idx, ka, ia, m, 64, hist, s);
    uint32_t *order = alt ? ia : idx, *other = alt ? idx : ia;
    k_gather_keys<<<g, 256, 0, s>>>(khi, order, m, ka);
    const bool alt2 = radix_sort_pairs(ka, order, klo, other, m, 64, hist, s);
    k_place_big<<<g, 256, 0, s>>>(big, alt2 ? klo : ka, alt2 ? other : order, m, w.first, cid, in_off, out);
    g_kernel_launches += 5;
    if (cudaStreamSynchronize(s) != cudaSuccess) rc = DT_ECUDA;
  } else {
    cudaGetLastError();
    rc = DT_ENOMEM;
  }
  cudaFree(big);
  cudaFree(khi);
  cudaFree(klo);
  cudaFree(ka);
  cudaFree(idx);
  cudaFree(ia);
  cudaFree(hist);
  return rc;
}

}  // namespace

void canon_ws_free(CanonWS& w) {
  cudaFree(w.ids);
  cudaFree(w.first);
  cudaFree(w.scan);
  cudaFree(w.count);
  w = CanonWS();
}

uint64_t canon_ws_bytes(const CanonWS& w) { return w.cap * 8 + w.scan_cap * 4 + (w.count ? 16 : 0); }

int canon_ws_reserve(CanonWS& w, uint64_t npts) {
  if (!w.count && cudaMalloc(&w.count, 16) != cudaSuccess) return DT_ENOMEM;
  const uint64_t need = npts + 1;
  if (need <= w.cap) return DT_OK;
  cudaFree(w.ids);
  cudaFree(w.first);
  cudaFree(w.scan);
  w.ids = w.first = w.scan = nullptr;
  w.cap = w.scan_cap = 0;
  const uint64_t scan = prefix_scratch_entries(need);
  if (cudaMalloc(&w.ids, need * 4) != cudaSuccess || cudaMalloc(&w.first, need * 4) != cudaSuccess ||
      cudaMalloc(&w.scan, scan * 4) != cudaSuccess)
    return DT_ENOMEM;
  w.cap = need;
  w.scan_cap = scan;
  return DT_OK;
}

int canon_count(const CanonIn& in, CanonWS& w, uint64_t* T, cudaStream_t s) {
  if (!w.count && cudaMalloc(&w.count, 16) != cudaSuccess) return DT_ENOMEM;
  unsigned long long c = 0;
  const unsigned g = grid_of(in.nslots, kCollectThreads * kCollectItems, 152u * 8);
  cudaMemsetAsync(w.count, 0, 16, s);
  if (in.clouds)
    k_canon_collect<true><<<g, kCollectThreads, 0, s>>>(in.tets, in.nslots, nullptr, in.npts, in.clouds, in.n_clouds,
                                                        nullptr, nullptr, nullptr, w.count);
  else
    k_canon_collect<false><<<g, kCollectThreads, 0, s>>>(in.tets, in.nslots, nullptr, in.npts, nullptr, 0, nullptr,
                                                         nullptr, nullptr, w.count);
  ++g_kernel_launches;
  cudaMemcpyAsync(&c, w.count, 8, cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return DT_ECUDA;
  *T = c;
  return DT_OK;
}

int canon_rows(const CanonIn& in, CanonWS& w, const CanonScratch& t, uint64_t cap, uint4* staged, uint4* out, uint64_t* T,
               unsigned long long* cloud_starts, cudaStream_t s) {
  int rc = canon_ws_reserve(w, in.npts);
  if (rc != DT_OK) return rc;
  unsigned long long c[2] = {0, 0};
  cudaMemsetAsync(w.count, 0, 16, s);
  cudaMemsetAsync(w.first, 0, (in.npts + 1) * 4, s);
  k_input_ids<<<grid_of(in.npts, 256, 152u * 16), 256, 0, s>>>(in.pts, in.npts, w.ids);
  const unsigned g = grid_of(in.nslots, kCollectThreads * kCollectItems, 152u * 8);
  if (in.clouds)
    k_canon_collect<true><<<g, kCollectThreads, 0, s>>>(in.tets, in.nslots, w.ids, in.npts, in.clouds, in.n_clouds,
                                                        t.rows, t.place, w.first, w.count);
  else
    k_canon_collect<false><<<g, kCollectThreads, 0, s>>>(in.tets, in.nslots, w.ids, in.npts, nullptr, 0, t.rows,
                                                         t.place, w.first, w.count);
  g_kernel_launches += 2;
  prefix_sum_exclusive(w.first, in.npts + 1, w.scan, s);
  if (cloud_starts) {
    k_cloud_starts<<<grid_of(in.n_clouds + 1, 256, 152u), 256, 0, s>>>(w.first, in.in_off, in.n_clouds, cloud_starts);
    ++g_kernel_launches;
  }
  cudaMemcpyAsync(c, w.count, 16, cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return DT_ECUDA;
  *T = c[0];
  if (c[0] > 0 && c[0] <= cap) {
    const uint64_t nt = (c[0] + kTileRows - 1) / kTileRows;
    k_canon_scatter<<<grid_of(c[0], 256, 152u * 16), 256, 0, s>>>(t.rows, t.place, c[0], w.first, staged);
    k_canon_bounds<<<grid_of(nt, 256, 152u * 16), 256, 0, s>>>(staged, c[0], w.first, nt, t.bounds);
    k_canon_order<<<(unsigned)nt, kOrderThreads, 0, s>>>(staged, out, t.bounds, w.first, in.cid, in.in_off);
    g_kernel_launches += 3;
    if (c[1]) rc = order_big(t.rows, c[0], w, in.cid, in.in_off, out, s);
  }
  // the scratch goes back as it came: zero
  cudaMemsetAsync(t.rows, 0, c[0] * 16, s);
  cudaMemsetAsync(t.place, 0, c[0] * 4, s);
  if (rc == DT_OK && cudaPeekAtLastError() != cudaSuccess) rc = DT_ECUDA;
  return rc;
}

}  // namespace dtg
