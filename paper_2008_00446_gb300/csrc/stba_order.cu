// Device side of a new cluster assignment (Sec. 4.1-4.2): the observations are re-ordered by (point,
// cluster, camera), the virtual points (distinct (point, cluster) pairs) are numbered, and the per-camera
// observation lists of the camera pass are rebuilt.  The (point, camera) order fixed at create is the base:
// inside a point run the new order is the stable sort of the base by cluster, so a virtual point is a run
// of equal clusters and its observations stay ordered by camera.  Every step is deterministic.
#include <climits>
#include <type_traits>

#include <cuda_runtime.h>

#include "stba_device.cuh"
#include "stba_internal.cuh"

namespace stba {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr int SUPER = 64;   // tiles whose counts are also kept as one sum

// Sums per scan tile: virtual-point starts (super: per SUPER tiles) and twice the camera-pair instances.
struct TileSums {
  unsigned long long* pairs;   // [ntiles]
  int* tile;                   // [ntiles]
  int* super;                  // [ntiles / SUPER + 1]
};

// New position of every base observation: its rank in the stable order by cluster inside its point run.
// Marks the first observation of every virtual point, counts these and the camera-pair instances (each twice) per
// scan tile, and carries the per-observation data over.
// Bound by its 100 bytes of scattered 4- to 16-byte accesses an observation: 31 us at 1.1 M observations (with the
// clusters and the counts from kernels of their own and one more copy of the observations 43 us).
template <typename real>
__global__ void __launch_bounds__(256) k_reorder(ReorderArgs A, TileSums S, const real* __restrict__ res_old,
                                                 real* __restrict__ res_new) {
  __shared__ unsigned wpairs[8];
  __shared__ int wfirst[2][8];
  __shared__ int key[256];   // clusters of the CTA's observations: most of a run is in the same CTA
  const int b0 = blockIdx.x * 256, bo = b0 + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int np = 0, same = 1;
  bool first = false;
  int cam = 0, kb = 0;
  if (bo < A.q) {
    cam = A.base_cam[bo];
    kb = A.cam_cluster[cam];
  }
  key[threadIdx.x] = kb;
  __syncthreads();
  if (bo < A.q) {
    const int i = A.obs_pt[bo];
    const int b = A.pt_off[i], e = A.pt_off[i + 1];
    int rank = 0;
    same = 0;
    first = true;
    for (int o = b; o < e; ++o) {
      const unsigned l = (unsigned)(o - b0);
      const int ko = l < 256u ? key[l] : A.cam_cluster[A.base_cam[o]];
      rank += (ko < kb) || (ko == kb && o < bo);
      first = first && !(ko == kb && o < bo);
      same += ko == kb;
    }
    np = b + rank;
    A.inv_new[bo] = np;
    A.nsing[bo] = same == 1 ? (np | INT_MIN) : np;
    A.obs_base[np] = bo;
    A.obs_cam[np] = cam;
    A.obs_perm[np] = A.base_src[bo];
    A.start[np] = first ? 1 : 0;
    if (A.obs_uv) reinterpret_cast<double2*>(A.obs_uv)[np] = reinterpret_cast<const double2*>(A.base_uv)[bo];
    if (A.obs_uvdf) A.obs_uvdf[np] = A.base_uvdf[bo];
    if (res_old) {   // residuals at the current x, stored in the order of the previous assignment
      using V2 = std::conditional_t<sizeof(real) == 4, float2, double2>;
      reinterpret_cast<V2*>(res_new)[np] = reinterpret_cast<const V2*>(res_old)[A.inv_old[bo]];
    }
  }
  // the CTA's sums first: thousands of atomics on one address queue in L2 (48 us with one per warp)
  const int t0 = b0 / SCAN_TILE, t = np / SCAN_TILE;
  const bool near = t == t0 || t == t0 + 1;
  const unsigned f0 = __ballot_sync(FULL_MASK, first && t == t0), f1 = __ballot_sync(FULL_MASK, first && t == t0 + 1);
  if (first && !near) {   // a run that began in an earlier tile, or goes on past the next
    atomicAdd(S.tile + t, 1);
    atomicAdd(S.super + t / SUPER, 1);
  }
  const unsigned p = __reduce_add_sync(FULL_MASK, (unsigned)(same - 1));
  if (lane == 0) {
    wfirst[0][w] = __popc(f0);
    wfirst[1][w] = __popc(f1);
    wpairs[w] = p;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    int c = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) c += wfirst[threadIdx.x][u];
    if (c) {
      atomicAdd(S.tile + t0 + threadIdx.x, c);
      atomicAdd(S.super + (t0 + threadIdx.x) / SUPER, c);
    }
  } else if (threadIdx.x == 2) {
    unsigned long long c = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) c += wpairs[u];
    if (c) atomicAdd(S.pairs + t0, c);
  }
}

// per tile of SCAN_TILE observations: the number of virtual-point starts
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_tiles(int q, const int* __restrict__ start,
                                                             int* __restrict__ tile_sum) {
  __shared__ int ws[SCAN_THREADS / 32];
  const int base = blockIdx.x * SCAN_TILE;
  int s = 0;
#pragma unroll
  for (int t = 0; t < SCAN_ITEMS; ++t) {
    const int o = base + t * SCAN_THREADS + threadIdx.x;
    s += o < q ? start[o] : 0;
  }
  for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(FULL_MASK, s, d);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < SCAN_THREADS / 32; ++w) t += ws[w];
    tile_sum[blockIdx.x] = t;
  }
}

// exclusive scan of the tile sums (one CTA, sequential chunks of 1024); the total goes to counts[0]
__global__ void __launch_bounds__(1024) k_scan_partials(int ntiles, int* __restrict__ tile_sum,
                                                        long long* __restrict__ counts) {
  __shared__ int ws[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int c0 = 0; c0 < ntiles; c0 += 1024) {
    const int i = c0 + threadIdx.x;
    const int v = i < ntiles ? tile_sum[i] : 0;
    int x = v;
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL_MASK, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
      int z = ws[lane];
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, z, d);
        if (lane >= d) z += y;
      }
      ws[lane] = z;
    }
    __syncthreads();
    const int incl = x + (w > 0 ? ws[w - 1] : 0) + carry;
    if (i < ntiles) tile_sum[i] = incl - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry = incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) counts[0] = carry;
}

// Eight consecutive ints from (to) a 16-byte aligned array of q, zeros past its end.
__device__ __forceinline__ void load8(const int* __restrict__ p, int base, int q, int (&v)[SCAN_ITEMS]) {
  if (base + SCAN_ITEMS <= q) {
    const int4 a = *reinterpret_cast<const int4*>(p + base), b = *reinterpret_cast<const int4*>(p + base + 4);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else {
#pragma unroll
    for (int t = 0; t < SCAN_ITEMS; ++t) v[t] = base + t < q ? p[base + t] : 0;
  }
}
__device__ __forceinline__ void store8(int* __restrict__ p, int base, int q, const int (&v)[SCAN_ITEMS]) {
  if (base + SCAN_ITEMS <= q) {
    *reinterpret_cast<int4*>(p + base) = make_int4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<int4*>(p + base + 4) = make_int4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int t = 0; t < SCAN_ITEMS; ++t)
      if (base + t < q) p[base + t] = v[t];
  }
}

// Virtual-point numbers: obs_vp, vp_off, vp_point, pt_vp_off, and their closing entries and count in the last
// tile's CTA.  A CTA adds up the tiles before its own itself (the super sums, then at most SUPER - 1 tiles), and a
// thread moves its eight consecutive entries as two 16-byte vectors: 13 us at 1.1 M observations; with 4-byte
// accesses 32 bytes apart, a kernel for the tiles' prefixes and one for the closing entries 27 us.
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_apply(ReorderArgs A, TileSums S,
                                                             long long* __restrict__ counts) {
  __shared__ int ws[SCAN_THREADS / 32], wp[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;   // contiguous items per thread
  int pre = 0;
  const int ns = blockIdx.x / SUPER;
  for (int t = threadIdx.x; t < ns; t += SCAN_THREADS) pre += S.super[t];
  for (int t = ns * SUPER + threadIdx.x; t < (int)blockIdx.x; t += SCAN_THREADS) pre += S.tile[t];
  pre = (int)__reduce_add_sync(FULL_MASK, (unsigned)pre);
  int v[SCAN_ITEMS], s = 0;
  load8(A.start, base, A.q, v);
#pragma unroll
  for (int t = 0; t < SCAN_ITEMS; ++t) s += v[t];
  int x = s;
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(FULL_MASK, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) ws[w] = x;
  if (lane == 0) wp[w] = pre;
  __syncthreads();
  int run = x - s, total = 0;   // run: starts before this thread's first item
#pragma unroll
  for (int u = 0; u < SCAN_THREADS / 32; ++u) {
    total += wp[u] + ws[u];
    run += wp[u] + (u < w ? ws[u] : 0);
  }
  if (base < A.q) {
    int vp[SCAN_ITEMS], pt[SCAN_ITEMS];
    load8(A.obs_pt, base, A.q, pt);
#pragma unroll
    for (int t = 0; t < SCAN_ITEMS; ++t) {
      const int o = base + t;
      run += v[t];   // 0 past the end
      vp[t] = run - 1;
      if (v[t]) {
        A.vp_off[run - 1] = o;
        A.vp_point[run - 1] = pt[t];
        if (A.pt_off[pt[t]] == o) A.pt_vp_off[pt[t]] = run - 1;
      }
    }
    store8(A.obs_vp, base, A.q, vp);
    if (A.base_vp) {
      int bo[SCAN_ITEMS];
      load8(A.obs_base, base, A.q, bo);
#pragma unroll
      for (int t = 0; t < SCAN_ITEMS; ++t)
        if (base + t < A.q) A.base_vp[bo[t]] = vp[t];
    }
  }
  if (threadIdx.x == 0 && S.pairs[blockIdx.x])
    atomicAdd(reinterpret_cast<unsigned long long*>(counts + 1), S.pairs[blockIdx.x]);
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    counts[0] = total;
    A.vp_off[total] = A.q;
    A.pt_vp_off[A.n] = total;
  }
}

// Camera lists: the observations of every camera (new positions), those of single-observation virtual
// points first, each group in base order -- a stable partition of every camera's run of cam_base.  Whether
// an observation is alone in its virtual point (no other observation of its point in its cluster) comes
// from k_reorder, packed with its new position.
__device__ __forceinline__ void place_obs(const ReorderArgs& A, int j, int e, int idx, int x) {
  const int o = x & INT_MAX;
  A.cam_obs[A.cam_off[j] + idx] = o;
  const size_t sl = 32 * (size_t)A.cam_warp_off[j] + idx;
  A.slots[sl] = o;
  A.slot_pv[sl] = make_int2(A.ept[e], A.obs_vp[o] | (x & INT_MIN));
}

// One CTA per camera: counts the single ones, then places CL_CHUNK observations at a time (ranks from warp
// ballots).  For problems whose cameras have at most CL_MAX observations each; one with many more would be walked
// by one CTA alone, so there the list is made by the scan over all observations (k_cam_flag .. k_cam_place).
// 21 us for 1000 cameras with 1.1 M observations, the five launches of the scan 40 us.
constexpr int CL_THREADS = 256, CL_ROWS = 8, CL_CHUNK = CL_THREADS * CL_ROWS, CL_MAX = 8 * CL_CHUNK;
__global__ void __launch_bounds__(CL_THREADS) k_cam_lists(ReorderArgs A) {
  __shared__ int cnt[CL_ROWS * (CL_THREADS / 32)];   // single ones of (row, warp), then their prefix
  __shared__ int total;
  const int j = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = A.cam_off[j], n = A.cam_off[j + 1] - b;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  int x[CL_ROWS];
  auto load = [&](int c0) {
#pragma unroll
    for (int t = 0; t < CL_ROWS; ++t) {
      const int e = c0 + CL_THREADS * t + threadIdx.x;
      x[t] = e < n ? A.nsing[A.cam_base[b + e]] : 0;
    }
  };
  int mine = 0;
  for (int c0 = (n - 1) / CL_CHUNK * CL_CHUNK; c0 >= 0; c0 -= CL_CHUNK) {   // ends with the first chunk in x
    load(c0);
#pragma unroll
    for (int t = 0; t < CL_ROWS; ++t) mine += x[t] < 0;
  }
  const int wsum = (int)__reduce_add_sync(FULL_MASK, (unsigned)mine);
  if (lane == 0 && wsum) atomicAdd(&total, wsum);
  __syncthreads();
  const int nsingle = total;
  int done = 0;   // single ones of the chunks before
  for (int c0 = 0; c0 < n; c0 += CL_CHUNK) {
    if (c0) load(c0);
    unsigned bal[CL_ROWS];
#pragma unroll
    for (int t = 0; t < CL_ROWS; ++t) {
      bal[t] = __ballot_sync(FULL_MASK, x[t] < 0);
      if (lane == 0) cnt[t * (CL_THREADS / 32) + w] = __popc(bal[t]);
    }
    __syncthreads();
    if (w == 0) {   // exclusive prefix of the 64 counts
      const int c0v = cnt[2 * lane], c1v = cnt[2 * lane + 1];
      int p = c0v + c1v;
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, p, d);
        if (lane >= d) p += y;
      }
      cnt[2 * lane] = p - c0v - c1v;
      cnt[2 * lane + 1] = p - c1v;
      if (lane == 31) total = p;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < CL_ROWS; ++t) {
      const int e = c0 + CL_THREADS * t + threadIdx.x;
      if (e >= n) break;
      const int before = done + cnt[t * (CL_THREADS / 32) + w] + __popc(bal[t] & ((1u << lane) - 1));
      place_obs(A, j, b + e, x[t] < 0 ? before : nsingle + e - before, x[t]);
    }
    done += total;
    __syncthreads();   // cnt and total are rewritten by the next chunk
  }
}

__global__ void k_cam_flag(ReorderArgs A, int* __restrict__ flag) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= A.q) return;
  const int x = A.nsing[A.cam_base[e]];   // one gather: the new position and whether it is alone
  A.eo[e] = x;                            // for k_cam_place
  flag[e] = x < 0 ? 1 : 0;
}

// excl[e] = number of flags before e (tile offsets from k_scan_partials); excl[q] = total
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_excl(int q, const int* __restrict__ flag,
                                                            const int* __restrict__ tile_off,
                                                            const long long* __restrict__ total,
                                                            int* __restrict__ excl) {
  __shared__ int ws[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
  int v[SCAN_ITEMS], s = 0;
#pragma unroll
  for (int t = 0; t < SCAN_ITEMS; ++t) {
    v[t] = base + t < q ? flag[base + t] : 0;
    s += v[t];
  }
  int x = s;
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(FULL_MASK, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  int woff = 0;
  for (int u = 0; u < w; ++u) woff += ws[u];
  int run = tile_off[blockIdx.x] + woff + x - s;
#pragma unroll
  for (int t = 0; t < SCAN_ITEMS; ++t) {
    if (base + t >= q) break;
    excl[base + t] = run;
    run += v[t];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) excl[q] = (int)total[0];
}

__global__ void k_cam_place(ReorderArgs A, const int* __restrict__ excl) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= A.q) return;
  const int j = A.ecam[e];
  const int b = A.cam_off[j], cnt = A.cam_off[j + 1] - b;
  const int before = excl[e] - excl[b];               // singles of camera j before e
  const int nsingle = excl[b + cnt] - excl[b];
  const int x = A.eo[e];
  place_obs(A, j, e, x < 0 ? before : nsingle + (e - b - before), x);
}

// chunks of the camera graph whose two cameras share a cluster
// a chunk is listed when its two cameras share a cluster that this process owns (every cluster unless sharded)
__global__ void k_chunk_flag(int nchunks, const int4* __restrict__ chunks, const int* __restrict__ cam_cluster,
                             const int* __restrict__ owned, int* __restrict__ flag) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nchunks) return;
  const int4 ch = chunks[c];
  const int k = cam_cluster[ch.x];
  flag[c] = (k == cam_cluster[ch.y] && owned[k]) ? 1 : 0;
}

__global__ void k_chunk_list(int nchunks, const int* __restrict__ flag, const int* __restrict__ excl,
                             int* __restrict__ active) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nchunks && flag[c]) active[excl[c]] = c;
}

// zeroes the per reals of the nv virtual points, nv read from the device counter
__global__ void __launch_bounds__(256) k_zero_vp(float4* __restrict__ p, const long long* __restrict__ counts,
                                                 int real_bytes, int per) {
  const long long n16 = (per * counts[0] * real_bytes + 15) / 16;   // the buffer holds per q reals, 16-byte padded
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n16; i += (long long)gridDim.x * blockDim.x)
    p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

}  // namespace

__global__ void k_base_vp(int q, const int* __restrict__ obs_base, const int* __restrict__ obs_vp, int* __restrict__ base_vp) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o < q) base_vp[obs_base[o]] = obs_vp[o];
}

void launch_base_vp(const int* obs_base, const int* obs_vp, int* base_vp, int q, cudaStream_t stream) {
  k_base_vp<<<(q + 255) / 256, 256, 0, stream>>>(q, obs_base, obs_vp, base_vp);
}

size_t reorder_tiles(int64_t q) {
  const size_t ntiles = (size_t)((q + SCAN_TILE - 1) / SCAN_TILE);
  return 3 * ntiles + ntiles / SUPER + 1;
}

void launch_list_chunks(const PairChunks& B, const int* cam_cluster, const int* owned, long long* nactive,
                        cudaStream_t stream) {
  const int n = B.nchunks;
  if (n <= 0) return;
  const int g = (n + 255) / 256, ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  k_chunk_flag<<<g, 256, 0, stream>>>(n, B.chunks, cam_cluster, owned, B.flag);
  k_scan_tiles<<<ntiles, SCAN_THREADS, 0, stream>>>(n, B.flag, B.tile_sum);
  k_scan_partials<<<1, 1024, 0, stream>>>(ntiles, B.tile_sum, nactive);
  k_scan_excl<<<ntiles, SCAN_THREADS, 0, stream>>>(n, B.flag, B.tile_sum, nactive, B.excl);
  k_chunk_list<<<g, 256, 0, stream>>>(n, B.flag, B.excl, const_cast<int*>(B.active));
}

void launch_zero_vp3(void* p, const long long* counts, int real_bytes, cudaStream_t stream) {
  k_zero_vp<<<2 * RED_BLOCKS, 256, 0, stream>>>(reinterpret_cast<float4*>(p), counts, real_bytes, 3);
}

template <typename real>
void launch_reorder(const ReorderArgs& A, int* key, int* tile_sum, long long* counts, const real* res_old,
                    real* res_new, cudaStream_t stream) {
  const int g = (A.q + 255) / 256;
  const int ntiles = (A.q + SCAN_TILE - 1) / SCAN_TILE;
  TileSums S;
  S.pairs = reinterpret_cast<unsigned long long*>(tile_sum);
  S.tile = tile_sum + 2 * (size_t)ntiles;
  S.super = S.tile + ntiles;
  cudaMemsetAsync(counts, 0, 3 * sizeof(long long), stream);
  cudaMemsetAsync(tile_sum, 0, reorder_tiles(A.q) * sizeof(int), stream);
  k_reorder<real><<<g, 256, 0, stream>>>(A, S, res_old, res_new);
  k_scan_apply<<<ntiles, SCAN_THREADS, 0, stream>>>(A, S, counts);
  if (A.max_cam_obs <= CL_MAX) {
    k_cam_lists<<<A.m, CL_THREADS, 0, stream>>>(A);
    return;
  }
  // flags, their exclusive scan, placement
  int* excl = A.start + A.q + 1;   // second half of the start buffer
  k_cam_flag<<<g, 256, 0, stream>>>(A, key);
  k_scan_tiles<<<ntiles, SCAN_THREADS, 0, stream>>>(A.q, key, tile_sum);
  k_scan_partials<<<1, 1024, 0, stream>>>(ntiles, tile_sum, counts + 2);
  k_scan_excl<<<ntiles, SCAN_THREADS, 0, stream>>>(A.q, key, tile_sum, counts + 2, excl);
  k_cam_place<<<g, 256, 0, stream>>>(A, excl);
}

template void launch_reorder<float>(const ReorderArgs&, int*, int*, long long*, const float*, float*, cudaStream_t);
template void launch_reorder<double>(const ReorderArgs&, int*, int*, long long*, const double*, double*,
                                     cudaStream_t);

}  // namespace stba
