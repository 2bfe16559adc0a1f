// Periodic on-device counting sort of particle slots by (cell tile, cell in
// tile).  The paper's particles wander between sub-domains one cell per step
// at most (§2, CFL argument); here the "sub-domains" are the push kernel's
// cell tiles, and regrouping the particles by tile every few steps keeps each
// tile's particles contiguous.  Integer-only: the result is exactly defined
// up to the order of particles sharing a cell.
//
//   hist     rank[p] = atomicAdd(&count[key(cell[p])], 1)   (dead slots: -1)
//   sums     run[t] = the tile's cell counts, summed and padded
//   groups   per 1024 tiles: slots, and work items for every candidate size
//   starts   tile_start = exclusive scan of run; *d_count = total; the size of
//            the push's work items is chosen and the items are written
//   offsets  count[key] <- tile_start[t] + exclusive scan within the tile;
//            the padding slots of each tile run get dst.cell = -1
//   permute  dst.cell[count[key] + rank[p]] = p    (the source of each slot)
//   gather   dst[q] = src[dst.cell[q]]             (every SoA array)
// The move is written as a gather: each destination slot reads its source,
// so the writes of every array are coalesced.  (A scatter that writes each
// particle to its new slot turns into a scatter of partial sectors once the
// particles have drifted for a few steps: 5x slower at 134M particles.)
// No block waits for another: the two scans over tiles are a launch for the
// groups' sums and one in which every block adds up the groups before it (one
// block did both before, 0.37 ms of a sort at 262,144 tiles).  Bound by the
// scattered 4-byte reads of the gather; 134M particles take 3.5 ms (4.45 with
// integer divisions in the keys and the one-block scans), 35M in a foil 0.66 ms
// (1.0).
#include <cuda_runtime.h>

#include "pic_device.cuh"

namespace pic {

namespace {

// The tile edges are powers of two (push_tile_shape), the grid's are not.
struct KeyMap {
  FastDiv d0, d1;
  int n0, n1;
  int s0, s1, s2;  // log2 of the tile edges
  int nt0, nt1;
  int tc;  // cells per tile
  __device__ __forceinline__ int key(int c) const {
    const int r = (int)d0.div((uint32_t)c);
    const int i = c - r * n0;
    const int k = (int)d1.div((uint32_t)r);
    const int j = r - k * n1;
    const int ti = i >> s0, tj = j >> s1, tk = k >> s2;
    const int tile = ti + nt0 * (tj + nt1 * tk);
    return tile * tc + (i - (ti << s0)) + (((j - (tj << s1)) + ((k - (tk << s2)) << s1)) << s0);
  }
};

__global__ void k_hist(KeyMap km, const int32_t *__restrict__ cell, const int64_t *__restrict__ d_count,
                       int32_t *__restrict__ count, int32_t *__restrict__ rank) {
  after_previous();
  const int64_t n = *d_count;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // every lane of a warp takes part in every pass
  for (int64_t p0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); p0 < n; p0 += stride) {
    const int64_t p = p0 + lane;
    const int c = p < n ? cell[p] : -1;
    const int key = c < 0 ? -1 : km.key(c);
    // aggregate lanes of the warp that share a key (sorted input: common)
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader && key >= 0) base = atomicAdd(&count[key], __popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (p < n) rank[p] = key < 0 ? -1 : base + __popc(peers & ((1u << lane) - 1u));
  }
}

// one warp per tile
__global__ void k_tile_sum(const int32_t *__restrict__ count, int64_t ntiles, int tc, uint32_t *__restrict__ run) {
  after_previous();
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= ntiles) return;
  const int32_t *c = count + t * tc;
  uint32_t s = 0;
  for (int i = lane; i < tc; i += 32) s += (uint32_t)c[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) run[t] = (s + kTilePad - 1) / kTilePad * kTilePad;  // padded run length
}

// Slots per work item of a run: the fewest equal pieces of at most `size`
// (runs, sizes and pieces are multiples of kTilePad); and how many they are.
__device__ __forceinline__ uint32_t item_slots(uint32_t run, uint32_t size) {
  if (run <= size) return run;
  const uint32_t pieces = (run + size - 1) / size;
  return ((run + pieces - 1) / pieces + kTilePad - 1) / kTilePad * kTilePad;
}
__device__ __forceinline__ uint32_t items_of(uint32_t run, uint32_t size) {
  if (run <= size) return run > 0;
  const uint32_t len = item_slots(run, size);
  return (run + len - 1) / len;
}

// What is summed over tiles: slots, work items for every candidate size, and
// the adjoint's items.
constexpr int kGroup = 1024;
constexpr int kVals = kItemCands + 2;
constexpr int kPart = 2;  // values of a block of k_tile_groups: the divisions are a serial chain
static_assert(kVals <= 32 && kVals % kPart == 0, "one warp per value, one lane per candidate");

__global__ void __launch_bounds__(kGroup)
    k_tile_groups(const uint32_t *__restrict__ run, int64_t ntiles, ItemPlan plan, uint32_t *__restrict__ part,
                  const int64_t *__restrict__ d_count, int64_t *__restrict__ n_src) {
  after_previous();
  __shared__ uint32_t s[kPart];
  const int v0 = blockIdx.y * kPart;
  if (threadIdx.x < kPart) s[threadIdx.x] = 0;
  if (blockIdx.x == 0 && v0 == 0 && threadIdx.x == 0) *n_src = *d_count;  // k_tile_starts rewrites it
  __syncthreads();
  const int64_t t = blockIdx.x * (int64_t)kGroup + threadIdx.x;
  const uint32_t r = t < ntiles ? run[t] : 0u;
#pragma unroll
  for (int k = 0; k < kPart; ++k) {
    const int v = v0 + k;
    uint32_t x = r;
    if (v > 0) x = items_of(r, v <= kItemCands ? (uint32_t)plan.cand[v - 1] : (uint32_t)kAdjItem);
    const uint32_t sum = __reduce_add_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0 && sum > 0) atomicAdd(&s[k], sum);
  }
  __syncthreads();
  if (threadIdx.x < kPart) part[blockIdx.x * kVals + v0 + threadIdx.x] = s[threadIdx.x];
}

// The size of the push's items is chosen here, where the tiles' runs are
// known: a fixed size left the last round of blocks nearly empty or split the
// items finer than needed (items for 16 blocks per SM against this rule: hot
// 2D plasma of 1.8M particles 0.137 -> 0.119 ms per push, FP64 64^3 3.03 ->
// 2.73 ms).
//
// Estimated time of a species of `slots` slots cut into `items`, in items (of
// their mean slots and plan.fixed more) that an SM's blocks share.  Measured
// with every size from 520 to 1920 slots in 2D FP32 (three blocks per SM): with
// two rounds of items or more the time is proportional to slots + 400 items
// within 5 % wherever the last round ends (a block that draws no item leaves
// its share to the others), SMs with one item more than others costing up to
// half of it; just above one round the second costs 0.4 of a round before its
// items; below one, two blocks on an SM take 0.85 of the time of three.  A
// block that has its SM to itself leaves it idle instead.
// (2D foil of 0.33M particles: 256 items 25.0 us per push, 416 items 20.9, 480
// items 26.9, 576 items 31.2.)  3D and FP64 runs are ranked by the same form: on
// nine of ten of them, 3D FP32 and FP64 and 2D FP64, CIC and TSC, every second
// size forced in turn, the choice was within 1 % of the fastest (FP64 40^3 of 8
// per cell 819 us, 838 to 1544 with the others; 64^3 FP32 180 and 229 to 611), and
// 5 % slower on one (48 x 40 x 32 TSC FP32 of 27 per cell, 156 us and 149).
__device__ __forceinline__ unsigned long long item_cost(const ItemPlan &pl, uint32_t slots, uint32_t items) {
  const uint32_t per = pl.blocks * pl.nsm, full = items / per, rem = items % per;
  const uint32_t most = (rem + pl.nsm - 1) / pl.nsm * pl.nsm;
  uint32_t unit = items;
  if (full == 0) unit = (per + most) / 2;
  else if (rem > 0) unit += pl.blocks == 1 ? per - rem : 2 * per / (5 * full * full) + (most - rem) / 2;
  return (unsigned long long)unit * (slots / items + pl.fixed);
}

// Exclusive block scan of three counters (1024 threads).
__device__ __forceinline__ void scan3(uint32_t (&v)[3], uint32_t (*sh)[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t own[3] = {v[0], v[1], v[2]};
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, v[q], o);
      if (lane >= o) v[q] += x;
    }
  if (lane == 31)
    for (int q = 0; q < 3; ++q) sh[warp][q] = v[q];
  __syncthreads();
  if (warp == 0) {
    uint32_t w[3] = {sh[lane][0], sh[lane][1], sh[lane][2]};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, w[q], o);
        if (lane >= o) w[q] += x;
      }
    for (int q = 0; q < 3; ++q) sh[lane][q] = w[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) v[q] += (warp > 0 ? sh[warp - 1][q] : 0u) - own[q];
}

// One tile per thread: its start slot, and its work items (of the push, and of
// the adjoint where adj.nwork > 0).
__global__ void __launch_bounds__(kGroup)
    k_tile_starts(const uint32_t *__restrict__ run, int64_t ntiles, int ngroups, ItemPlan plan,
                  const uint32_t *__restrict__ part, int64_t *__restrict__ tile_start, int64_t *__restrict__ d_count,
                  WorkList push, WorkList adj) {
  after_previous();
  __shared__ uint32_t s_before[kVals], s_total[kVals], s_scan[32][3];
  __shared__ int s_pick;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kVals) {
    uint32_t before = 0, total = 0;
    for (int g = lane; g < ngroups; g += 32) {
      const uint32_t x = part[g * kVals + warp];
      total += x;
      if (g < (int)blockIdx.x) before += x;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0) {
      s_before[warp] = before;
      s_total[warp] = total;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int best = lane;
    unsigned long long least = ~0ull;
    if (lane < kItemCands && s_total[0] > 0) least = item_cost(plan, s_total[0], s_total[1 + lane]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long c = __shfl_xor_sync(0xffffffffu, least, o);
      const int j = __shfl_xor_sync(0xffffffffu, best, o);
      if (c < least || (c == least && j < best)) {
        least = c;
        best = j;
      }
    }
    if (lane == 0) s_pick = best;
  }
  __syncthreads();
  const int pick = s_pick;
  const uint32_t size = (uint32_t)plan.cand[pick];
  const int64_t t = blockIdx.x * (int64_t)kGroup + threadIdx.x;
  const uint32_t r = t < ntiles ? run[t] : 0u;
  uint32_t at[3] = {r, items_of(r, size), adj.nwork > 0 ? items_of(r, kAdjItem) : 0u};
  scan3(at, s_scan);
  const uint32_t first = s_before[0] + at[0];
  if (t < ntiles) tile_start[t] = first;
  const auto write = [&](const WorkList &w, uint32_t i, uint32_t len) {
    for (uint32_t p = 0; p < r; p += len, ++i) {
      w.work_tile[i] = (int32_t)t;
      w.work_pb[i] = (int64_t)first + p;
      w.work_n[i] = (int32_t)(r - p < len ? r - p : len);
    }
  };
  write(push, s_before[1 + pick] + at[1], item_slots(r, size));
  if (adj.nwork > 0) write(adj, s_before[kVals - 1] + at[2], item_slots(r, kAdjItem));
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    tile_start[ntiles] = s_total[0];
    *d_count = s_total[0];
    *push.count = (int32_t)s_total[1 + pick];
    if (adj.nwork > 0) *adj.count = (int32_t)s_total[kVals - 1];
  }
}

// one warp per tile: count[key] <- absolute start slot of the key; the
// tile's padding slots in the destination are marked dead
__global__ void k_offsets(int32_t *__restrict__ count, int64_t ntiles, int tc, const int64_t *__restrict__ tile_start,
                          int32_t *__restrict__ dst_cell) {
  after_previous();
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= ntiles) return;
  int32_t *c = count + t * tc;
  int64_t run = tile_start[t];
  for (int base = 0; base < tc; base += 32) {
    const int i = base + lane;
    const int v = i < tc ? c[i] : 0;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (i < tc) c[i] = (int32_t)(run + incl - v);
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (run + lane < tile_start[t + 1]) dst_cell[run + lane] = -1;
}

__global__ void k_permute(KeyMap km, const int32_t *__restrict__ cell, const int64_t *__restrict__ n_src,
                          const int32_t *__restrict__ count, const int32_t *__restrict__ rank,
                          int32_t *__restrict__ dst_cell, int64_t capacity, Counters *ctr) {
  after_previous();
  const int64_t n = *n_src;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int r = rank[p];
    if (r < 0) continue;
    const int64_t q = (int64_t)count[km.key(cell[p])] + r;
    if (!PIC_CHECK(q >= 0 && q < capacity, ctr)) continue;
    dst_cell[q] = (int32_t)p;  // slots stay below 2^31
  }
}

template <class R>
__global__ void k_gather(int dims, Particles src, Particles dst, const int64_t *__restrict__ n_dst,
                         const int64_t *__restrict__ n_src, Counters *ctr) {
  after_previous();
  const int64_t n = *n_dst;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int p = dst.cell[q];
    if (p < 0) continue;  // tile padding: stays a dead slot
    if (!PIC_CHECK(p < *n_src, ctr)) continue;
    dst.cell[q] = src.cell[p];
    dst.id[q] = src.id[p];
    static_cast<R *>(dst.w)[q] = static_cast<const R *>(src.w)[p];
    for (int d = 0; d < 3; ++d) {
      if (d < dims) static_cast<R *>(dst.off[d])[q] = static_cast<const R *>(src.off[d])[p];
      static_cast<R *>(dst.u[d])[q] = static_cast<const R *>(src.u[d])[p];
    }
  }
}

}  // namespace

// n_src, run[ntiles], part[groups][kVals]
size_t sort_tmp_bytes(int64_t ntiles) {
  const int64_t groups = (ntiles + kGroup - 1) / kGroup;
  return sizeof(int64_t) + sizeof(uint32_t) * (size_t)(ntiles + groups * kVals);
}

cudaError_t launch_sort(const Grid &g, const Particles &src, const Particles &dst, int64_t *d_count,
                        int64_t capacity, int32_t *keys, int32_t *rank, int64_t *tile_start, void *tmp,
                        const WorkSplit &ws, Counters *ctr, cudaStream_t st, int *nlaunch) {
  KeyMap km;
  km.d0 = make_fastdiv((uint32_t)g.n[0]);
  km.d1 = make_fastdiv((uint32_t)g.n[1]);
  km.n0 = g.n[0];
  km.n1 = g.n[1];
  int *const lg[3] = {&km.s0, &km.s1, &km.s2};
  for (int d = 0; d < 3; ++d) {
    *lg[d] = 0;
    while ((1 << *lg[d]) < g.tile[d]) ++*lg[d];
    if ((1 << *lg[d]) != g.tile[d]) return cudaErrorInvalidValue;
  }
  km.nt0 = g.ntile[0];
  km.nt1 = g.ntile[1];
  km.tc = g.tile[0] * g.tile[1] * g.tile[2];
  int64_t *n_src = static_cast<int64_t *>(tmp);
  uint32_t *run = reinterpret_cast<uint32_t *>(n_src + 1), *part = run + g.ntiles;
  const int groups = (int)((g.ntiles + kGroup - 1) / kGroup);
  const int64_t nkeys = g.ntiles * km.tc;
  cudaError_t e = cudaMemsetAsync(keys, 0, sizeof(int32_t) * nkeys, st);
  if (e != cudaSuccess) return e;
  const int nsm = ws.plan.nsm;
  const int64_t want = (capacity + 255) / 256;
  const int nb = (int)(want < (int64_t)nsm * 16 ? (want > 0 ? want : 1) : (int64_t)nsm * 16);
  launch_next(k_hist, nb, 256, 0, st, km, src.cell, d_count, keys, rank);
  const unsigned wb = (unsigned)((g.ntiles * 32 + 255) / 256);
  launch_next(k_tile_sum, wb, 256, 0, st, keys, g.ntiles, km.tc, run);
  launch_next(k_tile_groups, dim3(groups, kVals / kPart), kGroup, 0, st, run, g.ntiles, ws.plan, part, d_count,
              n_src);
  launch_next(k_tile_starts, groups, kGroup, 0, st, run, g.ntiles, groups, ws.plan, part, tile_start, d_count, ws,
              ws.adj);
  launch_next(k_offsets, wb, 256, 0, st, keys, g.ntiles, km.tc, tile_start, dst.cell);
  launch_next(k_permute, nb, 256, 0, st, km, src.cell, n_src, keys, rank, dst.cell, capacity, ctr);
  if (g.prec == 1)
    launch_next(k_gather<double>, nb, 256, 0, st, g.dims, src, dst, d_count, n_src, ctr);
  else
    launch_next(k_gather<float>, nb, 256, 0, st, g.dims, src, dst, d_count, n_src, ctr);
  if (nlaunch) *nlaunch = 7;
  return cudaGetLastError();
}

}  // namespace pic
