// Classification of the 8^3-cell Eulerian tiles after the Gauss points of each
// have been counted (the tiles of a packed plan are those of all its
// structures, each with the neighbours on its own periodic grid):
//   non-empty  the tile holds points              -> spread push / interp work
//   near       a tile of its 3x3x3 neighbourhood holds points
//                                                   -> its faces are merged
//   far        otherwise                          -> its faces are zero
// A non-empty tile is cut into work items ("chunks") of consecutive points
// (item_points), so that a densely populated tile (mesh singularities
// concentrate points) is shared by several CTAs, and a small structure by
// many.  A tile's items own consecutive scratch blocks, the first of which is
// the tile's slot.  Two kernels: per-CTA counts, then every CTA
// finds its output offsets from the counts of the CTAs before it and writes
// its part of the work list and of the near-tile list.
#include "ib_device.cuh"

namespace ibfe {
namespace {

constexpr int kT = 256;  // tiles per CTA
constexpr int kCounts = 3;  // per-CTA counts: work items, near tiles, points

// Block-wide exclusive scans of K integers at once (one pair of barriers for
// all of them); total[k] receives the block sum of v[k].  tmp: K * 32 ints.
template <int K>
__device__ __forceinline__ void block_scan_k(const int (&v)[K], int (&pre)[K], int (&total)[K],
                                             int* tmp) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    x[k] = v[k];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(full, x[k], o);
      if (lane >= o) x[k] += y;
    }
    if (lane == 31) tmp[k * 32 + warp] = x[k];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      int w = lane < nw ? tmp[k * 32 + lane] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(full, w, o);
        if (lane >= o) w += y;
      }
      tmp[k * 32 + lane] = w;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    total[k] = tmp[k * 32 + nw - 1];
    pre[k] = (warp > 0 ? tmp[k * 32 + warp - 1] : 0) + x[k] - v[k];
  }
  __syncthreads();
}

// i in [-1, n]: its periodic image in [0, n)
__device__ __forceinline__ int wrap_one(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <bool kPacked>
__global__ void __launch_bounds__(kT) k_classify(GridDev g, const InstDev* __restrict__ inst,
                                                 const int32_t* __restrict__ tile_inst,
                                                 const int32_t* __restrict__ points, int ntiles,
                                                 int32_t* __restrict__ nonempty,
                                                 int32_t* __restrict__ near,
                                                 int32_t* __restrict__ bcount, ItemRule rule) {
  chain_wait();
  chain_next();
  __shared__ int sum[kCounts];
  if (threadIdx.x < kCounts) sum[threadIdx.x] = 0;
  const int t = blockIdx.x * kT + threadIdx.x;
  int nr = 0, nch = 0, npt = 0;
  if (t < ntiles) {
    const TileGeo geo = tile_geo<kPacked>(g, inst, tile_inst, t);
    const int nt0 = geo.nt[0], nt1 = geo.nt[1], nt2 = geo.nt[2];
    int tx, ty, tz;
    tile_coords(geo, t, tx, ty, tz);
    npt = points[t];
    const int per = item_points(npt, rule);
    nch = (npt + per - 1) / per;
    // all 27 neighbours' counts loaded at once (most tiles are far from the
    // structure and would otherwise wait for 27 dependent round trips)
    nr = 0;
#pragma unroll
    for (int a = -1; a <= 1; ++a)
#pragma unroll
      for (int b = -1; b <= 1; ++b)
#pragma unroll
        for (int c = -1; c <= 1; ++c) {
          const int nb = geo.base + wrap_one(tx + c, nt0) +
                         nt0 * (wrap_one(ty + b, nt1) + nt1 * wrap_one(tz + a, nt2));
          nr |= __ldg(points + nb) > 0;
        }
    nonempty[t] = nch;
    near[t] = nr;
  }
  __syncthreads();
  const unsigned full = 0xffffffffu;
  const int v[kCounts] = {__reduce_add_sync(full, nch), __reduce_add_sync(full, nr),
                          __reduce_add_sync(full, npt)};
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < kCounts; ++k)
      if (v[k]) atomicAdd(sum + k, v[k]);
  }
  __syncthreads();
  if (threadIdx.x < kCounts) bcount[kCounts * blockIdx.x + threadIdx.x] = sum[threadIdx.x];
}

// counters: [0] work items, [3] near tiles; the work counters (1: push; 2, 4, 5,
// 7: interpolations) are zeroed for the calls that follow this binning, with
// the tiles' largest values and finished items, and the point counts for the
// next binning.  The tiles' point ranges: start = points of the tiles before,
// end = start + points.
__global__ void __launch_bounds__(kT) k_compact(const int32_t* __restrict__ nonempty,
                                                const int32_t* __restrict__ near, int ntiles,
                                                const int32_t* __restrict__ bcount, int nblocks,
                                                int32_t* __restrict__ points,
                                                uint32_t* __restrict__ vmax,
                                                int32_t* __restrict__ done,
                                                int32_t* __restrict__ start,
                                                int32_t* __restrict__ end,
                                                int32_t* __restrict__ slot,
                                                int4* __restrict__ work, ItemRule rule,
                                                int32_t* __restrict__ list_near,
                                                int32_t* __restrict__ counters) {
  chain_wait();
  chain_next();
  __shared__ int tmp[kCounts * 32];
  __shared__ int base[2 * kCounts];  // counts of the CTAs before this one, and of all
  if (threadIdx.x < 2 * kCounts) base[threadIdx.x] = 0;
  __syncthreads();
  int sums[2 * kCounts] = {};
  for (int b = threadIdx.x; b < nblocks; b += kT) {
#pragma unroll
    for (int k = 0; k < kCounts; ++k) {
      const int a = bcount[kCounts * b + k];
      if (b < (int)blockIdx.x) sums[k] += a;
      sums[kCounts + k] += a;
    }
  }
#pragma unroll
  for (int k = 0; k < 2 * kCounts; ++k) {
    const int v = __reduce_add_sync(0xffffffffu, sums[k]);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(base + k, v);
  }
  __syncthreads();
  const int t2 = base[kCounts], t3 = base[kCounts + 1];
  const int t = blockIdx.x * kT + threadIdx.x;
  const int np = t < ntiles ? points[t] : 0;
  const int per = item_points(np, rule);
  const int cnt[kCounts] = {t < ntiles ? nonempty[t] : 0, t < ntiles ? near[t] : 0, np};
  int cpre[kCounts], ctot[kCounts];
  block_scan_k<kCounts>(cnt, cpre, ctot, tmp);
  const int ne = cnt[0], first = base[0] + cpre[0], s0 = base[2] + cpre[2];
  if (t < ntiles) {
    points[t] = 0;
    vmax[t] = 0u;
    done[t] = 0;
    start[t] = s0;
    end[t] = s0 + np;
    slot[t] = ne ? first : -1;
    for (int j = 0; j < ne; ++j)
      work[first + j] = make_item(s0 + j * per, min(per, np - j * per), t, first + j, ne);
    if (cnt[1]) list_near[base[1] + cpre[1]] = t;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    counters[0] = t2;
    counters[3] = t3;
    counters[1] = counters[2] = counters[4] = counters[5] = counters[7] = 0;
  }
}

}  // namespace

int classify_blocks(int ntiles) { return (ntiles + kT - 1) / kT; }

// Work item size of a plan with Q points: full items (kChunk points) where
// they give every SM several, smaller ones where they would leave SMs idle
// (the transfer kernels take one item per CTA at a time).  FP32: 1.5 items
// per SM in steps of 128 (a 16-point group per warp of the accumulation);
// below that the items' fixed costs (a 41 KB block written and merged) win.
// Accumulation / interpolation in us, items of 1024, 512, 256, 128 points:
// 115 k points at 128^3 30 / 25, 30 / 18, 32 / 18, 36 / 20; 102 k points of
// tetrahedra at 104^3 42 / 26, 33 / 20, 38 / 22, 51 / 23; 1.38 M points at
// 256^3 149 / 110, 158 / 118, 177 / 124, 192 / 132.  FP64: 4 items per SM of a
// whole GB300 in steps of 64 (FP64 arithmetic alone takes microseconds per point
// and SM); its sums are grouped by item, so that their bits must not follow from
// the SMs that a part of the GPU, or another one, has.
constexpr int kFullSMs = 152;
int item_size(int precision, int64_t Q, int sms) {
  const int gran = precision == IB_FP64 ? 64 : 128;
  const int64_t items = precision == IB_FP64 ? 4 * kFullSMs : sms + sms / 2;
  const int64_t item = ((Q + items - 1) / items + gran - 1) / gran * gran;
  return (int)(item < gran ? gran : (item > kChunk ? kChunk : item));
}

// a tile of n points has at most 1 + n / min(item, kMinChunk) items
int64_t max_work_items(int ntiles, int64_t Q, int item) {
  const int64_t m = ntiles + Q / (item < kMinChunk ? item : kMinChunk) + 1;
  return Q > 0 && m > Q ? Q : m;
}

ib_status launch_classify_tiles(ib_plan* p, cudaStream_t s) {
  const int nt = p->ntiles, nb = classify_blocks(nt);
  auto classify = p->n_inst > 1 ? k_classify<true> : k_classify<false>;
  chain_launch(classify, nb, kT, 0, s, p->grid, p->inst, p->tile_inst, p->tile_cnt, nt,
               p->tile_nonempty, p->tile_near, p->tile_bcount, item_rule(p));
  chain_launch(k_compact, nb, kT, 0, s, p->tile_nonempty, p->tile_near, nt, p->tile_bcount, nb,
               p->tile_cnt, p->tile_vmax, p->tile_done, p->tile_start, p->tile_end, p->tile_slot,
               p->items, item_rule(p), p->tile_list_near, p->tile_counters);
  return cudaGetLastError() == cudaSuccess ? IB_OK : IB_ERR_CUDA;
}

}  // namespace ibfe
