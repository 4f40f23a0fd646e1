// Host side of the hyperelastic nodal force (Section 4.4) and its adjoints:
// the choice of kernel instantiation per call, and the deterministic
// per-material reductions of energies and parameter gradients.  The device
// code is in fe_kernel.cuh.
#include <algorithm>

#include "dfloat.cuh"
#include "ib_device.cuh"

namespace ibfe {
namespace {

// Deterministic per-material sums of per-element partials, one launch.
// Material m's elements lie in the range mrange[m] (the whole mesh for a plan
// of one structure; its instance's elements in a packed plan), cut into at
// most kReduceCTAs chunks of at least kRedMin elements; CTA per_mat m + b sums
// its chunk b (one grid dimension: a packed plan may have more materials than
// the others hold): each thread its elements in order, then one warp per value the threads'
// sums (eight per lane, then a shuffle tree).  The CTA that completes its
// material's count adds the chunks' sums, again one warp per value in a fixed
// order.  The partition and the trees depend only on the range, so an
// instance of a packed plan gets the bits of a plan of its own.
//
// FP64 adds run at 1/64 of the FP32 rate on GB300, and this kernel runs
// beside the spreading: a value takes 12 warp-wide adds per CTA (every warp's
// own tree for each value took 50), and materials have their own CTAs instead
// of being visited in turn by all of them.  Packed sweep of 16 shells, beside
// the spreading: 346 + 20 us before (two levels, every CTA through every
// material); 256^3 backward 125 + 6 us.
__device__ __forceinline__ double warp_tree(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;  // valid in lane 0
}

constexpr int kRedThreads = 256;
constexpr int kRedMin = 1024;

template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_reduce(const T* __restrict__ part,
                                                        const int32_t* __restrict__ mat_id,
                                                        const int2* __restrict__ mrange, int E,
                                                        int nvals, int per_mat, double* rpart,
                                                        int* count, double* __restrict__ out) {
  chain_wait();
  __shared__ double sh[kParamRow][kRedThreads];
  __shared__ bool last;
  const int m = blockIdx.x / per_mat, b = blockIdx.x % per_mat;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int2 r = mrange[m];
  const int len = r.y - r.x;
  const int chunk = max(kRedMin, (len + kReduceCTAs - 1) / kReduceCTAs);
  const int nblk = max(1, (len + chunk - 1) / chunk);
  if (b >= nblk) return;
  const int e0 = r.x + b * chunk, e1 = min(r.y, e0 + chunk);
  double s[kParamRow];
#pragma unroll
  for (int k = 0; k < kParamRow; ++k) s[k] = 0.0;
#pragma unroll 2
  for (int e = e0 + threadIdx.x; e < e1; e += kRedThreads)
    if ((mat_id ? __ldg(mat_id + e) : 0) == m) {
#pragma unroll
      for (int k = 0; k < kParamRow; ++k)
        if (k < nvals) s[k] += double(__ldg(part + (int64_t)k * E + e));
    }
#pragma unroll
  for (int k = 0; k < kParamRow; ++k)
    if (k < nvals) sh[k][threadIdx.x] = s[k];
  __syncthreads();
  double* mine = rpart + (int64_t)m * kReduceCTAs * kParamRow;
  for (int k = warp; k < nvals; k += kRedThreads / 32) {
    double v = 0.0;
#pragma unroll
    for (int t = 0; t < kRedThreads / 32; ++t) v += sh[k][32 * t + lane];
    v = warp_tree(v);
    if (lane == 0) {
      if (nblk == 1)
        out[m * kParamRow + k] = v;
      else
        mine[b * kParamRow + k] = v;
    }
  }
  if (nblk == 1) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(count + m, 1) + 1 == nblk;
    if (last) count[m] = 0;  // for the next call
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int k = warp; k < nvals; k += kRedThreads / 32) {
    double v = 0.0;
    for (int i = lane; i < nblk; i += 32) v += __ldcg(mine + i * kParamRow + k);
    v = warp_tree(v);
    if (lane == 0) out[m * kParamRow + k] = v;
  }
}

// The smallest instantiated law set covering the material table (every
// model in it, the active term if a material has T_a != 0 or the parameter
// gradients are wanted: they include d/dT_a).
int law_set(const ib_plan* p, const MatTable& mt, bool params) {
  int need = params ? kLawAct : 0;
  if (p->mat_dev) need |= p->mat_need;  // packed plans: the device table's laws
  for (int m = 0; m < mt.n; ++m) {
    need |= 1 << mt.model[m];
    if (mt.p[m][kTa] != 0.0) need |= kLawAct;
  }
  if ((need & ~kLawBase) == 0) return kLawBase;
  if ((need & ~kLawBaseAct) == 0) return kLawBaseAct;
  return kLawAll;
}

}  // namespace

#define IBFE_FE_ARGS p, mt, xa, off, v, out, s
#define HEX IB_ELEM_HEX8

namespace {
// IB_FP32_SPLIT_DFVOL plans: every law, the exact volumetric invariant; one
// instantiation per element and output.
constexpr int kLawVol = kLawAll | kLawVolX;
template <int T>
ib_status vol_force(ib_plan* p, const MatTable& mt, const void* xa, const float* off,
                    const void* v, void* out, bool energy, bool adj, bool params,
                    cudaStream_t s) {
  if (adj)
    return params ? fe_run<float, df, false, true, true, kLawVol, T>(IBFE_FE_ARGS)
                  : fe_run<float, df, false, true, false, kLawVol, T>(IBFE_FE_ARGS);
  return energy ? fe_run<float, df, true, false, false, kLawVol, T>(IBFE_FE_ARGS)
                : fe_run<float, df, false, false, false, kLawVol, T>(IBFE_FE_ARGS);
}

// Tetrahedral meshes (P1 and P2): one instantiation per precision and
// output (all laws).
template <int T>
ib_status tet_force(ib_plan* p, const MatTable& mt, const void* xa, const float* off,
                    const void* v, void* out, bool energy, bool adj, bool params,
                    cudaStream_t s) {
  constexpr int L = kLawAll;
  if (p->precision == IB_FP64) {
    if (adj)
      return params ? fe_run<double, double, false, true, true, L, T>(IBFE_FE_ARGS)
                    : fe_run<double, double, false, true, false, L, T>(IBFE_FE_ARGS);
    return energy ? fe_run<double, double, true, false, false, L, T>(IBFE_FE_ARGS)
                  : fe_run<double, double, false, false, false, L, T>(IBFE_FE_ARGS);
  }
  if (p->precision == IB_FP32_SPLIT_F32STAB) {
    if (adj)
      return params ? fe_run<float, float, false, true, true, L, T>(IBFE_FE_ARGS)
                    : fe_run<float, float, false, true, false, L, T>(IBFE_FE_ARGS);
    return energy ? fe_run<float, float, true, false, false, L, T>(IBFE_FE_ARGS)
                  : fe_run<float, float, false, false, false, L, T>(IBFE_FE_ARGS);
  }
  if (p->precision == IB_FP32_SPLIT_DFVOL) return vol_force<T>(p, mt, xa, off, v, out, energy,
                                                               adj, params, s);
  if (adj)
    return params ? fe_run<float, df, false, true, true, L, T>(IBFE_FE_ARGS)
                  : fe_run<float, df, false, true, false, L, T>(IBFE_FE_ARGS);
  return energy ? fe_run<float, df, true, false, false, L, T>(IBFE_FE_ARGS)
                : fe_run<float, df, false, false, false, L, T>(IBFE_FE_ARGS);
}
}  // namespace

ib_status launch_fe_force(ib_plan* p, const MatTable& mt, const void* xa, const float* off,
                          void* out, bool energy, cudaStream_t s) {
  const void* v = nullptr;
  if (p->elem == IB_ELEM_TET4)
    return tet_force<IB_ELEM_TET4>(p, mt, xa, off, v, out, energy, false, false, s);
  if (p->elem == IB_ELEM_TET10)
    return tet_force<IB_ELEM_TET10>(p, mt, xa, off, v, out, energy, false, false, s);
  const int set = law_set(p, mt, false);
  if (p->precision == IB_FP32_SPLIT_DFVOL)
    return vol_force<HEX>(p, mt, xa, off, v, out, energy, false, false, s);
  if (p->precision == IB_FP64)
    return energy ? fe_run<double, double, true, false, false, kLawAll, HEX>(IBFE_FE_ARGS)
                  : fe_run<double, double, false, false, false, kLawAll, HEX>(IBFE_FE_ARGS);
  if (p->precision == IB_FP32_SPLIT_F32STAB) {
    if (energy) return fe_run<float, float, true, false, false, kLawAll, HEX>(IBFE_FE_ARGS);
    return set == kLawBase
               ? fe_run<float, float, false, false, false, kLawBase, HEX>(IBFE_FE_ARGS)
               : fe_run<float, float, false, false, false, kLawAll, HEX>(IBFE_FE_ARGS);
  }
  if (energy) return fe_run<float, df, true, false, false, kLawAll, HEX>(IBFE_FE_ARGS);
  if (set == kLawBase)
    return fe_run<float, df, false, false, false, kLawBase, HEX>(IBFE_FE_ARGS);
  if (set == kLawBaseAct)
    return fe_run<float, df, false, false, false, kLawBaseAct, HEX>(IBFE_FE_ARGS);
  return fe_run<float, df, false, false, false, kLawAll, HEX>(IBFE_FE_ARGS);
}

ib_status launch_fe_force_adj(ib_plan* p, const MatTable& mt, const void* xa, const float* off,
                              const void* v, void* out, bool params, cudaStream_t s) {
  if (p->elem == IB_ELEM_TET4)
    return tet_force<IB_ELEM_TET4>(p, mt, xa, off, v, out, false, true, params, s);
  if (p->elem == IB_ELEM_TET10)
    return tet_force<IB_ELEM_TET10>(p, mt, xa, off, v, out, false, true, params, s);
  const int set = law_set(p, mt, params);
  if (p->precision == IB_FP32_SPLIT_DFVOL)
    return vol_force<HEX>(p, mt, xa, off, v, out, false, true, params, s);
  if (p->precision == IB_FP64)
    return params ? fe_run<double, double, false, true, true, kLawAll, HEX>(IBFE_FE_ARGS)
                  : fe_run<double, double, false, true, false, kLawAll, HEX>(IBFE_FE_ARGS);
  if (p->precision == IB_FP32_SPLIT_F32STAB)
    return params ? fe_run<float, float, false, true, true, kLawAll, HEX>(IBFE_FE_ARGS)
                  : fe_run<float, float, false, true, false, kLawAll, HEX>(IBFE_FE_ARGS);
  if (params)
    return set == kLawBaseAct
               ? fe_run<float, df, false, true, true, kLawBaseAct, HEX>(IBFE_FE_ARGS)
               : fe_run<float, df, false, true, true, kLawAll, HEX>(IBFE_FE_ARGS);
  if (set == kLawBase) return fe_run<float, df, false, true, false, kLawBase, HEX>(IBFE_FE_ARGS);
  if (set == kLawBaseAct)
    return fe_run<float, df, false, true, false, kLawBaseAct, HEX>(IBFE_FE_ARGS);
  return fe_run<float, df, false, true, false, kLawAll, HEX>(IBFE_FE_ARGS);
}

#undef HEX
#undef IBFE_FE_ARGS

ib_status launch_reduce_parts(ib_plan* p, int nvals, int n_mats, cudaStream_t s,
                              bool real_parts, double* out) {
  if (n_mats > p->mat_cap) return IB_ERR_INVALID_ARG;
  if (!out) out = p->ered;
  if (p->E == 0) {
    cudaMemsetAsync(out, 0, sizeof(double) * kParamRow * n_mats, s);
    return cudaGetLastError() == cudaSuccess ? IB_OK : IB_ERR_CUDA;
  }
  // chunks any material can have: the whole mesh's
  const int nblk = std::min(kReduceCTAs, (p->E + kRedMin - 1) / kRedMin);
  const unsigned grid = (unsigned)nblk * (unsigned)n_mats;
  // FP32 partials are widened exactly: the sums are those of their doubles
  if (real_parts && p->precision != IB_FP64)
    chain_launch(k_reduce<float>, grid, kRedThreads, 0, s, reinterpret_cast<const float*>(p->epart),
                 p->mat_id, p->mat_range, p->E, nvals, nblk, p->rpart, p->red_count, out);
  else
    chain_launch(k_reduce<double>, grid, kRedThreads, 0, s, p->epart, p->mat_id, p->mat_range, p->E,
                 nvals, nblk, p->rpart, p->red_count, out);
  return cudaGetLastError() == cudaSuccess ? IB_OK : IB_ERR_CUDA;
}

}  // namespace ibfe
