// Direct (Fourier) solve of the fluid step: tables, workspace and launcher
// (spectral.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstring>

#include "ibfe.h"

namespace ibfe {

constexpr int kSpecMaxPasses = 8;

// One transform length: its radices in pass order, each pass's stride,
// twiddle step and reciprocal of the stride, and the table exp(-2 pi i j / n).
struct SpecDim {
  int n, np;
  int rad[kSpecMaxPasses], q[kSpecMaxPasses], tws[kSpecMaxPasses];
  unsigned magic[kSpecMaxPasses];
  const float2* tw;
};

struct SpecArgs {
  SpecDim x, y, z;
  // symbols (Re D, Im D, |D|^2, 0) of the forward differences, in the order
  // the modes are stored in (x: natural; y, z: digit-reversed)
  const float4 *symx, *symy, *symz;
  const int* posx;       // place of mode k in a transformed x line
  float2* spec;          // [4][n2][n1][pitch] modes 0 .. n0/2 of the four fields; then the tables
  int pitch;
  int xskew;             // shared-memory skew of the x lines per first-pass block
  int zsh, zen;          // shared-memory swap of the z lines
  int ahead;             // planes that a CTA of the y transforms prefetches ahead
  float alpha, nu;       // rho / dt, mu / h^2
  float inv_n, pscale;   // 1 / cells, -h / dt
};

struct Spectral {
  SpecArgs a;
  size_t smem_x, smem_y, smem_z;
  int threads_x, threads_y, threads_z;
};

// Lattices the direct solve takes: every length even, at most 1024, with no
// prime factor above 5.
bool spectral_supports(const int n[3]);
// IB_ERR_CAPACITY: no room for the workspace (the caller keeps its V-cycles).
// up: a stream of the caller's that nothing is queued on (the tables' upload,
// waited for)
ib_status spectral_create(Spectral* sp, const int n[3], double h, double rho, double mu,
                          double dt, cudaStream_t up);
void spectral_destroy(Spectral* sp);
// keep: leave the increment w in the rows of a.spec (for the residuals)
ib_status spectral_step(const Spectral* sp, const float* u, const float* f, float* un, float* p,
                        bool keep, cudaStream_t s);
// partial sums of the squared residuals and right-hand sides, four per CTA
void launch_spectral_resid(const Spectral* sp, const float* u, const float* f, const float* p,
                           double a, double nu, double dtoh, double* part, int ctas,
                           cudaStream_t s);

}  // namespace ibfe
