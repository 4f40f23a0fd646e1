// Direct solve of the fluid step (Section 4.2) on the periodic MAC grid, FP32.
//
// On a periodic lattice the Helmholtz and Poisson operators of Chorin's
// projection are circulant, so one discrete Fourier transform diagonalises
// the whole step.  It is solved for the increment w = u^{n+1} - u^n:
//   (a - mu Lap_h) d = f + mu Lap_h u^n                 (a = rho / dt, u* = u^n + d)
//   Lap_h p = (div_h u^n + div_h d) / dt
//   w = d - dt grad_h p
// The four right-hand fields r_c = f_c + mu Lap_h u_c (c = 0..2) and
// r_3 = h div_h u^n are formed from the stencils in FP32 before the transform:
// div_h u is a difference of neighbours (no cancellation against transformed
// velocities, whose rounding would enter p multiplied by |u| / dt), and the
// transform's rounding is relative to the increment, not to u.
// With the forward-difference symbols D_d = exp(2 pi i k_d / n_d) - 1 and
// S = sum_d |D_d|^2, per mode
//   d_c = r_c / (a + mu S / h^2),   q = (r_3 + sum_d D_d d_d) / S   (0 at k = 0),
//   w_c = d_c - conj(D_c) q,        p = -(h / dt) q.
//
// Five kernels (each reads and writes every mode once):
//   k_spec_rhs    stencils and the x transform; two rows of a field make one
//                 complex line, unpacked to n0/2 + 1 modes per row
//   k_spec_y<0>   y transform, 16 adjacent modes x one line per thread group
//   k_spec_solve  z transform of the four fields, the algebra above and the
//                 inverse z transform, without leaving the SM
//   k_spec_y<1>   inverse y transform
//   k_spec_out    inverse x transform, u_next = u + w and p
// Transforms are in place: decimation in frequency forward (natural order in,
// digit-reversed order out), decimation in time backward, so no pass permutes
// anything and a butterfly owns its places; the symbols are tabulated in the
// order the modes are stored in.  Each transform's first pass reads global
// memory and its last pass writes it.
//
// Order of the planes: each kernel starts with what the one before it wrote
// last, which L2 still holds (k_spec_y<0> and k_spec_out walk the planes
// backwards): at 256^3 k_spec_out 157 -> 140 us.  Loads that would wait for
// memory behind the transforms are asked for early: k_spec_out's velocity rows
// at its start (177 -> 157 us), the rows that k_spec_rhs is the first to read
// (171 -> 163), the y transforms' lines one wave of CTAs ahead (106 -> 91).  A wave ahead for k_spec_rhs (171 -> 204), the solve (158 -> 168)
// and k_spec_out's modes (140 -> 159) costs more than it hides.
//
// Measured on GB300 (us; V-cycles of fluid.cu before, this after, steps back to
// back): 32^3 632 -> 22, 192^3 3416 -> 284, 256^3 6550 -> 610.  At 256^3 the five
// kernels take 164, 83, 151, 83 and 133 us (ncu) for 0.64, 0.50, 0.50, 0.50 and
// 0.69 GB: 3.9, 6.0, 3.3, 6.0 and 5.2 TB/s; k_spec_rhs and the solve issue on 56
// and 58% of their cycles beside their loads' latency (bank conflicts and L1
// requests taken out of k_spec_rhs change nothing).  Choices measured before
// the lengths were compiled in: x lines use radices up to 8 (48 registers, 5
// CTAs per SM: 184 against 250 us with radix 16 for k_spec_out); y lines up to
// 16 (two passes at 256: 104 against 114..130 us); the z transform holds four
// fields, 3 CTAs per SM (175 us; 2: 208, 4 with spills: 211).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <utility>
#include <vector>

#include "ib_internal.cuh"
#include "spectral.cuh"

namespace ibfe {
namespace {

constexpr int kTX = 16;   // modes per tile of the y transform (128-byte rows)
constexpr int kTZ = 8;    // modes per tile of the z transform (four fields in shared memory)
constexpr int kMaxN = 1024;

// Sums and differences of both parts in one instruction (the packed FP32
// arithmetic of this GPU; each part is rounded as by its own instruction).
// The compiler forms none from the scalar code: the solve at 192^3 75.6 ->
// 72.2 us, the inverse y transform 59.7 -> 56.3.  Products stay scalar: a
// complex one would need its factors swapped and doubled in registers.
__device__ __forceinline__ unsigned long long as_pair(float2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ float2 from_pair(unsigned long long r) {
  float2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
  return a;
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_pair(a)), "l"(as_pair(b)));
  return from_pair(r);
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_pair(a)), "l"(as_pair(b)));
  return from_pair(r);
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// a times -i (forward) or i (inverse)
template <bool kInv>
__device__ __forceinline__ float2 rot(float2 a) {
  return kInv ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// R-point transforms in registers, natural order (exponent sign - forward, + inverse)
template <int R, bool kInv>
struct Dft;
template <bool kInv>
struct Dft<2, kInv> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  }
};
template <bool kInv>
struct Dft<3, kInv> {
  static __device__ __forceinline__ void run(float2* v) {
    constexpr float s3 = 0.86602540378443864676f;  // sin(2 pi / 3)
    const float2 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const float2 m = make_float2(v[0].x - 0.5f * t.x, v[0].y - 0.5f * t.y);
    const float2 s = rot<kInv>(make_float2(s3 * d.x, s3 * d.y));
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, s);
    v[2] = csub(m, s);
  }
};
template <bool kInv>
struct Dft<4, kInv> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    const float2 t2 = cadd(v[1], v[3]), t3 = rot<kInv>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[1] = cadd(t1, t3);
    v[2] = csub(t0, t2);
    v[3] = csub(t1, t3);
  }
};
template <bool kInv>
struct Dft<5, kInv> {
  static __device__ __forceinline__ void run(float2* v) {
    constexpr float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    constexpr float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
    const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const float2 t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const float2 m1 = make_float2(v[0].x + c1 * t1.x + c2 * t2.x, v[0].y + c1 * t1.y + c2 * t2.y);
    const float2 m2 = make_float2(v[0].x + c2 * t1.x + c1 * t2.x, v[0].y + c2 * t1.y + c1 * t2.y);
    const float2 e1 = rot<kInv>(make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y));
    const float2 e2 = rot<kInv>(make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y));
    v[0] = make_float2(v[0].x + t1.x + t2.x, v[0].y + t1.y + t2.y);
    v[1] = cadd(m1, e1);
    v[4] = csub(m1, e1);
    v[2] = cadd(m2, e2);
    v[3] = csub(m2, e2);
  }
};

// cos and sin of 2 pi j / R for the composite radices
template <int R>
__device__ constexpr float kCosT(int j) {
  constexpr float c16[16] = {1.f, 0.92387953251128675613f, 0.70710678118654752440f,
                             0.38268343236508977173f, 0.f, -0.38268343236508977173f,
                             -0.70710678118654752440f, -0.92387953251128675613f, -1.f,
                             -0.92387953251128675613f, -0.70710678118654752440f,
                             -0.38268343236508977173f, 0.f, 0.38268343236508977173f,
                             0.70710678118654752440f, 0.92387953251128675613f};
  constexpr float c6[6] = {1.f, 0.5f, -0.5f, -1.f, -0.5f, 0.5f};
  return R == 6 ? c6[j % 6] : c16[(j * (16 / (R == 6 ? 16 : R))) % 16];
}
template <int R>
__device__ constexpr float kSinT(int j) {
  constexpr float s3 = 0.86602540378443864676f;
  constexpr float s6[6] = {0.f, s3, s3, 0.f, -s3, -s3};
  // sin(2 pi j / 16) = cos(2 pi (j - 4) / 16)
  return R == 6 ? s6[j % 6] : kCosT<16>((j * (16 / (R == 6 ? 16 : R)) + 12) % 16);
}

// R = R1 R2: n = R2 n1 + n2, k = k1 + R1 k2
template <int R1, int R2, bool kInv>
struct DftC {
  static __device__ __forceinline__ void run(float2* v) {
    constexpr int R = R1 * R2;
    float2 t[R];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      float2 a[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) a[n1] = v[R2 * n1 + n2];
      Dft<R1, kInv>::run(a);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) {
        const int e = n2 * k1;
        if (e == 0)
          t[k1 * R2 + n2] = a[k1];
        else if (4 * e == R)
          t[k1 * R2 + n2] = rot<kInv>(a[k1]);
        else
          t[k1 * R2 + n2] =
              cmul(a[k1], make_float2(kCosT<R>(e), kInv ? kSinT<R>(e) : -kSinT<R>(e)));
      }
    }
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      Dft<R2, kInv>::run(t + k1 * R2);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) v[k1 + R1 * k2] = t[k1 * R2 + k2];
    }
  }
};
template <bool kInv>
struct Dft<6, kInv> : DftC<3, 2, kInv> {};
template <bool kInv>
struct Dft<8, kInv> : DftC<2, 4, kInv> {};
template <bool kInv>
struct Dft<16, kInv> : DftC<4, 4, kInv> {};

// Passes of a transform of length n along dimension d: the radices (their
// product n, at least two of them; np = 0 if n has a prime factor above 5), in
// descending order, fewest passes first, then the smallest sum.  x (d = 0):
// radices up to 8; y: up to 16; z: the last one at most 5 (the solve holds
// four fields' last butterflies in registers).
struct Plan {
  int np;
  int rad[kSpecMaxPasses], q[kSpecMaxPasses], tws[kSpecMaxPasses];
  unsigned magic[kSpecMaxPasses];
};
__host__ __device__ constexpr void plan_search(int left, int depth, int sum, int first, int last,
                                               int (&cur)[kSpecMaxPasses], int& best_sum,
                                               Plan& best) {
  constexpr int all[7] = {16, 8, 6, 5, 4, 3, 2};
  if (left == 1) {
    if (depth < 2 || cur[depth - 1] > last) return;
    if (best.np == 0 || depth < best.np || (depth == best.np && sum < best_sum)) {
      best.np = depth;
      best_sum = sum;
      for (int i = 0; i < depth; ++i) best.rad[i] = cur[i];
    }
    return;
  }
  if (depth >= kSpecMaxPasses) return;
  for (int r : all) {
    if (r > first || left % r || (depth > 0 && r > cur[depth - 1])) continue;
    cur[depth] = r;
    plan_search(left / r, depth + 1, sum + r, first, last, cur, best_sum, best);
  }
}
__host__ __device__ constexpr Plan make_plan(int n, int d) {
  Plan p = {};
  int cur[kSpecMaxPasses] = {}, best = 0, odd = n;
  while (odd % 2 == 0) odd /= 2;
  while (odd % 3 == 0) odd /= 3;
  while (odd % 5 == 0) odd /= 5;
  if (odd != 1) return p;
  plan_search(n, 0, 0, d == 0 ? 8 : 16, d == 0 ? 8 : (d == 1 ? 16 : 5), cur, best, p);
  int L = n;
  for (int i = 0; i < p.np; ++i) {
    p.q[i] = L / p.rad[i];
    p.tws[i] = n / L;
    p.magic[i] = (1u << 20) / p.q[i] + 1;
    L /= p.rad[i];
  }
  return p;
}

// Threads of a CTA whose columns are `w` wide: one butterfly of the first
// (largest) radix each, or an equal number each.
__host__ __device__ constexpr int col_threads(int n, int r0, int w) {
  const int rows = n / r0;
  int t = (rows + 256 / w - 1) / (256 / w);
  while (rows % t && t < rows) ++t;
  const int th = w * (rows / t);
  return th < 32 ? 32 : th;
}

// Threads of the x and y kernels' CTAs, known with the length, and how many
// such CTAs 48 registers a thread let an SM hold.  Bounding each instance by
// its own CTA instead of 256 threads gives the 192-thread ones 56 registers at
// the same occupancy: the forward y transform at 192^3 58 -> 51 us, the
// inverse x transform 72 -> 69.
template <int N, int d>
constexpr int cta_threads() {
  if constexpr (N == 0)
    return 256;
  else
    return col_threads(N, make_plan(N, d).rad[0], 16);
}
constexpr int ctas_at_48(int threads) { return 1280 / threads; }

// One pass over blocks of L = R Q places: butterfly j takes the places
// b R Q + m + r Q, r < R, with b = j / Q and m = j mod Q.  magic = 2^20 / Q + 1
// divides by Q exactly for j < n <= 1024.
struct Pass {
  int R, Q, tws;   // radix, stride, twiddle step n / L
  unsigned magic;
};

// The transforms along dimension d, of length N: known at compile time (2^k, 3 2^k
// and 5 2^k from 32 to 512: strides, addresses and trip counts are
// immediates, some 30% fewer instructions per pass), or N = 0: any length, the
// plan read from the arguments.
template <int N, int d>
struct Dim {
  static constexpr Plan P = make_plan(N, d);
};
template <int d>
struct Dim<0, d> {};

// Butterflies j0, j0 + step, ... of one pass on NF lines that share their
// twiddles (the fields of the z transform; 1 elsewhere).  A.place(p0, Q) gives
// the butterfly's address base, A.ld / A.st move place p0 + r Q of line c.
// Forward: transform, then twiddles; inverse: conjugate twiddles, then
// transform.
template <int R, bool kInv, int NF, bool kKnown, typename In, typename Out>
__device__ __forceinline__ void pass_r(const Pass P, int n, int j0, int step,
                                       const float2* __restrict__ tw, const In& in,
                                       const Out& out) {
  if (kKnown) __builtin_assume(j0 >= 0 && j0 < step);
#pragma unroll 1
  for (int j = j0; j < n / R; j += step) {
    const int b = kKnown ? (int)((unsigned)j / (unsigned)P.Q) : (int)(((unsigned)j * P.magic) >> 20);
    const int m = j - b * P.Q, p0 = b * R * P.Q + m;
    constexpr bool kHold = NF > 1 && R <= 8;  // twiddles kept over the lines
    float2 w[kHold ? R : 1];
    if (kHold && P.Q > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) w[r] = __ldg(tw + m * r * P.tws);
    }
    auto twid = [&](int r) { return kHold ? w[r] : __ldg(tw + m * r * P.tws); };
    const auto pi = in.place(p0, P.Q);
    const auto po = out.place(p0, P.Q);
#pragma unroll 1
    for (int c = 0; c < NF; ++c) {
      float2 v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = in.ld(pi, c, r);
      if (kInv && P.Q > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = cmulc(v[r], twid(r));
      }
      Dft<R, kInv>::run(v);
      if (!kInv && P.Q > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = cmul(v[r], twid(r));
      }
#pragma unroll
      for (int r = 0; r < R; ++r) out.st(po, c, r, v[r]);
    }
  }
}

// Pass i of the transform (i known at compile time when N is).
template <int N, int d, int i, bool kInv, int NF, typename In, typename Out>
__device__ __forceinline__ void known_pass(int j0, const float2* __restrict__ tw, const In& in,
                                           const Out& out, int step) {
  constexpr Plan P = Dim<N, d>::P;
  pass_r<P.rad[i], kInv, NF, true>(Pass{P.rad[i], P.q[i], P.tws[i], P.magic[i]}, N, j0, step, tw,
                                   in, out);
}
template <bool kInv, int NF, bool k16, typename In, typename Out>
__device__ __forceinline__ void any_pass(const SpecDim& D, int i, int j0, int step, const In& in,
                                         const Out& out) {
  const Pass P{D.rad[i], D.q[i], D.tws[i], D.magic[i]};
  switch (P.R) {
    case 2: pass_r<2, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 3: pass_r<3, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 4: pass_r<4, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 5: pass_r<5, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 6: pass_r<6, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 8: pass_r<8, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out); break;
    case 16:
      if constexpr (k16) pass_r<16, kInv, NF, false>(P, D.n, j0, step, D.tw, in, out);
      break;
  }
}

// Passes [from, to) of a transform within shared memory, in execution order
// (pass e executes the plan's pass e forward, np - 1 - e inverse), a barrier
// after each.
template <int N, int d, bool kInv, int NF, int e, int to, typename S>
__device__ __forceinline__ void known_passes(int j0, int step, const float2* tw, const S& s) {
  if constexpr (e < to) {
    constexpr int np = Dim<N, d>::P.np;
    known_pass<N, d, kInv ? np - 1 - e : e, kInv, NF>(j0, tw, s, s, step);
    __syncthreads();
    known_passes<N, d, kInv, NF, e + 1, to>(j0, step, tw, s);
  }
}

// A base address and the steps between the butterfly's places (even and odd r
// start from a and b).
struct Place {
  int a, b, step;
  __device__ __forceinline__ int at(int r) const { return ((r & 1) ? b : a) + r * step; }
};

// Column of a [place][mode] array in global memory, masked beyond the last mode
struct GlobalCol {
  float2* g;
  int pitch;        // between places
  int64_t field;    // between the lines c
  bool on;
  __device__ __forceinline__ Place place(int p0, int Q) const {
    const int a = p0 * pitch;
    return Place{a, a, Q * pitch};
  }
  __device__ __forceinline__ float2 ld(const Place& p, int c, int r) const {
    return on ? g[c * field + p.at(r)] : make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void st(const Place& p, int c, int r, float2 v) const {
    if (on) g[c * field + p.at(r)] = v;
  }
};

// Column of a [place][width] array in shared memory.  width 16: a half-warp's
// 16 columns of one place fill the 32 banks.  width 8: two places share them,
// and the places whose (p >> sh) is odd swap with their neighbour (p ^ 1), so
// that butterflies 2^sh places apart (the last pass) differ in parity; every
// other pass's stride is a multiple of 2^sh, so the swap is one of two bases.
// en = 0: no swap (odd last radix: neighbours already differ).
__host__ __device__ constexpr int swap_shift(int last) { return last == 4 ? 2 : 1; }
__host__ __device__ constexpr int swap_on(int last) { return last % 2 == 0 ? 1 : 0; }
template <int kW>
struct SharedCol {
  float2* s;
  int field, sh, en;
  __device__ __forceinline__ Place place(int p0, int Q) const {
    if (kW == 16) return Place{p0 * kW, p0 * kW, Q * kW};
    const int a = p0 ^ ((p0 >> sh) & en);
    return Place{a * kW, (a ^ ((Q >> sh) & en)) * kW, Q * kW};
  }
  __device__ __forceinline__ float2 ld(const Place& p, int c, int r) const {
    return s[c * field + p.at(r)];
  }
  __device__ __forceinline__ void st(const Place& p, int c, int r, float2 v) const {
    s[c * field + p.at(r)] = v;
  }
};

// Lines of the x transforms, [place][16 lines] with a row pitch of 17 (the
// load and store phases run along the places) and one more skew per block of
// the first pass's stride Q1: consecutive modes lie Q1 places apart, and
// 17 Q1 + skew = 1 (mod 16) spreads them over the banks.
constexpr int kXL = 16;  // lines: four row pairs x four fields
constexpr int kXP = kXL + 1;
__host__ __device__ constexpr int line_skew(int Q1) { return ((1 - Q1) % 16 + 16) % 16; }
template <int N>
struct LineSmem {
  float2* s;
  int Q1, skew;
  unsigned magic1;
  __device__ __forceinline__ LineSmem(const SpecArgs& A, float2* p) : s(p) {
    if constexpr (N > 0) {
      Q1 = Dim<N, 0>::P.q[0];
      skew = line_skew(Dim<N, 0>::P.q[0]);
      magic1 = 0;
    } else {
      Q1 = A.x.q[0];
      skew = A.xskew;
      magic1 = A.x.magic[0];
    }
  }
  __device__ __forceinline__ int addr(int p) const {
    return p * kXP + (N > 0 ? (int)((unsigned)p / (unsigned)Q1) : (int)(((unsigned)p * magic1) >> 20)) * skew;
  }
  __device__ __forceinline__ Place place(int p0, int Q) const {
    const int a = addr(p0);
    return Place{a, a, Q * kXP + (Q == Q1 ? skew : 0)};
  }
  __device__ __forceinline__ float2 ld(const Place& p, int, int r) const { return s[p.at(r)]; }
  __device__ __forceinline__ void st(const Place& p, int, int r, float2 v) const {
    s[p.at(r)] = v;
  }
};

__device__ __forceinline__ int up(int i, int n) { return i + 1 == n ? 0 : i + 1; }
__device__ __forceinline__ int dn(int i, int n) { return i == 0 ? n - 1 : i - 1; }

// kV adjacent cells of a row (kV = 2: 8-byte aligned)
template <int kV>
__device__ __forceinline__ void ld_cells(float* v, const float* __restrict__ g) {
  if (kV == 2) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(g));
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = __ldg(g);
  }
}

// Requests to bring memory to L2: the 128-byte line at g; the 16-byte blocks
// that lie within [g, g + bytes).
__device__ __forceinline__ void prefetch_line(const void* g) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(g));
}
__device__ __forceinline__ void prefetch_rows(const void* g, int bytes) {
  const uintptr_t a = (reinterpret_cast<uintptr_t>(g) + 15) & ~(uintptr_t)15;
  const uintptr_t e = (reinterpret_cast<uintptr_t>(g) + bytes) & ~(uintptr_t)15;
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)(e - a))
                 : "memory");
}

// The lines a warp of a CTA of `threads` threads takes are first_line(warp),
// and from there every (threads / 32)-th.  CTAs are multiples of 16 threads (a
// column each per place): the half warp that some end in takes no line, as the
// full warps take them all.  (The threads are read from the launch: with the
// compile-time number in the kernels' line loops 256^3 610 -> 624 us.)
__host__ __device__ constexpr int first_line(int warp, int threads) {
  return warp < threads / 32 ? warp : kXL;
}
constexpr bool each_line_once() {
  for (int threads = 32; threads <= 256; threads += 16)
    for (int l = 0; l < kXL; ++l) {
      int takers = 0;
      for (int w = 0; w < (threads + 31) / 32; ++w)
        for (int k = first_line(w, threads); k < kXL; k += threads / 32) takers += k == l;
      if (takers != 1) return false;
    }
  return true;
}
static_assert(each_line_once(), "two warps on a line would race on its places and modes");

// Transforms the 16 lines held in shared memory.
template <bool kInv, int N>
__device__ __forceinline__ void line_passes(const SpecArgs& A, float2* z) {
  const LineSmem<N> L(A, z + (threadIdx.x & (kXL - 1)));
  if constexpr (N > 0) {
    constexpr int step = col_threads(N, Dim<N, 0>::P.rad[0], kXL) / kXL;
    known_passes<N, 0, kInv, 1, 0, Dim<N, 0>::P.np>(threadIdx.x / kXL, step, A.x.tw, L);
  } else {
    for (int i = 0; i < A.x.np; ++i) {
      any_pass<kInv, 1, false>(A.x, kInv ? A.x.np - 1 - i : i, threadIdx.x / kXL,
                               blockDim.x / kXL, L, L);
      __syncthreads();
    }
  }
}

// Row pairs 4 b .. 4 b + 3 of plane k (b = blockIdx.x): the four fields'
// right-hand sides as complex lines (first row of the pair real, second
// imaginary), their x transform, and the modes 0 .. n0/2 of every row.  Line
// l = 4 (pair) + field.
template <int kV, int N>
__global__ void __launch_bounds__(cta_threads<N, 0>(), ctas_at_48(cta_threads<N, 0>()))
    k_spec_rhs(SpecArgs A, const float* __restrict__ u,
                                                  const float* __restrict__ f) {
  chain_wait();
  chain_next();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* z = reinterpret_cast<float2*>(smem_raw);
  const LineSmem<N> L(A, z);
  const int n0 = N > 0 ? N : A.x.n, n1 = A.y.n, n2 = A.z.n;
  const int k = blockIdx.y, jp0 = blockIdx.x * 4, np = min(4, n1 / 2 - jp0);
  const int cells = n0 * n1 * n2;
  // the rows that no CTA of an earlier plane has read: u above, f here
  if (threadIdx.x < 6 && (threadIdx.x < 3 || f))
    prefetch_rows((threadIdx.x < 3 ? u + threadIdx.x * cells + up(k, n2) * n1 * n0
                                   : f + (threadIdx.x - 3) * cells + k * n1 * n0) +
                      2 * jp0 * n0,
                  sizeof(float) * 2 * np * n0);
  const int kp = up(k, n2) * n1, km = dn(k, n2) * n1, kc = k * n1;
  // a thread forms kV cells of a row pair; work (pair, cells) laid out flat
  const int nv = n0 / kV;
  int rp = threadIdx.x / nv, iv = threadIdx.x - rp * nv;
  while (rp < 4) {
    const int i = iv * kV;
    if (rp < np) {
      const int ip = i + kV == n0 ? 0 : i + kV, im = dn(i, n0);
      const int j = 2 * (jp0 + rp);
      const int r0 = (kc + j) * n0, r1 = r0 + n0;
      const int ra = (kc + dn(j, n1)) * n0 + i, rc = (kc + up(j + 1, n1)) * n0 + i;
      const int ru = (kp + j) * n0 + i, rd = (km + j) * n0 + i;
      float div0[kV], div1[kV];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float* uc = u + c * cells;
        float v0[kV + 1], v1[kV + 1], y2[kV], z0[kV], z1[kV];
        ld_cells<kV>(v0, uc + r0 + i);
        ld_cells<kV>(v1, uc + r1 + i);
        v0[kV] = __ldg(uc + r0 + ip);
        v1[kV] = __ldg(uc + r1 + ip);
        ld_cells<kV>(y2, uc + rc);
        ld_cells<kV>(z0, uc + ru);
        ld_cells<kV>(z1, uc + ru + n0);
#pragma unroll
        for (int e = 0; e < kV; ++e) {
          if (c == 0) div0[e] = v0[e + 1] - v0[e], div1[e] = v1[e + 1] - v1[e];
          if (c == 1) div0[e] += v1[e] - v0[e], div1[e] += y2[e] - v1[e];
          if (c == 2) div0[e] += z0[e] - v0[e], div1[e] += z1[e] - v1[e];
        }
        float g0[kV], g1[kV];
        if (f) {
          ld_cells<kV>(g0, f + c * cells + r0 + i);
          ld_cells<kV>(g1, f + c * cells + r1 + i);
        } else {
#pragma unroll
          for (int e = 0; e < kV; ++e) g0[e] = g1[e] = 0.f;
        }
        if (A.nu != 0.f) {
          // second differences as sums of first differences
          float ym[kV], q0[kV], q1[kV];
          ld_cells<kV>(ym, uc + ra);
          ld_cells<kV>(q0, uc + rd);
          ld_cells<kV>(q1, uc + rd + n0);
          float w0 = v0[0] - __ldg(uc + r0 + im), w1 = v1[0] - __ldg(uc + r1 + im);
#pragma unroll
          for (int e = 0; e < kV; ++e) {
            const float x0 = v0[e + 1] - v0[e], x1 = v1[e + 1] - v1[e];
            const float dy = v1[e] - v0[e];
            g0[e] = fmaf(A.nu, (x0 - w0) + (dy - (v0[e] - ym[e])) +
                                   ((z0[e] - v0[e]) - (v0[e] - q0[e])), g0[e]);
            g1[e] = fmaf(A.nu, (x1 - w1) + ((y2[e] - v1[e]) - dy) +
                                   ((z1[e] - v1[e]) - (v1[e] - q1[e])), g1[e]);
            w0 = x0;
            w1 = x1;
          }
        }
#pragma unroll
        for (int e = 0; e < kV; ++e) z[L.addr(i + e) + 4 * rp + c] = make_float2(g0[e], g1[e]);
      }
#pragma unroll
      for (int e = 0; e < kV; ++e) z[L.addr(i + e) + 4 * rp + 3] = make_float2(div0[e], div1[e]);
    } else {  // lines past the last pair of the plane
#pragma unroll
      for (int e = 0; e < kV; ++e)
#pragma unroll
        for (int c = 0; c < 4; ++c) z[L.addr(i + e) + 4 * rp + c] = make_float2(0.f, 0.f);
    }
    for (iv += blockDim.x; iv >= nv; iv -= nv) ++rp;
  }
  __syncthreads();
  line_passes<false, N>(A, z);
  // z_k = a_k + i b_k of the two real rows a, b:
  //   2 a_k = z_k + conj z_{n-k},  2 b_k = -i (z_k - conj z_{n-k})
  // (the factor 2 is in inv_n)
  const int nx = n0 / 2 + 1;
  const int lane = threadIdx.x & 31, threads = (int)blockDim.x;
  for (int l = first_line(threadIdx.x >> 5, threads); l < 4 * np; l += threads / 32) {
    float2* o = A.spec + ((int64_t)((l & 3) * n2 + k) * n1 + 2 * (jp0 + (l >> 2))) * A.pitch;
    const float2* zl = z + l;
#pragma unroll 4
    for (int kx = lane; kx < nx; kx += 32) {
      const float2 a = zl[__ldg(A.posx + kx)];
      const float2 b = zl[__ldg(A.posx + (kx ? n0 - kx : 0))];
      o[kx] = make_float2(a.x + b.x, a.y - b.y);
      o[A.pitch + kx] = make_float2(a.y + b.y, b.x - a.x);
    }
  }
}

// One line of n1 places x kTX adjacent modes of one field and plane.
constexpr bool has16(int n, int d) { return n == 0 || make_plan(n, d).rad[0] == 16; }
template <bool kInv, int N>
__global__ void __launch_bounds__(cta_threads<N, 1>(),
                                  has16(N, 1) ? 768 / cta_threads<N, 1>()
                                              : ctas_at_48(cta_threads<N, 1>()))
    k_spec_y(SpecArgs A) {
  chain_wait();
  chain_next();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n1 = N > 0 ? N : A.y.n, n2 = A.z.n;
  const int col = threadIdx.x & (kTX - 1), j0 = threadIdx.x / kTX;
  const int kx = blockIdx.x * kTX + col;
  const int k = kInv ? blockIdx.z : n2 - 1 - blockIdx.z;
  const GlobalCol g{A.spec + (int64_t)(blockIdx.y * n2 + k) * n1 * A.pitch + kx, A.pitch, 0,
                    kx <= A.x.n / 2};
  // one wave of CTAs ahead, where the modes come from memory
  if ((int)blockIdx.z + A.ahead < n2)
    for (int r = threadIdx.x; r < n1; r += blockDim.x)
      prefetch_line(A.spec + ((int64_t)(blockIdx.y * n2 + (kInv ? k + A.ahead : k - A.ahead)) * n1 +
                              r) * A.pitch + blockIdx.x * kTX);
  const SharedCol<kTX> s{reinterpret_cast<float2*>(smem_raw) + col, 0, 0, 0};
  if constexpr (N > 0) {
    constexpr int np = Dim<N, 1>::P.np, step = col_threads(N, Dim<N, 1>::P.rad[0], kTX) / kTX;
    known_pass<N, 1, kInv ? np - 1 : 0, kInv, 1>(j0, A.y.tw, g, s, step);
    __syncthreads();
    known_passes<N, 1, kInv, 1, 1, np - 1>(j0, step, A.y.tw, s);
    known_pass<N, 1, kInv ? 0 : np - 1, kInv, 1>(j0, A.y.tw, s, g, step);
  } else {
    const int np = A.y.np, step = blockDim.x / kTX;
    any_pass<kInv, 1, true>(A.y, kInv ? np - 1 : 0, j0, step, g, s);
    __syncthreads();
    for (int i = 1; i + 1 < np; ++i) {
      any_pass<kInv, 1, true>(A.y, kInv ? np - 1 - i : i, j0, step, s, s);
      __syncthreads();
    }
    any_pass<kInv, 1, true>(A.y, kInv ? 0 : np - 1, j0, step, s, g);
  }
}

// Last forward pass (stride 1, no twiddles) of the four fields, the solve and
// the first inverse pass over the same places, in registers.
template <int R>
__device__ __forceinline__ void solve_pass(const SpecArgs& A, const SharedCol<kTZ>& s, int n2,
                                           int j0, int step, float2 dx, float2 dy, float sxy) {
#pragma unroll 1
  for (int j = j0; j < n2 / R; j += step) {
    float2 v[4][R];
    const int p0 = j * R, par = j & s.en;  // p0 >> sh = j for the even radices
    float2* q0 = s.s + p0 * kTZ;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[c][r] = q0[c * s.field + (r ^ par) * kTZ];
      Dft<R, false>::run(v[c]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 w = __ldg(A.symz + p0 + r);  // (Re D_z, Im D_z, |D_z|^2, 0)
      const float2 dz = make_float2(w.x, w.y);
      const float S = sxy + w.z;
      const float hm = A.inv_n / fmaf(A.nu, S, A.alpha);
      const float2 d0 = make_float2(v[0][r].x * hm, v[0][r].y * hm);
      const float2 d1 = make_float2(v[1][r].x * hm, v[1][r].y * hm);
      const float2 d2 = make_float2(v[2][r].x * hm, v[2][r].y * hm);
      const float2 t = cadd(cadd(cmul(dx, d0), cmul(dy, d1)), cmul(dz, d2));
      const float iS = S > 0.f ? 1.f / S : 0.f;
      const float2 q = make_float2(fmaf(v[3][r].x, A.inv_n, t.x) * iS,
                                   fmaf(v[3][r].y, A.inv_n, t.y) * iS);
      v[0][r] = csub(d0, cmulc(q, dx));
      v[1][r] = csub(d1, cmulc(q, dy));
      v[2][r] = csub(d2, cmulc(q, dz));
      v[3][r] = make_float2(q.x * A.pscale, q.y * A.pscale);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Dft<R, true>::run(v[c]);
#pragma unroll
      for (int r = 0; r < R; ++r) q0[c * s.field + (r ^ par) * kTZ] = v[c][r];
    }
  }
}

template <int N>
__global__ void __launch_bounds__(256, 3) k_spec_solve(SpecArgs A) {
  chain_wait();
  chain_next();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n2 = N > 0 ? N : A.z.n;
  const int col = threadIdx.x & (kTZ - 1), j0 = threadIdx.x / kTZ;
  const int kx = blockIdx.x * kTZ + col;
  const bool on = kx <= A.x.n / 2;
  const int plane = A.y.n * A.pitch;
  const GlobalCol g{A.spec + (int64_t)blockIdx.y * A.pitch + kx, plane, (int64_t)n2 * plane, on};
  SharedCol<kTZ> s{reinterpret_cast<float2*>(smem_raw) + col, n2 * kTZ, A.zsh, A.zen};
  if constexpr (N > 0) {
    s.sh = swap_shift(Dim<N, 2>::P.rad[Dim<N, 2>::P.np - 1]);
    s.en = swap_on(Dim<N, 2>::P.rad[Dim<N, 2>::P.np - 1]);
  }
  const float4 wx = __ldg(A.symx + (on ? kx : 0)), wy = __ldg(A.symy + blockIdx.y);
  const float2 dx = make_float2(wx.x, wx.y), dy = make_float2(wy.x, wy.y);
  const float sxy = wx.z + wy.z;
  if constexpr (N > 0) {
    constexpr int np = Dim<N, 2>::P.np, step = col_threads(N, Dim<N, 2>::P.rad[0], kTZ) / kTZ;
    known_pass<N, 2, 0, false, 4>(j0, A.z.tw, g, s, step);
    __syncthreads();
    known_passes<N, 2, false, 4, 1, np - 1>(j0, step, A.z.tw, s);
    solve_pass<Dim<N, 2>::P.rad[Dim<N, 2>::P.np - 1]>(A, s, n2, j0, step, dx, dy, sxy);
    __syncthreads();
    known_passes<N, 2, true, 4, 1, np - 1>(j0, step, A.z.tw, s);
    known_pass<N, 2, 0, true, 4>(j0, A.z.tw, s, g, step);
  } else {
    const int np = A.z.np, step = blockDim.x / kTZ;
    any_pass<false, 4, true>(A.z, 0, j0, step, g, s);
    __syncthreads();
    for (int i = 1; i + 1 < np; ++i) {
      any_pass<false, 4, true>(A.z, i, j0, step, s, s);
      __syncthreads();
    }
    switch (A.z.rad[np - 1]) {
      case 2: solve_pass<2>(A, s, n2, j0, step, dx, dy, sxy); break;
      case 3: solve_pass<3>(A, s, n2, j0, step, dx, dy, sxy); break;
      case 4: solve_pass<4>(A, s, n2, j0, step, dx, dy, sxy); break;
      case 5: solve_pass<5>(A, s, n2, j0, step, dx, dy, sxy); break;
    }
    __syncthreads();
    for (int i = np - 2; i > 0; --i) {
      any_pass<true, 4, true>(A.z, i, j0, step, s, s);
      __syncthreads();
    }
    any_pass<true, 4, true>(A.z, 0, j0, step, s, g);
  }
}

// Inverse x transform of four row pairs (plane k) of the four fields,
// u_next = u + w and p.  kKeep: the increment w is also left in the rows of
// spec (for the residuals).
template <bool kKeep, int N>
__global__ void __launch_bounds__(cta_threads<N, 0>(), ctas_at_48(cta_threads<N, 0>()))
    k_spec_out(SpecArgs A, const float* u, float* un,
                                                  float* __restrict__ p) {
  chain_wait();
  chain_next();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* z = reinterpret_cast<float2*>(smem_raw);
  const LineSmem<N> L(A, z);
  const int n0 = N > 0 ? N : A.x.n, n1 = A.y.n, n2 = A.z.n;
  const int k = n2 - 1 - blockIdx.y, jp0 = blockIdx.x * 4, np = min(4, n1 / 2 - jp0);
  const int nx = n0 / 2 + 1;
  const int cells = n0 * n1 * n2;
  if (threadIdx.x < 3)
    prefetch_rows(u + threadIdx.x * cells + (k * n1 + 2 * jp0) * n0, sizeof(float) * 2 * np * n0);
  // a warp takes a line, four groups of 32 modes of both rows in flight
  const int lane = threadIdx.x & 31, threads = (int)blockDim.x;
  for (int l = first_line(threadIdx.x >> 5, threads); l < kXL; l += threads / 32) {
    const bool on = l < 4 * np;
    const float2* g =
        A.spec + ((int64_t)((l & 3) * n2 + k) * n1 + 2 * (jp0 + (on ? l >> 2 : 0))) * A.pitch;
    float2* zl = z + l;
    for (int k0 = lane; k0 < nx; k0 += 128) {
      float2 a[4], b[4];
      int pa[4], pb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kx = k0 + 32 * q;
        a[q] = b[q] = make_float2(0.f, 0.f);
        pa[q] = pb[q] = 0;
        if (kx < nx) {
          if (on) {
            a[q] = g[kx];
            b[q] = g[A.pitch + kx];
          }
          pa[q] = __ldg(A.posx + kx);
          pb[q] = __ldg(A.posx + (kx ? n0 - kx : 0));
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kx = k0 + 32 * q;
        if (kx >= nx) break;
        // z_k = a_k + i b_k, z_{n-k} = conj a_k + i conj b_k; real at k = 0, n/2
        if (kx == 0 || 2 * kx == n0) {
          zl[pa[q]] = make_float2(a[q].x, b[q].x);
        } else {
          zl[pa[q]] = make_float2(a[q].x - b[q].y, a[q].y + b[q].x);
          zl[pb[q]] = make_float2(a[q].x + b[q].y, b[q].x - a[q].y);
        }
      }
    }
  }
  __syncthreads();
  line_passes<true, N>(A, z);
  int rp = threadIdx.x / n0, i = threadIdx.x - rp * n0;
  while (rp < np) {
    const int row = (k * n1 + 2 * (jp0 + rp)) * n0 + i;
    const float2* zi = z + L.addr(i) + 4 * rp;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2 w = zi[c];
      const float a = u[c * cells + row] + w.x, b = u[c * cells + row + n0] + w.y;
      un[c * cells + row] = a;
      un[c * cells + row + n0] = b;
      if (kKeep) {
        float* o = reinterpret_cast<float*>(A.spec + ((int64_t)(c * n2 + k) * n1 +
                                                      2 * (jp0 + rp)) * A.pitch);
        o[i] = w.x;
        o[2 * A.pitch + i] = w.y;
      }
    }
    const float2 w = zi[3];
    p[row] = w.x;
    p[row + n0] = w.y;
    for (i += blockDim.x; i >= n0; i -= n0) ++rp;
  }
}

// Squared residuals and right-hand sides of both solves, per CTA in fixed
// order: part[4 b ..] = (Helmholtz residual, its rhs, Poisson residual, rhs).
// u: the velocity before the step; w (rows of spec): the increment.
__global__ void __launch_bounds__(256) k_spec_resid(SpecArgs A, const float* __restrict__ u,
                                                    const float* __restrict__ f,
                                                    const float* __restrict__ p, double a,
                                                    double nu, double dtoh,
                                                    double* __restrict__ part) {
  __shared__ double sh[4][8];
  const int n0 = A.x.n, n1 = A.y.n, n2 = A.z.n, cells = n0 * n1 * n2;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  auto at = [&](int i, int j, int k) { return (k * n1 + j) * n0 + i; };
  // d = w + dt grad p (u* = u + d)
  auto d = [&](int c, int i, int j, int k) {
    const float w = reinterpret_cast<const float*>(
        A.spec + ((int64_t)(c * n2 + k) * n1 + j) * A.pitch)[i];
    const int b = c == 0 ? at(dn(i, n0), j, k) : (c == 1 ? at(i, dn(j, n1), k) : at(i, j, dn(k, n2)));
    return double(w) + dtoh * (double(p[at(i, j, k)]) - double(p[b]));
  };
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cells; t += gridDim.x * blockDim.x) {
    const int i = t % n0, j = (t / n0) % n1, k = t / (n0 * n1);
    const int ip = up(i, n0), im = dn(i, n0), jp = up(j, n1), jm = dn(j, n1), kp = up(k, n2),
              km = dn(k, n2);
    for (int c = 0; c < 3; ++c) {
      const float* uc = u + c * cells;
      const double uu = uc[t];
      const double lu = double(uc[at(ip, j, k)]) + uc[at(im, j, k)] + uc[at(i, jp, k)] +
                        uc[at(i, jm, k)] + uc[at(i, j, kp)] + uc[at(i, j, km)] - 6.0 * uu;
      const double dc = d(c, i, j, k);
      const double ld = d(c, ip, j, k) + d(c, im, j, k) + d(c, i, jp, k) + d(c, i, jm, k) +
                        d(c, i, j, kp) + d(c, i, j, km) - 6.0 * dc;
      const double fc = f ? double(f[c * cells + t]) : 0.0;
      const double rhs = a * uu + fc;
      const double res = fc + nu * lu - (a * dc - nu * ld);
      acc[0] += res * res;
      acc[1] += rhs * rhs;
    }
    const double dv = (double(u[at(ip, j, k)]) - u[t]) +
                      (double(u[cells + at(i, jp, k)]) - u[cells + t]) +
                      (double(u[2 * cells + at(i, j, kp)]) - u[2 * cells + t]) +
                      (d(0, ip, j, k) - d(0, i, j, k)) + (d(1, i, jp, k) - d(1, i, j, k)) +
                      (d(2, i, j, kp) - d(2, i, j, k));
    const double lp = double(p[at(ip, j, k)]) + p[at(im, j, k)] + p[at(i, jp, k)] +
                      p[at(i, jm, k)] + p[at(i, j, kp)] + p[at(i, j, km)] - 6.0 * double(p[t]);
    const double res = dv - dtoh * lp;  // both scaled by h
    acc[2] += res * res;
    acc[3] += dv * dv;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], o);
    if (lane == 0) sh[c][warp] = acc[c];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += sh[threadIdx.x][w];
    part[4 * blockIdx.x + threadIdx.x] = s;
  }
}

// f(std::integral_constant<int, N>): N the length where it has compile-time
// transforms (2^k, 3 2^k and 5 2^k from 32 to 512: the lattices that halve well,
// which users pick), else 0, any length.  Measured at 192^3: 328 us a step
// against 362 us with every length from the arguments; 128^3 115 / 131 us.
template <int N, typename F>
bool if_length(int n, F&& f) {
  if (n != N) return false;
  f(std::integral_constant<int, N>{});
  return true;
}
template <int... N, typename F>
void one_length(std::integer_sequence<int, N...>, int n, F&& f) {
  if (!(if_length<N>(n, f) || ...)) f(std::integral_constant<int, 0>{});
}
template <typename F>
void with_length(int n, F&& f) {
  one_length(std::integer_sequence<int, 32, 40, 48, 64, 80, 96, 128, 160, 192, 256, 320, 384,
                                   512>{}, n, f);
}

size_t z_smem(int n2) { return sizeof(float2) * 4 * kTZ * (size_t)n2; }
constexpr size_t kMaxSmem = 227 * 1024;

bool ok(cudaError_t e) { return e == cudaSuccess; }

}  // namespace

bool spectral_supports(const int n[3]) {
  for (int d = 0; d < 3; ++d)
    if (n[d] % 2 || n[d] > kMaxN || make_plan(n[d], d).np == 0) return false;
  return z_smem(n[2]) <= kMaxSmem;
}

ib_status spectral_create(Spectral* sp, const int n[3], double h, double rho, double mu,
                          double dt, cudaStream_t up) {
  SpecArgs& A = sp->a;
  SpecDim* dims[3] = {&A.x, &A.y, &A.z};
  const double pi = 3.14159265358979323846;
  std::vector<unsigned char> host;
  auto put = [&](const void* src, size_t bytes) {
    const size_t at = (host.size() + 15) / 16 * 16;
    host.resize(at + bytes);
    std::memcpy(host.data() + at, src, bytes);
    return at;
  };
  size_t tw_at[3], sym_at[3], pos_at = 0;
  for (int d = 0; d < 3; ++d) {
    const int N = n[d];
    SpecDim& D = *dims[d];
    const Plan P = make_plan(N, d);
    D.n = N;
    D.np = P.np;
    std::copy(P.rad, P.rad + kSpecMaxPasses, D.rad);
    std::copy(P.q, P.q + kSpecMaxPasses, D.q);
    std::copy(P.tws, P.tws + kSpecMaxPasses, D.tws);
    std::copy(P.magic, P.magic + kSpecMaxPasses, D.magic);
    std::vector<float2> tw(N);
    for (int j = 0; j < N; ++j)
      tw[j] = make_float2((float)std::cos(2 * pi * j / N), (float)-std::sin(2 * pi * j / N));
    // place p of the transformed line holds mode freq[p]
    std::vector<int> freq(N), pos(N);
    for (int p = 0; p < N; ++p) {
      int k = 0, w = 1, r = p;
      for (int i = 0; i < D.np; ++i) {
        k += w * (r / D.q[i]);
        r %= D.q[i];
        w *= D.rad[i];
      }
      freq[p] = k;
      pos[k] = p;
    }
    std::vector<float4> sym(N);
    for (int p = 0; p < N; ++p) {
      const int k = d == 0 ? p : freq[p];  // x modes are stored in order
      const double s = std::sin(pi * k / N), c = std::cos(pi * k / N);
      // D = exp(2 i t) - 1 = 2 i s exp(i t), |D|^2 = 4 s^2
      sym[p] = make_float4((float)(-2 * s * s), (float)(2 * s * c), (float)(4 * s * s), 0.f);
    }
    tw_at[d] = put(tw.data(), sizeof(float2) * N);
    sym_at[d] = put(sym.data(), sizeof(float4) * N);
    if (d == 0) {  // shared-memory address of each mode (LineSmem::addr)
      A.xskew = line_skew(D.q[0]);
      for (int& q : pos) q = q * kXP + q / D.q[0] * A.xskew;
      pos_at = put(pos.data(), sizeof(int) * N);
    }
  }
  A.pitch = (n[0] / 2 + 1 + 3) / 4 * 4;  // rows start on 32-byte sectors
  const size_t spec = (sizeof(float2) * 4 * (size_t)n[2] * n[1] * A.pitch + 255) / 256 * 256;
  if (const ib_status f = injected("modes")) return f;
  if (const cudaError_t e = cudaMalloc((void**)&A.spec, spec + host.size())) {
    A.spec = nullptr;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? IB_ERR_CAPACITY : IB_ERR_CUDA;
  }
  char* const t = reinterpret_cast<char*>(A.spec) + spec;  // the tables behind the modes
  // The tables are on the device when the solver is handed out, whatever stream
  // it is first used on.  A plain copy from pageable memory may return with its
  // last part still on the way, in the order of the legacy stream alone, which
  // non-blocking streams do not wait for; one wait per solver.
  if (!ok(cudaMemcpyAsync(t, host.data(), host.size(), cudaMemcpyHostToDevice, up)) ||
      !ok(cudaStreamSynchronize(up)))
    return IB_ERR_CUDA;
  for (int d = 0; d < 3; ++d) dims[d]->tw = reinterpret_cast<const float2*>(t + tw_at[d]);
  A.symx = reinterpret_cast<const float4*>(t + sym_at[0]);
  A.symy = reinterpret_cast<const float4*>(t + sym_at[1]);
  A.symz = reinterpret_cast<const float4*>(t + sym_at[2]);
  A.posx = reinterpret_cast<const int*>(t + pos_at);
  A.alpha = (float)(rho / dt);
  A.nu = (float)(mu / (h * h));
  A.inv_n = (float)(0.5 / ((double)n[0] * n[1] * n[2]));
  A.pscale = (float)(-h / dt);
  // shared-memory swap of the z lines (even last radices 2 and 4)
  const int last = A.z.rad[A.z.np - 1];
  A.zsh = swap_shift(last);
  A.zen = swap_on(last);
  sp->smem_x = sizeof(float2) * (size_t)(kXP * n[0] + A.x.rad[0] * A.xskew);
  sp->smem_y = sizeof(float2) * kTX * n[1];
  sp->smem_z = z_smem(n[2]);
  sp->threads_x = col_threads(n[0], A.x.rad[0], kXL);
  sp->threads_y = col_threads(n[1], A.y.rad[0], kTX);
  sp->threads_z = col_threads(n[2], A.z.rad[0], kTZ);
  // lines longer than the default 48 KB of shared memory holds
  auto opt = [](size_t smem, auto... k) {
    return smem <= 48 * 1024 ||
           (ok(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem)) && ...);
  };
  // Planes whose CTAs of the y transforms are resident at once: what a CTA asks
  // for ahead belongs to the CTA that takes its place.  Only for modes that L2
  // does not hold (256^3: 106 -> 91 and 113 -> 99 us; 128^3, held, 17.2 -> 17.8).
  int dev = 0, sms = 0, l2 = 0, per_sm = 1;
  if (!ok(cudaGetDevice(&dev)) ||
      !ok(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
      !ok(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev)))
    return IB_ERR_CUDA;
  const bool beyond_l2 = spec > (size_t)l2;
  bool good = true;
  with_length(n[0], [&](auto N) {
    constexpr int L = decltype(N)::value;
    good = good && opt(sp->smem_x, k_spec_rhs<1, L>, k_spec_rhs<2, L>, k_spec_out<false, L>,
                       k_spec_out<true, L>);
  });
  with_length(n[1], [&](auto N) {
    constexpr int L = decltype(N)::value;
    good = good && opt(sp->smem_y, k_spec_y<false, L>, k_spec_y<true, L>) &&
           (!beyond_l2 ||
            ok(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spec_y<true, L>,
                                                             sp->threads_y, sp->smem_y)));
  });
  with_length(n[2], [&](auto N) {
    good = good && opt(sp->smem_z, k_spec_solve<decltype(N)::value>);
  });
  const int plane = (n[0] / 2 + kTX) / kTX * 4;  // CTAs of a plane
  A.ahead = beyond_l2 ? (per_sm * sms + plane - 1) / plane : n[2];
  return good ? IB_OK : IB_ERR_CUDA;
}

void spectral_destroy(Spectral* sp) {
  cudaFree(sp->a.spec);
  sp->a.spec = nullptr;
}

ib_status spectral_step(const Spectral* sp, const float* u, const float* f, float* un, float* p,
                        bool keep, cudaStream_t s) {
  const SpecArgs& A = sp->a;
  const int n1 = A.y.n, n2 = A.z.n, nx = A.x.n / 2 + 1;
  const dim3 gx((n1 / 2 + 3) / 4, n2);
  const int ty = (nx + kTX - 1) / kTX, tz = (nx + kTZ - 1) / kTZ;
  // cell pairs by 8-byte loads where the arrays' bases allow (rows are even)
  const bool pairs = ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(f)) & 7) == 0;
  const dim3 gy(ty, 4, n2), gz(tz, n1);
  with_length(A.x.n, [&](auto N) {
    constexpr int L = decltype(N)::value;
    chain_launch(pairs ? k_spec_rhs<2, L> : k_spec_rhs<1, L>, gx, sp->threads_x, sp->smem_x, s, A,
                 u, f);
  });
  with_length(A.y.n, [&](auto N) {
    chain_launch(k_spec_y<false, decltype(N)::value>, gy, sp->threads_y, sp->smem_y, s, A);
  });
  with_length(A.z.n, [&](auto N) {
    chain_launch(k_spec_solve<decltype(N)::value>, gz, sp->threads_z, sp->smem_z, s, A);
  });
  with_length(A.y.n, [&](auto N) {
    chain_launch(k_spec_y<true, decltype(N)::value>, gy, sp->threads_y, sp->smem_y, s, A);
  });
  with_length(A.x.n, [&](auto N) {
    constexpr int L = decltype(N)::value;
    chain_launch(keep ? k_spec_out<true, L> : k_spec_out<false, L>, gx, sp->threads_x, sp->smem_x,
                 s, A, u, un, p);
  });
  return ok(cudaGetLastError()) ? IB_OK : IB_ERR_CUDA;
}

void launch_spectral_resid(const Spectral* sp, const float* u, const float* f, const float* p,
                           double a, double nu, double dtoh, double* part, int ctas,
                           cudaStream_t s) {
  k_spec_resid<<<ctas, 256, 0, s>>>(sp->a, u, f, p, a, nu, dtoh, part);
}

}  // namespace ibfe
