// chem.cu -- per-cell kernels around the trace: the hydrogen-only ionisation
// update (Eq. "dndt", Step 6 of Sec. 3.1), the absorber-density refresh
// n_HI = n_H x_HI, and conversion of the rates for the caller.
#include <cuda_runtime.h>
#include <stdint.h>

#include "f2.cuh"
#include "rt_internal.cuh"

namespace rtg {

// One substep, FP64 path, from the closed form below: for cells outside the
// range of chem_cell_fp64's corrections.
__device__ __noinline__ double2 chem_substep_fp64(double x, double z, double a, double b, double hk) {
  const double D = __dadd_rn(__dmul_rn(b, b), __dmul_rn(__dmul_rn(4.0, a), __dadd_rn(z, hk)));
  const double sq = __dsqrt_rn(D);
  const double xn = __ddiv_rn(__dmul_rn(2.0, __dadd_rn(a, x)), __dadd_rn(__dadd_rn(__dmul_rn(2.0, a), b), sq));
  const double zn = __ddiv_rn(__dmul_rn(2.0, __dadd_rn(z, hk)), __dadd_rn(b, sq));
  return xn <= zn ? make_double2(xn, __dsub_rn(1.0, xn)) : make_double2(__dsub_rn(1.0, zn), zn);
}

// One cell, FP64 path.  The FP64 pipe bounds this kernel, and the closed form
// of a substep (below) takes two quotients and a square root on it.  Instead
// the fraction that is the smaller one after the substep is guessed in FP32
// and corrected twice by Newton's method, the residual of the implicit
// equation in FP64 and the step in FP32 (the derivative at the root is
// -sqrt(D) or sqrt(D)): the first leaves ~1e-13, the second the rounding of
// its residual,
//   x-form: (a (1 - x')^2 + x) - b x',   z-form: (a z' + b) z' - (z + hk),
// whose terms are the size of the result's own.  (The guess decides which
// fraction that is: where a substep takes a cell past 1/2, the other one as
// one minus the corrected one would only be good to 2^-53 of 1.)  8 to 10 FP64
// operations a substep instead of ~45: 128^3 cells, 10 substeps, 1410 -> 440
// us.  Against the recursion in 113 bits the mean error over 10 substeps is
// 1.5e-16 in x_HI and 1.7e-16 in x_HII, the largest 2.1e-15 and 3.5e-15; the
// closed form's 1.8e-16, 1.9e-16, 3.6e-15 and 3.7e-15.  The largest of one
// substep: 6.2e-16 and 4.7e-16, the closed form's 5.8e-16 and 5.1e-16.
__device__ __forceinline__ void chem_cell_fp64(double& x, double& z, double n, double kc, double h, int nsub,
                                               double alpha) {
  const double a = __dmul_rn(__dmul_rn(h, alpha), n);
  const double hk = __dmul_rn(h, kc);
  const double b = __dadd_rn(1.0, hk);
  const bool fits = a < 1e6 && hk >= 0.0 && hk < 1e18;
  const double tab = __dadd_rn(__dmul_rn(2.0, a), b);
  const float af = f32_chop(a), bf = f32_chop(b), hkf = f32_chop(hk);
  int i = 0;
  // fractions further from 1 in sum than rounding takes them (a caller may give
  // both): a form that holds one of them only would drop what the other says.
  // (Tested as integers: with three FP64 operations instead of one 192^3 cells
  // took 50 us longer.)
  const double sum = __dadd_rn(x, z);
  const unsigned sh = (unsigned)__double2hiint(sum), sl = (unsigned)__double2loint(sum);
  if (!((sh == 0x3FF00000u && sl <= 1u) || (sh == 0x3FEFFFFFu && sl >= 0xFFFFFFFEu))) {
    const double2 v = chem_substep_fp64(x, z, a, b, hk);
    x = v.x;
    z = v.y;
    if (x != x) return;  // not a number: so it stays
    i = 1;
  }
  for (; i < nsub; ++i) {
    const float xf = f32_chop(x), wf = f32_chop(z) + hkf;
    const float D = fmaf(4.0f * af, wf, bf * bf);
    const float rs = rsqrtf(D), sq = D * rs;
    const float gx = __fdividef(2.0f * (af + xf), 2.0f * af + bf + sq);
    const bool xform = gx < 0.5f;
    const float g0 = xform ? gx : __fdividef(2.0f * wf, bf + sq);
    // the corrections are FP32 numbers: the second one, 1e-13 of the result and
    // needed to 1e-3, stays above their range's end from 1e-22 on
    if (!fits || !(g0 >= 1e-22f)) {
      const double2 v = chem_substep_fp64(x, z, a, b, hk);
      x = v.x;
      z = v.y;
      continue;
    }
    double v = f64_wide(g0);
    if (xform) {
      v = __dadd_rn(v, f64_wide(rs * f32_chop(__fma_rn(__fma_rn(a, v, -tab), v, __dadd_rn(a, x)))));
      const double u = __dsub_rn(1.0, v);
      v = __dadd_rn(v, f64_wide(rs * f32_chop(__fma_rn(-b, v, __fma_rn(__dmul_rn(a, u), u, x)))));
      x = v;
      z = __dsub_rn(1.0, v);
    } else {
      const double c = -__dadd_rn(z, hk);
      v = __dsub_rn(v, f64_wide(rs * f32_chop(__fma_rn(__fma_rn(a, v, b), v, c))));
      v = __dsub_rn(v, f64_wide(rs * f32_chop(__fma_rn(__fma_rn(a, v, b), v, c))));
      z = v;
      x = __dsub_rn(1.0, v);
    }
  }
}

// x == 1 and z == 0 (either sign), compared as bit patterns
__device__ __forceinline__ bool is_neutral(double x, double z) {
  return __double_as_longlong(x) == 0x3FF0000000000000LL && (__double_as_longlong(z) << 1) == 0;
}

// One cell, FP32-mixed path: FP32 solution + one double-float Newton
// correction per substep (see chem_mixed_kernel).  x, z and n arrive and
// leave in FP64 (converted through their bit fields, off the FP64 pipe); in
// between, only the smaller of the two fractions is carried, as a double-float
// pair s.  ha and h2 are h alpha_B and h as pairs.  Returns
// n_HI = n_H x_HI as a pair.
__device__ __forceinline__ F2 chem_cell_mixed(double& x, double& z, double n, float kc, F2 ha, F2 h2, int nsub) {
  const F2 n2 = f2_from_double_bits(n);
  const F2 a = f2_mul(ha, n2);
  const F2 hk = f2_mul_f(h2, kc);
  const F2 one = {1.0f, 0.0f};
  const F2 b = f2_add(one, hk);
  const F2 two_a_b = f2_add(F2{2.0f * a.hi, 2.0f * a.lo}, b);
  const float a2 = 2.0f * a.hi, a4 = 4.0f * a.hi, bb = b.hi * b.hi;
  const F2 x0 = f2_from_double_bits(x), z0 = f2_from_double_bits(z);
  bool sx = x0.hi < 0.5f;  // s holds x_HI (else x_HII)
  F2 s = sx ? x0 : z0;
  float w0 = z0.hi + hk.hi;  // z + hk of the first substep
  // the residual (a v + B) v + sg (s + C) of the form that s is in: x-form
  // B = -(2a + b), C = a, sg = 1; z-form B = b, C = hk, sg = -1
  F2 B = sx ? F2{-two_a_b.hi, -two_a_b.lo} : b;
  F2 C = sx ? a : hk;
  float sg = sx ? 1.0f : -1.0f;
  for (int i = 0; i < nsub; ++i) {
    F2 c = two_sum(s.hi, C.hi);
    c = fast_two_sum(c.hi, __fadd_rn(c.lo, __fadd_rn(s.lo, C.lo)));
    // the FP32 guess needs only ~1e-7: approximate root and quotient (D >= 1,
    // the denominator >= 2)
    const float wf = i == 0 ? w0 : (sx ? (1.0f - s.hi) + hk.hi : c.hi);
    const float D = fmaf(a4, wf, bb);
    const float v = 2.0f * c.hi * rcp_approx(fmaf(D, rsqrt_approx(D), fabsf(B.hi)));
    const float ph = __fmul_rn(a.hi, v);
    const float pl = fmaf(a.lo, v, fmaf(a.hi, v, -ph));
    F2 q = two_sum(B.hi, ph);
    q = fast_two_sum(q.hi, __fadd_rn(q.lo, __fadd_rn(pl, B.lo)));
    const float rh = __fmul_rn(q.hi, v);
    const F2 r = fast_two_sum(rh, fmaf(q.lo, v, fmaf(q.hi, v, -rh)));
    const float f = __fadd_rn(fmaf(sg, c.hi, r.hi), fmaf(sg, c.lo, r.lo));  // the high parts cancel exactly
    // Newton's step with the second-order term, the quotient to FP32 rounding
    const float fp = fmaf(a2, v, B.hi);
    const float rf = rcp_approx(fp);
    const float q0 = __fmul_rn(f, rf);
    float d = -fmaf(fmaf(-q0, fp, f), rf, q0);
    d = fmaf(-(a.hi * d) * d, rf, d);
    s = fast_two_sum(v, d);
    if (sx ? s.hi >= 0.5f : s.hi > 0.5f) {  // to the other form: its fraction is the smaller now
      s = f2_sub(one, s);
      sx = !sx;
      B = sx ? F2{-two_a_b.hi, -two_a_b.lo} : b;
      C = sx ? a : hk;
      sg = -sg;
    }
  }
  const F2 xp = sx ? s : f2_sub(one, s);
  const F2 zp = sx ? f2_sub(one, s) : s;
  x = f2_to_double_bits(xp);
  z = f2_to_double_bits(zp);
  return f2_mul(n2, xp);
}

// Backward Euler on dx/dt = alpha_B n_H (1 - x)^2 - k x, x = x_HI,
// z = x_HII, over nsub substeps h with k frozen.  With a = h alpha_B n_H and
// b = 1 + h k the implicit step solves a x'^2 - (2a + b) x' + (a + x) = 0;
// its physical root, written without cancellation, is
//   x' = 2(a + x) / (2a + b + sqrt(D)),  z' = 2(z + hk) / (b + sqrt(D)),
//   D = b^2 + 4a(z + hk),
// and the smaller of x', z' is kept with the other as its complement, so both
// fractions keep their relative accuracy as either tends to 0.
template <typename KT, typename NT>
__global__ void chem_kernel(long long ncell, const double* __restrict__ nH, double* __restrict__ xHI,
                            double* __restrict__ xHII, const KT* __restrict__ K, NT* __restrict__ nhi,
                            double h, int nsub, double alpha) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    double x = xHI[c], z = xHII[c];
    const KT kc = K[c];
    // no radiation and fully neutral: every substep returns (1, 0) exactly
    if (kc == (KT)0 && z == 0.0 && x == 1.0) continue;
    const double n = nH[c];
    chem_cell_fp64(x, z, n, (double)kc, h, nsub, alpha);
    xHI[c] = x;
    xHII[c] = z;
    nhi[c] = (NT)__dmul_rn(n, x);
  }
}

// Bound by its issue slots.  The two forms share one sequence of ~60
// instructions a substep (their operands change where a cell changes form),
// the residual's pairs are only renormalised where that shows in the result,
// and the Newton step's quotient is an approximate reciprocal with one
// residual: 128^3 cells, 10 substeps, the whole call 102 -> 70 us.  Over 10
// substeps the error against 113 bits is 4.2e-13 at most and 6.0e-15 on average
// in x_HI, 5.1e-13 and 4.9e-15 in x_HII (4.2e-13, 6.0e-15, 1.5e-12 and 4.9e-15
// before).  (A cell that passes 1/2 in one of the last two substeps keeps the
// fraction that has become the smaller one to ~1e-14 of 1, not of itself.)
//
// Same backward-Euler step for the FP32-mixed path, solved by FP32 + one
// Newton correction: the smaller fraction is first obtained in FP32 from its
// cancellation-free formula, then corrected once with the residual of the
// implicit equation evaluated in double-float arithmetic,
//   x-form: g(x') = a x'^2 - (2a + b) x' + (a + x),  g' = 2a x' - (2a + b),
//   z-form: f(z') = a z'^2 + b z' - (z + hk),         f' = 2a z' + b.
// From a ~1e-7 relative guess one Newton step leaves ~1e-14 (the residual's
// double-float rounding, ~2^-48 of its largest term), so the carried state
// stays within ~1e-13 of the FP64 recursion while the substeps run on the
// FP32 pipe.  FP64 arithmetic is left only in one addition per stored
// fraction: the state's conversions to and from pairs move bit fields
// (f2.cuh), since the FP64 pipe, a small fraction of the FP32 one, otherwise
// bounds the kernel.
__global__ void chem_mixed_kernel(long long ncell, const double* __restrict__ nH, double* __restrict__ xHI,
                                  double* __restrict__ xHII, const float2* __restrict__ K,
                                  float2* __restrict__ nhi, float4 hh, int nsub) {
  const F2 ha = {hh.x, hh.y}, h2 = {hh.z, hh.w};
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    double x = xHI[c], z = xHII[c];
    const float kc = K[c].x;
    if (kc == 0.0f && is_neutral(x, z)) continue;
    const F2 nx = chem_cell_mixed(x, z, nH[c], kc, ha, h2, nsub);
    xHI[c] = x;
    xHII[c] = z;
    nhi[c] = make_float2(nx.hi, nx.lo);
  }
}

// Range tests on the bit patterns (FP64 comparisons run on the FP64 pipe and
// bound the kernels that make them; with these tests a 256^3 check takes 24
// instead of 69 us, its commit 118 instead of 162): a finite
// number >= 0, a number in [0, 1] (either zero included).
__device__ __forceinline__ bool good_density(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return u < 0x7FF0000000000000ULL || u == 0x8000000000000000ULL;
}
__device__ __forceinline__ bool good_fraction(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return u <= 0x3FF0000000000000ULL || u == 0x8000000000000000ULL;
}

template <typename NT>
__global__ void refresh_nhi_kernel(long long ncell, const double* __restrict__ nH,
                                   const double* __restrict__ xHI, NT* __restrict__ nhi) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x)
    nhi[c] = (NT)__dmul_rn(nH[c], xHI[c]);
}

// FP32-mixed grids keep n_HI as a pair: FP32 rounding and remainder of the
// FP64 product.
__global__ void refresh_nhi_pair_kernel(long long ncell, const double* __restrict__ nH,
                                        const double* __restrict__ xHI, float2* __restrict__ nhi) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const F2 v = f2_from_double_bits(__dmul_rn(nH[c], xHI[c]));
    nhi[c] = make_float2(v.hi, v.lo);
  }
}

// FP32 pairs (rounded value, remainder) of an FP64 absorber density.
__global__ void pair_kernel(long long ncell, const double* __restrict__ src, float2* __restrict__ dst) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const F2 v = f2_from_double_bits(src[c]);
    dst[c] = make_float2(v.hi, v.lo);
  }
}

// First cell whose density is negative, NaN or infinite (atomicMin into bad).
__global__ void check_density_kernel(long long n, const double* __restrict__ a, unsigned long long* __restrict__ bad) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const double v = a[c];
    if (!good_density(v)) atomicMin(bad, (unsigned long long)c);
  }
}

template <typename ST>
__global__ void convert_kernel(long long n, const ST* __restrict__ src, double* __restrict__ dst) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    dst[c] = (double)src[c];
}

// Gamma of an FP32-mixed grid, eV/s, in erg/s as FP32: the product with scale
// as an FP32 pair, rounded (the FP64 pipe is a small fraction of the FP32 one).
// Small results (an optically thick cell's) would lose the product's low part
// below the FP32 range and are formed 2^64 times larger; results below the
// FP32 normal range, infinities and values that are not numbers go through
// FP64, out of line so that its instructions are not predicated into every
// cell.
__device__ __noinline__ float scale64(float v, double scale) { return (float)((double)v * scale); }
__device__ __forceinline__ float scale32(float v, double scale, float sh, float sl) {
  float p = __fmul_rn(v, sh), up = 1.0f;
  if (!(fabsf(p) >= 1e-30f && fabsf(p) <= 3e38f)) {
    if (v == 0.0f) return 0.0f;
    if (!(fabsf(p) >= 2.4e-38f && fabsf(p) <= 3e38f) || sh < 1e-20f) return scale64(v, scale);
    v *= 18446744073709551616.0f;  // 2^64
    p = __fmul_rn(v, sh);
    up = 5.4210108624275222e-20f;  // 2^-64
  }
  return __fmul_rn(__fadd_rn(p, fmaf(v, sl, fmaf(v, sh, -p))), up);
}
// k_ph, Gamma (times scale) and x_HI for the caller, each where its output is
// given.  MIXED: kg holds (k_ph, Gamma) pairs, else K and G are FP64 arrays.
template <bool MIXED, typename DT>
__global__ void read_rates_kernel(long long n, const void* __restrict__ K, const double* __restrict__ G,
                                  const double* __restrict__ x, DT* __restrict__ ok, DT* __restrict__ og,
                                  DT* __restrict__ ox, double scale) {
  const float sh = (float)scale, sl = (float)(scale - (double)sh);
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    if (MIXED) {
      if (ok || og) {
        const float2 v = ((const float2*)K)[c];
        if (ok) ok[c] = (DT)v.x;
        if (og) og[c] = sizeof(DT) == 4 ? (DT)scale32(v.y, scale, sh, sl) : (DT)((double)v.y * scale);
      }
    } else {
      if (ok) ok[c] = (DT)((const double*)K)[c];
      if (og) og[c] = (DT)(scale == 1.0 ? G[c] : G[c] * scale);
    }
    if (ox) ox[c] = (DT)x[c];
  }
}
// The FP32 outputs of an FP32-mixed grid four cells at a time (16-byte
// accesses), for 16-byte aligned outputs; the last n % 4 cells by block 0.
// Bound by memory: 28 bytes a cell, 71 us for 256^3 (6.6 TB/s).
// One cell a thread with FP64 conversions and products took 140 us, the FP64
// pipe's time.
__global__ void read_rates4_kernel(long long n, const float2* __restrict__ kg, const double* __restrict__ x,
                                   float* __restrict__ ok, float* __restrict__ og, float* __restrict__ ox,
                                   double scale) {
  const float sh = (float)scale, sl = (float)(scale - (double)sh);
  const long long n4 = n / 4;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n4; i += (long long)gridDim.x * blockDim.x) {
    if (ok || og) {
      const float4 a = ((const float4*)kg)[2 * i], b = ((const float4*)kg)[2 * i + 1];
      if (ok) ((float4*)ok)[i] = make_float4(a.x, a.z, b.x, b.z);
      if (og)
        ((float4*)og)[i] = make_float4(scale32(a.y, scale, sh, sl), scale32(a.w, scale, sh, sl),
                                       scale32(b.y, scale, sh, sl), scale32(b.w, scale, sh, sl));
    }
    if (ox) {
      const double2 u = ((const double2*)x)[2 * i], v = ((const double2*)x)[2 * i + 1];
      ((float4*)ox)[i] = make_float4(f2_from_double_bits(u.x).hi, f2_from_double_bits(u.y).hi,
                                     f2_from_double_bits(v.x).hi, f2_from_double_bits(v.y).hi);
    }
  }
  const long long c = 4 * n4 + threadIdx.x;
  if (blockIdx.x == 0 && c < n) {
    if (ok) ok[c] = kg[c].x;
    if (og) og[c] = scale32(kg[c].y, scale, sh, sl);
    if (ox) ox[c] = f2_from_double_bits(x[c]).hi;
  }
}

// The caller's k_ph and Gamma (times scale), each where it is given, into an
// FP32-mixed grid.
template <typename ST>
__global__ void write_rates_kernel(long long n, const ST* __restrict__ k, const ST* __restrict__ g,
                                   float2* __restrict__ kg, double scale) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    if (k && g) kg[c] = make_float2((float)k[c], (float)((double)g[c] * scale));
    else if (k) kg[c].x = (float)k[c];
    else kg[c].y = (float)((double)g[c] * scale);
  }
}

__global__ void complement_kernel(long long n, const double* __restrict__ x, double* __restrict__ out) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    out[c] = __dsub_rn(1.0, x[c]);
}

// Range check of a gas state: bad[0] = first cell whose n_H is negative, NaN
// or infinite (nH may be NULL), bad[1] = first cell whose x_HI lies outside
// [0, 1] or is NaN; entries stay at ~0 when every cell passes.
__global__ void check_state_kernel(long long n, const double* __restrict__ nH, const double* __restrict__ x,
                                   unsigned long long* __restrict__ bad) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    if (nH) {
      const double v = nH[c];
      if (!good_density(v)) atomicMin(&bad[0], (unsigned long long)c);
    }
    const double xv = x[c];
    if (!good_fraction(xv)) atomicMin(&bad[1], (unsigned long long)c);
  }
}

// The same check two cells at a time (16-byte loads, twice the bytes in
// flight per thread), for 16-byte aligned arrays of an even length.
__global__ void check_state2_kernel(long long n2, const double2* __restrict__ nH, const double2* __restrict__ x,
                                    unsigned long long* __restrict__ bad) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n2; i += (long long)gridDim.x * blockDim.x) {
    if (nH) {
      const double2 v = nH[i];
      if (!good_density(v.x)) atomicMin(&bad[0], (unsigned long long)(2 * i));
      if (!good_density(v.y)) atomicMin(&bad[0], (unsigned long long)(2 * i + 1));
    }
    const double2 xv = x[i];
    if (!good_fraction(xv.x)) atomicMin(&bad[1], (unsigned long long)(2 * i));
    if (!good_fraction(xv.y)) atomicMin(&bad[1], (unsigned long long)(2 * i + 1));
  }
}

// Commit of a gas state uploaded without waiting (rt_set_state_async), run
// after check_state_kernel has left the first failing cells in
// ctl[CTL_CHECK_N] and ctl[CTL_CHECK_X] (~0 = none).  When every cell passed,
// the staged arrays replace the grid's -- n_H only when sn is given, x_HII
// from sz or as 1 - x_HI -- and the absorber density n_HI = n_H x_HI is
// refreshed (FP64, or the FP32 pair on the mixed path).  Otherwise nothing
// changes and the rejection is latched in ctl[CTL_SET_ERR] (the first one
// keeps its failing cells), where the next trace and rt_synchronize find it.
// The block that finishes last (CTL_COMMIT_DONE) sets the check words back
// to ~0 for the next upload, after every block has read them.  With `verdict`
// (rt_set_state, whose caller waits) the outcome goes there instead.
__device__ __forceinline__ bool commit_verdict(unsigned long long* ctl, unsigned long long* verdict) {
  const unsigned long long bn = ctl[CTL_CHECK_N], bx = ctl[CTL_CHECK_X];
  if (verdict) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      verdict[0] = bn;
      verdict[1] = bx;
    }
    return bn == ~0ULL && bx == ~0ULL;
  }
  if (bn == ~0ULL && bx == ~0ULL) return true;
  if (blockIdx.x == 0 && threadIdx.x == 0 &&
      atomicCAS(&ctl[CTL_SET_ERR], 0ULL, (unsigned long long)RT_ERR_INVALID_ARG) == 0ULL) {
    ctl[CTL_SET_BADN] = bn;
    ctl[CTL_SET_BADX] = bx;
  }
  return false;
}
__device__ __forceinline__ void commit_finish(unsigned long long* ctl) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&ctl[CTL_COMMIT_DONE], 1ULL) == (unsigned long long)gridDim.x - 1ULL;
    if (last) {
      __threadfence();
      ctl[CTL_CHECK_N] = ~0ULL;
      ctl[CTL_CHECK_X] = ~0ULL;
      ctl[CTL_COMMIT_DONE] = 0ULL;
    }
  }
}
template <bool PAIR>
__global__ void commit_state_kernel(long long n, unsigned long long* ctl, unsigned long long* verdict,
                                    const double* __restrict__ sn, const double* __restrict__ sx, const double* __restrict__ sz,
                                    double* __restrict__ nH, double* __restrict__ xHI, double* __restrict__ xHII,
                                    void* __restrict__ nhi) {
  const bool ok = commit_verdict(ctl, verdict);
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; ok && c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const double h = sn ? sn[c] : nH[c];
    if (sn) nH[c] = h;
    const double x = sx[c];
    xHI[c] = x;
    xHII[c] = sz ? sz[c] : __dsub_rn(1.0, x);
    const double v = __dmul_rn(h, x);
    if (PAIR) {
      const F2 p = f2_from_double_bits(v);
      ((float2*)nhi)[c] = make_float2(p.hi, p.lo);
    } else {
      ((double*)nhi)[c] = v;
    }
  }
  commit_finish(ctl);
}

// The same commit two cells at a time (16-byte accesses), for 16-byte
// aligned arrays of an even length.
template <bool PAIR>
__global__ void commit_state2_kernel(long long n2, unsigned long long* ctl, unsigned long long* verdict,
                                     const double2* __restrict__ sn, const double2* __restrict__ sx, const double2* __restrict__ sz,
                                     double2* __restrict__ nH, double2* __restrict__ xHI, double2* __restrict__ xHII,
                                     void* __restrict__ nhi) {
  const bool ok = commit_verdict(ctl, verdict);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; ok && i < n2;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 h = sn ? sn[i] : nH[i];
    if (sn) nH[i] = h;
    const double2 x = sx[i];
    xHI[i] = x;
    xHII[i] = sz ? sz[i] : make_double2(__dsub_rn(1.0, x.x), __dsub_rn(1.0, x.y));
    const double v0 = __dmul_rn(h.x, x.x), v1 = __dmul_rn(h.y, x.y);
    if (PAIR) {
      const F2 p0 = f2_from_double_bits(v0), p1 = f2_from_double_bits(v1);
      ((float4*)nhi)[i] = make_float4(p0.hi, p0.lo, p1.hi, p1.lo);
    } else {
      ((double2*)nhi)[i] = make_double2(v0, v1);
    }
  }
  commit_finish(ctl);
}

// Commit of a state uploaded straight into the grid's alternate buffers
// (rt_set_state_async from host memory without n_H; the host has already
// made x and z the grid's arrays).  Every block checks its cells' x_HI and
// writes their n_HI = n_H x_HI (and x_HII = 1 - x_HI when none was uploaded)
// as if the state passed; the block that finishes last (CTL_COMMIT_DONE)
// takes the verdict.  A rejected state is undone by that block -- the
// previous state copied into x and z and n_HI recomputed from it, so the
// grid ends as it was -- and latched in ctl[CTL_SET_ERR].  Either way it
// points the grid's device descriptor at x and z and sets the check words
// back to ~0.
template <bool PAIR>
__global__ void check_refresh_kernel(long long n, unsigned long long* __restrict__ ctl, const double* __restrict__ nH,
                                     double* __restrict__ x, double* __restrict__ z, int z_given,
                                     const double* __restrict__ x_old, const double* __restrict__ z_old,
                                     void* __restrict__ nhi, InstDev* __restrict__ inst) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    const double xv = x[c];
    if (!good_fraction(xv)) atomicMin(&ctl[CTL_CHECK_X], (unsigned long long)c);
    if (!z_given) z[c] = __dsub_rn(1.0, xv);
    const double v = __dmul_rn(nH[c], xv);
    if (PAIR) {
      const F2 p = f2_from_double_bits(v);
      ((float2*)nhi)[c] = make_float2(p.hi, p.lo);
    } else {
      ((double*)nhi)[c] = v;
    }
  }
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&ctl[CTL_COMMIT_DONE], 1ULL) == (unsigned long long)gridDim.x - 1ULL;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const unsigned long long bx = ctl[CTL_CHECK_X];
  if (bx != ~0ULL) {
    if (threadIdx.x == 0 && atomicCAS(&ctl[CTL_SET_ERR], 0ULL, (unsigned long long)RT_ERR_INVALID_ARG) == 0ULL) {
      ctl[CTL_SET_BADN] = ~0ULL;
      ctl[CTL_SET_BADX] = bx;
    }
    for (long long c = threadIdx.x; c < n; c += blockDim.x) {
      const double xv = x_old[c];
      x[c] = xv;
      z[c] = z_old[c];
      const double v = __dmul_rn(nH[c], xv);
      if (PAIR) {
        const F2 p = f2_from_double_bits(v);
        ((float2*)nhi)[c] = make_float2(p.hi, p.lo);
      } else {
        ((double*)nhi)[c] = v;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    inst->xHI = x;
    inst->xHII = z;
    ctl[CTL_CHECK_N] = ~0ULL;
    ctl[CTL_CHECK_X] = ~0ULL;
    ctl[CTL_COMMIT_DONE] = 0ULL;
  }
}

// Adaptive RT timestep (Sec. 3.4), step 1, Eq. "dtelec": per cell
// eps / |k_ph + n_e alpha_B| (C_H = 0, n_e = n_H (1 - x_HI)) where the cell's
// optical depth sdx n_HI exceeds tau_front, else dt_max; never above dt_max.
// The value is FP32 (a timestep needs no more), in units of dt_max when
// dt_max is finite (so cells outside the front hold exactly 1).  The front
// test is the FP64 one (a cell's side of the threshold must not depend on
// rounding), taken in FP32 where that proves it.
struct StepArgs {
  double sdx, tau_front;
  float sdx32;         // 0 where FP32 cannot hold it or its products
  float hi32, lo32;    // above hi32 in FP32 proves a front cell, below lo32 proves none (inf, -1: never)
  float eps, alpha, dt_max, unit;
  float dt_max_units;  // dt_max / unit
};
// (out of line, or its FP64 instructions would be predicated into every cell)
__device__ __noinline__ bool front_fp64(double nh, double x, double sdx, double tau_front) {
  return sdx * nh * x > tau_front;
}
__device__ __forceinline__ float cell_timestep(double nh64, double x64, float k, const StepArgs& p) {
  const float nh = f2_from_double_bits(nh64).hi, x = f2_from_double_bits(x64).hi;
  const float rate = fabsf(k + nh * (1.0f - x) * p.alpha);
  // within 2^-21 of sdx n_HI where that comes near tau_front: sdx and sdx n_H
  // are below 1e25 and tau_front above 1e-12, so n_H and x are normal there
  // (beyond, not a number: neither side is proven)
  const float t1 = p.sdx32 * nh;
  const float t = t1 < 1e25f ? t1 * x : __int_as_float(0x7fffffff);
  bool front = t > p.hi32;
  if (!front && !(t < p.lo32)) front = front_fp64(nh64, x64, p.sdx, p.tau_front);
  float dt = p.dt_max;
  if (front && rate > 0.0f) {
    dt = fminf(p.dt_max, p.eps / rate);
    if (dt != p.dt_max) return dt / p.unit;
  }
  return p.dt_max_units;
}

// A block's minimum into the grid's: atomicMin on the bit patterns, which order
// like the positive floats; the block that finishes last moves the minimum to
// out[1] and resets the running one.
__device__ __forceinline__ void timestep_finish(float best, unsigned int* out, unsigned long long* done) {
  for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) atomicMin(&out[0], __float_as_uint(best));
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(done, 1ULL) == (unsigned long long)gridDim.x - 1ULL) {
      __threadfence();
      out[1] = atomicExch(&out[0], 0x7f800000u);
      *done = 0ULL;
    }
  }
}

// Steps 1-3 in one pass over tiles: the per-cell timestep of a tile and its
// halo in shared memory, the 3^3 Gaussian (exp(-|d|^2/2), renormalised over
// neighbours inside the grid), and its minimum over the grid.
// Bound by its issue slots (the per-cell timestep of 1.7 cells a cell, mostly).
// The weights are products over the axes, so a plane's sum is three sums of
// rows and passes on to the planes beside it; the cells outside hold 0 and the
// norm is the same product of sums over ones, so a uniform field comes back
// unchanged to the bit.  128^3, per call: 255 us with the field in a scratch
// array and the filter in a second kernel, 68 us with 27 tested neighbours a
// cell and the FP64 front test in line, now 40 us (256^3: 290 -> 199).
constexpr int kTileX = 32, kTileY = 8, kTileZ = 8;
template <typename KT>
__global__ void __launch_bounds__(256) timestep_kernel(int nx, int ny, int nz, const double* __restrict__ nH,
                                                       const double* __restrict__ xHI, const KT* __restrict__ K,
                                                       int kstride, StepArgs p, unsigned int* __restrict__ out,
                                                       unsigned long long* __restrict__ done) {
  __shared__ float tile[kTileZ + 2][kTileY + 2][kTileX + 2];
  const float w = 0.60653066f;  // e^-1/2
  const int tx = (nx + kTileX - 1) / kTileX, ty = (ny + kTileY - 1) / kTileY, tz = (nz + kTileZ - 1) / kTileZ;
  const long long tiles = (long long)tx * ty * tz;
  float best = __int_as_float(0x7f800000);
  for (long long b = blockIdx.x; b < tiles; b += gridDim.x) {
    const int x0 = (int)(b % tx) * kTileX, y0 = (int)((b / tx) % ty) * kTileY, z0 = (int)(b / ((long long)tx * ty)) * kTileZ;
    __syncthreads();
    for (int t = threadIdx.x; t < (kTileZ + 2) * (kTileY + 2) * (kTileX + 2); t += 256) {
      const int i = t % (kTileX + 2), j = (t / (kTileX + 2)) % (kTileY + 2), k = t / ((kTileX + 2) * (kTileY + 2));
      const int x = x0 + i - 1, y = y0 + j - 1, z = z0 + k - 1;
      float v = 0.0f;
      if (x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz) {
        const long long c = x + (long long)nx * (y + (long long)ny * z);
        v = cell_timestep(nH[c], xHI[c], (float)K[c * kstride], p);
      }
      tile[k][j][i] = v;
    }
    __syncthreads();
    const int i = threadIdx.x % kTileX, j = threadIdx.x / kTileX;
    const int x = x0 + i, y = y0 + j;
    if (x < nx && y < ny) {
      const float cx = (float)((x > 0) + (x < nx - 1)), cy = (float)((y > 0) + (y < ny - 1));
      const float wx = fmaf(w, cx, 1.0f), wxy = fmaf(w, cy * wx, wx);
      const auto plane = [&](int k) {
        float r[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) r[d] = fmaf(w, tile[k][j + d][i] + tile[k][j + d][i + 2], tile[k][j + d][i + 1]);
        return fmaf(w, r[0] + r[2], r[1]);
      };
      const int nk = nz - z0 < kTileZ ? nz - z0 : kTileZ;
      float below = plane(0), here = plane(1);
      for (int k = 0; k < nk; ++k) {
        const float above = plane(k + 2);
        const float cz = (float)((z0 + k > 0) + (z0 + k < nz - 1));
        best = fminf(best, fmaf(w, below + above, here) / fmaf(w, cz * wxy, wxy));
        below = here;
        here = above;
      }
    }
  }
  timestep_finish(best, out, done);
}

// The same in two passes over a field in memory, for grids that fill the tiles
// badly (see launch_timestep).
template <typename KT>
__global__ void __launch_bounds__(256) cell_timestep_kernel(long long n, const double* __restrict__ nH,
                                                            const double* __restrict__ xHI, const KT* __restrict__ K,
                                                            int kstride, StepArgs p, float* __restrict__ field) {
  for (long long c = blockIdx.x * 256LL + threadIdx.x; c < n; c += gridDim.x * 256LL)
    field[c] = cell_timestep(nH[c], xHI[c], (float)K[c * kstride], p);
}
__global__ void __launch_bounds__(256) filter_min_kernel(int nx, int ny, int nz, const float* __restrict__ field,
                                                         unsigned int* __restrict__ out,
                                                         unsigned long long* __restrict__ done) {
  const float w = 0.60653066f;  // e^-1/2
  const long long n = (long long)nx * ny * nz;
  float best = __int_as_float(0x7f800000);
  for (long long c = blockIdx.x * 256LL + threadIdx.x; c < n; c += gridDim.x * 256LL) {
    const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((long long)nx * ny));
    const auto row = [&](int j, int k) {
      if (j < 0 || j >= ny || k < 0 || k >= nz) return 0.0f;
      const float* f = field + (x + (long long)nx * (j + (long long)ny * k));
      return fmaf(w, (x > 0 ? f[-1] : 0.0f) + (x < nx - 1 ? f[1] : 0.0f), f[0]);
    };
    const auto plane = [&](int k) { return fmaf(w, row(y - 1, k) + row(y + 1, k), row(y, k)); };
    const float cx = (float)((x > 0) + (x < nx - 1)), cy = (float)((y > 0) + (y < ny - 1)),
                cz = (float)((z > 0) + (z < nz - 1));
    const float wx = fmaf(w, cx, 1.0f), wxy = fmaf(w, cy * wx, wx);
    best = fminf(best, fmaf(w, plane(z - 1) + plane(z + 1), plane(z)) / fmaf(w, cz * wxy, wxy));
  }
  timestep_finish(best, out, done);
}

// Whether rt_timestep takes the two passes (and so needs a field of nx ny nz
// floats): where the tiles hold more than 2.5 times the grid's cells, as those
// of a grid of a few cells across do.  Bound by the loads of the 27 neighbours,
// the passes take 30 us + 15 ps a cell whatever the shape, the tiles 10 ps a
// cell that they hold: 12x300x300 (2.7 times) 51 in tiles and 41 us in two passes,
// 2x1024x1024 (16 times) 349 and 64 us, 1x1x20000000 (256 times) 19500 and 290 us;
// 16x256x256 (2 times) 40 and 40 us, 40x300x300 (1.6 times) 80 and 91 us, 256^3 199 and
// 348 us.  (Two passes over a field allocated in each call: 150, 177 and 559 us
// for the first three.)
bool timestep_two_passes(int nx, int ny, int nz) {
  const auto tiles = [](int d, int t) { return (double)((d + t - 1) / t) * t / d; };
  return tiles(nx, kTileX) * tiles(ny, kTileY) * tiles(nz, kTileZ) > 2.5;
}

// The minimum (bits of a float) into out[1]; out[0] holds +inf between calls,
// *done 0; field: null, or what timestep_two_passes asks for.
cudaError_t launch_timestep(int nx, int ny, int nz, const double* nH, const double* xHI, const void* K, int fp64_rates,
                            double sdx, double tau_front, float eps, float alpha, float dt_max, float unit,
                            unsigned int* out, unsigned long long* done, float* field, cudaStream_t st) {
  StepArgs p = {sdx, tau_front, 0.0f, INFINITY, -1.0f, eps, alpha, dt_max, unit, dt_max / unit};
  if (sdx > 1e-30 && sdx < 1e25) {
    const float tau32 = (float)tau_front;
    p.sdx32 = (float)sdx;
    if (tau32 > 1e-12f) {
      p.hi32 = tau32 * (1.0f + 1e-6f);
      p.lo32 = tau32 * (1.0f - 1e-6f);
    } else if (tau_front == 0.0) {
      p.hi32 = 0.0f;
    }
  }
  if (field) {
    const long long n = (long long)nx * ny * nz;
    const int g = (int)(n < 152 * 8 * 256 ? (n + 255) / 256 : 152 * 8);
    if (fp64_rates)
      cell_timestep_kernel<double><<<g, 256, 0, st>>>(n, nH, xHI, (const double*)K, 1, p, field);
    else
      cell_timestep_kernel<float><<<g, 256, 0, st>>>(n, nH, xHI, (const float*)K, 2, p, field);
    filter_min_kernel<<<g, 256, 0, st>>>(nx, ny, nz, field, out, done);
    return cudaGetLastError();
  }
  const long long tiles = (long long)((nx + kTileX - 1) / kTileX) * ((ny + kTileY - 1) / kTileY) *
                          ((nz + kTileZ - 1) / kTileZ);
  const int g = (int)(tiles < 152 * 8 ? tiles : 152 * 8);
  if (fp64_rates)
    timestep_kernel<double><<<g, 256, 0, st>>>(nx, ny, nz, nH, xHI, (const double*)K, 1, p, out, done);
  else
    timestep_kernel<float><<<g, 256, 0, st>>>(nx, ny, nz, nH, xHI, (const float*)K, 2, p, out, done);
  return cudaGetLastError();
}

// h alpha_B and h as FP32 pairs (host side), for the mixed update kernels
static float4 step_pairs(double h, double alpha) {
  const double ha = h * alpha;
  const float a_hi = (float)ha, h_hi = (float)h;
  return make_float4(a_hi, (float)(ha - (double)a_hi), h_hi, (float)(h - (double)h_hi));
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

static int grid_for(long long n, int block) {
  long long g = (n + block - 1) / block;
  if (g > 152 * 32) g = 152 * 32;
  if (g < 1) g = 1;
  return (int)g;
}

cudaError_t launch_chem(int precision, long long ncell, const double* nH, double* xHI, double* xHII,
                        const void* K, void* nhi, double h, int nsub, double alpha, cudaStream_t st) {
  const int block = 256, grid = grid_for(ncell, block);
  if (precision == RT_FP64)
    chem_kernel<double, double><<<grid, block, 0, st>>>(ncell, nH, xHI, xHII, (const double*)K,
                                                         (double*)nhi, h, nsub, alpha);
  else
    chem_mixed_kernel<<<grid, block, 0, st>>>(ncell, nH, xHI, xHII, (const float2*)K, (float2*)nhi,
                                              step_pairs(h, alpha), nsub);
  return cudaGetLastError();
}

cudaError_t launch_refresh(int precision, long long ncell, const double* nH, const double* xHI,
                           void* nhi, cudaStream_t st) {
  const int block = 256, grid = grid_for(ncell, block);
  if (precision == RT_FP64)
    refresh_nhi_kernel<double><<<grid, block, 0, st>>>(ncell, nH, xHI, (double*)nhi);
  else
    refresh_nhi_pair_kernel<<<grid, block, 0, st>>>(ncell, nH, xHI, (float2*)nhi);
  return cudaGetLastError();
}

cudaError_t launch_pair(long long n, const double* src, void* dst, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  pair_kernel<<<grid, block, 0, st>>>(n, src, (float2*)dst);
  return cudaGetLastError();
}

cudaError_t launch_check_density(long long n, const double* a, unsigned long long* bad, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  check_density_kernel<<<grid, block, 0, st>>>(n, a, bad);
  return cudaGetLastError();
}

// Step 2 of a trace in one launch: the rate arrays (nbytes each, 16-byte
// aligned; b may be null) and the budget words (acc, cnt) to zero.
__global__ void zero_fields_kernel(uint4* __restrict__ a, uint4* __restrict__ b, size_t n16, size_t nbytes,
                                   unsigned long long* __restrict__ acc, int nacc, unsigned long long* __restrict__ cnt,
                                   int ncnt) {
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x) {
    a[i] = z;
    if (b) b[i] = z;
  }
  if (blockIdx.x == 0) {
    for (size_t t = 16 * n16 + threadIdx.x; t < nbytes; t += blockDim.x) {
      ((unsigned char*)a)[t] = 0;
      if (b) ((unsigned char*)b)[t] = 0;
    }
    for (int t = threadIdx.x; t < nacc; t += blockDim.x) acc[t] = 0ULL;
    for (int t = threadIdx.x; t < ncnt; t += blockDim.x) cnt[t] = 0ULL;
  }
}

cudaError_t launch_zero_fields(void* a, void* b, size_t nbytes, void* acc, int nacc, void* cnt, int ncnt,
                               cudaStream_t st) {
  if (((uintptr_t)a & 15u) || ((uintptr_t)b & 15u)) return cudaErrorInvalidValue;
  const size_t n16 = nbytes / 16;
  long long blocks = (long long)((n16 + 255) / 256);
  if (blocks > 152 * 4) blocks = 152 * 4;
  if (blocks < 1) blocks = 1;
  zero_fields_kernel<<<(int)blocks, 256, 0, st>>>((uint4*)a, (uint4*)b, n16, nbytes, (unsigned long long*)acc, nacc,
                                                  (unsigned long long*)cnt, ncnt);
  return cudaGetLastError();
}

// Adds delta to one device word (the trace self-test's phantom package).
__global__ void add_word_kernel(unsigned long long* w, unsigned long long delta) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *w += delta;
}

cudaError_t launch_add_word(unsigned long long* w, unsigned long long delta, cudaStream_t st) {
  add_word_kernel<<<1, 32, 0, st>>>(w, delta);
  return cudaGetLastError();
}

cudaError_t launch_check_state(long long n, const double* nH, const double* x, unsigned long long* bad,
                               cudaStream_t st) {
  const int block = 256;
  if (n % 2 == 0 && aligned16(nH) && aligned16(x))
    check_state2_kernel<<<grid_for(n / 2, block), block, 0, st>>>(n / 2, (const double2*)nH, (const double2*)x, bad);
  else
    check_state_kernel<<<grid_for(n, block), block, 0, st>>>(n, nH, x, bad);
  return cudaGetLastError();
}

cudaError_t launch_commit_state(int precision, long long n, unsigned long long* ctl, unsigned long long* verdict,
                               const double* sn, const double* sx, const double* sz, double* nH, double* xHI,
                               double* xHII, void* nhi, cudaStream_t st) {
  const int block = 256;
  if (n % 2 == 0 && aligned16(sn) && aligned16(sx) && aligned16(sz) && aligned16(nH) && aligned16(xHI) &&
      aligned16(xHII) && aligned16(nhi)) {
    const long long n2 = n / 2;
    const int grid = grid_for(n2, block);
    if (precision == RT_FP64)
      commit_state2_kernel<false><<<grid, block, 0, st>>>(n2, ctl, verdict, (const double2*)sn, (const double2*)sx,
                                                          (const double2*)sz, (double2*)nH, (double2*)xHI,
                                                          (double2*)xHII, nhi);
    else
      commit_state2_kernel<true><<<grid, block, 0, st>>>(n2, ctl, verdict, (const double2*)sn, (const double2*)sx,
                                                         (const double2*)sz, (double2*)nH, (double2*)xHI,
                                                         (double2*)xHII, nhi);
    return cudaGetLastError();
  }
  const int grid = grid_for(n, block);
  if (precision == RT_FP64)
    commit_state_kernel<false><<<grid, block, 0, st>>>(n, ctl, verdict, sn, sx, sz, nH, xHI, xHII, nhi);
  else
    commit_state_kernel<true><<<grid, block, 0, st>>>(n, ctl, verdict, sn, sx, sz, nH, xHI, xHII, nhi);
  return cudaGetLastError();
}

cudaError_t launch_check_refresh(int precision, long long n, unsigned long long* ctl, const double* nH, double* x,
                                 double* z, int z_given, const double* x_old, const double* z_old, void* nhi,
                                 InstDev* inst, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  if (precision == RT_FP64)
    check_refresh_kernel<false><<<grid, block, 0, st>>>(n, ctl, nH, x, z, z_given, x_old, z_old, nhi, inst);
  else
    check_refresh_kernel<true><<<grid, block, 0, st>>>(n, ctl, nH, x, z, z_given, x_old, z_old, nhi, inst);
  return cudaGetLastError();
}

cudaError_t launch_complement(long long n, const double* x, double* out, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  complement_kernel<<<grid, block, 0, st>>>(n, x, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Batched forms: one launch for every grid of a batch.  blockIdx.y selects the
// grid (its descriptor in `inst`), blocks of a row stride over its cells.
// ---------------------------------------------------------------------------

// Step 2 for every grid: zero the rates (esz bytes of k_ph and of Gamma per
// cell, together in one array where G is null), the budget sums and the
// counters.
__device__ __forceinline__ void zero_rates(void* K, void* G, size_t bytes) {
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  uint4* const a = (uint4*)K;
  uint4* const b = (uint4*)G;
  const size_t n16 = bytes / 16;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x) {
    a[i] = z;
    if (b) b[i] = z;
  }
  if (blockIdx.x == 0)
    for (size_t t = 16 * n16 + 4 * threadIdx.x; t < bytes; t += 4 * blockDim.x) {
      *(unsigned int*)((char*)K + t) = 0u;
      if (G) *(unsigned int*)((char*)G + t) = 0u;
    }
}
__global__ void batch_zero_kernel(const InstDev* __restrict__ inst, int esz) {
  const InstDev I = inst[blockIdx.y];
  const size_t bytes = (size_t)I.nx * I.ny * I.nz * esz;
  zero_rates(I.K, I.G, I.G ? bytes : 2 * bytes);
  for (int t = 0; t < 2; ++t)  // helium photon types, where the grid has them
    if (I.Khe[t]) zero_rates(I.Khe[t], I.Ghe[t], I.Ghe[t] ? bytes : 2 * bytes);
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < 8; i += blockDim.x) I.acc[i] = 0.0;
    for (int i = threadIdx.x; i < kCntWords; i += blockDim.x) I.cnt[i] = 0ULL;
  }
}

template <bool MIXED>
__global__ void batch_chem_kernel(const InstDev* __restrict__ inst, double h, int nsub, double alpha, float4 hh) {
  const InstDev I = inst[blockIdx.y];
  const F2 ha = {hh.x, hh.y}, h2 = {hh.z, hh.w};
  const long long n = (long long)I.nx * I.ny * I.nz;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    double x = I.xHI[c], z = I.xHII[c];
    if (MIXED) {
      const float kc = ((const float2*)I.K)[c].x;
      if (kc == 0.0f && is_neutral(x, z)) continue;
      const F2 nx = chem_cell_mixed(x, z, I.nH[c], kc, ha, h2, nsub);
      ((double*)I.xHI)[c] = x;
      I.xHII[c] = z;
      ((float2*)I.nhi)[c] = make_float2(nx.hi, nx.lo);
    } else {
      const double kc = ((const double*)I.K)[c];
      if (kc == 0.0 && z == 0.0 && x == 1.0) continue;
      const double nh = I.nH[c];
      chem_cell_fp64(x, z, nh, kc, h, nsub, alpha);
      ((double*)I.xHI)[c] = x;
      I.xHII[c] = z;
      ((double*)I.nhi)[c] = __dmul_rn(nh, x);
    }
  }
}

cudaError_t launch_batch_zero(const InstDev* inst, int ninst, int precision, long long max_cells, cudaStream_t st) {
  if (ninst <= 0) return cudaSuccess;
  const int esz = precision == RT_FP64 ? 8 : 4;
  long long bx = (max_cells * esz / 4 + 255) / 256;
  if (bx > 64) bx = 64;
  if (bx < 1) bx = 1;
  batch_zero_kernel<<<dim3((unsigned)bx, (unsigned)ninst), 256, 0, st>>>(inst, esz);
  return cudaGetLastError();
}

cudaError_t launch_batch_chem(const InstDev* inst, int ninst, int precision, long long max_cells, double h,
                              int nsub, double alpha, cudaStream_t st) {
  if (ninst <= 0) return cudaSuccess;
  // blocks per grid for ~4096 cells each (up to 1024): a grid's cells are
  // spread over blocks in proportion to its size, so the largest grids of a
  // batch do not finish last on a few blocks; the blocks a smaller grid does
  // not need return at once.  (64 blocks per grid took 4.0 vs 2.5 ms on the
  // 64-grid batch.)
  long long bx = (max_cells + 4095) / 4096;
  if (bx > 1024) bx = 1024;
  if (bx < 1) bx = 1;
  if (precision == RT_FP64)
    batch_chem_kernel<false><<<dim3((unsigned)bx, (unsigned)ninst), 256, 0, st>>>(inst, h, nsub, alpha,
                                                                                   step_pairs(h, alpha));
  else
    batch_chem_kernel<true><<<dim3((unsigned)bx, (unsigned)ninst), 256, 0, st>>>(inst, h, nsub, alpha,
                                                                                  step_pairs(h, alpha));
  return cudaGetLastError();
}

// Outputs of element type dtype; null ones are left out.
cudaError_t launch_read_rates(int precision, long long n, const void* K, const void* G, const double* x, void* ok,
                              void* og, void* ox, int dtype, double scale, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  const double* g = (const double*)G;
  // four cells a thread where every array allows 16-byte accesses
  if (precision == RT_FP32_MIXED && dtype == RT_DTYPE_F32 && aligned16(K) && aligned16(x) && aligned16(ok) &&
      aligned16(og) && aligned16(ox)) {
    read_rates4_kernel<<<grid_for(n / 4, block), block, 0, st>>>(n, (const float2*)K, x, (float*)ok, (float*)og,
                                                                 (float*)ox, scale);
    return cudaGetLastError();
  }
  if (precision == RT_FP64) {
    if (dtype == RT_DTYPE_F64)
      read_rates_kernel<false, double><<<grid, block, 0, st>>>(n, K, g, x, (double*)ok, (double*)og, (double*)ox, scale);
    else
      read_rates_kernel<false, float><<<grid, block, 0, st>>>(n, K, g, x, (float*)ok, (float*)og, (float*)ox, scale);
  } else {
    if (dtype == RT_DTYPE_F64)
      read_rates_kernel<true, double><<<grid, block, 0, st>>>(n, K, g, x, (double*)ok, (double*)og, (double*)ox, scale);
    else
      read_rates_kernel<true, float><<<grid, block, 0, st>>>(n, K, g, x, (float*)ok, (float*)og, (float*)ox, scale);
  }
  return cudaGetLastError();
}

cudaError_t launch_write_rates(long long n, const void* k, const void* g, int dtype, void* kg, double scale,
                               cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  if (dtype == RT_DTYPE_F64)
    write_rates_kernel<double><<<grid, block, 0, st>>>(n, (const double*)k, (const double*)g, (float2*)kg, scale);
  else
    write_rates_kernel<float><<<grid, block, 0, st>>>(n, (const float*)k, (const float*)g, (float2*)kg, scale);
  return cudaGetLastError();
}

// src of element type src_dtype into an FP64 array
cudaError_t launch_convert(long long n, const void* src, int src_dtype, void* dst, cudaStream_t st) {
  const int block = 256, grid = grid_for(n, block);
  if (src_dtype == RT_DTYPE_F64)
    convert_kernel<double><<<grid, block, 0, st>>>(n, (const double*)src, (double*)dst);
  else
    convert_kernel<float><<<grid, block, 0, st>>>(n, (const float*)src, (double*)dst);
  return cudaGetLastError();
}

}  // namespace rtg
