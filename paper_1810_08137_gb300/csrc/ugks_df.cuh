// Double-FP32 arithmetic of the DF64 form beyond the scalar core of ugks_dfcore.cuh
// (error-free transformations, sums, products): division, lazily normalised running sums,
// e^x, and the same operations on packed FP32 pairs (two velocities per lane); then the DF64
// form's kernels.
#pragma once

#include "ugks_dfcore.cuh"

namespace ugks {

// a / b: quotient q1 of the high parts, one correction from the remainder a - q1 b.  With r good to
// about an ulp (one Newton step) q1 is within an ulp of a.hi / b.hi, so a.hi - q1 b.hi is exact in
// one FMA; the rest of the remainder is added in FP32, 2^-24 of a correction of 2^-24: about 2^-48.
__device__ __forceinline__ df df_div(df a, df b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b.hi));
  r = __fmaf_rn(r, __fmaf_rn(-b.hi, r, 1.f), r);  // one Newton step: r to ~2^-24
  const float q1 = __fmul_rn(a.hi, r);
  const float e = __fmaf_rn(-q1, b.hi, a.hi);
  const float rem = __fmaf_rn(-q1, b.lo, __fadd_rn(e, a.lo));
  return fast_two_sum(q1, __fmul_rn(rem, r));
}
// Running sum acc + a b without renormalising: the rounding error of the high-part sum and
// the product's low parts go to acc.lo, which is left to grow (by at most an ulp of acc.hi
// per term); df_norm restores |lo| <= ulp(hi)/2 once the sum is complete.
__device__ __forceinline__ df df_acc(df acc, df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float pl = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)));
  const df s = two_sum(acc.hi, p);
  return {s.hi, __fadd_rn(acc.lo, __fadd_rn(s.lo, pl))};
}
__device__ __forceinline__ df df_norm(df a) { return two_sum(a.hi, a.lo); }

// e^x for x <= 0 (Maxwellian factors), about 2^-44 relative: x = k ln2 + r with
// |r| <= ln2 / 2, e^r = (e^(r/8))^8, e^(r/8) by its Taylor series to the 8th power in Horner
// form with double-FP32 coefficients 1/n (the first term left out is below 2^-50 for
// |r/8| <= 0.0434; each squaring doubles the relative error).  0 below x = -87.
__device__ __forceinline__ df df_exp(df x) {
  // ln 2 = kLn2Hi + kLn2Mid + kLn2Lo to about 2^-62; kLn2Hi has 15 significant bits, so
  // k kLn2Hi is exact for |k| < 2^9
  constexpr float kLn2Hi = 6.9314575e-01f, kLn2Mid = 1.4286068e-06f, kLn2Lo = 5.497923e-14f;
  // 1/n = kInvHi[n] + kInvLo[n]
  constexpr float kInvHi[9] = {0.f, 1.f, 5.e-01f, 3.3333334e-01f, 2.5e-01f, 2.e-01f, 1.6666667e-01f,
                               1.4285715e-01f, 1.25e-01f};
  constexpr float kInvLo[9] = {0.f, 0.f, 0.f, -9.934108e-09f, 0.f, -2.9802323e-09f, -4.967054e-09f,
                               -6.386212e-09f, 0.f};
  if (x.hi < -87.f) return {0.f, 0.f};
  const float k = rintf(__fmul_rn(x.hi, 1.442695e+00f));
  df r = df_add(x, df_of(-__fmul_rn(k, kLn2Hi)));
  r = df_sub(r, two_prod(k, kLn2Mid));
  r = df_add(r, df_of(-__fmul_rn(k, kLn2Lo)));
  const df t = {__fmul_rn(r.hi, 0.125f), __fmul_rn(r.lo, 0.125f)};
  // Horner: 1 + t (1 + t/2 (1 + t/3 (... (1 + t/8))))
  df p = df_of(1.f);
#pragma unroll
  for (int n = 8; n >= 1; n--) p = df_fma(df_mul(p, t), df{kInvHi[n], kInvLo[n]}, df_of(1.f));
  p = df_mul(p, p);
  p = df_mul(p, p);
  p = df_mul(p, p);
  const float s = __int_as_float(((int)k + 127) << 23);  // 2^k, k >= -126
  return {__fmul_rn(p.hi, s), __fmul_rn(p.lo, s)};
}

// =====================================================================================
// DF64 form of the step: f stored as double-FP32 pairs (DF4), the per-velocity arithmetic of
// the sums (S1, S7), the micro flux (S6, S8) and the implicit update (Eq. 3) in double-FP32
// on the FP32 pipe; the interface (S2-S5) and cell (Eq. 4) scalars in FP64 (the shared
// kernels, which write double-FP32 copies of their records).  The kernels follow the FP64
// form's kernels step for step: warp per cell, lane = u index, loop over the v rows.
// =====================================================================================
__device__ __forceinline__ df dfv(float2 a) { return {a.x, a.y}; }
__device__ __forceinline__ df dh(const DF4& v) { return {v.hh, v.hl}; }
__device__ __forceinline__ df db(const DF4& v) { return {v.bh, v.bl}; }
__device__ __forceinline__ DF4 mk4(df h, df b) {
  DF4 o;
  o.hh = h.hi; o.hl = h.lo; o.bh = b.hi; o.bl = b.lo;
  return o;
}
__device__ __forceinline__ DF4 split4(double h, double b) { return mk4(df_of(h), df_of(b)); }
__device__ __forceinline__ df df_half(df a) { return {0.5f * a.hi, 0.5f * a.lo}; }  // exact
__device__ __forceinline__ df df_zero() { return {0.f, 0.f}; }

// van Leer half slope d1 d2 / (d1 + d2) if d1 d2 > 0 else 0, d1 = c - a, d2 = b - c
__device__ __forceinline__ df vl_df(df a, df c, df b) {
  const df d1 = df_sub(c, a), d2 = df_sub(b, c);
  const df p = df_mul(d1, d2);
  const df r = df_div(p, df_add(d1, d2));
  return p.hi > 0.f ? r : df_zero();
}

// Ghost ring: the FP64 form's, stored as double-FP32 pairs
__device__ __forceinline__ DF4 ghost_value(DF4*, double h, double b) { return split4(h, b); }

// State conversion (set-up and checkpoint paths): FP64 rows [cell][q][(h, b)] of rows
// j0 .. j0+nrows-1 <-> double-FP32 f with its ghost ring; a block takes a cell at a time.
__global__ void k_rows_to_df(const double* __restrict__ src, DF4* __restrict__ dst, Params P, int j0,
                             int nrows) {
  for (int c = blockIdx.x; c < P.nx * nrows; c += gridDim.x) {
    const int r = c / P.nx, i = c - r * P.nx;
    const double* s = src + (size_t)c * P.nq * 2;
    DF4* d = dst + ((size_t)(j0 + r + 2) * P.ex + i + 2) * P.nq;
    for (int q = threadIdx.x; q < P.nq; q += blockDim.x) d[q] = split4(s[2 * q], s[2 * q + 1]);
  }
}
__global__ void k_df_to_rows(const DF4* __restrict__ src, double* __restrict__ dst, Params P, int j0,
                             int nrows) {
  for (int c = blockIdx.x; c < P.nx * nrows; c += gridDim.x) {
    const int r = c / P.nx, i = c - r * P.nx;
    const DF4* s = src + ((size_t)(j0 + r + 2) * P.ex + i + 2) * P.nq;
    double* d = dst + (size_t)c * P.nq * 2;
    for (int q = threadIdx.x; q < P.nq; q += blockDim.x) {
      const DF4 v = s[q];
      d[2 * q] = to_double(dh(v));
      d[2 * q + 1] = to_double(db(v));
    }
  }
}
// Pointwise Maxwellian of (rho, U, V, T) per cell (FP64, stored as double-FP32) and W.
__global__ void k_init_maxwellian_df(Params P, const double* __restrict__ prim, DF4* __restrict__ f,
                                     double* __restrict__ W, int nwe) {
  const int nc = P.nx * P.ny;
  const int cell = blockIdx.x;
  if (cell >= nc) return;
  const int i = cell % P.nx, j = cell / P.nx;
  const double rho = prim[cell], U = prim[nc + cell], V = prim[2 * nc + cell], T = prim[3 * nc + cell];
  const double lam = 1.0 / T, G = rho * lam / kPi, bf = P.K / (2.0 * lam);
  DF4* dst = f + fcell(P, i, j) * P.nq;
  for (int q = threadIdx.x; q < P.nq; q += blockDim.x) {
    const int k = q % P.nu, m = q / P.nu;
    const double du = P.u[k] - U, dv = P.v[m] - V;
    const double gh = G * exp(-lam * (du * du + dv * dv));
    dst[q] = split4(gh, bf * gh);
  }
  if (threadIdx.x == 0) {
    const int w = wcell(P, i, j);
    W[w] = rho;
    W[nwe + w] = rho * U;
    W[2 * nwe + w] = rho * V;
    W[3 * nwe + w] = rho * (0.5 * (U * U + V * V) + (P.K + 2) / (4.0 * lam));
  }
}

}  // namespace ugks
