// Double-FP32 arithmetic of the DF64 form beyond the scalar core of ugks_dfcore.cuh
// (error-free transformations, sums, products): lazily normalised running sums, e^x, and the sums
// kernel's operations on packed FP32 pairs; then the DF64 form's ghost value, state conversion and
// initial state (its step kernels are those of ugks_tile.cuh).
#pragma once

#include "ugks_dfcore.cuh"

namespace ugks {

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
// on the FP32 pipe; the interface (S2-S5) in FP64 and double-FP32 and the cell scalars (Eq. 4) in
// FP64 (the shared kernels, which write double-FP32 copies of their records).  The sums and the
// update run on the FP64 form's kernels (ugks_tile.cuh, arithmetic NumDF).
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

// ---- the same operations on two numbers at a time (packed FP32 pairs: one instruction for both),
// lane by lane the scalar operation's results ----
struct df2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ df2 two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b), bb = sub2(s, a);
  return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ df2 fast_two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ df2 df2_add(df2 a, df2 b) {
  const df2 s = two_sum2(a.hi, b.hi);
  return fast_two_sum2(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ df2 df2_sub(df2 a, df2 b) {  // df_add(a, -b)
  const float2 s = sub2(a.hi, b.hi), bb = sub2(s, a.hi);
  const float2 e = sub2(sub2(a.hi, sub2(s, bb)), add2(b.hi, bb));
  return fast_two_sum2(s, add2(e, sub2(a.lo, b.lo)));
}
// a b without renormalising: product of the high parts, and its rounding error plus the cross terms
__device__ __forceinline__ df2 df2_prod(df2 a, df2 b) {
  const float2 p = mul2(a.hi, b.hi);
  return {p, fma2(a.lo, b.hi, fma2(a.hi, b.lo, fma2(a.hi, b.hi, neg2(p))))};
}
__device__ __forceinline__ df2 df2_mul(df2 a, df2 b) {
  const df2 p = df2_prod(a, b);
  return fast_two_sum2(p.hi, p.lo);
}
__device__ __forceinline__ df2 df2_acc(df2 acc, df2 a, df2 b) {
  const df2 p = df2_prod(a, b), s = two_sum2(acc.hi, p.hi);
  return {s.hi, add2(acc.lo, add2(s.lo, p.lo))};
}
// van Leer half slope d1 d2 / (d1 + d2) if d1 d2 > 0 else 0, d1 = c - a, d2 = b - c.  The quotient p / t:
// q1 of the high parts, one correction from the remainder p - q1 t.  With r good to about an ulp (one
// Newton step) q1 is within an ulp of p.hi / t.hi, so p.hi - q1 t.hi is exact in one FMA; the low parts'
// share, formed by itself, is added in FP32, 2^-24 of a correction of 2^-24.  Over 3.6e7 quotients the
// error is 0.80 x 2^-48 rms, 9.1 at most (0.81 and 9.0 with the remainder as a double-FP32 difference of
// 13 instructions; with the low parts added one after the other 0.81 and 10.0).
__device__ __forceinline__ df2 vl2_df(df2 a, df2 c, df2 b) {
  const df2 d1 = df2_sub(c, a), d2 = df2_sub(b, c), p = df2_mul(d1, d2), t = df2_add(d1, d2);
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(t.hi.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(t.hi.y));
  const float2 nt = neg2(t.hi);
  r = fma2(r, fma2(nt, r, f2(1.f)), r);
  const float2 q1 = mul2(p.hi, r), nq = neg2(q1);
  const float2 rem = add2(fma2(nq, t.hi, p.hi), fma2(nq, t.lo, p.lo));
  df2 o = fast_two_sum2(q1, mul2(rem, r));
  if (!(p.hi.x > 0.f)) o.hi.x = o.lo.x = 0.f;
  if (!(p.hi.y > 0.f)) o.hi.y = o.lo.y = 0.f;
  return o;
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
      d[2 * q] = f64_of_any(v.hh) + f64_of_any(v.hl);
      d[2 * q + 1] = f64_of_any(v.bh) + f64_of_any(v.bl);
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
