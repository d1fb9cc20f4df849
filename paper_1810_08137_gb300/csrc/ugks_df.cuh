// Double-FP32 arithmetic of the DF64 form beyond the scalar core of ugks_dfcore.cuh
// (error-free transformations, sums, products): division, lazily normalised running sums,
// e^x, and the same operations on packed FP32 pairs (two velocities per lane); then the DF64
// form's kernels.
#pragma once

#include "ugks_dfcore.cuh"

namespace ugks {

// a / b: quotient of the high parts, one correction from the double-FP32 remainder
__device__ __forceinline__ df df_div(df a, df b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b.hi));
  r = __fmaf_rn(r, __fmaf_rn(-b.hi, r, 1.f), r);  // one Newton step: r to ~2^-24
  const float q1 = __fmul_rn(a.hi, r);
  const df rem = df_sub(a, df_mul(b, q1));
  return fast_two_sum(q1, __fmul_rn(rem.hi, r));
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

// ---- two double-FP32 numbers at once (two velocities of a lane), on packed FP32 pairs ----
// The operations of the scalar double-FP32 type, lane by lane: each packed instruction does
// the same operation on the .x and .y parts, so the results equal the scalar ones bitwise.
struct df2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ df2 two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  const float2 bb = sub2(s, a);
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
__device__ __forceinline__ df2 df2_neg(df2 a) { return {neg2(a.hi), neg2(a.lo)}; }
__device__ __forceinline__ df2 df2_sub(df2 a, df2 b) { return df2_add(a, df2_neg(b)); }
__device__ __forceinline__ df2 df2_mul(df2 a, df2 b) {
  const float2 p = mul2(a.hi, b.hi);
  const float2 e = fma2(a.lo, b.hi, fma2(a.hi, b.lo, fma2(a.hi, b.hi, neg2(p))));
  return fast_two_sum2(p, e);
}
// a b + c
__device__ __forceinline__ df2 df2_fma(df2 a, df2 b, df2 c) {
  const float2 p = mul2(a.hi, b.hi);
  const float2 pl = fma2(a.lo, b.hi, fma2(a.hi, b.lo, fma2(a.hi, b.hi, neg2(p))));
  const df2 s = two_sum2(c.hi, p);
  return fast_two_sum2(s.hi, add2(s.lo, add2(c.lo, pl)));
}
__device__ __forceinline__ df2 df2_bcast(df a) { return {make_float2(a.hi, a.hi), make_float2(a.lo, a.lo)}; }
__device__ __forceinline__ df2 df2_of(df a, df b) { return {make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }
__device__ __forceinline__ df df2_x(df2 a) { return {a.hi.x, a.lo.x}; }
__device__ __forceinline__ df df2_y(df2 a) { return {a.hi.y, a.lo.y}; }
__device__ __forceinline__ df2 df2_zero() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

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
// j0 .. j0+nrows-1 <-> double-FP32 f with its ghost ring; grid-stride over velocity-cells.
__global__ void k_rows_to_df(const double* __restrict__ src, DF4* __restrict__ dst, Params P, int j0,
                             int nrows) {
  const long n = (long)P.nx * nrows * P.nq;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const long c = t / P.nq;
    const int q = (int)(t - c * P.nq);
    const int r = (int)(c / P.nx), i = (int)(c - (long)r * P.nx);
    dst[((size_t)(j0 + r + 2) * P.ex + i + 2) * P.nq + q] = split4(src[2 * t], src[2 * t + 1]);
  }
}
__global__ void k_df_to_rows(const DF4* __restrict__ src, double* __restrict__ dst, Params P, int j0,
                             int nrows) {
  const long n = (long)P.nx * nrows * P.nq;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const long c = t / P.nq;
    const int q = (int)(t - c * P.nq);
    const int r = (int)(c / P.nx), i = (int)(c - (long)r * P.nx);
    const DF4 v = src[((size_t)(j0 + r + 2) * P.ex + i + 2) * P.nq + q];
    dst[2 * t] = (double)v.hh + (double)v.hl;
    dst[2 * t + 1] = (double)v.bh + (double)v.bl;
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

// -------------------------------------------------------------------------------------
// S6 + S8 in double-FP32: the FP64 form's face-flux kernel (k_face_flux) -- one warp per
// interior cell, lane = u index, the v loop split at v = 0; the cell forms the micro flux
// X = Q g + Mt4 f_up - Mt5 d of its downwind x- and y-face for every velocity (and of the
// ghost- or wall-side faces of a boundary cell) into the face-flux buffers, from its slopes in
// the slope buffer and the double-FP32 face records.  The Maxwellian factors come from
// df_exp; nothing here runs on the FP64 pipe.
// -------------------------------------------------------------------------------------
__device__ __forceinline__ df neg_lam_sq(df lam, df d) { return df_neg(df_mul(lam, df_mul(d, d))); }

// Q in v for fixed u on an x face (un = u, ut = v) or a y face (un = v, ut = u), double-FP32
__device__ __forceinline__ void poly_v_df(const float2* c, df u, bool xface, df* q) {
  if (xface) {
    q[0] = df_fma(u, df_fma(u, df_fma(u, dfv(c[6]), dfv(c[3])), dfv(c[1])), dfv(c[0]));
    q[1] = df_fma(u, df_fma(u, dfv(c[7]), dfv(c[4])), dfv(c[2]));
    q[2] = df_fma(u, dfv(c[6]), dfv(c[5]));
    q[3] = dfv(c[7]);
  } else {
    q[0] = df_fma(u, df_fma(u, df_fma(u, dfv(c[7]), dfv(c[5])), dfv(c[2])), dfv(c[0]));
    q[1] = df_fma(u, df_fma(u, dfv(c[6]), dfv(c[4])), dfv(c[1]));
    q[2] = df_fma(u, dfv(c[7]), dfv(c[3]));
    q[3] = dfv(c[6]);
  }
}
__device__ __forceinline__ df horner3_df(const df* q, df v) {
  return df_fma(df_fma(df_fma(q[3], v, q[2]), v, q[1]), v, q[0]);
}

struct FaceKD {
  df Mt4, Mt5, bf;
  int wall;
};

__global__ void __launch_bounds__(128) k_face_flux_df(Params P, const DF4* __restrict__ f,
                                                      const FaceRecD* __restrict__ fxr,
                                                      const FaceRecD* __restrict__ fyr,
                                                      const DF4* __restrict__ sl, DF4* __restrict__ Xx,
                                                      DF4* __restrict__ Xy) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nv = P.nv, nu = P.nu, nq = P.nq, nx = P.nx, ny = P.ny;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float2* tu = P.gdf;
  const float2* tv = P.gdf + 2 * nu;
  df* ev = reinterpret_cast<df*>(smraw) + warp * 4 * nv;  // [4][nv]: x W, x E, y S, y N factors in v
  const int cell = blockIdx.x * kWarpsPerBlock + warp;
  if (cell >= nx * ny) return;
  const int i = cell % nx, j = cell / nx;
  const FaceRecD& RW = fxr[(size_t)j * (nx + 1) + i];
  const FaceRecD& RE = fxr[(size_t)j * (nx + 1) + i + 1];
  const FaceRecD& RS = fyr[(size_t)j * nx + i];
  const FaceRecD& RN = fyr[(size_t)(j + 1) * nx + i];
  for (int m = lane; m < nv; m += 32) {
    const df vv = dfv(tv[m]);
    ev[0 * nv + m] = df_exp(neg_lam_sq(dfv(RW.lam), df_sub(vv, dfv(RW.Ut))));  // x faces: ut = v
    ev[1 * nv + m] = df_exp(neg_lam_sq(dfv(RE.lam), df_sub(vv, dfv(RE.Ut))));
    ev[2 * nv + m] = df_exp(neg_lam_sq(dfv(RS.lam), df_sub(vv, dfv(RS.Un))));  // y faces: un = v
    ev[3 * nv + m] = df_exp(neg_lam_sq(dfv(RN.lam), df_sub(vv, dfv(RN.Un))));
  }
  __syncwarp();
  auto faceK = [](const FaceRecD& R) { return FaceKD{dfv(R.Mt4), dfv(R.Mt5), dfv(R.bfac), R.wall}; };
  const FaceKD KW = faceK(RW), KE = faceK(RE), KS = faceK(RS), KN = faceK(RN);
  const df tdx = dfv(P.df_tdx), tdy = dfv(P.df_tdy), dtT = dfv(P.df_dt);
  const long rs = (long)P.ex * nq;
  const DF4* fc0 = f + fcell(P, i, j) * nq;
  const DF4* sl0 = sl + (size_t)wcell(P, i, j) * nq * 2;  // this cell's slopes
  DF4* xw0 = Xx + ((size_t)j * (nx + 1) + i) * nq;        // W face of the cell; E face: + nq
  DF4* ys0 = Xy + ((size_t)j * nx + i) * nq;              // S face; N face: + nx nq
  const bool pW = P.bc_kind[0] == 2, pE = P.bc_kind[1] == 2, pS = P.bc_kind[2] == 2, pN = P.bc_kind[3] == 2;

  // X of a face for the two velocities of a lane (packed): face value (fh, fb) and slope term
  // (dh_, db_) of its upwind side; inc: the gas side is upwind (a wall face then passes
  // dt f_up, else dt g_wall)
  const df2 dt2 = df2_bcast(dtT);
  bool act_ = false;  // this lane's u index is a real one (set per chunk of 32 u)
  auto flux = [&](const FaceKD& F, const df (&qh)[4], const df (&qb)[4], df2 vv, df2 g, df2 fh, df2 fb,
                  df2 dh_, df2 db_, bool inc, df2& xh, df2& xb) {
    if (F.wall) {
      xh = inc ? df2_mul(dt2, fh) : df2_mul(dt2, g);
      xb = inc ? df2_mul(dt2, fb) : df2_mul(dt2, df2_mul(df2_bcast(F.bf), g));
      return;
    }
    auto horner = [&](const df (&q)[4]) {
      return df2_fma(df2_fma(df2_fma(df2_bcast(q[3]), vv, df2_bcast(q[2])), vv, df2_bcast(q[1])), vv,
                     df2_bcast(q[0]));
    };
    const df2 m4 = df2_bcast(F.Mt4), m5 = df2_bcast(F.Mt5);
    xh = df2_sub(df2_fma(horner(qh), g, df2_mul(m4, fh)), df2_mul(m5, dh_));
    xb = df2_sub(df2_fma(horner(qb), g, df2_mul(m4, fb)), df2_mul(m5, db_));
  };
  // store the pair of a face's fluxes: row A always, row B when it is a real row
  auto put = [&](DF4* base, size_t qA, size_t qB, bool hasB, df2 xh, df2 xb) {
    if (!act_) return;
    base[qA] = mk4(df2_x(xh), df2_x(xb));
    if (hasB) base[qB] = mk4(df2_y(xh), df2_y(xb));
  };
  auto gfac = [](const FaceRecD& R, df u, float2 U) {
    return df_mul(dfv(R.G), df_exp(neg_lam_sq(dfv(R.lam), df_sub(u, dfv(U)))));
  };

  for (int k0 = 0; k0 < nu; k0 += 32) {
    const int k = k0 + lane;
    const bool act = k < nu;
    const int kk = act ? k : nu - 1;
    act_ = act;
    const df u = dfv(tu[kk]);
    df gu[4];
    gu[0] = gfac(RW, u, RW.Un);
    gu[1] = gfac(RE, u, RE.Un);
    gu[2] = gfac(RS, u, RS.Ut);
    gu[3] = gfac(RN, u, RN.Ut);
    const bool up = u.hi > 0.f;     // downwind x-face: E for u > 0, W otherwise
    const int xs = up ? 0 : 1;      // upwind side of the x-face records
    const FaceRecD& RXd = up ? RE : RW;
    const FaceRecD& RXg = up ? RW : RE;
    const FaceKD KXd = up ? KE : KW, KXg = up ? KW : KE;
    const df gXd = up ? gu[1] : gu[0], gXg = up ? gu[0] : gu[1];
    const df* evXd = ev + (up ? nv : 0);
    const df* evXg = ev + (up ? 0 : nv);
    DF4* xd0 = up ? xw0 + nq : xw0;
    DF4* xg0 = up ? xw0 : xw0 + nq;
    df qX[2][4];
#pragma unroll
    for (int c = 0; c < 2; c++) poly_v_df(RXd.Q[xs][c], u, true, qX[c]);
    const long xo = up ? -(long)nq : (long)nq;  // x-upwind neighbour in f, in q
    const bool xg = up ? i == 0 : i == nx - 1;  // it is a ghost cell (or a wall)
    const bool xz = (up && i == 0 && pW) || (!up && i == nx - 1 && pE);
    const df cu = df_mul(u, tdx);

    auto half = [&](auto vup_tag, int m0, int m1) {
      constexpr bool VUP = decltype(vup_tag)::value;  // downwind y-face: N for v > 0, S otherwise
      constexpr int ys = VUP ? 0 : 1;
      const FaceRecD& RYd = VUP ? RN : RS;
      const FaceRecD& RYg = VUP ? RS : RN;
      const FaceKD& KYd = VUP ? KN : KS;
      const FaceKD& KYg = VUP ? KS : KN;
      const df gYd = VUP ? gu[3] : gu[2], gYg = VUP ? gu[2] : gu[3];
      const df* evYd = ev + (VUP ? 3 : 2) * nv;
      const df* evYg = ev + (VUP ? 2 : 3) * nv;
      DF4* yd0 = VUP ? ys0 + (size_t)nx * nq : ys0;
      DF4* yg0 = VUP ? ys0 : ys0 + (size_t)nx * nq;
      df qY[2][4];
#pragma unroll
      for (int c = 0; c < 2; c++) poly_v_df(RYd.Q[ys][c], u, false, qY[c]);
      const long yo = VUP ? -rs : rs;                             // y-upwind neighbour in f
      const long yso = VUP ? -(long)P.wx * nq : (long)P.wx * nq;  // ... in the slope buffer
      const bool yg = VUP ? j == 0 : j == ny - 1;
      const bool yz = (VUP && j == 0 && pS) || (!VUP && j == ny - 1 && pN);
      // two rows at a time (packed pairs; an odd last row is paired with itself)
      for (int m = m0; m < m1; m += 2) {
        const bool hasB = m + 1 < m1;
        const int mB = hasB ? m + 1 : m;
        const df2 vv = df2_of(dfv(tv[m]), dfv(tv[mB]));
        const size_t qA = (size_t)m * nu + kk, qB = (size_t)mB * nu + kk;
        const DF4* pA = fc0 + qA;
        const DF4* pB = fc0 + qB;
        const DF4 cA = pA[0], cB = pB[0];
        const DF4* sA = sl0 + 2 * qA;
        const DF4* sB = sl0 + 2 * qB;
        const DF4 aA = sA[0], bA = sA[1], aB = sB[0], bB = sB[1];  // half slopes r_x, r_y
        const df2 ch = df2_of(dh(cA), dh(cB)), cb = df2_of(db(cA), db(cB));
        const df2 axh = df2_of(dh(aA), dh(aB)), axb = df2_of(db(aA), db(aB));
        const df2 ayh = df2_of(dh(bA), dh(bB)), ayb = df2_of(db(bA), db(bB));
        const df2 cv = df2_mul(vv, df2_bcast(tdy));
        const df2 cu2 = df2_bcast(cu);
        const df2 dch = df2_fma(cu2, axh, df2_mul(cv, ayh)), dcb = df2_fma(cu2, axb, df2_mul(cv, ayb));
        df2 xh, xb;
        // downwind x face: f_up = f + r_x (u > 0) or f - r_x (u < 0)
        flux(KXd, qX[0], qX[1], vv, df2_mul(df2_bcast(gXd), df2_of(evXd[m], evXd[mB])),
             up ? df2_add(ch, axh) : df2_sub(ch, axh), up ? df2_add(cb, axb) : df2_sub(cb, axb), dch, dcb,
             true, xh, xb);
        put(xd0, qA, qB, hasB, xh, xb);
        if (xg) {
          const DF4 xuA = pA[xo], xuB = pB[xo];
          DF4 auA = sA[2 * xo], buA = sA[2 * xo + 1], auB = sB[2 * xo], buB = sB[2 * xo + 1];
          if (xz) auA = buA = auB = buB = mk4(df_zero(), df_zero());
          const df2 uxh = df2_of(dh(auA), dh(auB)), uxb = df2_of(db(auA), db(auB));
          const df2 uyh = df2_of(dh(buA), dh(buB)), uyb = df2_of(db(buA), db(buB));
          const df2 duh = df2_fma(cu2, uxh, df2_mul(cv, uyh)), dub = df2_fma(cu2, uxb, df2_mul(cv, uyb));
          const df2 gh_ = df2_of(dh(xuA), dh(xuB)), gb_ = df2_of(db(xuA), db(xuB));
          df qg[2][4];
#pragma unroll
          for (int cc = 0; cc < 2; cc++) poly_v_df(RXg.Q[xs][cc], u, true, qg[cc]);
          flux(KXg, qg[0], qg[1], vv, df2_mul(df2_bcast(gXg), df2_of(evXg[m], evXg[mB])),
               up ? df2_add(gh_, uxh) : df2_sub(gh_, uxh), up ? df2_add(gb_, uxb) : df2_sub(gb_, uxb), duh,
               dub, false, xh, xb);
          put(xg0, qA, qB, hasB, xh, xb);
        }
        // downwind y face: f_up = f + r_y (v > 0) or f - r_y (v < 0)
        flux(KYd, qY[0], qY[1], vv, df2_mul(df2_bcast(gYd), df2_of(evYd[m], evYd[mB])),
             VUP ? df2_add(ch, ayh) : df2_sub(ch, ayh), VUP ? df2_add(cb, ayb) : df2_sub(cb, ayb), dch, dcb,
             true, xh, xb);
        put(yd0, qA, qB, hasB, xh, xb);
        if (yg) {
          const DF4 yuA = pA[yo], yuB = pB[yo];
          DF4 avA = sA[2 * yso], bvA = sA[2 * yso + 1], avB = sB[2 * yso], bvB = sB[2 * yso + 1];
          if (yz) avA = bvA = avB = bvB = mk4(df_zero(), df_zero());
          const df2 vxh = df2_of(dh(avA), dh(avB)), vxb = df2_of(db(avA), db(avB));
          const df2 vyh = df2_of(dh(bvA), dh(bvB)), vyb = df2_of(db(bvA), db(bvB));
          const df2 dvh = df2_fma(cu2, vxh, df2_mul(cv, vyh)), dvb = df2_fma(cu2, vxb, df2_mul(cv, vyb));
          const df2 gh_ = df2_of(dh(yuA), dh(yuB)), gb_ = df2_of(db(yuA), db(yuB));
          df qg[2][4];
#pragma unroll
          for (int cc = 0; cc < 2; cc++) poly_v_df(RYg.Q[ys][cc], u, false, qg[cc]);
          flux(KYg, qg[0], qg[1], vv, df2_mul(df2_bcast(gYg), df2_of(evYg[m], evYg[mB])),
               VUP ? df2_add(gh_, vyh) : df2_sub(gh_, vyh), VUP ? df2_add(gb_, vyb) : df2_sub(gb_, vyb),
               dvh, dvb, false, xh, xb);
          put(yg0, qA, qB, hasB, xh, xb);
        }
      }
    };
    half(std::integral_constant<bool, false>{}, 0, P.m_pos);
    half(std::integral_constant<bool, true>{}, P.m_pos, nv);
  }
}

// Eq. 3 in double-FP32 from the four face fluxes of each velocity-cell (the FP64 form's
// k_cell_update): f^{n+1} = f^n + inv [flux + cg1 (g^{n+1} - f^n) + cgn (g^n - f^n)].
__global__ void __launch_bounds__(128) k_cell_update_df(Params P, const DF4* __restrict__ f,
                                                        DF4* __restrict__ fo,
                                                        const CellRecD* __restrict__ cr,
                                                        const DF4* __restrict__ Xx,
                                                        const DF4* __restrict__ Xy) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nv = P.nv, nu = P.nu, nq = P.nq, nx = P.nx, ny = P.ny;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float2* tu = P.gdf;
  const float2* tv = P.gdf + 2 * nu;
  df* ev = reinterpret_cast<df*>(smraw) + warp * 2 * nv;  // [2][nv]: g^n, g^{n+1} factors in v
  const int cell = blockIdx.x * kWarpsPerBlock + warp;
  if (cell >= nx * ny) return;
  const int i = cell % nx, j = cell / nx;
  const CellRecD& C = cr[cell];
  for (int m = lane; m < nv; m += 32) {
    const df vv = dfv(tv[m]);
    ev[m] = df_exp(neg_lam_sq(dfv(C.lamn), df_sub(vv, dfv(C.Vn))));
    ev[nv + m] = df_exp(neg_lam_sq(dfv(C.lam1), df_sub(vv, dfv(C.V1))));
  }
  __syncwarp();
  const df inv = dfv(C.inv), cg1 = dfv(C.cg1), cgn = dfv(C.cgn);
  const df cg1b = df_mul(cg1, dfv(C.b1)), cgnb = df_mul(cgn, dfv(C.bn));
  const df idx = dfv(P.df_idx), idy = dfv(P.df_idy);
  const DF4* fc0 = f + fcell(P, i, j) * nq;
  DF4* fo0 = fo + fcell(P, i, j) * nq;
  const DF4* xw0 = Xx + ((size_t)j * (nx + 1) + i) * nq;
  const DF4* ys0 = Xy + ((size_t)j * nx + i) * nq;
  for (int k0 = 0; k0 < nu; k0 += 32) {
    const int k = k0 + lane;
    const bool act = k < nu;
    const int kk = act ? k : nu - 1;
    const df u = dfv(tu[kk]);
    const df gun = df_mul(dfv(C.Gn), df_exp(neg_lam_sq(dfv(C.lamn), df_sub(u, dfv(C.Un)))));
    const df gu1 = df_mul(dfv(C.G1), df_exp(neg_lam_sq(dfv(C.lam1), df_sub(u, dfv(C.U1)))));
    const df2 fxu = df2_bcast(df_mul(u, idx));
    const df2 gun2 = df2_bcast(gun), gu12 = df2_bcast(gu1);
    const df2 inv2 = df2_bcast(inv), cg12 = df2_bcast(cg1), cgn2 = df2_bcast(cgn);
    const df2 cg1b2 = df2_bcast(cg1b), cgnb2 = df2_bcast(cgnb);
    // two rows at a time (packed pairs; an odd last row is paired with itself)
    for (int m = 0; m < nv; m += 2) {
      const bool hasB = m + 1 < nv;
      const int mB = hasB ? m + 1 : m;
      const df2 fyv = df2_mul(df2_of(dfv(tv[m]), dfv(tv[mB])), df2_bcast(idy));
      const size_t qA = (size_t)m * nu + kk, qB = (size_t)mB * nu + kk;
      const DF4 cA = fc0[qA], cB = fc0[qB];
      const DF4 WA = xw0[qA], EA = xw0[nq + qA], SA = ys0[qA], NA = ys0[(size_t)nx * nq + qA];
      const DF4 WB = xw0[qB], EB = xw0[nq + qB], SB = ys0[qB], NB = ys0[(size_t)nx * nq + qB];
      const df2 flh = df2_fma(fxu, df2_sub(df2_of(dh(WA), dh(WB)), df2_of(dh(EA), dh(EB))),
                              df2_mul(fyv, df2_sub(df2_of(dh(SA), dh(SB)), df2_of(dh(NA), dh(NB)))));
      const df2 flb = df2_fma(fxu, df2_sub(df2_of(db(WA), db(WB)), df2_of(db(EA), db(EB))),
                              df2_mul(fyv, df2_sub(df2_of(db(SA), db(SB)), df2_of(db(NA), db(NB)))));
      const df2 gnh = df2_mul(gun2, df2_of(ev[m], ev[mB])), g1h = df2_mul(gu12, df2_of(ev[nv + m], ev[nv + mB]));
      const df2 ch = df2_of(dh(cA), dh(cB)), cb = df2_of(db(cA), db(cB));
      const df2 dhh = df2_mul(inv2, df2_add(flh, df2_add(df2_mul(cg12, df2_sub(g1h, ch)),
                                                         df2_mul(cgn2, df2_sub(gnh, ch)))));
      const df2 dbb = df2_mul(inv2, df2_add(flb, df2_add(df2_sub(df2_mul(cg1b2, g1h), df2_mul(cg12, cb)),
                                                         df2_sub(df2_mul(cgnb2, gnh), df2_mul(cgn2, cb)))));
      const df2 nh = df2_add(ch, dhh), nb = df2_add(cb, dbb);
      if (act) {
        fo0[qA] = mk4(df2_x(nh), df2_x(nb));
        if (hasB) fo0[qB] = mk4(df2_y(nh), df2_y(nb));
      }
    }
  }
}

}  // namespace ugks
