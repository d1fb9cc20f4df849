// Velocity sums and update of the FP64 and DF64 forms, one source for both arithmetics.
//
// S1 + S7 with one thread per cell: the FP32-f form's sums_tile_body (ugks_f32.cuh) in FP64 or
// double-FP32 arithmetic, plus the slope buffer the face-flux kernel reads.  A block owns a tile of
// 8 x 4 cells (lane = cell) and one quadrant of velocity space, so it feeds one x side and one y
// side; its four warps take a share of the quadrant's rows each, and the interface kernel adds the
// two quadrants of a side.  Bound by arithmetic: FP64 64 pipe instructions per velocity-cell, the
// pipe 90 % busy (100x50x28^2 624 -> 512 us against a warp per cell); DF64 by the FMA pipe (64 %) and
// FP32 issue (55 %), so h and b, or two powers of u, go through packed pairs (200x100x28^2 538 -> 409 ->
// 369 us, 60x30x101^2 712 -> 559 -> 508 us: a warp per cell, a thread per cell, packed pairs).  The
// weights w v^n are those rounded once (formed from rounded v and w they put 13 % more error on rho V
// than on rho U of the transposed flow).
#pragma once

namespace ugks {

// Arithmetic of a form's velocity values: Num::V (8 bytes) and a 16-byte (h, b) of them.
struct NumF64 {
  using V = double;
  using H = double2;  // (h, b) in global and shared memory
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V h(const H& a) { return a.x; }
  static __device__ __forceinline__ V b(const H& a) { return a.y; }
  static __device__ __forceinline__ H pack(V h, V b) { return make_double2(h, b); }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ V sub(V a, V b) { return a - b; }
  static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
  static __device__ __forceinline__ V mad(V a, V b, V c) { return fma(a, b, c); }
  static __device__ __forceinline__ V acc(V c, V a, V b) { return fma(a, b, c); }
  static __device__ __forceinline__ V norm(V a) { return a; }
  static __device__ __forceinline__ V half(V a) { return 0.5 * a; }
  static __device__ __forceinline__ V neg(V a) { return -a; }
  static __device__ __forceinline__ V vl(V a, V c, V b) { return vl_half(a, c, b); }
  static __device__ __forceinline__ double f64(V a) { return a; }
  // two values at a time: (h, b) of a velocity, or two powers of u
  using V2 = double2;
  static __device__ __forceinline__ V2 pair(const H& a) { return a; }
  static __device__ __forceinline__ V2 of(V x, V y) { return make_double2(x, y); }
  static __device__ __forceinline__ V x(V2 a) { return a.x; }
  static __device__ __forceinline__ V y(V2 a) { return a.y; }
  static __device__ __forceinline__ H pack2(V2 a) { return a; }
  static __device__ __forceinline__ V2 acc2(V2 c, V2 a, V2 b) { return of(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)); }
  static __device__ __forceinline__ V2 vl2(V2 a, V2 c, V2 b) { return of(vl(a.x, c.x, b.x), vl(a.y, c.y, b.y)); }
  static __device__ __forceinline__ V ld(const V* p) { return *p; }
  using Face = FaceRec;
  using Cell = CellRec;
  static constexpr bool kShakhov = true;
  static __device__ __forceinline__ V val(double a) { return a; }  // a record's field
  static __device__ __forceinline__ V exp(V a) { return ::exp(a); }
  static __device__ __forceinline__ V u(const Params& P, int k) { return P.u[k]; }
  static __device__ __forceinline__ V v(const Params& P, int m) { return P.v[m]; }
  static __device__ __forceinline__ V tdx(const Params& P) { return P.d_tdx; }
  static __device__ __forceinline__ V tdy(const Params& P) { return P.d_tdy; }
  static __device__ __forceinline__ V idx(const Params& P) { return P.d_idx; }
  static __device__ __forceinline__ V idy(const Params& P) { return P.d_idy; }
  static __device__ __forceinline__ V dt(const Params& P) { return P.dt; }
  // [nu][6]: w_u u^m (m = 0..4; half at u = 0) and u; [nv][2]: v and w_v (half at v = 0)
  static __device__ __forceinline__ const V* utab(const Params& P) { return P.mvd + 5 * P.nv; }
  // [5][nv]: w_v v^n, each rounded once
  static __device__ __forceinline__ const V* vpow(const Params& P) { return P.mvd; }
};
struct NumDF {
  using V = df;
  using H = DF4;
  static __device__ __forceinline__ V zero() { return df_zero(); }
  static __device__ __forceinline__ V h(const H& a) { return dh(a); }
  static __device__ __forceinline__ V b(const H& a) { return db(a); }
  static __device__ __forceinline__ H pack(V h, V b) { return mk4(h, b); }
  static __device__ __forceinline__ V add(V a, V b) { return df_add(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return df_sub(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return df_mul(a, b); }
  static __device__ __forceinline__ V mad(V a, V b, V c) { return df_fma(a, b, c); }
  static __device__ __forceinline__ V acc(V c, V a, V b) { return df_acc(c, a, b); }  // not normalised
  static __device__ __forceinline__ V norm(V a) { return df_norm(a); }
  static __device__ __forceinline__ V half(V a) { return df_half(a); }
  static __device__ __forceinline__ V neg(V a) { return df_neg(a); }
  static __device__ __forceinline__ double f64(V a) { return to_double(a); }
  using V2 = df2;
  static __device__ __forceinline__ V2 pair(const H& a) {
    return {make_float2(a.hh, a.bh), make_float2(a.hl, a.bl)};
  }
  static __device__ __forceinline__ V2 of(V x, V y) { return {make_float2(x.hi, y.hi), make_float2(x.lo, y.lo)}; }
  static __device__ __forceinline__ V x(V2 a) { return {a.hi.x, a.lo.x}; }
  static __device__ __forceinline__ V y(V2 a) { return {a.hi.y, a.lo.y}; }
  static __device__ __forceinline__ H pack2(V2 a) { return {a.hi.x, a.hi.y, a.lo.x, a.lo.y}; }
  static __device__ __forceinline__ V2 acc2(V2 c, V2 a, V2 b) { return df2_acc(c, a, b); }
  static __device__ __forceinline__ V2 vl2(V2 a, V2 c, V2 b) { return vl2_df(a, c, b); }
  static __device__ __forceinline__ V ld(const V* p) { return dfv(*reinterpret_cast<const float2*>(p)); }
  using Face = FaceRecD;
  using Cell = CellRecD;
  static constexpr bool kShakhov = false;
  static __device__ __forceinline__ V val(float2 a) { return dfv(a); }
  static __device__ __forceinline__ V exp(V a) { return df_exp(a); }
  static __device__ __forceinline__ V u(const Params& P, int k) { return dfv(__ldg(P.gdf + k)); }
  static __device__ __forceinline__ V v(const Params& P, int m) { return dfv(__ldg(P.gdf + 2 * P.nu + m)); }
  static __device__ __forceinline__ V tdx(const Params& P) { return dfv(P.df_tdx); }
  static __device__ __forceinline__ V tdy(const Params& P) { return dfv(P.df_tdy); }
  static __device__ __forceinline__ V idx(const Params& P) { return dfv(P.df_idx); }
  static __device__ __forceinline__ V idy(const Params& P) { return dfv(P.df_idy); }
  static __device__ __forceinline__ V dt(const Params& P) { return dfv(P.df_dt); }
  static __device__ __forceinline__ const V* utab(const Params& P) {
    return reinterpret_cast<const V*>(P.gdf + 2 * P.nu + 6 * P.nv);
  }
  static __device__ __forceinline__ const V* vpow(const Params& P) {
    return reinterpret_cast<const V*>(P.gdf + 2 * P.nu + P.nv);
  }
};

constexpr int kCellPart = 4 * 32;  // partial sums of a cell: [quadrant][x side 16, y side 16]
constexpr size_t kCellSumsWarp = (size_t)kTileStages * kTileStageF4 * 16 + 32 * kTileOut * 8;

// part: [(nx+2)(ny+2) cells (W indexing)][kCellPart].  Block: (tile, quadrant), quadrant fastest;
// quadrant bit 0: u <= 0 (W side, else u >= 0, E side), bit 1: v <= 0 (S, else N).  The u = 0 column
// and the v = 0 row enter both of their halves with half weight.
template <class N>
__global__ void __launch_bounds__(128, 3) k_sums_cell(Params P, const typename N::H* __restrict__ f,
                                                      double* __restrict__ part,
                                                      typename N::H* __restrict__ slopes) {
  using V = typename N::V;
  using V2 = typename N::V2;
  using H = typename N::H;
  extern __shared__ __align__(16) unsigned char cell_sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ntx = tiles_x(P), tile = blockIdx.x >> 2, quad = blockIdx.x & 3;
  const bool un = quad & 1, vn = quad & 2;
  const int nu = P.nu, nv = P.nv, nq = P.nq;
  const int x0 = (tile % ntx) * kTileX - 1, y0 = (tile / ntx) * kTileY - 1;
  const int tx = lane & 7, ty = lane >> 3, i = x0 + tx, j = y0 + ty;
  const bool xg = i < 0 || i >= P.nx, yg = j < 0 || j >= P.ny;
  // cells whose sums are read: not corner ghosts, ghosts behind a wall, past the end
  const bool need = i <= P.nx && j <= P.ny && !(xg && yg) && !(i < 0 && P.bc_kind[0] == 1) &&
                    !(i >= P.nx && P.bc_kind[1] == 1) && !(j < 0 && P.bc_kind[2] == 1) &&
                    !(j >= P.ny && P.bc_kind[3] == 1);
  // a cell next to a pressure ghost (zero slopes) reads itself in place of its neighbours
  const bool zs = (i < 0 && P.bc_kind[0] == 2) || (i >= P.nx && P.bc_kind[1] == 2) ||
                  (j < 0 && P.bc_kind[2] == 2) || (j >= P.ny && P.bc_kind[3] == 2);
  unsigned char* wsm = cell_sm + warp * kCellSumsWarp;
  H* st = reinterpret_cast<H*>(wsm);
  V* out = reinterpret_cast<V*>(wsm + kTileStages * kTileStageF4 * 16) + lane;  // [32][kTileOut]
  const int own = ((ty + 1) * kTileRow + tx + 1) * kTilePitch;
  const int ox = zs ? 0 : kTilePitch, oy = zs ? 0 : kTileRow * kTilePitch;

  // staging: lane (column lane / 4, slot lane % 4) copies its column of the 6 rows and one halo
  // cell; rows and columns past the ghost ring repeat its last one
  static_assert(kTileSlots == 4, "one column of the tile per 4 lanes");
  const int sl = lane & 3, lc = lane >> 2;
  const size_t rs = (size_t)P.ex * nq;
  const int xlast = P.nx + 1, yspan = P.ny + 2 - y0;
  const int hx = lc < 4 ? x0 - 1 : min(x0 + kTileX, xlast), hr = lc & 3;
  const H* gcol = f + ((size_t)(y0 + 1) * P.ex + min(x0 + lc, xlast) + 2) * nq + sl;  // row y0 - 1
  const H* ghal = f + ((size_t)(min(y0 + hr, P.ny + 1) + 2) * P.ex + hx + 2) * nq + sl;
  const uint32_t dcol = smem_addr(st + (1 + lc) * kTilePitch + sl);
  const uint32_t dhal = smem_addr(st + ((1 + hr) * kTileRow + (lc < 4 ? 0 : kTileX + 1)) * kTilePitch + sl);

  const int k0 = un ? 0 : P.k_neg, k1 = un ? P.k_pos : nu;      // u columns of the quadrant
  const int ms = vn ? 0 : P.m_neg, nm = (vn ? P.m_pos : P.nv) - ms;  // its rows, and this warp's share
  const int m0 = ms + nm * warp / kWarpsPerBlock, m1 = ms + nm * (warp + 1) / kWarpsPerBlock;
  const V* ut = N::utab(P);
  const V* vt = ut + 6 * nu;
  const V* vp = N::vpow(P);
  const V tdx = N::tdx(P), tdy = N::tdy(P);
  H* slc = slopes + (size_t)wcell(P, need ? i : 0, need ? j : 0) * nq * 2;

  int pm = m0, pk = k0;  // next stage to be copied
  uint32_t pslot = 0;
  auto copy_stage = [&]() {
    if (pm < m1 && pk < k1) {
      if (pk + sl < k1) {
        const size_t s0 = (size_t)pm * nu + pk;
        const H* g = gcol + s0;
        uint32_t d = dcol + pslot;
#pragma unroll
        for (int r = 0; r < kTileY + 2; r++) {
          cp_async16_cg_u(d, g);
          d += kTileRow * kTilePitch * 16;
          if (r < yspan) g += rs;
        }
        cp_async16_cg_u(dhal + pslot, ghal + s0);
      }
      pk += kTileSlots;
      if (pk >= k1) {
        pk = k0;
        pm++;
      }
      pslot ^= kTileStageF4 * 16;
    }
    cp_async_commit();
  };

#pragma unroll 1
  for (int e = 0; e < 32; e++) out[e * kTileOut] = N::zero();
  copy_stage();
  const H* c = st + own;
  int cflip = kTileStageF4;
  for (int m = m0; m < m1; m++) {
    // sums over u^n of the value and its two half slopes: (h, b) for n < 2 or 3, then h of two powers
    V2 a0, a1, a23, x0s, x1s, x2s, x34, y0s, y1s, y23;
    a0 = a1 = a23 = x0s = x1s = x2s = x34 = y0s = y1s = y23 = N::of(N::zero(), N::zero());
    // slopes of a velocity of two quadrants (u = 0 or v = 0) are written by the upper one
    const bool wrow = need && !(vn && m >= P.m_neg);
#pragma unroll 1
    for (int k = k0; k < k1; k += kTileSlots) {
      __syncwarp();  // every lane is done with the stage refilled next
      copy_stage();
      cp_async_wait<1>();
      __syncwarp();
      const int n = min(kTileSlots, k1 - k);
#pragma unroll 1
      for (int q = 0; q < n; q++) {
        const H C = c[q], Wn = c[q - ox], E = c[q + ox], S = c[q - oy], Nn = c[q + oy];
        const V* t = ut + 6 * (k + q);
        const V w0 = N::ld(t), w1 = N::ld(t + 1), w2 = N::ld(t + 2), w3 = N::ld(t + 3), w4 = N::ld(t + 4);
        const V2 cc = N::pair(C);
        const V2 rx = N::vl2(N::pair(Wn), cc, N::pair(E)), ry = N::vl2(N::pair(S), cc, N::pair(Nn));
        if (wrow && !(un && k + q >= P.k_neg)) {
          H* q2 = slc + 2 * ((size_t)m * nu + k + q);
          q2[0] = N::pack2(rx);
          q2[1] = N::pack2(ry);
        }
        const V2 w00 = N::of(w0, w0), w11 = N::of(w1, w1), w22 = N::of(w2, w2), w23 = N::of(w2, w3);
        a0 = N::acc2(a0, w00, cc); a1 = N::acc2(a1, w11, cc); a23 = N::acc2(a23, w23, N::of(N::x(cc), N::x(cc)));
        x0s = N::acc2(x0s, w00, rx); x1s = N::acc2(x1s, w11, rx); x2s = N::acc2(x2s, w22, rx);
        x34 = N::acc2(x34, N::of(w3, w4), N::of(N::x(rx), N::x(rx)));
        y0s = N::acc2(y0s, w00, ry); y1s = N::acc2(y1s, w11, ry); y23 = N::acc2(y23, w23, N::of(N::x(ry), N::x(ry)));
      }
      c += cflip;
      cflip = -cflip;
    }
    // the row's part of the 32 face sums
    auto nx_ = [](V2 a) { return N::norm(N::x(a)); };
    auto ny_ = [](V2 a) { return N::norm(N::y(a)); };
    const V A0 = nx_(a0), A1 = nx_(a1), A2 = nx_(a23), A3 = ny_(a23), Ab0 = ny_(a0), Ab1 = ny_(a1);
    const V X0 = nx_(x0s), X1 = nx_(x1s), X2 = nx_(x2s), X3 = nx_(x34), X4 = ny_(x34);
    const V Xb0 = ny_(x0s), Xb1 = ny_(x1s), Xb2 = ny_(x2s);
    const V Y0 = nx_(y0s), Y1 = nx_(y1s), Y2 = nx_(y23), Y3 = ny_(y23), Yb0 = ny_(y0s), Yb1 = ny_(y1s);
    // tangential slopes without their factor 2/dy or 2/dx, energy components as (w/2) (q2 + b0) +
    // (w v^2/2) q0
    const V w = vt[2 * m + 1], w1 = vp[nv + m], w2 = vp[2 * nv + m], vty = N::mul(vt[2 * m], tdy);
    const V hw = N::half(w), hw1 = N::half(w1), hw2 = N::half(w2), hw3 = N::half(vp[3 * nv + m]);
    auto put = [&](int e, V g, V x) { out[e * kTileOut] = N::norm(N::acc(out[e * kTileOut], g, x)); };
    auto put2 = [&](int e, V g, V x, V g_, V x_) {
      out[e * kTileOut] = N::norm(N::acc(N::acc(out[e * kTileOut], g_, x_), g, x));
    };
    {  // x side: W0, tangential slope, Sf, Ss
      auto F = [&](V a, V x) { return un ? N::sub(a, x) : N::add(a, x); };
      const V F0 = F(A0, X0), F1 = F(A1, X1), F2 = F(A2, X2), F3 = F(A3, X3), B0 = F(Ab0, Xb0), B1 = F(Ab1, Xb1);
      put(kOffW0, w, F0); put(kOffW0 + 1, w, F1); put(kOffW0 + 2, w1, F0);
      put2(kOffW0 + 3, hw, N::add(F2, B0), hw2, F0);
      put(kOffSt, w, Y0); put(kOffSt + 1, w, Y1); put(kOffSt + 2, w1, Y0);
      put2(kOffSt + 3, hw, N::add(Y2, Yb0), hw2, Y0);
      put(kOffSf, w, F1); put(kOffSf + 1, w, F2); put(kOffSf + 2, w1, F1);
      put2(kOffSf + 3, hw, N::add(F3, B1), hw2, F1);
      const V Z1 = N::mad(tdx, X2, N::mul(vty, Y1)), Z2 = N::mad(tdx, X3, N::mul(vty, Y2));
      const V Z3 = N::mad(tdx, X4, N::mul(vty, Y3)), Zb = N::mad(tdx, Xb2, N::mul(vty, Yb1));
      put(kOffSs, w, Z1); put(kOffSs + 1, w, Z2); put(kOffSs + 2, w1, Z1);
      put2(kOffSs + 3, hw, N::add(Z3, Zb), hw2, Z1);
    }
    {  // y side
      auto F = [&](V a, V y) { return vn ? N::sub(a, y) : N::add(a, y); };
      const V F0 = F(A0, Y0), F1 = F(A1, Y1), FB = N::add(F(A2, Y2), F(Ab0, Yb0));
      put(16 + kOffW0, w, F0); put(16 + kOffW0 + 1, w, F1); put(16 + kOffW0 + 2, w1, F0);
      put2(16 + kOffW0 + 3, hw, FB, hw2, F0);
      put(16 + kOffSt, w, X0); put(16 + kOffSt + 1, w, X1); put(16 + kOffSt + 2, w1, X0);
      put2(16 + kOffSt + 3, hw, N::add(X2, Xb0), hw2, X0);
      put(16 + kOffSf, w1, F0); put(16 + kOffSf + 1, w1, F1); put(16 + kOffSf + 2, w2, F0);
      put2(16 + kOffSf + 3, hw1, FB, hw3, F0);
      const V D0 = N::mad(tdx, X1, N::mul(vty, Y0)), D1 = N::mad(tdx, X2, N::mul(vty, Y1));
      const V D2 = N::mad(tdx, X3, N::mul(vty, Y2)), Db = N::mad(tdx, Xb1, N::mul(vty, Yb0));
      put(16 + kOffSs, w1, D0); put(16 + kOffSs + 1, w1, D1); put(16 + kOffSs + 2, w2, D0);
      put2(16 + kOffSs + 3, hw1, N::add(D2, Db), hw3, D0);
    }
  }
  cp_async_wait<0>();
  const unsigned ok = __ballot_sync(kFull, need);
  __syncthreads();
  // the warps' sums, added in order: each warp writes eight cells, lane = entry
  const double scale = (lane & 12) != kOffSt ? 1.0 : lane < 16 ? P.d_tdy : P.d_tdx;
  const unsigned char* all = cell_sm + kTileStages * kTileStageF4 * 16 + sizeof(V) * lane * kTileOut;
#pragma unroll 1
  for (int t = 8 * warp; t < 8 * warp + 8; t++)
    if (ok >> t & 1) {
      double r = 0.0;
#pragma unroll
      for (int w = 0; w < kWarpsPerBlock; w++)
        r += N::f64(reinterpret_cast<const V*>(all + w * kCellSumsWarp)[t]);
      r *= scale;
      part[(size_t)wcell(P, x0 + (t & 7), y0 + (t >> 3)) * kCellPart + quad * 32 + lane] = r;
    }
}

// -------------------------------------------------------------------------------------
// S6 + S8 and Eq. 3 of the FP64 and DF64 forms in two passes: every (face, velocity) micro flux
// once.
// k_face_flux: one block per interior cell; for each velocity the cell forms the flux
// X = Q g + Mt4 f_up - Mt5 d_up (or the wall flux) through its downwind x-face and y-face from
// its own reconstruction, and a cell next to the boundary also forms the flux whose upwind side
// is the ghost cell or the wall.  Every face and velocity is written by exactly one block, into
// Xx [(nx+1) ny][nq] and Xy [nx (ny+1)][nq] (face-major, velocity innermost).  k_cell_update then
// reads the four fluxes of each velocity-cell and applies Eq. 3.
// Both are bound by arithmetic: the FP64 form by the FP64 pipe (2 operations per clock and SM),
// the DF64 form by the FP32 pipe.  Lanes run over the flattened
// velocities (a lane per u would leave 12 of 32 idle at nu = 20), and all that depends on u or v
// alone comes from tables in shared memory (one kind per warp), so a velocity-cell costs 28 FP64
// instructions for its two faces: per face 3 for Q_h, 2 for Q_b = X2 Q_h + linear, 1 for g and 4 per
// component, with f_up and d_up folded into the coefficients of the cell value and its two half
// slopes (67 before), 36 with the tables; k_cell_update 20 (24 with tables, 30 before).  A block per
// cell shares the tables and spreads small meshes evenly.  Both passes, FP64: 100x50x28^2 0.820 ->
// 0.447 ms (a warp per cell 0.518), 40x20x20^2 163 -> 70 us (90); FP64 pipe 94 % and 86 % busy.  DF64:
// 200x100x28^2 815 -> 573 us, 60x30x101^2 1478 -> 728 us (1125).
// -------------------------------------------------------------------------------------
// Q at fixed u as a polynomial in v, from a record's eight coefficients: x face (un = u, ut = v) or
// y face (un = v, ut = u).
template <class N, typename C>
__device__ __forceinline__ void poly_in_v(const C* c, typename N::V u, bool xface, typename N::V* q) {
  auto k = [&](int i) { return N::val(c[i]); };
  const int n1 = xface ? 1 : 2, n2 = xface ? 3 : 5, n3 = xface ? 6 : 7;  // powers of u
  const int t1 = xface ? 2 : 1, t2 = xface ? 5 : 3, t3 = xface ? 7 : 6;  // powers of v
  q[0] = N::mad(u, N::mad(u, N::mad(u, k(n3), k(n2)), k(n1)), k(0));
  q[1] = N::mad(u, N::mad(u, k(t3), k(4)), k(t1));
  q[2] = N::mad(u, k(n3), k(t2));
  q[3] = k(t3);
}

// Tables of k_face_flux (doubles, one after the other): per u index, the downwind x-face
// (kFluxX arrays), then the downwind y-face for v <= 0 and for v > 0 (kFluxX arrays each), then
// the factors of g of the upwind faces (x, y for v <= 0, y for v > 0; boundary cells only); per v
// index kFluxM values.
// The u tables hold up to kFluxUB values of u at a time (a larger grid is walked in blocks of u), so
// that their arrays lie at fixed distances and a wide velocity grid does not cost residency.
constexpr int kFluxUB = 40;
constexpr int kFluxX = 8;  // q0 q1 q2 q3 (Q_h in v), l0 l1 (Q_b - X2 Q_h), c1 (coefficient of r_x), g
constexpr int kFluxU = 3 * kFluxX + 3;
constexpr int kFluxM = 8;  // v; factors of g: W, E, downwind y, upwind y; coefficient of r_y: W, E, downwind y
__host__ __device__ constexpr size_t face_flux_doubles(int nv) { return kFluxU * kFluxUB + (size_t)kFluxM * nv; }

template <class N>
__global__ void __launch_bounds__(128, 4) k_face_flux(Params P, const typename N::H* __restrict__ f,
                                                      const typename N::Face* __restrict__ fxr,
                                                      const typename N::Face* __restrict__ fyr,
                                                      const typename N::H* __restrict__ sl,
                                                      typename N::H* __restrict__ Xx,
                                                      typename N::H* __restrict__ Xy) {
  using V = typename N::V;
  using H = typename N::H;
  using Face = typename N::Face;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nv = P.nv, nu = P.nu, nq = P.nq, nx = P.nx, ny = P.ny, mpos = P.m_pos;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V* tu = reinterpret_cast<V*>(smraw);
  V* tm = tu + kFluxU * kFluxUB;
  const int cell = blockIdx.x;
  const int i = cell % nx, j = cell / nx;
  const Face& RW = fxr[(size_t)j * (nx + 1) + i];
  const Face& RE = fxr[(size_t)j * (nx + 1) + i + 1];
  const Face& RS = fyr[(size_t)j * nx + i];
  const Face& RN = fyr[(size_t)(j + 1) * nx + i];
  const bool edge = i == 0 || i == nx - 1 || j == 0 || j == ny - 1;
  auto val = [](const auto& x) { return N::val(x); };
  auto gauss = [](V lam, V d) { return N::exp(N::neg(N::mul(lam, N::mul(d, d)))); };
  const V tdx = N::tdx(P), tdy = N::tdy(P), dtv = N::dt(P);

  // the block's tables, one kind per warp: x-face, y-face for v <= 0, y-face for v > 0, v
  for (int m = lane; m < (warp == 3 ? nv : 0); m += 32) {
    const V v = N::v(P, m), cv = N::mul(v, tdy);
    const bool vp = m >= mpos;
    const Face& RD = vp ? RN : RS;
    const Face& RG = vp ? RS : RN;
    auto vg = [&](const Face& R, V U) { return gauss(val(R.lam), N::sub(v, U)); };
    V* t = tm + kFluxM * m;
    t[0] = v;
    t[1] = vg(RW, val(RW.Ut));
    t[2] = vg(RE, val(RE.Ut));
    t[3] = vg(RD, val(RD.Un));
    t[4] = edge ? vg(RG, val(RG.Un)) : N::zero();
    t[5] = N::neg(N::mul(val(RW.Mt5), cv));
    t[6] = N::neg(N::mul(val(RE.Mt5), cv));
    t[7] = N::sub(vp ? val(RD.Mt4) : N::neg(val(RD.Mt4)), N::mul(val(RD.Mt5), cv));
  }
  const V MW = val(RW.Mt4), ME = val(RE.Mt4), MS = val(RS.Mt4), MN = val(RN.Mt4);
  const V XW = val(RW.bfac), XE = val(RE.bfac), XS = val(RS.bfac), XN = val(RN.bfac);
  const H* fc0 = f + fcell(P, i, j) * nq;
  const H* sl0 = sl + (size_t)wcell(P, i, j) * nq * 2;  // this cell's slopes
  H* xw0 = Xx + ((size_t)j * (nx + 1) + i) * nq;        // W face of the cell; E face: + nq
  H* ys0 = Xy + ((size_t)j * nx + i) * nq;              // S face; N face: + nx nq
  const size_t ynf = (size_t)nx * nq;
  const int kpos = P.k_pos;

  const int blocks = (nu + kFluxUB - 1) / kFluxUB;
  for (int ub = 0; ub < blocks; ub++) {
    const int kb = nu * ub / blocks, kw = nu * (ub + 1) / blocks - kb;  // this block's values of u
    if (ub) __syncthreads();  // the tables of the previous block of u are no longer read
    // u tables: Q at fixed u as a polynomial in v; a wall face passes dt f_up (Mt4 = dt, no Q)
    for (int kk = lane; kk < (warp < 3 ? kw : 0); kk += 32) {
      const int k = kb + kk;
      const V u = N::u(P, k), cu = N::mul(u, tdx);
      const bool up = k >= P.k_pos;
      // coefficient of a slope: +-Mt4 (the face value) - Mt5 c
      auto coef = [&](const Face& R, int sg, V c) {
        const V m5 = N::mul(val(R.Mt5), c);
        return sg == 0 ? N::neg(m5) : N::sub(sg > 0 ? val(R.Mt4) : N::neg(val(R.Mt4)), m5);
      };
      auto face = [&](const Face& R, int side, bool xface, V c1, V* t) {
        const auto* h = R.Q[side][0];
        const auto* b = R.Q[side][1];
        V q[4] = {N::zero(), N::zero(), N::zero(), N::zero()}, l0 = N::zero(), l1 = N::zero(), g = N::zero();
        if (!R.wall) {
          const V bf = val(R.bfac);
          auto diff = [&](int c) { return N::sub(val(b[c]), N::mul(bf, val(h[c]))); };
          const V dn = diff(1), dt = diff(2);
          poly_in_v<N>(h, u, xface, q);
          l0 = N::mad(u, xface ? dn : dt, diff(0));
          l1 = xface ? dt : dn;
          g = N::mul(val(R.G), gauss(val(R.lam), N::sub(u, val(xface ? R.Un : R.Ut))));
        }
#pragma unroll
        for (int e = 0; e < 4; e++) t[e * kFluxUB + kk] = q[e];
        t[4 * kFluxUB + kk] = l0;
        t[5 * kFluxUB + kk] = l1;
        t[6 * kFluxUB + kk] = c1;
        t[7 * kFluxUB + kk] = g;
      };
      const Face& RF = warp == 0 ? (up ? RE : RW) : warp == 1 ? RS : RN;
      face(RF, warp == 0 ? (up ? 0 : 1) : warp == 1 ? 1 : 0, warp == 0, coef(RF, warp ? 0 : up ? 1 : -1, cu),
           tu + warp * kFluxX * kFluxUB);
      if (edge) {  // the upwind faces: x, y for v <= 0 (N), y for v > 0 (S)
        const Face& RG = warp == 0 ? (up ? RW : RE) : warp == 1 ? RN : RS;
        tu[(3 * kFluxX + warp) * kFluxUB + kk] =
            N::mul(val(RG.G), gauss(val(RG.lam), N::sub(u, val(warp == 0 ? RG.Un : RG.Ut))));
      }
    }
    __syncthreads();
    const int dm = 128 / kw, dk = 128 - dm * kw;  // 128 velocities on
    int m = threadIdx.x / kw, kk = threadIdx.x - m * kw;
    while (m < nv) {
      const int k = kb + kk, q = m * nu + k;
      const bool up = k >= kpos, vp = m >= mpos;  // u > 0, v > 0
      const V* mt = tm + kFluxM * m;
      const V v = mt[0];
      const H c = fc0[q], a = sl0[2 * q], b = sl0[2 * q + 1];  // half slopes r_x, r_y (h, b)
      // X of a face from its u table, coefficient c2 of r_y, Mt4, X2 = <xi^2> and v factor of g
      auto flux = [&](const V* t, V c2, V m4, V x2, V ev) {
        const V qh = N::mad(N::mad(N::mad(t[3 * kFluxUB], v, t[2 * kFluxUB]), v, t[kFluxUB]), v, t[0]);
        const V qb = N::mad(x2, qh, N::mad(t[5 * kFluxUB], v, t[4 * kFluxUB]));
        const V c1 = t[6 * kFluxUB], g = N::mul(t[7 * kFluxUB], ev);
        return N::pack(N::mad(qh, g, N::mad(c2, N::h(b), N::mad(c1, N::h(a), N::mul(m4, N::h(c))))),
                       N::mad(qb, g, N::mad(c2, N::b(b), N::mad(c1, N::b(a), N::mul(m4, N::b(c))))));
      };
      (up ? xw0 + nq : xw0)[q] = flux(tu + kk, mt[up ? 6 : 5], up ? ME : MW, up ? XE : XW, mt[up ? 2 : 1]);
      (vp ? ys0 + ynf : ys0)[q] = flux(tu + (vp ? 2 : 1) * kFluxX * kFluxUB + kk, mt[7], vp ? MN : MS,
                                       vp ? XN : XS, mt[3]);
      if (edge) {
        // faces whose upwind side is a ghost cell or a wall
        const V u = N::u(P, k), cu = N::mul(u, tdx), cv = N::mul(v, tdy);
        auto ghost = [&](const Face& R, int side, bool xface, bool zero, V g, H fu, H au, H bu, bool plus) {
          if (R.wall) return N::pack(N::mul(dtv, g), N::mul(dtv, N::mul(val(R.bfac), g)));
          if (zero) au = bu = N::pack(N::zero(), N::zero());
          const V m4 = val(R.Mt4), m5 = val(R.Mt5);
          auto comp = [&](const auto* Q, V f0, V ax, V by) {
            V p[4];
            poly_in_v<N>(Q, u, xface, p);
            const V r = xface ? ax : by, fv = plus ? N::add(f0, r) : N::sub(f0, r);
            const V d = N::mad(cu, ax, N::mul(cv, by));
            const V qq = N::mad(N::mad(N::mad(p[3], v, p[2]), v, p[1]), v, p[0]);
            return N::sub(N::mad(qq, g, N::mul(m4, fv)), N::mul(m5, d));
          };
          return N::pack(comp(R.Q[side][0], N::h(fu), N::h(au), N::h(bu)),
                         comp(R.Q[side][1], N::b(fu), N::b(au), N::b(bu)));
        };
        if (up ? i == 0 : i == nx - 1) {
          const Face& R = up ? RW : RE;
          const long xo = up ? -(long)nq : (long)nq;
          (up ? xw0 : xw0 + nq)[q] = ghost(R, up ? 0 : 1, true, P.bc_kind[up ? 0 : 1] == 2,
                                           N::mul(tu[3 * kFluxX * kFluxUB + kk], mt[up ? 1 : 2]), fc0[q + xo],
                                           sl0[2 * (q + xo)], sl0[2 * (q + xo) + 1], up);
        }
        if (vp ? j == 0 : j == ny - 1) {
          const Face& R = vp ? RS : RN;
          const long yo = (vp ? -1L : 1L) * P.ex * nq, yso = (vp ? -1L : 1L) * P.wx * nq;
          (vp ? ys0 : ys0 + ynf)[q] = ghost(R, vp ? 0 : 1, false, P.bc_kind[vp ? 2 : 3] == 2,
                                            N::mul(tu[(3 * kFluxX + (vp ? 2 : 1)) * kFluxUB + kk], mt[4]), fc0[q + yo],
                                            sl0[2 * (q + yso)], sl0[2 * (q + yso) + 1], vp);
        }
      }
      m += dm;
      kk += dk;
      if (kk >= kw) {
        kk -= kw;
        m++;
      }
    }
  }
}

// Eq. 3 from the four face fluxes of each velocity-cell (k_face_flux): the increment
// f^{n+1} - f^n = inv (flux + cg1 (g^{n+1} - f^n) + cgn (g^n - f^n)) with inv folded into the
// coefficients; 20 FP64 instructions per velocity-cell.  The differences from f^n are formed first:
// rounding then acts on the increment, and a state at its equilibrium stays as it is (A1 g^{n+1} + An g^n
// - (A1 + An) f^n is two instructions shorter and rounds at the size of f: 13 % more error in f at
// dt/2tau of 5 and more).  Tables of the block's cell: per u index inv u/dx, g^n and g^{n+1} factors;
// per v index the same with v/dy.
__host__ __device__ constexpr size_t cell_update_doubles(int nu, int nv) { return 3 * ((size_t)nu + nv); }

template <class N>
__global__ void __launch_bounds__(128) k_cell_update(Params P, const typename N::H* __restrict__ f,
                                                     typename N::H* __restrict__ fo,
                                                     const typename N::Cell* __restrict__ cr,
                                                     const typename N::H* __restrict__ Xx,
                                                     const typename N::H* __restrict__ Xy) {
  using V = typename N::V;
  using H = typename N::H;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nv = P.nv, nu = P.nu, nq = P.nq, nx = P.nx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V* tu = reinterpret_cast<V*>(smraw);
  V* tm = tu + 3 * nu;
  const int cell = blockIdx.x;
  const int i = cell % nx, j = cell / nx;
  const typename N::Cell& C = cr[cell];
  auto val = [](const auto& x) { return N::val(x); };
  auto gauss = [](V lam, V d) { return N::exp(N::neg(N::mul(lam, N::mul(d, d)))); };
  const V inv = val(C.inv), ix = N::mul(inv, N::idx(P)), iy = N::mul(inv, N::idy(P));
  // one kind of table per warp: u with g^n, u with g^{n+1}, v with g^n, v with g^{n+1}
  for (int t = lane; t < (warp < 2 ? nu : nv); t += 32) {
    const V x = warp < 2 ? N::u(P, t) : N::v(P, t);
    const V lam = val(warp & 1 ? C.lam1 : C.lamn);
    const V c0 = val(warp == 0 ? C.Un : warp == 1 ? C.U1 : warp == 2 ? C.Vn : C.V1);
    const V g = gauss(lam, N::sub(x, c0));
    if (warp == 0) tu[t] = N::mul(ix, x);
    if (warp == 2) tm[t] = N::mul(iy, x);
    if (warp < 2) tu[(1 + warp) * nu + t] = N::mul(val(warp ? C.G1 : C.Gn), g);
    else tm[(warp - 1) * nv + t] = g;
  }
  __syncthreads();
  const V A1 = N::mul(inv, val(C.cg1)), An = N::mul(inv, val(C.cgn)), b1 = val(C.b1), bn = val(C.bn);
  const H* fc0 = f + fcell(P, i, j) * nq;
  H* fo0 = fo + fcell(P, i, j) * nq;
  const H* xw0 = Xx + ((size_t)j * (nx + 1) + i) * nq;
  const H* ys0 = Xy + ((size_t)j * nx + i) * nq;
  const size_t ynf = (size_t)nx * nq;
  const int dm = 128 / nu, dk = 128 - dm * nu;  // 128 velocities on
  int m = threadIdx.x / nu, k = threadIdx.x - m * nu;
  for (int q = threadIdx.x; q < nq; q += 128) {
    const H c = fc0[q], XW = xw0[q], XE = xw0[nq + q], XS = ys0[q], XN = ys0[ynf + q];
    const V au = tu[k], av = tm[m];
    const V gn = N::mul(tu[nu + k], tm[nv + m]), g1 = N::mul(tu[2 * nu + k], tm[2 * nv + m]);
    const V flh = N::mad(au, N::sub(N::h(XW), N::h(XE)), N::mul(av, N::sub(N::h(XS), N::h(XN))));
    const V flb = N::mad(au, N::sub(N::b(XW), N::b(XE)), N::mul(av, N::sub(N::b(XS), N::b(XN))));
    const V ch = N::h(c), cb = N::b(c);
    V dh_, db_;
    bool shk = false;
    if constexpr (N::kShakhov) shk = P.shk;
    if (!shk) {
      const V nb = N::neg(cb);
      dh_ = N::mad(A1, N::sub(g1, ch), N::mad(An, N::sub(gn, ch), flh));
      db_ = N::mad(A1, N::mad(b1, g1, nb), N::mad(An, N::mad(bn, gn, nb), flb));
    } else if constexpr (N::kShakhov) {  // g+_h = g_h (1 + S_h), g+_b = g_h (b + S_b), heat flux of f^n
      const double u = P.u[k], v = P.v[m];
      double cu = u - C.Un, cv = v - C.Vn, cq = cu * C.qx + cv * C.qy, c2 = 2.0 * C.lamn * (cu * cu + cv * cv);
      const double shn = C.an * cq * (c2 - 4.0), sbn = C.an * cq * C.bn * (c2 - 2.0);
      cu = u - C.U1; cv = v - C.V1;
      cq = cu * C.qx + cv * C.qy; c2 = 2.0 * C.lam1 * (cu * cu + cv * cv);
      const double sh1 = C.a1 * cq * (c2 - 4.0), sb1 = C.a1 * cq * C.b1 * (c2 - 2.0);
      dh_ = fma(A1, fma(g1, sh1, g1 - ch), fma(An, fma(gn, shn, gn - ch), flh));
      db_ = fma(A1, fma(g1, C.b1 + sb1, -cb), fma(An, fma(gn, C.bn + sbn, -cb), flb));
    }
    fo0[q] = N::pack(N::add(ch, dh_), N::add(cb, db_));
    m += dm;
    k += dk;
    if (k >= nu) {
      k -= nu;
      m++;
    }
  }
}

}  // namespace ugks
