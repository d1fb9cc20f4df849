// S1 + S7 of the FP64 and DF64 forms with one thread per cell: the FP32-f form's sums_tile_body
// (ugks_f32.cuh) in FP64 or double-FP32 arithmetic, plus the slope buffer these forms' face-flux
// kernels read.  A block owns a tile of 8 x 4 cells (lane = cell) and one quadrant of velocity
// space, so it feeds one x side and one y side; its four warps take a share of the quadrant's
// rows each, and the interface kernel adds the two quadrants of a side.
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
  static __device__ __forceinline__ V tdx(const Params& P) { return P.d_tdx; }
  static __device__ __forceinline__ V tdy(const Params& P) { return P.d_tdy; }
  // [nu][6]: w_u u^m (m = 0..4; half at u = 0) and u; [nv][2]: v and w_v (half at v = 0)
  static __device__ __forceinline__ const V* utab(const Params& P) { return P.mvd + 5 * P.nv; }
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
  static __device__ __forceinline__ V vl(V a, V c, V b) { return vl_df(a, c, b); }
  static __device__ __forceinline__ double f64(V a) { return to_double(a); }
  static __device__ __forceinline__ V tdx(const Params& P) { return dfv(P.df_tdx); }
  static __device__ __forceinline__ V tdy(const Params& P) { return dfv(P.df_tdy); }
  static __device__ __forceinline__ const V* utab(const Params& P) {
    return reinterpret_cast<const V*>(P.gdf + 2 * P.nu + 6 * P.nv);
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
  using H = typename N::H;
  extern __shared__ __align__(16) unsigned char cell_sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ntx = tiles_x(P), tile = blockIdx.x >> 2, quad = blockIdx.x & 3;
  const bool un = quad & 1, vn = quad & 2;
  const int nu = P.nu, nq = P.nq;
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
    V A0, A1, A2, A3, X0, X1, X2, X3, X4, Y0, Y1, Y2, Y3, Ab0, Ab1, Xb0, Xb1, Xb2, Yb0, Yb1;
    A0 = A1 = A2 = A3 = X0 = X1 = X2 = X3 = X4 = Y0 = Y1 = Y2 = Y3 = N::zero();
    Ab0 = Ab1 = Xb0 = Xb1 = Xb2 = Yb0 = Yb1 = N::zero();
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
        const V w0 = t[0], w1 = t[1], w2 = t[2], w3 = t[3], w4 = t[4];
        const V ch = N::h(C), cb = N::b(C);
        const V rxh = N::vl(N::h(Wn), ch, N::h(E)), rxb = N::vl(N::b(Wn), cb, N::b(E));
        const V ryh = N::vl(N::h(S), ch, N::h(Nn)), ryb = N::vl(N::b(S), cb, N::b(Nn));
        if (wrow && !(un && k + q >= P.k_neg)) {
          H* q2 = slc + 2 * ((size_t)m * nu + k + q);
          q2[0] = N::pack(rxh, rxb);
          q2[1] = N::pack(ryh, ryb);
        }
        A0 = N::acc(A0, w0, ch); A1 = N::acc(A1, w1, ch); A2 = N::acc(A2, w2, ch); A3 = N::acc(A3, w3, ch);
        X0 = N::acc(X0, w0, rxh); X1 = N::acc(X1, w1, rxh); X2 = N::acc(X2, w2, rxh);
        X3 = N::acc(X3, w3, rxh); X4 = N::acc(X4, w4, rxh);
        Y0 = N::acc(Y0, w0, ryh); Y1 = N::acc(Y1, w1, ryh); Y2 = N::acc(Y2, w2, ryh); Y3 = N::acc(Y3, w3, ryh);
        Ab0 = N::acc(Ab0, w0, cb); Ab1 = N::acc(Ab1, w1, cb);
        Xb0 = N::acc(Xb0, w0, rxb); Xb1 = N::acc(Xb1, w1, rxb); Xb2 = N::acc(Xb2, w2, rxb);
        Yb0 = N::acc(Yb0, w0, ryb); Yb1 = N::acc(Yb1, w1, ryb);
      }
      c += cflip;
      cflip = -cflip;
    }
    // the row's part of the 32 face sums
    auto nz = [](V& a) { a = N::norm(a); };
    nz(A0); nz(A1); nz(A2); nz(A3); nz(X0); nz(X1); nz(X2); nz(X3); nz(X4); nz(Y0); nz(Y1); nz(Y2); nz(Y3);
    nz(Ab0); nz(Ab1); nz(Xb0); nz(Xb1); nz(Xb2); nz(Yb0); nz(Yb1);
    const V v = vt[2 * m], w = vt[2 * m + 1];
    const V vv = N::mul(v, v), wv = N::mul(w, v), vty = N::mul(v, tdy);
    auto put = [&](int e, V g, V x) { out[e * kTileOut] = N::norm(N::acc(out[e * kTileOut], g, x)); };
    auto en = [&](V q2, V q0, V b0) { return N::half(N::add(N::mad(vv, q0, q2), b0)); };
    {  // x side: W0, tangential slope, Sf, Ss
      auto F = [&](V a, V x) { return un ? N::sub(a, x) : N::add(a, x); };
      const V F0 = F(A0, X0), F1 = F(A1, X1), F2 = F(A2, X2), F3 = F(A3, X3), B0 = F(Ab0, Xb0), B1 = F(Ab1, Xb1);
      put(kOffW0, w, F0); put(kOffW0 + 1, w, F1); put(kOffW0 + 2, wv, F0); put(kOffW0 + 3, w, en(F2, F0, B0));
      const V wt = N::mul(w, tdy), wvt = N::mul(wv, tdy);
      put(kOffSt, wt, Y0); put(kOffSt + 1, wt, Y1); put(kOffSt + 2, wvt, Y0); put(kOffSt + 3, wt, en(Y2, Y0, Yb0));
      put(kOffSf, w, F1); put(kOffSf + 1, w, F2); put(kOffSf + 2, wv, F1); put(kOffSf + 3, w, en(F3, F1, B1));
      const V Z1 = N::mad(tdx, X2, N::mul(vty, Y1)), Z2 = N::mad(tdx, X3, N::mul(vty, Y2));
      const V Z3 = N::mad(tdx, X4, N::mul(vty, Y3)), Zb = N::mad(tdx, Xb2, N::mul(vty, Yb1));
      put(kOffSs, w, Z1); put(kOffSs + 1, w, Z2); put(kOffSs + 2, wv, Z1); put(kOffSs + 3, w, en(Z3, Z1, Zb));
    }
    {  // y side
      auto F = [&](V a, V y) { return vn ? N::sub(a, y) : N::add(a, y); };
      const V F0 = F(A0, Y0), F1 = F(A1, Y1), F2 = F(A2, Y2), B0 = F(Ab0, Yb0);
      const V ef = en(F2, F0, B0), wvv = N::mul(w, vv);
      put(16 + kOffW0, w, F0); put(16 + kOffW0 + 1, w, F1); put(16 + kOffW0 + 2, wv, F0); put(16 + kOffW0 + 3, w, ef);
      const V wt = N::mul(w, tdx), wvt = N::mul(wv, tdx);
      put(16 + kOffSt, wt, X0); put(16 + kOffSt + 1, wt, X1); put(16 + kOffSt + 2, wvt, X0);
      put(16 + kOffSt + 3, wt, en(X2, X0, Xb0));
      put(16 + kOffSf, wv, F0); put(16 + kOffSf + 1, wv, F1); put(16 + kOffSf + 2, wvv, F0);
      put(16 + kOffSf + 3, wv, ef);
      const V D0 = N::mad(tdx, X1, N::mul(vty, Y0)), D1 = N::mad(tdx, X2, N::mul(vty, Y1));
      const V D2 = N::mad(tdx, X3, N::mul(vty, Y2)), Db = N::mad(tdx, Xb1, N::mul(vty, Yb0));
      put(16 + kOffSs, wv, D0); put(16 + kOffSs + 1, wv, D1); put(16 + kOffSs + 2, wvv, D0);
      put(16 + kOffSs + 3, wv, en(D2, D0, Db));
    }
  }
  cp_async_wait<0>();
  const unsigned ok = __ballot_sync(kFull, need);
  __syncthreads();
  // the warps' sums, added in order: each warp writes eight cells, lane = entry
  const unsigned char* all = cell_sm + kTileStages * kTileStageF4 * 16 + sizeof(V) * lane * kTileOut;
#pragma unroll 1
  for (int t = 8 * warp; t < 8 * warp + 8; t++)
    if (ok >> t & 1) {
      double r = 0.0;
#pragma unroll
      for (int w = 0; w < kWarpsPerBlock; w++)
        r += N::f64(reinterpret_cast<const V*>(all + w * kCellSumsWarp)[t]);
      part[(size_t)wcell(P, x0 + (t & 7), y0 + (t >> 3)) * kCellPart + quad * 32 + lane] = r;
    }
}

}  // namespace ugks
