// C-ABI implementation of the GB300 UGKS library (declarations and contracts in
// include/ugks.h).  Host side: validation, velocity grid, time step, device state,
// step orchestration.  Device side: ugks_kernels.cuh.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <cmath>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "../../include/ugks.h"
#include "ugks_kernels.cuh"
#include "ugks_f32.cuh"
#include "ugks_df.cuh"
#include "ugks_tile.cuh"
#include "ugks_batch.cuh"

using namespace ugks;

struct ugks_batch_ctx;
struct ugks_ctx {
  ugks_config cfg;
  Params P;
  cudaStream_t stream = nullptr;
  int prec = 0;
  size_t t2 = 16;        // FP64 form: bytes per (h, b) pair in device f
  size_t fcells = 0;     // cells of the f buffers (ghost ring 2)
  int nwe = 0;           // cells of the W buffers (ghost ring 1)
  void* f[2] = {nullptr, nullptr};
  double* W[2] = {nullptr, nullptr};
  int cur = 0;
  double* sums = nullptr;
  double2* slopes = nullptr;  // FP64 form: van Leer slopes kept by the sums kernel for the update
  double2* xflux = nullptr;   // FP64 form: micro flux of every face and velocity, x faces then y
  FaceRec* fxr = nullptr;
  FaceRec* fyr = nullptr;
  double* Fx = nullptr;
  double* Fy = nullptr;
  CellRec* cells = nullptr;
  FaceRecF* fxf = nullptr;   // FP32 form: float face and cell records for the walk kernel
  FaceRecF* fyf = nullptr;
  CellRecF* cellf = nullptr;
  double* mt4 = nullptr;     // Mt4 per face (x faces then y faces)
  FaceRecD* fxd = nullptr;   // DF64 form: double-FP32 face and cell records, grid tables
  FaceRecD* fyd = nullptr;
  CellRecD* celld = nullptr;
  float2* gdf = nullptr;
  int nchunk_neg = 0, nchunk_pos = 0;
  int walk_rows = kWalkRows; // FP32 form: rows per tile of the walk (stepped alone)
  int sums_split = 1;        // FP32 form: warps per cell of the sums kernel (velocity-space split)
  bool sums_tiled = false;   // FP32 form: sums with one thread per cell
  double* hs = nullptr;      // Shakhov model: heat-flux moment sums, kNHeat per cell
  CellShkF* cshk = nullptr;  // Shakhov model, FP32-f form: per-cell Shakhov factors
  // FP32 form: the step runs the batch kernels over a one-instance table, so an instance
  // stepped alone executes exactly the code it executes inside a batch
  SlotDev* d_slot = nullptr;
  BatchWork* d_work = nullptr;
  int grid1[16] = {0};       // per step kernel: blocks of its launch
  int device = -1;                  // device current at its creation
  ugks_batch_ctx* owner = nullptr;  // batch this instance is a slot of
  double* rpart = nullptr;
  int nrblocks = 0;
  int face_block = 128;      // faces and cells per block of the interface and cell kernels
  int cell_block = 128;
  int* err = nullptr;
  double* d_grid = nullptr;  // u[nu], v[nv], wu[nu], wv[nv], [5][nv] wv v^n
  double* stage = nullptr;   // FP64 staging for FP32 state conversion: two halves, stage_bytes
  double2* grefd = nullptr;  // FP32 form: g_ref per velocity in FP64 (state conversion)
  cudaStream_t xstream = nullptr;     // FP32 form: host <-> staging copies
  cudaEvent_t ev_copied[2] = {nullptr, nullptr}, ev_free[2] = {nullptr, nullptr};
  float4* gref4 = nullptr;   // FP32 form: g_ref per slot of the paired-row layout
  float* ftab = nullptr;     // FP32 form: velocity tables (pwt, uwf)
  size_t stage_bytes = 0;
  std::vector<double> hu, hv, hwu, hwv;
  size_t bytes = 0;
  long steps_done = 0;
  std::string last_error;
  // one captured graph per ping-pong parity of the step (replayed on `stream`)
  cudaStream_t cap_stream = nullptr;
  cudaGraphExec_t graph[2] = {nullptr, nullptr};
  // tracing: one set of UGKS_NKERNELS+1 events per profiled step
  bool profiling = false;
  std::vector<cudaEvent_t> events;
  size_t events_used = 0;
};

namespace {

ugks_status fail(ugks_ctx* h, ugks_status s, const std::string& msg) {
  if (h) h->last_error = msg;
  return s;
}

ugks_status cuda_fail(ugks_ctx* h, cudaError_t e, const char* where) {
  return fail(h, UGKS_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define CK(call)                                                \
  do {                                                          \
    cudaError_t e_ = (call);                                    \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call);      \
  } while (0)

void axis(int n, double lo, double hi, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  if (n == 1) { x[0] = 0.5 * (lo + hi); w[0] = 1.0; return; }
  const double d = (hi - lo) / (n - 1), c = 0.5 * (lo + hi);
  for (int k = 0; k < n; k++) {
    x[k] = c + (k - 0.5 * (n - 1)) * d;  // symmetric about the centre
    w[k] = (k == 0 || k == n - 1) ? 0.5 * d : d;
  }
}

// Prandtl number of a configuration: pr <= 0 (a zero-initialised field) means BGK, 1.
double shakhov_pr(const ugks_config* c) { return c->pr > 0.0 ? c->pr : 1.0; }

const char* validate(const ugks_config* c) {
  if (!c) return "cfg is NULL";
  if (c->nx < 1 || c->ny < 1) return "nx, ny must be >= 1";
  if ((long)c->nx * c->ny > 400000000L) return "too many cells";
  if (c->nu < 1 || c->nv < 1 || c->nu > kMaxAxis || c->nv > kMaxAxis) return "nu, nv must be in [1, 512]";
  if ((long)c->nu * c->nv > kMaxNq) return "nu*nv must be <= 65536";
  if (!(c->lx > 0) || !(c->ly > 0)) return "lx, ly must be > 0";
  if (c->nu > 1 && !(c->umax > c->umin)) return "umax must exceed umin";
  if (c->nv > 1 && !(c->vmax > c->vmin)) return "vmax must exceed vmin";
  if (c->K < 0 || c->K > 8) return "K must be in [0, 8]";
  if (!(c->kn > 0) || !isfinite(c->kn)) return "kn must be finite and > 0";
  if (!(c->alpha > 0) || !(c->omega >= 0) || !(c->omega < 2.5)) return "bad omega/alpha";
  if (!(c->dt > 0) && !(c->cfl > 0)) return "need cfl > 0 or dt > 0";
  if (c->precision != UGKS_FP64 && c->precision != UGKS_FP32F && c->precision != UGKS_DF64)
    return "bad precision";
  if (!std::isfinite(c->pr)) return "pr must be finite";
  if (shakhov_pr(c) != 1.0 && c->precision == UGKS_DF64)
    return "Shakhov model (pr != 1): UGKS_FP64 or UGKS_FP32F form only";
  for (int s = 0; s < 4; s++) {
    const ugks_bc& b = c->bc[s];
    if (b.kind < 0 || b.kind > 2) return "bad boundary kind";
    if (b.kind == UGKS_BC_PRESSURE && (!(b.rho > 0) || !(b.T > 0))) return "pressure boundary needs rho, T > 0";
    if (b.kind == UGKS_BC_WALL && !(b.T > 0)) return "wall needs T > 0";
  }
  if ((c->bc[0].kind == UGKS_BC_PERIODIC) != (c->bc[1].kind == UGKS_BC_PERIODIC)) return "periodic W/E must be paired";
  if ((c->bc[2].kind == UGKS_BC_PERIODIC) != (c->bc[3].kind == UGKS_BC_PERIODIC)) return "periodic S/N must be paired";
  if (c->bc[0].kind == UGKS_BC_PERIODIC && c->nx < 2) return "periodic x needs nx >= 2";
  if (c->bc[2].kind == UGKS_BC_PERIODIC && c->ny < 2) return "periodic y needs ny >= 2";
  return nullptr;
}

// Derived constants of P (after K, dx, dy, dt and mu_ref are set).
void set_derived(Params& P) {
  P.inv_kp2 = 1.0 / (P.K + 2);
  P.half_dt_mu = P.dt / (2.0 * P.mu_ref);
  P.quarter_dt_mu = P.dt / (4.0 * P.mu_ref);
  P.d_tdx = 2.0 / P.dx;
  P.d_tdy = 2.0 / P.dy;
  P.d_idx = 1.0 / P.dx;
  P.d_idy = 1.0 / P.dy;
}

// Bytes of one half of the FP32 form's host staging buffer: about 32 MiB, at least one mesh
// row of FP64 f and at most half the mesh, rounded up to 256 bytes so that both halves are
// aligned for any access.
size_t stage_half_bytes(size_t row_d, size_t ny) {
  size_t want = (size_t)64 << 20;
  if (want < 2 * row_d) want = 2 * row_d;
  if (want > row_d * ny) want = row_d * ny;
  if (want < 2 * row_d) want = 2 * row_d;  // two halves of at least one row each
  return ((want / 2) + 255) & ~(size_t)255;
}

// Row pairs of the FP32 paired-row layout for a velocity axis: (v < 0 half, all).  Each half
// of the v axis (v < 0, v >= 0) is padded to an even number of rows.
std::pair<int, int> f32_row_pairs(int nv, double vmin, double vmax) {
  std::vector<double> v, w;
  axis(nv, vmin, vmax, v, w);
  int mneg = 0;
  for (int m = 0; m < nv; m++)
    if (v[m] < 0) mneg = m + 1;
  const int pn = (mneg + 1) / 2;
  return {pn, pn + (nv - mneg + 1) / 2};
}

// Threads per block of the interface and cell kernels (one thread per face or cell) for n faces or
// cells in a launch: one warp where whole blocks would leave SMs of a GB300 (152) idle, since their FP64
// chains are bound by one SM's FP64 pipe (2 operations per clock).  40x20 cells 14.9 -> 12.8 us.  The
// cell blocks fix the order in which a residual is added up and the device bytes of an instance, so
// they depend on the instance alone, not on the device; a face's result does not depend on its block.
int small_block(long n) { return n < 152 * 128 ? 32 : 128; }

// Velocity sums per cell: the FP64 and DF64 forms' BGK sums kernel keeps its four quadrants apart (the
// Shakhov model's kernel, kNSum of them, gets the same room: the model adds only its own buffers).
int sums_per_cell(const ugks_config* c) { return c->precision != UGKS_FP32F ? kCellPart : kNSum; }

// Device bytes ugks_create allocates for cfg (cudaMalloc sizes, without allocator rounding).
size_t predict_bytes(const ugks_config* c) {
  const size_t nx = c->nx, ny = c->ny, nq = (size_t)c->nu * c->nv, nc = nx * ny;
  const bool f32 = c->precision == UGKS_FP32F, dfm = c->precision == UGKS_DF64;
  const size_t pr_all = f32_row_pairs(c->nv, c->vmin, c->vmax).second, fs = pr_all * c->nu;
  const size_t fslot = f32 ? fs * sizeof(float4) : nq * sizeof(double2);  // f bytes per cell
  const size_t fcells = (nx + 4) * (ny + 4), nwe = (nx + 2) * (ny + 2);
  const size_t nfx = (nx + 1) * ny, nfy = nx * (ny + 1), cb = small_block(nc), nrb = (nc + cb - 1) / cb;
  size_t b = 2 * fcells * fslot + 2 * 4 * sizeof(double) * nwe + sizeof(double) * sums_per_cell(c) * nwe;
  if (shakhov_pr(c) != 1.0) b += sizeof(double) * kNHeat * nwe + (f32 ? sizeof(CellShkF) * nc : 0);
  b += f32 ? sizeof(FaceRecF) * (nfx + nfy) : (dfm ? sizeof(FaceRecD) : sizeof(FaceRec)) * (nfx + nfy);
  b += sizeof(double) * 4 * (nfx + nfy) + sizeof(double) * (nfx + nfy);
  b += f32 ? sizeof(CellRecF) * nc : (dfm ? sizeof(CellRecD) : sizeof(CellRec)) * nc;
  if (dfm) b += sizeof(float2) * (8 * (size_t)c->nu + 8 * (size_t)c->nv);
  b += sizeof(double) * 8 * nrb + sizeof(int) + sizeof(double) * (8 * (size_t)c->nu + 9 * (size_t)c->nv);
  if (!f32) b += nwe * nq * 2 * sizeof(double2) + (nfx + nfy) * nq * sizeof(double2);  // slopes, face fluxes
  if (f32) {
    const size_t row_d = nx * nq * 2 * sizeof(double);
    b += 2 * stage_half_bytes(row_d, ny) + sizeof(float4) * fs + sizeof(double2) * nq +
         sizeof(float) * (12 * (pr_all + 1) + 14 * (size_t)c->nu);
    b += sizeof(SlotDev) + sizeof(BatchWork);
  }
  return b;
}

template <typename T>
size_t smem_sums(int nv) {
  (void)nv;
  return sums_smem_bytes<T>();
}
template <typename T>
size_t smem_update(int nv) {
  return (1 + 6 * kWarpsPerBlock) * (size_t)nv * sizeof(T);
}
static_assert(face_flux_doubles(kMaxAxis) * sizeof(double) <= 48 * 1024 &&
                  cell_update_doubles(kMaxAxis, kMaxAxis) * sizeof(double) <= 48 * 1024,
              "update tables: no raised shared-memory limit");

// dynamic shared memory limits of the FP64 form's sums and update kernels
cudaError_t set_smem_limits_fp64(int nv) {
  cudaError_t e = cudaFuncSetAttribute(k_sums<double, double2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_sums<double>(nv));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sums_cell<NumF64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(kWarpsPerBlock * kCellSumsWarp));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_update<double, double2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)smem_update<double>(nv));
}

// The ghost ring is one launch, timed as ghost_x; ghost_y keeps its place and counts no launch.
const char* const kKernelNames[UGKS_NKERNELS] = {"ghost_x", "ghost_y", "sums", "faces", "cells",
                                                   "update"};
constexpr int kNoKernel = 1;

// Records event `k` of the current profiled step (no-op when not profiling).
cudaError_t mark(ugks_ctx* h, int k) {
  if (!h->profiling) return cudaSuccess;
  const size_t idx = h->events_used + k;
  while (h->events.size() <= idx) {
    cudaEvent_t e;
    cudaError_t r = cudaEventCreate(&e);
    if (r != cudaSuccess) return r;
    h->events.push_back(e);
  }
  return cudaEventRecord(h->events[idx], h->stream);
}

cudaError_t launch_step_f32(ugks_ctx* h, cudaStream_t st);
cudaError_t setup_single_f32(ugks_ctx* h);
cudaError_t upload_single_f32(ugks_ctx* h);
int auto_sums_split(const Params& P, int sms);
bool use_sums_tiles(const Params& P, int split, int sms);
SlotDev slot_desc(const ugks_ctx* h, int par, int walk_rows, int walk_vtile = 0);
ugks_status upload_owner(ugks_ctx* h);

template <class N>
void launch_sums_cell(const Params& P, const typename N::H* f, double* part, typename N::H* slopes, cudaStream_t st) {
  k_sums_cell<N><<<4 * tiles_x(P) * tiles_y(P), 32 * kWarpsPerBlock, kWarpsPerBlock * kCellSumsWarp, st>>>(
      P, f, part, slopes);
}

// The update in two passes: every face flux once, then Eq. 3 per velocity-cell.
template <class N>
void launch_update(const Params& P, const typename N::H* fi, typename N::H* fo, const typename N::Face* fx,
                   const typename N::Face* fy, const typename N::Cell* cells, const typename N::H* slopes,
                   typename N::H* Xx, typename N::H* Xy, cudaStream_t st) {
  const int nc = P.nx * P.ny;
  k_face_flux<N><<<nc, 128, face_flux_doubles(P.nv) * sizeof(double), st>>>(P, fi, fx, fy, slopes, Xx, Xy);
  k_cell_update<N><<<nc, 128, cell_update_doubles(P.nu, P.nv) * sizeof(double), st>>>(P, fi, fo, cells, Xx, Xy);
}

template <typename T>
cudaError_t launch_step(ugks_ctx* h, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    return launch_step_f32(h, st);
  } else {
  using T2 = typename Vec2<T>::type;
  const Params& P = h->P;
  T2* fi = static_cast<T2*>(h->f[h->cur]);
  T2* fo = static_cast<T2*>(h->f[h->cur ^ 1]);
  double* Wi = h->W[h->cur];
  double* Wo = h->W[h->cur ^ 1];
  cudaError_t r;
  if ((r = mark(h, 0)) != cudaSuccess) return r;
  k_ghost<T2><<<ghost_cells(P), 128, 0, st>>>(P, fi, Wi, h->nwe);
  if ((r = mark(h, 1)) != cudaSuccess) return r;
  if ((r = mark(h, 2)) != cudaSuccess) return r;
  const int nce = (P.nx + 2) * (P.ny + 2);
  double* sums = h->sums;
  const int nf = (P.nx + 1) * P.ny + P.nx * (P.ny + 1), fb = (nf + h->face_block - 1) / h->face_block;
  if (P.shk) {  // the Shakhov model's heat-flux sums run one warp per cell
    k_sums<T, T2><<<(nce + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock, smem_sums<T>(P.nv), st>>>(
        P, fi, sums, reinterpret_cast<T2*>(h->slopes));
    if ((r = mark(h, 3)) != cudaSuccess) return r;
    k_faces<kRecF64, false><<<fb, h->face_block, 0, st>>>(P, sums, Wi, h->nwe, h->fxr, h->fyr, h->Fx, h->Fy, h->mt4);
  } else {
    launch_sums_cell<NumF64>(P, fi, sums, reinterpret_cast<T2*>(h->slopes), st);
    if ((r = mark(h, 3)) != cudaSuccess) return r;
    k_faces<kRecF64, true><<<fb, h->face_block, 0, st>>>(P, sums, Wi, h->nwe, h->fxr, h->fyr, h->Fx, h->Fy, h->mt4);
  }
  if ((r = mark(h, 4)) != cudaSuccess) return r;
  k_cells<<<h->nrblocks, h->cell_block, 0, st>>>(P, Wi, Wo, h->nwe, h->Fx, h->Fy, h->cells, h->rpart, h->err,
                                       h->cellf, h->mt4);
  if ((r = mark(h, 5)) != cudaSuccess) return r;
  T2* Xx = reinterpret_cast<T2*>(h->xflux);
  T2* Xy = Xx + (size_t)(P.nx + 1) * P.ny * P.nq;
  launch_update<NumF64>(P, fi, fo, h->fxr, h->fyr, h->cells, reinterpret_cast<T2*>(h->slopes), Xx, Xy, st);
  if ((r = mark(h, 6)) != cudaSuccess) return r;
  if (h->profiling) h->events_used += UGKS_NKERNELS + 1;
  return cudaGetLastError();
  }
}

// DF64 form: ghost ring, double-FP32 sums, FP64 interface and cell scalars (double-FP32
// records), double-FP32 face fluxes and Eq. 3.
cudaError_t set_smem_limits_df() {
  return cudaFuncSetAttribute(k_sums_cell<NumDF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(kWarpsPerBlock * kCellSumsWarp));
}

cudaError_t launch_step_df(ugks_ctx* h, cudaStream_t st) {
  const Params& P = h->P;
  DF4* fi = static_cast<DF4*>(h->f[h->cur]);
  DF4* fo = static_cast<DF4*>(h->f[h->cur ^ 1]);
  double* Wi = h->W[h->cur];
  double* Wo = h->W[h->cur ^ 1];
  DF4* sl = reinterpret_cast<DF4*>(h->slopes);
  cudaError_t r;
  if ((r = mark(h, 0)) != cudaSuccess) return r;
  k_ghost<DF4><<<ghost_cells(P), 128, 0, st>>>(P, fi, Wi, h->nwe);
  if ((r = mark(h, 1)) != cudaSuccess) return r;
  if ((r = mark(h, 2)) != cudaSuccess) return r;
  launch_sums_cell<NumDF>(P, fi, h->sums, sl, st);
  if ((r = mark(h, 3)) != cudaSuccess) return r;
  const int nf = (P.nx + 1) * P.ny + P.nx * (P.ny + 1);
  k_faces<kRecDF, true><<<(nf + h->face_block - 1) / h->face_block, h->face_block, 0, st>>>(P, h->sums, Wi, h->nwe, h->fxd, h->fyd, h->Fx, h->Fy,
                                                    h->mt4);
  if ((r = mark(h, 4)) != cudaSuccess) return r;
  k_cells<<<h->nrblocks, h->cell_block, 0, st>>>(P, Wi, Wo, h->nwe, h->Fx, h->Fy, nullptr, h->rpart, h->err, nullptr,
                                       h->mt4, h->celld);
  if ((r = mark(h, 5)) != cudaSuccess) return r;
  DF4* Xx = reinterpret_cast<DF4*>(h->xflux);
  DF4* Xy = Xx + (size_t)(P.nx + 1) * P.ny * P.nq;
  launch_update<NumDF>(P, fi, fo, h->fxd, h->fyd, h->celld, sl, Xx, Xy, st);
  if ((r = mark(h, 6)) != cudaSuccess) return r;
  if (h->profiling) h->events_used += UGKS_NKERNELS + 1;
  return cudaGetLastError();
}

// One step of the handle's form, enqueued on st.
cudaError_t launch_any(ugks_ctx* h, cudaStream_t st) {
  if (h->prec == UGKS_FP64) return launch_step<double>(h, st);
  if (h->prec == UGKS_DF64) return launch_step_df(h, st);
  return launch_step<float>(h, st);
}

constexpr int kConvBlocks = 1216;  // blocks of the state conversion kernels: 8 per SM
// 16-byte alignment of a caller's FP64 rows (the state conversion kernels then move each
// (h, b) pair as one 16-byte access)
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <typename T2>
__global__ void k_init_maxwellian(Params P, const double* __restrict__ prim, T2* __restrict__ f,
                                  double* __restrict__ W, int nwe) {
  const int nc = P.nx * P.ny;
  const int cell = blockIdx.x;
  if (cell >= nc) return;
  const int i = cell % P.nx, j = cell / P.nx;
  const double rho = prim[cell], U = prim[nc + cell], V = prim[2 * nc + cell], T = prim[3 * nc + cell];
  const double lam = 1.0 / T, G = rho * lam / kPi, bf = P.K / (2.0 * lam);
  T2* dst = f + fcell(P, i, j) * P.nq;
  for (int q = threadIdx.x; q < P.nq; q += blockDim.x) {
    const int k = q % P.nu, m = q / P.nu;
    const double du = P.u[k] - U, dv = P.v[m] - V;
    const double gh = G * exp(-lam * (du * du + dv * dv));
    double rh, rb;
    ref_maxwellian(P, P.u[k], P.v[m], rh, rb);
    T2 o;
    o.x = gh - rh;
    o.y = bf * gh - rb;
    dst[q] = o;
  }
  if (threadIdx.x == 0) {
    const int w = wcell(P, i, j);
    W[w] = rho;
    W[nwe + w] = rho * U;
    W[2 * nwe + w] = rho * V;
    W[3 * nwe + w] = rho * (0.5 * (U * U + V * V) + (P.K + 2) / (4.0 * lam));
  }
}

__global__ void k_prim(Params P, const double* __restrict__ W, int nwe, double* __restrict__ out) {
  const int nc = P.nx * P.ny;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nc) return;
  const int w = wcell(P, c % P.nx, c / P.nx);
  const double r = W[w], U = W[nwe + w] / r, V = W[2 * nwe + w] / r;
  const double lam = (P.K + 2) * r / (4.0 * (W[3 * nwe + w] - 0.5 * r * (U * U + V * V)));
  out[c] = r;
  out[nc + c] = U;
  out[2 * nc + c] = V;
  out[3 * nc + c] = 1.0 / lam;
}

// W between its ghosted buffers and the caller's [4][nc] device rows, in one launch.
__global__ void k_copy_W(Params P, double* __restrict__ Wg, int nwe, double* __restrict__ Wc, bool out) {
  const int nc = P.nx * P.ny, t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nc) return;
  const int w = wcell(P, t % P.nx, t / P.nx);
  for (int c = 0; c < 4; c++) {
    if (out) Wc[(size_t)c * nc + t] = Wg[(size_t)c * nwe + w];
    else Wg[(size_t)c * nwe + w] = Wc[(size_t)c * nc + t];
  }
}

// FP64 form: the ghosted f buffer and the caller's device rows (8-byte aligned), a block per cell.
__global__ void k_copy_f(Params P, double2* __restrict__ fg, double* __restrict__ fc, bool out) {
  for (int c = blockIdx.x; c < P.nx * P.ny; c += gridDim.x) {
    double* g = reinterpret_cast<double*>(fg + fcell(P, c % P.nx, c / P.nx) * P.nq);
    double* u = fc + (size_t)c * P.nq * 2;
    for (int q = threadIdx.x; q < 2 * P.nq; q += blockDim.x) {
      if (out) u[q] = g[q];
      else g[q] = u[q];
    }
  }
}

// Whether a kernel of the handle may move the caller's device rows itself: memory of the handle's own
// device from the first byte to the last, 8-byte aligned, with that device current.  Everything else
// (another GPU's memory, managed or host memory, odd addresses) goes through the runtime's copies,
// which reach it or refuse it without a fault.
bool own_rows(const ugks_ctx* h, const void* p, size_t bytes) {
  int dev = -1;
  cudaPointerAttributes a0, a1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != h->device || (reinterpret_cast<uintptr_t>(p) & 7) != 0 ||
      cudaPointerGetAttributes(&a0, p) != cudaSuccess ||
      cudaPointerGetAttributes(&a1, static_cast<const char*>(p) + bytes - 1) != cudaSuccess) {
    cudaGetLastError();  // clear the error of an unknown pointer
    return false;
  }
  return a0.type == cudaMemoryTypeDevice && a1.type == cudaMemoryTypeDevice && a0.device == h->device &&
         a1.device == h->device;
}

ugks_status copy_W_in(ugks_ctx* h, const double* W, cudaMemcpyKind kind) {
  const Params& P = h->P;
  if (kind == cudaMemcpyDeviceToDevice && own_rows(h, W, 4 * sizeof(double) * P.nx * P.ny)) {
    k_copy_W<<<(P.nx * P.ny + 127) / 128, 128, 0, h->stream>>>(P, h->W[h->cur], h->nwe, const_cast<double*>(W), false);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  for (int c = 0; c < 4; c++) {
    double* dst = h->W[h->cur] + (size_t)c * h->nwe + wcell(P, 0, 0);
    CK(cudaMemcpy2DAsync(dst, P.wx * sizeof(double), W + (size_t)c * P.nx * P.ny, P.nx * sizeof(double),
                         P.nx * sizeof(double), P.ny, kind, h->stream));
  }
  return UGKS_OK;
}

ugks_status copy_W_out(ugks_ctx* h, double* W, cudaMemcpyKind kind) {
  const Params& P = h->P;
  if (kind == cudaMemcpyDeviceToDevice && own_rows(h, W, 4 * sizeof(double) * P.nx * P.ny)) {
    k_copy_W<<<(P.nx * P.ny + 127) / 128, 128, 0, h->stream>>>(P, h->W[h->cur], h->nwe, W, true);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  for (int c = 0; c < 4; c++) {
    const double* src = h->W[h->cur] + (size_t)c * h->nwe + wcell(P, 0, 0);
    CK(cudaMemcpy2DAsync(W + (size_t)c * P.nx * P.ny, P.nx * sizeof(double), src, P.wx * sizeof(double),
                         P.nx * sizeof(double), P.ny, kind, h->stream));
  }
  return UGKS_OK;
}

// Device address of `bytes` bytes of host memory at p that kernels can read and write
// directly: page-locked or registered host memory (on this GB300 node reached over
// NVLink-C2C), whose first and last byte map into one contiguous device range.  nullptr for
// pageable memory, which goes through the staging buffer instead.
void* device_view(const void* p, size_t bytes) {
  cudaPointerAttributes a0, a1;
  if (cudaPointerGetAttributes(&a0, p) != cudaSuccess ||
      cudaPointerGetAttributes(&a1, static_cast<const char*>(p) + bytes - 1) != cudaSuccess) {
    cudaGetLastError();  // clear the error of an unknown pointer
    return nullptr;
  }
  if (a0.type != cudaMemoryTypeHost || a1.type != cudaMemoryTypeHost || !a0.devicePointer ||
      static_cast<char*>(a1.devicePointer) != static_cast<char*>(a0.devicePointer) + bytes - 1)
    return nullptr;
  return a0.devicePointer;
}

ugks_status copy_f_in(ugks_ctx* h, const double* f, bool from_host) {
  const Params& P = h->P;
  const size_t row_d = (size_t)P.nx * P.nq * 2 * sizeof(double);
  const cudaMemcpyKind kind = from_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  if (h->prec == UGKS_FP64 && !from_host && own_rows(h, f, row_d * P.ny)) {
    k_copy_f<<<kConvBlocks, 256, 0, h->stream>>>(P, static_cast<double2*>(h->f[h->cur]), const_cast<double*>(f), false);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  if (h->prec == UGKS_FP64) {
    char* dst = static_cast<char*>(h->f[h->cur]) + ((size_t)2 * P.ex + 2) * P.nq * h->t2;
    CK(cudaMemcpy2DAsync(dst, (size_t)P.ex * P.nq * h->t2, f, row_d, row_d, P.ny, kind, h->stream));
    return UGKS_OK;
  }
  if (h->prec == UGKS_DF64) {
    // host rows pass through the slope buffer (32 B per velocity-cell >= 16 B of FP64 rows)
    const double* src = f;
    if (from_host) {
      CK(cudaMemcpyAsync(h->slopes, f, row_d * P.ny, cudaMemcpyHostToDevice, h->stream));
      src = reinterpret_cast<const double*>(h->slopes);
    }
    k_rows_to_df<<<kConvBlocks, 256, 0, h->stream>>>(src, static_cast<DF4*>(h->f[h->cur]), P, 0, P.ny);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  float4* dst = static_cast<float4*>(h->f[h->cur]);
  const double* src = from_host ? static_cast<const double*>(device_view(f, row_d * P.ny)) : f;
  if (src) {  // device memory, or host memory the conversion kernel reads in place
    if (aligned16(src))
      k_rows_to_f32<true><<<kConvBlocks, 256, 0, h->stream>>>(src, dst, P, h->grefd, 0, P.ny);
    else
      k_rows_to_f32<false><<<kConvBlocks, 256, 0, h->stream>>>(src, dst, P, h->grefd, 0, P.ny);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  // two staging halves: the copy of chunk k+1 (copy stream) overlaps the conversion of
  // chunk k (library stream)
  const size_t half = h->stage_bytes / 2;
  const int rows = (int)(half / row_d);
  int k = 0;
  for (int j0 = 0; j0 < P.ny; j0 += rows, k++) {
    const int nr = (j0 + rows <= P.ny) ? rows : P.ny - j0;
    const int b = k & 1;
    double* buf = h->stage + b * (half / sizeof(double));
    CK(cudaStreamWaitEvent(h->xstream, h->ev_free[b], 0));
    CK(cudaMemcpyAsync(buf, f + (size_t)j0 * P.nx * P.nq * 2, nr * row_d, cudaMemcpyHostToDevice, h->xstream));
    CK(cudaEventRecord(h->ev_copied[b], h->xstream));
    CK(cudaStreamWaitEvent(h->stream, h->ev_copied[b], 0));
    k_rows_to_f32<true><<<kConvBlocks, 256, 0, h->stream>>>(buf, dst, P, h->grefd, j0, nr);
    CK(cudaGetLastError());
    CK(cudaEventRecord(h->ev_free[b], h->stream));
  }
  return UGKS_OK;
}

ugks_status copy_f_out(ugks_ctx* h, double* f, bool to_host) {
  const Params& P = h->P;
  const size_t row_d = (size_t)P.nx * P.nq * 2 * sizeof(double);
  const cudaMemcpyKind kind = to_host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  if (h->prec == UGKS_FP64 && !to_host && own_rows(h, f, row_d * P.ny)) {
    k_copy_f<<<kConvBlocks, 256, 0, h->stream>>>(P, static_cast<double2*>(h->f[h->cur]), f, true);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  if (h->prec == UGKS_FP64) {
    const char* src = static_cast<const char*>(h->f[h->cur]) + ((size_t)2 * P.ex + 2) * P.nq * h->t2;
    CK(cudaMemcpy2DAsync(f, row_d, src, (size_t)P.ex * P.nq * h->t2, row_d, P.ny, kind, h->stream));
    return UGKS_OK;
  }
  if (h->prec == UGKS_DF64) {
    double* dst = to_host ? reinterpret_cast<double*>(h->slopes) : f;
    k_df_to_rows<<<kConvBlocks, 256, 0, h->stream>>>(static_cast<const DF4*>(h->f[h->cur]), dst, P, 0, P.ny);
    CK(cudaGetLastError());
    if (to_host) CK(cudaMemcpyAsync(f, dst, row_d * P.ny, cudaMemcpyDeviceToHost, h->stream));
    return UGKS_OK;
  }
  const float4* src = static_cast<const float4*>(h->f[h->cur]);
  double* dst = to_host ? static_cast<double*>(device_view(f, row_d * P.ny)) : f;
  if (dst) {  // device memory, or host memory the conversion kernel writes in place
    if (aligned16(dst))
      k_f32_to_rows<true><<<kConvBlocks, 256, 0, h->stream>>>(src, dst, P, h->grefd, 0, P.ny);
    else
      k_f32_to_rows<false><<<kConvBlocks, 256, 0, h->stream>>>(src, dst, P, h->grefd, 0, P.ny);
    CK(cudaGetLastError());
    return UGKS_OK;
  }
  // conversion of chunk k+1 (library stream) overlaps the copy of chunk k (copy stream);
  // the caller synchronises the library stream, which waits for the last copy
  const size_t half = h->stage_bytes / 2;
  const int rows = (int)(half / row_d);
  int k = 0;
  for (int j0 = 0; j0 < P.ny; j0 += rows, k++) {
    const int nr = (j0 + rows <= P.ny) ? rows : P.ny - j0;
    const int b = k & 1;
    double* buf = h->stage + b * (half / sizeof(double));
    CK(cudaStreamWaitEvent(h->stream, h->ev_free[b], 0));
    k_f32_to_rows<true><<<kConvBlocks, 256, 0, h->stream>>>(src, buf, P, h->grefd, j0, nr);
    CK(cudaGetLastError());
    CK(cudaEventRecord(h->ev_copied[b], h->stream));
    CK(cudaStreamWaitEvent(h->xstream, h->ev_copied[b], 0));
    CK(cudaMemcpyAsync(f + (size_t)j0 * P.nx * P.nq * 2, buf, nr * row_d, cudaMemcpyDeviceToHost, h->xstream));
    CK(cudaEventRecord(h->ev_free[b], h->xstream));
  }
  for (int b = 0; b < 2; b++) CK(cudaStreamWaitEvent(h->stream, h->ev_free[b], 0));
  return UGKS_OK;
}

ugks_status check_err(ugks_ctx* h) {
  int e = 0;
  CK(cudaMemcpyAsync(&e, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (e & 2) return fail(h, UGKS_ETIMEOUT, "a bounded wait of the update walk for its record copies gave up");
  if (e) return fail(h, UGKS_ENUMERIC, "numerical failure: rho <= 0, T <= 0 or NaN in a cell");
  return UGKS_OK;
}

}  // namespace

// -------------------------------------------------------------------------------------
// Scratch for ugks_step_noalloc: a fixed device array, no allocation at call time.
// -------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[UGKS_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[kMaxDevices] = {nullptr};

// Device address of the scratch array on the current device.  Outside stream capture the
// address is looked up on every call, so that a context that was torn down and created again
// (cudaDeviceReset, or a host framework recreating the primary context) never leaves a stale
// address behind: the module is loaded again there and the array may move.  While `st` is
// being captured the lookup (which may load the module) is not made, and the address of the
// last call outside capture on this device is used; with none the call fails.
cudaError_t noalloc_scratch(cudaStream_t st, void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();  // e.g. the legacy stream while another stream captures globally
    cs = cudaStreamCaptureStatusActive;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (cs == cudaStreamCaptureStatusNone) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = p;
  } else if (!g_noalloc_ptr[dev]) {
    return cudaErrorStreamCaptureUnsupported;
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

}  // namespace

extern "C" {

ugks_status ugks_step_noalloc(const ugks_config* cfg, const double* f_in, const double* W_in,
                              double* f_out, double* W_out, void* cuda_stream) {
  const char* bad = validate(cfg);
  if (!bad && shakhov_pr(cfg) != 1.0) bad = "the Shakhov model (pr != 1) needs ugks_create";
  if (bad || !f_in || !W_in || !f_out || !W_out || cfg->precision != UGKS_FP64) {
    fprintf(stderr, "ugks_step_noalloc: %s\n",
            bad ? bad : (cfg->precision != UGKS_FP64 ? "precision must be UGKS_FP64" : "NULL buffer"));
    return UGKS_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // host-side setup in fixed-size arrays (no heap)
  Params P;
  memset(&P, 0, sizeof P);
  P.nx = cfg->nx; P.ny = cfg->ny; P.nu = cfg->nu; P.nv = cfg->nv; P.nq = cfg->nu * cfg->nv;
  P.K = cfg->K;
  P.ex = cfg->nx + 4;
  P.wx = cfg->nx + 2;
  P.dx = cfg->lx / cfg->nx;
  P.dy = cfg->ly / cfg->ny;
  double grid[4 * kMaxAxis + 5 * kMaxAxis];  // u, v, wu, wv, then [5][nv] wv v^n
  double* hu = grid;
  double* hv = grid + P.nu;
  double* hwu = grid + P.nu + P.nv;
  double* hwv = grid + 2 * P.nu + P.nv;
  auto fill_axis = [](int n, double lo, double hi, double* x, double* w) {
    if (n == 1) { x[0] = 0.5 * (lo + hi); w[0] = 1.0; return; }
    const double d = (hi - lo) / (n - 1), c = 0.5 * (lo + hi);
    for (int k = 0; k < n; k++) {
      x[k] = c + (k - 0.5 * (n - 1)) * d;
      w[k] = (k == 0 || k == n - 1) ? 0.5 * d : d;
    }
  };
  fill_axis(P.nu, cfg->umin, cfg->umax, hu, hwu);
  fill_axis(P.nv, cfg->vmin, cfg->vmax, hv, hwv);
  double* hwn = grid + 2 * (P.nu + P.nv);
  for (int n = 0; n < 5; n++)
    for (int m = 0; m < P.nv; m++) hwn[n * P.nv + m] = hwv[m] * std::pow(hv[m], n);
  const int ngrid = 2 * (P.nu + P.nv) + 5 * P.nv;  // doubles in the grid block
  double um = 0, vm = 0;
  for (int k = 0; k < P.nu; k++) um = fmax(um, fabs(hu[k]));
  for (int m = 0; m < P.nv; m++) vm = fmax(vm, fabs(hv[m]));
  if (cfg->dt > 0) P.dt = cfg->dt;
  else {
    if (!(um / P.dx + vm / P.dy > 0)) return UGKS_EINVAL;
    P.dt = cfg->cfl / (um / P.dx + vm / P.dy);
  }
  const double a = cfg->alpha, om = cfg->omega;
  P.mu_ref = 5.0 * (a + 1.0) * (a + 2.0) * sqrt(M_PI) / (4.0 * a * (5.0 - 2.0 * om) * (7.0 - 2.0 * om)) * cfg->kn;
  P.omega = om;
  P.omega_half = om == 0.5;
  set_derived(P);
  for (int sd = 0; sd < 4; sd++) {
    P.bc_kind[sd] = cfg->bc[sd].kind;
    P.bc_rho[sd] = cfg->bc[sd].rho;
    P.bc_T[sd] = cfg->bc[sd].T;
    P.bc_U[sd] = cfg->bc[sd].U;
    if (cfg->bc[sd].kind != UGKS_BC_WALL) continue;
    const double lam = 1.0 / cfg->bc[sd].T, Uw = cfg->bc[sd].U;
    for (int m = 0; m < P.nv; m++)
      for (int k = 0; k < P.nu; k++) {
        const double u = hu[k], v = hv[m], w = hwu[k] * hwv[m];
        const double un = sd < 2 ? u : v, ut = sd < 2 ? v : u;
        const bool outgoing = (sd == 0 || sd == 2) ? un > 0 : un < 0;
        if (!outgoing) continue;
        const double gh = lam / M_PI * exp(-lam * ((ut - Uw) * (ut - Uw) + un * un));
        const double gb = P.K / (2.0 * lam) * gh;
        P.wall_mom[sd][0] += w * un * gh;
        P.wall_mom[sd][1] += w * un * u * gh;
        P.wall_mom[sd][2] += w * un * v * gh;
        P.wall_mom[sd][3] += w * un * (0.5 * (u * u + v * v) * gh + 0.5 * gb);
      }
  }
  P.m_pos = P.nv;
  for (int m = 0; m < P.nv; m++)
    if (hv[m] > 0) { P.m_pos = m; break; }
  for (int m = 0; m < P.nv; m++)
    if (hv[m] < 0) P.m_neg = m + 1;

  // carve the scratch array
  const int nx = P.nx, ny = P.ny, nq = P.nq, nc = nx * ny;
  const int nwe = (nx + 2) * (ny + 2), nfx = (nx + 1) * ny, nfy = nx * (ny + 1);
  const int nrb = (nc + 127) / 128;
  const size_t fb = (size_t)(nx + 4) * (ny + 4) * nq * sizeof(double2);
  size_t off[16], need = 0;
  const size_t sz[13] = {fb, fb, 4 * sizeof(double) * nwe, 4 * sizeof(double) * nwe,
                         sizeof(double) * kNSum * (size_t)nwe, sizeof(FaceRec) * (size_t)nfx,
                         sizeof(FaceRec) * (size_t)nfy, sizeof(double) * 4 * (size_t)nfx,
                         sizeof(double) * 4 * (size_t)nfy, sizeof(double) * (size_t)(nfx + nfy),
                         sizeof(CellRec) * (size_t)nc, sizeof(double) * 8 * (size_t)nrb,
                         sizeof(double) * ngrid + sizeof(int)};
  for (int b = 0; b < 13; b++) { off[b] = need; need += align256(sz[b]); }
  if (need > UGKS_NOALLOC_SCRATCH_BYTES) {
    fprintf(stderr, "ugks_step_noalloc: problem needs %zu bytes of scratch, the fixed maximum is %u\n",
            need, (unsigned)UGKS_NOALLOC_SCRATCH_BYTES);
    return UGKS_EINVAL;
  }
  void* base = nullptr;
  cudaError_t e = noalloc_scratch(st, &base);
  if (e != cudaSuccess) {
    fprintf(stderr, "ugks_step_noalloc: scratch address: %s\n", cudaGetErrorString(e));
    return UGKS_ECUDA;
  }
  char* sb = static_cast<char*>(base);
  double2* f0 = reinterpret_cast<double2*>(sb + off[0]);
  double2* f1 = reinterpret_cast<double2*>(sb + off[1]);
  double* W0 = reinterpret_cast<double*>(sb + off[2]);
  double* W1 = reinterpret_cast<double*>(sb + off[3]);
  double* sums = reinterpret_cast<double*>(sb + off[4]);
  FaceRec* fxr = reinterpret_cast<FaceRec*>(sb + off[5]);
  FaceRec* fyr = reinterpret_cast<FaceRec*>(sb + off[6]);
  double* Fx = reinterpret_cast<double*>(sb + off[7]);
  double* Fy = reinterpret_cast<double*>(sb + off[8]);
  double* mt4 = reinterpret_cast<double*>(sb + off[9]);
  CellRec* cells = reinterpret_cast<CellRec*>(sb + off[10]);
  double* rpart = reinterpret_cast<double*>(sb + off[11]);
  double* dgrid = reinterpret_cast<double*>(sb + off[12]);
  int* err = reinterpret_cast<int*>(dgrid + ngrid);
  P.mvd = dgrid + 2 * (P.nu + P.nv);
  P.u = dgrid;
  P.v = dgrid + P.nu;
  P.wu = dgrid + P.nu + P.nv;
  P.wv = dgrid + 2 * P.nu + P.nv;

#define NA_CK(call)                                                                     \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) {                                                            \
      fprintf(stderr, "ugks_step_noalloc: %s: %s\n", #call, cudaGetErrorString(e_));   \
      return UGKS_ECUDA;                                                                \
    }                                                                                   \
  } while (0)
  NA_CK(cudaMemcpyAsync(dgrid, grid, sizeof(double) * ngrid, cudaMemcpyHostToDevice, st));
  NA_CK(cudaMemsetAsync(err, 0, sizeof(int), st));
  // the previous call's contents stay in the array: clear the f ring so every cell the
  // kernels read is defined
  NA_CK(cudaMemsetAsync(f0, 0, fb, st));
  NA_CK(cudaMemsetAsync(W0, 0, 4 * sizeof(double) * nwe, st));
  const size_t row = (size_t)nx * nq * sizeof(double2);
  NA_CK(cudaMemcpy2DAsync(reinterpret_cast<char*>(f0) + ((size_t)2 * P.ex + 2) * nq * sizeof(double2),
                          (size_t)P.ex * nq * sizeof(double2), f_in, row, row, ny, cudaMemcpyDeviceToDevice, st));
  for (int c = 0; c < 4; c++)
    NA_CK(cudaMemcpy2DAsync(W0 + (size_t)c * nwe + wcell(P, 0, 0), P.wx * sizeof(double),
                            W_in + (size_t)c * nc, nx * sizeof(double), nx * sizeof(double), ny,
                            cudaMemcpyDeviceToDevice, st));
  NA_CK(set_smem_limits_fp64(P.nv));
  k_ghost<double2><<<ghost_cells(P), 128, 0, st>>>(P, f0, W0, nwe);
  k_sums<double, double2><<<(nwe + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock,
                            smem_sums<double>(P.nv), st>>>(P, f0, sums, nullptr);
  k_faces<kRecF64, false><<<(nfx + nfy + 127) / 128, 128, 0, st>>>(P, sums, W0, nwe, fxr, fyr, Fx, Fy, mt4);
  k_cells<<<nrb, 128, 0, st>>>(P, W0, W1, nwe, Fx, Fy, cells, rpart, err, nullptr, mt4);
  // slopes are formed again in the update kernel: the scratch array holds no slope buffer
  k_update<double, double2><<<(nc + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock,
                              smem_update<double>(P.nv), st>>>(P, f0, f1, fxr, fyr, cells);
  NA_CK(cudaGetLastError());
  NA_CK(cudaMemcpy2DAsync(f_out, row, reinterpret_cast<char*>(f1) + ((size_t)2 * P.ex + 2) * nq * sizeof(double2),
                          (size_t)P.ex * nq * sizeof(double2), row, ny, cudaMemcpyDeviceToDevice, st));
  for (int c = 0; c < 4; c++)
    NA_CK(cudaMemcpy2DAsync(W_out + (size_t)c * nc, nx * sizeof(double), W1 + (size_t)c * nwe + wcell(P, 0, 0),
                            P.wx * sizeof(double), nx * sizeof(double), ny, cudaMemcpyDeviceToDevice, st));
  int herr = 0;
  NA_CK(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  NA_CK(cudaStreamSynchronize(st));
#undef NA_CK
  if (herr) {
    fprintf(stderr, "ugks_step_noalloc: numerical failure (rho <= 0, T <= 0 or NaN)\n");
    return UGKS_ENUMERIC;
  }
  return UGKS_OK;
}

// -------------------------------------------------------------------------------------
// FP64 arithmetic rate of the device (the roofline of the FP64 form's kernels): every
// thread runs 8 independent chains of dependent FP64 fused multiply-adds.
// -------------------------------------------------------------------------------------
__global__ void k_fp64_rate(double* out, int iters, double a, double b) {
  double x[8];
#pragma unroll
  for (int k = 0; k < 8; k++) x[k] = threadIdx.x * 1e-3 + k;
  for (int i = 0; i < iters; i++) {
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = fma(x[k], a, b);
  }
  double r = 0.0;
#pragma unroll
  for (int k = 0; k < 8; k++) r += x[k];
  if (r == 1.2345e300) out[0] = r;  // keeps the chains live; never true for these inputs
}

ugks_status ugks_fp64_rate(void* cuda_stream, double* gflops) {
  if (!gflops) return UGKS_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return UGKS_ECUDA;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return UGKS_ECUDA;
  if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return UGKS_ECUDA; }
  const int blocks = sms * 8, threads = 256, iters = 4096;
  cudaError_t e = cudaSuccess;
  float best = 1e30f;
  for (int rep = 0; rep < 4 && e == cudaSuccess; rep++) {  // first launch: warm-up
    e = cudaEventRecord(e0, st);
    if (e == cudaSuccess) {
      k_fp64_rate<<<blocks, threads, 0, st>>>(nullptr, iters, 0.999999, 1e-7);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess && rep > 0 && ms < best) best = ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e != cudaSuccess) return UGKS_ECUDA;
  *gflops = 2.0 * 8.0 * iters * (double)blocks * threads / (best * 1e-3) / 1e9;
  return UGKS_OK;
}

ugks_status ugks_create(const ugks_config* cfg, void* cuda_stream, ugks_handle* out) {
  if (!out) return UGKS_EINVAL;
  *out = nullptr;
  const char* bad = validate(cfg);
  if (bad) {
    fprintf(stderr, "ugks_create: %s\n", bad);
    return UGKS_EINVAL;
  }
  ugks_ctx* h = new ugks_ctx();
  h->cfg = *cfg;
  h->stream = static_cast<cudaStream_t>(cuda_stream);
  h->prec = cfg->precision;
  cudaGetDevice(&h->device);
  h->t2 = sizeof(double2);  // FP64 form (the FP32-f form stores float4 slots of two velocities)
  Params& P = h->P;
  memset(&P, 0, sizeof P);
  P.nx = cfg->nx; P.ny = cfg->ny; P.nu = cfg->nu; P.nv = cfg->nv; P.nq = cfg->nu * cfg->nv;
  P.K = cfg->K;
  P.ex = cfg->nx + 4;
  P.wx = cfg->nx + 2;
  P.dx = cfg->lx / cfg->nx;
  P.dy = cfg->ly / cfg->ny;
  axis(cfg->nu, cfg->umin, cfg->umax, h->hu, h->hwu);
  axis(cfg->nv, cfg->vmin, cfg->vmax, h->hv, h->hwv);
  double um = 0, vm = 0;
  for (double x : h->hu) um = fmax(um, fabs(x));
  for (double x : h->hv) vm = fmax(vm, fabs(x));
  if (cfg->dt > 0) P.dt = cfg->dt;
  else {
    if (!(um / P.dx + vm / P.dy > 0)) { delete h; return UGKS_EINVAL; }
    P.dt = cfg->cfl / (um / P.dx + vm / P.dy);
  }
  const double a = cfg->alpha, om = cfg->omega;
  P.mu_ref = 5.0 * (a + 1.0) * (a + 2.0) * sqrt(M_PI) / (4.0 * a * (5.0 - 2.0 * om) * (7.0 - 2.0 * om)) * cfg->kn;
  P.omega = om;
  P.omega_half = om == 0.5;
  P.pr = shakhov_pr(cfg);
  P.shk = P.pr != 1.0;
  P.shk_c = (1.0 - P.pr) * 4.0 / (P.K + 4.0);
  set_derived(P);
  P.f_tdx = (float)(2.0 / P.dx);
  P.f_tdy = (float)(2.0 / P.dy);
  P.f_idx = (float)(1.0 / P.dx);
  P.f_idy = (float)(1.0 / P.dy);
  P.f_dt = (float)P.dt;
  P.walk_wait_polls = kWalkWaitPolls;
  for (int s = 0; s < 4; s++) {
    P.bc_kind[s] = cfg->bc[s].kind;
    P.bc_rho[s] = cfg->bc[s].rho;
    P.bc_T[s] = cfg->bc[s].T;
    P.bc_U[s] = cfg->bc[s].U;
    if (cfg->bc[s].kind != UGKS_BC_WALL) continue;
    // discrete moments of the outgoing wall Maxwellian (rho = 1), natural frame
    const double lam = 1.0 / cfg->bc[s].T, Uw = cfg->bc[s].U;
    double m[4] = {0, 0, 0, 0};
    for (int mm = 0; mm < P.nv; mm++)
      for (int k = 0; k < P.nu; k++) {
        const double u = h->hu[k], v = h->hv[mm], w = h->hwu[k] * h->hwv[mm];
        const double un = s < 2 ? u : v, ut = s < 2 ? v : u;
        const bool outgoing = (s == 0 || s == 2) ? un > 0 : un < 0;
        if (!outgoing) continue;
        const double gh = lam / M_PI * exp(-lam * ((ut - Uw) * (ut - Uw) + un * un));
        const double gb = P.K / (2.0 * lam) * gh;
        m[0] += w * un * gh;
        m[1] += w * un * u * gh;
        m[2] += w * un * v * gh;
        m[3] += w * un * (0.5 * (u * u + v * v) * gh + 0.5 * gb);
      }
    for (int c = 0; c < 4; c++) P.wall_mom[s][c] = m[c];
  }

  P.m_pos = P.nv;
  for (int m = 0; m < P.nv; m++)
    if (h->hv[m] > 0) { P.m_pos = m; break; }
  P.m_neg = 0;
  for (int m = 0; m < P.nv; m++)
    if (h->hv[m] < 0) P.m_neg = m + 1;
  P.k_pos = P.nu;
  for (int k = 0; k < P.nu; k++)
    if (h->hu[k] > 0) { P.k_pos = k; break; }
  for (int k = 0; k < P.nu; k++)
    if (h->hu[k] < 0) P.k_neg = k + 1;
  {
    const std::pair<int, int> rp = f32_row_pairs(P.nv, cfg->vmin, cfg->vmax);
    P.pr_neg = rp.first;
    P.pr_all = rp.second;
    P.fs = P.pr_all * P.nu;
  }
  // FP32 walk: chunks of 32 slots within each half of the v axis
  h->nchunk_neg = (P.pr_neg * P.nu + 31) / 32;
  h->nchunk_pos = ((P.pr_all - P.pr_neg) * P.nu + 31) / 32;
  std::vector<float4> gref_host;
  std::vector<double2> grefd_host;
  if (h->prec == UGKS_FP32F) {
    double rr = cfg->ref_rho, rU = cfg->ref_U, rV = cfg->ref_V, rT = cfg->ref_T;
    if (!(rT > 0) || !(rr > 0)) { rr = 1.0; rU = 0.0; rV = 0.0; rT = 1.0; }
    P.use_ref = 1;
    P.ref_lam = 1.0 / rT;
    P.ref_G = rr * P.ref_lam / M_PI;
    P.ref_U = rU;
    P.ref_V = rV;
    P.ref_bf = P.K / (2.0 * P.ref_lam);
    const double kLog2e = 1.4426950408889634;
    P.ref_E[0] = std::log2(P.ref_G) - P.ref_lam * (rU * rU + rV * rV) * kLog2e;
    P.ref_E[1] = 2.0 * P.ref_lam * rU * kLog2e;
    P.ref_E[2] = 2.0 * P.ref_lam * rV * kLog2e;
    P.ref_E[3] = -P.ref_lam * kLog2e;
    P.ref_iG = 1.0 / P.ref_G;
    P.ref_E0u = -P.ref_lam * (rU * rU + rV * rV) * kLog2e;
    grefd_host.resize((size_t)P.nq);
    for (int m = 0; m < P.nv; m++)
      for (int k = 0; k < P.nu; k++) {
        const double u = h->hu[k], v = h->hv[m], w = h->hwu[k] * h->hwv[m];
        double gh, gb;
        ref_maxwellian(P, u, v, gh, gb);
        grefd_host[(size_t)m * P.nu + k] = make_double2(gh, gb);
        const double psi[4] = {gh, u * gh, v * gh, 0.5 * (u * u + v * v) * gh + 0.5 * gb};
        const double hs[4] = {u > 0 ? 1.0 : (u < 0 ? 0.0 : 0.5), u < 0 ? 1.0 : (u > 0 ? 0.0 : 0.5),
                              v > 0 ? 1.0 : (v < 0 ? 0.0 : 0.5), v < 0 ? 1.0 : (v > 0 ? 0.0 : 0.5)};
        const double un[4] = {u, u, v, v};
        for (int sd = 0; sd < 4; sd++)
          for (int c = 0; c < 4; c++) {
            P.refsum[sd][kOffW0 + c] += hs[sd] * w * psi[c];
            P.refsum[sd][kOffSf + c] += hs[sd] * w * un[sd] * psi[c];
          }
        if (P.shk) {  // Shakhov: raw heat-flux moments of g_ref per side and over the cell
          const double mh[10] = {u * u, u * v, v * v, u * u * u, u * u * v, u * v * v, v * v * v, 0, 0, 0};
          for (int sd = 0; sd < 4; sd++) {
            for (int t = 0; t < 7; t++) P.refheat[sd][t] += hs[sd] * w * mh[t] * gh;
            P.refheat[sd][7] += hs[sd] * w * gb;
            P.refheat[sd][8] += hs[sd] * w * u * gb;
            P.refheat[sd][9] += hs[sd] * w * v * gb;
          }
          const double mc[10] = {1.0, u, v, u * u, u * v, v * v, u * u * u, u * u * v, u * v * v, v * v * v};
          for (int t = 0; t < 10; t++) P.refheat[4][t] += w * mc[t] * gh;
          P.refheatC[0] += w * gb;
          P.refheatC[1] += w * u * gb;
          P.refheatC[2] += w * v * gb;
        }
      }
    for (int c = 0; c < 4; c++) {
      P.refpair[0][c] = P.refsum[kSumE / 16][kOffW0 + c] + P.refsum[kSumW / 16][kOffW0 + c];
      P.refpair[0][4 + c] = P.refsum[kSumE / 16][kOffSf + c] + P.refsum[kSumW / 16][kOffSf + c];
      P.refpair[1][c] = P.refsum[kSumN / 16][kOffW0 + c] + P.refsum[kSumS / 16][kOffW0 + c];
      P.refpair[1][4 + c] = P.refsum[kSumN / 16][kOffSf + c] + P.refsum[kSumS / 16][kOffSf + c];
    }
    for (int ax = 0; ax < 2; ax++)
      for (int t = 0; t < 10; t++) P.refheatpair[ax][t] = P.refheat[2 * ax][t] + P.refheat[2 * ax + 1][t];
    // g_ref per slot of the paired-row layout (h, h', b, b')
    gref_host.resize((size_t)P.fs);
    for (int pr = 0; pr < P.pr_all; pr++)
      for (int k = 0; k < P.nu; k++) {
        const double2 g0 = grefd_host[(size_t)prow(P, 2 * pr) * P.nu + k];
        const double2 g1 = grefd_host[(size_t)prow(P, 2 * pr + 1) * P.nu + k];
        gref_host[(size_t)pr * P.nu + k] = make_float4((float)g0.x, (float)g1.x, (float)g0.y, (float)g1.y);
      }
  }

  cudaError_t e;
  auto alloc = [&](void** p, size_t n) -> bool {
    e = cudaMalloc(p, n);
    if (e != cudaSuccess) return false;
    h->bytes += n;
    return true;
  };
  h->fcells = (size_t)(P.nx + 4) * (P.ny + 4);
  h->nwe = (P.nx + 2) * (P.ny + 2);
  const size_t fbytes = h->fcells * (h->prec == UGKS_FP32F ? P.fs * sizeof(float4) : P.nq * sizeof(double2));
  const int nfx = (P.nx + 1) * P.ny, nfy = P.nx * (P.ny + 1), nc = P.nx * P.ny;
  h->face_block = small_block(nfx + nfy);
  h->cell_block = small_block(nc);
  h->nrblocks = (nc + h->cell_block - 1) / h->cell_block;
  const bool f32 = h->prec == UGKS_FP32F, dfm = h->prec == UGKS_DF64;
  bool ok = alloc(&h->f[0], fbytes) && alloc(&h->f[1], fbytes) &&
            alloc((void**)&h->W[0], 4 * sizeof(double) * h->nwe) &&
            alloc((void**)&h->W[1], 4 * sizeof(double) * h->nwe) &&
            alloc((void**)&h->sums, sizeof(double) * sums_per_cell(cfg) * (size_t)h->nwe) &&
            (!P.shk || alloc((void**)&h->hs, sizeof(double) * kNHeat * (size_t)h->nwe)) &&
            (f32 || alloc((void**)&h->slopes, sizeof(double2) * 2 * (size_t)h->nwe * P.nq)) &&
            (f32 || alloc((void**)&h->xflux, sizeof(double2) * (size_t)(nfx + nfy) * P.nq)) &&
            (f32 ? alloc((void**)&h->fxf, sizeof(FaceRecF) * (size_t)nfx)
                 : dfm ? alloc((void**)&h->fxd, sizeof(FaceRecD) * (size_t)nfx)
                       : alloc((void**)&h->fxr, sizeof(FaceRec) * (size_t)nfx)) &&
            (f32 ? alloc((void**)&h->fyf, sizeof(FaceRecF) * (size_t)nfy)
                 : dfm ? alloc((void**)&h->fyd, sizeof(FaceRecD) * (size_t)nfy)
                       : alloc((void**)&h->fyr, sizeof(FaceRec) * (size_t)nfy)) &&
            alloc((void**)&h->Fx, sizeof(double) * 4 * (size_t)nfx) &&
            alloc((void**)&h->Fy, sizeof(double) * 4 * (size_t)nfy) &&
            alloc((void**)&h->mt4, sizeof(double) * (size_t)(nfx + nfy)) &&
            (!(f32 && P.shk) || alloc((void**)&h->cshk, sizeof(CellShkF) * (size_t)nc)) &&
            (f32 ? alloc((void**)&h->cellf, sizeof(CellRecF) * (size_t)nc)
                 : dfm ? alloc((void**)&h->celld, sizeof(CellRecD) * (size_t)nc)
                       : alloc((void**)&h->cells, sizeof(CellRec) * (size_t)nc)) &&
            (!dfm || alloc((void**)&h->gdf, sizeof(float2) * (8 * (size_t)P.nu + 8 * (size_t)P.nv))) &&
            alloc((void**)&h->rpart, sizeof(double) * 8 * (size_t)h->nrblocks) &&
            alloc((void**)&h->err, sizeof(int)) &&
            alloc((void**)&h->d_grid, sizeof(double) * (8 * (size_t)P.nu + 9 * (size_t)P.nv));
  if (ok && h->prec == UGKS_FP32F) {
    const size_t row_d = (size_t)P.nx * P.nq * 2 * sizeof(double);
    h->stage_bytes = 2 * stage_half_bytes(row_d, P.ny);
    ok = alloc((void**)&h->stage, h->stage_bytes) && alloc((void**)&h->gref4, sizeof(float4) * (size_t)P.fs) &&
         alloc((void**)&h->grefd, sizeof(double2) * (size_t)P.nq) &&
         alloc((void**)&h->ftab, sizeof(float) * (12 * ((size_t)P.pr_all + 1) + 14 * (size_t)P.nu));
    if (ok) {
      e = cudaStreamCreateWithFlags(&h->xstream, cudaStreamNonBlocking);
      for (int b = 0; b < 2 && e == cudaSuccess; b++) {
        e = cudaEventCreateWithFlags(&h->ev_copied[b], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_free[b], cudaEventDisableTiming);
      }
      ok = e == cudaSuccess;
    }
  }
  if (!ok) {
    ugks_destroy(h);
    fprintf(stderr, "ugks_create: device allocation failed: %s\n", cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? UGKS_ENOMEM : UGKS_ECUDA;
  }
  std::vector<double> grid;
  grid.insert(grid.end(), h->hu.begin(), h->hu.end());
  grid.insert(grid.end(), h->hv.begin(), h->hv.end());
  grid.insert(grid.end(), h->hwu.begin(), h->hwu.end());
  grid.insert(grid.end(), h->hwv.begin(), h->hwv.end());
  for (int n = 0; n < 5; n++)
    for (int m = 0; m < P.nv; m++) grid.push_back(h->hwv[m] * std::pow(h->hv[m], n));
  // tables of the thread-per-cell sums: [nu][6] w_u u^m (m = 0..4, half at u = 0) and u, [nv][2] v
  // and w_v (half at v = 0)
  std::vector<double> cell_tab;
  for (int k = 0; k < P.nu; k++) {
    for (int n = 0; n < 5; n++)
      cell_tab.push_back((h->hu[k] == 0.0 ? 0.5 : 1.0) * h->hwu[k] * std::pow(h->hu[k], n));
    cell_tab.push_back(h->hu[k]);
  }
  for (int m = 0; m < P.nv; m++) {
    cell_tab.push_back(h->hv[m]);
    cell_tab.push_back((h->hv[m] == 0.0 ? 0.5 : 1.0) * h->hwv[m]);
  }
  grid.insert(grid.end(), cell_tab.begin(), cell_tab.end());
  P.mvd = h->d_grid + 2 * (P.nu + P.nv);
  P.hs = h->hs;
  P.cshk = h->cshk;
  P.u = h->d_grid;
  P.v = h->d_grid + P.nu;
  P.wu = h->d_grid + P.nu + P.nv;
  P.wv = h->d_grid + 2 * P.nu + P.nv;
  P.gref4 = h->gref4;
  P.grefd = h->grefd;
  auto sp = [](double x) {  // a double-FP32 pair
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
  };
  P.df_tdx = sp(2.0 / P.dx);
  P.df_tdy = sp(2.0 / P.dy);
  std::vector<float2> gdf_host;
  if (dfm) {
    // u[nu], wu[nu], v[nv], [5][nv] wv v^n and the mesh constants as double-FP32 pairs
    for (double x : h->hu) gdf_host.push_back(sp(x));
    for (double x : h->hwu) gdf_host.push_back(sp(x));
    for (double x : h->hv) gdf_host.push_back(sp(x));
    for (int n = 0; n < 5; n++)
      for (int m = 0; m < P.nv; m++) gdf_host.push_back(sp(h->hwv[m] * std::pow(h->hv[m], n)));
    for (double x : cell_tab) gdf_host.push_back(sp(x));
    P.gdf = h->gdf;
    P.df_idx = sp(1.0 / P.dx);
    P.df_idy = sp(1.0 / P.dy);
    P.df_dt = sp(P.dt);
  }
  std::vector<float> ftab_host;
  if (h->ftab) {
    // [pr_all][12]: (w0 w0' w1 w1') (w2 w2' w3 w3') (w4 w4' v v'), then [nu][12]: (w0 w0 w1 w1)
    // (w2 w2 w3 w3) (w4 w4 u u) and a row of zeros, then u[nu], wu[nu]
    ftab_host.assign(12 * ((size_t)P.pr_all + 1) + 14 * (size_t)P.nu, 0.f);
    const bool v0 = P.m_pos > P.m_neg;
    for (int pr = 0; pr < P.pr_all; pr++)
      for (int h2 = 0; h2 < 2; h2++) {
        const int r = 2 * pr + h2, m = prow(P, r);
        const bool real = padrow(P, m) == r;  // padded rows repeat a row with zero weight
        const double vv = h->hv[m];
        double w = real ? h->hwv[m] : 0.0;
        if (real && v0 && m == P.m_neg) w *= 0.5;  // v = 0: half to each half of the v axis
        float* t = &ftab_host[12 * (size_t)pr];
        for (int n = 0; n < 5; n++) t[2 * n + h2] = (float)(w * std::pow(vv, n));
        t[10 + h2] = (float)vv;
      }
    for (int k = 0; k < P.nu; k++) {
      float* t = &ftab_host[12 * ((size_t)P.pr_all + k)];
      const double w = h->hu[k] == 0.0 ? 0.5 * h->hwu[k] : h->hwu[k];  // u = 0: half to each half
      for (int n = 0; n < 5; n++) t[2 * n] = t[2 * n + 1] = (float)(w * std::pow(h->hu[k], n));
      t[10] = t[11] = (float)h->hu[k];
      float* uwf = &ftab_host[12 * ((size_t)P.pr_all + P.nu + 1)];
      uwf[k] = (float)h->hu[k];
      uwf[P.nu + k] = (float)h->hwu[k];
    }
    P.pwt = reinterpret_cast<const float4*>(h->ftab);
    P.uwt4 = P.pwt + 3 * (size_t)P.pr_all;
    P.uwf = h->ftab + 12 * ((size_t)P.pr_all + P.nu + 1);
  }
  auto setup = [&]() -> cudaError_t {
    cudaError_t r;
    if ((r = cudaMemcpyAsync(h->d_grid, grid.data(), grid.size() * sizeof(double), cudaMemcpyHostToDevice,
                             h->stream)) != cudaSuccess) return r;
    for (int b = 0; b < 2; b++) {
      if ((r = cudaMemsetAsync(h->f[b], 0, fbytes, h->stream)) != cudaSuccess) return r;
      if ((r = cudaMemsetAsync(h->W[b], 0, 4 * sizeof(double) * h->nwe, h->stream)) != cudaSuccess) return r;
    }
    if ((r = cudaMemsetAsync(h->rpart, 0, sizeof(double) * 8 * h->nrblocks, h->stream)) != cudaSuccess) return r;
    // slopes of cells the sums kernel never forms (wall ghosts, corners) stay zero
    if (h->slopes && (r = cudaMemsetAsync(h->slopes, 0, sizeof(double2) * 2 * (size_t)h->nwe * P.nq,
                                          h->stream)) != cudaSuccess)
      return r;
    if (h->gref4 && (r = cudaMemcpyAsync(h->gref4, gref_host.data(), sizeof(float4) * gref_host.size(),
                                        cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
      return r;
    if (h->ftab && (r = cudaMemcpyAsync(h->ftab, ftab_host.data(), sizeof(float) * ftab_host.size(),
                                        cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
      return r;
    if (h->grefd && (r = cudaMemcpyAsync(h->grefd, grefd_host.data(), sizeof(double2) * grefd_host.size(),
                                         cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
      return r;
    if (h->gdf && (r = cudaMemcpyAsync(h->gdf, gdf_host.data(), sizeof(float2) * gdf_host.size(),
                                       cudaMemcpyHostToDevice, h->stream)) != cudaSuccess)
      return r;
    if ((r = cudaMemsetAsync(h->err, 0, sizeof(int), h->stream)) != cudaSuccess) return r;
    if (h->prec == UGKS_FP64 && (r = set_smem_limits_fp64(P.nv)) != cudaSuccess) return r;
    if (h->prec == UGKS_DF64 && (r = set_smem_limits_df()) != cudaSuccess) return r;
    if ((r = cudaStreamSynchronize(h->stream)) != cudaSuccess) return r;
    return h->prec == UGKS_FP32F ? setup_single_f32(h) : cudaSuccess;
  };
  e = setup();
  if (e != cudaSuccess) {
    fprintf(stderr, "ugks_create: %s\n", cudaGetErrorString(e));
    ugks_destroy(h);
    return UGKS_ECUDA;
  }
  *out = h;
  return UGKS_OK;
}

void ugks_destroy(ugks_handle h) {
  if (!h) return;
  void* ptrs[] = {h->f[0], h->f[1], h->W[0], h->W[1], h->sums, h->slopes, h->xflux, h->fxr, h->fyr, h->Fx, h->Fy,
                  h->cells, h->rpart, h->err, h->d_grid, h->stage, h->gref4, h->grefd, h->fxf, h->fyf,
                  h->cellf, h->mt4, h->ftab, h->d_slot, h->d_work, h->fxd, h->fyd, h->celld, h->gdf,
                  h->hs, h->cshk};
  if (h->stream) cudaStreamSynchronize(h->stream);
  if (h->xstream) {
    cudaStreamSynchronize(h->xstream);
    cudaStreamDestroy(h->xstream);
  }
  for (int b = 0; b < 2; b++) {
    if (h->ev_copied[b]) cudaEventDestroy(h->ev_copied[b]);
    if (h->ev_free[b]) cudaEventDestroy(h->ev_free[b]);
  }
  for (void* p : ptrs)
    if (p) cudaFree(p);
  for (cudaEvent_t e : h->events) cudaEventDestroy(e);
  for (int b = 0; b < 2; b++)
    if (h->graph[b]) cudaGraphExecDestroy(h->graph[b]);
  if (h->cap_stream) {
    cudaStreamSynchronize(h->cap_stream);
    cudaStreamDestroy(h->cap_stream);
  }
  delete h;
}

const char* ugks_last_error(ugks_handle h) { return h ? h->last_error.c_str() : "null handle"; }

size_t ugks_device_bytes(ugks_handle h) { return h ? h->bytes : 0; }

ugks_status ugks_get_grid(ugks_handle h, double* dt, double* u, double* v, double* w) {
  if (!h) return UGKS_EINVAL;
  if (dt) *dt = h->P.dt;
  if (u) memcpy(u, h->hu.data(), sizeof(double) * h->P.nu);
  if (v) memcpy(v, h->hv.data(), sizeof(double) * h->P.nv);
  if (w)
    for (int m = 0; m < h->P.nv; m++)
      for (int k = 0; k < h->P.nu; k++) w[m * h->P.nu + k] = h->hwu[k] * h->hwv[m];
  return UGKS_OK;
}

// A new state clears the failures recorded for the previous one.
ugks_status clear_err(ugks_ctx* h) {
  CK(cudaMemsetAsync(h->err, 0, sizeof(int), h->stream));
  return UGKS_OK;
}

ugks_status ugks_set_state(ugks_handle h, const double* f_host, const double* W_host) {
  if (!h || !f_host || !W_host) return fail(h, UGKS_EINVAL, "set_state: NULL argument");
  if (clear_err(h)) return UGKS_ECUDA;
  ugks_status s = copy_f_in(h, f_host, true);
  if (s) return s;
  s = copy_W_in(h, W_host, cudaMemcpyHostToDevice);
  if (s) return s;
  CK(cudaStreamSynchronize(h->stream));
  return UGKS_OK;
}

ugks_status ugks_set_state_device(ugks_handle h, const double* f_dev, const double* W_dev) {
  if (!h || !f_dev || !W_dev) return fail(h, UGKS_EINVAL, "set_state_device: NULL argument");
  if (clear_err(h)) return UGKS_ECUDA;
  ugks_status s = copy_f_in(h, f_dev, false);
  if (s) return s;
  return copy_W_in(h, W_dev, cudaMemcpyDeviceToDevice);
}

ugks_status ugks_init_maxwellian(ugks_handle h, const double* rho, const double* U, const double* V,
                                 const double* T) {
  if (!h || !rho || !U || !V || !T) return fail(h, UGKS_EINVAL, "init_maxwellian: NULL argument");
  if (clear_err(h)) return UGKS_ECUDA;
  const Params& P = h->P;
  const int nc = P.nx * P.ny;
  for (int c = 0; c < nc; c++)
    if (!(rho[c] > 0) || !(T[c] > 0)) return fail(h, UGKS_EINVAL, "init_maxwellian: rho and T must be > 0");
  double* prim = h->sums;  // scratch: sums holds >= 64 * nc doubles
  const double* src[4] = {rho, U, V, T};
  for (int c = 0; c < 4; c++)
    CK(cudaMemcpyAsync(prim + (size_t)c * nc, src[c], nc * sizeof(double), cudaMemcpyHostToDevice, h->stream));
  if (h->prec == UGKS_FP64)
    k_init_maxwellian<double2><<<nc, 128, 0, h->stream>>>(P, prim, static_cast<double2*>(h->f[h->cur]),
                                                          h->W[h->cur], h->nwe);
  else if (h->prec == UGKS_DF64)
    k_init_maxwellian_df<<<nc, 128, 0, h->stream>>>(P, prim, static_cast<DF4*>(h->f[h->cur]), h->W[h->cur],
                                                    h->nwe);
  else
    k_init_maxwellian_p<<<nc, 128, 0, h->stream>>>(P, prim, static_cast<float4*>(h->f[h->cur]),
                                                   h->W[h->cur], h->nwe);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(h->stream));
  return UGKS_OK;
}

// Capture one step per ping-pong parity into a graph (private capture stream; the graphs
// are replayed on the handle's stream, which may be the legacy default stream).
static cudaError_t build_graphs(ugks_ctx* h) {
  cudaError_t e;
  if (!h->cap_stream && (e = cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking)) != cudaSuccess)
    return e;
  const int cur0 = h->cur;
  for (int par = 0; par < 2; par++) {
    h->cur = par;
    cudaGraph_t g = nullptr;
    if ((e = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) break;
    const cudaError_t el = launch_any(h, h->cap_stream);
    e = cudaStreamEndCapture(h->cap_stream, &g);
    if (el != cudaSuccess) e = el;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&h->graph[par], g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) break;
  }
  h->cur = cur0;
  return e;
}

ugks_status ugks_step(ugks_handle h, int nsteps) {
  if (!h || nsteps < 0) return fail(h, UGKS_EINVAL, "step: bad argument");
  if (!h->profiling && !h->graph[1]) {
    cudaError_t e = build_graphs(h);
    if (e != cudaSuccess) return cuda_fail(h, e, "step graph capture");
  }
  for (int s = 0; s < nsteps; s++) {
    cudaError_t e;
    if (h->profiling)  // direct launches so that the tracing events sit between kernels
      e = launch_any(h, h->stream);
    else
      e = cudaGraphLaunch(h->graph[h->cur], h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "step launch");
    h->cur ^= 1;
    h->steps_done++;
  }
  return UGKS_OK;
}

ugks_status ugks_set_wait_limit(ugks_handle h, long long polls) {
  if (!h || polls < 0) return fail(h, UGKS_EINVAL, "set_wait_limit: bad argument");
  h->P.walk_wait_polls = polls > (1LL << 30) ? (1 << 30) : (int)polls;
  if (h->d_slot) {  // the FP32-f step reads its parameters from its slot descriptor
    CK(cudaStreamSynchronize(h->stream));
    const SlotDev S = slot_desc(h, h->cur, h->walk_rows);
    CK(cudaMemcpy(h->d_slot, &S, sizeof(SlotDev), cudaMemcpyHostToDevice));
  }
  return upload_owner(h);
}

ugks_status ugks_set_sums_split(ugks_handle h, int warps) {
  if (!h || !(warps == 0 || warps == 1 || warps == 2 || warps == 4))
    return fail(h, UGKS_EINVAL, "set_sums_split: warps must be 0, 1, 2 or 4");
  if (!h->d_slot) return fail(h, UGKS_EINVAL, "set_sums_split: FP32-f form only");
  if (h->P.shk && warps > 1) return fail(h, UGKS_EINVAL, "set_sums_split: one warp per cell for the Shakhov model");
  CK(cudaStreamSynchronize(h->stream));
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  h->sums_split = warps == 0 ? auto_sums_split(h->P, sms) : warps;
  h->sums_tiled = use_sums_tiles(h->P, h->sums_split, sms);
  CK(upload_single_f32(h));
  for (int b = 0; b < 2; b++)  // the captured steps hold the old grid: capture them again
    if (h->graph[b]) {
      CK(cudaGraphExecDestroy(h->graph[b]));
      h->graph[b] = nullptr;
    }
  return upload_owner(h);
}

int ugks_get_sums_split(ugks_handle h) { return (h && h->d_slot) ? h->sums_split : 0; }

ugks_status ugks_sync(ugks_handle h) {
  if (!h) return UGKS_EINVAL;
  return check_err(h);
}

ugks_status ugks_moments(ugks_handle h, double* W_host, double* prim_host) {
  if (!h || !W_host) return fail(h, UGKS_EINVAL, "moments: NULL argument");
  ugks_status s = copy_W_out(h, W_host, cudaMemcpyDeviceToHost);
  if (s) return s;
  if (prim_host) {
    const int nc = h->P.nx * h->P.ny;
    k_prim<<<(nc + 127) / 128, 128, 0, h->stream>>>(h->P, h->W[h->cur], h->nwe, h->sums);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(prim_host, h->sums, 4 * sizeof(double) * nc, cudaMemcpyDeviceToHost, h->stream));
  }
  return check_err(h);
}

ugks_status ugks_get_state(ugks_handle h, double* f_host, double* W_host) {
  if (!h || !f_host || !W_host) return fail(h, UGKS_EINVAL, "get_state: NULL argument");
  ugks_status s = copy_f_out(h, f_host, true);
  if (s) return s;
  s = copy_W_out(h, W_host, cudaMemcpyDeviceToHost);
  if (s) return s;
  return check_err(h);
}

ugks_status ugks_get_state_device(ugks_handle h, double* f_dev, double* W_dev) {
  if (!h || !f_dev || !W_dev) return fail(h, UGKS_EINVAL, "get_state_device: NULL argument");
  ugks_status s = copy_f_out(h, f_dev, false);
  if (s) return s;
  return copy_W_out(h, W_dev, cudaMemcpyDeviceToDevice);
}

ugks_status ugks_residual(ugks_handle h, double res[4]) {
  if (!h || !res) return fail(h, UGKS_EINVAL, "residual: NULL argument");
  std::vector<double> part((size_t)8 * h->nrblocks);
  CK(cudaMemcpyAsync(part.data(), h->rpart, part.size() * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  ugks_status s = check_err(h);
  if (s) return s;
  const int nc = h->P.nx * h->P.ny;
  for (int c = 0; c < 4; c++) {
    double ss = 0, mx = 0;
    for (int b = 0; b < h->nrblocks; b++) {
      ss += part[(size_t)b * 8 + c];
      mx = fmax(mx, part[(size_t)b * 8 + 4 + c]);
    }
    res[c] = h->steps_done ? sqrt(ss / nc) / fmax(mx, 1e-300) : 0.0;
  }
  return UGKS_OK;
}

ugks_status ugks_profile(ugks_handle h, int enable) {
  if (!h) return UGKS_EINVAL;
  CK(cudaStreamSynchronize(h->stream));
  h->profiling = enable != 0;
  h->events_used = 0;
  return UGKS_OK;
}

ugks_status ugks_kernel_times(ugks_handle h, double* ms, long* launches) {
  if (!h) return UGKS_EINVAL;
  CK(cudaStreamSynchronize(h->stream));
  double acc[UGKS_NKERNELS] = {0};
  const size_t per = UGKS_NKERNELS + 1, nsets = h->events_used / per;
  for (size_t s = 0; s < nsets; s++)
    for (int k = 0; k < UGKS_NKERNELS; k++) {
      if (k == kNoKernel) continue;
      float t = 0.f;
      CK(cudaEventElapsedTime(&t, h->events[s * per + k], h->events[s * per + k + 1]));
      acc[k] += t;
    }
  for (int k = 0; k < UGKS_NKERNELS; k++) {
    if (ms) ms[k] = acc[k];
    if (launches) launches[k] = k == kNoKernel ? 0 : (long)nsets;
  }
  return UGKS_OK;
}

const char* ugks_kernel_name(int i) { return (i >= 0 && i < UGKS_NKERNELS) ? kKernelNames[i] : ""; }

}  // extern "C"

// =====================================================================================
// Batch of independent instances (FP32-f form)
// =====================================================================================
struct ugks_batch_ctx {
  cudaStream_t stream = nullptr;
  cudaStream_t cap_stream = nullptr;
  int max_slots = 0;
  size_t budget = 0, used = 0;
  std::vector<ugks_ctx*> ctx;       // per slot, nullptr when free
  std::vector<int> walk_rows;       // per slot: cell tile of the walk (rows), 0: automatic
  std::vector<int> eff_rows;        // per slot: rows in use
  std::vector<int> walk_vtile;      // per slot: velocity tile of the walk (chunks, 0 = all)
  bool persistent = false;          // one cooperative launch per step (else phase launches)
  int grid_step = 0;                // co-resident blocks of the persistent step kernel
  BarrierDev* d_bar = nullptr;      // its grid barrier (count, gen, wait limit, timeout flag)
  SlotDev* d_slots = nullptr;
  std::vector<SlotDev> h_slots;     // their host copies
  BatchWork* d_work = nullptr;
  BatchWork h_work;
  int par = 0;                      // parity of the next step
  cudaGraphExec_t graph[2] = {nullptr, nullptr};  // captured step, per parity
  int grid[16] = {0};               // per step kernel: resident blocks
  int kinds = 0;                    // kinds of the active instances (the captured launches)
  std::string last_error;
};

namespace {

// Kernels of the FP32-f step: a phase has one kernel per kind of instance
enum StepKernel { kGhost, kSumsTile, kSumsWarp, kSumsShk, kFaces, kFacesShk, kCells, kStrip, kStripShk,
                  kStepKernels };
struct StepKernelInfo {
  const void* fn;
  size_t smem;   // dynamic shared memory
  int phase;
  int kinds;     // kinds of instances it serves (bits of instance_kind)
};
// 1: BGK, one thread per cell in the sums; 2: BGK, one or more warps per cell; 4: Shakhov
int instance_kind(const ugks_ctx* h) { return h->P.shk ? 4 : (h->sums_tiled ? 1 : 2); }
const StepKernelInfo kStepInfo[kStepKernels] = {
    {(const void*)kb_ghost, 0, 0, 7},          {(const void*)kb_sums_tile, kTileSmem, 1, 1},
    {(const void*)kb_sums, 0, 1, 2},           {(const void*)kb_sums_shk, 0, 1, 4},
    {(const void*)kb_faces, 0, 2, 3},          {(const void*)kb_faces_shk, 0, 2, 4},
    {(const void*)kb_cells, 0, 3, 7},          {(const void*)kb_strip, kStripSmem, 4, 3},
    {(const void*)kb_strip_shk, kStripSmem, 4, 4}};

// Shared-memory limits of the step kernels, and their resident blocks on the whole device.
cudaError_t step_grids(int* grid) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  for (int k = 0; k < kStepKernels && e == cudaSuccess; k++) {
    int nb = 0;
    if (kStepInfo[k].smem)
      e = cudaFuncSetAttribute(kStepInfo[k].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepInfo[k].smem);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kStepInfo[k].fn, 128, kStepInfo[k].smem);
    grid[k] = (nb > 0 ? nb : 1) * sms;
  }
  return e;
}

cudaError_t launch_kernel(int k, int grid, const SlotDev* slots, const BatchWork* work, int par, cudaStream_t st) {
  void* args[3] = {(void*)&slots, (void*)&work, (void*)&par};
  return cudaLaunchKernel(kStepInfo[k].fn, dim3(grid), dim3(128), args, kStepInfo[k].smem, st);
}

ugks_status bfail(ugks_batch_ctx* b, ugks_status s, const std::string& m) {
  if (b) b->last_error = m;
  return s;
}

#define BCK(call)                                                                        \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) return bfail(b, UGKS_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

SlotDev slot_desc(const ugks_ctx* h, int par, int walk_rows, int walk_vtile) {
  SlotDev S;
  memset(&S, 0, sizeof S);
  S.P = h->P;
  S.f[0] = static_cast<float4*>(h->f[0]);
  S.f[1] = static_cast<float4*>(h->f[1]);
  S.W[0] = h->W[0];
  S.W[1] = h->W[1];
  S.sums = h->sums;
  S.fxf = h->fxf;
  S.fyf = h->fyf;
  S.cellf = h->cellf;
  S.Fx = h->Fx;
  S.Fy = h->Fy;
  S.mt4 = h->mt4;
  S.rpart = h->rpart;
  S.err = h->err;
  S.nwe = h->nwe;
  S.nrblocks = h->nrblocks;
  S.face_block = h->face_block;
  S.cell_block = h->cell_block;
  S.nchunk_neg = h->nchunk_neg;
  S.nchunk_pos = h->nchunk_pos;
  S.walk_rows = walk_rows;
  S.walk_vtile = walk_vtile;
  S.sums_split = h->sums_split;
  S.sums_tiled = h->sums_tiled;
  S.cur = h->cur ^ par;
  return S;
}

// The captured steps are captured again at the next step.
void drop_graphs(ugks_batch_ctx* b) {
  for (int par = 0; par < 2; par++)
    if (b->graph[par]) {
      cudaGraphExecDestroy(b->graph[par]);
      b->graph[par] = nullptr;
    }
}

// Rows per tile of the walk for an instance that has `warps` resident warps to itself.  With
// two waves or more of tiles of kWalkRows rows: equal tiles of at most that many (longer ones lose
// the L2 hits of the strips' halos: 800x400x28^2 1.717 ms at 64 rows, 1.803 at 128; shorter ones
// pay for their first face row and halo rows more often: 333x167x37^2 0.519 ms at 64, 0.549 at 14).
// Below that the warps walk their tiles side by side and a step takes waves x (rows + 0.8) row
// times: 40x20x20^2 one tile of 20 rows -> 1 row, 38.9 -> 14.1 us; 100x50x28^2 50 -> 10 rows,
// 80 -> 39 us.
int auto_walk_rows(const Params& P, int nchunk, long warps) {
  const long per = (long)((P.nx + kStripW - 1) / kStripW) * nchunk;
  const int tiles = (P.ny + kWalkRows - 1) / kWalkRows;
  int best = (P.ny + tiles - 1) / tiles;
  if (per * tiles >= 2 * warps) return best;
  double best_t = 1e300;
  for (int rows = 1; rows <= (P.ny < kWalkRows ? P.ny : kWalkRows); rows++) {
    const long items = per * ((P.ny + rows - 1) / rows);
    const double t = (double)((items + warps - 1) / warps) * (rows + 0.8);
    if (t <= best_t) {
      best_t = t;
      best = rows;
    }
  }
  return best;
}

// Choose the walk tiles, rebuild the work table of the active slots and upload it together with
// every slot's descriptor (stream-ordered, one wait): the table's block counts and the captured
// kernels follow from the same descriptors that the device reads, whatever was set on an instance
// since the last upload.  An instance without a set tile gets its share of the resident warps by
// its velocity-cells.  An admission changes every share, so that single descriptors uploaded one
// by one would cost a copy and a wait per slot.
ugks_status upload_work(ugks_batch_ctx* b) {
  BatchWork& w = b->h_work;
  double total = 0.0;
  long faces = 0;
  for (ugks_ctx* h : b->ctx)
    if (h) {
      total += (double)h->P.nx * h->P.ny * h->P.nq;
      faces += (long)(h->P.nx + 1) * h->P.ny + (long)h->P.nx * (h->P.ny + 1);
    }
  // the faces per block follow from all instances' faces: a batch's blocks have four warps, and with
  // one of them at work 64 serving requests took 625 us a step instead of 599, 16 uneven instances
  // 4.18 ms instead of 4.13 (12 requests, below the line, 156 us instead of 162)
  const int face_block = small_block(faces);
  w.n = 0;
  int kinds = 0, last = 0;
  for (int p = 0; p < kPhases; p++) w.start[p][0] = 0;
  for (int s = 0; s < b->max_slots; s++) {
    const ugks_ctx* h = b->ctx[s];
    if (!h) continue;
    int rows = b->walk_rows[s];
    if (rows <= 0) {
      const double share = (double)h->P.nx * h->P.ny * h->P.nq / total;
      const long warps = (long)(share * b->grid[kStrip] * kWarpsPerBlock);
      rows = auto_walk_rows(h->P, h->nchunk_neg + h->nchunk_pos, warps < 1 ? 1 : warps);
    }
    b->eff_rows[s] = rows;
    b->h_slots[s] = slot_desc(h, b->par, rows, b->walk_vtile[s]);
    b->h_slots[s].face_block = face_block;
    kinds |= instance_kind(h);
    last = s + 1;
    const int a = w.n++;
    w.slot[a] = s;
    for (int p = 0; p < kPhases; p++) {
      const long next = (long)w.start[p][a] + phase_blocks(b->h_slots[s], p);
      if (next > 0x7fffffffL) return bfail(b, UGKS_EINVAL, "batch too large for the work table");
      w.start[p][a + 1] = (int)next;
    }
  }
  if (last)
    BCK(cudaMemcpyAsync(b->d_slots, b->h_slots.data(), sizeof(SlotDev) * last, cudaMemcpyHostToDevice, b->stream));
  BCK(cudaMemcpyAsync(b->d_work, &w, sizeof(BatchWork), cudaMemcpyHostToDevice, b->stream));
  BCK(cudaStreamSynchronize(b->stream));  // host memory reused by the next update
  if (kinds != b->kinds && !b->persistent) drop_graphs(b);  // other kernels
  b->kinds = kinds;
  return UGKS_OK;
}

// A setting of an instance in a batch takes effect in the batch's steps.
ugks_status upload_owner(ugks_ctx* h) {
  if (!h->owner) return UGKS_OK;
  const ugks_status r = upload_work(h->owner);
  return r ? fail(h, r, h->owner->last_error) : UGKS_OK;
}

cudaError_t launch_batch(ugks_batch_ctx* b, cudaStream_t st) {
  if (b->persistent) {
    // one cooperative launch: every block is resident, so the grid barriers can complete
    cudaError_t e = cudaMemsetAsync(b->d_bar, 0, 2 * sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof lc);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    lc.gridDim = dim3(b->grid_step);
    lc.blockDim = dim3(128);
    lc.dynamicSmemBytes = kStepSmem;
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kb_step, (const SlotDev*)b->d_slots, (const BatchWork*)b->d_work, b->par, b->d_bar);
  }
  for (int k = 0; k < kStepKernels; k++)
    if (kStepInfo[k].kinds & b->kinds) {
      const cudaError_t e = launch_kernel(k, b->grid[k], b->d_slots, b->d_work, b->par, st);
      if (e != cudaSuccess) return e;
    }
  return cudaGetLastError();
}

// Warps per cell of the FP32-f sums kernel chosen from the mesh and the device: split the
// velocity space of each cell over 2 or 4 warps while the cells alone would fill fewer than
// two waves of the kernel's resident warps (sms x 5 blocks x 4 warps) and every warp keeps at
// least two FP32 chunks of row pairs per half of the v axis.
int auto_sums_split(const Params& P, int sms) {
  if (P.shk) return 1;  // the Shakhov model's heat-flux sums run one warp per cell
  const long cells = (long)(P.nx + 2) * (P.ny + 2), resident = (long)sms * 5 * kWarpsPerBlock;
  int pmin = P.pr_neg < P.pr_all - P.pr_neg ? P.pr_neg : P.pr_all - P.pr_neg;
  if (pmin == 0) pmin = P.pr_all;
  int split = 1;
  while (split < kWarpsPerBlock && cells * split < 2 * resident && pmin >= 2 * split * kSumChunkPairs)
    split *= 2;
  return split;
}

// Sums with one thread per cell (sums_tile_body) where its tiles keep the device busy: from one
// and a half blocks per SM.  Measured, warp per cell -> thread per cell, 28^2 velocities: 120x60
// (256 tiles) 42.9 -> 40.8 us, 140x70 60.8 -> 49.5 us, 166x83 (462, just past a wave of resident
// blocks) 77.3 -> 71.6 us, 800x400 1456 -> 947 us; 120x60 at 16^2 26.8 -> 22.2 us, at 37^2 100.8 -> 72.6
// us, at 64^2 175.9 -> 151.4 us.  Below, a block has an SM to itself and its four warps do not fill it.
bool use_sums_tiles(const Params& P, int split, int sms) {
  return !P.shk && split == 1 && 2L * tiles_x(P) * tiles_y(P) >= 3L * sms;
}

// Slot descriptor, one-instance work table and grid sizes of the FP32-f step (uploaded again
// when a tile shape or the sums split changes).
cudaError_t upload_single_f32(ugks_ctx* h) {
  cudaError_t e;
  int cap[kStepKernels];
  if ((e = step_grids(cap)) != cudaSuccess) return e;
  h->walk_rows = auto_walk_rows(h->P, h->nchunk_neg + h->nchunk_pos, (long)cap[kStrip] * kWarpsPerBlock);
  const SlotDev S = slot_desc(h, h->cur, h->walk_rows);
  BatchWork w;
  memset(&w, 0, sizeof w);
  w.n = 1;
  w.slot[0] = 0;
  for (int p = 0; p < kPhases; p++) w.start[p][1] = phase_blocks(S, p);
  for (int k = 0; k < kStepKernels; k++) {
    const int want = w.start[kStepInfo[k].phase][1];
    h->grid1[k] = want < 1 ? 1 : (want < cap[k] ? want : cap[k]);
  }
  if ((e = cudaMemcpy(h->d_slot, &S, sizeof(SlotDev), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  return cudaMemcpy(h->d_work, &w, sizeof(BatchWork), cudaMemcpyHostToDevice);
}

cudaError_t setup_single_f32(ugks_ctx* h) {
  cudaError_t e = cudaMalloc((void**)&h->d_slot, sizeof(SlotDev));
  if (e != cudaSuccess) return e;
  h->bytes += sizeof(SlotDev);
  if ((e = cudaMalloc((void**)&h->d_work, sizeof(BatchWork))) != cudaSuccess) return e;
  h->bytes += sizeof(BatchWork);
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  h->sums_split = auto_sums_split(h->P, sms);
  h->sums_tiled = use_sums_tiles(h->P, h->sums_split, sms);
  return upload_single_f32(h);
}

cudaError_t launch_step_f32(ugks_ctx* h, cudaStream_t st) {
  cudaError_t r;
  const int kind = instance_kind(h);
  int next = 0;  // next event: the ring is the first of the step's six named parts, the second is empty
  for (int k = 0; k < kStepKernels; k++) {
    if (!(kStepInfo[k].kinds & kind)) continue;
    while (next <= (kStepInfo[k].phase ? kStepInfo[k].phase + 1 : 0))
      if ((r = mark(h, next++)) != cudaSuccess) return r;
    if ((r = launch_kernel(k, h->grid1[k], h->d_slot, h->d_work, h->cur, st)) != cudaSuccess) return r;
  }
  if ((r = mark(h, 6)) != cudaSuccess) return r;
  if (h->profiling) h->events_used += UGKS_NKERNELS + 1;
  return cudaGetLastError();
}

cudaError_t capture_batch(ugks_batch_ctx* b) {
  cudaError_t e;
  if (!b->cap_stream && (e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking)) != cudaSuccess)
    return e;
  cudaGraph_t g = nullptr;
  if ((e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return e;
  const cudaError_t el = launch_batch(b, b->cap_stream);
  e = cudaStreamEndCapture(b->cap_stream, &g);
  if (el != cudaSuccess) e = el;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph[b->par], g, 0);
  if (g) cudaGraphDestroy(g);
  return e;
}

// Default wait of the persistent step's grid barriers: about 1 s of 128 ns polls.
constexpr unsigned long long kDefaultWaitPolls = 8000000ull;

int velocity_class(const ugks_config& c) {
  const int nq = c.nu * c.nv;
  return nq <= 576 ? 0 : (nq <= 1600 ? 1 : (nq <= 4096 ? 2 : 3));
}

}  // namespace

extern "C" {

size_t ugks_state_bytes(const ugks_config* cfg) {
  return validate(cfg) ? 0 : predict_bytes(cfg);
}

ugks_status ugks_batch_create(int max_slots, size_t hbm_budget, void* cuda_stream, ugks_batch* out) {
  if (!out || max_slots < 1 || max_slots > kMaxSlots) return UGKS_EINVAL;
  *out = nullptr;
  ugks_batch_ctx* b = new ugks_batch_ctx();
  b->stream = static_cast<cudaStream_t>(cuda_stream);
  b->max_slots = max_slots;
  b->budget = hbm_budget;
  b->ctx.assign(max_slots, nullptr);
  b->walk_rows.assign(max_slots, 0);
  b->eff_rows.assign(max_slots, 0);
  b->h_slots.resize(max_slots);
  b->walk_vtile.assign(max_slots, 0);
  memset(&b->h_work, 0, sizeof(BatchWork));
  cudaError_t e = cudaMalloc((void**)&b->d_slots, sizeof(SlotDev) * max_slots);
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_work, sizeof(BatchWork));
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_work, 0, sizeof(BatchWork), b->stream);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = step_grids(b->grid);
  // persistent step: every block must be resident at once (cooperative launch)
  int coop = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kb_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepSmem);
  if (e == cudaSuccess) {
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kb_step, 128, kStepSmem);
    b->grid_step = nb * sms;
    b->persistent = coop && nb > 0;
  }
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->d_bar, sizeof(BarrierDev));
  if (e == cudaSuccess) {
    BarrierDev bar;
    memset(&bar, 0, sizeof bar);
    bar.limit = kDefaultWaitPolls;
    e = cudaMemcpyAsync(b->d_bar, &bar, sizeof bar, cudaMemcpyHostToDevice, b->stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) {
    fprintf(stderr, "ugks_batch_create: %s\n", cudaGetErrorString(e));
    ugks_batch_destroy(b);
    return e == cudaErrorMemoryAllocation ? UGKS_ENOMEM : UGKS_ECUDA;
  }
  *out = b;
  return UGKS_OK;
}

void ugks_batch_destroy(ugks_batch b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (ugks_ctx* h : b->ctx)
    if (h) ugks_destroy(h);
  drop_graphs(b);
  if (b->cap_stream) {
    cudaStreamSynchronize(b->cap_stream);
    cudaStreamDestroy(b->cap_stream);
  }
  if (b->d_slots) cudaFree(b->d_slots);
  if (b->d_work) cudaFree(b->d_work);
  if (b->d_bar) cudaFree(b->d_bar);
  delete b;
}

const char* ugks_batch_last_error(ugks_batch b) { return b ? b->last_error.c_str() : "null batch"; }

size_t ugks_batch_bytes_used(ugks_batch b) { return b ? b->used : 0; }

ugks_status ugks_batch_admit(ugks_batch b, const ugks_config* cfg, int* slot) {
  if (!b || !cfg || !slot) return bfail(b, UGKS_EINVAL, "admit: NULL argument");
  const char* bad = validate(cfg);
  if (bad) return bfail(b, UGKS_EINVAL, std::string("admit: ") + bad);
  if (cfg->precision != UGKS_FP32F) return bfail(b, UGKS_EINVAL, "admit: batch instances use UGKS_FP32F");
  const size_t need = predict_bytes(cfg);
  if (b->budget && b->used + need > b->budget) return bfail(b, UGKS_ENOMEM, "admit: over the HBM budget");
  int s = -1;
  for (int k = 0; k < b->max_slots; k++)
    if (!b->ctx[k]) { s = k; break; }
  if (s < 0) return bfail(b, UGKS_ENOMEM, "admit: no free slot");
  ugks_ctx* h = nullptr;
  const ugks_status st = ugks_create(cfg, b->stream, &h);
  if (st) return bfail(b, st, "admit: instance allocation failed");
  b->ctx[s] = h;
  b->used += h->bytes;
  int cls_rows = 0, cls_vt = 0;
  for (int k = 0; k < b->max_slots; k++)  // tuned tile of the same velocity class, if any
    if (k != s && b->ctx[k] && velocity_class(b->ctx[k]->cfg) == velocity_class(*cfg)) {
      cls_rows = b->walk_rows[k];
      cls_vt = b->walk_vtile[k];
    }
  b->walk_rows[s] = cls_rows;
  b->walk_vtile[s] = cls_vt;
  h->owner = b;
  ugks_status r = upload_work(b);
  if (r) {  // undo the admission: the caller gets no slot index to retire
    const std::string msg = b->last_error;
    cudaStreamSynchronize(b->stream);
    b->used -= h->bytes;
    ugks_destroy(h);
    b->ctx[s] = nullptr;
    upload_work(b);  // best effort: the table of the instances still admitted
    return bfail(b, r, "admit: " + msg);
  }
  *slot = s;
  return UGKS_OK;
}

ugks_status ugks_batch_retire(ugks_batch b, int slot) {
  if (!b || slot < 0 || slot >= b->max_slots || !b->ctx[slot]) return bfail(b, UGKS_EINVAL, "retire: bad slot");
  BCK(cudaStreamSynchronize(b->stream));
  b->used -= b->ctx[slot]->bytes;
  ugks_destroy(b->ctx[slot]);
  b->ctx[slot] = nullptr;
  return upload_work(b);
}

ugks_handle ugks_batch_instance(ugks_batch b, int slot) {
  if (!b || slot < 0 || slot >= b->max_slots) return nullptr;
  return b->ctx[slot];
}

ugks_status ugks_batch_step(ugks_batch b, int nsteps) {
  if (!b || nsteps < 0) return bfail(b, UGKS_EINVAL, "batch step: bad argument");
  for (int k = 0; k < nsteps; k++) {
    if (!b->graph[b->par]) {
      const cudaError_t e = capture_batch(b);
      if (e != cudaSuccess) return bfail(b, UGKS_ECUDA, std::string("batch capture: ") + cudaGetErrorString(e));
    }
    BCK(cudaGraphLaunch(b->graph[b->par], b->stream));
    b->par ^= 1;
    for (ugks_ctx* h : b->ctx)
      if (h) { h->cur ^= 1; h->steps_done++; }
  }
  return UGKS_OK;
}

ugks_status ugks_batch_sync(ugks_batch b) {
  if (!b) return UGKS_EINVAL;
  BCK(cudaStreamSynchronize(b->stream));
  int berr = 0;
  BCK(cudaMemcpy(&berr, &b->d_bar->err, sizeof(int), cudaMemcpyDeviceToHost));
  if (berr) {
    BCK(cudaMemset(&b->d_bar->err, 0, sizeof(int)));
    return bfail(b, UGKS_ETIMEOUT,
                 "a grid barrier of the persistent step gave up waiting; the instances' states "
                 "are undefined (set them again)");
  }
  for (ugks_ctx* h : b->ctx)
    if (h) {
      const ugks_status s = check_err(h);
      if (s) return bfail(b, s, "numerical failure in an instance");
    }
  return UGKS_OK;
}

ugks_status ugks_batch_set_walk_rows(ugks_batch b, int slot, int rows) {
  if (!b || slot < 0 || slot >= b->max_slots || !b->ctx[slot] || rows < 1) return bfail(b, UGKS_EINVAL, "bad tile");
  b->walk_rows[slot] = rows;
  return upload_work(b);
}

int ugks_batch_get_walk_rows(ugks_batch b, int slot) {
  return (b && slot >= 0 && slot < b->max_slots && b->ctx[slot]) ? b->eff_rows[slot] : 0;
}

ugks_status ugks_batch_set_walk_vtile(ugks_batch b, int slot, int chunks) {
  if (!b || slot < 0 || slot >= b->max_slots || !b->ctx[slot] || chunks < 0)
    return bfail(b, UGKS_EINVAL, "bad velocity tile");
  b->walk_vtile[slot] = chunks;
  return upload_work(b);
}

int ugks_batch_get_walk_vtile(ugks_batch b, int slot) {
  return (b && slot >= 0 && slot < b->max_slots && b->ctx[slot]) ? b->walk_vtile[slot] : -1;
}

ugks_status ugks_batch_set_persistent(ugks_batch b, int enable) {
  if (!b) return UGKS_EINVAL;
  if (enable && !(b->grid_step > 0))
    return bfail(b, UGKS_EINVAL, "persistent step: cooperative launch unavailable on this device");
  BCK(cudaStreamSynchronize(b->stream));
  if ((enable != 0) != b->persistent) drop_graphs(b);
  b->persistent = enable != 0;
  return UGKS_OK;
}

int ugks_batch_get_persistent(ugks_batch b) { return b && b->persistent ? 1 : 0; }

ugks_status ugks_batch_set_wait_limit(ugks_batch b, unsigned long long polls) {
  if (!b) return UGKS_EINVAL;
  BCK(cudaStreamSynchronize(b->stream));
  BCK(cudaMemcpy(&b->d_bar->limit, &polls, sizeof polls, cudaMemcpyHostToDevice));
  return UGKS_OK;
}

ugks_status ugks_batch_tune(ugks_batch b, int trial_steps, double* best_ms) {
  if (!b || trial_steps < 1) return bfail(b, UGKS_EINVAL, "tune: bad argument");
  // cell tile (rows of the walk) x velocity tile (32-slot chunks per tile, 0 = all)
  static const int cand_rows[4] = {16, 32, 64, 128};
  static const int cand_vt[3] = {0, 2, 1};
  cudaEvent_t e0, e1;
  BCK(cudaEventCreate(&e0));
  BCK(cudaEventCreate(&e1));
  float best_total = 0.f;
  ugks_status r = UGKS_OK;
  for (int cls = 0; cls < 4 && !r; cls++) {
    bool any = false;
    for (int s = 0; s < b->max_slots; s++) any |= b->ctx[s] && velocity_class(b->ctx[s]->cfg) == cls;
    if (!any) continue;
    int best_r = kWalkRows, best_v = 0;
    float best_t = 1e30f;
    auto apply = [&](int rows, int vt) -> ugks_status {
      for (int s = 0; s < b->max_slots; s++)
        if (b->ctx[s] && velocity_class(b->ctx[s]->cfg) == cls) {
          b->walk_rows[s] = rows;
          b->walk_vtile[s] = vt;
        }
      return upload_work(b);
    };
    for (int ci = 0; ci < 4 && !r; ci++)
      for (int vi = 0; vi < 3 && !r; vi++) {
        if ((r = apply(cand_rows[ci], cand_vt[vi]))) break;
        if ((r = ugks_batch_step(b, 1))) break;  // warm-up of this shape
        if (cudaEventRecord(e0, b->stream) != cudaSuccess) { r = bfail(b, UGKS_ECUDA, "tune: event"); break; }
        if ((r = ugks_batch_step(b, trial_steps))) break;
        float t = 0.f;
        if (cudaEventRecord(e1, b->stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
          r = bfail(b, UGKS_ECUDA, "tune: timing");
          break;
        }
        if (t < best_t) { best_t = t; best_r = cand_rows[ci]; best_v = cand_vt[vi]; }
      }
    if (!r) r = apply(best_r, best_v);
    best_total = best_t / trial_steps;
  }
  // step mode: one persistent launch (four grid barriers per step) against the phase
  // launches; the barriers cost more than the launches when the batch holds little work
  if (!r && b->grid_step > 0) {
    float t_mode[2] = {0.f, 0.f};
    for (int m = 0; m < 2 && !r; m++) {
      if ((r = ugks_batch_set_persistent(b, m))) break;
      if ((r = ugks_batch_step(b, 1))) break;
      float t = 0.f;
      if (cudaEventRecord(e0, b->stream) != cudaSuccess) { r = bfail(b, UGKS_ECUDA, "tune: event"); break; }
      if ((r = ugks_batch_step(b, trial_steps))) break;
      if (cudaEventRecord(e1, b->stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
          cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
        r = bfail(b, UGKS_ECUDA, "tune: timing");
        break;
      }
      t_mode[m] = t;
    }
    if (!r) r = ugks_batch_set_persistent(b, t_mode[1] <= t_mode[0] ? 1 : 0);
    if (!r) best_total = fminf(t_mode[0], t_mode[1]) / trial_steps;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (r) return r;
  if (best_ms) *best_ms = best_total;
  return ugks_batch_sync(b);
}

}  // extern "C"
