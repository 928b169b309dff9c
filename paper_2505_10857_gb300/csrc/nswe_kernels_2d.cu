// CUDA kernels (sm_103a) of the 2D NMGM (Section 4), FP64: the residual of
// Eq. 20 with dimension-by-dimension characteristic WENO3, LLF fluxes at the
// two Gauss points of each edge and the S2/S3 source quadratures; the FD
// Jacobians J21 and J9 (Eq. 21); Galerkin coarse operators by 2x2
// aggregation (Eq. 24); multicolour 3x3 block SOR (Eq. 22); restriction and
// prolongation (Eq. 24-25); a dense LU with partial pivoting on the coarsest
// grid; the App. A interpolation in tensor form (Eq. A.3).
//
// A 2D problem is large (512 x 256 cells = 131k cells, 85-200 MB of Jacobian),
// so every phase is a grid-wide kernel over cells; the host sequences them.
#include <atomic>
#include <cmath>
#include <type_traits>
#include <utility>

#include "nswe_fp64.cuh"
#include "nswe_internal.h"

namespace nswe {

// Programmatic dependent launch of the 2D kernels (on by default).
std::atomic<int> g_pdl2{1};
void set_pdl_2d(int on) { g_pdl2.store(on ? 1 : 0); }
int get_pdl_2d() { return g_pdl2.load(); }

// Stencil offset tables (dx, dy), sorted by dy then dx; index = position in
// the block storage J[(k*9 + l*3 + m)*n + c].
__constant__ int c_off_j9[9][2] = {{0, -2}, {0, -1}, {-2, 0}, {-1, 0}, {0, 0}, {1, 0}, {2, 0}, {0, 1}, {0, 2}};
__constant__ int c_off_j21[21][2] = {{-1, -2}, {0, -2}, {1, -2}, {-2, -1}, {-1, -1}, {0, -1}, {1, -1},
                                     {2, -1},  {-2, 0}, {-1, 0}, {0, 0},   {1, 0},   {2, 0},   {-2, 1},
                                     {-1, 1},  {0, 1},  {1, 1},  {2, 1},   {-1, 2},  {0, 2},   {1, 2}};
__constant__ int c_off_p5[5][2] = {{0, -1}, {-1, 0}, {0, 0}, {1, 0}, {0, 1}};
__constant__ int c_off_p9[9][2] = {{-1, -1}, {0, -1}, {1, -1}, {-1, 0}, {0, 0}, {1, 0}, {-1, 1}, {0, 1}, {1, 1}};

namespace {

// Programmatic dependent launch (sm_90 and later): every 2D kernel first
// waits until the kernel before it on the stream has completed and its
// writes are visible (griddepcontrol.wait), then lets the kernel after it
// begin launching (griddepcontrol.launch_dependents), so that a launch's
// set-up overlaps the previous kernel instead of following it. Both are
// no-ops for a launch without the programmatic-serialization attribute.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr double kZeta2 = 1e-6;
constexpr double kGs2 = 0.28867513459481288225;   // 1/(2 sqrt 3)
constexpr double kTq = 0.14433756729740644113;    // 1/(4 sqrt 3)
__device__ constexpr double kLag2[2][4] = {
    {(-kGs2 - 1.5) / 36.0, -(13.0 / 12.0) * (-kGs2 - 0.5), (13.0 / 12.0) * (-kGs2 + 0.5), -(-kGs2 + 1.5) / 36.0},
    {(kGs2 - 1.5) / 36.0, -(13.0 / 12.0) * (kGs2 - 0.5), (13.0 / 12.0) * (kGs2 + 0.5), -(kGs2 + 1.5) / 36.0}};

__device__ __forceinline__ int st_size(int st) { return st == ST_J9 ? 9 : st == ST_J21 ? 21 : st == ST_P5 ? 5 : 9; }
__device__ __forceinline__ int st_off(int st, int k, int d) {
  return st == ST_J9 ? c_off_j9[k][d] : st == ST_J21 ? c_off_j21[k][d] : st == ST_P5 ? c_off_p5[k][d] : c_off_p9[k][d];
}
__device__ __forceinline__ int st_center(int st) { return st == ST_J9 ? 4 : st == ST_J21 ? 10 : st == ST_P5 ? 2 : 4; }

struct Geo2 {
  int Nx, Ny;
  double dx, dy, g;
  const double *gq;
  const int *bck;
  const double *bcs;
};

__device__ __forceinline__ Geo2 make_geo2(const ProbDev2 &P, int l) {
  Geo2 G;
  G.Nx = P.lev[l].Nx;
  G.Ny = P.lev[l].Ny;
  G.dx = P.lev[l].dx;
  G.dy = P.lev[l].dy;
  G.g = P.g;
  G.gq = P.lev[l].gq;
  G.bck = P.lev[l].bck;
  G.bcs = P.bcs;
  return G;
}

__device__ double block_sum2(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}

}  // namespace
}  // namespace nswe

#include "nswe_tile2d.cuh"

namespace nswe {
namespace {

// ---------------------------------------------------------------------------- kernels

__global__ void __launch_bounds__(kTile2Threads, 1) k2_residual(const ProbDev2 *P, int level, const double *U,
                                                                double *R, double *partials, int TX, int TY) {
  pdl_enter();
  residual_tiles2(P, level, U, R, partials, TX, TY, blockIdx.x, gridDim.x);
}

// res = the sum of the partials / cells: strided over the block, then the
// block's fixed-order sum (one thread adding 512 partials took 36 us).
__device__ __forceinline__ void finish_block2(const double *partials, int nparts, int n, double *res) {
  __shared__ double red[33];
  double v = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) v += partials[i];
  const double s = block_sum2(v, red);
  if (threadIdx.x == 0) *res = s / n;
}

__global__ void __launch_bounds__(kThreads) k2_finish(const double *partials, int nparts, int n, double *res) {
  pdl_enter();
  finish_block2(partials, nparts, n, res);
}

template <typename TJ, bool FROZEN>
__global__ void __launch_bounds__(kTile2Threads, 1) k2_jacobian(const ProbDev2 *P, int level, int st, const double *U,
                                                                double eps, double alpha, const double *R, TJ *J,
                                                                int cm, int TX, int TY) {
  pdl_enter();
  jacobian_tiles2<TJ, FROZEN>(P, level, st, U, eps, alpha, R, J, cm, TX, TY, blockIdx.x, gridDim.x);
}

// Rounded products, the last steps of a smoother update and divisions,
// written out so that all kernels of the smoother round alike.
__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double div_r(double a, double b) { return fast_div(a, b, fast_rcp(b)); }
__device__ __forceinline__ float div_r(float a, float b) { return __fdiv_rn(a, b); }
// Row (d0, d1, d2) of the inverse diagonal block times r.
template <typename T>
__device__ __forceinline__ T dinv_row(T d0, T d1, T d2, T r0, T r1, T r2) {
  return fma(d2, r2, fma(d0, r0, mul_r(d1, r1)));
}
// `reps` relaxations x := (1 - omega) x - omega t.
template <typename T>
__device__ __forceinline__ T relax(T x, T t, T omega, int reps) {
  const T keep = T(1.0) - omega, wt = mul_r(omega, t);
  for (int s = 0; s < reps; ++s) x = fma(keep, x, -wt);
  return x;
}

// Galerkin coarse operator (Eq. 24), one item per (coarse cell, entry of its
// 3x3 blocks): sums over the four fine cells of the aggregate and their
// blocks, in that order. With the stencil known at compile time the coarse
// block of every term is too, and the loads issue together; one thread per
// coarse cell searching each term's block took 62 us at 64 x 32 in FP64.
template <int ST>
__device__ constexpr int off_c(int k, int d) {
  constexpr int j9[9][2] = {{0, -2}, {0, -1}, {-2, 0}, {-1, 0}, {0, 0}, {1, 0}, {2, 0}, {0, 1}, {0, 2}};
  constexpr int p5[5][2] = {{0, -1}, {-1, 0}, {0, 0}, {1, 0}, {0, 1}};
  constexpr int p9[9][2] = {{-1, -1}, {0, -1}, {1, -1}, {-1, 0}, {0, 0}, {1, 0}, {-1, 1}, {0, 1}, {1, 1}};
  constexpr int j21[21][2] = {{-1, -2}, {0, -2}, {1, -2}, {-2, -1}, {-1, -1}, {0, -1}, {1, -1},
                              {2, -1},  {-2, 0}, {-1, 0}, {0, 0},   {1, 0},   {2, 0},  {-2, 1},
                              {-1, 1},  {0, 1},  {1, 1},  {2, 1},   {-1, 2},  {0, 2},  {1, 2}};
  return ST == ST_J9 ? j9[ST == ST_J9 ? k : 0][d] : ST == ST_P5 ? p5[ST == ST_P5 ? k : 0][d]
                     : ST == ST_P9 ? p9[ST == ST_P9 ? k : 0][d] : j21[k][d];
}
// The coarse block that a fine cell (a, b) of its aggregate couples to through block k.
template <int ST>
__device__ constexpr int coarse_block(int a, int b, int k) {
  constexpr int CS = (ST == ST_J9 || ST == ST_P5) ? ST_P5 : ST_P9;
  const int ox = a + off_c<ST>(k, 0), oy = b + off_c<ST>(k, 1);
  const int fx = ox < 0 ? (ox - 1) / 2 : ox / 2, fy = oy < 0 ? (oy - 1) / 2 : oy / 2;
  for (int t = 0; t < (CS == ST_P5 ? 5 : 9); ++t)
    if (off_c<CS>(t, 0) == fx && off_c<CS>(t, 1) == fy) return t;
  return -1;
}

template <typename T, int ST>
__device__ __forceinline__ void coarse_op_items2(int Nx, int Ny, const T *Jf, T *Jc, int cm, int first, int stride) {
  constexpr int K = ST == ST_J9 ? 9 : ST == ST_J21 ? 21 : ST == ST_P5 ? 5 : 9;
  constexpr int Kc = (ST == ST_J9 || ST == ST_P5) ? 5 : 9;
  const int Ncx = Nx / 2, nc = Ncx * (Ny / 2);
  const size_t Sf = blk_stride(cm, Nx, Ny);
  for (int w = first; w < 9 * nc; w += stride) {
    const int e = w / nc, cc = w % nc, I = cc % Ncx, Jy = cc / Ncx;
    T acc[Kc];
#pragma unroll
    for (int t = 0; t < Kc; ++t) acc[t] = T(0.0);
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {
      const int a = ab & 1, b = ab >> 1, xi = 2 * I + a, yi = 2 * Jy + b;
      const T *J = Jf + (size_t)e * Sf + blk_pos(cm, Nx, Ny, xi, yi);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int ex = xi + off_c<ST>(k, 0), ey = yi + off_c<ST>(k, 1);
        const bool in = ex >= 0 && ex < Nx && ey >= 0 && ey < Ny;
        const T v = J[(size_t)(k * 9) * Sf];
        acc[coarse_block<ST>(a, b, k)] += in ? v : T(0.0);
      }
    }
#pragma unroll
    for (int t = 0; t < Kc; ++t) Jc[(size_t)(t * 9 + e) * nc + cc] = acc[t];
  }
}

template <typename T>
__device__ __forceinline__ void coarse_op_cells2(int Nx, int Ny, int st, const T *Jf, T *Jc, int cm, int first,
                                                 int stride) {
  if (st == ST_J9) coarse_op_items2<T, ST_J9>(Nx, Ny, Jf, Jc, cm, first, stride);
  else if (st == ST_P5) coarse_op_items2<T, ST_P5>(Nx, Ny, Jf, Jc, cm, first, stride);
  else if (st == ST_J21) coarse_op_items2<T, ST_J21>(Nx, Ny, Jf, Jc, cm, first, stride);
  else coarse_op_items2<T, ST_P9>(Nx, Ny, Jf, Jc, cm, first, stride);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_coarse_op(int Nx, int Ny, int st, const T *Jf, T *Jc, int cm) {
  pdl_enter();
  coarse_op_cells2<T>(Nx, Ny, st, Jf, Jc, cm, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename T>
__device__ __forceinline__ void dinv_cells2(int Nx, int Ny, int st, const T *J, T *Dinv, int cm, int first,
                                            int stride) {
  const int kc = st_center(st), ncell = Nx * Ny;
  const size_t n = blk_stride(cm, Nx, Ny);  // the stride of J and Dinv
  for (int q = first; q < ncell; q += stride) {
    const size_t c = blk_pos(cm, Nx, Ny, q % Nx, q / Nx);
    T a[9];
    for (int e = 0; e < 9; ++e) a[e] = J[(size_t)(kc * 9 + e) * n + c];
    // cofactors over the determinant
    const auto minor = [](T p, T q, T r, T t) { return fma(p, q, -mul_r(r, t)); };
    const T c00 = minor(a[4], a[8], a[5], a[7]), c01 = minor(a[5], a[6], a[3], a[8]),
            c02 = minor(a[3], a[7], a[4], a[6]);
    const T det = fma(a[2], c02, fma(a[0], c00, mul_r(a[1], c01)));
    const T inv[9] = {c00, minor(a[2], a[7], a[1], a[8]), minor(a[1], a[5], a[2], a[4]),
                      c01, minor(a[0], a[8], a[2], a[6]), minor(a[2], a[3], a[0], a[5]),
                      c02, minor(a[1], a[6], a[0], a[7]), minor(a[0], a[4], a[1], a[3])};
#pragma unroll
    for (int e = 0; e < 9; ++e) Dinv[(size_t)e * n + c] = div_r(inv[e], det);
  }
}

__global__ void __launch_bounds__(kThreads) k2_dinv(int Nx, int Ny, int st, const double *J, double *Dinv, int cm) {
  pdl_enter();
  dinv_cells2<double>(Nx, Ny, st, J, Dinv, cm, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// The inverse diagonal blocks of the levels l0 .. L - 1 of a hierarchy in one
// launch: block x of the grid takes blocks of the level that block0 puts it in.
template <typename T>
__global__ void __launch_bounds__(kThreads) k2_dinv_levels(const __grid_constant__ Tail2<T> t, int l0) {
  pdl_enter();
  int l = l0;
  while (l + 1 < t.L && (int)blockIdx.x >= t.off[l + 1]) ++l;
  const int nb = t.off[l + 1] - t.off[l];
  dinv_cells2<T>(t.Nx[l], t.Ny[l], t.st[l], t.J[l], t.Dinv[l], l == l0 ? t.cm : 0,
                 (blockIdx.x - t.off[l]) * blockDim.x + threadIdx.x, nb * blockDim.x);
}

// The cells of colour col, enumerated directly so that every lane of a warp
// updates a cell (an FP64 warp instruction costs the same whatever its
// active lanes): mode 0, the stencil's own colouring; mode 1, (i + j) mod Kc;
// mode 2, (j - i + Nx - 1) mod Kc. The J9 and 5-point colourings are mode 1
// with Kc = 3 and 2; the J21 and 9-point colourings are tensor products of
// residues, (i mod P) + P (j mod P) with P = 3 and 2.
__device__ __forceinline__ void sor_items(int Nx, int Ny, int st, int &mode, int &Kc, int col, int &P, int &W,
                                          int &items) {
  if (mode == 0 && (st == ST_J9 || st == ST_P5)) {
    mode = 1;
    Kc = st == ST_J9 ? 3 : 2;
  }
  if (mode == 0) {
    P = st == ST_J21 ? 3 : 2;
    const int a = col % P, b = col / P;
    W = Nx > a ? (Nx - a + P - 1) / P : 0;
    const int H = Ny > b ? (Ny - b + P - 1) / P : 0;
    items = W * H;
  } else {
    P = 0;
    W = (Nx + Kc - 1) / Kc;
    items = W * Ny;
  }
}

// Cell (i, j) of item t of a colour pass (the enumeration of sor_items);
// false if the item lies beyond the grid.
__device__ __forceinline__ bool sor_item_cell(int Nx, int mode, int Kc, int col, int P, int W, int t, int &i, int &j) {
  if (mode == 0) {
    i = col % P + (t % W) * P;
    j = col / P + (t / W) * P;
    return true;
  }
  j = t / W;
  const int a = mode == 1 ? col - j : j + Nx - 1 - col;
  i = ((a % Kc) + Kc) % Kc + (t % W) * Kc;
  return i < Nx;
}

// One colour pass of the block SOR (Eq. 22), relaxation applied reps times
// (consecutive visits of a colour see the same neighbours), with three lanes
// per cell: lane l of a cell's group forms component l of r = R + sum_k J_k
// dU_k, the group exchanges r by shuffles, and lane l updates dU component l. Ten cells per warp (lanes 30, 31 idle). On
// small grids this spreads a pass over three times as many warps, each with a
// third of the dependent FP64 instructions: an FP64 warp instruction holds
// its SMSP's FP64 unit for tens of cycles, so the length of one thread's
// chain, not the total work, bounds such a pass.
// STC >= 0: the stencil fixed at compile time: the operator's loads all issue
// together, before those of dU; -1: the stencil st of the call. early: the
// kernel before this one on the stream is a pass of the same smoothing, which
// changes only dU, so the operator and the right-hand side are read before
// waiting for it (pdl_enter is called here then). A pass of 512 x 256 is 8 us
// of FP64 issue behind a launch gap and a trip to memory: 17.0 us with the
// loads issued block by block after the wait, 14.2 so; 256 x 128 7.2 -> 4.4.
template <typename T, int STC>
__device__ __forceinline__ void sor_pass_split(int Nx, int Ny, int st_arg, const T *J, const T *Dinv, const T *R,
                                               T *dU, double omega_d, int mode, int Kc, int col, int reps,
                                               int warp0, int warps, int cm, bool early = false) {
  const int st = STC >= 0 ? STC : st_arg;
  int P, W, items;
  sor_items(Nx, Ny, st, mode, Kc, col, P, W, items);
  const T omega = T(omega_d);
  const int lane = threadIdx.x & 31, g = lane / 3, l = lane - 3 * g, src = 3 * g;
  const int n = Nx * Ny, K = st_size(st), kc = st_center(st);
  for (int w = warp0; w * 10 < items; w += warps) {  // warp-uniform
    const int t = w * 10 + g;
    int i = 0, j = 0;
    const bool on = lane < 30 && t < items && sor_item_cell(Nx, mode, Kc, col, P, W, t, i, j);
    const int c = j * Nx + i;
    const size_t S = blk_stride(cm, Nx, Ny), pc = blk_pos(cm, Nx, Ny, i, j);  // J, Dinv
    T r = on ? R[l * n + c] : T(0.0);
    T D[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) D[m] = on ? Dinv[(size_t)(l * 3 + m) * S + pc] : T(0.0);
    if constexpr (STC >= 0) {
      constexpr int KC = STC == ST_J9 ? 9 : STC == ST_P5 ? 5 : 21, C0 = KC / 2;
      T Jr[KC][3], x[KC][3];
      auto inside = [&](int k) {
        const int p = i + off_c<STC>(k, 0), q = j + off_c<STC>(k, 1);
        return on && p >= 0 && p < Nx && q >= 0 && q < Ny;
      };
#pragma unroll
      for (int k = 0; k < KC; ++k)
#pragma unroll
        for (int m = 0; m < 3; ++m)
          if (k != C0) Jr[k][m] = inside(k) ? J[(size_t)(k * 9 + l * 3 + m) * S + pc] : T(0.0);
      if (early) pdl_enter();
#pragma unroll
      for (int k = 0; k < KC; ++k)
#pragma unroll
        for (int m = 0; m < 3; ++m)
          if (k != C0)
            x[k][m] = inside(k) ? dU[m * n + c + off_c<STC>(k, 1) * Nx + off_c<STC>(k, 0)] : T(0.0);
#pragma unroll
      for (int k = 0; k < KC; ++k)
#pragma unroll
        for (int m = 0; m < 3; ++m)
          if (k != C0) r = fma(Jr[k][m], x[k][m], r);
    } else if (on) {
      for (int k = 0; k < K; ++k) {
        if (k == kc) continue;
        const int p = i + st_off(st, k, 0), q = j + st_off(st, k, 1);
        if (p < 0 || p >= Nx || q < 0 || q >= Ny) continue;
        const int cp = q * Nx + p;
        const T x0 = dU[cp], x1 = dU[n + cp], x2 = dU[2 * n + cp];
        r = fma(J[(size_t)(k * 9 + l * 3 + 0) * S + pc], x0, r);
        r = fma(J[(size_t)(k * 9 + l * 3 + 1) * S + pc], x1, r);
        r = fma(J[(size_t)(k * 9 + l * 3 + 2) * S + pc], x2, r);
      }
    }
    const T r0 = __shfl_sync(0xffffffffu, r, min(src, 31));
    const T r1 = __shfl_sync(0xffffffffu, r, min(src + 1, 31));
    const T r2 = __shfl_sync(0xffffffffu, r, min(src + 2, 31));
    if (on) {
      const T tl = dinv_row(D[0], D[1], D[2], r0, r1, r2);
      dU[l * n + c] = relax(dU[l * n + c], tl, omega, reps);
    }
  }
}

template <typename T, int STC>
__global__ void __launch_bounds__(kThreads) k2_sor_split(int Nx, int Ny, int st, const T *J, const T *Dinv,
                                                         const T *R, T *dU, double omega, int mode, int Kc, int col,
                                                         int reps, int cm, int early) {
  if (STC < 0 || !early) pdl_enter();
  sor_pass_split<T, STC>(Nx, Ny, st, J, Dinv, R, dU, omega, mode, Kc, col, reps,
                         (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5, cm, early);
}

template <typename T>
__device__ void restrict_cells2(int Nx, int Ny, int st, const T *J, const T *R, const T *dU, T *Rc, T *dUc, int first,
                                int stride, int cm = 0) {
  const int n = Nx * Ny, Ncx = Nx / 2, nc = Ncx * (Ny / 2), K = st_size(st);
  const size_t S = blk_stride(cm, Nx, Ny);  // J
  for (int cc = first; cc < nc; cc += stride) {
    const int I = cc % Ncx, Jy = cc / Ncx;
    T s[3] = {T(0.0), T(0.0), T(0.0)};
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        const int xi = 2 * I + a, yi = 2 * Jy + b, c = yi * Nx + xi;
        const size_t pc = blk_pos(cm, Nx, Ny, xi, yi);
        T r[3] = {R[c], R[n + c], R[2 * n + c]};
        for (int k = 0; k < K; ++k) {
          const int p = xi + st_off(st, k, 0), q = yi + st_off(st, k, 1);
          if (p < 0 || p >= Nx || q < 0 || q >= Ny) continue;
          const int cp = q * Nx + p;
          const T x0 = dU[cp], x1 = dU[n + cp], x2 = dU[2 * n + cp];
#pragma unroll
          for (int l = 0; l < 3; ++l) {
            r[l] = fma(J[(size_t)(k * 9 + l * 3 + 0) * S + pc], x0, r[l]);
            r[l] = fma(J[(size_t)(k * 9 + l * 3 + 1) * S + pc], x1, r[l]);
            r[l] = fma(J[(size_t)(k * 9 + l * 3 + 2) * S + pc], x2, r[l]);
          }
        }
        s[0] += r[0];
        s[1] += r[1];
        s[2] += r[2];
      }
    // the oracle accumulates the four children in row-major fine order
    for (int l = 0; l < 3; ++l) {
      Rc[l * nc + cc] = s[l];
      dUc[l * nc + cc] = T(0.0);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_restrict(int Nx, int Ny, int st, const T *J, const T *R, const T *dU,
                                                        T *Rc, T *dUc, int cm) {
  pdl_enter();
  restrict_cells2<T>(Nx, Ny, st, J, R, dU, Rc, dUc, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x,
                     cm);
}

template <typename T>
__device__ void prolong_cells2(int Nx, int Ny, T *dU, const T *dUc, int first, int stride) {
  const int n = Nx * Ny, Ncx = Nx / 2, nc = Ncx * (Ny / 2);
  for (int c = first; c < n; c += stride) {
    const int cc = (c / Nx / 2) * Ncx + (c % Nx) / 2;
    for (int l = 0; l < 3; ++l) dU[l * n + c] += dUc[l * nc + cc];
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_prolong(int Nx, int Ny, T *dU, const T *dUc) {
  pdl_enter();
  prolong_cells2<T>(Nx, Ny, dU, dUc, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// A cell-contiguous J9 (81 planes) in colour-major storage. Items run along
// the destination's rows (plane, colour, row j, slot), so writes coalesce; the
// reads of a row's three colours share their sectors through L2.
template <typename T>
__global__ void __launch_bounds__(kThreads) k2_colour_major(int Nx, int Ny, const T *J, T *Jcm) {
  pdl_enter();
  const int W = (Nx + 2) / 3;
  const long S = 3L * Ny * W, count = 81 * S;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count; t += (long)gridDim.x * blockDim.x) {
    const long pl = t / S;
    const int r = (int)(t - pl * S), slot = r % W, cj = r / W, j = cj % Ny, c = cj / Ny;
    const int i = 3 * slot + (c - j % 3 + 3) % 3;
    if (i < Nx) Jcm[t] = J[pl * Nx * Ny + (long)j * Nx + i];
  }
}

// Dense system A (row-major, unknown 3c+m) assembled from a block operator:
// zero it, then scatter the blocks.
template <typename T>
__global__ void __launch_bounds__(kThreads) k2_zero(long count, T *A) {
  pdl_enter();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count; t += (long)gridDim.x * blockDim.x) A[t] = T(0.0);
}

template <typename T>
__device__ __forceinline__ void scatter_items2(int Nx, int Ny, int st, const T *J, T *A, int first, int stride) {
  const int n = Nx * Ny, N3 = 3 * n, K = st_size(st);
  for (int t = first; t < n * K; t += stride) {
    const int c = t % n, k = t / n, i = c % Nx, j = c / Nx;
    const int p = i + st_off(st, k, 0), q = j + st_off(st, k, 1);
    if (p < 0 || p >= Nx || q < 0 || q >= Ny) continue;
    const int cp = q * Nx + p;
    for (int l = 0; l < 3; ++l)
      for (int m = 0; m < 3; ++m) A[(size_t)(3 * c + l) * N3 + 3 * cp + m] = J[(size_t)(k * 9 + l * 3 + m) * n + c];
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_scatter(int Nx, int Ny, int st, const T *J, T *A) {
  pdl_enter();
  scatter_items2<T>(Nx, Ny, st, J, A, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// LU with partial pivoting (ties to the lowest row) of A (n x n, global
// memory), by the calling thread block. piv[k] = pivot row; flag = 1 on an
// exact zero pivot.
template <typename T>
__device__ void lu_block2(int N3, T *A, int *piv, int *flag) {
  __shared__ T sv[32];
  __shared__ int si[32];
  __shared__ int s_p;
  for (int k = 0; k < N3; ++k) {
    T best = T(-1.0);
    int bi = N3;
    for (int i = k + threadIdx.x; i < N3; i += blockDim.x) {
      const T v = fabs(A[(size_t)i * N3 + k]);
      if (v > best) {
        best = v;
        bi = i;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const T ov = __shfl_down_sync(0xffffffffu, best, o);
      const int oi = __shfl_down_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    }
    if ((threadIdx.x & 31) == 0) {
      sv[threadIdx.x >> 5] = best;
      si[threadIdx.x >> 5] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      T b = sv[0];
      int p = si[0];
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
        if (sv[w] > b || (sv[w] == b && si[w] < p)) {
          b = sv[w];
          p = si[w];
        }
      s_p = p;
      piv[k] = p;
      if (A[(size_t)p * N3 + k] == T(0.0)) *flag = 1;
    }
    __syncthreads();
    const int p = s_p;
    // Swap only the active columns: earlier multipliers stay where they were
    // computed, which is what the interleaved forward solve expects.
    if (p != k)
      for (int c = k + threadIdx.x; c < N3; c += blockDim.x) {
        const T t = A[(size_t)k * N3 + c];
        A[(size_t)k * N3 + c] = A[(size_t)p * N3 + c];
        A[(size_t)p * N3 + c] = t;
      }
    __syncthreads();
    const T d = A[(size_t)k * N3 + k];
    for (int i = k + 1 + threadIdx.x; i < N3; i += blockDim.x) A[(size_t)i * N3 + k] = div_r(A[(size_t)i * N3 + k], d);
    __syncthreads();
    const int rows = N3 - k - 1;
    for (int t = threadIdx.x; t < rows * rows; t += blockDim.x) {
      const int i = k + 1 + t / rows, c = k + 1 + t % rows;
      A[(size_t)i * N3 + c] = fma(-A[(size_t)i * N3 + k], A[(size_t)k * N3 + c], A[(size_t)i * N3 + c]);
    }
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_lu(int N3, T *A, int *piv, int *flag) {
  pdl_enter();
  lu_block2<T>(N3, A, piv, flag);
}

// The row of largest |a| among the lanes' (a, row), ties to the lowest row: the
// bit patterns of non-negative values order as the values (a NaN counts as 0),
// so the integer reductions of the warp find it.
__device__ __forceinline__ int pivot_row2(float a, int row) {
  const unsigned key = a == a ? __float_as_uint(a) & 0x7fffffffu : 0u;
  const unsigned m = __reduce_max_sync(0xffffffffu, row >= 0 ? key : 0u);
  return (int)__reduce_min_sync(0xffffffffu, row >= 0 && key == m ? (unsigned)row : 0xffffffffu);
}
__device__ __forceinline__ int pivot_row2(double a, int row) {
  const unsigned hi = a == a ? (unsigned)__double2hiint(a) & 0x7fffffffu : 0u;
  const unsigned lo = a == a ? (unsigned)__double2loint(a) : 0u;
  const unsigned mh = __reduce_max_sync(0xffffffffu, row >= 0 ? hi : 0u);
  const unsigned ml = __reduce_max_sync(0xffffffffu, row >= 0 && hi == mh ? lo : 0u);
  return (int)__reduce_min_sync(0xffffffffu, row >= 0 && hi == mh && lo == ml ? (unsigned)row : 0xffffffffu);
}
// |a| > |b| as the keys above order them.
__device__ __forceinline__ bool larger2(float a, float b) { return !(b == b) ? a == a && a != 0.0f : fabsf(a) > fabsf(b); }
__device__ __forceinline__ bool larger2(double a, double b) {
  const unsigned long long ka = a == a ? (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull : 0ull;
  const unsigned long long kb = b == b ? (unsigned long long)__double_as_longlong(b) & 0x7fffffffffffffffull : 0ull;
  return ka > kb;
}

// The dense coarsest system of block operator J (cell-contiguous) assembled
// in shared memory, factored there as lu_block2 does (the same pivots and
// updates), and written to A; by one block of kLu2Threads. Every warp finds
// the pivot itself and forms the multipliers of its own rows (one lane each),
// so a step without an exchange of rows has one barrier; four warps up to 128
// unknowns, one per FP64 unit.
template <typename T>
__device__ void lu_smem_block2(int Nx, int Ny, int st, const T *J, T *A, int *piv, int *flag) {
  extern __shared__ __align__(16) unsigned char g_lu2_smem[];
  T *M = reinterpret_cast<T *>(g_lu2_smem);
  const int n = Nx * Ny, N3 = 3 * n, ld = N3 + 1, K = st_size(st);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int t = threadIdx.x; t < N3 * ld; t += blockDim.x) M[t] = T(0.0);
  __syncthreads();
  for (int t = threadIdx.x; t < 9 * n * K; t += blockDim.x) {
    const int c = t % n, ke = t / n, k = ke / 9, e = ke % 9, p = c % Nx + st_off(st, k, 0), q = c / Nx + st_off(st, k, 1);
    if (p >= 0 && p < Nx && q >= 0 && q < Ny) M[(3 * c + e / 3) * ld + 3 * (q * Nx + p) + e % 3] = J[(size_t)ke * n + c];
  }
  __syncthreads();
  for (int k = 0; k < N3; ++k) {
    T best = T(0.0);
    int row = -1;
    for (int i = k + lane; i < N3; i += 32) {
      const T a = M[i * ld + k];
      if (row < 0 || larger2(a, best)) {
        best = a;
        row = i;
      }
    }
    const int p = pivot_row2(best, row);
    if (threadIdx.x == 0) {
      piv[k] = p;
      if (M[p * ld + k] == T(0.0)) *flag = 1;
    }
    if (p != k) {  // block-uniform; only the active columns, as lu_block2
      __syncthreads();
      for (int c = k + threadIdx.x; c < N3; c += blockDim.x) {
        const T t = M[k * ld + c];
        M[k * ld + c] = M[p * ld + c];
        M[p * ld + c] = t;
      }
      __syncthreads();
    }
    // rows k + 1 + warp, + nw, ...: at most 32 of them (lu2_smem). The matrix
    // is banded: rows whose multiplier is zero and columns whose pivot-row
    // entries are zero keep their values, unless the other factor is not finite.
    const int first = k + 1 + warp, rows = first < N3 ? (N3 - first + nw - 1) / nw : 0;
    T mult = T(0.0);
    if (lane < rows) {
      const T a = M[(first + lane * nw) * ld + k], d = M[k * ld + k];
      mult = a == T(0.0) && d != T(0.0) && isfinite(d) ? T(0.0) : -div_r(a, d);
    }
    const unsigned nz = __ballot_sync(0xffffffffu, mult != T(0.0));
    const bool odd_mult = __any_sync(0xffffffffu, !isfinite(mult));
    for (int c0 = k + 1; c0 < N3; c0 += 32) {
      const int c = c0 + lane;
      const T u = c < N3 ? M[k * ld + c] : T(0.0);
      if (!odd_mult && !__any_sync(0xffffffffu, u != T(0.0))) continue;
      const unsigned todo = __any_sync(0xffffffffu, !isfinite(u)) ? 0xffffffffu : nz;
      for (int q = 0; q < rows; q += 4) {
        if (!((todo >> q) & 15u)) continue;
        T *a = M + (first + q * nw) * ld + c, v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = q + i < rows && c < N3 ? a[i * nw * ld] : T(0.0);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = fma(__shfl_sync(0xffffffffu, mult, (q + i) & 31), u, v[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (q + i < rows && c < N3) a[i * nw * ld] = v[i];
      }
    }
    __syncthreads();  // every warp has searched column k: it may take the multipliers
    if (lane < rows) M[(first + lane * nw) * ld + k] = -mult;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < N3 * N3; t += blockDim.x) A[t] = M[(t / N3) * ld + t % N3];
}

constexpr int kLu2Threads = 256;
inline int lu2_threads(int N3) { return N3 <= 128 ? 128 : kLu2Threads; }

template <typename T>
__global__ void __launch_bounds__(kLu2Threads, 1) k2_lu_smem(int Nx, int Ny, int st, const T *J, T *A, int *piv,
                                                             int *flag) {
  pdl_enter();
  lu_smem_block2<T>(Nx, Ny, st, J, A, piv, flag);
}

}  // namespace
}  // namespace nswe

#include "nswe_cluster2d.cuh"

namespace nswe {
namespace {

extern __shared__ __align__(16) unsigned char g_lus2_smem[];

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_lu_solve(int n, const T *A, const int *piv, const T *R, T *dU) {
  pdl_enter();
  lu_solve_block<T>(n, A, 3 * n, 1, piv, R, reinterpret_cast<T *>(g_lus2_smem), dU);
}

template <typename T>
__global__ void __launch_bounds__(kTail2Threads, 1) k2_vcycle_tail(const __grid_constant__ Tail2<T> t, int nu1, int nu2,
                                                                  double omega, int Kc, int cycles) {
  vcycle_cluster2<T>(t, nu1, nu2, omega, Kc, cycles);
}

__global__ void __launch_bounds__(kThreads) k2_to_f32(long count, const double *src, float *dst) {
  pdl_enter();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < count; t += (long)gridDim.x * blockDim.x)
    dst[t] = float(src[t]);
}

template <typename T>
__device__ __forceinline__ void update_cells2(int n, double *U, const T *dU, double tau, int *flag, int first,
                                              int stride) {
  for (int c = first; c < n; c += stride) {
    const double h = U[c] + tau * double(dU[c]);
    U[c] = h;
    U[n + c] += tau * double(dU[n + c]);
    U[2 * n + c] += tau * double(dU[2 * n + c]);
    if (!(h > 0.0)) atomicOr(flag, 1);
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k2_update(int n, double *U, const T *dU, double tau, int *flag) {
  pdl_enter();
  update_cells2<T>(n, U, dU, tau, flag, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(kThreads) k2_interp(const ProbDev2 *P, int coarse_level, const double *Uc,
                                                      double *Uf) {
  pdl_enter();
  const Geo2 Gc = make_geo2(*P, coarse_level);
  const int Ncx = Gc.Nx, Ncy = Gc.Ny, Nfx = 2 * Ncx, nf = 4 * Ncx * Ncy;
  const double w[2][3] = {{0.125, 1.0, -0.125}, {-0.125, 1.0, 0.125}};
  for (int cc = blockIdx.x * blockDim.x + threadIdx.x; cc < Ncx * Ncy; cc += gridDim.x * blockDim.x) {
    const int I = cc % Ncx, Jc = cc / Ncx;
    double nb[3][3][3];
    for (int q = -1; q <= 1; ++q)
      for (int p = -1; p <= 1; ++p) {
        int src, code;
        cell_meta(Gc, Uc, I + p, Jc + q, nb[q + 1][p + 1], src, code);
      }
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        const int cf = (2 * Jc + b) * Nfx + 2 * I + a;
        for (int m = 0; m < 3; ++m) {
          double s = 0.0;
          for (int q = 0; q < 3; ++q) {
            double row = 0.0;
            for (int p = 0; p < 3; ++p) row += w[a][p] * nb[q][p][m];
            s += w[b][q] * row;
          }
          Uf[m * nf + cf] = s;
        }
      }
  }
}

int grid2(long items) {
  long b = (items + kThreads - 1) / kThreads;
  return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

// Launches a 2D kernel. Launched from the host (not into a stream capture)
// and with the switch on, it carries programmatic stream serialization: it
// may begin launching while the previous kernel on the stream still runs,
// and waits for that kernel in pdl_enter(). Measured on the host-launched
// V-cycles this removes a quarter of their time on 64 x 32 to 256 x 128;
// replayed from a CUDA graph, where the gaps between kernel nodes are
// already short, the same edges made a nested solve 3 % slower, so launches
// into a capture keep ordinary stream order.
template <typename... KArgs, typename... Args>
void launchk2s(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool pdl = g_pdl2.load(std::memory_order_relaxed) && cudaStreamIsCapturing(s, &cs) == cudaSuccess &&
                   cs == cudaStreamCaptureStatusNone;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
void launchk2(void (*kern)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args &&...args) {
  launchk2s(kern, grid, block, 0, s, std::forward<Args>(args)...);
}

// Raises a kernel's limit of dynamic shared memory to that of an SM (227 KB
// less a little static), and with `clusters` allows cluster sizes above 8;
// once per device.
template <typename... KArgs>
cudaError_t raise_smem(std::atomic<unsigned> &raised, void (*kern)(KArgs...), bool clusters = false) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned bit = 1u << (dev & 31);
  if (raised.load(std::memory_order_acquire) & bit) return cudaSuccess;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTile2MaxSmem))) return e;
  if (clusters && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))) return e;
  raised.fetch_or(bit, std::memory_order_release);
  return cudaSuccess;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_tile2(std::atomic<unsigned> &raised, void (*kern)(KArgs...), int grid, size_t smem, cudaStream_t s,
                         Args &&...args) {
  const cudaError_t e = raise_smem(raised, kern);
  if (e != cudaSuccess) return e;
  launchk2s(kern, grid, kTile2Threads, smem, s, std::forward<Args>(args)...);
  return cudaGetLastError();
}

}  // namespace

// The tile of a residual (NF = 1) or Jacobian (NF flux variants) of an Nx x Ny
// level: the least estimated time over tiles that fit shared memory. A block
// holds an SM; its time is the FP64 warp instructions of its largest sub-
// partition, phase by phase (the halo's included), and the tiles run in
// rounds of one per SM. So large grids take the largest tile that fills the
// SMs evenly, small grids tiles of a few cells. Results do not depend on the
// tile, the order of the partial sums of res does.
static Tile2Shape tile2_choose(int Nx, int Ny, int NF, int K) {
  const bool jac = NF > 1;
  const int NV = jac ? 10 : 1;
  Tile2Shape best{0, 0, 0, 0};
  long best_cost = 0;
  size_t off[8];
  auto rounds4 = [](long items) { return (items + 127) / 128; };  // warps per sub-partition
  static const int side[] = {3, 4, 6, 8, 10, 12, 16, 20, 24, 28, 32};
  for (int cx : side)
    for (int cy : side) {
      // the same number of tiles, evenly sized
      const int nx = (Nx + cx - 1) / cx, ny = (Ny + cy - 1) / cy, TX = (Nx + nx - 1) / nx, TY = (Ny + ny - 1) / ny;
      const size_t smem = sizeof(double) * tile2_doubles(TX, TY, NV, NF, jac, off);
      if (smem > (size_t)kTile2MaxSmem) continue;
      const long nI = (long)(TX + 2) * (TY + 2), nP = (long)(TX + 3) * (TY + 2) + (long)(TY + 3) * (TX + 2);
      const long nF = (long)(TX + 1) * TY + (long)(TY + 1) * TX, cells = (long)TX * TY;
      long cost = 40 + 190 * rounds4(nP) + 130 * rounds4(NF * nF) + (jac ? 85 * rounds4(3L * K * cells) : 100 * rounds4(cells));
      if (jac) cost += 60 * rounds4(36 * nI);
      cost *= ((long)nx * ny + kSmCount - 1) / kSmCount;
      if (!best.TX || cost < best_cost) {
        best_cost = cost;
        best = Tile2Shape{TX, TY, nx * ny, smem};
      }
    }
  return best;
}

Tile2Shape tile2_residual_shape(int Nx, int Ny) {
  Tile2Shape t = tile2_choose(Nx, Ny, 1, 0);
  if (t.blocks > 1024) t.blocks = 1024;  // partial sums; the blocks stride over the tiles
  return t;
}
Tile2Shape tile2_jacobian_shape(int Nx, int Ny, int st) {
  return st == ST_J21 ? tile2_choose(Nx, Ny, 37, 21) : tile2_choose(Nx, Ny, 25, 9);
}

cudaError_t launch2_residual(const ProbDev2 *p, int level, int Nx, int Ny, const double *U, double *R, double *res,
                             double *partials, cudaStream_t s) {
  static std::atomic<unsigned> raised{0};
  const Tile2Shape t = tile2_residual_shape(Nx, Ny);
  const cudaError_t e = launch_tile2(raised, k2_residual, t.blocks, t.smem, s, p, level, U, R, partials, t.TX, t.TY);
  if (e != cudaSuccess) return e;
  if (res) launchk2(k2_finish, 1, kThreads, s, partials, t.blocks, Nx * Ny, res);
  return cudaGetLastError();
}

template <typename TJ>
cudaError_t launch2_jacobian(const ProbDev2 *p, int level, int Nx, int Ny, int st, const double *U, double eps,
                             double alpha, const double *R, TJ *J, bool frozen, int cm, cudaStream_t s) {
  static std::atomic<unsigned> raised[2];
  const Tile2Shape t = tile2_jacobian_shape(Nx, Ny, st);
  auto kern = frozen ? k2_jacobian<TJ, true> : k2_jacobian<TJ, false>;
  return launch_tile2(raised[frozen ? 1 : 0], kern, t.blocks, t.smem, s, p, level, st, U, eps, alpha, R, J, cm, t.TX,
                      t.TY);
}

template <typename T>
cudaError_t launch2_coarse_op(int Nx, int Ny, int st, const T *Jf, T *Jc, int cm, cudaStream_t s) {
  launchk2(k2_coarse_op<T>, grid2(9L * (Nx / 2) * (Ny / 2)), kThreads, s, Nx, Ny, st, Jf, Jc, cm);
  return cudaGetLastError();
}

cudaError_t launch2_dinv(int Nx, int Ny, int st, const double *J, double *Dinv, int cm, cudaStream_t s) {
  launchk2(k2_dinv, grid2((long)Nx * Ny), kThreads, s, Nx, Ny, st, J, Dinv, cm);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_dinv_levels(Tail2<T> t, int l0, int cm0, cudaStream_t s) {
  int blocks = 0;
  for (int l = l0; l < t.L; ++l) {
    t.off[l] = blocks;
    blocks += grid2((long)t.Nx[l] * t.Ny[l]);
  }
  t.off[t.L] = blocks;
  t.cm = cm0;
  if (blocks) launchk2(k2_dinv_levels<T>, blocks, kThreads, s, t, l0);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_sor(int Nx, int Ny, int st, const T *J, const T *Dinv, const T *R, T *dU, double omega, int mode,
                        int Kc, int col, int reps, int cm, bool early, cudaStream_t s) {
  // Items of the pass as the kernel enumerates them (see sor_items).
  long items;
  if (mode == 0 && (st == ST_J9 || st == ST_P5)) items = (long)((Nx + (st == ST_J9 ? 3 : 2) - 1) / (st == ST_J9 ? 3 : 2)) * Ny;
  else if (mode == 0) items = (long)((Nx + 2) / (st == ST_J21 ? 3 : 2) + 1) * ((Ny + 2) / (st == ST_J21 ? 3 : 2) + 1);
  else items = (long)((Nx + Kc - 1) / Kc) * Ny;
  // three lanes per cell; one warp per block on small passes so that the
  // block scheduler spreads the warps over the SMs
  const long warps = (items + 9) / 10;
  const int bs = warps <= 4L * kSmCount ? 32 : 128;
  const unsigned grid = (unsigned)((warps * 32 + bs - 1) / bs);
  if (st == ST_J9)
    launchk2(k2_sor_split<T, ST_J9>, grid, bs, s, Nx, Ny, st, J, Dinv, R, dU, omega, mode, Kc, col, reps, cm,
             (int)early);
  else if (st == ST_P5)
    launchk2(k2_sor_split<T, ST_P5>, grid, bs, s, Nx, Ny, st, J, Dinv, R, dU, omega, mode, Kc, col, reps, cm,
             (int)early);
  else
    launchk2(k2_sor_split<T, -1>, grid, bs, s, Nx, Ny, st, J, Dinv, R, dU, omega, mode, Kc, col, reps, cm,
             (int)early);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_restrict(int Nx, int Ny, int st, const T *J, const T *R, const T *dU, T *Rc, T *dUc, int cm,
                             cudaStream_t s) {
  launchk2(k2_restrict<T>, grid2((long)(Nx / 2) * (Ny / 2)), kThreads, s, Nx, Ny, st, J, R, dU, Rc, dUc, cm);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_prolong(int Nx, int Ny, T *dU, const T *dUc, cudaStream_t s) {
  launchk2(k2_prolong<T>, grid2((long)Nx * Ny), kThreads, s, Nx, Ny, dU, dUc);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_colour_major(int Nx, int Ny, const T *J, T *Jcm, cudaStream_t s) {
  launchk2(k2_colour_major<T>, grid2(81 * (long)blk_stride(1, Nx, Ny)), kThreads, s, Nx, Ny, J, Jcm);
  return cudaGetLastError();
}

// Shared memory of the factorisation of an N3 x N3 system (0: too large for it).
template <typename T>
size_t lu2_smem(int N3) {
  const size_t b = sizeof(T) * (size_t)N3 * (N3 + 1);
  return b <= (size_t)kTile2MaxSmem && N3 <= kLu2Threads ? b : 0;  // (at most 32 rows per warp)
}

template <typename T>
cudaError_t launch2_dense_factor(int Nx, int Ny, int st, const T *J, T *A, int *piv, int *flag, cudaStream_t s) {
  static std::atomic<unsigned> raised{0};
  const long N3 = 3L * Nx * Ny;
  if (const size_t smem = lu2_smem<T>((int)N3)) {
    const cudaError_t e = raise_smem(raised, k2_lu_smem<T>);
    if (e != cudaSuccess) return e;
    launchk2s(k2_lu_smem<T>, 1, lu2_threads((int)N3), smem, s, Nx, Ny, st, J, A, piv, flag);
    return cudaGetLastError();
  }
  launchk2(k2_zero<T>, grid2(N3 * N3), kThreads, s, N3 * N3, A);
  launchk2(k2_scatter<T>, grid2((long)Nx * Ny * (st == ST_J21 ? 21 : 9)), kThreads, s, Nx, Ny, st, J, A);
  launchk2(k2_lu<T>, 1, kThreads, s, (int)N3, A, piv, flag);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_dense_solve(int n, const T *A, const int *piv, const T *R, T *dU, cudaStream_t s) {
  launchk2s(k2_lu_solve<T>, 1, kThreads, sizeof(T) * 9 * (size_t)n, s, n, A, piv, R, dU);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch2_update(int n, double *U, const T *dU, double tau, int *flag, cudaStream_t s) {
  launchk2(k2_update<T>, grid2(n), kThreads, s, n, U, dU, tau, flag);
  return cudaGetLastError();
}

template <typename T>
int plan_tail2(Tail2<T> &t, int l0, int cm0, long max_cells, int max_ctas) {
  const size_t cap = kTile2MaxSmem / sizeof(T);
  const int N3 = 3 * t.Nx[t.L] * t.Ny[t.L];
  const size_t xs = 3 * (size_t)N3;
  t.l0 = l0;
  t.cm = cm0;
  t.ls = t.L;
  for (int m = l0; m < t.L; ++m)
    if ((long)t.Nx[m] * t.Ny[m] <= max_cells && band2_values(t.Nx[m], t.Ny[m], t.st[m], max_ctas, sizeof(T)) + xs <= cap) {
      t.ls = m;
      break;
    }
  t.ctas = t.ls < t.L ? (t.Ny[t.ls] / 2 < max_ctas ? t.Ny[t.ls] / 2 : max_ctas) : 1;
  // The larger levels keep their place for the whole launch as long as the
  // smaller ones fit beside them; those that do not all fit share one place
  // and are loaded again for each smoothing.
  size_t val[NSWE_MAX_LEVELS], rest[NSWE_MAX_LEVELS + 1], most[NSWE_MAX_LEVELS + 1], sum = 0;
  rest[t.L] = most[t.L] = 0;
  for (int m = t.L - 1; m >= t.ls; --m) {
    val[m] = band2_values(t.Nx[m], t.Ny[m], t.st[m], t.ctas, sizeof(T));
    rest[m] = rest[m + 1] + val[m];
    most[m] = most[m + 1] > val[m] ? most[m + 1] : val[m];
  }
  t.shared_from = t.ls;
  while (t.shared_from < t.L && sum + rest[t.shared_from] + xs > cap &&
         sum + val[t.shared_from] + most[t.shared_from + 1] + xs <= cap)
    sum += val[t.shared_from++];
  const bool all = sum + rest[t.shared_from] + xs <= cap;
  size_t at = 0;
  for (int m = t.ls; m < t.L; ++m) {
    t.off[m] = (int)at;
    if (all || m < t.shared_from) at += val[m];
  }
  if (!all) at += most[t.shared_from];
  if (all) t.shared_from = t.L;
  // a warp per ten cells of the largest colour pass, at least the direct solve's rows
  int groups = (N3 + 31) / 32;
  for (int m = t.ls; m < t.L; ++m) {
    const int pairs = t.Ny[m] / 2, nA = pairs < t.ctas ? pairs : t.ctas, rows = 2 * ((pairs + nA - 1) / nA);
    const int g = (band2_slots(t.Nx[m], t.st[m], rows) + 9) / 10;
    groups = g > groups ? g : groups;
  }
  t.threads = groups <= 4 ? 128 : groups <= 8 ? 256 : kTail2Threads;
  t.lu_off = (int)at;
  t.lu_smem = t.lu_off + (size_t)N3 * (N3 + 1) + xs <= cap;
  t.smem = sizeof(T) * (t.lu_off + (t.lu_smem ? (size_t)N3 * (N3 + 1) : 0) + xs);
  return t.ls;
}

namespace {
// One cluster of `ctas` CTAs per problem, `count` problems. Behind the coarsest
// factorisation, and with the overlap switch on, the cluster begins its way
// down while the factorisation runs and waits for it before the direct solve;
// into a capture too, where this is one edge per V-cycle.
template <typename... KArgs, typename... Args>
cudaError_t launch_clusters2(std::atomic<unsigned> &raised, void (*kern)(KArgs...), int count, int ctas, int threads,
                             size_t smem, bool after_factor, cudaStream_t s, Args &&...args) {
  cudaError_t e = raise_smem(raised, kern, true);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)count * (unsigned)ctas, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = after_factor && g_pdl2.load(std::memory_order_relaxed) ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
}  // namespace

int max_cluster_ctas() {
  static std::atomic<unsigned> raised{0};
  static std::atomic<int> known[32];  // per device; 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  std::atomic<int> *slot = dev < 32 ? known + dev : nullptr;
  int n = slot ? slot->load(std::memory_order_relaxed) : 0;
  if (n) return n;
  auto kern = k2_vcycle_tail<double>;
  const bool raisable = raise_smem(raised, kern, true) == cudaSuccess;
  if (!raisable) (void)cudaGetLastError();
  for (n = raisable ? kMaxClusterCtas : 1; n > 1; n /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n, 1, 1);
    cfg.blockDim = dim3(kTail2Threads, 1, 1);
    cfg.dynamicSmemBytes = kTile2MaxSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)n;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0) break;
    (void)cudaGetLastError();
  }
  if (slot) slot->store(n, std::memory_order_relaxed);
  return n;
}

template <typename T>
cudaError_t launch2_vcycle_tail(const Tail2<T> &t, int nu1, int nu2, double omega, int Kc, int cycles,
                                bool after_factor, cudaStream_t s) {
  static std::atomic<unsigned> raised{0};
  return launch_clusters2(raised, k2_vcycle_tail<T>, 1, t.ctas, t.threads, t.smem, after_factor, s, t, nu1, nu2,
                          omega, Kc, cycles);
}

cudaError_t launch2_to_f32(long count, const double *src, float *dst, cudaStream_t s) {
  launchk2(k2_to_f32, grid2(count), kThreads, s, count, src, dst);
  return cudaGetLastError();
}

#define NSWE_2D_INSTANTIATE(T)                                                                                    \
  template cudaError_t launch2_jacobian<T>(const ProbDev2 *, int, int, int, int, const double *, double, double, \
                                           const double *, T *, bool, int, cudaStream_t);                        \
  template cudaError_t launch2_coarse_op<T>(int, int, int, const T *, T *, int, cudaStream_t);                   \
  template cudaError_t launch2_sor<T>(int, int, int, const T *, const T *, const T *, T *, double, int, int, int, \
                                      int, int, bool, cudaStream_t);                                             \
  template cudaError_t launch2_restrict<T>(int, int, int, const T *, const T *, const T *, T *, T *, int,        \
                                           cudaStream_t);                                                        \
  template cudaError_t launch2_prolong<T>(int, int, T *, const T *, cudaStream_t);                               \
  template cudaError_t launch2_colour_major<T>(int, int, const T *, T *, cudaStream_t);                          \
  template cudaError_t launch2_dense_factor<T>(int, int, int, const T *, T *, int *, int *, cudaStream_t);       \
  template cudaError_t launch2_dense_solve<T>(int, const T *, const int *, const T *, T *, cudaStream_t);         \
  template cudaError_t launch2_dinv_levels<T>(Tail2<T>, int, int, cudaStream_t);                                 \
  template int plan_tail2<T>(Tail2<T> &, int, int, long, int);                                                   \
  template cudaError_t launch2_update<T>(int, double *, const T *, double, int *, cudaStream_t);                 \
  template cudaError_t launch2_vcycle_tail<T>(const Tail2<T> &, int, int, double, int, int, bool, cudaStream_t);
NSWE_2D_INSTANTIATE(double)
NSWE_2D_INSTANTIATE(float)
#undef NSWE_2D_INSTANTIATE

cudaError_t launch2_interp(const ProbDev2 *p, int coarse_level, int nc, const double *Uc, double *Uf,
                           cudaStream_t s) {
  launchk2(k2_interp, grid2(nc), kThreads, s, p, coarse_level, Uc, Uf);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------- batched (lockstep) kernels

namespace {

// The task owning this block (tasks sorted by b0) and the block's index in
// it; null when the task's problem is masked off.
template <typename T>
__device__ __forceinline__ const BTask2<T> *btask2(const BTask2<T> *tasks, int ntask, const int *done, int &lb) {
  int lo = 0, hi = ntask - 1;
  const int b = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].b0 <= b) lo = mid;
    else hi = mid - 1;
  }
  const BTask2<T> *t = tasks + lo;
  lb = b - t->b0;
  return (done && done[t->prob]) ? nullptr : t;
}

__global__ void __launch_bounds__(kTile2Threads, 1) kb2_residual(const BTask2<double> *tasks, int ntask,
                                                                 const int *done) {
  pdl_enter();
  int lb;
  const BTask2<double> *t = btask2(tasks, ntask, done, lb);
  if (t) residual_tiles2(t->P, t->level, t->U, t->R64, t->partials, t->TX, t->TY, lb, t->nb);
}

// One task per block: res[prob] = the sum of its partials / cells (as k2_finish).
__global__ void __launch_bounds__(kThreads) kb2_finish(const BTask2<double> *tasks, int ntask, const int *done,
                                                       double *res) {
  pdl_enter();
  const BTask2<double> &t = tasks[blockIdx.x];
  if (done && done[t.prob]) return;
  finish_block2(t.partials, t.nb, t.Nx * t.Ny, res + t.prob);
}

template <typename TJ, bool FROZEN>
__global__ void __launch_bounds__(kTile2Threads, 1) kb2_jacobian(const BTask2<TJ> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<TJ> *t = btask2(tasks, ntask, done, lb);
  if (t)
    jacobian_tiles2<TJ, FROZEN>(t->P, t->level, t->st, t->U, t->eps, t->alpha, t->R64, t->J, t->cm, t->TX, t->TY, lb,
                                t->nb);
}

__global__ void __launch_bounds__(kThreads) kb2_to_f32(const BTask2<float> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<float> *t = btask2(tasks, ntask, done, lb);
  if (!t) return;
  const long count = 3L * t->Nx * t->Ny;
  for (long c = lb * (long)blockDim.x + threadIdx.x; c < count; c += (long)t->nb * blockDim.x)
    t->R32[c] = float(t->R64[c]);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_zero_du(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (!t) return;
  const long count = 3L * t->Nx * t->Ny;
  for (long c = lb * (long)blockDim.x + threadIdx.x; c < count; c += (long)t->nb * blockDim.x) t->dU[c] = T(0.0);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_coarse_op(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t) coarse_op_cells2<T>(t->Nx, t->Ny, t->st, t->J, t->Jc, t->cm, lb * blockDim.x + threadIdx.x, t->nb * blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_dinv(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t) dinv_cells2<T>(t->Nx, t->Ny, t->st, t->J, t->Dinv, t->cm, lb * blockDim.x + threadIdx.x, t->nb * blockDim.x);
}

template <typename T, int STC>
__global__ void __launch_bounds__(kB2SorThreads) kb2_sor_split(const BTask2<T> *tasks, int ntask, const int *done,
                                                               int st, double omega, int mode, int Kc, int col,
                                                               int reps) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t)
    sor_pass_split<T, STC>(t->Nx, t->Ny, st, t->J, t->Dinv, t->R, t->dU, omega, mode, Kc, col, reps,
                           (lb * blockDim.x + threadIdx.x) >> 5, (t->nb * blockDim.x) >> 5, t->cm);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_restrict(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t)
    restrict_cells2<T>(t->Nx, t->Ny, t->st, t->J, t->R, t->dU, t->Rc, t->dUc, lb * blockDim.x + threadIdx.x,
                       t->nb * blockDim.x, t->cm);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_prolong(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t) prolong_cells2<T>(t->Nx, t->Ny, t->dU, t->dUc, lb * blockDim.x + threadIdx.x, t->nb * blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kTail2Threads, 1) kb2_vcycle_tail(const Tail2<T> *tails, const BTask2<T> *tasks,
                                                                   const int *done, int nu1, int nu2, double omega,
                                                                   int Kc, int cycles) {
  const int i = blockIdx.x / cooperative_groups::this_cluster().num_blocks();
  if (done && done[tasks[i].prob]) return;  // the whole cluster
  vcycle_cluster2<T>(tails[i], nu1, nu2, omega, Kc, cycles);
}

template <typename T>
__global__ void __launch_bounds__(kLu2Threads, 1) kb2_lu_smem(const BTask2<T> *tasks, const int *done, int *flags) {
  pdl_enter();
  const BTask2<T> &t = tasks[blockIdx.x];
  if (done && done[t.prob]) return;
  lu_smem_block2<T>(t.Nx, t.Ny, t.st, t.J, t.A, t.piv, flags + t.prob);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_dense_zero(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (!t) return;
  const long N3 = 3L * t->Nx * t->Ny, count = N3 * N3;
  for (long c = lb * (long)blockDim.x + threadIdx.x; c < count; c += (long)t->nb * blockDim.x) t->A[c] = T(0.0);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_scatter(const BTask2<T> *tasks, int ntask, const int *done) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t) scatter_items2<T>(t->Nx, t->Ny, t->st, t->J, t->A, lb * blockDim.x + threadIdx.x, t->nb * blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_lu(const BTask2<T> *tasks, const int *done, int *flags) {
  pdl_enter();
  const BTask2<T> &t = tasks[blockIdx.x];
  if (done && done[t.prob]) return;
  lu_block2<T>(3 * t.Nx * t.Ny, t.A, t.piv, flags + t.prob);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_lu_solve(const BTask2<T> *tasks, const int *done) {
  pdl_enter();
  const BTask2<T> &t = tasks[blockIdx.x];
  if (done && done[t.prob]) return;
  const int n = t.Nx * t.Ny;
  lu_solve_block<T>(n, t.A, 3 * n, 1, t.piv, t.R, reinterpret_cast<T *>(g_lus2_smem), t.dU);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) kb2_update(const BTask2<T> *tasks, int ntask, const int *done,
                                                       int *flags) {
  pdl_enter();
  int lb;
  const BTask2<T> *t = btask2(tasks, ntask, done, lb);
  if (t)
    update_cells2<T>(t->Nx * t->Ny, t->U, t->dU, t->tau, flags + t->prob, lb * blockDim.x + threadIdx.x,
                     t->nb * blockDim.x);
}

}  // namespace

int b2_grid(long items) { return grid2(items); }

cudaError_t launchb2_residual(const Batch2Launch<double> &b, const int *done, double *res, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  static std::atomic<unsigned> raised{0};
  const cudaError_t e = launch_tile2(raised, kb2_residual, b.blocks, b.smem, s, b.tasks, b.ntask, done);
  if (e != cudaSuccess) return e;
  launchk2(kb2_finish, b.ntask, kThreads, s, b.tasks, b.ntask, done, res);
  return cudaGetLastError();
}

template <typename TJ>
cudaError_t launchb2_jacobian(const Batch2Launch<TJ> &b, const int *done, bool frozen, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  static std::atomic<unsigned> raised[2];
  auto kern = frozen ? kb2_jacobian<TJ, true> : kb2_jacobian<TJ, false>;
  return launch_tile2(raised[frozen ? 1 : 0], kern, b.blocks, b.smem, s, b.tasks, b.ntask, done);
}

cudaError_t launchb2_to_f32(const Batch2Launch<float> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_to_f32, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_zero_du(const Batch2Launch<T> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_zero_du<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_coarse_op(const Batch2Launch<T> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_coarse_op<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_dinv(const Batch2Launch<T> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_dinv<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_sor(const Batch2Launch<T> &b, const int *done, int st, double omega, int mode, int Kc, int col,
                         int reps, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  if (st == ST_J9)
    launchk2(kb2_sor_split<T, ST_J9>, b.blocks, kB2SorThreads, s, b.tasks, b.ntask, done, st, omega, mode, Kc, col, reps);
  else if (st == ST_P5)
    launchk2(kb2_sor_split<T, ST_P5>, b.blocks, kB2SorThreads, s, b.tasks, b.ntask, done, st, omega, mode, Kc, col, reps);
  else
    launchk2(kb2_sor_split<T, -1>, b.blocks, kB2SorThreads, s, b.tasks, b.ntask, done, st, omega, mode, Kc, col, reps);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_restrict(const Batch2Launch<T> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_restrict<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_prolong(const Batch2Launch<T> &b, const int *done, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_prolong<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_vcycle_tail(const Tail2<T> *tails, const BTask2<T> *tasks, int ntask, int ctas, int threads,
                                 size_t smem, const int *done, int nu1, int nu2, double omega, int Kc, int cycles,
                                 bool after_factor, cudaStream_t s) {
  if (ntask == 0) return cudaSuccess;
  static std::atomic<unsigned> raised{0};
  return launch_clusters2(raised, kb2_vcycle_tail<T>, ntask, ctas, threads, smem, after_factor, s, tails, tasks, done,
                          nu1, nu2, omega, Kc, cycles);
}

template <typename T>
cudaError_t launchb2_dense_factor(const Batch2Launch<T> &zero, const Batch2Launch<T> &scatter, const BTask2<T> *tasks,
                                  int ntask, int max_cells, const int *done, int *flags, cudaStream_t s) {
  if (ntask == 0) return cudaSuccess;
  static std::atomic<unsigned> raised{0};
  if (const size_t smem = lu2_smem<T>(3 * max_cells)) {
    const cudaError_t e = raise_smem(raised, kb2_lu_smem<T>);
    if (e != cudaSuccess) return e;
    launchk2s(kb2_lu_smem<T>, ntask, lu2_threads(3 * max_cells), smem, s, tasks, done, flags);
    return cudaGetLastError();
  }
  launchk2(kb2_dense_zero<T>, zero.blocks, kThreads, s, zero.tasks, zero.ntask, done);
  launchk2(kb2_scatter<T>, scatter.blocks, kThreads, s, scatter.tasks, scatter.ntask, done);
  launchk2(kb2_lu<T>, ntask, kThreads, s, tasks, done, flags);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_dense_solve(const BTask2<T> *tasks, int ntask, int max_cells, const int *done, cudaStream_t s) {
  if (ntask == 0) return cudaSuccess;
  launchk2s(kb2_lu_solve<T>, ntask, kThreads, sizeof(T) * 9 * (size_t)max_cells, s, tasks, done);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launchb2_update(const Batch2Launch<T> &b, const int *done, int *flags, cudaStream_t s) {
  if (b.ntask == 0) return cudaSuccess;
  launchk2(kb2_update<T>, b.blocks, kThreads, s, b.tasks, b.ntask, done, flags);
  return cudaGetLastError();
}

#define NSWE_B2_INSTANTIATE(T)                                                                                     \
  template cudaError_t launchb2_jacobian<T>(const Batch2Launch<T> &, const int *, bool, cudaStream_t);            \
  template cudaError_t launchb2_zero_du<T>(const Batch2Launch<T> &, const int *, cudaStream_t);                   \
  template cudaError_t launchb2_coarse_op<T>(const Batch2Launch<T> &, const int *, cudaStream_t);                 \
  template cudaError_t launchb2_dinv<T>(const Batch2Launch<T> &, const int *, cudaStream_t);                      \
  template cudaError_t launchb2_sor<T>(const Batch2Launch<T> &, const int *, int, double, int, int, int, int,     \
                                       cudaStream_t);                                                             \
  template cudaError_t launchb2_restrict<T>(const Batch2Launch<T> &, const int *, cudaStream_t);                  \
  template cudaError_t launchb2_prolong<T>(const Batch2Launch<T> &, const int *, cudaStream_t);                   \
  template cudaError_t launchb2_vcycle_tail<T>(const Tail2<T> *, const BTask2<T> *, int, int, int, size_t,         \
                                               const int *, int, int, double, int, int, bool, cudaStream_t);      \
  template cudaError_t launchb2_dense_factor<T>(const Batch2Launch<T> &, const Batch2Launch<T> &,                 \
                                                const BTask2<T> *, int, int, const int *, int *, cudaStream_t);   \
  template cudaError_t launchb2_dense_solve<T>(const BTask2<T> *, int, int, const int *, cudaStream_t);           \
  template cudaError_t launchb2_update<T>(const Batch2Launch<T> &, const int *, int *, cudaStream_t);
NSWE_B2_INSTANTIATE(double)
NSWE_B2_INSTANTIATE(float)
#undef NSWE_B2_INSTANTIATE

}  // namespace nswe
