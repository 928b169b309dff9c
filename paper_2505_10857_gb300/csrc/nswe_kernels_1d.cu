// CUDA kernels (sm_103a) of the 1D NMGM: WENO3 finite-volume residual,
// regularized FD Jacobian J3/J5, geometric multigrid V-cycle with
// multicolour block SOR, and the nested Newton solve (Algorithm 3), all FP64.
//
// Execution model: every building block is a "CTA-level" routine that loops
// over its work items with a block-wide stride, so the same code serves the
// standalone grid kernels (residual, Jacobian: many blocks per problem) and
// the persistent solve kernel, where one thread block runs a whole nested
// solve of one problem with __syncthreads() between phases and no host
// round trip. Problem data and workspace stay in device memory (L2 resident
// for the 1D sizes); the coarsest factorisation lives in shared memory.
#include <cooperative_groups.h>

#include <cmath>
#include <type_traits>

#include "nswe_fp64.cuh"
#include "nswe_internal.h"

namespace nswe {
namespace {

constexpr double kZeta = 1e-6;  // WENO epsilon (Section 3.1)

// Rounded products and sums. Where a sum takes a product that the compiler
// could fuse into it, or one of two products, the rounding is written out:
// left to the compiler it differed between the solve kernel's launch shapes
// (by their register budgets), so that a problem's bits depended on the number
// of problems launched with it.
__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_r(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_r(float a, float b) { return __fadd_rn(a, b); }

// Lagrange weights of the cubic through t = -3/2, -1/2, 1/2, 3/2 evaluated at
// the Gauss points t = -/+ 1/(2 sqrt 3) (Eq. 9). With t^2 = 1/12 the basis
// reduces to (t - 3/2)/36, -(13/12)(t - 1/2), (13/12)(t + 1/2), -(t + 3/2)/36.
constexpr double kGs = 0.28867513459481288225;  // 1/(2 sqrt 3)
__device__ constexpr double kLag[2][4] = {
    {(-kGs - 1.5) / 36.0, -(13.0 / 12.0) * (-kGs - 0.5), (13.0 / 12.0) * (-kGs + 0.5), -(-kGs + 1.5) / 36.0},
    {(kGs - 1.5) / 36.0, -(13.0 / 12.0) * (kGs - 0.5), (13.0 / 12.0) * (kGs + 0.5), -(kGs + 1.5) / 36.0}};

struct Geo {
  int N;
  double dx, g;
  const double *sf;   // [N+1] width at faces
  const double *gq;   // [3][2][N] sigma, sigma_x, b_x at the Gauss points
  const double *isf;  // [N+1] 1/sigma at faces
  const double *cgf;  // [N+1] sqrt(g/sigma) at faces
  const double *igq;  // [2][N] 1/sigma at the Gauss points
  int bl, br;
  double blh, blq, brh, brq;
  int flux;  // NSWE_FLUX_HLL or NSWE_FLUX_LLF
  // FP32 copies of the level's state and geometry, read by the FP32 Jacobian
  // passes instead of converting the FP64 values at every use (a conversion
  // from FP64 occupies the narrow FP64 pipe); nullptr: convert at use. The
  // copies hold exactly the converted values, so both give the same bits.
  const float *U32;    // [2][N]
  const float *isf32;  // [N+1]
  const float *cgf32;  // [N+1]
  const float *igq32;  // [2][N]
  const float *gq32;   // [2: sigma_x, b_x][2][N]
  float g32, hdx32;    // float(g), 0.5f * float(dx)
};

__device__ __forceinline__ Geo make_geo(const ProbDev &P, int l) {
  Geo G;
  G.U32 = G.isf32 = G.cgf32 = G.igq32 = G.gq32 = nullptr;
  G.g32 = G.hdx32 = 0.0f;
  G.N = P.lev[l].N;
  G.dx = P.lev[l].dx;
  G.g = P.g;
  G.sf = P.lev[l].sf;
  G.gq = P.lev[l].gq;
  G.isf = P.lev[l].gd;
  G.cgf = G.isf + G.N + 1;
  G.igq = G.cgf + G.N + 1;
  G.bl = P.bl;
  G.br = P.br;
  G.blh = P.blh;
  G.blq = P.blq;
  G.brh = P.brh;
  G.brq = P.brq;
  G.flux = P.flux;
  return G;
}

// Ghost state from the boundary data and the adjacent interior cell.
__device__ __forceinline__ void ghost(int kind, double bh, double bq, double sb, double He, double Qe,
                                      double &H, double &Q) {
  if (kind == NSWE_BC_DISCHARGE) {
    H = He;
    Q = bq;
  } else if (kind == NSWE_BC_DEPTH) {
    H = mul_r(sb, bh);
    Q = Qe;
  } else if (kind == NSWE_BC_STATE) {
    H = mul_r(sb, bh);
    Q = bq;
  } else {
    H = He;
    Q = Qe;
  }
}

// WENO3 in one cell from averages a, b, c (cells k-1, k, k+1), Eq. 7-8 with
// the linear weights (1/3, 2/3) for U^+_{k-1/2} and (2/3, 1/3) for
// U^-_{k+1/2}. With the differences d0 = c - b, d1 = b - a and
// s_r = (zeta + beta_r)^2, beta_r = d_r^2, the weighted means are
//   U^+_{k-1/2} = b - (s1 d0 + 2 s0 d1) / (2 (s1 + 2 s0)),
//   U^-_{k+1/2} = b + (2 s1 d0 + s0 d1) / (2 (2 s1 + s0));
// both quotients share one reciprocal. The FP64 pipe bounds every kernel
// that calls this (64 cycles per warp instruction): 21 instruction slots
// instead of the 33 of the candidate polynomials, and a small correction is
// rounded instead of the value itself.
template <typename T>
struct Slope {
  T d, s;  // difference and (zeta + d^2)^2
};

template <typename T>
__device__ __forceinline__ Slope<T> slope(T d) {
  const T e = fma(d, d, T(kZeta));
  return {d, e * e};
}

template <typename T>
__device__ __forceinline__ void weno3(T b, const Slope<T> &S0, const Slope<T> &S1, T &up, T &um) {
  const T x = S1.s * S0.d, y = S0.s * S1.d;
  const T D1 = fma(T(2.0), S0.s, S1.s), D2 = fma(T(2.0), S1.s, S0.s);
  const T hinv = T(0.5) * rcp_t(D1 * D2);
  up = fma(-fma(T(2.0), y, x), D2 * hinv, b);
  um = fma(fma(T(2.0), x, y), D1 * hinv, b);
}

template <typename T>
__device__ __forceinline__ void weno3(T a, T b, T c, T &up, T &um) {
  weno3<T>(b, slope<T>(c - b), slope<T>(b - a), up, um);
}

// FP32: the candidate polynomials with the normalised weights w0 = s1/(s1 +
// 2 s0), v0 = 2 s1/(2 s1 + s0). The FP32 pipe bounds no kernel here, and the
// difference quotients of the FP32 Jacobian show every rounding (2e-5 of its
// largest block), so its passes keep their sequence of operations.
template <>
__device__ __forceinline__ void weno3<float>(float a, float b, float c, float &up, float &um) {
  float d0 = c - b, d1 = b - a;
  float e0 = fmaf(d0, d0, float(kZeta)), e1 = fmaf(d1, d1, float(kZeta));
  float s0 = mul_r(e0, e0), s1 = mul_r(e1, e1);
  float p0 = fmaf(1.5f, b, -0.5f * c), p1 = fmaf(0.5f, a, 0.5f * b);  // U^(0), U^(1) at k-1/2
  float q0 = fmaf(0.5f, b, 0.5f * c), q1 = fmaf(1.5f, b, -0.5f * a);  // U^(0), U^(1) at k+1/2
  float D1 = fmaf(2.0f, s0, s1), D2 = fmaf(2.0f, s1, s0);
  float inv = 1.0f / mul_r(D1, D2);
  up = mul_r(fmaf(s1, p0, mul_r(2.0f * s0, p1)), mul_r(D2, inv));
  um = mul_r(fmaf(2.0f * s1, q0, mul_r(s0, q1)), mul_r(D1, inv));
}

// Quantities of one interface state entering the flux at a face of width
// sigma: velocity u = Q/H, the wave speeds lo = u - c and hi = u + c with the
// celerity c = sqrt(g H/sigma), and the physical flux F = (Q, Q^2/H +
// g H^2/(2 sigma)) (Eq. 4). One reciprocal square root r = H^(-1/2) gives
// both 1/H = r^2 and c = sqrt(g/sigma) H r; cg = sqrt(g/sigma), isg = 1/sigma
// and hg = g/(2 sigma) are per-face values. r2 = 1/H, hr = H r, c and the
// pressure term P = g H^2/(2 sigma) are kept, so that a state differing only
// in Q (fstate_q) costs four instructions. Sum says which product of u -+ c the
// wave speeds take unrounded, for each kernel as it is fastest.
enum class Sum { kRounded, kFusedC, kFusedU };

template <typename T>
struct FState {
  T H, Q, u, c, lo, hi, F1, r2, hr, P;
};

template <typename T>
struct Face {
  T isg, cg, g, hg;
};

template <typename T>
__device__ __forceinline__ Face<T> face(T isg, T cg, T g) {
  return {isg, cg, g, T(0.5) * g * isg};
}

// The state of `b` with its discharge replaced by Q.
template <Sum S, typename T>
__device__ __forceinline__ FState<T> fstate_q(const FState<T> &b, T Q, const Face<T> &f) {
  FState<T> s = b;
  s.Q = Q;
  s.u = mul_r(Q, b.r2);
  s.lo = S == Sum::kFusedC ? fma(-f.cg, b.hr, s.u) : S == Sum::kFusedU ? fma(Q, b.r2, -b.c) : add_r(s.u, -b.c);
  s.hi = S == Sum::kFusedC ? fma(f.cg, b.hr, s.u) : S == Sum::kFusedU ? fma(Q, b.r2, b.c) : add_r(s.u, b.c);
  s.F1 = fma(Q, s.u, b.P);
  return s;
}

template <Sum S, typename T>
__device__ __forceinline__ FState<T> fstate(T H, T Q, const Face<T> &f) {
  FState<T> s;
  s.H = H;
  const T r = rsqrt_t(H);
  s.r2 = mul_r(r, r);
  s.hr = mul_r(H, r);
  s.c = mul_r(f.cg, s.hr);
  if constexpr (std::is_same<T, float>::value) s.P = (0.5f * f.g * H) * (H * f.isg);  // as weno3<float>
  else s.P = (f.hg * H) * H;
  return fstate_q<S>(s, Q, f);
}

// Ordering keys of FP64 values on the integer pipe (the FP64 pipe is the
// narrow one): for finite x, key(x) orders as x, with key(-0) = -1 just
// below key(+0) = 0. Selecting by key gives fmin / fmax of two finite values
// (either zero for a pair of zeros), and x >= 0 is key(x) >= -1.
__device__ __forceinline__ long long okey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double kmin(double a, double b) { return okey(a) <= okey(b) ? a : b; }
__device__ __forceinline__ double kmax(double a, double b) { return okey(a) >= okey(b) ? a : b; }
__device__ __forceinline__ bool knonneg(double a) { return okey(a) >= -1LL; }
__device__ __forceinline__ bool knonpos(double a) { return okey(a) <= 0LL; }
__device__ __forceinline__ float kmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float kmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ bool knonneg(float a) { return a >= 0.0f; }
__device__ __forceinline__ bool knonpos(float a) { return a <= 0.0f; }

// HLL flux of two interface states: S_L = min(u_L - c_L, u_R - c_R),
// S_R = max(u_L + c_L, u_R + c_R), upwind fluxes outside the fan, the HLL
// average inside, written as the left flux and a correction: with
// w = -S_L / (S_R - S_L), F = F_L + w (F_R - F_L - S_R (U_R - U_L)).
template <typename T>
__device__ __forceinline__ void hll_states(const FState<T> &L, const FState<T> &R, T &F0, T &F1) {
  const T SL = kmin(L.lo, R.lo);
  const T SR = kmax(L.hi, R.hi);
  if (knonneg(SL)) {
    F0 = L.Q;
    F1 = L.F1;
  } else if (knonpos(SR)) {
    F0 = R.Q;
    F1 = R.F1;
  } else {
    if constexpr (std::is_same<T, float>::value) {  // as weno3<float>
      const T iw = 1.0f / (SR - SL);
      const T SLR = mul_r(SL, SR);
      F0 = mul_r(fma(SLR, R.H - L.H, fma(SR, L.Q, -mul_r(SL, R.Q))), iw);
      F1 = mul_r(fma(SLR, R.Q - L.Q, fma(SR, L.F1, -mul_r(SL, R.F1))), iw);
      return;
    }
    const T w = -SL * rcp_t(SR - SL);
    const T dQ = R.Q - L.Q;
    F0 = fma(w, fma(-SR, R.H - L.H, dQ), L.Q);
    F1 = fma(w, fma(-SR, dQ, R.F1 - L.F1), L.F1);
  }
}

// Numerical flux of two interface states: HLL, or LLF: the mean of the
// physical fluxes minus a (U_R - U_L) / 2, a = max(|u_L| + c_L, |u_R| + c_R).
// FLUX fixes the choice at compile time (NSWE_FLUX_HLL or NSWE_FLUX_LLF),
// or -1 takes it from `flux` (the standalone kernels).
template <int FLUX, typename T>
__device__ __forceinline__ void num_flux(const FState<T> &L, const FState<T> &R, int flux, T &F0, T &F1) {
  if (FLUX == NSWE_FLUX_LLF || (FLUX < 0 && flux == NSWE_FLUX_LLF)) {
    const T a = fmax(fabs(L.u) + L.c, fabs(R.u) + R.c);
    F0 = T(0.5) * (L.Q + R.Q) - T(0.5) * a * (R.H - L.H);
    F1 = T(0.5) * (L.F1 + R.F1) - T(0.5) * a * (R.Q - L.Q);
  } else {
    hll_states(L, R, F0, F1);
  }
}

// Level data in the precision T of a pass: FP64 values as stored; FP32
// values from the copies when the level has them, else converted at use.
template <typename T> struct GeoT;
template <> struct GeoT<double> {
  static __device__ __forceinline__ double u(const Geo &G, const double *U, int i) { return U[i]; }
  static __device__ __forceinline__ double isf(const Geo &G, int f) { return G.isf[f]; }
  static __device__ __forceinline__ double cgf(const Geo &G, int f) { return G.cgf[f]; }
  static __device__ __forceinline__ double igq(const Geo &G, int i) { return G.igq[i]; }
  static __device__ __forceinline__ double sigx(const Geo &G, int i) { return G.gq[2 * G.N + i]; }
  static __device__ __forceinline__ double bx(const Geo &G, int i) { return G.gq[4 * G.N + i]; }
  static __device__ __forceinline__ double g(const Geo &G) { return G.g; }
  static __device__ __forceinline__ double hdx(const Geo &G) { return 0.5 * G.dx; }
};
template <> struct GeoT<float> {
  static __device__ __forceinline__ float u(const Geo &G, const double *U, int i) {
    return G.U32 ? G.U32[i] : float(U[i]);
  }
  static __device__ __forceinline__ float isf(const Geo &G, int f) { return G.isf32 ? G.isf32[f] : float(G.isf[f]); }
  static __device__ __forceinline__ float cgf(const Geo &G, int f) { return G.cgf32 ? G.cgf32[f] : float(G.cgf[f]); }
  static __device__ __forceinline__ float igq(const Geo &G, int i) { return G.igq32 ? G.igq32[i] : float(G.igq[i]); }
  static __device__ __forceinline__ float sigx(const Geo &G, int i) {
    return G.gq32 ? G.gq32[i] : float(G.gq[2 * G.N + i]);
  }
  static __device__ __forceinline__ float bx(const Geo &G, int i) {
    return G.gq32 ? G.gq32[2 * G.N + i] : float(G.gq[4 * G.N + i]);
  }
  static __device__ __forceinline__ float g(const Geo &G) { return G.isf32 ? G.g32 : float(G.g); }
  static __device__ __forceinline__ float hdx(const Geo &G) { return G.isf32 ? G.hdx32 : 0.5f * float(G.dx); }
};

// Two-point Gauss source of cell j (Eq. 9): S = (dx/2) sum_q [g h^2 sigma_x/2
// - g sigma h b_x] at the Gauss points, h = H_h/sigma, H_h the cubic through
// the interface values p0..p3 of H at t = -3/2, -1/2, 1/2, 3/2. With
// H_h = sigma h this is sum_q H_h (A_q H_h - B_q), A_q = dx g sigma_x /
// (4 sigma^2) and B_q = dx g b_x / 2 of the cell (1/sigma is per-cell
// geometry), which a Jacobian pass forms once for its perturbed sources.
template <typename T>
struct SrcCell {
  T A[2], B[2];
};

template <typename T>
__device__ __forceinline__ SrcCell<T> src_cell(const Geo &G, int j) {
  SrcCell<T> c;
  const T gd = GeoT<T>::g(G) * GeoT<T>::hdx(G);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const T is = GeoT<T>::igq(G, q * G.N + j);
    c.A[q] = (T(0.5) * gd) * GeoT<T>::sigx(G, q * G.N + j) * (is * is);
    c.B[q] = gd * GeoT<T>::bx(G, q * G.N + j);
  }
  return c;
}

// FP32: the terms as they stand in Eq. 9 (as weno3<float>).
template <>
struct SrcCell<float> {
  float is[2], sigx[2], bx[2], g, hdx;
};

template <>
__device__ __forceinline__ SrcCell<float> src_cell<float>(const Geo &G, int j) {
  SrcCell<float> c;
  c.g = GeoT<float>::g(G);
  c.hdx = GeoT<float>::hdx(G);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    c.is[q] = GeoT<float>::igq(G, q * G.N + j);
    c.sigx[q] = GeoT<float>::sigx(G, q * G.N + j);
    c.bx[q] = GeoT<float>::bx(G, q * G.N + j);
  }
  return c;
}

__device__ __forceinline__ float source_at(const SrcCell<float> &c, float p0, float p1, float p2, float p3) {
  float S = 0.0f;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float Hh = fmaf(float(kLag[q][0]), p0, mul_r(float(kLag[q][1]), p1));
    Hh = fmaf(float(kLag[q][3]), p3, fmaf(float(kLag[q][2]), p2, Hh));
    float h = mul_r(Hh, c.is[q]);
    S = add_r(S, fmaf(mul_r(mul_r(0.5f * c.g, h), h), c.sigx[q], -mul_r(mul_r(c.g, Hh), c.bx[q])));
  }
  return S;
}

// The FP32 source_at leaves out the factor dx/2: the source, and d less the
// source in one rounding.
__device__ __forceinline__ float source_value(const SrcCell<float> &c, float S) { return mul_r(S, c.hdx); }
__device__ __forceinline__ float less_source(const SrcCell<float> &c, float d, float S) { return fmaf(-S, c.hdx, d); }
template <typename T>
__device__ __forceinline__ T source_value(const SrcCell<T> &, T S) {
  return S;
}
template <typename T>
__device__ __forceinline__ T less_source(const SrcCell<T> &, T d, T S) {
  return d - S;
}

template <typename T>
__device__ __forceinline__ T source_at(const SrcCell<T> &c, T p0, T p1, T p2, T p3) {
  T S[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const T Hh = fma(T(kLag[q][3]), p3, fma(T(kLag[q][0]), p0, fma(T(kLag[q][2]), p2, T(kLag[q][1]) * p1)));
    const T t = fma(c.A[q], Hh, -c.B[q]);
    S[q] = q == 0 ? Hh * t : fma(Hh, t, S[0]);
  }
  return S[1];
}

// ----------------------------------------------------------------------------
// Block-level helpers.

// Fixed-order block sum (warp shuffles, then warps in index order).
__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    red[32] = s;
  }
  __syncthreads();
  double s = red[32];
  __syncthreads();
  return s;
}

// ----------------------------------------------------------------------------
// Teams: the threads that share one problem's phases. BlockTeam is one
// thread block (the batched form: one problem per block). ClusterTeam is a
// thread-block cluster of up to 16 CTAs on as many SMs (the latency form:
// one problem per cluster): the per-cell loops of a phase are strided over
// all its threads, phases are separated by cluster barriers (release /
// acquire at cluster scope, so the global writes of one phase are visible to
// every CTA in the next), and the smallest levels and the coarsest LU run on
// the leader CTA alone with block barriers. Every cluster barrier is reached
// by all threads of the cluster: the branches around them depend only on
// values that are the same in every CTA (sizes, and res, flags and counters
// reduced over the cluster).
struct BlockTeam {
  __device__ __forceinline__ int tid() const { return threadIdx.x; }
  __device__ __forceinline__ int size() const { return blockDim.x; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ bool lead() const { return true; }
  static constexpr bool kMulti = false;
  // the same sum in every thread (fixed order)
  __device__ __forceinline__ double sum(double v, double *red) const { return block_sum(v, red); }
  __device__ __forceinline__ bool any(bool b) const { return __syncthreads_or(b) != 0; }
};

struct ClusterTeam {
  int rank, n;
  __device__ __forceinline__ int tid() const { return rank * (int)blockDim.x + (int)threadIdx.x; }
  __device__ __forceinline__ int size() const { return n * (int)blockDim.x; }
  __device__ __forceinline__ void sync() const { cooperative_groups::this_cluster().sync(); }
  __device__ __forceinline__ bool lead() const { return rank == 0; }
  static constexpr bool kMulti = true;
  // CTA partials in rank order: every thread adds the same values in the same
  // order. red[33] holds this CTA's partial until all CTAs have read it.
  __device__ double sum(double v, double *red) const {
    const double part = block_sum(v, red);
    if (threadIdx.x == 0) red[33] = part;
    sync();
    auto cl = cooperative_groups::this_cluster();
    double s = 0.0;
    for (int r = 0; r < n; ++r) s += *cl.map_shared_rank(red + 33, r);
    sync();
    return s;
  }
  __device__ bool any(bool b) const {
    __shared__ int s_any;
    const int mine = __syncthreads_or(b);
    if (threadIdx.x == 0) s_any = mine;
    sync();
    auto cl = cooperative_groups::this_cluster();
    int a = 0;
    for (int r = 0; r < n; ++r) a |= *cl.map_shared_rank(&s_any, r);
    sync();
    return a != 0;
  }
  // the leader's value of a flag in every thread (after the leader wrote it)
  __device__ int lead_value(const int *flag) const {
    const int v = *cooperative_groups::this_cluster().map_shared_rank(const_cast<int *>(flag), 0);
    sync();
    return v;
  }
};

// ----------------------------------------------------------------------------
// Regularized FD Jacobian (Eq. 12-13) in three passes that share work between
// neighbouring cells. Perturbing U_i in component m changes only the
// component-m reconstructions of cells i-1, i, i+1 (WENO3 is component-wise,
// ghost states copy the same component of the edge cell), hence only the
// fluxes of faces i-1..i+2 and the sources of cells i-1..i+1. So:
//   A  per cell k = -1..N: reconstructions of the base state and of the
//      three states with cell k-1, k or k+1 perturbed (same component);
//   B  per face f = 0..N: the base flux and the 8 fluxes with one of cells
//      f-2..f+1 perturbed in one component;
//   C  per block (j, i): R_j of the perturbed state from two face fluxes and
//      the Gauss source, minus the base R_j, over eps, plus alpha ||R_j||_1 I
//      on the diagonal.
// Each perturbed R_j is the same arithmetic on the same values as a full
// re-evaluation of the local residual, at a fraction of the cost.
// FP64 issue bounds the passes: about 510 instruction slots per cell for J3
// (744 with the candidate polynomials, full HLL averages and CUDA's divisions):
// 2^20 cells 1491 -> 1105 us, the 608-problem solve launch 443 -> 354 ms.

template <typename T>
struct JW {
  T *rec;  // [2 comps][4 variants][2: up, um][N+2], cell k at k+1
  T *flx;  // [9 variants][2 comps][N+1]
  int N;
  __device__ __forceinline__ T &r(int m, int v, int o, int k) const {
    return rec[((m * 4 + v) * 2 + o) * (N + 2) + (k + 1)];
  }
  __device__ __forceinline__ T &f(int w, int l, int face) const { return flx[(w * 2 + l) * (N + 1) + face]; }
};

template <typename T>
__device__ __forceinline__ JW<T> jw_view(double *base, int N) {
  JW<T> W;
  W.rec = reinterpret_cast<T *>(base);
  W.flx = W.rec + 16 * (size_t)(N + 2);
  W.N = N;
  return W;
}

// Component m of cell kk (ghosts included) of the state with interior cell
// ip perturbed by eps in component m (ip = -1: no perturbation).
template <typename T>
__device__ __forceinline__ T pval(const Geo &G, const double *U, int m, int kk, int ip, double eps, T eps_t) {
  const int N = G.N;
  if (kk >= 0 && kk < N) {
    T x = GeoT<T>::u(G, U, m * N + kk);
    return kk == ip ? x + eps_t : x;
  }
  const int e = kk < 0 ? 0 : N - 1;
  double He = U[e], Qe = U[N + e];
  if (e == ip) {
    if (m == 0) He += eps;
    else Qe += eps;
  }
  double Hg, Qg;
  if (kk < 0) ghost(G.bl, G.blh, G.blq, G.sf[0], He, Qe, Hg, Qg);
  else ghost(G.br, G.brh, G.brq, G.sf[N], He, Qe, Hg, Qg);
  return T(m == 0 ? Hg : Qg);
}

// Pass A. Variant v = 0: base; v = 1, 2, 3: cell k + v - 2 perturbed. One
// item forms the four variants of a cell and component: perturbing cell k-1
// (k+1) leaves the difference d0 (d1) and its smoothness term. Next to the
// boundary the ghost cells follow the perturbed edge cell; the differences
// kept are zero there (two ghost cells are equal), as in the base state.
template <typename T>
__device__ void jac_pass_a(const Geo &G, const double *U, double eps, const JW<T> &W, int first, int stride) {
  const int N = G.N, items = (N + 2) * 2;
  const T eps_t = T(eps);
  for (int it = first; it < items; it += stride) {
    const int m = it >= N + 2, k = it - m * (N + 2) - 1;
    T a, b, c, a1, b1, c1, a2, b2, c2, a3, b3, c3;  // window of the base state and what each variant has in its place
    if (k > 0 && k < N - 1) {
      a = GeoT<T>::u(G, U, m * N + k - 1);
      b = b1 = b3 = GeoT<T>::u(G, U, m * N + k);
      c = GeoT<T>::u(G, U, m * N + k + 1);
      a2 = a3 = a;
      c1 = c2 = c;
      a1 = a + eps_t;
      b2 = b + eps_t;
      c3 = c + eps_t;
    } else {
      auto at = [&](int kk, int ip) { return pval<T>(G, U, m, kk, ip, eps, eps_t); };
      a = at(k - 1, -1);
      b = at(k, -1);
      c = at(k + 1, -1);
      a1 = at(k - 1, k - 1);
      b1 = at(k, k - 1);
      c1 = at(k + 1, k - 1);
      a2 = at(k - 1, k);
      b2 = at(k, k);
      c2 = at(k + 1, k);
      a3 = at(k - 1, k + 1);
      b3 = at(k, k + 1);
      c3 = at(k + 1, k + 1);
    }
    // variant v has the difference (and smoothness) at the `kept` side of the base state
    const Slope<T> S0 = slope<T>(c - b), S1 = slope<T>(b - a);
    auto rec = [&](T va, T vb, T vc, bool keep0, bool keep1, T &vup, T &vum) {
      if constexpr (std::is_same<T, float>::value)
        weno3<float>(va, vb, vc, vup, vum);
      else
        weno3<T>(vb, keep0 ? S0 : slope<T>(vc - vb), keep1 ? S1 : slope<T>(vb - va), vup, vum);
    };
    T up, um;
    rec(a, b, c, true, true, up, um);
    W.r(m, 0, 0, k) = up;
    W.r(m, 0, 1, k) = um;
    if (k >= 1) {
      rec(a1, b1, c1, true, false, up, um);
      W.r(m, 1, 0, k) = up;
      W.r(m, 1, 1, k) = um;
    }
    if (k >= 0 && k < N) {
      rec(a2, b2, c2, false, false, up, um);
      W.r(m, 2, 0, k) = up;
      W.r(m, 2, 1, k) = um;
    }
    if (k < N - 1) {
      rec(a3, b3, c3, false, true, up, um);
      W.r(m, 3, 0, k) = up;
      W.r(m, 3, 1, k) = um;
    }
  }
}

// Reconstruction variant of cell kk under a perturbation of cell i.
__device__ __forceinline__ int rec_variant(int i, int kk) {
  int d = i - kk;
  return (d >= -1 && d <= 1) ? d + 2 : 0;
}

// Pass B, one face per item. Variant w = 0: base; w = 1 + 2p + m: cell
// f - 2 + p perturbed in component m. The left state comes from cell f-1
// (perturbed for p = 0, 1, 2), the right state from cell f (p = 1, 2, 3);
// the per-state HLL quantities of the base states serve all variants that do
// not perturb that side.
template <typename T, int FLUX>
__device__ void jac_pass_b(const Geo &G, const JW<T> &W, int first, int stride) {
  // The fused forms shorten the FP64 solve's chains: 608 problems of 4096 cells
  // 365 -> 361 ms.
  constexpr bool kFused = FLUX == NSWE_FLUX_HLL && std::is_same<T, double>::value;
  constexpr Sum kBase = kFused ? Sum::kFusedC : Sum::kRounded, kQ = kFused ? Sum::kFusedU : Sum::kRounded;
  const int N = G.N;
  const T g = GeoT<T>::g(G);
  for (int f = first; f <= N; f += stride) {
    const Face<T> fc = face<T>(GeoT<T>::isf(G, f), GeoT<T>::cgf(G, f), g);
    const FState<T> Lb = fstate<kBase>(W.r(0, 0, 1, f - 1), W.r(1, 0, 1, f - 1), fc);
    const FState<T> Rb = fstate<kBase>(W.r(0, 0, 0, f), W.r(1, 0, 0, f), fc);
    T F0, F1;
    num_flux<FLUX>(Lb, Rb, G.flux, F0, F1);
    W.f(0, 0, f) = F0;
    W.f(0, 1, f) = F1;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int i = f - 2 + p;
      if (i < 0 || i >= N) continue;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        // a Q perturbation (m = 1) leaves H, 1/H, c and the pressure term of
        // the base state
        FState<T> Ls = Lb, Rs = Rb;
        if (p <= 2)
          Ls = m == 0 ? fstate<Sum::kFusedC>(W.r(0, p + 1, 1, f - 1), Lb.Q, fc)
                      : fstate_q<kQ>(Lb, W.r(1, p + 1, 1, f - 1), fc);
        if (p >= 1)
          Rs = m == 0 ? fstate<Sum::kFusedC>(W.r(0, p, 0, f), Rb.Q, fc) : fstate_q<kQ>(Rb, W.r(1, p, 0, f), fc);
        num_flux<FLUX>(Ls, Rs, G.flux, F0, F1);
        const int w = 1 + 2 * p + m;
        W.f(w, 0, f) = F0;
        W.f(w, 1, f) = F1;
      }
    }
  }
}

// Flux variant at face `face` for a perturbation of cell i, component m.
__device__ __forceinline__ int flux_variant(int i, int m, int face) {
  int p = i - face + 2;
  return (p >= 0 && p <= 3) ? 1 + 2 * p + m : 0;
}

// Pass C, one cell j per item: the base R_j (written when Rout is given),
// then for each block k (cell i = j + k - hw) R_j of the state with U_i
// perturbed, from two face fluxes and the Gauss source, minus the base R_j,
// over eps, plus alpha ||R_j||_1 I on the diagonal. The regularisation uses
// Rreg when given (the FP64 residual of a mixed-precision step), else the
// pass's own base residual. Returns the partial sum of ||R_j||_1 of the
// cells that wrote R.
template <typename T>
__device__ double jac_pass_c(const Geo &G, int nb, double eps, double alpha, const JW<T> &W, const double *Rreg,
                             double *Rout, T *J, int first, int stride) {
  const int N = G.N, hw = (nb - 1) / 2;
  const T ieps = T(1.0) / T(eps);
  double acc = 0.0;
  for (int j = first; j < N; j += stride) {
    const SrcCell<T> sc = src_cell<T>(G, j);
    const T Sb =
        source_value(sc, source_at(sc, W.r(0, 0, 0, j - 1), W.r(0, 0, 0, j), W.r(0, 0, 1, j), W.r(0, 0, 1, j + 1)));
    const T R0 = W.f(0, 0, j + 1) - W.f(0, 0, j);
    const T R1 = W.f(0, 1, j + 1) - W.f(0, 1, j) - Sb;
    if (Rout) {
      Rout[j] = double(R0);
      Rout[N + j] = double(R1);
      acc += fabs(double(R0)) + fabs(double(R1));
    }
    // on the diagonal: v + alpha ||R_j||_1
    const T norm = Rreg ? T(alpha * (fabs(Rreg[j]) + fabs(Rreg[N + j]))) : fabs(R0) + fabs(R1);
    auto regularised = [&](T v) { return Rreg ? add_r(v, norm) : fma(T(alpha), norm, v); };
    for (int k = 0; k < nb; ++k) {
      const int i = j + k - hw;
      if (i < 0 || i >= N) {
#pragma unroll
        for (int e = 0; e < 4; ++e) J[(k * 4 + e) * N + j] = T(0.0);
        continue;
      }
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        T S = Sb;
        if (m == 0) {
          const int v0 = rec_variant(i, j - 1), v1 = rec_variant(i, j), v2 = rec_variant(i, j + 1);
          S = source_at(sc, W.r(0, v0, 0, j - 1), W.r(0, v1, 0, j), W.r(0, v1, 1, j), W.r(0, v2, 1, j + 1));
        }
        const int wr = flux_variant(i, m, j + 1), wl = flux_variant(i, m, j);
        const T P0 = W.f(wr, 0, j + 1) - W.f(wl, 0, j);
        const T d1 = W.f(wr, 1, j + 1) - W.f(wl, 1, j);
        const T P1 = m == 0 ? less_source(sc, d1, S) : d1 - S;
        T v0 = mul_r(P0 - R0, ieps), v1 = mul_r(P1 - R1, ieps);
        if (i == j) {
          if (m == 0) v0 = regularised(v0);
          else v1 = regularised(v1);
        }
        J[(k * 4 + 0 * 2 + m) * N + j] = v0;
        J[(k * 4 + 1 * 2 + m) * N + j] = v1;
      }
    }
  }
  return acc;
}

// ----------------------------------------------------------------------------
// FP64 residual in three passes over a compact workspace (the residual of a
// mixed-precision Newton step): reconstructions once per cell, fluxes once
// per face, then sources and differences per cell. Same arithmetic as the
// base variant of the Jacobian passes.
struct RW {
  double *rec;  // [2 comps][2: up, um][N+2], cell k at k+1
  double *flx;  // [2 comps][N+1]
  int N;
  __device__ __forceinline__ double &r(int m, int o, int k) const { return rec[(m * 2 + o) * (N + 2) + (k + 1)]; }
  __device__ __forceinline__ double &f(int l, int face) const { return flx[l * (N + 1) + face]; }
};

// FP32 copies of a mixed-precision level (Geo::U32 and the geometry): 10 N + 2
// floats placed after the FP64 residual's workspace, within jw_doubles(N).
__host__ __device__ inline size_t f32_area_offset(size_t N) {
  const size_t rw = (jw_doubles(N) / 2 + 2) / 2 * 2;
  return (rw + 4 * (N + 2) + 2 * (N + 1) + 3) / 4 * 4;
}

// Points G's FP32 copies at their place in the Jacobian workspace jw.
__device__ __forceinline__ float *attach_f32(Geo &G, double *jw) {
  float *A = reinterpret_cast<float *>(jw + f32_area_offset((size_t)G.N));
  const int N = G.N;
  G.U32 = A;
  G.isf32 = A + 2 * N;
  G.cgf32 = G.isf32 + N + 1;
  G.igq32 = G.cgf32 + N + 1;
  G.gq32 = G.igq32 + 2 * N;
  G.g32 = float(G.g);
  G.hdx32 = 0.5f * float(G.dx);
  return A;
}

// Writes the FP32 copies of state U and of G's geometry into A (attach_f32's
// layout), items strided.
__device__ void fill_f32(const Geo &G, const double *U, float *A, int first, int stride) {
  const int N = G.N;
  float *U32 = A, *isf = A + 2 * N, *cgf = isf + N + 1, *igq = cgf + N + 1, *gq = igq + 2 * N;
  for (int t = first; t < 4 * N; t += stride) {
    if (t < 2 * N) {
      U32[t] = float(U[t]);
      igq[t] = float(G.igq[t]);
    }
    if (t <= N) {
      isf[t] = float(G.isf[t]);
      cgf[t] = float(G.cgf[t]);
    }
    gq[t] = float(G.gq[2 * N + t]);  // sigma_x and b_x planes
  }
}

// Placed after the FP32 Jacobian workspace of the same level.
__device__ __forceinline__ RW rw_view(double *jw, int N) {
  RW W;
  W.rec = jw + (jw_doubles((size_t)N) / 2 + 2) / 2 * 2;
  W.flx = W.rec + 4 * (size_t)(N + 2);
  W.N = N;
  return W;
}

__device__ void res_pass_a(const Geo &G, const double *U, const RW &W, int first, int stride) {
  const int N = G.N, items = (N + 2) * 2;
  for (int it = first; it < items; it += stride) {
    const int k = it % (N + 2) - 1, m = it / (N + 2);
    double up, um;
    weno3<double>(pval<double>(G, U, m, k - 1, -1, 0.0, 0.0), pval<double>(G, U, m, k, -1, 0.0, 0.0),
                  pval<double>(G, U, m, k + 1, -1, 0.0, 0.0), up, um);
    W.r(m, 0, k) = up;
    W.r(m, 1, k) = um;
  }
}

template <int FLUX>
__device__ void res_pass_b(const Geo &G, const RW &W, int first, int stride) {
  for (int f = first; f <= G.N; f += stride) {
    double F0, F1;
    const Face<double> fc = face(G.isf[f], G.cgf[f], G.g);
    num_flux<FLUX>(fstate<Sum::kRounded>(W.r(0, 1, f - 1), W.r(1, 1, f - 1), fc),
                   fstate<Sum::kRounded>(W.r(0, 0, f), W.r(1, 0, f), fc), G.flux, F0, F1);
    W.f(0, f) = F0;
    W.f(1, f) = F1;
  }
}

__device__ double res_pass_c(const Geo &G, const RW &W, double *R, int first, int stride) {
  const int N = G.N;
  double acc = 0.0;
  for (int j = first; j < N; j += stride) {
    const double S = source_at<double>(src_cell<double>(G, j), W.r(0, 0, j - 1), W.r(0, 0, j), W.r(0, 1, j), W.r(0, 1, j + 1));
    const double R0 = W.f(0, j + 1) - W.f(0, j);
    const double R1 = W.f(1, j + 1) - W.f(1, j) - S;
    R[j] = R0;
    R[N + j] = R1;
    acc += fabs(R0) + fabs(R1);
  }
  return acc;
}

// Derived geometry of every level (1/sigma and sqrt(g/sigma) at faces, 1/sigma
// at the Gauss points), items strided over the finest level's faces.
__device__ void geom_derive_items(const ProbDev &P, int first, int stride) {
  for (int l = 0; l < P.levels; ++l) {
    const LevelDev &Lv = P.lev[l];
    const int N = Lv.N;
    double *isf = Lv.gd, *cgf = isf + N + 1, *igq = cgf + N + 1;
    for (int t = first; t <= N; t += stride) {
      isf[t] = 1.0 / Lv.sf[t];
      cgf[t] = sqrt(P.g * isf[t]);
    }
    for (int t = first; t < 2 * N; t += stride) {
      const int q = t / N, j = t % N;
      igq[t] = 1.0 / Lv.gq[(0 * 2 + q) * N + j];
    }
  }
}

// Inverse of the diagonal 2x2 blocks of cells first, first + stride, .. < end, times -omega: the factor with which the
// smoother applies them.
template <typename T>
__device__ void dinv_cells(int N, int nb, const T *J, T *Dinv, double omega, int first, int end, int stride) {
  const int hw = (nb - 1) / 2;
  for (int j = first; j < end; j += stride) {
    T a = J[(hw * 4 + 0) * N + j], b = J[(hw * 4 + 1) * N + j];
    T c = J[(hw * 4 + 2) * N + j], d = J[(hw * 4 + 3) * N + j];
    const T s = T(-omega) * rcp_t(fma(a, d, -(b * c)));
    Dinv[0 * N + j] = d * s;
    Dinv[1 * N + j] = -b * s;
    Dinv[2 * N + j] = -c * s;
    Dinv[3 * N + j] = a * s;
  }
}

// Galerkin coarse operator (Eq. 17): sums of fine blocks over aggregate pairs.
// An interior aggregate (2j, 2j+1) of a three-block fine level has the
// coarse blocks J_-1(2j), J_0(2j) + J_+1(2j) + J_-1(2j+1) + J_0(2j+1) and
// J_+1(2j+1), summed in the order of the general loop below.
template <typename T>
__device__ void coarse_op_cells(int Nf, int nbf, const T *Jf, int Nc, T *Jc, int first, int end, int stride) {
  const int hf = (nbf - 1) / 2;
  for (int j = first; j < end; j += stride) {
    if (nbf == 3 && j > 0 && 2 * j + 2 < Nf) {
      const int x0 = 2 * j, x1 = 2 * j + 1;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        Jc[(0 * 4 + e) * Nc + j] = Jf[(0 * 4 + e) * Nf + x0];
        Jc[(1 * 4 + e) * Nc + j] =
            ((Jf[(1 * 4 + e) * Nf + x0] + Jf[(2 * 4 + e) * Nf + x0]) + Jf[(0 * 4 + e) * Nf + x1]) +
            Jf[(1 * 4 + e) * Nf + x1];
        Jc[(2 * 4 + e) * Nc + j] = Jf[(2 * 4 + e) * Nf + x1];
      }
      continue;
    }
    T a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0}, a2[4] = {0, 0, 0, 0};
    for (int a = 0; a < 2; ++a) {
      int xi = 2 * j + a;
      if (xi >= Nf) break;
      for (int k = 0; k < nbf; ++k) {
        int eta = xi + k - hf;
        if (eta < 0 || eta >= Nf) continue;
        int kc = eta / 2 - j + 1;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          T v = Jf[(k * 4 + e) * Nf + xi];
          if (kc == 0) a0[e] += v;
          else if (kc == 1) a1[e] += v;
          else a2[e] += v;
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Jc[(0 * 4 + e) * Nc + j] = a0[e];
      Jc[(1 * 4 + e) * Nc + j] = a1[e];
      Jc[(2 * 4 + e) * Nc + j] = a2[e];
    }
  }
}

// Block SOR update (Eq. 19) of the cells of one colour (j mod C == col),
// x := (1 - omega) x - omega D^-1 r, applied `reps` times in a row. Cells of
// one colour do not couple, so a repeated visit of the same colour sees the
// same neighbour values: the correction t = -omega D^-1 r is computed once
// and the relaxation applied reps times, which is the sequence of reps
// separate passes. -omega is in the stored inverse (dinv_cells), so a visit
// costs 14 FP64 instructions with two neighbours. zero: dU is all zero (the
// first pass after a restriction), and the neighbour sums are left out.
template <typename T>
__device__ void sor_colour(int N, int nb, const T *J, const T *Dinv, const T *R, T *dU, double omega_d, int C,
                           int col, int reps, bool zero, int first, int stride) {
  const T keep = T(1.0) - T(omega_d);
  const int hw = (nb - 1) / 2;
  for (int j = col + C * first; j < N; j += C * stride) {
    T r0 = R[j], r1 = R[N + j];
    T x0 = T(0.0), x1 = T(0.0);
    if (!zero) {
      for (int k = 0; k < nb; ++k) {
        int i = j + k - hw;
        if (k == hw || i < 0 || i >= N) continue;
        const T y0 = dU[i], y1 = dU[N + i];
        r0 = fma(J[(k * 4 + 0) * N + j], y0, r0);
        r0 = fma(J[(k * 4 + 1) * N + j], y1, r0);
        r1 = fma(J[(k * 4 + 2) * N + j], y0, r1);
        r1 = fma(J[(k * 4 + 3) * N + j], y1, r1);
      }
      x0 = dU[j];
      x1 = dU[N + j];
    }
    const T t0 = fma(Dinv[0 * N + j], r0, Dinv[1 * N + j] * r1);
    const T t1 = fma(Dinv[2 * N + j], r0, Dinv[3 * N + j] * r1);
    for (int r = 0; r < reps; ++r) {
      x0 = fma(keep, x0, t0);
      x1 = fma(keep, x1, t1);
    }
    dU[j] = x0;
    dU[N + j] = x1;
  }
}

// Defect restriction (Eq. 17) and zero coarse correction.
template <typename T>
__device__ void restrict_cells(int Nf, int nb, const T *J, const T *R, const T *dU, int Nc, T *Rc, T *dUc,
                               int first, int stride) {
  const int hw = (nb - 1) / 2;
  for (int j = first; j < Nc; j += stride) {
    T s0 = T(0.0), s1 = T(0.0);
    for (int a = 0; a < 2; ++a) {
      int xi = 2 * j + a;
      if (xi >= Nf) break;
      T r0 = R[xi], r1 = R[Nf + xi];
      for (int k = 0; k < nb; ++k) {
        int eta = xi + k - hw;
        if (eta < 0 || eta >= Nf) continue;
        T x0 = dU[eta], x1 = dU[Nf + eta];
        r0 = fma(J[(k * 4 + 0) * Nf + xi], x0, r0);
        r0 = fma(J[(k * 4 + 1) * Nf + xi], x1, r0);
        r1 = fma(J[(k * 4 + 2) * Nf + xi], x0, r1);
        r1 = fma(J[(k * 4 + 3) * Nf + xi], x1, r1);
      }
      s0 += r0;
      s1 += r1;
    }
    Rc[j] = s0;
    Rc[Nc + j] = s1;
    dUc[j] = T(0.0);
    dUc[Nc + j] = T(0.0);
  }
}

// Prolongation (Eq. 18).
template <typename T>
__device__ void prolong_cells(int Nf, T *dU, int Nc, const T *dUc, int first, int stride) {
  for (int xi = first; xi < Nf; xi += stride) {
    dU[xi] += dUc[xi / 2];
    dU[Nf + xi] += dUc[Nc + xi / 2];
  }
}

// App. A (Eq. A.2): fine averages from the coarse quadratic; the domain ends
// use the coarse level's ghost states.
__device__ void interp_cells(const Geo &Gc, const double *Uc, double *Uf, int first, int stride) {
  const int Nc = Gc.N, Nf = 2 * Nc;
  const double *Hc = Uc, *Qc = Uc + Nc;
  for (int c = first; c < Nc; c += stride) {
    double hm, qm, hp, qp;
    double h0 = Hc[c], q0 = Qc[c];
    if (c > 0) {
      hm = Hc[c - 1];
      qm = Qc[c - 1];
    } else {
      ghost(Gc.bl, Gc.blh, Gc.blq, Gc.sf[0], Hc[0], Qc[0], hm, qm);
    }
    if (c < Nc - 1) {
      hp = Hc[c + 1];
      qp = Qc[c + 1];
    } else {
      ghost(Gc.br, Gc.brh, Gc.brq, Gc.sf[Nc], Hc[Nc - 1], Qc[Nc - 1], hp, qp);
    }
    Uf[2 * c] = hm / 8.0 + h0 - hp / 8.0;
    Uf[2 * c + 1] = -hm / 8.0 + h0 + hp / 8.0;
    Uf[Nf + 2 * c] = qm / 8.0 + q0 - qp / 8.0;
    Uf[Nf + 2 * c + 1] = -qm / 8.0 + q0 + qp / 8.0;
  }
}

// ----------------------------------------------------------------------------
// Coarsest direct solve: LU with partial pivoting (ties to the lowest row) of
// the block-banded system, unknown u = 2j + m, in LAPACK-style band storage
// (kl sub-diagonals, 2 kl super-diagonals after fill-in). A banded matrix
// keeps its zeros outside the band through the elimination, so this performs
// the same pivots and updates as a dense LU. The elimination is a sequence of
// n pivot steps; one warp runs it, its lanes covering the entries of a step
// (the kl multipliers, the kl x 2kl updated entries, the 2kl back-substitution
// updates). GB300 issues an FP64 warp instruction at the same cost whatever
// its active lanes, so spreading each step over lanes, rather than running it
// on one thread, divides the FP64 work of the solve by about the band width.
// Every entry sees the same operations in the same order as in a serial
// elimination.

template <typename T>
struct Band {
  T *ab;    // [ldab][n]
  int *piv;      // [n]
  T *x;     // [n]
  T *rinv;  // [n] reciprocals of the pivots
  int n, kl, ldab;
  __device__ __forceinline__ T &A(int r, int c) const { return ab[(2 * kl + r - c) * n + c]; }
};

// Order key of |a|: for non-negative floating-point values the bit patterns,
// read as unsigned integers, are ordered as the values (NaN keys are dropped
// to 0, so a NaN never wins a pivot search).
__device__ __forceinline__ unsigned long long abs_key(double a) {
  return a == a ? (unsigned long long)(__double_as_longlong(a) & 0x7fffffffffffffffLL) : 0ull;
}

// Pivot steps k0 .. k1 - 1 of the factorisation by warp 0 (lanes 0..31, all of
// them calling). Returns true if a pivot was exactly zero.
template <typename T>
__device__ bool band_lu_warp(const Band<T> &B, int k0, int k1) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int n = B.n, kl = B.kl, w2 = 2 * kl, upd = kl * w2;
  bool sing = false;
  for (int k = k0; k < k1; ++k) {
    const int imax = min(n - 1, k + kl), cmax = min(n - 1, k + w2);
    // Pivot: the first row of largest |A(i, k)|, i = k..imax (kl <= 7).
    unsigned long long key = 0;
    int p = 0x7fffffff;
    if (lane <= kl && k + lane <= imax) {
      key = abs_key(B.A(k + lane, k));
      p = k + lane;
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const unsigned long long ok = __shfl_xor_sync(FULL, key, o);
      const int op = __shfl_xor_sync(FULL, p, o);
      if (ok > key || (ok == key && op < p)) {
        key = ok;
        p = op;
      }
    }
    p = __shfl_sync(FULL, p, 0);
    if (lane == 0) B.piv[k] = p;
    if (p != k)
      for (int c = k + lane; c <= cmax; c += 32) {
        const T t = B.A(k, c);
        B.A(k, c) = B.A(p, c);
        B.A(p, c) = t;
      }
    __syncwarp();
    // One division for 1/d (lane 0) and the multipliers A(k+i, k)/d (lane i).
    const T d = B.A(k, k);
    const bool mrow = lane >= 1 && lane <= kl && k + lane <= imax;
    const T rd = rcp_t(d);
    const T q = lane == 0 ? rd : (mrow ? fast_div(B.A(k + lane, k), d, rd) : T(0.0));
    if (lane == 0) {
      B.rinv[k] = q;
      if (d == T(0.0)) sing = true;
    }
    if (mrow) B.A(k + lane, k) = q;
    // A(k+i, k+c) -= l_i A(k, k+c), i = 1..kl, c = 1..2kl.
    for (int e0 = 0; e0 < upd; e0 += 32) {
      const int e = e0 + lane, i = 1 + e / w2, c = 1 + e % w2;
      const T l = __shfl_sync(FULL, q, min(i, 31));
      if (e < upd && k + i <= imax && k + c <= cmax) B.A(k + i, k + c) -= l * B.A(k, k + c);
    }
    __syncwarp();
  }
  return __shfl_sync(FULL, sing, 0);
}

// x (B.x, length n) := A^{-1} x with the stored factors, by warp 0. The back
// substitution is column oriented: once x_i is known, the rows above it take
// their A(r, i) x_i terms, so each row subtracts its terms from the farthest
// column to the nearest, the order of the row-oriented loop.
template <typename T>
__device__ void band_lu_solve_warp(const Band<T> &B) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int n = B.n, kl = B.kl;
  for (int k = 0; k < n; ++k) {
    const int p = B.piv[k];
    if (p != k && lane == 0) {
      const T t = B.x[k];
      B.x[k] = B.x[p];
      B.x[p] = t;
    }
    __syncwarp();
    const T xk = B.x[k];
    if (lane >= 1 && lane <= kl && k + lane < n) B.x[k + lane] -= B.A(k + lane, k) * xk;
    __syncwarp();
  }
  for (int i = n - 1; i >= 0; --i) {
    T xi = T(0.0);
    if (lane == 0) {
      xi = B.x[i] * B.rinv[i];
      B.x[i] = xi;
    }
    xi = __shfl_sync(FULL, xi, 0);
    const int r = i - lane;
    if (lane >= 1 && lane <= 2 * kl && r >= 0) B.x[r] -= B.A(r, i) * xi;
    __syncwarp();
  }
}

// FP32 instantiation: one thread runs the elimination with the active rows in
// registers (a window of kl+1 rows). FP32 instructions issue at full rate, so
// the serial recurrence is shorter than its warp-parallel form, whose
// shuffles and warp barriers then dominate.
template <int KL, typename T>
__device__ bool band_lu_serial(const Band<T> &B) {
  constexpr int W = 2 * KL + 1;
  const int n = B.n;
  T w[KL + 1][W];
#pragma unroll
  for (int i = 0; i <= KL; ++i)
#pragma unroll
    for (int c = 0; c < W; ++c) w[i][c] = (i < n && c < n) ? B.A(i, c) : T(0.0);
  bool sing = false;
  for (int k = 0; k < n; ++k) {
    int p = 0;
    T best = fabs(w[0][0]);
#pragma unroll
    for (int i = 1; i <= KL; ++i)
      if (k + i < n && fabs(w[i][0]) > best) {
        best = fabs(w[i][0]);
        p = i;
      }
    B.piv[k] = k + p;
#pragma unroll
    for (int i = 1; i <= KL; ++i)
      if (p == i)
#pragma unroll
        for (int c = 0; c < W; ++c) {
          T t = w[0][c];
          w[0][c] = w[i][c];
          w[i][c] = t;
        }
    const T d = w[0][0];
    if (d == T(0.0)) sing = true;
    B.rinv[k] = T(1.0) / d;
#pragma unroll
    for (int i = 1; i <= KL; ++i)
      if (k + i < n) {
        const T l = w[i][0] / d;
        B.A(k + i, k) = l;
#pragma unroll
        for (int c = 1; c < W; ++c) w[i][c] -= l * w[0][c];
      }
#pragma unroll
    for (int c = 0; c < W; ++c)
      if (k + c < n) B.A(k, k + c) = w[0][c];
    // Slide the window one row and one column.
#pragma unroll
    for (int i = 0; i < KL; ++i) {
#pragma unroll
      for (int c = 0; c < W - 1; ++c) w[i][c] = w[i + 1][c + 1];
      w[i][W - 1] = T(0.0);
    }
    const int r = k + KL + 1;
#pragma unroll
    for (int c = 0; c < W; ++c) w[KL][c] = (r < n && k + 1 + c < n) ? B.A(r, k + 1 + c) : T(0.0);
  }
  return sing;
}

// The same serial factorisation working on the band storage in place (any
// kl); used for the 5-block Jacobian of a direct solve on the coarsest level.
template <typename T>
__device__ bool band_lu_serial_smem(const Band<T> &B) {
  const int n = B.n, kl = B.kl;
  bool sing = false;
  for (int k = 0; k < n; ++k) {
    const int imax = min(n - 1, k + kl), cmax = min(n - 1, k + 2 * kl);
    int p = k;
    for (int i = k + 1; i <= imax; ++i)
      if (fabs(B.A(i, k)) > fabs(B.A(p, k))) p = i;
    B.piv[k] = p;
    if (p != k)
      for (int c = k; c <= cmax; ++c) {
        T t = B.A(k, c);
        B.A(k, c) = B.A(p, c);
        B.A(p, c) = t;
      }
    const T d = B.A(k, k);
    if (d == T(0.0)) sing = true;
    B.rinv[k] = T(1.0) / d;
    for (int i = k + 1; i <= imax; ++i) {
      const T l = B.A(i, k) / d;
      B.A(i, k) = l;
      for (int c = k + 1; c <= cmax; ++c) B.A(i, c) -= l * B.A(k, c);
    }
  }
  return sing;
}

// x (B.x, length n) := A^{-1} x with the stored factors (one thread).
template <int KL, typename T>
__device__ void band_lu_solve_serial(const Band<T> &B) {
  constexpr int W = 2 * KL + 1;
  const int n = B.n;
  T X[KL + 1];
#pragma unroll
  for (int i = 0; i <= KL; ++i) X[i] = i < n ? B.x[i] : T(0.0);
  for (int k = 0; k < n; ++k) {
    const int p = B.piv[k] - k;
#pragma unroll
    for (int i = 1; i <= KL; ++i)
      if (p == i) {
        T t = X[0];
        X[0] = X[i];
        X[i] = t;
      }
#pragma unroll
    for (int i = 1; i <= KL; ++i)
      if (k + i < n) X[i] -= B.A(k + i, k) * X[0];
    B.x[k] = X[0];
#pragma unroll
    for (int i = 0; i < KL; ++i) X[i] = X[i + 1];
    X[KL] = (k + KL + 1 < n) ? B.x[k + KL + 1] : T(0.0);
  }
  T Y[W - 1];  // Y[c] = x[i + 1 + c]
#pragma unroll
  for (int c = 0; c < W - 1; ++c) Y[c] = T(0.0);
  for (int i = n - 1; i >= 0; --i) {
    T s = B.x[i];
#pragma unroll
    for (int c = W - 2; c >= 1; --c)
      if (i + 1 + c < n) s -= B.A(i, i + 1 + c) * Y[c];
    if (i + 1 < n) s -= B.A(i, i + 1) * Y[0];
    const T xi = s * B.rinv[i];
    B.x[i] = xi;
#pragma unroll
    for (int c = W - 2; c >= 1; --c) Y[c] = Y[c - 1];
    Y[0] = xi;
  }
}

__shared__ int s_sing;

// Assemble the band matrix from J (all threads).
template <typename T>
__device__ void band_assemble(Band<T> &B, int N, int nb, const T *J) {
  const int hw = (nb - 1) / 2;
  B.n = 2 * N;
  B.kl = 2 * hw + 1;
  B.ldab = 3 * B.kl + 1;
  const int n = B.n;
  if (threadIdx.x == 0) s_sing = 0;
  for (int t = threadIdx.x; t < B.ldab * n; t += blockDim.x) B.ab[t] = T(0.0);
  __syncthreads();
  for (int t = threadIdx.x; t < N * nb * 4; t += blockDim.x) {
    int j = t % N, ke = t / N, k = ke / 4, e = ke % 4, l = e / 2, m = e % 2;
    int i = j + k - hw;
    if (i < 0 || i >= N) continue;
    B.A(2 * j + l, 2 * i + m) = J[(k * 4 + e) * N + j];
  }
  __syncthreads();
}

// Pivot steps k0 .. k1 - 1 of the assembled matrix by the calling warp (in
// FP32 its first thread runs all of them with the first). Sets s_sing if a
// pivot was exactly zero.
template <typename T>
__device__ void band_lu_steps(const Band<T> &B, int k0, int k1) {
  bool sing = false;
  if constexpr (std::is_same<T, double>::value) {
    sing = band_lu_warp<T>(B, k0, k1);
  } else {
    if (k0 == 0 && k1 > 0 && (threadIdx.x & 31) == 0)
      sing = B.kl == 3 ? band_lu_serial<3, T>(B) : band_lu_serial_smem<T>(B);
    __syncwarp();
  }
  if (sing && (threadIdx.x & 31) == 0) s_sing = 1;
}

// Assemble (all threads), then factor (warp 0). Returns true if a pivot was
// exactly zero (all threads).
template <typename T>
__device__ bool band_factor(Band<T> &B, int N, int nb, const T *J) {
  band_assemble(B, N, nb, J);
  if (threadIdx.x < 32) band_lu_steps(B, 0, B.n);
  __syncthreads();
  return s_sing != 0;
}

// dU = -J^{-1} R with the stored factors (warp 0 solves in FP64, thread 0 in
// FP32; all threads call).
template <typename T>
__device__ void band_solve(const Band<T> &B, int N, const T *R, T *dU) {
  for (int t = threadIdx.x; t < N; t += blockDim.x) {
    B.x[2 * t] = -R[t];
    B.x[2 * t + 1] = -R[N + t];
  }
  __syncthreads();
  if constexpr (std::is_same<T, double>::value) {
    if (threadIdx.x < 32) band_lu_solve_warp<T>(B);
  } else if (threadIdx.x == 0) {
    if (B.kl == 3) band_lu_solve_serial<3, T>(B);
    else band_lu_solve_serial<5, T>(B);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < N; t += blockDim.x) {
    dU[t] = B.x[2 * t];
    dU[N + t] = B.x[2 * t + 1];
  }
  __syncthreads();
}

// ----------------------------------------------------------------------------
// Multigrid hierarchy view: level l0 (the system being solved) uses the
// caller's J/R/dU, levels l0+1..L the problem's workspace.
// In the FP32 instantiation the workspace arrays (sized for FP64) hold FP32
// values.
template <typename T>
struct MG {
  int l0, L;
  int N[NSWE_MAX_LEVELS], nb[NSWE_MAX_LEVELS];
  T *J[NSWE_MAX_LEVELS], *Dinv[NSWE_MAX_LEVELS], *R[NSWE_MAX_LEVELS], *dU[NSWE_MAX_LEVELS];
};

template <typename T>
__device__ void mg_bind(MG<T> &mg, const ProbDev &P, int l0, int nb0, const T *J, const T *R, T *dU) {
  mg.l0 = l0;
  mg.L = P.levels - 1;
  for (int l = l0; l <= mg.L; ++l) {
    mg.N[l] = P.lev[l].N;
    mg.nb[l] = (l == l0) ? nb0 : 3;
    mg.J[l] = (l == l0) ? const_cast<T *>(J) : reinterpret_cast<T *>(P.lev[l].J);
    mg.R[l] = (l == l0) ? const_cast<T *>(R) : reinterpret_cast<T *>(P.lev[l].R);
    mg.dU[l] = (l == l0) ? dU : reinterpret_cast<T *>(P.lev[l].dU);
    mg.Dinv[l] = reinterpret_cast<T *>(P.lev[l].Dinv);
  }
}

// ----------------------------------------------------------------------------
// Legs: the smoothing of one level with the restriction behind it (down) or
// the prolongation before it (up) as one pass without barriers. A warp takes
// a tile of 16 cell pairs, two lanes per pair (one per component), holds the
// pairs' operator rows, right-hand side and correction in registers and runs
// all colour passes on them, neighbours' values by shuffles. Values spoil from
// the tile's edges by one cell per pass: with at most five passes (two
// symmetric steps of the two-colour smoother) and the restriction, 3 pairs on
// either side, so tiles overlap by 6 pairs and each writes its inner ones; at
// the domain's ends nothing spoils. What a tile reads is never what another
// writes: a leg's result goes to another buffer than its source.
// Why: on few SMs a pass is a barrier (0.2 us in a cluster), a trip to L2 for
// operator and correction (0.4 us) and 14 FP64 instructions of 64 cycles; a
// leg pays the first two once instead of six times and, with two lanes per
// cell, 7 instructions per pass, for 1.6 times the arithmetic. A full batch,
// one block per problem, is bound by the FP64 pipe and smooths pass by pass.
// Cells see the operations of sor_colour, restrict_cells and prolong_cells in
// their order.
// GB300: a 4096-cell solve on 16 CTAs 77.3 -> 69.4 ms.
constexpr int kLegPairs = 16, kLegOwn = 10, kLegHalo = 3, kLegSteps = 2;

__host__ __device__ inline int leg_tiles(int N) {
  return N / 2 <= kLegPairs ? 1 : (N / 2 - kLegPairs + kLegOwn - 1) / kLegOwn + 1;
}
// Whether a level is smoothed by legs.
__host__ __device__ inline bool leg_level(int nb, const nswe_params &prm) {
  return nb == 3 && prm.nu1 >= 1 && prm.nu1 <= kLegSteps && prm.nu2 >= 1 && prm.nu2 <= kLegSteps;
}

// One tile. src: the correction on entry (null: zero). Down: Rc receives the
// restricted defect. UP: dUc, the coarse correction, is added first.
template <typename T, bool UP>
__device__ __forceinline__ void leg_tile(int N, const T *J, const T *Dinv, const T *R, const T *src, T *dst,
                                         const T *dUc, T *Rc, int steps, T keep, int tile, int tiles) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, p = lane >> 1, c = lane & 1, pairs = N / 2;
  const int P = kLegOwn * tile + p, je = 2 * P, jo = je + 1;
  const bool in = P < pairs;
  auto blk = [&](int k, int q, int j, bool on) { return on ? J[(k * 4 + 2 * c + q) * N + j] : T(0.0); };
  const bool left = in && je > 0, right = in && jo < N - 1;
  const T em0 = blk(0, 0, je, left), em1 = blk(0, 1, je, left), ep0 = blk(2, 0, je, in), ep1 = blk(2, 1, je, in);
  const T om0 = blk(0, 0, jo, in), om1 = blk(0, 1, jo, in), op0 = blk(2, 0, jo, right), op1 = blk(2, 1, jo, right);
  auto at = [&](const T *A, int i) { return in ? A[i] : T(0.0); };
  const T ed0 = at(Dinv, 2 * c * N + je), ed1 = at(Dinv, (2 * c + 1) * N + je);
  const T od0 = at(Dinv, 2 * c * N + jo), od1 = at(Dinv, (2 * c + 1) * N + jo);
  const T re = at(R, c * N + je), ro = at(R, c * N + jo);
  T xe = T(0.0), xo = T(0.0);
  if (src) {
    xe = at(src, c * N + je);
    xo = at(src, c * N + jo);
  }
  if (UP) {
    const T xc = at(dUc, c * pairs + P);
    xe += xc;
    xo += xc;
  }
  // both components of a lane's value and of the value of the pair before / after it
  auto both = [&](T v, int pp, T &v0, T &v1) {
    const int at0 = 2 * min(max(pp, 0), kLegPairs - 1);
    v0 = __shfl_sync(FULL, v, at0);
    v1 = __shfl_sync(FULL, v, at0 + 1);
  };
  T a0, a1, b0, b1;  // neighbours before and after
  auto relax = [&](T r, T d0, T d1, T x, int reps) {
    const T other = __shfl_xor_sync(FULL, r, 1);
    const T r0 = c ? other : r, r1 = c ? r : other;
    const T t = fma(d0, r0, d1 * r1);
    x = fma(keep, x, t);
    return reps == 2 ? fma(keep, x, t) : x;
  };
  for (int v = 0; v <= 2 * steps; ++v) {
    const int reps = v == 0 || v == 2 * steps ? 1 : 2;
    if ((v & 1) == 0) {
      T r = re;
      if (UP || src || v > 0) {
        both(xo, p - 1, a0, a1);
        both(xo, p, b0, b1);
        r = fma(ep1, b1, fma(ep0, b0, fma(em1, a1, fma(em0, a0, r))));
      }
      xe = relax(r, ed0, ed1, xe, reps);
    } else {
      both(xe, p, a0, a1);
      both(xe, p + 1, b0, b1);
      const T r = fma(op1, b1, fma(op0, b0, fma(om1, a1, fma(om0, a0, ro))));
      xo = relax(r, od0, od1, xo, reps);
    }
  }
  const bool own = in && (p >= kLegHalo || tile == 0) && (p < kLegHalo + kLegOwn || tile == tiles - 1);
  if (own) {
    dst[c * N + je] = xe;
    dst[c * N + jo] = xo;
  }
  if (!UP) {
    T l0, l1, e0, e1, o0, o1, n0, n1;
    both(xo, p - 1, l0, l1);
    both(xe, p, e0, e1);
    both(xo, p, o0, o1);
    both(xe, p + 1, n0, n1);
    const T ec0 = blk(1, 0, je, in), ec1 = blk(1, 1, je, in), oc0 = blk(1, 0, jo, in), oc1 = blk(1, 1, jo, in);
    const T se = fma(ep1, o1, fma(ep0, o0, fma(ec1, e1, fma(ec0, e0, fma(em1, l1, fma(em0, l0, re))))));
    const T so = fma(op1, n1, fma(op0, n0, fma(oc1, o1, fma(oc0, o0, fma(om1, e1, fma(om0, e0, ro))))));
    if (own) Rc[c * pairs + P] = se + so;
  }
}

// The leg's tiles `warp`, `warp` + warps, ...
template <typename T, bool UP>
__device__ void leg(int N, const T *J, const T *Dinv, const T *R, const T *src, T *dst, const T *dUc, T *Rc,
                    int steps, double omega, int warp, int warps) {
  const int tiles = leg_tiles(N);
  for (int t = warp; t < tiles; t += warps)
    leg_tile<T, UP>(N, J, Dinv, R, src, dst, dUc, Rc, steps, T(1.0) - T(omega), t, tiles);
}

// Where the up leg of a level leaves its correction: beside the level's
// operator in its storage (20 N values of FP64, of which J3 takes 12 N and a
// mixed step's right-hand side 2 N). The other levels' stays in dU.
template <typename T>
__device__ __forceinline__ T *leg_out(T *J, int N) {
  return J + 14 * (size_t)N;
}

// Coarse operators of the levels below l0 and diagonal inverses, block `part`
// of `parts`: its share of the coarsest cells and the cells below them on
// every level, which need nothing from outside.
template <typename T>
__device__ void mg_setup_part(const MG<T> &mg, double omega, int part, int parts) {
  const int NL = mg.N[mg.L], c0 = NL * part / parts, c1 = NL * (part + 1) / parts;
  for (int l = mg.l0 + 1; l <= mg.L; ++l) {
    const int sh = mg.L - l;
    coarse_op_cells(mg.N[l - 1], mg.nb[l - 1], mg.J[l - 1], mg.N[l], mg.J[l], (c0 << sh) + (int)threadIdx.x, c1 << sh,
                    (int)blockDim.x);
    __syncthreads();
  }
  for (int l = mg.l0; l < mg.L; ++l) {
    const int sh = mg.L - l;
    dinv_cells(mg.N[l], mg.nb[l], mg.J[l], mg.Dinv[l], omega, (c0 << sh) + (int)threadIdx.x, c1 << sh,
               (int)blockDim.x);
  }
}

// Coarse operators, diagonal inverses and the coarsest factorisation; done
// once per Newton step since J is fixed during its V-cycles. Returns whether
// a pivot was exactly zero, in every thread of the team. A cluster may leave
// the pivot steps to the first V-cycle (later): false is returned then.
template <typename T, class TM = BlockTeam>
__device__ bool mg_setup(const MG<T> &mg, Band<T> &B, double omega, const TM &team = TM(), bool later = false) {
  if constexpr (TM::kMulti) {
    mg_setup_part(mg, omega, team.rank, team.n);
    team.sync();
    if (later) {
      if (team.lead()) band_assemble(B, mg.N[mg.L], mg.nb[mg.L], mg.J[mg.L]);
      return false;
    }
    if (team.lead()) band_factor(B, mg.N[mg.L], mg.nb[mg.L], mg.J[mg.L]);
    team.sync();  // the leader's factors and flag are done
    return team.lead_value(&s_sing) != 0;
  } else {
    for (int l = mg.l0 + 1; l <= mg.L; ++l) {
      coarse_op_cells(mg.N[l - 1], mg.nb[l - 1], mg.J[l - 1], mg.N[l], mg.J[l], (int)threadIdx.x, mg.N[l],
                      (int)blockDim.x);
      __syncthreads();
    }
    for (int l = mg.l0; l < mg.L; ++l)
      dinv_cells(mg.N[l], mg.nb[l], mg.J[l], mg.Dinv[l], omega, (int)threadIdx.x, mg.N[l], (int)blockDim.x);
    return band_factor(B, mg.N[mg.L], mg.nb[mg.L], mg.J[mg.L]);
  }
}

// `steps` symmetric multicolour SOR steps (colours 0..C-1 then C-1..0 each);
// consecutive visits of one colour run as one pass. zero: dU is all zero.
template <typename T, class TM = BlockTeam>
__device__ void sor_smooth(const MG<T> &mg, int l, int steps, double omega, bool zero, const TM &team = TM()) {
  const int nb = mg.nb[l], C = (nb - 1) / 2 + 1;
  int prev = -1, reps = 0;
  for (int s = 0; s < steps; ++s)
    for (int pass = 0; pass < 2 * C; ++pass) {
      const int col = pass < C ? pass : 2 * C - 1 - pass;
      if (col == prev) {
        ++reps;
        continue;
      }
      if (prev >= 0) {
        sor_colour(mg.N[l], nb, mg.J[l], mg.Dinv[l], mg.R[l], mg.dU[l], omega, C, prev, reps, zero, team.tid(),
                   team.size());
        team.sync();
        zero = false;
      }
      prev = col;
      reps = 1;
    }
  if (prev >= 0) {
    sor_colour(mg.N[l], nb, mg.J[l], mg.Dinv[l], mg.R[l], mg.dU[l], omega, C, prev, reps, zero, team.tid(),
               team.size());
    team.sync();
  }
}

// Algorithm 2 from level l0 by one block, pass by pass. zero: dU of level l0
// is all zero (that of a coarser level always is, by the restriction).
template <typename T>
__device__ void mg_vcycle(const MG<T> &mg, const Band<T> &B, const nswe_params &prm, bool zero) {
  for (int l = mg.l0; l < mg.L; ++l) {
    sor_smooth(mg, l, prm.nu1, prm.omega, zero || l > mg.l0);
    restrict_cells(mg.N[l], mg.nb[l], mg.J[l], mg.R[l], mg.dU[l], mg.N[l + 1], mg.R[l + 1], mg.dU[l + 1],
                   threadIdx.x, blockDim.x);
    __syncthreads();
  }
  band_solve(B, mg.N[mg.L], mg.R[mg.L], mg.dU[mg.L]);
  for (int l = mg.L - 1; l >= mg.l0; --l) {
    prolong_cells(mg.N[l], mg.dU[l], mg.N[l + 1], mg.dU[l + 1], threadIdx.x, blockDim.x);
    __syncthreads();
    sor_smooth(mg, l, prm.nu2, prm.omega, false);
  }
}

// Algorithm 2 from level ls >= l0 with legs: by a cluster, or by one block in
// FP32, whose pipe does not bound the smoothing. Levels that can be take legs
// (leg_level), the others (the full Jacobian's own level, more than two
// smoothing steps) go pass by pass. The levels of at most a tile per warp of a
// block, and of less than team_cells cells where they go pass by pass, run on
// the leader CTA with block barriers, and the coarsest solve. out0: the
// correction of level l0, on return and (unless zero) on entry; for a level
// smoothed by passes it is mg.dU[l0]. ready: called by the leader before the
// coarsest solve. factor: the coarsest matrix is assembled but not factored:
// while the cluster runs the legs on the way down, the leader's first warp
// takes the pivot steps in their place, as many beside each leg as it is long
// (a chain of 2 N_L steps of 900 cycles each, otherwise waited for: a
// 4096-cell solve on 16 CTAs 69.4 -> 52.6 ms).
template <typename T, class TM, typename F>
__device__ void mg_vcycle_legs(const MG<T> &mg, const Band<T> &B, const nswe_params &prm, bool zero, T *out0,
                               const TM &team, int team_cells, int ls, bool factor, F &&ready) {
  const int nw = (int)blockDim.x >> 5;
  auto lead_level = [&](int l) {
    return leg_level(mg.nb[l], prm) ? leg_tiles(mg.N[l]) <= nw : mg.N[l] < team_cells;
  };
  int lt = ls;
  if constexpr (TM::kMulti)
    while (lt < mg.L && !lead_level(lt)) ++lt;
  int rounds = 0, done = 0, pivots = 0;  // legs' rounds of tiles: of all levels, so far; pivot steps taken
  const int lu_warps = factor ? 1 : 0;
  auto leg_rounds = [&](int l) {
    const int w = (team.size() >> 5) - lu_warps;
    return leg_level(mg.nb[l], prm) ? (leg_tiles(mg.N[l]) + w - 1) / w : 0;
  };
  if (factor)
    for (int l = ls; l < lt; ++l) rounds += leg_rounds(l);
  auto out = [&](int l) {
    return l == mg.l0 ? out0 : l < mg.L && leg_level(mg.nb[l], prm) ? leg_out(mg.J[l], mg.N[l]) : mg.dU[l];
  };
  auto down = [&](int l, const auto &tm) {
    if (leg_level(mg.nb[l], prm)) {
      const int skip = l < lt ? lu_warps : 0, warp = (tm.tid() >> 5) - skip;
      if (skip) {
        done += leg_rounds(l);
        const int k = 2 * mg.N[mg.L] * done / rounds;
        if (warp < 0) band_lu_steps(B, pivots, k);
        pivots = k;
      }
      if (warp >= 0)
        leg<T, false>(mg.N[l], mg.J[l], mg.Dinv[l], mg.R[l], l > mg.l0 || zero ? nullptr : out0, mg.dU[l], nullptr,
                      mg.R[l + 1], prm.nu1, prm.omega, warp, (tm.size() >> 5) - skip);
      tm.sync();
      return;
    }
    sor_smooth(mg, l, prm.nu1, prm.omega, zero || l > mg.l0, tm);
    restrict_cells(mg.N[l], mg.nb[l], mg.J[l], mg.R[l], mg.dU[l], mg.N[l + 1], mg.R[l + 1], mg.dU[l + 1], tm.tid(),
                   tm.size());
    tm.sync();
  };
  auto up = [&](int l, const auto &tm) {
    if (leg_level(mg.nb[l], prm)) {
      leg<T, true>(mg.N[l], mg.J[l], mg.Dinv[l], mg.R[l], mg.dU[l], out(l), out(l + 1), nullptr, prm.nu2, prm.omega,
                   tm.tid() >> 5, tm.size() >> 5);
      tm.sync();
      return;
    }
    prolong_cells(mg.N[l], mg.dU[l], mg.N[l + 1], out(l + 1), tm.tid(), tm.size());
    tm.sync();
    sor_smooth(mg, l, prm.nu2, prm.omega, false, tm);
  };
  if constexpr (TM::kMulti)
    for (int l = ls; l < lt; ++l) down(l, team);
  if (team.lead()) {
    for (int l = lt; l < mg.L; ++l) down(l, BlockTeam());
    ready();
    if (factor && pivots < B.n) {
      if (threadIdx.x < 32) band_lu_steps(B, pivots, B.n);
      __syncthreads();
    }
    band_solve(B, mg.N[mg.L], mg.R[mg.L], mg.dU[mg.L]);
    for (int l = mg.L - 1; l >= lt; --l) up(l, BlockTeam());
  }
  if constexpr (TM::kMulti) {
    team.sync();
    for (int l = lt - 1; l >= ls; --l) up(l, team);
  }
}

// Band storage in dynamic shared memory, sized by the host for the coarsest
// level: ab [ldab_cap * n_cap], x [n_cap], rinv [n_cap], piv [n_cap].
extern __shared__ double g_dyn_smem[];

template <typename T>
__device__ __forceinline__ Band<T> band_view(int n_cap, int ldab_cap) {
  Band<T> B;
  B.ab = reinterpret_cast<T *>(g_dyn_smem);
  B.x = B.ab + (size_t)ldab_cap * n_cap;
  B.rinv = B.x + n_cap;
  B.piv = reinterpret_cast<int *>(B.rinv + n_cap);
  B.n = B.kl = B.ldab = 0;
  return B;
}

// ----------------------------------------------------------------------------
// Kernels.

constexpr int kVcThreads = 128;       // a warp per SM sub-partition: the FP64 pipe sets a leg's time
// Larger levels are launches over the chip: four rounds of a cluster's 16 x 4
// warps cost less than a launch and its gap per leg (4096 cells, 205 tiles:
// 146 us with 256 here, 157 with 64).
constexpr int kVcClusterTiles = 256;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The standalone residual by tiles of cells in shared memory: every WENO
// reconstruction formed once (one per cell and component), then every face
// flux and, on other warps, every source, then the differences. The FP64 pipe
// bounds it: about 110 instruction slots per cell against 220 where each cell
// rebuilds its neighbours' reconstructions and both its fluxes. Small levels
// take tiles of 31 cells (32 faces: one warp), so that one channel spreads over
// many SMs and the chain of a warp is one reconstruction and one flux; levels
// that fill the chip that way take 254 (512 reconstructions for 256 threads).
// The blocks of a level of at most 16 tiles are one cluster and form res too
// (res given); else their sums go to `partials` for k_finish_res.
constexpr int kResTileSmall = 31, kResThreadsSmall = 128, kResTile = 254, kResThreads = 256;
constexpr int kResMaxBlocks = 1024;  // partial sums of a context

template <int TILE, int THREADS>
__global__ void __launch_bounds__(THREADS) k_residual(const ProbDev *P, int level, const double *U, double *R,
                                                      double *partials, double *res) {
  __shared__ double rec[2][2][TILE + 2], flx[2][TILE + 1], src[TILE], red[34];
  const Geo G = make_geo(*P, level);
  const int N = G.N;
  double acc = 0.0;
  for (int t0 = blockIdx.x * TILE; t0 < N; t0 += gridDim.x * TILE) {
    const int cells = min(TILE, N - t0), w = cells + 2;
    for (int it = threadIdx.x; it < 2 * w; it += THREADS) {
      const int m = it >= w, i = it - m * w, k = t0 + i - 1;
      auto at = [&](int kk) { return pval<double>(G, U, m, kk, -1, 0.0, 0.0); };
      weno3<double>(at(k - 1), at(k), at(k + 1), rec[m][0][i], rec[m][1][i]);  // cell t0 + i - 1
    }
    __syncthreads();
    const int first_src = (cells + 1 + 31) & ~31;
    for (int it = threadIdx.x; it < first_src + cells; it += THREADS) {
      if (it <= cells) {
        const int f = t0 + it;
        const Face<double> fc = face(G.isf[f], G.cgf[f], G.g);
        num_flux<-1>(fstate<Sum::kRounded>(rec[0][1][it], rec[1][1][it], fc),
                     fstate<Sum::kRounded>(rec[0][0][it + 1], rec[1][0][it + 1], fc), G.flux, flx[0][it], flx[1][it]);
      } else if (it >= first_src) {
        const int i = it - first_src;
        src[i] = source_at(src_cell<double>(G, t0 + i), rec[0][0][i], rec[0][0][i + 1], rec[0][1][i + 1],
                           rec[0][1][i + 2]);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cells; i += THREADS) {
      const double R0 = flx[0][i + 1] - flx[0][i];
      const double R1 = flx[1][i + 1] - flx[1][i] - src[i];
      R[t0 + i] = R0;
      R[N + t0 + i] = R1;
      acc += fabs(R0) + fabs(R1);
    }
    __syncthreads();  // the tile is read before the next one is built
  }
  const double s = block_sum(acc, red);
  if (!res) {
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
    return;
  }
  auto cl = cooperative_groups::this_cluster();
  if (threadIdx.x == 0) red[33] = s;
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x < 32) {
    double v = threadIdx.x < cl.num_blocks() ? *cl.map_shared_rank(red + 33, threadIdx.x) : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) *res = v / N;
  }
  cl.sync();  // no block leaves while its sum may be read
}

// res from the block sums, by one block (one thread took 36 us for 1024).
__global__ void __launch_bounds__(kThreads) k_finish_res(const double *partials, int n, int N, double *res) {
  __shared__ double red[33];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += partials[i];
  const double s = block_sum(v, red);
  if (threadIdx.x == 0) *res = s / N;
}

__global__ void __launch_bounds__(kThreads) k_geom_derive(const ProbDev *P) {
  geom_derive_items(*P, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// The derived geometry of many problems in one launch: block b derives
// tasks[b].prob.
__global__ void __launch_bounds__(kThreads) k_geom_derive_batch(const SolveTask *tasks) {
  geom_derive_items(*tasks[blockIdx.x].prob, threadIdx.x, blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_jac_a(const ProbDev *P, int level, const double *U, double eps) {
  Geo G = make_geo(*P, level);
  jac_pass_a<T>(G, U, eps, jw_view<T>(P->jw, G.N), blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_jac_b(const ProbDev *P, int level) {
  Geo G = make_geo(*P, level);
  jac_pass_b<T, -1>(G, jw_view<T>(P->jw, G.N), blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_jac_c(const ProbDev *P, int level, int nb, double eps, double alpha,
                                                    const double *Rreg, double *R, T *J, double *partials) {
  __shared__ double red[33];
  Geo G = make_geo(*P, level);
  double acc = jac_pass_c<T>(G, nb, eps, alpha, jw_view<T>(P->jw, G.N), Rreg, R, J,
                             blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  double s = block_sum(acc, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// A standalone V-cycle: coarse operators and inverses (k_vc_setup, a block per
// coarsest cell), the coarsest factorisation (k_vc_factor, one block, left in
// the Jacobian workspace), then k_vc_cluster with the levels that one cluster
// of 16 blocks takes, started beside the factorisation; larger levels are
// launches of their own before and after it (k_vc_leg). One block for all of
// it took 513 us for 4096 cells, this 121.
// The factors lie at the front of the workspace: ab, rinv, piv of Band.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_vc_setup(const ProbDev *P, int level, int nb, const T *J,
                                                       double omega) {
  MG<T> mg;
  mg_bind<T>(mg, *P, level, nb, J, nullptr, nullptr);
  mg_setup_part(mg, omega, blockIdx.x, gridDim.x);
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_vc_factor(const ProbDev *P, int *status, int n_cap, int ldab_cap) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Band<T> B = band_view<T>(n_cap, ldab_cap);
  const LevelDev &Lv = P->lev[P->levels - 1];
  const bool sing = band_factor(B, Lv.N, 3, reinterpret_cast<const T *>(Lv.J));
  Band<T> G = B;
  G.ab = reinterpret_cast<T *>(P->jw);
  G.rinv = G.ab + (size_t)B.ldab * B.n;
  G.piv = reinterpret_cast<int *>(G.rinv + B.n);
  for (int t = threadIdx.x; t < B.ldab * B.n; t += blockDim.x) G.ab[t] = B.ab[t];
  for (int t = threadIdx.x; t < B.n; t += blockDim.x) {
    G.rinv[t] = B.rinv[t];
    G.piv[t] = B.piv[t];
  }
  if (threadIdx.x == 0) *status = sing ? NSWE_ESINGULAR : NSWE_OK;
}

// ls: the first level of the cluster (l0 = level: all of them).
template <typename T>
__global__ void __launch_bounds__(kVcThreads, 1)
    k_vc_cluster(const ProbDev *P, int level, int ls, int nb, const T *J, const T *R, T *dU,
                 const __grid_constant__ nswe_params prm, int n_cap, int ldab_cap) {
  const auto cl = cooperative_groups::this_cluster();
  const ClusterTeam team{(int)cl.block_rank(), (int)cl.num_blocks()};
  MG<T> mg;
  mg_bind<T>(mg, *P, level, nb, J, R, leg_level(nb, prm) ? reinterpret_cast<T *>(P->lev[level].dU) : dU);
  Band<T> B = band_view<T>(n_cap, ldab_cap);
  B.n = 2 * mg.N[mg.L];
  B.kl = 3;
  B.ldab = 10;
  mg_vcycle_legs<T>(mg, B, prm, false, dU, team, 0, ls, false, [&] {
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the factors are there
    const T *ab = reinterpret_cast<const T *>(P->jw), *rinv = ab + (size_t)B.ldab * B.n;
    const int *piv = reinterpret_cast<const int *>(rinv + B.n);
    for (int t = threadIdx.x; t < B.ldab * B.n; t += blockDim.x) B.ab[t] = ab[t];
    for (int t = threadIdx.x; t < B.n; t += blockDim.x) {
      B.rinv[t] = rinv[t];
      B.piv[t] = piv[t];
    }
    __syncthreads();
  });
}

// The coarsest level's own system: the direct solve.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_vc_direct(int N, int nb, const T *J, const T *R, T *dU, int *status,
                                                        int n_cap, int ldab_cap) {
  Band<T> B = band_view<T>(n_cap, ldab_cap);
  const bool sing = band_factor(B, N, nb, J);
  band_solve(B, N, R, dU);
  if (threadIdx.x == 0) *status = sing ? NSWE_ESINGULAR : NSWE_OK;
}

// One leg of one level on the whole chip; level l0 takes the caller's arrays.
template <typename T, bool UP>
__global__ void __launch_bounds__(kVcThreads, 4) k_vc_leg(const ProbDev *P, int l, int l0, const T *J, const T *R, T *dU,
                                                       int steps, double omega) {
  const LevelDev &Lv = P->lev[l], &Lc = P->lev[l + 1];
  const int N = Lv.N, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = (gridDim.x * blockDim.x) >> 5;
  T *const Jl = l == l0 ? const_cast<T *>(J) : reinterpret_cast<T *>(Lv.J);
  const T *const Rl = l == l0 ? R : reinterpret_cast<const T *>(Lv.R);
  T *const mid = reinterpret_cast<T *>(Lv.dU), *const out = l == l0 ? dU : leg_out(Jl, N);
  const T *const Dinv = reinterpret_cast<const T *>(Lv.Dinv);
  T *const Jc = reinterpret_cast<T *>(Lc.J);
  if (UP)
    leg<T, true>(N, Jl, Dinv, Rl, mid, out,
                 l + 1 == P->levels - 1 ? reinterpret_cast<const T *>(Lc.dU) : leg_out(Jc, Lc.N), nullptr, steps,
                 omega, warp, warps);
  else
    leg<T, false>(N, Jl, Dinv, Rl, l == l0 ? out : nullptr, mid, nullptr, reinterpret_cast<T *>(Lc.R), steps, omega,
                  warp, warps);
}

// The team of the calling thread and the index of its problem: a block per
// problem, or a cluster per problem (clusters tile the grid along x).
template <class TM>
__device__ __forceinline__ TM make_team(int &task_index);
template <>
__device__ __forceinline__ BlockTeam make_team<BlockTeam>(int &task_index) {
  task_index = blockIdx.x;
  return BlockTeam{};
}
template <>
__device__ __forceinline__ ClusterTeam make_team<ClusterTeam>(int &task_index) {
  const auto cl = cooperative_groups::this_cluster();
  ClusterTeam t{(int)cl.block_rank(), (int)cl.num_blocks()};
  task_index = blockIdx.x / t.n;
  return t;
}

// Algorithm 3 for one problem per team (a thread block, or a cluster of
// blocks: TM). T is the precision of the Jacobian and the multigrid solve of
// each Newton step: with T = double the whole step is FP64; with T = float
// the residual, the convergence test and the update U += tau dU stay FP64
// while the FD Jacobian (Eq. 12-13), the coarse operators, the smoother and
// the coarsest LU run in FP32. FLUX: the numerical flux of every task of the
// launch (compile-time, so that the HLL kernels carry no LLF code).
// team_cells: of the levels smoothed pass by pass, a cluster team runs those
// with at least that many cells on all its CTAs, the others on the leader CTA.
template <typename T, int THREADS, int MINB, int FLUX, class TM = BlockTeam>
__global__ void __launch_bounds__(THREADS, MINB)
    k_solve(const SolveTask *tasks, nswe_params launch_prm, int n_cap, int ldab_cap, int team_cells) {
  constexpr bool kMixed = std::is_same<T, float>::value;
  __shared__ double red[34];
  __shared__ nswe_params s_prm;
  const unsigned long long t_start = global_ns();
  int ti;
  const TM team = make_team<TM>(ti);
  const SolveTask task = tasks[ti];
  const ProbDev &P = *task.prob;
  if (threadIdx.x == 0) s_prm = task.prm ? *task.prm : launch_prm;
  if (task.derive) geom_derive_items(P, team.tid(), team.size());
  team.sync();  // (a cluster team: also every CTA has started before any shared-memory access across CTAs)
  const nswe_params &prm = s_prm;
  const int L = P.levels - 1;
  const int s0 = (prm.nest_start < 0 || prm.nest_start > L) ? L : prm.nest_start;
  const int nb = prm.jacobian == NSWE_JAC_FULL ? 5 : 3;
  Band<T> B = band_view<T>(n_cap, ldab_cap);

  int iters[NSWE_MAX_LEVELS], lstat[NSWE_MAX_LEVELS];
  double lres[NSWE_MAX_LEVELS];
  for (int l = 0; l < NSWE_MAX_LEVELS; ++l) {
    iters[l] = 0;
    lstat[l] = NSWE_OK;
    lres[l] = 0.0;
  }
  int vcycles = 0, total = 0, fatal = 0;

  {
    const int Ns = P.lev[s0].N;
    for (int t = team.tid(); t < 2 * Ns; t += team.size()) P.lev[s0].U[t] = task.U0[t];
    team.sync();
  }

  for (int l = s0; l >= 0 && !fatal; --l) {
    const LevelDev &Lv = P.lev[l];
    Geo G = make_geo(P, l);
    const int N = G.N;
    if (l < s0) {
      interp_cells(make_geo(P, l + 1), P.lev[l + 1].U, Lv.U, team.tid(), team.size());
      team.sync();
    }
    // Mixed path: the FP32 Jacobian reads FP32 copies of the state (kept up
    // to date by the update) and of the level's geometry.
    float *U32 = nullptr;
    if constexpr (kMixed) {
      U32 = attach_f32(G, P.jw);
      fill_f32(G, Lv.U, U32, team.tid(), team.size());
      team.sync();
    }
    const JW<T> W = jw_view<T>(P.jw, N);
    T *const J = reinterpret_cast<T *>(Lv.J);
    T *const dU = reinterpret_cast<T *>(Lv.dU);
    // Right-hand side of the linear solve: the FP64 residual itself, or its
    // FP32 copy in the unused upper part of J's storage (J takes 4 nb N of
    // the 40 N floats there).
    T *const Rs = kMixed ? J + (size_t)4 * nb * N : reinterpret_cast<T *>(Lv.R);
    // FP64 path: R, J and res at the current state in one pass (Eq. 10,
    // 12-13). Mixed path: only the FP64 residual and res here.
    auto residual_step = [&]() -> double {
      double acc;
      if constexpr (kMixed) {
        const RW RWv = rw_view(P.jw, N);
        res_pass_a(G, Lv.U, RWv, team.tid(), team.size());
        team.sync();
        res_pass_b<FLUX>(G, RWv, team.tid(), team.size());
        team.sync();
        acc = res_pass_c(G, RWv, Lv.R, team.tid(), team.size());
      } else {
        jac_pass_a<T>(G, Lv.U, prm.eps[l], W, team.tid(), team.size());
        team.sync();
        jac_pass_b<T, FLUX>(G, W, team.tid(), team.size());
        team.sync();
        acc = jac_pass_c<T>(G, nb, prm.eps[l], prm.alpha, W, nullptr, Lv.R, J, team.tid(), team.size());
      }
      return team.sum(acc, red) / N;
    };
    double res = residual_step();
    int n = 0, st = NSWE_OK;
    while (true) {
      if constexpr (kMixed) {
        // FP32 Jacobian at the current state, regularised with the FP64 R.
        jac_pass_a<T>(G, Lv.U, prm.eps[l], W, team.tid(), team.size());
        team.sync();
        jac_pass_b<T, FLUX>(G, W, team.tid(), team.size());
        team.sync();
        jac_pass_c<T>(G, nb, prm.eps[l], prm.alpha, W, Lv.R, nullptr, J, team.tid(), team.size());
        for (int t = team.tid(); t < 2 * N; t += team.size()) Rs[t] = T(Lv.R[t]);
        team.sync();
      }
      MG<T> mg;
      mg_bind<T>(mg, P, l, nb, J, Rs, dU);
      // (a cluster factors the coarsest system beside its first V-cycle)
      const bool later = TM::kMulti && l < L && prm.nu3 >= 1;
      bool sing = mg_setup<T, TM>(mg, B, prm.omega, team, later);
      if (!later) team.sync();
      if (sing) {
        st = NSWE_ESINGULAR;
        break;
      }
      T *x = dU;  // where the correction ends
      if (l == L) {
        if (team.lead()) band_solve<T>(B, N, Rs, dU);
        if constexpr (TM::kMulti) team.sync();
      } else if constexpr (TM::kMulti || kMixed) {
        if (leg_level(nb, prm)) x = leg_out(J, N);
        if (!leg_level(nb, prm) || prm.nu3 < 1) {
          for (int t = team.tid(); t < 2 * N; t += team.size()) x[t] = T(0.0);
          team.sync();
        }
        for (int m = 0; m < prm.nu3; ++m) {
          mg_vcycle_legs<T, TM>(mg, B, prm, m == 0, x, team, team_cells, l, later && m == 0, [] {});
          if constexpr (TM::kMulti)
            if (m == 0 && (sing = team.lead_value(&s_sing) != 0)) break;
          ++vcycles;
        }
        if (sing) {
          st = NSWE_ESINGULAR;
          break;
        }
      } else {
        for (int t = team.tid(); t < 2 * N; t += team.size()) dU[t] = T(0.0);
        team.sync();
        for (int m = 0; m < prm.nu3; ++m) {
          mg_vcycle<T>(mg, B, prm, m == 0);
          ++vcycles;
        }
      }
      bool bad = false;
      for (int j = team.tid(); j < N; j += team.size()) {
        double h = fma(prm.tau, double(x[j]), Lv.U[j]);
        Lv.U[j] = h;
        Lv.U[N + j] = fma(prm.tau, double(x[N + j]), Lv.U[N + j]);
        if constexpr (kMixed) {
          U32[j] = float(h);
          U32[N + j] = float(Lv.U[N + j]);
        }
        if (!(h > 0.0)) bad = true;
      }
      bad = team.any(bad);
      ++n;
      if (bad) {
        st = NSWE_ENEGDEPTH;
        break;
      }
      // res of the new state (on the FP64 path its Jacobian serves the next
      // step and is not needed once res < tol).
      res = residual_step();
      if (!(res == res) || isinf(res)) {
        st = NSWE_ENAN;
        break;
      }
      if (res < prm.tol) break;
      if (n >= prm.n_max) {
        st = NSWE_ENOTCONV;
        break;
      }
    }
    iters[l] = n;
    lres[l] = res;
    lstat[l] = st;
    total += n;
    if (st == NSWE_ENAN || st == NSWE_ENEGDEPTH || st == NSWE_ESINGULAR) fatal = st;
  }

  if (!fatal) {
    const int N0 = P.lev[0].N;
    for (int t = team.tid(); t < 2 * N0; t += team.size()) task.U[t] = P.lev[0].U[t];
  }
  if (threadIdx.x == 0 && team.lead() && task.info) {
    nswe_info inf;
    for (int l = 0; l < NSWE_MAX_LEVELS; ++l) {
      inf.iters[l] = iters[l];
      inf.res[l] = lres[l];
      inf.level_status[l] = lstat[l];
    }
    inf.status = fatal ? fatal : lstat[0];
    inf.total_iters = total;
    inf.vcycles = vcycles;
    inf.t_start_ns = t_start;
    inf.t_end_ns = global_ns();
    *task.info = inf;
  }
  if (task.done) {
    // Every thread's result writes are visible system-wide before the flag.
    __threadfence_system();
    team.sync();
    if (threadIdx.x == 0 && team.lead()) *reinterpret_cast<volatile int *>(task.done) = 1;
  }
  if constexpr (TM::kMulti) team.sync();  // no CTA leaves while another may read its shared memory
}

// A launch of `blocks` blocks in clusters of `ctas`; at: storage of its attribute.
cudaLaunchConfig_t cluster_config(int blocks, int ctas, int threads, size_t smem, cudaStream_t s,
                                  cudaLaunchAttribute *at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

int grid_for(int items) {
  int b = (items + kThreads - 1) / kThreads;
  return b < 1 ? 1 : (b > 1024 ? 1024 : b);
}

}  // namespace

cudaError_t launch_geom_derive(const ProbDev *p, int finest_cells, cudaStream_t s) {
  k_geom_derive<<<grid_for(2 * finest_cells + 1), kThreads, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_geom_derive_batch(const SolveTask *tasks, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_geom_derive_batch<<<count, kThreads, 0, s>>>(tasks);
  return cudaGetLastError();
}

cudaError_t launch_residual(const ProbDev *p, int level, int N, const double *U, double *R, double *res,
                            double *partials, int max_ctas, cudaStream_t s) {
  const int small = (N + kResTileSmall - 1) / kResTileSmall;
  if (small > 4 * kSmCount) {
    const int tiles = (N + kResTile - 1) / kResTile, grid = tiles < kResMaxBlocks ? tiles : kResMaxBlocks;
    k_residual<kResTile, kResThreads><<<grid, kResThreads, 0, s>>>(p, level, U, R, partials, nullptr);
    if (res) k_finish_res<<<1, kThreads, 0, s>>>(partials, grid, N, res);
    return cudaGetLastError();
  }
  auto kern = k_residual<kResTileSmall, kResThreadsSmall>;
  if (!res || small > max_ctas) {
    kern<<<small, kResThreadsSmall, 0, s>>>(p, level, U, R, partials, nullptr);
    if (res) k_finish_res<<<1, kThreads, 0, s>>>(partials, small, N, res);
    return cudaGetLastError();
  }
  if (small > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = cluster_config(small, small, kResThreadsSmall, 0, s, at);
  return cudaLaunchKernelEx(&cfg, kern, p, level, U, R, partials, res);
}

cudaError_t launch_jacobian(const ProbDev *p, int level, int N, int nb, const double *U, double eps,
                            double alpha, double *R, double *J, double *res, double *partials, cudaStream_t s) {
  k_jac_a<double><<<grid_for((N + 2) * 2), kThreads, 0, s>>>(p, level, U, eps);
  k_jac_b<double><<<grid_for(N + 1), kThreads, 0, s>>>(p, level);
  const int grid = grid_for(N * nb);
  k_jac_c<double><<<grid, kThreads, 0, s>>>(p, level, nb, eps, alpha, nullptr, R, J, partials);
  if (res) k_finish_res<<<1, kThreads, 0, s>>>(partials, grid, N, res);
  return cudaGetLastError();
}

cudaError_t launch_jacobian_f32(const ProbDev *p, int level, int N, int nb, const double *U, double eps,
                                double alpha, double *R, float *J, double *res, double *partials, int max_ctas,
                                cudaStream_t s) {
  // The residual's reduction has consumed `partials` (stream order) before
  // the FP32 pass C reuses it (it writes zeros there).
  cudaError_t e = launch_residual(p, level, N, U, R, res, partials, max_ctas, s);
  if (e != cudaSuccess) return e;
  k_jac_a<float><<<grid_for((N + 2) * 2), kThreads, 0, s>>>(p, level, U, eps);
  k_jac_b<float><<<grid_for(N + 1), kThreads, 0, s>>>(p, level);
  k_jac_c<float><<<grid_for(N * nb), kThreads, 0, s>>>(p, level, nb, eps, alpha, R, nullptr, J, partials);
  return cudaGetLastError();
}

size_t band_smem_bytes(int n_cap, int ldab_cap) {
  return sizeof(double) * ((size_t)ldab_cap * n_cap + 2 * (size_t)n_cap) + sizeof(int) * (size_t)n_cap;
}

namespace {
template <typename T>
cudaError_t vcycle_t(const ProbDev *p, int level, int levels, int N, int nb, const T *J, const T *R, T *dU,
                     const nswe_params &prm, int *status, int max_ctas, cudaStream_t s) {
  const int L = levels - 1, NL = N >> (L - level), n_cap = 2 * NL;
  const int ldab_cap = 3 * (level == L && nb == 5 ? 5 : 3) + 1;
  const size_t smem = band_smem_bytes(n_cap, ldab_cap);
  if (level == L) {
    k_vc_direct<T><<<1, kThreads, smem, s>>>(N, nb, J, R, dU, status, n_cap, ldab_cap);
    return cudaGetLastError();
  }
  k_vc_setup<T><<<NL, kThreads, 0, s>>>(p, level, nb, J, prm.omega);
  // Levels of more than kVcClusterTiles tiles are launches over the chip.
  int ls = level;
  while (ls < L && leg_level(ls == level ? nb : 3, prm) && leg_tiles(N >> (ls - level)) > kVcClusterTiles) ++ls;
  auto grid = [&](int l) { return (leg_tiles(N >> (l - level)) + kVcThreads / 32 - 1) / (kVcThreads / 32); };
  for (int l = level; l < ls; ++l)
    k_vc_leg<T, false><<<grid(l), kVcThreads, 0, s>>>(p, l, level, J, R, dU, prm.nu1, prm.omega);
  k_vc_factor<T><<<1, kThreads, smem, s>>>(p, status, n_cap, ldab_cap);
  auto kern = k_vc_cluster<T>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = cluster_config(max_ctas, max_ctas, kVcThreads, smem, s, at);
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if ((e = cudaStreamIsCapturing(s, &cs)) != cudaSuccess) return e;
  if (cs == cudaStreamCaptureStatusNone) cfg.numAttrs = 2;  // (a capture keeps stream order)
  if ((e = cudaLaunchKernelEx(&cfg, kern, p, level, ls, nb, J, R, dU, prm, n_cap, ldab_cap)) != cudaSuccess) return e;
  for (int l = ls - 1; l >= level; --l)
    k_vc_leg<T, true><<<grid(l), kVcThreads, 0, s>>>(p, l, level, J, R, dU, prm.nu2, prm.omega);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_vcycle(const ProbDev *p, int level, int levels, int N, int nb, const double *J, const double *R,
                          double *dU, const nswe_params &prm, int *status, int max_ctas, cudaStream_t s) {
  return vcycle_t<double>(p, level, levels, N, nb, J, R, dU, prm, status, max_ctas, s);
}

cudaError_t launch_vcycle_f32(const ProbDev *p, int level, int levels, int N, int nb, const float *J, const float *R,
                              float *dU, const nswe_params &prm, int *status, int max_ctas, cudaStream_t s) {
  return vcycle_t<float>(p, level, levels, N, nb, J, R, dU, prm, status, max_ctas, s);
}

cudaError_t launch_solve(const SolveTask *tasks, int count, const nswe_params &prm, int max_coarse_cells,
                         cudaStream_t s) {
  return launch_solve_sized(tasks, count, prm, max_coarse_cells, prm.jacobian == NSWE_JAC_FULL ? 5 : 3, kShapeAuto, s);
}

namespace {
template <int SHAPE, int FLUX = NSWE_FLUX_HLL>
void launch_shape(const SolveTask *tasks, int count, const nswe_params &prm, int n_cap, int ldab_cap, size_t smem,
                  cudaStream_t s) {
  constexpr int TH = kSolveShapeThreads[SHAPE], MB = kSolveShapeBlocks[SHAPE];
  if (prm.precision == NSWE_PREC_MIXED)
    k_solve<float, TH, MB, FLUX><<<count, TH, smem, s>>>(tasks, prm, n_cap, ldab_cap, 0);
  else
    k_solve<double, TH, MB, FLUX><<<count, TH, smem, s>>>(tasks, prm, n_cap, ldab_cap, 0);
}
}  // namespace

namespace {
template <typename T>
cudaError_t launch_cluster_t(const SolveTask *tasks, int count, const nswe_params &prm, int n_cap, int ldab_cap,
                             size_t smem, int ctas, int team_cells, cudaStream_t s) {
  auto kern = k_solve<T, kClusterThreads, 1, NSWE_FLUX_HLL, ClusterTeam>;
  if (ctas > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = cluster_config(count * ctas, ctas, kClusterThreads, smem, s, at);
  return cudaLaunchKernelEx(&cfg, kern, tasks, prm, n_cap, ldab_cap, team_cells);
}
}  // namespace

cudaError_t launch_solve_cluster(const SolveTask *tasks, int count, const nswe_params &prm, int max_coarse_cells,
                                 int max_nb, int ctas, int team_cells, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  const int n_cap = 2 * max_coarse_cells, ldab_cap = 3 * (max_nb == 5 ? 5 : 3) + 1;
  const size_t smem = band_smem_bytes(n_cap, ldab_cap);
  if (prm.precision == NSWE_PREC_MIXED)
    return launch_cluster_t<float>(tasks, count, prm, n_cap, ldab_cap, smem, ctas, team_cells, s);
  return launch_cluster_t<double>(tasks, count, prm, n_cap, ldab_cap, smem, ctas, team_cells, s);
}

cudaError_t launch_solve_sized(const SolveTask *tasks, int count, const nswe_params &prm, int max_coarse_cells,
                               int max_nb, int shape, cudaStream_t s, int flux) {
  const int n_cap = 2 * max_coarse_cells, ldab_cap = 3 * (max_nb == 5 ? 5 : 3) + 1;
  const size_t smem = band_smem_bytes(n_cap, ldab_cap);
  if (flux == NSWE_FLUX_LLF) {  // a comparison option: the default shape only
    launch_shape<0, NSWE_FLUX_LLF>(tasks, count, prm, n_cap, ldab_cap, smem, s);
    return cudaGetLastError();
  }
  if (shape == kShapeAuto) shape = count <= 2 * kSmCount ? 2 : 0;
  switch (shape) {
  case 1: launch_shape<1>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  case 2: launch_shape<2>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  case 3: launch_shape<3>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  case 4: launch_shape<4>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  case 5: launch_shape<5>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  default: launch_shape<0>(tasks, count, prm, n_cap, ldab_cap, smem, s); break;
  }
  return cudaGetLastError();
}

}  // namespace nswe
