// The residual (Eq. 20) and the FD Jacobian (Eq. 12-13, 21) of the 2D scheme,
// one tile of cells per thread block, with every reconstruction and every
// face flux formed once.
//
// R of a cell needs, per direction, the characteristic WENO3 values of three
// neighbouring lines at four interfaces, and these combined at the two Gauss
// points of two faces. Evaluated cell by cell that is 36 one-sided
// reconstructions per cell where the cell's own share is 4, and for the J9 of
// Eq. 21 another 27 perturbed residuals. Here a block builds in shared memory
//   1 the tile's cells with two ghost layers,
//   2 the interface values of all its lines (both directions, both sides),
//   3 (Jacobian) the interface values with one of their three stencil cells
//     perturbed in one component,
//   4 the fluxes of its faces: unperturbed, and with one cell that the face
//     reads perturbed in one component,
//   5 and each cell's residual or blocks from two face fluxes and the source.
// A perturbed value is what the perturbed local residual of Eq. 12 would have
// there, by the same expressions, so each entry is that residual's. The
// products and sums are written out as fused or rounded (__dmul_rn, fma), so
// that every kernel built from this file rounds alike: a batch's problems get
// the bits they get alone, and the differences over eps = 1e-6, in which one
// rounding weighs 1e10 times as much, do not change with the compiler's choice.
//
// Bound: FP64 issue (64 cycles per warp instruction and SM sub-partition).
// Of it the halo costs (1 + 2/TX)(1 + 2/TY) in steps 2-3 and 1 + 1/TX in step
// 4; the tile is chosen per grid size by tile2_choose. Against one cell (or
// one cell and block) per thread with every line rebuilt, on GB300: residual
// 1253 -> 202 us at 512 x 256 and 314 -> 25 us at 96 x 40; with the Jacobian,
// 512 x 256: J9 13.1 -> 3.8 ms, frozen J9 14.1 -> 3.3 ms, J21 25.8 -> 5.6 ms;
// 96 x 40: J9 1.01 -> 0.19 ms, J21 1.95 -> 0.24 ms. J9 is bound by the 25
// flux variants of each face (two LLF fluxes each), about 60 FP64
// instructions per Gauss point.
//
// Ghost cells follow the interior cell that they copy or mirror, so every
// cell of the tile carries the index of its source cell and, per component,
// whether it holds the source's value, its negative or boundary data. "Cell
// cp perturbed" then perturbs every stencil position whose source is cp, and
// a consumer finds the variant of a line that reads cp by comparing sources:
// walls, corners and grids of four cells need no case of their own.
#pragma once

namespace nswe {
namespace {

constexpr int kTile2Threads = 512;

// Cell (i, j), two ghost layers (x rule, then y rule at corners), with its
// source cell (-1: boundary data only) and 2 bits per component: 0 boundary
// data, 1 the source's value, 2 its negative.
__device__ __forceinline__ void bc_post_code(int kind, const double *st, double o[3], int normal, int &code) {
  if (kind == NSWE_BC2_REFLECT) {
    o[normal] = -o[normal];
    const int c = (code >> (2 * normal)) & 3;
    if (c) code ^= 3 << (2 * normal);
  } else if (kind == NSWE_BC2_DISCHARGE) {
    o[1] = st[1];
    o[2] = st[2];
    code &= 3;
  } else if (kind == NSWE_BC2_DEPTH) {
    o[0] = st[0];
    code &= ~3;
  }
}

__device__ __forceinline__ void cell_meta(const Geo2 &G, const double *U, int i, int j, double o[3], int &src,
                                          int &code) {
  const int Nx = G.Nx, Ny = G.Ny, n = Nx * Ny;
  int xk = 0, xs = 0, yk = 0, ys = 0;
  src = -1;
  code = 0;
  if (i < 0 || i >= Nx) {
    xs = i < 0 ? 0 : 1;
    xk = G.bck[xs * Ny + min(max(j, 0), Ny - 1)];
    if (xk == NSWE_BC2_INFLOW) {
      o[0] = G.bcs[xs * 3];
      o[1] = G.bcs[xs * 3 + 1];
      o[2] = G.bcs[xs * 3 + 2];
      return;
    }
    i = (xk == NSWE_BC2_REFLECT) ? (i < 0 ? -1 - i : 2 * Nx - 1 - i) : (i < 0 ? 0 : Nx - 1);
  }
  if (j < 0 || j >= Ny) {
    ys = j < 0 ? 2 : 3;
    yk = G.bck[2 * Ny + (ys - 2) * Nx + i];
    if (yk != NSWE_BC2_INFLOW) j = (yk == NSWE_BC2_REFLECT) ? (j < 0 ? -1 - j : 2 * Ny - 1 - j) : (j < 0 ? 0 : Ny - 1);
  }
  if (yk == NSWE_BC2_INFLOW) {
    o[0] = G.bcs[ys * 3];
    o[1] = G.bcs[ys * 3 + 1];
    o[2] = G.bcs[ys * 3 + 2];
  } else {
    src = j * Nx + i;
    code = 1 | 1 << 2 | 1 << 4;
#pragma unroll
    for (int m = 0; m < 3; ++m) o[m] = U[m * n + src];
    if (yk) bc_post_code(yk, G.bcs + ys * 3, o, 2, code);
  }
  if (xk) bc_post_code(xk, G.bcs + xs * 3, o, 1, code);
}

// One tile: interior cells [x0, x0 + a) x [y0, y0 + b). Direction d (0: x, 1:
// y) has lines r = -1 .. T(d) (transverse to d, index r + 1) of cells al = -2
// .. A(d) + 1, and interfaces q between the cells al = q - 2 and q - 1.
// U^- at q = 1 .. A + 2 reads cells q-3 .. q-1, U^+ at q = 0 .. A + 1 reads
// cells q-2 .. q: A + 2 of each per line.
struct Tile2d {
  int x0, y0, a, b, W;
  __device__ __forceinline__ int A(int d) const { return d == 0 ? a : b; }
  __device__ __forceinline__ int T(int d) const { return d == 0 ? b : a; }
  __device__ __forceinline__ int cells() const { return W * (b + 4); }
  __device__ __forceinline__ int cell(int d, int al, int r) const {
    return d == 0 ? (r + 2) * W + al + 2 : (al + 2) * W + r + 2;
  }
  __device__ __forceinline__ int nI(int d) const { return (A(d) + 2) * (T(d) + 2); }  // one side's interface values
  __device__ __forceinline__ int nF(int d) const { return (A(d) + 1) * T(d); }        // faces q = 1 .. A + 1
  __device__ __forceinline__ int nP(int d) const { return (A(d) + 3) * (T(d) + 2); }  // interfaces, either side
  __device__ __forceinline__ int iI(int d, int line, int q, int side) const { return line * (A(d) + 2) + q - 1 + side; }
  __device__ __forceinline__ int iP(int d, int line, int q) const { return line * (A(d) + 3) + q; }
};

// Shared-memory planes of a tile. Values are stored plane by plane (slot and
// component major, interface or face minor), so that the threads of a warp,
// which take neighbouring interfaces of one slot, read consecutive words.
struct Smem2d {
  double *C;         // [3][cells]
  int *src;          // [cells]
  int *code;         // [cells]
  double *V0, *V1;   // per direction [2 sides][NV][3][nI]
  double *F0, *F1;   // [NF][3][nF]
  double *E0, *E1;   // steps 2-3, in F's place: [5][nP] un, ut, c, 1/(2c), 1/h of each interface
  double *Q0, *Q1;   //                          [2 sides][12][nI] Wr, and the weights of the frozen linearisation
  double *S0, *S1;   // [a * b] unperturbed source
  __device__ __forceinline__ double *V(int d) const { return d ? V1 : V0; }
  __device__ __forceinline__ double *F(int d) const { return d ? F1 : F0; }
  __device__ __forceinline__ double *E(int d) const { return d ? E1 : E0; }
  __device__ __forceinline__ double *Q(int d) const { return d ? Q1 : Q0; }
  __device__ __forceinline__ double *S(int d) const { return d ? S1 : S0; }
};

// Doubles of shared memory of a tile of a x b cells (the host's and the
// kernel's size): NV interface values, NF flux variants, aux doubles per
// one-sided value and eig per interface while the variants are formed.
__host__ __device__ inline size_t tile2_doubles(int a, int b, int NV, int NF, bool jac, size_t off[8]) {
  const size_t cells = (size_t)(a + 4) * (b + 4);
  const size_t nI0 = (size_t)(a + 2) * (b + 2), nI1 = nI0;
  const size_t nF0 = (size_t)(a + 1) * b, nF1 = (size_t)(b + 1) * a;
  const size_t nP0 = (size_t)(a + 3) * (b + 2), nP1 = (size_t)(b + 3) * (a + 2);
  size_t o = 3 * cells;
  off[0] = o;  // src and code
  o += cells;
  off[1] = o;  // V[0]
  o += 2 * (size_t)NV * 3 * nI0;
  off[2] = o;  // V[1]
  o += 2 * (size_t)NV * 3 * nI1;
  off[3] = o;  // S[0], S[1]
  o += jac ? 2 * (size_t)a * b : 0;
  const size_t fl = (size_t)NF * 3 * (nF0 + nF1), aux = jac ? 5 * (nP0 + nP1) + 24 * (nI0 + nI1) : 0;
  off[4] = o;                               // F[0]
  off[5] = o + (size_t)NF * 3 * nF0;        // F[1]
  off[6] = o + (jac ? 5 * (nP0 + nP1) : 0); // Q[0] (E[0], E[1] at off[4])
  off[7] = nP0;
  return o + (fl > aux ? fl : aux);
}

__device__ __forceinline__ Smem2d tile2_smem(double *base, const Tile2d &t, int NV, int NF, bool jac) {
  size_t off[8];
  tile2_doubles(t.a, t.b, NV, NF, jac, off);
  Smem2d s;
  s.C = base;
  s.src = reinterpret_cast<int *>(base + off[0]);
  s.code = s.src + t.cells();
  s.V0 = base + off[1];
  s.V1 = base + off[2];
  s.S0 = base + off[3];
  s.S1 = s.S0 + t.a * t.b;
  s.F0 = base + off[4];
  s.F1 = base + off[5];
  s.E0 = base + off[4];
  s.E1 = s.E0 + 5 * off[7];
  s.Q0 = base + off[6];
  s.Q1 = s.Q0 + 24 * (size_t)t.nI(0);
  return s;
}

// ---- step 1
__device__ __forceinline__ void tile2_load(const Geo2 &G, const double *U, const Tile2d &t, const Smem2d &s) {
  const int nc = t.cells();
  for (int it = threadIdx.x; it < nc; it += blockDim.x) {
    double o[3];
    int src, code;
    cell_meta(G, U, t.x0 - 2 + it % t.W, t.y0 - 2 + it / t.W, o, src, code);
    s.C[it] = o[0];
    s.C[nc + it] = o[1];
    s.C[2 * nc + it] = o[2];
    s.src[it] = src;
    s.code[it] = code;
  }
}

// The eigenvectors at an interface, from the mean of its two cells.
struct Eig2 {
  double un, ut, c, i2c, ih;
};

__device__ __forceinline__ Eig2 eig2(const double a[3], const double b[3], double g) {
  Eig2 e;
  const double h = 0.5 * (a[0] + b[0]);
  e.ih = fast_rcp(h);
  e.un = __dmul_rn(0.5 * (a[1] + b[1]), e.ih);
  e.ut = __dmul_rn(0.5 * (a[2] + b[2]), e.ih);
  e.c = fast_sqrt(__dmul_rn(g, h));
  e.i2c = 0.5 * fast_rcp(e.c);
  return e;
}

// Characteristic variable f of the state u.
__device__ __forceinline__ double char2(const Eig2 &e, int f, const double u[3]) {
  if (f == 1) return fma(-e.ut, u[0], u[2]);
  if (f == 0) {
    const double X = __dmul_rn(e.un + e.c, e.i2c);
    return fma(X, u[0], -__dmul_rn(e.i2c, u[1]));
  }
  const double X = __dmul_rn(e.c - e.un, e.i2c);
  return fma(X, u[0], __dmul_rn(e.i2c, u[1]));
}

// One-sided WENO3 (Eq. 7-8) of the values (a, b, c): the nonlinear weights'
// s0, s1 and normalisation w (as weno3: D1 or D2 over D1 D2), and the value
// with given weights. SIDE 0: U^- (right of the middle cell), 1: U^+ (left).
template <int SIDE>
__device__ __forceinline__ void weno2_weights(double a, double b, double c, double &s0, double &s1, double &w) {
  const double d0 = c - b, d1 = b - a;
  const double e0 = fma(d0, d0, kZeta2), e1 = fma(d1, d1, kZeta2);
  s0 = __dmul_rn(e0, e0);
  s1 = __dmul_rn(e1, e1);
  const double D1 = fma(2.0, s0, s1), D2 = fma(2.0, s1, s0);
  const double inv = fast_rcp(__dmul_rn(D1, D2));
  w = __dmul_rn(SIDE == 0 ? D1 : D2, inv);
}
template <int SIDE, bool FROZEN>
__device__ __forceinline__ double weno2_value(double a, double b, double c, double s0, double s1, double w) {
  if (SIDE == 0) {
    const double q0 = fma(0.5, b, 0.5 * c), q1 = fma(1.5, b, -0.5 * a);
    return __dmul_rn(FROZEN ? fma(s0, q1, __dmul_rn(2.0 * s1, q0)) : fma(2.0 * s1, q0, __dmul_rn(s0, q1)), w);
  }
  const double p0 = fma(1.5, b, -0.5 * c), p1 = fma(0.5, a, 0.5 * b);
  return __dmul_rn(fma(s1, p0, __dmul_rn(2.0 * s0, p1)), w);
}

__device__ __forceinline__ void from_char2(const Eig2 &e, const double Wr[3], double out[3]) {
  out[0] = __dadd_rn(Wr[0], Wr[2]);
  out[1] = fma(e.un - e.c, Wr[0], __dmul_rn(e.un + e.c, Wr[2]));
  out[2] = fma(e.ut, Wr[2], fma(e.ut, Wr[0], Wr[1]));
}

// A cell's state in direction d's order: depth, normal and tangential momentum.
__device__ __forceinline__ void cell3(const Smem2d &s, int nc, int c, int d, double u[3]) {
  u[0] = s.C[c];
  u[1] = s.C[(1 + d) * nc + c];
  u[2] = s.C[(2 - d) * nc + c];
}
// Component m of the state in direction d's order, and back.
__device__ __forceinline__ int local2(int d, int m) { return m == 0 || d == 0 ? m : 3 - m; }

// ---- step 2: one side's unperturbed value at an interface; u[0..2] its
// stencil cells. JAC: Wr, and for the frozen linearisation the weights, are
// kept for step 3.
template <int SIDE, bool JAC, bool FROZEN>
__device__ __forceinline__ void rec_base2(const Tile2d &t, const Smem2d &s, int d, int idx, const Eig2 &e,
                                          const double u0[3], const double u1[3], const double u2[3], int NV) {
  const int nI = t.nI(d);
  double Wr[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const double a = char2(e, f, u0), b = char2(e, f, u1), c = char2(e, f, u2);
    double s0, s1, w;
    weno2_weights<SIDE>(a, b, c, s0, s1, w);
    Wr[f] = weno2_value<SIDE, FROZEN>(a, b, c, s0, s1, w);
    if (JAC) {
      double *Q = s.Q(d) + (size_t)SIDE * 12 * nI + idx;
      Q[f * nI] = Wr[f];
      if (FROZEN) {
        Q[(3 + 3 * f) * nI] = s0;
        Q[(4 + 3 * f) * nI] = s1;
        Q[(5 + 3 * f) * nI] = w;
      }
    }
  }
  double out[3];
  from_char2(e, Wr, out);
  double *V = s.V(d) + (size_t)SIDE * NV * 3 * nI + idx;
#pragma unroll
  for (int m = 0; m < 3; ++m) V[m * nI] = out[m];
}

template <bool JAC, bool FROZEN>
__device__ __forceinline__ void tile2_base(const Geo2 &G, const Tile2d &t, const Smem2d &s, int NV) {
  const int np0 = t.nP(0), np = np0 + t.nP(1), nc = t.cells();
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    const int d = p >= np0 ? 1 : 0, pp = d ? p - np0 : p;
    const int A = t.A(d), line = pp / (A + 3), q = pp % (A + 3), r = line - 1;
    double ul[3], ua[3], ub[3], ur[3];  // cells q-3 .. q (the outer two clamped; used by the sides that exist)
    cell3(s, nc, t.cell(d, max(q - 3, -2), r), d, ul);
    cell3(s, nc, t.cell(d, q - 2, r), d, ua);
    cell3(s, nc, t.cell(d, q - 1, r), d, ub);
    cell3(s, nc, t.cell(d, min(q, A + 1), r), d, ur);
    const Eig2 e = eig2(ua, ub, G.g);
    if (JAC) {
      double *E = s.E(d) + t.iP(d, line, q);
      const int nP = t.nP(d);
      E[0] = e.un;
      E[nP] = e.ut;
      E[2 * nP] = e.c;
      E[3 * nP] = e.i2c;
      E[4 * nP] = e.ih;
    }
    if (q >= 1) rec_base2<0, JAC, FROZEN>(t, s, d, t.iI(d, line, q, 0), e, ul, ua, ub, NV);
    if (q <= A + 1) rec_base2<1, JAC, FROZEN>(t, s, d, t.iI(d, line, q, 1), e, ua, ub, ur, NV);
  }
}

// ---- step 3: the value with stencil position sp's source cell perturbed in
// component m (of direction d's order). A momentum component leaves the characteristic variables that
// do not contain it, and a cell outside the mean leaves the eigenvectors: what
// does not change is taken from step 2.
template <int SIDE, bool FROZEN>
__device__ __forceinline__ void rec_variant2(const Geo2 &G, const Tile2d &t, const Smem2d &s, int d, int line, int q,
                                             int sp, int m, double eps, int NV) {
  const int nI = t.nI(d), nP = t.nP(d), nc = t.cells(), r = line - 1;
  const int idx = t.iI(d, line, q, SIDE), mg = local2(d, m);
  double *V = s.V(d) + (size_t)SIDE * NV * 3 * nI + idx;
  const double *Q = s.Q(d) + (size_t)SIDE * 12 * nI + idx;
  const double *Ep = s.E(d) + t.iP(d, line, q);
  double u[3][3];
  int hit = 0;  // stencil positions whose value changes
  const int al0 = q - 3 + SIDE, cs = s.src[t.cell(d, al0 + sp, r)];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int c = t.cell(d, al0 + p, r);
    cell3(s, nc, c, d, u[p]);
    const int code = (s.code[c] >> (2 * mg)) & 3;
    if (code && s.src[c] == cs) {
      hit |= 1 << p;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k == m) u[p][k] = code == 1 ? u[p][k] + eps : u[p][k] - eps;
    }
  }
  double out[3] = {V[0], V[nI], V[2 * nI]};
  if (hit) {
    Eig2 e{Ep[0], Ep[nP], Ep[2 * nP], Ep[3 * nP], Ep[4 * nP]};
    // the interface's own two cells: positions 1, 2 of U^-, 0, 1 of U^+
    const bool mean = !FROZEN && (hit & (SIDE == 0 ? 6 : 3));
    const double *ma = u[SIDE == 0 ? 1 : 0], *mb = u[SIDE == 0 ? 2 : 1];
    if (mean) {
      if (m == 0) e = eig2(ma, mb, G.g);
      else if (m == 1) e.un = __dmul_rn(0.5 * (ma[1] + mb[1]), e.ih);
      else e.ut = __dmul_rn(0.5 * (ma[2] + mb[2]), e.ih);
    }
    double Wr[3] = {Q[0], Q[nI], Q[2 * nI]};
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (m != 0 && (m == 1) == (f == 1)) continue;  // a variable without this component
      const double a = char2(e, f, u[0]), b = char2(e, f, u[1]), c = char2(e, f, u[2]);
      double s0, s1, w;
      if (FROZEN) {
        s0 = Q[(3 + 3 * f) * nI];
        s1 = Q[(4 + 3 * f) * nI];
        w = Q[(5 + 3 * f) * nI];
      } else {
        weno2_weights<SIDE>(a, b, c, s0, s1, w);
      }
      Wr[f] = weno2_value<SIDE, FROZEN>(a, b, c, s0, s1, w);
    }
    if (m == 2) out[2] = fma(e.ut, Wr[2], fma(e.ut, Wr[0], Wr[1]));
    else from_char2(e, Wr, out);
  }
  V += (size_t)(1 + 3 * sp + m) * 3 * nI;
#pragma unroll
  for (int k = 0; k < 3; ++k) V[k * nI] = out[k];
}

// Items ordered slot by slot: a warp's threads share (sp, m), and with them
// the branch taken above.
template <bool FROZEN>
__device__ __forceinline__ void tile2_variants(const Geo2 &G, const Tile2d &t, const Smem2d &s, double eps, int NV) {
  const int n0 = t.nI(0), n1 = t.nI(1), per = 2 * (n0 + n1);
  for (int w = threadIdx.x; w < 9 * per; w += blockDim.x) {
    const int slot = w / per, x = w % per, sp = slot / 3, m = slot % 3;
    const int side = x >= n0 + n1 ? 1 : 0, y = side ? x - (n0 + n1) : x, d = y >= n0 ? 1 : 0, z = d ? y - n0 : y;
    const int A = t.A(d), line = z / (A + 2), q = z % (A + 2) + 1 - side;
    if (side == 0) rec_variant2<0, FROZEN>(G, t, s, d, line, q, sp, m, eps, NV);
    else rec_variant2<1, FROZEN>(G, t, s, d, line, q, sp, m, eps, NV);
  }
}

// The slot of a line's value at interface q when interior cell cp is
// perturbed in component m: 0 (unperturbed) if its stencil does not read cp.
__device__ __forceinline__ int slot2(const Tile2d &t, const Smem2d &s, int d, int line, int q, int side, int cp,
                                     int m) {
  const int al0 = q - 3 + side, r = line - 1;
  int slot = 0;
#pragma unroll
  for (int p = 2; p >= 0; --p)
    if (s.src[t.cell(d, al0 + p, r)] == cp) slot = 1 + 3 * p + m;
  return slot;
}

__device__ __forceinline__ void val2(const Tile2d &t, const Smem2d &s, int d, int line, int q, int side, int slot,
                                     int NV, double v[3]) {
  const int nI = t.nI(d);
  const double *V = s.V(d) + ((size_t)side * NV + slot) * 3 * nI + t.iI(d, line, q, side);
  v[0] = V[0];
  v[1] = V[nI];
  v[2] = V[2 * nI];
}

// LLF flux of the states L, R in direction order (depth, normal, tangential).
__device__ __forceinline__ void llf2(const double L[3], const double R[3], double g, double F[3]) {
  const double iL = fast_rcp(L[0]), iR = fast_rcp(R[0]);
  const double uL = __dmul_rn(L[1], iL), vL = __dmul_rn(L[2], iL), uR = __dmul_rn(R[1], iR), vR = __dmul_rn(R[2], iR);
  const double FL[2] = {L[1], fma(__dmul_rn(0.5 * g, L[0]), L[0], __dmul_rn(L[1], uL))};
  const double FR[3] = {R[1], fma(__dmul_rn(0.5 * g, R[0]), R[0], __dmul_rn(R[1], uR)), __dmul_rn(R[1], vR)};
  const double a =
      0.5 * fmax(fabs(uL) + fast_sqrt(__dmul_rn(g, L[0])), fabs(uR) + fast_sqrt(__dmul_rn(g, R[0])));
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const double sum = m == 2 ? fma(L[1], vL, FR[2]) : __dadd_rn(FL[m < 2 ? m : 0], FR[m]);
    F[m] = fma(0.5, sum, -__dmul_rn(a, R[m] - L[m]));
  }
}

// ---- step 4: the flux of face q on cell line r (of the tile's T(d) lines),
// the mean over its two Gauss points, with interior cell cp perturbed in
// component m (of direction d's order; cp < 0: unperturbed).
__device__ __forceinline__ void face_flux2(const Geo2 &G, const Tile2d &t, const Smem2d &s, int d, int r, int q, int cp,
                                           int m, int NV, double fl[3]) {
  double L[3][3], R[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int sl = cp < 0 ? 0 : slot2(t, s, d, r + k, q, 0, cp, m), sr = cp < 0 ? 0 : slot2(t, s, d, r + k, q, 1, cp, m);
    val2(t, s, d, r + k, q, 0, sl, NV, L[k]);
    val2(t, s, d, r + k, q, 1, sr, NV, R[k]);
  }
  fl[0] = fl[1] = fl[2] = 0.0;
#pragma unroll
  for (int gp = 0; gp < 2; ++gp) {
    const double sg = gp == 0 ? -kTq : kTq;
    double l[3], rr[3], F[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      l[k] = fma(sg, L[2][k] - L[0][k], L[1][k]);
      rr[k] = fma(sg, R[2][k] - R[0][k], R[1][k]);
    }
    llf2(l, rr, G.g, F);
#pragma unroll
    for (int k = 0; k < 3; ++k) fl[k] = fma(0.5, F[k], fl[k]);
  }
}

// The cells that face q of line r reads, for the Jacobian's stencil: position
// p = 0 .. 3 along the face's direction (cells q-3 .. q) on line r + dr. J9
// keeps the cross of the two cells beside the face.
__device__ __forceinline__ void flux_variant2(bool full, int w, int &dr, int &p) {
  if (full) {
    dr = w / 4 - 1;
    p = w % 4;
  } else {
    dr = w < 4 ? 0 : (w < 6 ? -1 : 1);
    p = w < 4 ? w : 1 + (w & 1);
  }
}
__device__ __forceinline__ int flux_slot2(bool full, int dr, int p, int m) {
  const int w = full ? 4 * (dr + 1) + p : (dr == 0 ? p : (dr < 0 ? 3 : 5) + p);
  return 1 + 3 * w + m;
}

// Source component 1 + d of cell (al, r) of direction d's coordinates, from
// the depth at four interfaces of three lines; c: the cell's global index.
__device__ __forceinline__ double source2(const Geo2 &G, const Tile2d &t, const Smem2d &s, int d, int al, int r, int c,
                                          int cp, int m, int NV) {
  const int n = G.Nx * G.Ny, nI = t.nI(d);
  double hq[2][4];
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int side = f < 2 ? 1 : 0, q = al + f;
    double v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int sl = cp < 0 ? 0 : slot2(t, s, d, r + k, q, side, cp, m);
      v[k] = s.V(d)[((size_t)side * NV + sl) * 3 * nI + t.iI(d, r + k, q, side)];
    }
#pragma unroll
    for (int gp = 0; gp < 2; ++gp) hq[gp][f] = fma(gp == 0 ? -kTq : kTq, v[2] - v[0], v[1]);
  }
  double acc = 0.0;
#pragma unroll
  for (int gp = 0; gp < 2; ++gp)
#pragma unroll
    for (int pp = 0; pp < 2; ++pp) {
      const double h01 = fma(kLag2[pp][0], hq[gp][0], __dmul_rn(kLag2[pp][1], hq[gp][1]));
      const double hv = fma(kLag2[pp][3], hq[gp][3], fma(kLag2[pp][2], hq[gp][2], h01));
      const int beta = d == 0 ? gp : pp, gamma = d == 0 ? pp : gp;
      acc = fma(__dmul_rn(G.g, hv), G.gq[(d * 4 + 2 * beta + gamma) * n + c], acc);
    }
  return -0.25 * acc;
}

__device__ __forceinline__ Tile2d tile2_at(const Geo2 &G, int TX, int TY, int tile) {
  const int nx = (G.Nx + TX - 1) / TX;
  Tile2d t;
  t.x0 = (tile % nx) * TX;
  t.y0 = (tile / nx) * TY;
  t.a = min(TX, G.Nx - t.x0);
  t.b = min(TY, G.Ny - t.y0);
  t.W = t.a + 4;
  return t;
}

extern __shared__ double g_tile2_smem[];

// Faces are numbered x first, then y.
__device__ __forceinline__ void face_of(const Tile2d &t, int f, int &d, int &r, int &q, int &i) {
  const int n0 = t.nF(0);
  d = f >= n0 ? 1 : 0;
  i = d ? f - n0 : f;
  r = i / (t.A(d) + 1);
  q = i % (t.A(d) + 1) + 1;
}

// The residual of Eq. 20 by block `bid` of `nblk` over tiles of TX x TY cells,
// its l1 partial sum in partials[bid].
__device__ __forceinline__ void residual_tiles2(const ProbDev2 *P, int level, const double *U, double *R,
                                                double *partials, int TX, int TY, int bid, int nblk) {
  __shared__ double red[33];
  const Geo2 G = make_geo2(*P, level);
  const int n = G.Nx * G.Ny, ntiles = ((G.Nx + TX - 1) / TX) * ((G.Ny + TY - 1) / TY);
  const double rdx = 1.0 / G.dx, rdy = 1.0 / G.dy;
  double acc = 0.0;
  for (int tile = bid; tile < ntiles; tile += nblk) {
    const Tile2d t = tile2_at(G, TX, TY, tile);
    const Smem2d s = tile2_smem(g_tile2_smem, t, 1, 1, false);
    __syncthreads();  // the previous tile's values are read
    tile2_load(G, U, t, s);
    __syncthreads();
    tile2_base<false, false>(G, t, s, 1);
    __syncthreads();
    const int nF0 = t.nF(0), nF = nF0 + t.nF(1);
    for (int f = threadIdx.x; f < nF; f += blockDim.x) {
      int d, r, q, i;
      face_of(t, f, d, r, q, i);
      double fl[3];
      face_flux2(G, t, s, d, r, q, -1, 0, 1, fl);
      const int nf = t.nF(d);
#pragma unroll
      for (int k = 0; k < 3; ++k) s.F(d)[k * nf + i] = fl[k];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < t.a * t.b; k += blockDim.x) {
      const int ci = k % t.a, cj = k / t.a, c = (t.y0 + cj) * G.Nx + t.x0 + ci;
      const double S[3] = {0.0, source2(G, t, s, 0, ci, cj, c, -1, 0, 1), source2(G, t, s, 1, cj, ci, c, -1, 0, 1)};
      const int fx = cj * (t.a + 1) + ci, fy = ci * (t.b + 1) + cj, ny = t.nF(1);
      double sum = 0.0;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double *Fx = s.F0 + m * nF0 + fx, *Fy = s.F1 + local2(1, m) * ny + fy;
        const double Rm = fast_div(Fx[1] - Fx[0], G.dx, rdx) + fast_div(Fy[1] - Fy[0], G.dy, rdy) - S[m];
        R[m * n + c] = Rm;
        sum += fabs(Rm);
      }
      acc += sum;
    }
  }
  const double sum = block_sum2(acc, red);
  if (threadIdx.x == 0) partials[bid] = sum;
}

// The Jacobian of Eq. 12-13 over tiles of TX x TY cells (FROZEN: the frozen
// linearisation); R: the residual at U, for the differences and the
// regularisation.
template <typename TJ, bool FROZEN>
__device__ __forceinline__ void jacobian_tiles2(const ProbDev2 *P, int level, int st, const double *U, double eps,
                                                double alpha, const double *R, TJ *J, int cm, int TX, int TY, int bid,
                                                int nblk) {
  constexpr int NV = 10;
  const Geo2 G = make_geo2(*P, level);
  const bool full = st == ST_J21;
  const int n = G.Nx * G.Ny, ntiles = ((G.Nx + TX - 1) / TX) * ((G.Ny + TY - 1) / TY);
  const int K = st_size(st), kc = st_center(st), NW = full ? 12 : 8, NF = 1 + 3 * NW;
  const size_t Sj = blk_stride(cm, G.Nx, G.Ny);
  const double rdx = 1.0 / G.dx, rdy = 1.0 / G.dy, ieps = 1.0 / eps;
  for (int tile = bid; tile < ntiles; tile += nblk) {
    const Tile2d t = tile2_at(G, TX, TY, tile);
    const Smem2d s = tile2_smem(g_tile2_smem, t, NV, NF, true);
    __syncthreads();
    tile2_load(G, U, t, s);
    __syncthreads();
    tile2_base<true, FROZEN>(G, t, s, NV);
    __syncthreads();
    tile2_variants<FROZEN>(G, t, s, eps, NV);
    __syncthreads();
    const int nF0 = t.nF(0), nF = nF0 + t.nF(1), ncell = t.a * t.b;
    for (int w = threadIdx.x; w < NF * nF + 2 * ncell; w += blockDim.x) {
      if (w >= NF * nF) {  // the unperturbed sources
        const int x = w - NF * nF, d = x >= ncell ? 1 : 0, k = d ? x - ncell : x, ci = k % t.a, cj = k / t.a;
        s.S(d)[k] = source2(G, t, s, d, d == 0 ? ci : cj, d == 0 ? cj : ci, (t.y0 + cj) * G.Nx + t.x0 + ci, -1, 0, NV);
        continue;
      }
      const int v = w / nF;
      int d, r, q, i, cp = -1, m = 0;
      face_of(t, w % nF, d, r, q, i);
      if (v > 0) {
        int dr, p;
        flux_variant2(full, (v - 1) / 3, dr, p);
        m = (v - 1) % 3;
        const int al = q - 3 + p, ln = r + dr;
        const int pi = t.x0 + (d == 0 ? al : ln), pj = t.y0 + (d == 0 ? ln : al);
        if (pi < 0 || pi >= G.Nx || pj < 0 || pj >= G.Ny) continue;  // no such cell: no block reads this
        cp = pj * G.Nx + pi;
      }
      double fl[3];
      face_flux2(G, t, s, d, r, q, cp, m, NV, fl);  // m and fl in direction d's order
      const int nf = t.nF(d);
#pragma unroll
      for (int k = 0; k < 3; ++k) s.F(d)[(size_t)(v * 3 + k) * nf + i] = fl[k];
    }
    __syncthreads();
    for (int w = threadIdx.x; w < 3 * K * ncell; w += blockDim.x) {
      const int x = w % ncell, km = w / ncell, k = km / 3, m = km % 3, ci = x % t.a, cj = x / t.a;
      const int gi = t.x0 + ci, gj = t.y0 + cj, c = gj * G.Nx + gi;
      const size_t pc = blk_pos(cm, G.Nx, G.Ny, gi, gj);
      const int ox = st_off(st, k, 0), oy = st_off(st, k, 1), pi = gi + ox, pj = gj + oy;
      if (pi < 0 || pi >= G.Nx || pj < 0 || pj >= G.Ny) {
#pragma unroll
        for (int l = 0; l < 3; ++l) J[(size_t)(k * 9 + l * 3 + m) * Sj + pc] = TJ(0.0);
        continue;
      }
      const int cp = pj * G.Nx + pi;
      double fd[2][3], sd[2];
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const int al = d == 0 ? ci : cj, r = d == 0 ? cj : ci, oa = d == 0 ? ox : oy, ol = d == 0 ? oy : ox;
        const int nf = t.nF(d), i = r * (t.A(d) + 1) + al;  // the cell's left face
        const bool near = ol >= -1 && ol <= 1;              // its lines read the perturbed cell
        const int ml = local2(d, m);
        const int vl = near && oa + 2 <= 3 ? flux_slot2(full, ol, oa + 2, ml) : 0;
        const int vr = near && oa + 1 >= 0 ? flux_slot2(full, ol, oa + 1, ml) : 0;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          const int lf = local2(d, l);
          fd[d][l] = s.F(d)[(size_t)(vr * 3 + lf) * nf + i + 1] - s.F(d)[(size_t)(vl * 3 + lf) * nf + i];
        }
        sd[d] = near ? source2(G, t, s, d, al, r, c, cp, ml, NV) : s.S(d)[x];
      }
      const double R0[3] = {R[c], R[n + c], R[2 * n + c]};
      const double Sm[3] = {0.0, sd[0], sd[1]};
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const double Rp = fast_div(fd[0][l], G.dx, rdx) + fast_div(fd[1][l], G.dy, rdy) - Sm[l];
        double v = __dmul_rn(Rp - R0[l], ieps);
        if (l == m && k == kc) v = __dadd_rn(v, __dmul_rn(alpha, fabs(R0[0]) + fabs(R0[1]) + fabs(R0[2])));
        J[(size_t)(k * 9 + l * 3 + m) * Sj + pc] = TJ(v);
      }
    }
  }
}

}  // namespace
}  // namespace nswe
