// The lower levels of a 2D V-cycle (Algorithm 2) on one thread-block cluster.
//
// A V-cycle with nu = 20 visits every level some 160 to 320 times (one colour
// pass each), and on levels of a few thousand cells a pass is a microsecond of
// arithmetic at most: as launches, or on one block, the passes cost their
// launch gaps, their round trips to L2 for J and dU, or one SM's FP64 rate.
// Here a cluster of up to 16 CTAs runs them. Each CTA owns a band of row pairs
// and keeps that band's off-diagonal blocks, inverse diagonal blocks,
// right-hand side and correction in shared memory for the whole smoothing (for
// the whole kernel where all levels fit). A pass reads its own band's shared
// memory, and for the rows beyond it the neighbours' (distributed shared
// memory, 220 cycles). Between passes stands one cluster barrier, whose release
// is restricted to shared memory: measured 140 to 200 cycles against 380 to 480
// with the full release and acquire of global memory too. Every cell sees the
// arithmetic of sor_pass_split.
//
// A pass is bound by the FP64 unit in FP64 (30 instructions of 64 cycles per
// warp and round of cells at J9) and by the latency of one warp's loads in
// FP32. V-cycles with nu = 20, GB300, before (a launch per pass, the last
// levels on one block) and after: FP64 32 x 16 3.11 -> 0.86 ms, 64 x 32 3.75 ->
// 1.11; FP32 32 x 16 1.64 -> 0.40, 64 x 32 3.18 -> 0.56, 128 x 64 3.15 -> 1.01;
// J21 at 64 x 32 FP64 15.8 -> 6.0, FP32 36.0 -> 2.1.
#pragma once

#include <cooperative_groups.h>

namespace nswe {
namespace {

extern __shared__ __align__(16) unsigned char g_tail2_smem[];

// Values at an offset (in T) of the block's shared memory; offsets rather
// than pointers, so that the accesses are known to be shared ones.
template <typename T>
__device__ __forceinline__ T *smem2() {
  return reinterpret_cast<T *>(g_tail2_smem);
}

// The band of one level owned by a CTA, in its shared memory: planes of `cap`
// values by cell, a stride that puts the three components' lanes of a colour's
// cells on different banks. Blocks reaching outside the grid are zero here: a
// pass then needs no test for the grid's sides (what it reads past a row's end
// is multiplied by zero; two zeros stand before and after the band's dU).
template <typename T>
struct Band2 {
  int Nx, Ny, st, y0, y1;  // rows [y0, y1); empty for the CTAs beyond the level's row pairs
  int cap;                 // stride of the planes
  int J, Dinv, R, dU;      // offsets: [(K - 1) 9], [9], [3], [3] planes
  int tab, slots;          // offset of the colour tables, entries per colour
  // dU of the CTAs owning the rows above y0 and below y1, shifted so that a
  // cell's index in this band leads to its place there (its own: none).
  const T *up, *down;
};

// Plane stride for `cells` cells with the zeros around dU: 11 mod 32.
__host__ __device__ inline int band2_stride(int cells) { return (cells + 4 + 20) / 32 * 32 + 11; }
__host__ __device__ inline int st_ncolours(int st) { return st == ST_J9 ? 3 : st == ST_J21 ? 9 : st == ST_P5 ? 2 : 4; }
// Entries of a colour's table for `rows` rows: the items of a colour pass
// (sor_items) of the stencil's own colouring.
__host__ __device__ inline int band2_slots(int Nx, int st, int rows) {
  const int C = st == ST_J9 || st == ST_J21 ? 3 : 2;
  return (Nx + C - 1) / C * (st == ST_J9 || st == ST_P5 ? rows : (rows + C - 1) / C);
}

// Values of T a level's band takes in a CTA's shared memory.
__host__ __device__ inline size_t band2_values(int Nx, int Ny, int st, int ctas, size_t sizeof_t) {
  const int K = st == ST_J9 ? 9 : st == ST_J21 ? 21 : st == ST_P5 ? 5 : 9;
  const int pairs = Ny / 2, nA = pairs < ctas ? pairs : ctas, rows = 2 * ((pairs + nA - 1) / nA);
  const size_t tab = 8 * (size_t)band2_slots(Nx, st, rows) * st_ncolours(st) / sizeof_t;
  return ((size_t)((K - 1) * 9 + 15) * band2_stride(rows * Nx) + tab + 1) / 2 * 2;
}

template <typename T>
__device__ __forceinline__ Band2<T> band2(const Tail2<T> &t, int l, int rank, int ctas) {
  Band2<T> b;
  b.Nx = t.Nx[l];
  b.Ny = t.Ny[l];
  b.st = t.st[l];
  const int pairs = b.Ny / 2, nA = min(pairs, ctas), rows = 2 * ((pairs + nA - 1) / nA);
  auto first = [&](int r) { return 2 * (pairs * r / nA); };
  b.y0 = rank < nA ? first(rank) : b.Ny;
  b.y1 = rank < nA ? first(rank + 1) : b.Ny;
  b.tab = t.off[l];  // 8-byte entries first
  b.slots = band2_slots(b.Nx, b.st, rows);
  b.cap = band2_stride(rows * b.Nx);
  b.J = b.tab + 8 / (int)sizeof(T) * b.slots * st_ncolours(b.st);
  b.Dinv = b.J + (st_size(b.st) - 1) * 9 * b.cap;
  b.R = b.Dinv + 9 * b.cap;
  b.dU = b.R + 3 * b.cap + 2;
  auto cl = cooperative_groups::this_cluster();
  b.up = b.down = smem2<T>() + b.dU;
  if (rank > 0 && rank < nA) b.up = cl.map_shared_rank(smem2<T>() + b.dU, rank - 1) + (b.y0 - first(rank - 1)) * b.Nx;
  if (rank + 1 < nA) b.down = cl.map_shared_rank(smem2<T>() + b.dU, rank + 1) - (b.y1 - b.y0) * b.Nx;
  return b;
}

// Item t of colour col of the band (three lanes' cell): its index in the band
// (-1: none; its rows then count as outside), and where its rows j - 2, j - 1, j + 1, j + 2 lie (2 bits each:
// 0 in the band, 1 in the CTA above, 2 in the one below, 3 outside the grid).
__device__ __forceinline__ int2 band2_item(int Nx, int Ny, int st, int y0, int y1, int mode, int Kc, int col,
                                           int t) {
  int P, W, items, i, j;
  sor_items(Nx, Ny, st, mode, Kc, col, P, W, items);
  if (mode == 0) {
    const int j0 = y0 + (col / P - y0 % P + P) % P;
    if (W == 0) return make_int2(-1, 255);
    i = col % P + (t % W) * P;
    j = j0 + (t / W) * P;
  } else {
    j = y0 + t / W;
    const int a = mode == 1 ? col - j : j + Nx - 1 - col;
    i = ((a % Kc) + Kc) % Kc + (t % W) * Kc;
  }
  if (i >= Nx || j >= y1) return make_int2(-1, 255);
  int where = 0;
  for (int r = 0; r < 4; ++r) {
    const int q = j + (r < 2 ? r - 2 : r - 1);
    where |= (q < 0 || q >= Ny ? 3 : q < y0 ? 1 : q >= y1 ? 2 : 0) << (2 * r);
  }
  return make_int2((j - y0) * Nx + i, where);
}

__device__ __forceinline__ void cluster_sync2() { cooperative_groups::this_cluster().sync(); }

// The band's colour tables, off-diagonal and inverse diagonal blocks.
template <typename T>
__device__ __forceinline__ void band2_load_op(const Tail2<T> &t, int l, const Band2<T> &b) {
  const int Nx = b.Nx, cells = (b.y1 - b.y0) * Nx, K = st_size(b.st), kc = st_center(b.st);
  T *sm = smem2<T>();
  int2 *tab = reinterpret_cast<int2 *>(sm + b.tab);
  for (int w = threadIdx.x; w < b.slots * st_ncolours(b.st); w += blockDim.x)
    tab[w] = band2_item(Nx, b.Ny, b.st, b.y0, b.y1, 0, 0, w / b.slots, w % b.slots);
  if (threadIdx.x < 6) {
    const int z = b.dU + threadIdx.x / 2 * b.cap + threadIdx.x % 2;
    sm[z - 2] = sm[z + cells] = T(0.0);
  }
  const int cm = l == t.l0 ? t.cm : 0;
  const size_t S = blk_stride(cm, Nx, b.Ny);
  const T *J = t.J[l], *Dinv = t.Dinv[l];
  const int planes = (K - 1) * 9 + 9;
#pragma unroll 4
  for (int w = threadIdx.x; w < planes * cells; w += blockDim.x) {
    const int p = w / cells, c = w % cells, x = c % Nx, y = b.y0 + c / Nx;
    const size_t pc = blk_pos(cm, Nx, b.Ny, x, y);
    T v;
    if (p < (K - 1) * 9) {
      const int k = p / 9 + (p / 9 >= kc ? 1 : 0), i = x + st_off(b.st, k, 0), j = y + st_off(b.st, k, 1);
      v = i >= 0 && i < Nx && j >= 0 && j < b.Ny ? J[(size_t)(p + (k > kc ? 9 : 0)) * S + pc] : T(0.0);
    } else {
      v = Dinv[(size_t)(p - (K - 1) * 9) * S + pc];
    }
    sm[b.J + p * b.cap + c] = v;
  }
}

// The band's right-hand side, and its correction: from global memory, or zero.
template <typename T>
__device__ __forceinline__ void band2_load_vec(const Tail2<T> &t, int l, const Band2<T> &b, bool rhs, bool zero) {
  const int n = b.Nx * b.Ny, cells = (b.y1 - b.y0) * b.Nx;
  T *sm = smem2<T>();
  for (int w = threadIdx.x; w < 3 * cells; w += blockDim.x) {
    const int m = w / cells, c = w % cells, at = m * n + b.y0 * b.Nx + c;
    if (rhs) sm[b.R + m * b.cap + c] = t.R[l][at];
    sm[b.dU + m * b.cap + c] = zero ? T(0.0) : t.dU[l][at];
  }
}

template <typename T>
__device__ __forceinline__ void band2_store(const Tail2<T> &t, int l, const Band2<T> &b) {
  const int n = b.Nx * b.Ny, cells = (b.y1 - b.y0) * b.Nx;
  for (int w = threadIdx.x; w < 3 * cells; w += blockDim.x) {
    const int m = w / cells, c = w % cells;
    t.dU[l][m * n + b.y0 * b.Nx + c] = smem2<T>()[b.dU + m * b.cap + c];
  }
}

// The coarse correction added to the band (Eq. 25).
template <typename T>
__device__ __forceinline__ void band2_prolong(const Tail2<T> &t, int l, const Band2<T> &b) {
  const T *dUc = t.dU[l + 1];
  const int nc = (b.Nx / 2) * (b.Ny / 2), cells = (b.y1 - b.y0) * b.Nx;
  for (int w = threadIdx.x; w < 3 * cells; w += blockDim.x) {
    const int m = w / cells, c = w % cells, y = b.y0 + c / b.Nx, x = c % b.Nx;
    smem2<T>()[b.dU + m * b.cap + c] += dUc[m * nc + (y / 2) * (b.Nx / 2) + x / 2];
  }
}

// One colour pass of the band's cells: three lanes per cell as sor_pass_split
// (in FP32 a thread per cell with vector loads was slower but for the largest
// level, 0.47 against 0.40 ms for a V-cycle at 32 x 16). TAB: the stencil's own
// colouring, whose items were listed by band2_load_op (finding an item's cell
// and neighbours took longer than its update).
template <typename T, int ST, bool TAB>
__device__ __forceinline__ void band2_pass(const Band2<T> &b, T omega, int mode, int Kc, int col, int reps) {
  constexpr int K = ST == ST_J9 ? 9 : ST == ST_J21 ? 21 : ST == ST_P5 ? 5 : 9;
  constexpr int kc = ST == ST_J9 ? 4 : ST == ST_J21 ? 10 : ST == ST_P5 ? 2 : 4;
  const int Nx = b.Nx, cap = b.cap, items = TAB ? b.slots : (Nx + Kc - 1) / Kc * (b.y1 - b.y0);
  T *dU = smem2<T>() + b.dU;
  const int2 *tab = reinterpret_cast<const int2 *>(smem2<T>() + b.tab) + (TAB ? col * b.slots : 0);
  const int lane = threadIdx.x & 31, g = lane / 3, l = lane - 3 * g, src = min(3 * g, 29);
  for (int w = threadIdx.x >> 5; w * 10 < items; w += blockDim.x >> 5) {  // warp-uniform
    const int t = w * 10 + g;
    int2 e = make_int2(-1, 255);
    if (lane < 30 && t < items) e = TAB ? tab[t] : band2_item(Nx, b.Ny, ST, b.y0, b.y1, mode, Kc, col, t);
    const bool on = e.x >= 0;
    const int c = on ? e.x : 0;
    const T *x[4];  // the dU of the cells above and below: rows j - 2, j - 1, j + 1, j + 2
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int at = (e.y >> (2 * r)) & 3, d = c + (at == 3 ? 0 : (r < 2 ? r - 2 : r - 1) * Nx);
      x[r] = (at == 1 ? b.up : at == 2 ? b.down : dU) + d;
    }
    const T *const J = smem2<T>() + b.J + 3 * l * cap + c, *const own = dU + c;
    T r = smem2<T>()[b.R + l * cap + c];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (k == kc) continue;
      const int ox = off_c<ST>(k, 0), oy = off_c<ST>(k, 1), jk = (k < kc ? k : k - 1) * 9;
      const T *xk = (oy == 0 ? own : x[oy < 0 ? oy + 2 : oy + 1]) + ox;
      r = fma(J[jk * cap], xk[0], r);
      r = fma(J[(jk + 1) * cap], xk[cap], r);
      r = fma(J[(jk + 2) * cap], xk[2 * cap], r);
    }
    const T r0 = __shfl_sync(0xffffffffu, r, src);
    const T r1 = __shfl_sync(0xffffffffu, r, src + 1);
    const T r2 = __shfl_sync(0xffffffffu, r, src + 2);
    const T *D = smem2<T>() + b.Dinv + 3 * l * cap + c;
    const T u = relax(own[l * cap], dinv_row(D[0], D[cap], D[2 * cap], r0, r1, r2), omega, reps);
    if (on) dU[l * cap + c] = u;
  }
}

// One colour pass and the barrier after it: the shared-memory writes of every
// CTA before it are visible to the others' reads of its shared memory after it.
template <typename T>
__device__ __forceinline__ void band2_pass_any(const Band2<T> &b, T omega, int mode, int Kc, int col, int reps) {
  if (mode == 0) {
    if (b.st == ST_J9) band2_pass<T, ST_J9, true>(b, omega, 0, 0, col, reps);
    else if (b.st == ST_P5) band2_pass<T, ST_P5, true>(b, omega, 0, 0, col, reps);
    else if (b.st == ST_P9) band2_pass<T, ST_P9, true>(b, omega, 0, 0, col, reps);
    else band2_pass<T, ST_J21, true>(b, omega, 0, 0, col, reps);
  } else if (b.st == ST_J9) {  // the directional schedule: cross stencils only
    band2_pass<T, ST_J9, false>(b, omega, mode, Kc, col, reps);
  } else {
    band2_pass<T, ST_P5, false>(b, omega, mode, Kc, col, reps);
  }
  __syncwarp();
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory");
}

// The colour passes of `steps` smoothing steps in the host's order (smooth2):
// pass(mode, Kc, colour, reps).
template <typename F>
__device__ __forceinline__ void each_pass2(int st, int steps, int Kc, F &&pass) {
  if (Kc >= 3 && (st == ST_J9 || st == ST_P5)) {
    for (int s = 0; s < steps; ++s)
      for (int d = 0; d < 4; ++d)
        for (int q = 0; q < Kc; ++q) pass((d % 2) + 1, Kc, d < 2 ? q : Kc - 1 - q, 1);
    return;
  }
  // half sweeps 0 .. C-1 and C-1 .. 0 in turn; the colour at which a half
  // sweep ends opens the next one, its two visits run as one
  const int C = st_ncolours(st), H = 4 * steps;
  if (H > 0) pass(0, 0, 0, 1);
  for (int h = 0; h < H; ++h) {
    const bool up = (h & 1) == 0;
    for (int q = 1; q < C; ++q) pass(0, 0, up ? q : C - 1 - q, q == C - 1 && h < H - 1 ? 2 : 1);
  }
}

// Defect restriction (Eq. 24) of the band's row pairs, the order of
// restrict_cells2; the operator comes from global memory.
template <typename T>
__device__ __forceinline__ void band2_restrict(const Tail2<T> &t, int l, const Band2<T> &b) {
  const int Nx = b.Nx, Ny = b.Ny, Ncx = Nx / 2, nc = Ncx * (Ny / 2), K = st_size(b.st);
  const int cm = l == t.l0 ? t.cm : 0;
  const size_t S = blk_stride(cm, Nx, Ny);
  const T *Jg = t.J[l], *sm = smem2<T>();
  const int items = 3 * Ncx * ((b.y1 - b.y0) / 2);
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    const int I = w % Ncx, q = w / Ncx, m = q % 3, Jy = b.y0 / 2 + q / 3;
    T s = T(0.0);
    for (int e = 0; e < 4; ++e) {
      const int xi = 2 * I + (e & 1), yi = 2 * Jy + (e >> 1), c = (yi - b.y0) * Nx + xi;
      const size_t pc = blk_pos(cm, Nx, Ny, xi, yi);
      T r = t.R[l][m * Nx * Ny + yi * Nx + xi];
      for (int k = 0; k < K; ++k) {
        const int ox = st_off(b.st, k, 0), oy = st_off(b.st, k, 1), y = yi + oy;
        if (xi + ox < 0 || xi + ox >= Nx || y < 0 || y >= Ny) continue;
        const T *x = (y < b.y0 ? b.up : y >= b.y1 ? b.down : sm + b.dU) + c + oy * Nx + ox;
        const T *J = Jg + (size_t)(k * 9 + m * 3) * S + pc;
        r = fma(J[0], x[0], r);
        r = fma(J[S], x[b.cap], r);
        r = fma(J[2 * S], x[2 * b.cap], r);
      }
      s += r;
    }
    t.R[l + 1][m * nc + Jy * Ncx + I] = s;
  }
}

// ---------------------------------------------------------------------------- coarsest direct solve

// dU = -A^{-1} R with the LU factors of lu_block2 (unknown 3c + m), by one
// block: row i on thread i (strided), one barrier per elimination step, the
// right-hand side double-buffered in x (3 N3 values of shared memory). A(i, k)
// at A[i rs + k cs].
template <typename T>
__device__ __forceinline__ void lu_solve_block(int n, const T *A, int rs, int cs, const int *piv, const T *R, T *x,
                                               T *dU) {
  const int N3 = 3 * n, nt = min((N3 + 31) / 32 * 32, (int)blockDim.x), tid = threadIdx.x;
  if (tid >= nt) return;
  auto bar = [&] { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); };
  T *xa = x, *xb = x + N3, *rinv = x + 2 * N3;
  for (int i = tid; i < N3; i += nt) {
    xa[i] = -R[(i % 3) * n + i / 3];
    rinv[i] = T(1.0) / A[(size_t)i * rs + (size_t)i * cs];
  }
  bar();
  for (int k = 0; k < N3; ++k) {
    const int p = piv[k];
    const T xk = xa[p], xo = xa[k];  // rows k and p change places
    for (int i = k + tid; i < N3; i += nt) {
      if (i == k) xb[i] = xk;
      else xb[i] = fma(-A[(size_t)i * rs + (size_t)k * cs], xk, i == p ? xo : xa[i]);
    }
    if (tid == 0) dU[(k % 3) * n + k / 3] = xk;
    T *s = xa;
    xa = xb;
    xb = s;
    bar();
  }
  for (int i = tid; i < N3; i += nt) xa[i] = dU[(i % 3) * n + i / 3];
  bar();
  for (int k = N3 - 1; k >= 0; --k) {
    const T xk = mul_r(xa[k], rinv[k]);
    for (int i = tid; i < k; i += nt) xb[i] = fma(-A[(size_t)i * rs + (size_t)k * cs], xk, xa[i]);
    if (tid == 0) dU[(k % 3) * n + k / 3] = xk;
    T *s = xa;
    xa = xb;
    xb = s;
    bar();
  }
}

// `cycles` V-cycles of the levels ls .. L by the calling cluster. The coarsest
// factorisation may still run when the kernel starts (launched with
// programmatic serialization right after it): it is waited for before its
// first use, so the smoothing on the way down hides it. Everything else the
// cluster reads was complete before the factorisation began.
template <typename T>
__device__ __forceinline__ void vcycle_cluster2(const Tail2<T> &t, int nu1, int nu2, double omega_d, int Kc,
                                                int cycles) {
  T *const smem = smem2<T>();
  auto cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
  const T omega = T(omega_d);
  const int nL = t.Nx[t.L] * t.Ny[t.L], N3 = 3 * nL;
  T *const As = smem + t.lu_off;  // factors (transposed, if they fit), then 3 N3 values of the solve
  T *const xs = As + (t.lu_smem ? (size_t)N3 * (N3 + 1) : 0);
  for (int l = t.ls; l < t.shared_from; ++l) band2_load_op(t, l, band2(t, l, rank, ctas));
  for (int cyc = 0; cyc < cycles; ++cyc) {
    for (int l = t.ls; l < t.L; ++l) {
      const Band2<T> b = band2(t, l, rank, ctas);
      const bool keep = l < t.shared_from;
      if (!keep) band2_load_op(t, l, b);
      band2_load_vec(t, l, b, l > t.ls || cyc == 0 || !keep, l > t.ls);
      cluster_sync2();
      each_pass2(b.st, nu1, Kc,
                 [&](int mode, int kc, int col, int reps) { band2_pass_any(b, omega, mode, kc, col, reps); });
      band2_restrict(t, l, b);
      if (!keep) band2_store(t, l, b);
      cluster_sync2();
    }
    if (rank == 0) {
      if (cyc == 0) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (t.lu_smem) {
          for (int w = threadIdx.x; w < N3 * N3; w += blockDim.x) As[(size_t)(w % N3) * (N3 + 1) + w / N3] = t.A[w];
          __syncthreads();
        }
      }
      if (t.lu_smem) lu_solve_block(nL, As, 1, N3 + 1, t.piv, t.R[t.L], xs, t.dU[t.L]);
      else lu_solve_block(nL, t.A, N3, 1, t.piv, t.R[t.L], xs, t.dU[t.L]);
    }
    cluster_sync2();
    for (int l = t.L - 1; l >= t.ls; --l) {
      const Band2<T> b = band2(t, l, rank, ctas);
      if (l >= t.shared_from) {
        band2_load_op(t, l, b);
        band2_load_vec(t, l, b, true, false);
        __syncthreads();
      }
      band2_prolong(t, l, b);
      cluster_sync2();
      each_pass2(b.st, nu2, Kc,
                 [&](int mode, int kc, int col, int reps) { band2_pass_any(b, omega, mode, kc, col, reps); });
      band2_store(t, l, b);
      cluster_sync2();
    }
  }
}

}  // namespace
}  // namespace nswe
