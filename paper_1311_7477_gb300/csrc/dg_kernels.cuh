// The hot-path kernels, templated on the arithmetic type T (double or float) and the
// number of nodes per cell and dimension N (1..5).
//
//   rhs_kernel       bracket J(psi, omega) (Eq. J) + viscous term + multistep update, fused, in
//                    fixed point on the integer pipe
//   apply_kernel     the LDG operator A or Delta_h on a field
//   cg_kernel        persistent cooperative conjugate-gradient Poisson solve (Sec. 6)
//   mixed_cg_kernel  float64 residual / float32 inner CG iterative refinement
//   invariants_*     V, E, Omega by quadrature (Eq. quantities, Eq. def_norm)
#pragma once

#include <type_traits>

#include "dg_device.cuh"
#include "dg_df.cuh"
#include "dg_fixed_tables.cuh"

namespace dgk {

constexpr int kThreads = 256;
// Threads of a standalone RHS block and the blocks per SM its registers are sized for (two tiles of
// 100 KB at n = 5, three of 68 KB at n = 4 fill an SM's shared memory; measured on 1000^2 cells:
// n = 5 1223 us with 320 threads, 1286 / 1282 with 416 / 512; n = 4 695 us with 256 threads and three
// blocks, 823 with 320 / 352 and two).
template <int N>
__host__ __device__ constexpr int rhs_threads() {
  return N == 5 ? 320 : 256;
}
template <int N>
__host__ __device__ constexpr int rhs_blocks() {
  return N == 5 ? 2 : 3;
}

// Copies an operator table (a kernel parameter or a global array) to shared memory: the
// solves index it with per-thread node numbers, which shared memory serves without the
// serialisation of divergent constant-bank reads.
template <class Tab>
__device__ __forceinline__ const Tab& stage_table(const Tab& src, unsigned char* dst) {
  static_assert(sizeof(Tab) % 4 == 0, "table size");
  const unsigned int* s = reinterpret_cast<const unsigned int*>(&src);
  unsigned int* d = reinterpret_cast<unsigned int*>(dst);
  for (int i = threadIdx.x; i < int(sizeof(Tab) / 4); i += blockDim.x) d[i] = s[i];
  __syncthreads();
  return *reinterpret_cast<const Tab*>(dst);
}

template <class Tab>
__host__ __device__ constexpr size_t table_bytes() {
  return (sizeof(Tab) + 15) & ~size_t(15);
}


__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }

// a*b - c*d with both products rounded separately (never contracted into an FMA), so that
// the bracket's antisymmetry J(f, g) = -J(g, f) and J(f, f) = 0 hold bitwise.
template <typename T>
__device__ __forceinline__ T prod_diff(T a, T b, T c, T d) {
  return sub_rn(mul_rn(a, b), mul_rn(c, d));
}

// =========================================================================================
// Right-hand side: R = -J(psi, omega) + D Delta_h omega and the update
//   omega_out = omega_base + dt (c_new R + sum_m c_hist[m] hist[m])
// (AB3: c = 23/12, -16/12, 5/12; the RK4 start-up stages use other coefficients).
// One thread block per tile of TY x TX cells; the tile and a one-cell halo ring (corners
// included: the second derivatives of J+x and Jx+ reach the diagonal neighbours) are staged
// in shared memory, all intermediate products stay there.
// =========================================================================================
struct RhsArgs {
  const double* psi;        // stream function; times sqrt(W) if psi_scaled
  const double* omega_in;   // vorticity at which R is evaluated (halo reads)
  const double* omega_base; // omega^k of the update (own nodes only; may alias omega_out)
  double* omega_out;        // updated vorticity, or J in bracket-only mode
  double* R_out;            // fresh R (may alias one hist buffer); may be null
  const double* hist[3];
  double c_new;
  double c_hist[3];
  int nhist;
  double dt;
  double visc;
  int psi_scaled;
  int bracket_only;
  int parts;                // bit 0: J++, bit 1: J+x, bit 2: Jx+ (0 = all three, J of Eq. J)
};

template <typename T, int N>
__host__ __device__ constexpr size_t rhs_smem_values(int TY, int TX) {
  return (size_t)(TY + 2) * (TX + 2) * (7 * (N * N + 1) + 12 * N);
}

// One box of the right-hand side in float64 (smem: rhs_smem_values<double, N>(G.TY, G.TX) values).
template <typename T, int N>
__device__ __forceinline__ void rhs_box_float(const Ops2D<T, N>& C, const Geom& G, const RhsArgs& A, const TileBox& B,
                                              unsigned char* smem_raw) {
  constexpr int NN = N * N;
  constexpr int CS = NN + 1;  // padded cell stride in shared memory
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int boxc = (G.TY + 2) * (G.TX + 2);
  T* sPsi = sm;
  T* sOm = sPsi + boxc * CS;
  T* sFx = sOm + boxc * CS;  // f_x, later h2 = f_x g - f g_x   (cells with rx in [0,TXe))
  T* sGx = sFx + boxc * CS;
  T* sFy = sGx + boxc * CS;  // f_y, later h1 = f g_y - f_y g   (cells with ry in [0,TYe))
  T* sGy = sFy + boxc * CS;
  T* sJ = sGy + boxc * CS;   // J++ on the tile
  T* t0 = sJ + boxc * CS;
  T *tPxR = t0, *tPxL = t0 + boxc * N, *tPyR = t0 + 2 * boxc * N, *tPyL = t0 + 3 * boxc * N;
  T *tOxR = t0 + 4 * boxc * N, *tOxL = t0 + 5 * boxc * N, *tOyR = t0 + 6 * boxc * N, *tOyL = t0 + 7 * boxc * N;
  T *tLxR = t0 + 8 * boxc * N, *tLxL = t0 + 9 * boxc * N, *tLyR = t0 + 10 * boxc * N, *tLyL = t0 + 11 * boxc * N;
  const int BW = B.BW;

  // S0: stage psi and omega on the tile with its full halo ring.
  stage_box<T, N>(G, B, sPsi, true, [&](size_t g, int k, bool) {
    const double v = A.psi[g];
    return A.psi_scaled ? T(v) * C.isw[k] : T(v);
  });
  stage_box<T, N>(G, B, sOm, true, [&](size_t g, int, bool) { return T(A.omega_in[g]); });
  __syncthreads();

  // S1: face traces for the first derivatives (every staged cell) and the viscous term.
  line_traces<T, N>(B, sPsi, sPsi, C.dx, C.dy, tPxR, tPxL, tPyR, tPyL, true);
  line_traces<T, N>(B, sOm, sOm, C.dx, C.dy, tOxR, tOxL, tOyR, tOyL, true);
  if (A.visc != 0.0) line_traces<T, N>(B, sOm, sOm, C.lx, C.ly, tLxR, tLxL, tLyR, tLyL, false);
  __syncthreads();
  if (G.bc) {  // Dirichlet: f^ = 0 on the boundary faces of the derivatives; LDG first cells
    dirichlet_ghost_traces<T, N>(G, B, tPxR, tPxL, tPyR, tPyL, true);
    dirichlet_ghost_traces<T, N>(G, B, tOxR, tOxL, tOyR, tOyL, true);
    if (A.visc != 0.0) dirichlet_first_traces<T, N>(B, sOm, sOm, C.lx, C.ly, tLxL, tLyL);
    __syncthreads();
  }

  // S2: f_x, g_x on rows [-1, TYe] x cols [0, TXe); f_y, g_y on rows [0, TYe) x cols [-1, TXe].
  {
    const int n1 = (B.TYe + 2) * B.TXe * NN;
    const int n2 = B.TYe * (B.TXe + 2) * NN;
    for (int i = threadIdx.x; i < n1 + n2; i += blockDim.x) {
      if (i < n1) {
        const int c = i / NN, k = i - (i / NN) * NN;
        const int ry = quot(c, B.mTXe) - 1, rx = c - (ry + 1) * B.TXe;
        const int lc = (ry + 1) * BW + rx + 1;
        const int a = k / N, b = k - (k / N) * N;
        sFx[lc * CS + k] = op_x_at<T, N>(sPsi, tPxR, tPxL, C.dx, lc, a, b);
        sGx[lc * CS + k] = op_x_at<T, N>(sOm, tOxR, tOxL, C.dx, lc, a, b);
      } else {
        const int ii = i - n1;
        const int c = ii / NN, k = ii - (ii / NN) * NN;
        const int w = B.TXe + 2;
        const int ry = c / w, rx = c - (c / w) * w - 1;
        const int lc = (ry + 1) * BW + rx + 1;
        const int a = k / N, b = k - (k / N) * N;
        sFy[lc * CS + k] = op_y_at<T, N>(sPsi, tPyR, tPyL, C.dy, lc, BW, a, b);
        sGy[lc * CS + k] = op_y_at<T, N>(sOm, tOyR, tOyL, C.dy, lc, BW, a, b);
      }
    }
  }
  __syncthreads();

  // Which parts enter (Eq. J): J = s (c0 J++ + J+x + Jx+) with J+x = D_x(f g_y) - D_y(f g_x),
  // Jx+ = D_y(f_x g) - D_x(f_y g); as h1 = a1 f g_y - b1 f_y g, h2 = a2 f_x g - b2 f g_x.
  const int parts = A.parts ? A.parts : 7;
  const bool use_pp = parts & 1, use_px = parts & 2, use_xp = parts & 4;
  const int nparts = int(use_pp) + int(use_px) + int(use_xp);
  // S3a: J++ = f_x g_y - f_y g_x on the tile.
  const int nin = B.TYe * B.TXe * NN;
  for (int i = threadIdx.x; i < nin; i += blockDim.x) {
    const int c = i / NN, k = i - (i / NN) * NN;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int o = ((ry + 1) * BW + rx + 1) * CS + k;
    sJ[o] = prod_diff(sFx[o], sGy[o], sFy[o], sGx[o]);
  }
  __syncthreads();

  // S3b: h1 = f g_y - f_y g (in place of f_y), h2 = f_x g - f g_x (in place of f_x).
  {
    const int n1 = B.TYe * (B.TXe + 2) * NN;
    const int n2 = (B.TYe + 2) * B.TXe * NN;
    for (int i = threadIdx.x; i < n1 + n2; i += blockDim.x) {
      if (i < n1) {
        const int c = i / NN, k = i - (i / NN) * NN;
        const int w = B.TXe + 2;
        const int ry = c / w, rx = c - (c / w) * w - 1;
        const int o = ((ry + 1) * BW + rx + 1) * CS + k;
        if (nparts == 3)
          sFy[o] = prod_diff(sPsi[o], sGy[o], sFy[o], sOm[o]);
        else
          sFy[o] = (use_px ? mul_rn(sPsi[o], sGy[o]) : T(0)) - (use_xp ? mul_rn(sFy[o], sOm[o]) : T(0));
      } else {
        const int ii = i - n1;
        const int c = ii / NN, k = ii - (ii / NN) * NN;
        const int ry = quot(c, B.mTXe) - 1, rx = c - (ry + 1) * B.TXe;
        const int o = ((ry + 1) * BW + rx + 1) * CS + k;
        if (nparts == 3)
          sFx[o] = prod_diff(sFx[o], sOm[o], sPsi[o], sGx[o]);
        else
          sFx[o] = (use_xp ? mul_rn(sFx[o], sOm[o]) : T(0)) - (use_px ? mul_rn(sPsi[o], sGx[o]) : T(0));
      }
    }
  }
  __syncthreads();

  // S4: traces of h1 along x and of h2 along y (reusing the psi trace arrays).
  line_traces<T, N>(B, sFy, sFx, C.dx, C.dy, tPxR, tPxL, tPyR, tPyL, false);
  __syncthreads();
  if (G.bc) {
    dirichlet_ghost_traces<T, N>(G, B, tPxR, tPxL, tPyR, tPyL, false);
    __syncthreads();
  }

  // S5: J = (J++ + D_x h1 + D_y h2) / 3 = (J++ + J+x + Jx+) / 3, the viscous term and the update.
  const T third = nparts == 3 ? T(1.0 / 3.0) : T(1);
  for (int i = threadIdx.x; i < nin; i += blockDim.x) {
    const int c = i / NN, k = i - (i / NN) * NN;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int lc = (ry + 1) * BW + rx + 1;
    const int a = k / N, b = k - (k / N) * N;
    const T dxh1 = op_x_at<T, N>(sFy, tPxR, tPxL, C.dx, lc, a, b);
    const T dyh2 = op_y_at<T, N>(sFx, tPyR, tPyL, C.dy, lc, BW, a, b);
    const T J = (((use_pp ? sJ[lc * CS + k] : T(0)) + dxh1) + dyh2) * third;
    const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
    if (A.bracket_only) {
      A.omega_out[g] = double(J);
      continue;
    }
    T R = -J;
    if (A.visc != 0.0) {
      const bool fx = G.bc && B.tx0 + rx == 0, fy = G.bc && B.ty0 + ry == 0;
      const T lap = op_x_at<T, N>(sOm, tLxR, tLxL, C.lx, lc, a, b, fx) +
                    op_y_at<T, N>(sOm, tLyR, tLyL, C.ly, lc, BW, a, b, fy);
      R = fma(-T(A.visc), lap, R);  // + D Delta_h omega, since -Delta_h = lx + ly
    }
    double incr = A.c_new * double(R);
    for (int m = 0; m < A.nhist; ++m) incr = fma(A.c_hist[m], double(A.hist[m][g]), incr);
    if (A.R_out) A.R_out[g] = double(R);
    A.omega_out[g] = fma(A.dt, incr, A.omega_base[g]);
  }
  __syncthreads();
}

// Cell stride of the fixed-point staging: odd, so that the lanes of a warp, which read the same
// node of consecutive cells, fall on distinct pairs of banks.
template <int N>
__host__ __device__ constexpr int fx_cell() {
  return (N * N) | 1;
}

// How far below a tile's largest value its cells may lie in fixed point, in bits.  Errors there are
// relative to the tile's largest value, in float64 to the values around the node.  Away from a cell 2^s
// times the others they pass those of the float64 tile at s = 6 (operators) and, for the bracket, whose
// two fields' bits add up, at s = 4, 4, 4, 3, 2 for n = 1..5, and double with each bit: at 14 bits they
// are still below 1e-12 of the values around the node.  A tile with a cell further down, its eight
// neighbours too (the zero line of a field does not count), is left to float64: the tail of a narrow
// vortex.  Such a tile takes four times as long (at a limit of 8 bits the whole far field of a
// Gaussian of a tenth of the box would be such tiles, at 14 a third; where zero lines of
// proportional fields cross, up to 13 bits occur).
constexpr int kFxRange = 14;

// The smallest non-zero magnitude word of what a thread staged, less 1 (zeros wrap around to the largest).
__device__ __forceinline__ unsigned fx_low(unsigned low, double v) { return min(low, fx_mag(v) - 1u); }
// The bits between the largest and the smallest non-zero value, from their magnitude words.
__device__ __forceinline__ int fx_spread(unsigned mag, unsigned low) {
  return mag ? max(1, int(mag >> 20)) - max(1, int((low + 1u) >> 20)) : 0;
}

// Whether a cell of the tile lies more than kFxRange bits below the largest value ef, eg of the staged
// fields f, g: the bits of both added, or (alone) those of g.  f may be null: g alone, on a box without
// corners.  e: one or two words per box cell of scratch.  In every thread, after a block synchronisation.
template <int N>
__device__ __noinline__ bool fx_far(const TileBox& B, const double* f, const double* g, int ef, int eg, bool alone,
                                    int* e) {
  constexpr int CS = fx_cell<N>();
  const int BWe = B.TXe + 2, BHe = B.TYe + 2, nb = BWe * BHe;
  const unsigned mw = magic_of(BWe);
  for (int u = threadIdx.x; u < (f ? 2 : 1) * nb; u += blockDim.x) {
    const int c = u < nb ? u : u - nb;
    const int br = quot(c, mw), bc = c - br * BWe;
    const bool corner = (br == 0 || br == BHe - 1) && (bc == 0 || bc == BWe - 1);
    unsigned m = 0;
    if (f || !corner) {
      const double* v = (u < nb ? g : f) + (br * B.BW + bc) * CS;
      for (int k = 0; k < N * N; ++k) m = max(m, fx_mag(v[k]));
    }
    e[u] = m ? max(1, int(m >> 20)) : 0;
  }
  __syncthreads();
  bool far = false;
  for (int c = threadIdx.x; c < B.TYe * B.TXe; c += blockDim.x) {
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    int mg = 0, mf = 0;
    for (int y = 0; y < 3; ++y)
      for (int x = 0; x < 3; ++x) {
        const int o = (ry + y) * BWe + rx + x;
        mg = max(mg, e[o]);
        if (f) mf = max(mf, e[nb + o]);
      }
    if (mg && alone) far |= eg - mg > kFxRange;
    if (mg && mf) far |= ef - mf + eg - mg > kFxRange;
  }
  return __syncthreads_or(far);
}

// A quick look before that one: whether a cell has no node near the largest values among the middle
// nodes of itself and its eight neighbours.  (The zero lines of resolved fields, which most tiles that
// come here have, end here.)  In every thread, after a block synchronisation.
template <int N>
__device__ __forceinline__ bool fx_lonely(const TileBox& B, const double* f, const double* g, int ef, int eg) {
  constexpr int CS = fx_cell<N>();
  bool lonely = false;
  for (int c = threadIdx.x; c < B.TYe * B.TXe; c += blockDim.x) {
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int o = (ry * B.BW + rx) * CS + N / 2 * (N + 1);
    int top = 0;
#pragma unroll
    for (int y = 0; y < 3; ++y)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const int i = o + (y * B.BW + x) * CS;
        top = max(top, ((__double2hiint(g[i]) >> 20) & 0x7ff) + (f ? (__double2hiint(f[i]) >> 20) & 0x7ff : 0));
      }
    lonely |= eg + (f ? ef : 0) - top > kFxRange;
  }
  return __syncthreads_or(lonely);
}

// The factors of the fixed-point LDG operators, 1 / hx^2 and 1 / hy^2.  ok: they lie in the range the
// fixed-point path covers.  stiff, lap: device tables (FxTable<n>) that replace fx_stiff and fx_lap
// on grids with a jump penalty tau != 0, else null.
struct FxScale {
  double cx, cy;
  int ok;
  const void *stiff, *lap;
};

// One LDG operator on all lines of a tile with a table in memory: x-lines to qx, y-lines to qy, cell
// (ry, rx) of the results at (ry * orow + rx + ooff).  Periodic grids (a penalty needs one).
template <int N>
__device__ __noinline__ void fx_lines_table(const FxTable<N>* O, const TileBox& B, const fx* sU, long long* qx,
                                            long long* qy, int orow, int ooff) {
  constexpr int CS = fx_cell<N>();
  const int nc = B.TYe * B.TXe;
  const unsigned mnc = magic_of(nc);
  for (int u = threadIdx.x; u < 2 * nc * N; u += blockDim.x) {
    asm volatile("" : "+l"(O));  // keeps the table out of registers across the lines
    const bool alongx = u < nc * N;
    const int v = alongx ? u : u - nc * N;
    const int ln = quot(v, mnc), c = v - ln * nc;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int st = alongx ? 1 : N, first = alongx ? ln * N : ln;
    long long* q = (alongx ? qx : qy) + (ry * orow + rx + ooff) * CS + first;
    fx_line<N>(*O, sU + ((ry + 1) * B.BW + rx + 1) * CS + first, st, alongx ? CS : B.BW * CS,
               [&](int i, long long y) { q[i * st] = y; });
  }
}

// What the fixed-point right-hand side (dg_fixed.cuh) takes from the grid.  The derivative and the
// Laplacian are tables of n on the reference cell, so every term of J carries the same factor
// 1 / (hx hy), applied once to the finished sum; likewise 1 / sqrt(W) is 1 / sqrt(w_a w_b) times
// one factor.
template <int N>
struct FxRhs {
  fx isw[N * N];   // 1 / sqrt(w_a w_b) = 2^(ei - 60) isw
  int ei;
  int ok;          // the factors lie in the range the fixed-point path covers
  double cj, cp;   // 1 / (hx hy), 2 / sqrt(hx hy)
  FxScale l;       // the Laplacian's
};

// Shared memory of one right-hand-side tile: five arrays over the box, or the float64 fallback's on
// the tile (up to 72 KB, three blocks per SM) or on single cells, whichever is larger.
template <int N>
__host__ __device__ constexpr size_t rhs_smem_bytes(int TY, int TX) {
  const size_t a = (size_t)(TY + 2) * (TX + 2) * 5 * fx_cell<N>() * 8;
  size_t b = rhs_smem_values<double, N>(TY, TX) * 8;
  if (b > 72 * 1024) b = rhs_smem_values<double, N>(1, 1) * 8;
  return a > b ? a : b;
}

// The tile in float64: for tiles whose values the fixed-point scale cannot hold (infinities, NaN,
// products near the ends of the float64 range, cells far below the others: kFxRange).  It needs more
// shared memory per cell than the fixed-point tile, so it runs on sub-tiles that fit.
template <int N>
__device__ __noinline__ void rhs_tile_float(const Ops2D<double, N>& C, const Geom& G, const RhsArgs& A, int tile,
                                            unsigned char* smem) {
  const TileBox B = make_box(G, tile);
  const size_t avail = rhs_smem_bytes<N>(G.TY, G.TX);
  Geom S = G;
  while (rhs_smem_values<double, N>(S.TY, S.TX) * 8 > avail) {
    if (S.TX >= S.TY)
      S.TX = (S.TX + 1) / 2;
    else
      S.TY = (S.TY + 1) / 2;
  }
  for (int y = 0; y < B.TYe; y += S.TY)
    for (int x = 0; x < B.TXe; x += S.TX) {
      TileBox b;
      b.ty0 = B.ty0 + y;
      b.tx0 = B.tx0 + x;
      b.TYe = min(S.TY, B.TYe - y);
      b.TXe = min(S.TX, B.TXe - x);
      b.BW = S.TX + 2;
      b.mTXe = magic_of(b.TXe);
      rhs_box_float<double, N>(C, S, A, b, smem);
    }
}

// J++ = f_x g_y - f_y g_x alone (parts == 1), left in sA with sF = 0.  The derivatives of a resolved
// field are far below the range their rows allow (h / 2^e of it), and a product rounded to 2^-60 of that
// range squared would be the whole error here (the sum of all parts rounds more elsewhere): so each
// field's derivatives are kept, and multiplied after a shift that fills 60 bits.  Returns the
// two fields' shifts, by which the result's unit is finer.  (Smooth fields, 512^2 cells, n = 5, against
// long double: relative error 6.9e-12 without the shifts, 3.2e-15 with; the float64 tile 1.9e-13.  1000^2
// cells, n = 4: 603 us, 745 through the phases of the whole J.)
template <int N>
__device__ __noinline__ int fx_jpp(const Geom& G, const TileBox& B, fx* sF, fx* sG, fx* sA, fx* sB, fx* sC,
                                   unsigned (*s_mag)[16]) {
  constexpr int CS = fx_cell<N>();
  constexpr FxTable<N> D = fx_deriv<N>();
  const int nc = B.TYe * B.TXe, dn = B.BW * CS;
  const unsigned mnc = magic_of(nc);
  unsigned hf = 0, hg = 0;
  // f_x to sA, g_x to sB, f_y to sC; then, f no longer needed, g_y to sF
  for (int part = 0; part < 2; ++part) {
    for (int u = threadIdx.x; u < (part ? 1 : 3) * nc * N; u += blockDim.x) {
      const int which = part ? 3 : u / (nc * N);
      const int v = part ? u : u - which * nc * N;
      const int ln = quot(v, mnc), c = v - ln * nc;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const bool alongx = which < 2;
      const int st = alongx ? 1 : N, o = ((ry + 1) * B.BW + rx + 1) * CS + (alongx ? ln * N : ln);
      const int pos = alongx ? B.tx0 + rx : B.ty0 + ry, len = alongx ? G.Nx : G.Ny;
      fx* out = (which == 0 ? sA : which == 1 ? sB : which == 2 ? sC : sF) + o;
      unsigned high = 0;
      fx_line_bounded<N>(D, ((which & 1) ? sG : sF) + o, st, alongx ? CS : dn, G.bc && pos == 0,
                         G.bc && pos == len - 1, [&](int i, long long y) {
                           const fx d = fx_split(y);
                           out[i * st] = d;
                           high |= unsigned(d.h ^ (d.h >> 31));
                         });
      ((which & 1) ? hg : hf) |= high;
    }
    __syncthreads();
  }
  hf = __reduce_or_sync(0xffffffffu, hf);
  hg = __reduce_or_sync(0xffffffffu, hg);
  const int lane = threadIdx.x & 31, nw = int(blockDim.x >> 5);
  if (lane == 0) {
    s_mag[0][threadIdx.x >> 5] = hf;
    s_mag[1][threadIdx.x >> 5] = hg;
  }
  __syncthreads();
  hf = __reduce_or_sync(0xffffffffu, lane < nw ? s_mag[0][lane] : 0u);
  hg = __reduce_or_sync(0xffffffffu, lane < nw ? s_mag[1][lane] : 0u);
  // high words below 2^(30 - s): values below 2^(60 - s)
  const int kf = max(0, min(__clz(int(hf)) - 2, 30)), kg = max(0, min(__clz(int(hg)) - 2, 30));
  for (int i = threadIdx.x; i < nc * N * N; i += blockDim.x) {
    const int c = i / (N * N), k = i - c * (N * N);
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int o = ((ry + 1) * B.BW + rx + 1) * CS + k;
    auto up = [&](const fx* p, int s) { return fx_split(fx_join(p[o]) << s); };
    reinterpret_cast<long long*>(sA)[o] = fx_prod_diff(up(sA, kf), up(sF, kg), up(sC, kf), up(sB, kg));
    reinterpret_cast<long long*>(sF)[o] = 0;
  }
  __syncthreads();
  return kf + kg;
}

// One tile of the right-hand side in fixed point (smem: rhs_smem_bytes<N>(G.TY, G.TX)).
//
// What bounds it: the integer pipe (60% busy with the multiply-adds on 512^2 cells, n = 5) and the
// synchronisations between phases; the float64 pipe only does the update (8%).  Per bracket, in float64
// (the same phases) and now: 1000^2 cells, n = 4 2396 and 710 us; 1000^2, n = 5 4.8 ms and 1.21 ms;
// 100^2, n = 4 38.9 and 16.4 us; 501 x 373, n = 3 158 (in double-float) and 74 us.  A thread computes a
// whole line of a cell (its n nodes along x or y):
// it reads the n values of the line and the neighbours' once, evaluates their face traces itself
// (as many multiply-adds as evaluating each trace once and storing it, one phase and 12 n arrays
// less), and takes its coefficients from the constant bank.  Phases (a block synchronisation after
// each):
//   stage f = psi and g = omega with their halo ring, find the tile's largest and smallest magnitudes
//   (and, where they are far apart, whether a cell is too far down: kFxRange), convert to fixed point;
//   x-lines of rows [-1, TYe]:  f_x, g_x, h2 = f_x g - f g_x;
//   y-lines of columns [-1, TXe]:  f_y, g_y, J++ = f_x g_y - f_y g_x, h1 = f g_y - f_y g;
//   x-lines of the tile: D_x h1 (over f); y-lines: J++ + D_y h2;   [viscous: lx g, ly g]
//   nodes: J, the update.
// J(f, f) = 0 and J(f, g) = -J(g, f) hold bitwise: equal and opposite products cancel exactly in
// the accumulators, and every rounding is odd.
//
// Gen: Dirichlet boundaries or a part of J only.  The common case (periodic, all of J) is compiled
// without either (1000^2 cells, n = 5: 1505 us with their selects around every trace and product and
// the tables as kernel parameters, 1286 without both).
template <int N, bool Gen>
__device__ __forceinline__ void rhs_tile(const FxRhs<N>& F, const Ops2D<double, N>& C, const Geom& G,
                                         const RhsArgs& A, int tile, unsigned char* smem) {
  constexpr int NN = N * N;
  constexpr int CS = fx_cell<N>();
  __shared__ unsigned s_mag[4][16];
  static_assert(rhs_threads<N>() <= 512 && kThreads <= 512, "warps of s_mag");
  __shared__ fx s_isw[NN];
  constexpr FxTable<N> D = fx_deriv<N>();
  constexpr FxTable<N> Lp = fx_lap<N>();
  const TileBox B = make_box(G, tile);
  const int BW = B.BW;
  const int boxc = (G.TY + 2) * BW;
  fx* sF = reinterpret_cast<fx*>(smem);
  fx* sG = sF + boxc * CS;
  fx* sA = sG + boxc * CS;  // f_x, then J++ (+ D_y h2)
  fx* sB = sA + boxc * CS;  // g_x, then h1, then lx g
  fx* sC = sB + boxc * CS;  // h2, then ly g

  const bool viscous = A.visc != 0.0 && !A.bracket_only;
  const int nw = int(blockDim.x >> 5), lane = threadIdx.x & 31;
  // stage the two fields and their largest and smallest magnitudes
  {
    double* rF = reinterpret_cast<double*>(sF);
    double* rG = reinterpret_cast<double*>(sG);
    unsigned mf = 0, mg = 0, nf = ~0u, ng = ~0u;
    const int BWe = B.TXe + 2, BHe = B.TYe + 2;
    const int rowlen = BWe * NN, total = BHe * rowlen;
    const unsigned mrow = magic_of(rowlen);
#pragma unroll 4
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int br = quot(i, mrow);
      const int j = i - br * rowlen;
      const int bc = j / NN, k = j - bc * NN;
      const int gy = B.ty0 + br - 1, gx = B.tx0 + bc - 1;
      const int o = (br * BW + bc) * CS + k;
      if (Gen && G.bc && (gy < 0 || gy >= G.Ny || gx < 0 || gx >= G.Nx)) {
        rF[o] = 0.0;
        rG[o] = 0.0;
        continue;
      }
      const size_t g = ((size_t)wrap_index(gy, G.Ny) * G.Nx + wrap_index(gx, G.Nx)) * NN + k;
      const double f = A.psi[g], w = A.omega_in[g];
      rF[o] = f;
      rG[o] = w;
      mf = max(mf, fx_mag(f));
      mg = max(mg, fx_mag(w));
      nf = fx_low(nf, f);
      ng = fx_low(ng, w);
    }
    mf = __reduce_max_sync(0xffffffffu, mf);
    mg = __reduce_max_sync(0xffffffffu, mg);
    nf = __reduce_min_sync(0xffffffffu, nf);
    ng = __reduce_min_sync(0xffffffffu, ng);
    if (A.psi_scaled && threadIdx.x < NN) s_isw[threadIdx.x] = F.isw[threadIdx.x];
    if ((threadIdx.x & 31) == 0) {
      s_mag[0][threadIdx.x >> 5] = mf;
      s_mag[1][threadIdx.x >> 5] = mg;
      s_mag[2][threadIdx.x >> 5] = nf;
      s_mag[3][threadIdx.x >> 5] = ng;
    }
  }
  __syncthreads();
  const unsigned mf = __reduce_max_sync(0xffffffffu, lane < nw ? s_mag[0][lane] : 0u);
  const unsigned mg = __reduce_max_sync(0xffffffffu, lane < nw ? s_mag[1][lane] : 0u);
  const unsigned nf = __reduce_min_sync(0xffffffffu, lane < nw ? s_mag[2][lane] : ~0u);
  const unsigned ng = __reduce_min_sync(0xffffffffu, lane < nw ? s_mag[3][lane] : ~0u);
  const int ef = max(1, int(mf >> 20)), eg = max(1, int(mg >> 20));
  // units of the fixed-point fields, 2^uf and 2^ug (of an all-zero field: any), of the products and of the
  // viscous term
  const int uf = mf ? ef - 1082 + (A.psi_scaled ? F.ei : 0) : 0, ug = mg ? eg - 1082 : 0;
  int uj = uf + ug + 2 * D.e + 60;
  const int ul = ug + (F.l.lap ? static_cast<const FxTable<N>*>(F.l.lap)->e : Lp.e);
  // magnitudes below 2^63: units within 2^+-600 keep every result and factor a normal number
  bool covered = F.ok && ef < 2047 && eg < 2047 && abs(uj) <= 600 && (!viscous || (F.l.ok && abs(ul) <= 600));
  if (covered && fx_spread(mf, nf) + fx_spread(mg, ng) > kFxRange) {
    const double *rF = reinterpret_cast<const double*>(sF), *rG = reinterpret_cast<const double*>(sG);
    if (fx_lonely<N>(B, rF, rG, ef, eg)) covered = !fx_far<N>(B, rF, rG, ef, eg, viscous, reinterpret_cast<int*>(sA));
  }
  if (!covered) {
    __syncthreads();  // the staging is reused
    rhs_tile_float<N>(C, G, A, tile, smem);
    return;
  }
  for (int i = threadIdx.x; i < boxc * CS; i += blockDim.x) {
    const fx f = sF[i], w = sG[i];  // raw bits: {low, high} words
    long long x = fx_from_bits(unsigned(f.l), unsigned(f.h), ef);
    if (A.psi_scaled) {
      const int k = i % CS;
      FxAcc s;
      fx_mac(s, s_isw[k < NN ? k : 0], fx_split(x));
      x = fx_round(s);
    }
    sF[i] = fx_split(x);
    sG[i] = fx_split(fx_from_bits(unsigned(w.l), unsigned(w.h), eg));
  }
  __syncthreads();

  // Which parts enter (Eq. J): J = s (c0 J++ + J+x + Jx+) with J+x = D_x(f g_y) - D_y(f g_x),
  // Jx+ = D_y(f_x g) - D_x(f_y g).
  const int parts = A.parts ? A.parts : 7;
  const int mpp = !Gen || (parts & 1) ? -1 : 0, mpx = !Gen || (parts & 2) ? -1 : 0, mxp = !Gen || (parts & 4) ? -1 : 0;
  const bool bc = Gen && G.bc;

  const int nc = B.TYe * B.TXe;
  const unsigned mnc = magic_of(nc);
  bool alone = false;
  if constexpr (Gen) {
    alone = parts == 1;
    if (alone) uj -= fx_jpp<N>(G, B, sF, sG, sA, sB, sC, s_mag);
  }
  if (!alone) {
    // x-lines of rows [-1, TYe]
    {
      const int nc = (B.TYe + 2) * B.TXe;
      const unsigned mnc = magic_of(nc);
      for (int u = threadIdx.x; u < nc * N; u += blockDim.x) {
        const int a = quot(u, mnc), c = u - a * nc;
        const int br = quot(c, B.mTXe), rx = c - br * B.TXe;
        const int o = (br * BW + rx + 1) * CS + a * N;
        fx fd[N];
        auto keep = [&](int i, long long y) { fd[i] = fx_split(y); };
        auto store = [&](int i, long long y) {
          const fx gd = fx_split(y);
          sA[o + i] = fd[i];
          sB[o + i] = gd;
          sC[o + i] = fx_split(fx_prod_diff(fd[i], fx_and(sG[o + i], mxp), fx_and(sF[o + i], mpx), gd));
        };
        if constexpr (Gen) {
          const bool first = bc && B.tx0 + rx == 0, last = bc && B.tx0 + rx == G.Nx - 1;
          fx_line_bounded<N>(D, sF + o, 1, CS, first, last, keep);
          fx_line_bounded<N>(D, sG + o, 1, CS, first, last, store);
        } else {
          fx_line<N>(D, sF + o, 1, CS, keep);
          fx_line<N>(D, sG + o, 1, CS, store);
        }
      }
    }
    __syncthreads();
    // y-lines of columns [-1, TXe]
    {
      const int w = B.TXe + 2, nc = B.TYe * w;
      const unsigned mnc = magic_of(nc), mw = magic_of(w);
      for (int u = threadIdx.x; u < nc * N; u += blockDim.x) {
        const int b = quot(u, mnc), c = u - b * nc;
        const int ry = quot(c, mw), bc_ = c - ry * w;
        const int o = ((ry + 1) * BW + bc_) * CS + b, dn = BW * CS;
        const bool inner = bc_ > 0 && bc_ <= B.TXe;
        fx fd[N];
        auto keep = [&](int i, long long y) { fd[i] = fx_split(y); };
        auto store = [&](int i, long long y) {
          const fx gd = fx_split(y);
          const int oi = o + i * N;
          if (inner)
            reinterpret_cast<long long*>(sA)[oi] = fx_prod_diff(fx_and(sA[oi], mpp), gd, fd[i], fx_and(sB[oi], mpp));
          sB[oi] = fx_split(fx_prod_diff(fx_and(sF[oi], mpx), gd, fd[i], fx_and(sG[oi], mxp)));
        };
        if constexpr (Gen) {
          const bool first = bc && B.ty0 + ry == 0, last = bc && B.ty0 + ry == G.Ny - 1;
          fx_line_bounded<N>(D, sF + o, N, dn, first, last, keep);
          fx_line_bounded<N>(D, sG + o, N, dn, first, last, store);
        } else {
          fx_line<N>(D, sF + o, N, dn, keep);
          fx_line<N>(D, sG + o, N, dn, store);
        }
      }
    }
    __syncthreads();
    // D_x h1 over f, J++ + D_y h2
    for (int u = threadIdx.x; u < 2 * nc * N; u += blockDim.x) {
      const bool alongx = u < nc * N;
      const int v = alongx ? u : u - nc * N;
      const int ln = quot(v, mnc), c = v - ln * nc;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const int cell = ((ry + 1) * BW + rx + 1) * CS;
      if (alongx) {
        const int o = cell + ln * N;
        auto put = [&](int i, long long y) { reinterpret_cast<long long*>(sF)[o + i] = y; };
        if constexpr (Gen)
          fx_line_bounded<N>(D, sB + o, 1, CS, bc && B.tx0 + rx == 0, bc && B.tx0 + rx == G.Nx - 1, put);
        else
          fx_line<N>(D, sB + o, 1, CS, put);
      } else {
        const int o = cell + ln;
        auto add = [&](int i, long long y) { reinterpret_cast<long long*>(sA)[o + i * N] += y; };
        if constexpr (Gen)
          fx_line_bounded<N>(D, sC + o, N, BW * CS, bc && B.ty0 + ry == 0, bc && B.ty0 + ry == G.Ny - 1, add);
        else
          fx_line<N>(D, sC + o, N, BW * CS, add);
      }
    }
    __syncthreads();
  }
  if (viscous && F.l.lap) {  // lx g over h1, ly g over h2
    fx_lines_table<N>(static_cast<const FxTable<N>*>(F.l.lap), B, sG, reinterpret_cast<long long*>(sB),
                      reinterpret_cast<long long*>(sC), BW, BW + 1);
    __syncthreads();
  } else if (viscous) {
    for (int u = threadIdx.x; u < 2 * nc * N; u += blockDim.x) {
      const bool alongx = u < nc * N;
      const int v = alongx ? u : u - nc * N;
      const int ln = quot(v, mnc), c = v - ln * nc;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const int cell = ((ry + 1) * BW + rx + 1) * CS;
      if (alongx) {
        const int o = cell + ln * N;
        auto put = [&](int i, long long y) { reinterpret_cast<long long*>(sB)[o + i] = y; };
        if constexpr (Gen)
          fx_ldg_bounded<N>(Lp, sG + o, 1, CS, bc ? B.tx0 + rx : 2, put);
        else
          fx_line<N>(Lp, sG + o, 1, CS, put);
      } else {
        const int o = cell + ln;
        auto put = [&](int i, long long y) { reinterpret_cast<long long*>(sC)[o + i * N] = y; };
        if constexpr (Gen)
          fx_ldg_bounded<N>(Lp, sG + o, N, BW * CS, bc ? B.ty0 + ry : 2, put);
        else
          fx_line<N>(Lp, sG + o, N, BW * CS, put);
      }
    }
    __syncthreads();
  }
  // nodes: J and the update
  const double cJ = (parts == 7 ? 1.0 / 3.0 : 1.0) * F.cj * (A.psi_scaled ? F.cp : 1.0) * fx_pow2(uj);
  const double cLx = A.visc * F.l.cx * fx_pow2(ul), cLy = A.visc * F.l.cy * fx_pow2(ul);
  const bool square = F.l.cx == F.l.cy;
  const int nin = nc * NN;
#pragma unroll 4
  for (int i = threadIdx.x; i < nin; i += blockDim.x) {
    const int c = i / NN, k = i - (i / NN) * NN;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int o = ((ry + 1) * BW + rx + 1) * CS + k;
    const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
    const double J =
        fx_to_double(reinterpret_cast<const long long*>(sA)[o] + reinterpret_cast<const long long*>(sF)[o]) * cJ;
    if (A.bracket_only) {
      A.omega_out[g] = J;
      continue;
    }
    // the node's other fields, loaded before they are needed
    const double base = A.omega_base[g];
    const double h0 = A.nhist > 0 ? A.hist[0][g] : 0.0, h1 = A.nhist > 1 ? A.hist[1][g] : 0.0,
                 h2 = A.nhist > 2 ? A.hist[2][g] : 0.0;
    double R = -J;
    if (viscous) {  // + D Delta_h omega, since -Delta_h = lx + ly
      const long long lx = reinterpret_cast<const long long*>(sB)[o], ly = reinterpret_cast<const long long*>(sC)[o];
      if (square)
        R = fma(-cLx, fx_to_double(lx + ly), R);
      else
        R = fma(-cLx, fx_to_double(lx), fma(-cLy, fx_to_double(ly), R));
    }
    double incr = A.c_new * R;
    if (A.nhist > 0) incr = fma(A.c_hist[0], h0, incr);
    if (A.nhist > 1) incr = fma(A.c_hist[1], h1, incr);
    if (A.nhist > 2) incr = fma(A.c_hist[2], h2, incr);
    if (A.R_out) A.R_out[g] = R;
    A.omega_out[g] = fma(A.dt, incr, base);
  }
  __syncthreads();
}

template <int N, bool Gen>
__global__ void __launch_bounds__(rhs_threads<N>(), rhs_blocks<N>()) rhs_kernel(const __grid_constant__ FxRhs<N> F,
                                                               const Ops2D<double, N>* __restrict__ C, const Geom G,
                                                               const __grid_constant__ RhsArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  rhs_tile<N, Gen>(F, *C, G, A, blockIdx.x, smem_raw);
}

// =========================================================================================
// One tile of an LDG operator on a float64 field in fixed point (dg_fixed.cuh).
// =========================================================================================

// Shared memory of the pass: the staged box and the two directions' results on the tile (or, before
// them, fx_far's word per box cell).
template <int N>
__host__ __device__ constexpr size_t fx_apply_bytes(int TY, int TX) {
  const size_t box = (size_t)(TY + 2) * (TX + 2), q = 2 * (size_t)TY * TX * fx_cell<N>() * 8;
  return box * fx_cell<N>() * 8 + (q > 4 * box ? q : (4 * box + 7) / 8 * 8);
}

// The lines of the tile in float64, for tiles the fixed-point scale cannot hold or not well enough.
template <int N>
__device__ __noinline__ void apply_lines_float(const Op1D<double, N>& ox, const Op1D<double, N>& oy, const Geom& G,
                                               const TileBox& B, const double* sU, double* qx, double* qy) {
  constexpr int CS = fx_cell<N>();
  const int nc = B.TYe * B.TXe;
  for (int u = threadIdx.x; u < 2 * nc * N; u += blockDim.x) {
    const bool alongx = u < nc * N;
    const int v = alongx ? u : u - nc * N;
    const int ln = v / nc, c = v - ln * nc;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const Op1D<double, N>& o = alongx ? ox : oy;
    const int st = alongx ? 1 : N, dc = alongx ? CS : B.BW * CS, first = alongx ? ln * N : ln;
    const double* w = sU + ((ry + 1) * B.BW + rx + 1) * CS + first;
    double* q = (alongx ? qx : qy) + (ry * G.TX + rx) * CS + first;
    const int pos = G.bc ? (alongx ? B.tx0 + rx : B.ty0 + ry) : 2;
    double tr = 0.0, tl = 0.0;
    for (int j = 0; j < N; ++j) {
      tr = fma(o.r[j], w[dc + j * st], tr);
      tl = fma(pos == 1 ? o.sf[j] : o.s[j], w[j * st - dc], tl);
    }
    for (int i = 0; i < N; ++i) {
      double acc = (pos == 0 ? o.af[i] : o.a[i]) * tr;
      acc = fma(o.d[i], tl, acc);
      for (int j = 0; j < N; ++j) acc = fma(pos == 0 ? o.Mf[i][j] : o.M[i][j], w[j * st], acc);
      q[i * st] = acc;
    }
  }
}

// Stages u = load(g, k, interior) on the tile and its plus-shaped halo, applies the operator (Lap:
// -Delta_h, else W^-1/2 A W^-1/2; ox, oy its float64 form) and hands (g, k, q) of the tile's nodes
// to out.  Local: tiles with cells far below the others (kFxRange) go to float64.  The solves do
// without: there errors count against the norm of the whole field, and 2^-60 of a tile's largest
// value is below 2^-53 of its norm.  smem: fx_apply_bytes<N>(G.TY, G.TX).
template <int N, bool Lap, bool Local, class LoadF, class OutF>
__device__ __forceinline__ void fx_tile_apply(const Op1D<double, N>& ox, const Op1D<double, N>& oy, const FxScale& S,
                                              const Geom& G, int tile, void* smem, LoadF&& load, OutF&& out) {
  constexpr int NN = N * N;
  constexpr int CS = fx_cell<N>();
  constexpr FxTable<N> O = Lap ? fx_lap<N>() : fx_stiff<N>();
  __shared__ unsigned s_mag[32];
  const TileBox B = make_box(G, tile);
  const int BW = B.BW, boxc = (G.TY + 2) * BW;
  fx* sU = static_cast<fx*>(smem);
  long long* qx = reinterpret_cast<long long*>(sU + boxc * CS);
  long long* qy = qx + G.TY * G.TX * CS;
  const int lane = threadIdx.x & 31, nw = int(blockDim.x >> 5);
  const FxTable<N>* tab = static_cast<const FxTable<N>*>(Lap ? S.lap : S.stiff);
  unsigned m = 0, low = ~0u;
  {
    double* rU = reinterpret_cast<double*>(sU);
    const int BWe = B.TXe + 2, BHe = B.TYe + 2;
    const int rowlen = BWe * NN, total = BHe * rowlen;
    const unsigned mrow = magic_of(rowlen);
#pragma unroll 4
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
      const int br = quot(i, mrow);
      const int j = i - br * rowlen;
      const int bc = j / NN, k = j - bc * NN;
      const bool rowhalo = (br == 0) || (br == BHe - 1), colhalo = (bc == 0) || (bc == BWe - 1);
      const int gy = B.ty0 + br - 1, gx = B.tx0 + bc - 1;
      const int o = (br * BW + bc) * CS + k;
      if (rowhalo && colhalo) {  // the 5-cell operators never read the corners
        if constexpr (Local) rU[o] = 0.0;
        continue;
      }
      double v = 0.0;  // Dirichlet: zero outside
      if (!(G.bc && (gy < 0 || gy >= G.Ny || gx < 0 || gx >= G.Nx)))
        v = load(((size_t)wrap_index(gy, G.Ny) * G.Nx + wrap_index(gx, G.Nx)) * NN + k, k, !(rowhalo || colhalo));
      rU[o] = v;
      m = max(m, fx_mag(v));
      if constexpr (Local) low = fx_low(low, v);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if constexpr (Local) low = __reduce_min_sync(0xffffffffu, low);
    if ((threadIdx.x & 31) == 0) {
      s_mag[threadIdx.x >> 5] = m;
      if constexpr (Local) s_mag[16 + (threadIdx.x >> 5)] = low;
    }
  }
  __syncthreads();
  m = __reduce_max_sync(0xffffffffu, lane < nw ? s_mag[lane] : 0u);
  const int em = max(1, int(m >> 20)), uq = m ? em - 1082 + (tab ? tab->e : O.e) : 0;
  bool covered = S.ok && em < 2047 && abs(uq) <= 600;
  if constexpr (Local) {
    low = __reduce_min_sync(0xffffffffu, lane < nw ? s_mag[16 + lane] : ~0u);
    const double* rU = reinterpret_cast<const double*>(sU);
    if (covered && fx_spread(m, low) > kFxRange && fx_lonely<N>(B, nullptr, rU, 0, em))
      covered = !fx_far<N>(B, nullptr, rU, 0, em, true, reinterpret_cast<int*>(qx));
  }
  const int nc = B.TYe * B.TXe;
  if (covered) {
    for (int i = threadIdx.x; i < boxc * CS; i += blockDim.x) {
      const fx w = sU[i];  // raw bits: {low, high} words
      sU[i] = fx_split(fx_from_bits(unsigned(w.l), unsigned(w.h), em));
    }
    __syncthreads();
    const unsigned mnc = magic_of(nc);
    if (tab) fx_lines_table<N>(tab, B, sU, qx, qy, G.TX, 0);
    for (int u = threadIdx.x; u < (tab ? 0 : 2 * nc * N); u += blockDim.x) {
      const bool alongx = u < nc * N;
      const int v = alongx ? u : u - nc * N;
      const int ln = quot(v, mnc), c = v - ln * nc;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const fx* w = sU + ((ry + 1) * BW + rx + 1) * CS;
      const int t = (ry * G.TX + rx) * CS;
      if (alongx) {
        auto put = [&](int i, long long y) { qx[t + ln * N + i] = y; };
        if (G.bc && B.tx0 + rx < 2)
          fx_ldg_bounded<N>(O, w + ln * N, 1, CS, B.tx0 + rx, put);
        else
          fx_line<N>(O, w + ln * N, 1, CS, put);
      } else {
        auto put = [&](int i, long long y) { qy[t + ln + i * N] = y; };
        if (G.bc && B.ty0 + ry < 2)
          fx_ldg_bounded<N>(O, w + ln, N, BW * CS, B.ty0 + ry, put);
        else
          fx_line<N>(O, w + ln, N, BW * CS, put);
      }
    }
  } else {
    apply_lines_float<N>(ox, oy, G, B, reinterpret_cast<const double*>(sU), reinterpret_cast<double*>(qx),
                         reinterpret_cast<double*>(qy));
  }
  __syncthreads();
  const double cx = S.cx * fx_pow2(uq), cy = S.cy * fx_pow2(uq);
  const bool square = S.cx == S.cy;
#pragma unroll 2
  for (int i = threadIdx.x; i < nc * NN; i += blockDim.x) {
    const int c = i / NN, k = i - c * NN;
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const int t = (ry * G.TX + rx) * CS + k;
    const long long a = qx[t], b = qy[t];
    double q;
    if (!covered)
      q = __longlong_as_double(a) + __longlong_as_double(b);
    else if (square)
      q = fx_to_double(a + b) * cx;
    else
      q = fma(fx_to_double(a), cx, fx_to_double(b) * cy);
    out(((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k, k, q);
  }
  __syncthreads();
}

// =========================================================================================
// Operator application: mode 0  y = A x = W^1/2 (W^-1/2 A W^-1/2) W^1/2 x,
//                       mode 1  y = Delta_h x = -(lx + ly) x.
// =========================================================================================
template <int N, bool Lap>
__global__ void __launch_bounds__(kThreads, 4) apply_kernel(const Ops2D<double, N>* __restrict__ C,
                                                         const FxScale S, const Geom G, const double* __restrict__ x,
                                                         double* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_sw[N * N];
  if constexpr (!Lap) {
    if (threadIdx.x < N * N) s_sw[threadIdx.x] = C->sw[threadIdx.x];
    __syncthreads();
  }
  fx_tile_apply<N, Lap, true>(
      Lap ? C->lx : C->kx, Lap ? C->ly : C->ky, S, G, blockIdx.x, smem_raw,
      [&](size_t g, int k, bool) { return Lap ? x[g] : x[g] * s_sw[k]; },
      [&](size_t g, int k, double q) { y[g] = Lap ? -q : q * s_sw[k]; });
}

// =========================================================================================
// Persistent conjugate-gradient solve of  Ahat y = b,  Ahat = W^-1/2 A W^-1/2  (plain CG on
// the symmetrically scaled system = CG on A psi = W omega preconditioned by W^-1, Sec. 6).
// Phases are separated by a capped grid barrier; dot products are block partials summed by
// every block in a fixed order (bit-identical scalars in all blocks, so every block takes the
// same branch).  Partial buffers alternate between two halves so that a block writing the
// next partial never races a slower block still reading the previous ones.
// =========================================================================================
constexpr int kRefineHistory = 48;  // sweeps recorded in SolveStatus

struct SolveStatus {
  long long total_iters;
  int last_iters;
  int max_iters;
  int flags;        // OR of all solves' flags
  int last_flags;
  int nsolves;
  int last_sweeps;  // refinement sweeps of the last mixed solve
  double last_rho;  // r.r of the last solve (scaled space)
  double last_rhob; // b.b
  // convergence history of the last mixed solve: r.r / b.b of the float64 residual before
  // sweep j (j = 0: of the initial guess) and the inner iterations of sweep j
  int hist_len;
  double hist_rr[kRefineHistory];
  int hist_it[kRefineHistory];
};

template <typename T>
struct CgVectors {
  T* y;      // solution (scaled space)
  T* r;      // residual
  T* p0;     // search directions (double-buffered: a phase reads one, writes the other)
  T* p1;
  T* q;      // Ahat p
};

template <typename T>
struct RhsSource {
  const double* omega;
  const T* rhs;
  T wbar;
};

template <typename T, int N>
__device__ __forceinline__ T rhs_at(const Ops2D<T, N>& C, const RhsSource<T>& B, size_t g, int k) {
  return B.rhs ? B.rhs[g] : C.sw[k] * (T(B.omega[g]) - B.wbar);
}

// Restarts from the true residual allowed after the recursive one has met the tolerance.
constexpr int kMaxRestarts = 20;

// ---- the two-level preconditioner --------------------------------------------------------
// In the scaled space (r~ = W^-1/2 r) the preconditioner M^-1 = B + P A_c^+ P^T of the
// unscaled system reads  z~ = Bt r~ + sqrt(W) (A_c^+ rc),  rc = sum over a cell's nodes of
// sqrt(W) r~  (= P^T r),  Bt = diag(sqrt W) A_cc^-1 diag(sqrt W)  (one n^2 x n^2 matrix for
// every cell), A_c = P^T A P the Galerkin coarse operator on the cells, diagonalised by the
// 2D DFT with eigenvalues ax[kx] + ay[ky] (constant mode dropped).
//
// The spectral preconditioner is M^-1 = Ahat^+ itself.  On the uniform periodic grid
// Ahat = I (x) Kx + Ky (x) I is block-circulant along both cell indices, so the DFT over cells
// turns each 1D operator into one n x n Hermitian matrix per wave number,
// Kx(kx) = M + e^{i th} a r^T + e^{-i th} d s^T (th = 2 pi kx / Nx), diagonalised on the host:
// Kx(kx) = Vx diag(lx) Vx^*, Ky(ky) = Vy diag(ly) Vy^*.  z~ = Ahat^+ r~ is then: a real DFT
// along x of the n^2 node fields and Vx^* per (cy, kx, a); a DFT along y, Vy^* per (ky, kx, j),
// division by ly_i + lx_j (the constant mode, the one pair whose sum is exactly 0, dropped),
// Vy and the inverse DFT along y; Vx and the inverse real DFT along x.  Three grid-wide phases
// over the spectrum S[kx][cy][a][j] (kx <= Nx/2).
enum : int { kPrecondJacobi = 0, kPrecondTwoLevel = 1, kPrecondSpectral = 2 };

template <typename T>
struct PrecondArgs {
  int kind;             // kPrecondTwoLevel or kPrecondSpectral
  const T* Bt;          // N^2 x N^2, row-major
  const Cplx<T>* twx;   // exp(-2 pi i m / Nx), m < Nx
  const Cplx<T>* twy;   // exp(-2 pi i m / Ny), m < Ny
  const T* ax;          // coarse eigenvalues: lambda(kx, ky) = ax[kx] + ay[ky]
  const T* ay;
  int log2x, log2y;     // log2 of Nx, Ny when powers of two, else -1 (direct DFT)
  T* z;                 // cell-block part of z~ (two-level) or all of z~ (spectral), one per dof
  T* rc;                // restricted residual (one per cell)
  T* uc;                // coarse correction (one per cell)
  Cplx<T>* C;           // coarse spectrum (Ny x (Nx/2 + 1))
  const Cplx<T>* Vx;    // spectral: Vx[kx][b][j], kx <= Nx/2 (column j = eigenvector j)
  const T* lx;          // lx[kx][j]
  const Cplx<T>* Vy;    // Vy[ky][a][i], ky < Ny
  const T* ly;          // ly[ky][i]
  Cplx<T>* S;           // spectrum, (Nx/2 + 1) x Ny x N x N
  // fixed-point spectral path (float64, power-of-two cell counts; null elsewhere): the same tables
  // in units of 2^-60, and the units' scales {top, exponent}: |value| < 2^top, value = integer 2^exponent
  const Cfx *fVx, *fVy, *ftwx, *ftwy;
  int2* EU;
  double lymin[2];      // the smallest ly, the smallest non-zero ly
};

// Shared memory and synchronisation of one persistent solve.
template <typename T>
struct SolveCtx {
  T *sU, *tXR, *tXL, *tYR, *tYL;  // tile staging
  Cplx<T>* line0;                 // DFT line buffers (alias the tile staging)
  Cplx<T>* line1;
  const T* Bs;                    // Bt staged in shared memory (null without preconditioner)
  T* red;
  BarrierState* bs;
  SyncState* sync;
  T* part;                        // 8 * vsize: two alternating halves of up to 3 sums and a magnitude
  int phase;
  unsigned int tbase;             // first ticket of the next dynamically scheduled phase
  int vrank, vsize;               // this block's rank and the block count of the (virtual) grid
  int cluster;                    // the whole grid is one thread-block cluster
  // float32 solves: if kdf is set (an OpsK<df, N> in shared memory), the operator Ahat is
  // applied in double-float arithmetic on the float32 vectors, staged in the 8-byte tile
  // buffers wU, wXR, wXL, wYR, wYL (the float64 context's staging region)
  const void* kdf;
  df *wU, *wXR, *wXL, *wYR, *wYL;
  FxScale ks;                     // factors of the fixed-point operator (float64 solves)
};

// The barrier between the phases of a solve: the hardware cluster barrier when the solve's
// blocks form one cluster (small grids), else the capped grid barrier.
template <typename T>
__device__ __forceinline__ bool solve_barrier(SolveCtx<T>& X) {
  if (X.cluster) {
    cluster_barrier();
    return true;
  }
  return grid_barrier(X.sync, X.bs, X.vsize);
}

// Dynamic distribution of a phase's work units over the blocks of a solve: each block takes
// the next unit from the ticket counter of the solve's SyncState until the units run out.
// Every block draws exactly one ticket past the last unit, so a phase consumes units + vsize
// tickets and every block knows where the next phase's tickets start (X.tbase, read from
// the counter by every block at the start of the solve, before its first barrier).  Units
// write disjoint outputs, so the results do not depend on which block takes which unit.
template <typename T>
__device__ __forceinline__ int next_unit(SolveCtx<T>& X, int units) {
  int* s = reinterpret_cast<int*>(X.red);
  __syncthreads();  // every thread has read the previous unit number
  if (threadIdx.x == 0) s[0] = int(atomicAdd(&X.sync->ticket, 1u) - X.tbase);
  __syncthreads();
  return s[0];
}

template <typename T>
__device__ __forceinline__ void end_units(SolveCtx<T>& X, int units) {
  X.tbase += unsigned(units) + unsigned(X.vsize);
}

template <typename T>
__device__ __forceinline__ unsigned int read_ticket(const SyncState* s) {
  return *reinterpret_cast<const volatile unsigned int*>(&s->ticket);
}

// Block partials of K sums -> grid barrier -> the sums in every block, in a fixed order that depends
// only on the block count.  red: 112 values.
// mag: also the largest magnitude word (fx_mag) of all blocks.
template <int K, typename T>
__device__ __forceinline__ bool reduce_sums(SolveCtx<T>& X, T (&v)[K], T (&out)[K], unsigned* mag = nullptr) {
  T* ph = X.part + (X.phase & 1) * 4 * X.vsize;
  unsigned* pm = reinterpret_cast<unsigned*>(ph + 3 * X.vsize);
  ++X.phase;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = int(blockDim.x >> 5);
#pragma unroll
  for (int j = 0; j < K; ++j) v[j] = warp_sum_down(v[j]);
  __syncthreads();  // the previous use of red has been read
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < K; ++j) X.red[32 * j + w] = v[j];
  }
  unsigned m = 0;
  if (mag) {
    m = __reduce_max_sync(0xffffffffu, *mag);
    if (lane == 0) reinterpret_cast<unsigned*>(X.red + 96)[w] = m;
  }
  __syncthreads();
  if (w == 0) {
    if (mag) {
      m = __reduce_max_sync(0xffffffffu, lane < nw ? reinterpret_cast<unsigned*>(X.red + 96)[lane] : 0u);
      if (lane == 0) __stcg(pm + X.vrank, m);
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const T t = warp_sum_down(lane < nw ? X.red[32 * j + lane] : T(0));
      if (lane == 0) __stcg(ph + K * X.vrank + j, t);
    }
  }
  if (!solve_barrier(X)) return false;
  if (mag) {
    m = 0;
    for (int i = lane; i < X.vsize; i += 32) m = max(m, __ldcg(pm + i));
    *mag = __reduce_max_sync(0xffffffffu, m);
  }
  if (X.vsize <= 128) {
    // few blocks: every warp adds all partials itself, without another block synchronisation
    T t[K] = {};
    for (int i = lane; i < X.vsize; i += 32)
#pragma unroll
      for (int j = 0; j < K; ++j) t[j] += __ldcg(ph + K * i + j);
#pragma unroll
    for (int j = 0; j < K; ++j) out[j] = __shfl_sync(0xffffffffu, warp_sum_down(t[j]), 0);
    return true;
  }
  T t[K] = {};
  for (int i = threadIdx.x; i < X.vsize; i += blockDim.x)
#pragma unroll
    for (int j = 0; j < K; ++j) t[j] += __ldcg(ph + K * i + j);
#pragma unroll
  for (int j = 0; j < K; ++j) t[j] = warp_sum_down(t[j]);
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < K; ++j) X.red[32 * j + w] = t[j];
  }
  __syncthreads();
  // every warp adds the warps' sums itself
#pragma unroll
  for (int j = 0; j < K; ++j)
    out[j] = __shfl_sync(0xffffffffu, warp_sum_down(lane < nw ? X.red[32 * j + lane] : T(0)), 0);
  return true;
}

template <typename T>
__device__ __forceinline__ bool reduce_all(SolveCtx<T>& X, T v0, T& out0) {
  T v[1] = {v0}, o[1];
  if (!reduce_sums<1>(X, v, o)) return false;
  out0 = o[0];
  return true;
}

template <typename T>
__device__ __forceinline__ bool reduce_all2(SolveCtx<T>& X, T v0, T v1, T& out0, T& out1) {
  T v[2] = {v0, v1}, o[2];
  if (!reduce_sums<2>(X, v, o)) return false;
  out0 = o[0];
  out1 = o[1];
  return true;
}

template <typename T>
__device__ __forceinline__ bool reduce_all3(SolveCtx<T>& X, T v0, T v1, T v2, T& out0, T& out1, T& out2) {
  T v[3] = {v0, v1, v2}, o[3];
  if (!reduce_sums<3>(X, v, o)) return false;
  out0 = o[0];
  out1 = o[1];
  out2 = o[2];
  return true;
}

// One CG tile pass in float32 or double-float: stage u = load(...) (plus-shaped halo), apply Ahat,
// hand (g, k, u, q) to out(...).
template <typename T, int N, class Tab, class LoadF, class OutF>
__device__ __forceinline__ void cg_tile_apply(const Tab& C, const Geom& G, int tile, SolveCtx<T>& X, LoadF&& load,
                                              OutF&& out) {
  constexpr int NN = N * N;
  const TileBox B = make_box(G, tile);
  stage_box<T, N>(G, B, X.sU, false, load);
  __syncthreads();
  line_traces<T, N>(B, X.sU, X.sU, C.kx, C.ky, X.tXR, X.tXL, X.tYR, X.tYL, false);
  __syncthreads();
  if (G.bc) {
    dirichlet_first_traces<T, N>(B, X.sU, X.sU, C.kx, C.ky, X.tXL, X.tYL);
    __syncthreads();
  }
  const int nin = B.TYe * B.TXe * NN;
  if constexpr (sizeof(T) == 4 && kThreads % NN == 0) {
    // float32: every node a thread visits is node k = threadIdx.x mod n^2 of its cell, so the
    // operator rows of that node are held in registers across the thread's cells (same
    // arithmetic and order as op_x_at / op_y_at)
    const int k = threadIdx.x % NN, a = k / N, b = k % N;
    T mx[N], my[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      mx[j] = C.kx.M[b][j];
      my[j] = C.ky.M[a][j];
    }
    const T xa = C.kx.a[b], xd = C.kx.d[b], ya = C.ky.a[a], yd = C.ky.d[a];
    for (int i = threadIdx.x; i < nin; i += kThreads) {
      const int c = i / NN;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const int lc = (ry + 1) * B.BW + rx + 1;
      const T* ux = X.sU + lc * (NN + 1) + a * N;
      const T* uy = X.sU + lc * (NN + 1) + b;
      T qx = xa * X.tXR[(lc + 1) * N + a];
      qx = fma(xd, X.tXL[(lc - 1) * N + a], qx);
      T qy = ya * X.tYR[(lc + B.BW) * N + b];
      qy = fma(yd, X.tYL[(lc - B.BW) * N + b], qy);
      if (G.bc && ((B.tx0 == 0 && rx == 0) || (B.ty0 == 0 && ry == 0))) {  // a Dirichlet boundary cell
        const bool fx = B.tx0 + rx == 0, fy = B.ty0 + ry == 0;
        const T* Mx = fx ? C.kx.Mf[b] : C.kx.M[b];
        const T* My = fy ? C.ky.Mf[a] : C.ky.M[a];
        qx = (fx ? C.kx.af[b] : xa) * X.tXR[(lc + 1) * N + a];
        qx = fma(xd, X.tXL[(lc - 1) * N + a], qx);
        qy = (fy ? C.ky.af[a] : ya) * X.tYR[(lc + B.BW) * N + b];
        qy = fma(yd, X.tYL[(lc - B.BW) * N + b], qy);
#pragma unroll
        for (int j = 0; j < N; ++j) qx = fma(Mx[j], ux[j], qx);
#pragma unroll
        for (int j = 0; j < N; ++j) qy = fma(My[j], uy[j * N], qy);
      } else {
#pragma unroll
        for (int j = 0; j < N; ++j) qx = fma(mx[j], ux[j], qx);
#pragma unroll
        for (int j = 0; j < N; ++j) qy = fma(my[j], uy[j * N], qy);
      }
      const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
      out(g, k, X.sU[lc * (NN + 1) + k], qx + qy);
    }
  } else {
    if (!G.bc) {
      for (int i = threadIdx.x; i < nin; i += blockDim.x) {
        const int c = i / NN, k = i - (i / NN) * NN;
        const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
        const int lc = (ry + 1) * B.BW + rx + 1;
        const int a = k / N, b = k - (k / N) * N;
        const T q = op_x_at<T, N>(X.sU, X.tXR, X.tXL, C.kx, lc, a, b) +
                    op_y_at<T, N>(X.sU, X.tYR, X.tYL, C.ky, lc, B.BW, a, b);
        const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
        out(g, k, X.sU[lc * (NN + 1) + k], q);
      }
    } else {  // Dirichlet: the first cell of a line takes its own blocks (Op1D::Mf, af)
      for (int i = threadIdx.x; i < nin; i += blockDim.x) {
        const int c = i / NN, k = i - (i / NN) * NN;
        const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
        const int lc = (ry + 1) * B.BW + rx + 1;
        const int a = k / N, b = k - (k / N) * N;
        const bool fx = B.tx0 + rx == 0, fy = B.ty0 + ry == 0;
        const T q = op_x_at<T, N>(X.sU, X.tXR, X.tXL, C.kx, lc, a, b, fx) +
                    op_y_at<T, N>(X.sU, X.tYR, X.tYL, C.ky, lc, B.BW, a, b, fy);
        const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
        out(g, k, X.sU[lc * (NN + 1) + k], q);
      }
    }
  }
  __syncthreads();
}

// One tile pass of the solve's operator, (g, k, u, q) handed to out: a float64 solve in fixed point
// (fx_tile_apply; u is loaded again, own(g)), a float32 one in float32 or -- with the compensated apply enabled -- in
// double-float arithmetic on the same float32 values, the result rounded to float32.  A float32 evaluation of Ahat u has an absolute error of about
// eps32 |Ahat| |u|, which on the smoothest modes of a fine grid (eigenvalue ~1 against
// |Ahat| ~ 1e7 at 1024^2 cells, n = 5) is as large as Ahat u itself; the double-float apply
// brings it down to ~eps32^2 |Ahat| |u|.
template <typename T, int N, class LoadF, class OwnF, class OutF>
__device__ __forceinline__ void solve_apply(const Ops2D<T, N>& C, const Geom& G, int tile, SolveCtx<T>& X,
                                            LoadF&& load, OwnF&& own, OutF&& out) {
  if constexpr (std::is_same<T, double>::value) {
    fx_tile_apply<N, false, false>(C.kx, C.ky, X.ks, G, tile, X.sU, load,
                                   [&](size_t g, int k, T q) { out(g, k, own(g), q); });
  } else {
    if (X.kdf) {
      SolveCtx<df> W;
      W.sU = X.wU;
      W.tXR = X.wXR;
      W.tXL = X.wXL;
      W.tYR = X.wYR;
      W.tYL = X.wYL;
      cg_tile_apply<df, N>(
          *static_cast<const OpsK<df, N>*>(X.kdf), G, tile, W,
          [&](size_t g, int k, bool interior) { return df(load(g, k, interior)); },
          [&](size_t g, int k, df u, df q) { out(g, k, u.hi, to_float(q)); });
      return;
    }
    cg_tile_apply<T, N>(C, G, tile, X, load, out);
  }
}

// Where the tile's residual is staged for the preconditioner's cell part: X.sU itself, or,
// with a float32 preconditioner in a float64 solve, a float32 copy in the (then unused) trace
// arrays.
template <typename T, typename TP>
__device__ __forceinline__ TP* pc_stage(SolveCtx<T>& X) {
  if constexpr (std::is_same<T, TP>::value)
    return X.sU;
  else
    return reinterpret_cast<TP*>(X.tXR);
}

// Cell part of the preconditioner on one tile whose interior residual is staged (X.sU, and its
// copy in the preconditioner's precision TP): z~ = Bt r~ on every cell, rc = sum sqrt(W) r~ per
// cell (to P.rc); returns the tile's r~ . z~_block (in T).
template <typename T, int N, typename TP = T>
__device__ __forceinline__ T pc_cells(const Ops2D<T, N>& C, const Geom& G, const TileBox& B,
                                      const PrecondArgs<TP>& P, SolveCtx<T>& X) {
  constexpr int NN = N * N;
  const TP* Bs = reinterpret_cast<const TP*>(X.Bs);
  const TP* su = pc_stage<T, TP>(X);
  T rz = T(0);
  const int nin = B.TYe * B.TXe * NN;
  if constexpr (sizeof(TP) == 4 && kThreads % NN == 0) {
    // float32: a thread's nodes all have k = threadIdx.x mod n^2, so its column of Bt stays in
    // registers (same arithmetic and order as below)
    const int k = threadIdx.x % NN;
    TP bk[NN];
#pragma unroll
    for (int j = 0; j < NN; ++j) bk[j] = Bs[j * NN + k];
    for (int i = threadIdx.x; i < nin; i += kThreads) {
      const int c = i / NN;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const int cell = ((ry + 1) * B.BW + rx + 1) * (NN + 1);
      const TP* u = su + cell;
      TP zj = TP(0);
#pragma unroll
      for (int j = 0; j < NN; ++j) zj = fma(bk[j], u[j], zj);
      const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
      __stcg(P.z + g, zj);
      rz = fma(X.sU[cell + k], T(zj), rz);
    }
  } else {
    for (int i = threadIdx.x; i < nin; i += blockDim.x) {
      const int c = i / NN, k = i - (i / NN) * NN;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const int cell = ((ry + 1) * B.BW + rx + 1) * (NN + 1);
      const TP* u = su + cell;
      TP zj = TP(0);
#pragma unroll
      for (int j = 0; j < NN; ++j) zj = fma(Bs[j * NN + k], u[j], zj);  // Bt is symmetric
      const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
      __stcg(P.z + g, zj);
      rz = fma(X.sU[cell + k], T(zj), rz);
    }
  }
  const int ncell = B.TYe * B.TXe;
  for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
    const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
    const TP* u = su + ((ry + 1) * B.BW + rx + 1) * (NN + 1);
    TP v = TP(0);
#pragma unroll
    for (int k = 0; k < NN; ++k) v = fma(TP(C.sw[k]), u[k], v);
    __stcg(P.rc + (size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx), v);
  }
  return rz;
}

template <typename T>
__device__ __forceinline__ Cplx<T> ld_cplx(const Cplx<T>* p) {
  return Cplx<T>{__ldcg(&p->re), __ldcg(&p->im)};
}

// An entry of the spectral preconditioner's n x n transforms.  In float64 through the
// read-only path (the compiler then keeps them out of registers: holding a whole float64
// transform per direction would spill); in float32 a plain load (measured faster).
template <typename T>
__device__ __forceinline__ Cplx<T> ld_table(const Cplx<T>* p) {
  if constexpr (sizeof(T) == 8)
    return Cplx<T>{__ldg(&p->re), __ldg(&p->im)};
  else
    return *p;
}

template <typename T>
__device__ __forceinline__ void st_cplx(Cplx<T>* p, Cplx<T> v) {
  __stcg(&p->re, v.re);
  __stcg(&p->im, v.im);
}

// Coarse solve uc = A_c^+ rc (rc real, one value per cell).  Two real rows a, b travel as
// one complex row a + i b: its DFT Z gives both spectra, A_k = (Z_k + conj Z_-k) / 2 and
// B_k = (Z_k - conj Z_-k) / 2i, of which the columns kx = 0 .. Nx/2 are kept (the others are
// their conjugates).  Then per kept column: DFT over y, division by the eigenvalues (the
// constant mode dropped), inverse DFT; finally per row pair the inverse DFT of
// A + i B (extended by conjugate symmetry) returns row a in the real and row b in the
// imaginary part.  Three grid-wide phases; the spectrum array holds Ny x (Nx/2 + 1) values.
// Returns sum uc . rc (in every block).
template <typename T, typename TR = T>
__device__ __forceinline__ bool pc_coarse(const Geom& G, const PrecondArgs<T>& P, SolveCtx<TR>& X, TR& ucrc) {
  const int Nx = G.Nx, Ny = G.Ny;
  Cplx<T>* L0 = reinterpret_cast<Cplx<T>*>(X.line0);  // the solve's DFT line buffers, in T
  Cplx<T>* L1 = reinterpret_cast<Cplx<T>*>(X.line1);
  const int Nh = Nx / 2, W = Nh + 1;  // kept columns
  const int npairs = (Ny + 1) / 2;
  for (int pr = X.vrank; pr < npairs; pr += X.vsize) {
    const int ra = 2 * pr, rb = 2 * pr + 1;
    const bool hasb = rb < Ny;
    for (int j = threadIdx.x; j < Nx; j += blockDim.x) {
      const T va = __ldcg(P.rc + (size_t)ra * Nx + j);
      const T vb = hasb ? __ldcg(P.rc + (size_t)rb * Nx + j) : T(0);
      L0[dft_slot(j, P.log2x)] = Cplx<T>{va, vb};
    }
    __syncthreads();
    dft_line(L0, L1, Nx, P.log2x, P.twx, false);
    for (int k = threadIdx.x; k < W; k += blockDim.x) {
      const Cplx<T> zk = L0[k], zm = L0[k == 0 ? 0 : Nx - k];
      st_cplx(&P.C[(size_t)ra * W + k], Cplx<T>{T(0.5) * (zk.re + zm.re), T(0.5) * (zk.im - zm.im)});
      if (hasb) st_cplx(&P.C[(size_t)rb * W + k], Cplx<T>{T(0.5) * (zk.im + zm.im), T(0.5) * (zm.re - zk.re)});
    }
    __syncthreads();
  }
  if (!solve_barrier(X)) return false;
  const T scale = T(1) / (T(Nx) * T(Ny));
  for (int col = X.vrank; col < W; col += X.vsize) {
    for (int j = threadIdx.x; j < Ny; j += blockDim.x) L0[dft_slot(j, P.log2y)] = ld_cplx(&P.C[(size_t)j * W + col]);
    __syncthreads();
    dft_line(L0, L1, Ny, P.log2y, P.twy, false);
    for (int ky = threadIdx.x; ky < Ny; ky += blockDim.x) {
      const T f = (col == 0 && ky == 0) ? T(0) : scale / (P.ax[col] + P.ay[ky]);
      const Cplx<T> v = L0[ky];
      L1[dft_slot(ky, P.log2y)] = Cplx<T>{v.re * f, v.im * f};
    }
    __syncthreads();
    dft_line(L1, L0, Ny, P.log2y, P.twy, true);
    for (int j = threadIdx.x; j < Ny; j += blockDim.x) st_cplx(&P.C[(size_t)j * W + col], L1[j]);
    __syncthreads();
  }
  if (!solve_barrier(X)) return false;
  TR acc = TR(0);
  for (int pr = X.vrank; pr < npairs; pr += X.vsize) {
    const int ra = 2 * pr, rb = 2 * pr + 1;
    const bool hasb = rb < Ny;
    for (int k = threadIdx.x; k < Nx; k += blockDim.x) {
      // A_k, B_k for k > Nx/2 are the conjugates of the kept columns Nx - k
      const bool kept = k < W;
      const int kk = kept ? k : Nx - k;
      Cplx<T> A = ld_cplx(&P.C[(size_t)ra * W + kk]);
      Cplx<T> B = hasb ? ld_cplx(&P.C[(size_t)rb * W + kk]) : Cplx<T>{T(0), T(0)};
      if (!kept) {
        A.im = -A.im;
        B.im = -B.im;
      }
      L0[dft_slot(k, P.log2x)] = Cplx<T>{A.re - B.im, A.im + B.re};
    }
    __syncthreads();
    dft_line(L0, L1, Nx, P.log2x, P.twx, true);
    for (int j = threadIdx.x; j < Nx; j += blockDim.x) {
      const size_t ca = (size_t)ra * Nx + j;
      const T ua = L0[j].re;
      __stcg(P.uc + ca, ua);
      acc = fma(TR(ua), TR(__ldcg(P.rc + ca)), acc);
      if (hasb) {
        const size_t cb = (size_t)rb * Nx + j;
        const T ub = L0[j].im;
        __stcg(P.uc + cb, ub);
        acc = fma(TR(ub), TR(__ldcg(P.rc + cb)), acc);
      }
    }
    __syncthreads();
  }
  return reduce_all(X, acc, ucrc);
}

// ---- the spectral preconditioner's three phases (see PrecondArgs) -------------------------
// Units of the row phases: (row pair pr, node row a): rows cy0 = 2 pr, cy1 = 2 pr + 1 travel as
// one complex line per node column b (real part row cy0, imaginary part row cy1), as in
// pc_coarse.  Shared memory: N lines of max(Nx, Ny) complex values (twice that for the direct
// DFT of a length that is not a power of two).

// Phase 1: S[kx][cy][a][j] = sum_b conj(Vx[kx][b][j]) DFT_x(r~[cy, ., a, b])[kx].
template <typename TP, int N, typename TR>
__device__ __forceinline__ void spectral_rows_fwd(const Geom& G, const PrecondArgs<TP>& P, const TR* r,
                                                  SolveCtx<TR>& X) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cplx<TP>* L0 = reinterpret_cast<Cplx<TP>*>(X.line0);
  Cplx<TP>* Lt = L0 + N * Nx;
  const int units = (Ny + 1) / 2 * N;
  for (int u = next_unit(X, units); u < units; u = next_unit(X, units)) {
    const int pr = u / N, a = u - pr * N;
    const int cy0 = 2 * pr, cy1 = cy0 + 1;
    const bool hasb = cy1 < Ny;
    for (int i = threadIdx.x; i < Nx * N; i += blockDim.x) {
      const int cx = i / N, b = i - cx * N;
      const TP va = TP(__ldcg(r + (((size_t)cy0 * Nx + cx) * N + a) * N + b));
      const TP vb = hasb ? TP(__ldcg(r + (((size_t)cy1 * Nx + cx) * N + a) * N + b)) : TP(0);
      L0[b * Nx + dft_slot(cx, P.log2x)] = Cplx<TP>{va, vb};
    }
    __syncthreads();
    fft_lines(L0, Lt, N, Nx, P.log2x, P.twx, false, false);
#pragma unroll 1
    for (int k = threadIdx.x; k < W; k += blockDim.x) {
      const int km = k == 0 ? 0 : Nx - k;
      Cplx<TP> A[N], B[N];
#pragma unroll
      for (int b = 0; b < N; ++b) {
        const Cplx<TP> zk = L0[b * Nx + k], zm = L0[b * Nx + km];
        A[b] = Cplx<TP>{TP(0.5) * (zk.re + zm.re), TP(0.5) * (zk.im - zm.im)};
        B[b] = Cplx<TP>{TP(0.5) * (zk.im + zm.im), TP(0.5) * (zm.re - zk.re)};
      }
      const Cplx<TP>* V = P.Vx + (size_t)k * N * N;
      Cplx<TP>* Sa = P.S + (((size_t)k * Ny + cy0) * N + a) * N;
      Cplx<TP>* Sb = P.S + (((size_t)k * Ny + cy1) * N + a) * N;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        Cplx<TP> ta{TP(0), TP(0)}, tb{TP(0), TP(0)};
#pragma unroll
        for (int b = 0; b < N; ++b) {
          const Cplx<TP> v = ld_table(V + b * N + j);  // conj(v) * x
          ta.re = fma(v.re, A[b].re, fma(v.im, A[b].im, ta.re));
          ta.im = fma(v.re, A[b].im, fma(-v.im, A[b].re, ta.im));
          tb.re = fma(v.re, B[b].re, fma(v.im, B[b].im, tb.re));
          tb.im = fma(v.re, B[b].im, fma(-v.im, B[b].re, tb.im));
        }
        st_cplx(Sa + j, ta);
        if (hasb) st_cplx(Sb + j, tb);
      }
    }
    __syncthreads();
  }
  end_units(X, units);
}

// Phase 2, per unit (kx, j): DFT along y of S[kx][.][a][j] for every a, then per ky
// t = Vy^* x, t_i *= scale / (ly_i + lx_j) (0 for the constant mode), x = Vy t, inverse DFT.
template <typename TP, int N, typename TR>
__device__ __forceinline__ void spectral_cols(const Geom& G, const PrecondArgs<TP>& P, SolveCtx<TR>& X) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cplx<TP>* L0 = reinterpret_cast<Cplx<TP>*>(X.line0);
  Cplx<TP>* Lt = L0 + N * Ny;
  const TP scale = TP(1) / (TP(Nx) * TP(Ny));
  for (int u = next_unit(X, W * N); u < W * N; u = next_unit(X, W * N)) {
    const int kx = u / N, j = u - kx * N;
    const Cplx<TP>* Sk = P.S + (size_t)kx * Ny * N * N;
    for (int i = threadIdx.x; i < Ny * N; i += blockDim.x) {
      const int cy = i / N, a = i - cy * N;
      L0[a * Ny + dft_slot(cy, P.log2y)] = ld_cplx(Sk + ((size_t)cy * N + a) * N + j);
    }
    __syncthreads();
    fft_lines(L0, Lt, N, Ny, P.log2y, P.twy, false, false);
    const TP lxj = P.lx[kx * N + j];
#pragma unroll 1
    for (int ky = threadIdx.x; ky < Ny; ky += blockDim.x) {
      const Cplx<TP>* V = P.Vy + (size_t)ky * N * N;
      Cplx<TP> t[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        Cplx<TP> acc{TP(0), TP(0)};
#pragma unroll
        for (int a = 0; a < N; ++a) {
          const Cplx<TP> v = ld_table(V + a * N + i), x = L0[a * Ny + ky];
          acc.re = fma(v.re, x.re, fma(v.im, x.im, acc.re));
          acc.im = fma(v.re, x.im, fma(-v.im, x.re, acc.im));
        }
        const TP den = P.ly[ky * N + i] + lxj;
        const TP f = den == TP(0) ? TP(0) : scale / den;
        t[i] = Cplx<TP>{acc.re * f, acc.im * f};
      }
#pragma unroll
      for (int a = 0; a < N; ++a) {
        Cplx<TP> acc{TP(0), TP(0)};
#pragma unroll
        for (int i = 0; i < N; ++i) acc = cadd(acc, cmul(ld_table(V + a * N + i), t[i]));
        L0[a * Ny + ky] = acc;
      }
    }
    __syncthreads();
    fft_lines(L0, Lt, N, Ny, P.log2y, P.twy, true, true);
    Cplx<TP>* Sw = P.S + (size_t)kx * Ny * N * N;
    for (int i = threadIdx.x; i < Ny * N; i += blockDim.x) {
      const int cy = i / N, a = i - cy * N;
      st_cplx(Sw + ((size_t)cy * N + a) * N + j, L0[a * Ny + dft_slot(cy, P.log2y)]);
    }
    __syncthreads();
  }
  end_units(X, W * N);
}

// Phase 3: z~[cy, ., a, b] = inverse real DFT_x of sum_j Vx[kx][b][j] S[kx][cy][a][j].
template <typename TP, int N, typename TR>
__device__ __forceinline__ void spectral_rows_inv(const Geom& G, const PrecondArgs<TP>& P, SolveCtx<TR>& X) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cplx<TP>* L0 = reinterpret_cast<Cplx<TP>*>(X.line0);
  Cplx<TP>* Lt = L0 + N * Nx;
  const int units = (Ny + 1) / 2 * N;
  for (int u = next_unit(X, units); u < units; u = next_unit(X, units)) {
    const int pr = u / N, a = u - pr * N;
    const int cy0 = 2 * pr, cy1 = cy0 + 1;
    const bool hasb = cy1 < Ny;
#pragma unroll 1
    for (int k = threadIdx.x; k < W; k += blockDim.x) {
      const Cplx<TP>* V = P.Vx + (size_t)k * N * N;
      const Cplx<TP>* Sa = P.S + (((size_t)k * Ny + cy0) * N + a) * N;
      const Cplx<TP>* Sb = P.S + (((size_t)k * Ny + cy1) * N + a) * N;
      Cplx<TP> ta[N], tb[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        ta[j] = ld_cplx(Sa + j);
        tb[j] = hasb ? ld_cplx(Sb + j) : Cplx<TP>{TP(0), TP(0)};
      }
      const bool mirror = k > 0 && 2 * k != Nx;  // Nx - k is a distinct bin
#pragma unroll
      for (int b = 0; b < N; ++b) {
        Cplx<TP> A{TP(0), TP(0)}, B{TP(0), TP(0)};
#pragma unroll
        for (int j = 0; j < N; ++j) {
          const Cplx<TP> v = ld_table(V + b * N + j);
          A = cadd(A, cmul(v, ta[j]));
          B = cadd(B, cmul(v, tb[j]));
        }
        // Z = A + i B at k; at Nx - k the spectra of the real rows are conj(A), conj(B)
        L0[b * Nx + k] = Cplx<TP>{A.re - B.im, A.im + B.re};
        if (mirror) L0[b * Nx + Nx - k] = Cplx<TP>{A.re + B.im, B.re - A.im};
      }
    }
    __syncthreads();
    fft_lines(L0, Lt, N, Nx, P.log2x, P.twx, true, true);
    for (int i = threadIdx.x; i < Nx * N; i += blockDim.x) {
      const int cx = i / N, b = i - cx * N;
      const Cplx<TP> zv = L0[b * Nx + dft_slot(cx, P.log2x)];
      __stcg(P.z + (((size_t)cy0 * Nx + cx) * N + a) * N + b, zv.re);
      if (hasb) __stcg(P.z + (((size_t)cy1 * Nx + cx) * N + a) * N + b, zv.im);
    }
    __syncthreads();
  }
  end_units(X, units);
}

// ---- the spectral preconditioner in fixed point (power-of-two cell counts) -------------------
//
// z~ = Ahat^+ r~ for float64 solves, on the integer pipe (dg_fixed.cuh): the DFTs and the n x n
// transforms of the three phases above, which held the float64 pipe for 60% of a solve, on complex
// 64-bit integers.  A unit's lines are one block-floating-point array: every pass ORs the
// magnitudes of what it writes, and the next one shifts by the few bits that keep its results
// within 2^63 (inputs below 2^60; a radix-4 butterfly grows a component at most 4 sqrt(2)).  Only
// the twiddle products round, one unit each; a float64 butterfly rounds every sum.
//
// Data and twiddles split at 32 bits, x = h 2^32 + l with a signed l (the low word as it is), w in
// units of 2^-62: w x = 4 wh xh + (wh xl + wl xh) 2^-30, three multiply-adds per real product as
// everywhere; |x| <= 2^62.5 and |w| <= 1 keep the second accumulator below 2^63.  The n x n
// transforms, whose rows sum ten products, keep the 30-bit split and inputs below 2^60.
struct Cll {
  long long re, im;
};

// Bits of a magnitude: the high word with the sign folded in (0: below 2^32).
__device__ __forceinline__ unsigned fx_high(long long v) {
  const int h = int(v >> 32);
  return unsigned(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned fx_high(const Cll& v) { return fx_high(v.re) | fx_high(v.im); }
__device__ __forceinline__ int fx_bits(unsigned high) { return high ? 64 - __clz(high) : 32; }

// The magnitudes of a complex value, ORed: as many bits as the larger one.
__device__ __forceinline__ unsigned long long fx_mag64(const Cll& v) {
  return (unsigned long long)(llabs(v.re) | llabs(v.im));
}

// v / 2^s rounded to nearest (s > 0), v 2^-s (s <= 0).
__device__ __forceinline__ long long fx_shift(long long v, int s) {
  if (s > 62) return 0;
  return s > 0 ? (v + (1ll << (s - 1))) >> s : v << -s;
}
// (a + b) / 2^s rounded, s >= 1; the sum may pass 2^63.
__device__ __forceinline__ long long fx_half(long long a, long long b, int s) {
  const long long h = (a >> 1) + (b >> 1) + (a & b & 1);
  return s > 1 ? (h + (1ll << (s - 2))) >> (s - 1) : h;
}
__device__ __forceinline__ Cll fx_shift(const Cll& v, int s) { return Cll{fx_shift(v.re, s), fx_shift(v.im, s)}; }

__device__ __forceinline__ Cfx fx_split(const Cll& v) { return Cfx{fx_split(v.re), fx_split(v.im)}; }
// The 32-bit split.
__device__ __forceinline__ fx fx_words(long long y) {
  return fx{int(y >> 32) + int(unsigned(y) >> 31), int(unsigned(y))};
}

// A complex sum of products w x (Conj: conj(w) x), rounded by get().
struct CfxAcc {
  FxAcc r{0, 1ll << 29}, i{0, 1ll << 29};
  template <bool Conj>
  __device__ __forceinline__ void mac(const Cfx& w, const Cfx& x) {
    const fx n = fx_neg(w.im);
    fx_mac(r, w.re, x.re);
    fx_mac(r, Conj ? w.im : n, x.im);
    fx_mac(i, w.re, x.im);
    fx_mac(i, Conj ? n : w.im, x.re);
  }
  __device__ __forceinline__ Cll get() const { return Cll{r.a1 + (r.a0 >> 30), i.a1 + (i.a0 >> 30)}; }
};

// w x (Conj: conj(w) x) of a twiddle in the 32-bit split.
template <bool Conj>
__device__ __forceinline__ Cll fx_cmul(const Cfx& w, const Cll& x) {
  const fx xr = fx_words(x.re), xi = fx_words(x.im), n = fx{-w.im.h, -w.im.l};
  FxAcc r{0, 1ll << 29}, i{0, 1ll << 29};
  fx_mac(r, w.re, xr);
  fx_mac(r, Conj ? w.im : n, xi);
  fx_mac(i, w.re, xi);
  fx_mac(i, Conj ? n : w.im, xr);
  return Cll{(r.a1 << 2) + (r.a0 >> 30), (i.a1 << 2) + (i.a0 >> 30)};
}

__device__ __forceinline__ Cll operator+(const Cll& a, const Cll& b) { return Cll{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Cll operator-(const Cll& a, const Cll& b) { return Cll{a.re - b.re, a.im - b.im}; }
// times -i (forward) or +i (inverse)
template <bool Inv>
__device__ __forceinline__ Cll fx_turn(const Cll& a) {
  return Inv ? Cll{-a.im, a.re} : Cll{a.im, -a.re};
}

__device__ __forceinline__ Cfx ld_cfx(const Cfx* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return Cfx{fx{v.x, v.y}, fx{v.z, v.w}};
}
__device__ __forceinline__ Cll ld_cll(const Cll* p) {
  const longlong2 v = __ldcg(reinterpret_cast<const longlong2*>(p));
  return Cll{v.x, v.y};
}
__device__ __forceinline__ void st_cll(Cll* p, const Cll& v) {
  __stcg(reinterpret_cast<longlong2*>(p), make_longlong2(v.re, v.im));
}
__device__ __forceinline__ Cll lds_cll(const Cll* p) {
  const longlong2 v = *reinterpret_cast<const longlong2*>(p);
  return Cll{v.x, v.y};
}
__device__ __forceinline__ void sts_cll(Cll* p, const Cll& v) {
  *reinterpret_cast<longlong2*>(p) = make_longlong2(v.re, v.im);
}

// v, unknown to the compiler.
__device__ __forceinline__ int opaque(int v) {
  asm volatile("" : "+r"(v));
  return v;
}

// The magnitudes a block's pass wrote, ORed into s_or[slot % 3] (the slot after next is cleared for
// the pass that will use it); call before the pass's block synchronisation.
__device__ __forceinline__ void fx_note(unsigned* s_or, int slot, unsigned high) {
  high = __reduce_or_sync(0xffffffffu, high);
  if ((threadIdx.x & 31) == 0 && high) atomicOr(&s_or[slot % 3], high);
  if (threadIdx.x == 0) s_or[(slot + 1) % 3] = 0;
}

// DFTs of `count` lines of length L = 2^log2L >= 2 in shared memory, by the whole block.  Inv ==
// false: decimation in time (bit-reversed input, natural output); Inv == true: conjugate twiddles and
// decimation in frequency (natural input, bit-reversed output).  slot: the s_or slot that holds
// the input's magnitudes; it is advanced to the output's.  Returns the bits shifted out (the
// result times 2^returned is the DFT of the input).
template <bool Inv>
__device__ __forceinline__ int fx_fft_lines(Cll* s, int count, int L, int log2L, const Cfx* tw, unsigned* s_or,
                                            int& slot) {
  const int tid = threadIdx.x, nth = blockDim.x;
  int total = 0;
  // the shift that brings the pass's inputs below 2^60 (up as well as down)
  auto next_shift = [&]() {
    const unsigned m = s_or[slot % 3];
    int sh = m ? fx_bits(m) - 60 : 0;
    if (sh < 0 && (total != 0 || sh > -4)) sh = 0;  // up only before the first pass, if worthwhile
    total += sh;
    ++slot;
    return sh;
  };
  auto radix2 = [&]() {  // span 1, every twiddle 1
    const int sh = next_shift(), hl = L >> 1;
    unsigned high = 0;
    for (int t = tid; t < count * hl; t += nth) {
      Cll* b = s + (t >> (log2L - 1)) * L + 2 * (t & (hl - 1));
      Cll u = lds_cll(b), v = lds_cll(b + 1);
      if (sh) {
        u = fx_shift(u, sh);
        v = fx_shift(v, sh);
      }
      const Cll x = u + v, y = u - v;
      sts_cll(b, x);
      sts_cll(b + 1, y);
      high |= fx_high(x) | fx_high(y);
    }
    fx_note(s_or, slot, high);
    __syncthreads();
  };
  const int q = L >> 2;
  auto radix4 = [&](int h, int lh) {  // spans h and 2 h
    const int sh = next_shift(), s4 = L / (4 * h);
    unsigned high = 0;
    for (int t = tid; t < count * q; t += nth) {
      const int line = t >> (log2L - 2), tt = t & (q - 1);
      const int grp = tt >> lh, pos = tt & (h - 1);
      Cll* b = s + line * L + grp * 4 * h + pos;
      Cll x0 = lds_cll(b), x1 = lds_cll(b + h), x2 = lds_cll(b + 2 * h), x3 = lds_cll(b + 3 * h);
      if (sh) {
        x0 = fx_shift(x0, sh);
        x1 = fx_shift(x1, sh);
        x2 = fx_shift(x2, sh);
        x3 = fx_shift(x3, sh);
      }
      Cll y0, y1, y2, y3;
      if constexpr (!Inv) {
        if (h > 1) {
          x1 = fx_cmul<false>(ld_cfx(tw + 2 * pos * s4), x1);
          x2 = fx_cmul<false>(ld_cfx(tw + pos * s4), x2);
          x3 = fx_cmul<false>(ld_cfx(tw + 3 * pos * s4), x3);
        }
        const Cll s1 = x0 + x1, s2 = x0 - x1, s3 = x2 + x3, s4v = fx_turn<false>(x2 - x3);
        y0 = s1 + s3;
        y2 = s1 - s3;
        y1 = s2 + s4v;
        y3 = s2 - s4v;
      } else {
        const Cll u0 = x0 + x2, u1 = x1 + x3, u2 = x0 - x2, u3 = fx_turn<true>(x1 - x3);
        y0 = u0 + u1;
        y1 = u0 - u1;
        y2 = u2 + u3;
        y3 = u2 - u3;
        if (h > 1) {
          y1 = fx_cmul<true>(ld_cfx(tw + 2 * pos * s4), y1);
          y2 = fx_cmul<true>(ld_cfx(tw + pos * s4), y2);
          y3 = fx_cmul<true>(ld_cfx(tw + 3 * pos * s4), y3);
        }
      }
      sts_cll(b, y0);
      sts_cll(b + h, y1);
      sts_cll(b + 2 * h, y2);
      sts_cll(b + 3 * h, y3);
      high |= fx_high(y0) | fx_high(y1) | fx_high(y2) | fx_high(y3);
    }
    fx_note(s_or, slot, high);
    __syncthreads();
  };
  if constexpr (!Inv) {
    int lh = 0;
    if (log2L & 1) {
      radix2();
      lh = 1;
    }
    for (; lh < log2L; lh += 2) radix4(1 << lh, lh);
  } else {
    int lh = log2L - 2;
    for (; lh >= 0; lh -= 2) radix4(1 << lh, lh);
    if (lh == -1) radix2();
  }
  return total;
}

// 2^60 / m for the significand 2^52 <= m < 2^53 of a float64, times 2^52 (a value in (2^59, 2^60]):
// a float32 reciprocal and two Newton steps in integers, correct to 4 units.
__device__ __forceinline__ long long fx_recip(unsigned long long m) {
  // D = m / 2^53 in [1/2, 1) as D 2^60; r0 ~ 1 / D in (1, 2] with 24 bits, as rh 2^-29
  const long long D = (long long)(m << 7);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f000000u | unsigned((m >> 29) & 0x7fffffu))));
  const unsigned rb = __float_as_uint(r);
  int rh = int(((rb & 0x7fffffu) | 0x800000u) << 6) << ((rb >> 23) - 127);  // r 2^29, r in (1, 2]
  const fx d{int(D >> 30), int(unsigned(D) & 0x3fffffffu)};
  // e = 1 - D r0 in units of 2^-59 (D r0 2^59 = D 2^60 rh 2^30 / 2^61 ...)
  const long long e = (1ll << 59) - ((long long)d.h * rh + (((long long)d.l * rh) >> 30));
  long long R = ((long long)rh << 30) + 2 * (e >> 30) * rh + (((e & 0x3fffffffll) * rh) >> 29);
  FxAcc s;
  fx_mac(s, d, fx{int(R >> 30), int(unsigned(R) & 0x3fffffffu)});
  const long long e1 = (1ll << 59) - (s.a1 + (s.a0 >> 30));
  R += (e1 * (R >> 30)) >> 29;
  return R;  // 2^59 / D = 2^112 / m
}

// Phase 1: S[kx][cy][a][j] as in spectral_rows_fwd.  r~ has its largest magnitude's biased exponent er
// and enters below 2^57; every unit leaves its S in a scale of its own, noted in EU[W n + unit].
template <int N>
__device__ __forceinline__ void fx_rows_fwd(const Geom& G, const PrecondArgs<double>& P, const double* r, int er,
                                            SolveCtx<double>& X, unsigned* s_or) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cll* L0 = reinterpret_cast<Cll*>(X.line0);
  const int units = (Ny + 1) / 2 * N;
  for (int u = next_unit(X, units); u < units; u = next_unit(X, units)) {
    const int pr = u / N, a = u - pr * N;
    const int cy0 = 2 * pr, cy1 = cy0 + 1;
    const bool hasb = cy1 < Ny;
    if (threadIdx.x < 3) s_or[threadIdx.x] = 0;
    __syncthreads();
    unsigned high = 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < Nx * N; i += blockDim.x) {
      const int cx = i / N, b = i - cx * N;
      const double va = __ldcg(r + (((size_t)cy0 * Nx + cx) * N + a) * N + b);
      const double vb = hasb ? __ldcg(r + (((size_t)cy1 * Nx + cx) * N + a) * N + b) : 0.0;
      const Cll v{fx_from_bits(__double2hiint(va), __double2loint(va), er) >> 3,
                  fx_from_bits(__double2hiint(vb), __double2loint(vb), er) >> 3};
      sts_cll(L0 + b * Nx + dft_slot(cx, P.log2x), v);
      high |= fx_high(v);
    }
    fx_note(s_or, 0, high);
    __syncthreads();
    int slot = 0;
    const int shifted = P.log2x ? fx_fft_lines<false>(L0, N, Nx, P.log2x, P.ftwx, s_or, slot) : 0;
    // the two real rows' spectra are halves of sums: below 2^60 after this shift
    const int sh = max(1, fx_bits(s_or[slot % 3]) + 1 - 60);
    if (threadIdx.x == 0) {
      const int e = er - 1079 + shifted + sh - 1;
      P.EU[W * N + u] = make_int2(e + 62, e);  // |S| < 2^62: n values below 2^60 in a unitary transform
    }
#pragma unroll 1
    for (int k = threadIdx.x; k < W; k += blockDim.x) {
      const int km = k == 0 ? 0 : Nx - k;
      Cfx A[N], B[N];
#pragma unroll
      for (int b = 0; b < N; ++b) {
        const Cll zk = lds_cll(L0 + b * Nx + k), zm = lds_cll(L0 + b * Nx + km);
        A[b] = fx_split(Cll{fx_half(zk.re, zm.re, sh), fx_half(zk.im, -zm.im, sh)});
        B[b] = fx_split(Cll{fx_half(zk.im, zm.im, sh), fx_half(zm.re, -zk.re, sh)});
      }
      // entry (b, j) at [(b N + j) W + k]: coalesced over the threads' k (the stride is opaque, so that
      // the addresses of all entries are not kept in registers across the loop)
      const Cfx* V = P.fVx + k;
      const int vs = opaque(W);
      Cll* Sa = reinterpret_cast<Cll*>(P.S) + (((size_t)k * Ny + cy0) * N + a) * N;
      Cll* Sb = Sa + (size_t)N * N;
#pragma unroll 1
      for (int j = 0; j < N; ++j) {
        CfxAcc ta, tb;
#pragma unroll
        for (int b = 0; b < N; ++b) {
          const Cfx v = ld_cfx(V + (b * N + j) * vs);
          ta.mac<true>(v, A[b]);
          tb.mac<true>(v, B[b]);
        }
        st_cll(Sa + j, ta.get());
        if (hasb) st_cll(Sb + j, tb.get());
      }
    }
    __syncthreads();
  }
  end_units(X, units);
}

// The largest `top` of n units' scales, in every thread.
__device__ __forceinline__ int fx_top(const int2* EU, int n) {
  int top = -(1 << 28);
  for (int i = threadIdx.x & 31; i < n; i += 32) top = max(top, __ldcg(EU + i).x);
  return __reduce_max_sync(0xffffffffu, top);
}

// Phase 2, per unit (kx, j), as in spectral_cols.  Every unit leaves its S in a scale of its own, noted
// in P.EU.  Its quotients y / (ly + lx), each formed from its own 60-bit significand, share a scale that
// a quotient by the smallest sum would fill.  Where the unit's content lies in high eigenvalues only,
// up to 2^27 times the smallest, they come out that much below: the unit is then done again in a finer
// scale (its input is still in S).
template <int N>
__device__ __forceinline__ void fx_cols(const Geom& G, const PrecondArgs<double>& P, SolveCtx<double>& X,
                                        unsigned* s_or) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cll* L0 = reinterpret_cast<Cll*>(X.line0);
  const int2* E1 = P.EU + W * N;
  const int top = fx_top(E1, (Ny + 1) / 2 * N);  // S is brought to integers below 2^60 of it
  const int e0 = top - 60 - P.log2x - P.log2y;   // (the inverse DFTs' 1 / (Nx Ny) included)
  for (int u = next_unit(X, W * N); u < W * N; u = next_unit(X, W * N)) {
    const int kx = u / N, j = u - kx * N;
    Cll* Sk = reinterpret_cast<Cll*>(P.S) + (size_t)kx * Ny * N * N;
    const double lxj = P.lx[kx * N + j];
    // the smallest non-zero sum is 2^p (1 .. 2): quotients of values below 2^62 are below 2^(62 - p)
    int qtop = 62 - ((__double2hiint(lxj + P.lymin[lxj == 0.0 ? 1 : 0]) >> 20) - 1023);
    int slot, shifted;
    for (int pass = 0;; ++pass) {
      if (threadIdx.x < 3) s_or[threadIdx.x] = 0;
      __syncthreads();
      unsigned high = 0;
#pragma unroll 4
      for (int i = threadIdx.x; i < Ny * N; i += blockDim.x) {
        const int cy = i / N, a = i - cy * N;
        const Cll v = fx_shift(ld_cll(Sk + ((size_t)cy * N + a) * N + j), top - 60 - __ldcg(E1 + (cy >> 1) * N + a).y);
        sts_cll(L0 + a * Ny + dft_slot(cy, P.log2y), v);
        high |= fx_high(v);
      }
      fx_note(s_or, 0, high);
      __syncthreads();
      slot = 0;
      shifted = P.log2y ? fx_fft_lines<false>(L0, N, Ny, P.log2y, P.ftwy, s_or, slot) : 0;
      const int bits = fx_bits(s_or[slot % 3]), sh = max(0, bits - 60);
      shifted += sh;
      ++slot;
      high = 0;
#pragma unroll 1
      for (int ky = threadIdx.x; ky < Ny; ky += blockDim.x) {
        const Cfx* V = P.fVy + ky;
        const int vs = opaque(Ny);
        Cfx x[N];
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = fx_split(fx_shift(lds_cll(L0 + a * Ny + ky), sh));
#pragma unroll 1
        for (int i = 0; i < N; ++i) {
          CfxAcc acc;
#pragma unroll
          for (int a = 0; a < N; ++a) acc.mac<true>(ld_cfx(V + (a * N + i) * vs), x[a]);
          const Cll y = acc.get();  // |y| < 2^62
          const double den = P.ly[ky * N + i] + lxj;
          const unsigned long long m = fx_mag64(y);
          Cfx t{fx{0, 0}, fx{0, 0}};
          if (den != 0.0 && m) {
            // den = r 2^(e - 52) and q = 2^112 / r: y / den = y q 2^(-60 - e) = t 2^(qtop - 60)
            const int hi = __double2hiint(den), by = 64 - __clzll((long long)m);
            const fx q = fx_split(fx_recip((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 |
                                           (unsigned)__double2loint(den)));
            const Cfx w = fx_split(fx_shift(y, by - 60));
            FxAcc re{0, 1ll << 29}, im{0, 1ll << 29};
            fx_mac(re, q, w.re);
            fx_mac(im, q, w.im);
            t = fx_split(fx_shift(Cll{re.a1 + (re.a0 >> 30), im.a1 + (im.a0 >> 30)}, qtop - by + (hi >> 20) - 1023));
          }
          // x is in registers: t takes its place
          *reinterpret_cast<int4*>(L0 + i * Ny + ky) = make_int4(t.re.h, t.re.l, t.im.h, t.im.l);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const int4 t = *reinterpret_cast<const int4*>(L0 + i * Ny + ky);
          x[i] = Cfx{fx{t.x, t.y}, fx{t.z, t.w}};
        }
#pragma unroll 1
        for (int a = 0; a < N; ++a) {
          CfxAcc acc;
#pragma unroll
          for (int i = 0; i < N; ++i) acc.mac<false>(ld_cfx(V + (a * N + i) * vs), x[i]);
          const Cll v = acc.get();
          sts_cll(L0 + a * Ny + ky, v);
          high |= fx_high(v);
        }
      }
      fx_note(s_or, slot, high);
      __syncthreads();
      // t and V t have the same norm: with `lost` bits missing, t 2^(lost - 5) stays below 2^60.  (Below
      // 2^32 the bits are not known: a second time may show that more are missing.)  With 20 of them
      // gone an application still gains 12 digits; a closer line would redo units of ordinary
      // fields (32^2 cells, n = 3, a steady state and noise: 13 missing; 71.8 us a step, 74.0 with 12)
      const int lost = min(bits, 60) - fx_bits(s_or[slot % 3]);
      if (lost <= 20 || pass == 3) break;
      qtop -= lost - 5;
      __syncthreads();  // every thread has read s_or
    }
    if (P.log2y) shifted += fx_fft_lines<true>(L0, N, Ny, P.log2y, P.ftwy, s_or, slot);
    if (threadIdx.x == 0) {
      // values below 2^32, zeros among them, count as 2^32: their magnitudes are not noted
      const int e = e0 + shifted + qtop - 60;
      P.EU[u] = make_int2(e + fx_bits(s_or[slot % 3]), e);
    }
    for (int i = threadIdx.x; i < Ny * N; i += blockDim.x) {
      const int cy = i / N, a = i - cy * N;
      st_cll(Sk + ((size_t)cy * N + a) * N + j, lds_cll(L0 + a * Ny + dft_slot(cy, P.log2y)));
    }
    __syncthreads();
  }
  end_units(X, W * N);
}

// Phase 3, as in spectral_rows_inv: the units' scales are brought to one, integers below 2^60.
template <int N>
__device__ __forceinline__ void fx_rows_inv(const Geom& G, const PrecondArgs<double>& P, SolveCtx<double>& X,
                                            unsigned* s_or) {
  const int Nx = G.Nx, Ny = G.Ny, W = Nx / 2 + 1;
  Cll* L0 = reinterpret_cast<Cll*>(X.line0);
  const int top = fx_top(P.EU, W * N);
  const int units = (Ny + 1) / 2 * N;
  for (int u = next_unit(X, units); u < units; u = next_unit(X, units)) {
    const int pr = u / N, a = u - pr * N;
    const int cy0 = 2 * pr, cy1 = cy0 + 1;
    const bool hasb = cy1 < Ny;
    if (threadIdx.x < 3) s_or[threadIdx.x] = 0;
    __syncthreads();
    unsigned high = 0;
#pragma unroll 1
    for (int k = threadIdx.x; k < W; k += blockDim.x) {
      const Cfx* V = P.fVx + k;
      const int vs = opaque(W);
      const Cll* Sa = reinterpret_cast<const Cll*>(P.S) + (((size_t)k * Ny + cy0) * N + a) * N;
      const Cll* Sb = Sa + (size_t)N * N;
      Cfx ta[N], tb[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int sh = top - 60 - __ldcg(P.EU + k * N + j).y;
        ta[j] = fx_split(fx_shift(ld_cll(Sa + j), sh));
        tb[j] = hasb ? fx_split(fx_shift(ld_cll(Sb + j), sh)) : Cfx{fx{0, 0}, fx{0, 0}};
      }
      const bool mirror = k > 0 && 2 * k != Nx;  // Nx - k is a distinct bin
#pragma unroll 1
      for (int b = 0; b < N; ++b) {
        CfxAcc ra, rb;
#pragma unroll
        for (int j = 0; j < N; ++j) {
          const Cfx v = ld_cfx(V + (b * N + j) * vs);
          ra.mac<false>(v, ta[j]);
          rb.mac<false>(v, tb[j]);
        }
        const Cll A = ra.get(), B = rb.get();
        // Z = A + i B at k; at Nx - k the spectra of the real rows are conj(A), conj(B) (|A|, |B| < 2^62)
        const Cll z{A.re - B.im, A.im + B.re};
        sts_cll(L0 + b * Nx + k, z);
        high |= fx_high(z);
        if (mirror) {
          const Cll c{A.re + B.im, B.re - A.im};
          sts_cll(L0 + b * Nx + Nx - k, c);
          high |= fx_high(c);
        }
      }
    }
    fx_note(s_or, 0, high);
    __syncthreads();
    int slot = 0;
    const int e = top - 60 + (P.log2x ? fx_fft_lines<true>(L0, N, Nx, P.log2x, P.ftwx, s_or, slot) : 0);
    for (int i = threadIdx.x; i < Nx * N; i += blockDim.x) {
      const int cx = i / N, b = i - cx * N;
      const Cll zv = lds_cll(L0 + b * Nx + dft_slot(cx, P.log2x));
      __stcg(P.z + (((size_t)cy0 * Nx + cx) * N + a) * N + b, fx_to_double(zv.re, e));
      if (hasb) __stcg(P.z + (((size_t)cy1 * Nx + cx) * N + a) * N + b, fx_to_double(zv.im, e));
    }
    __syncthreads();
  }
  end_units(X, units);
}

// z~ = Ahat^+ r~ (spectral preconditioner): the three phases and the sum r~ . z~ (in every block).
template <typename TP, int N, typename TR>
__device__ __forceinline__ bool pc_spectral(const Geom& G, const PrecondArgs<TP>& P, const TR* r, SolveCtx<TR>& X,
                                            TR& rz) {
  spectral_rows_fwd<TP, N, TR>(G, P, r, X);
  if (!solve_barrier(X)) return false;
  spectral_cols<TP, N, TR>(G, P, X);
  if (!solve_barrier(X)) return false;
  spectral_rows_inv<TP, N, TR>(G, P, X);
  if (!solve_barrier(X)) return false;
  // r~ . z~ in a fixed order over the dofs (the units above were scheduled dynamically)
  const size_t ndof = (size_t)G.Nx * G.Ny * N * N;
  TR acc = TR(0);
  for (size_t i = (size_t)X.vrank * blockDim.x + threadIdx.x; i < ndof; i += (size_t)X.vsize * blockDim.x)
    acc = fma(TR(__ldcg(P.z + i)), __ldcg(r + i), acc);
  return reduce_all(X, acc, rz);
}

// z~ = M^-1 r~ for the residual currently in r; returns r~ . z~ in rz.
template <typename T, int N, typename TP = T>
__device__ __forceinline__ bool pc_apply(const Ops2D<T, N>& C, const Geom& G, const PrecondArgs<TP>& P, const T* r,
                                         SolveCtx<T>& X, T& rz) {
  constexpr int NN = N * N;
  if (P.kind == kPrecondSpectral) return pc_spectral<TP, N, T>(G, P, r, X, rz);
  const int ntiles = G.tilesX * G.tilesY;
  TP* su = pc_stage<T, TP>(X);
  T rzb = T(0);
  for (int t = X.vrank; t < ntiles; t += X.vsize) {
    const TileBox B = make_box(G, t);
    const int nin = B.TYe * B.TXe * NN;
    for (int i = threadIdx.x; i < nin; i += blockDim.x) {
      const int c = i / NN, k = i - (i / NN) * NN;
      const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
      const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
      const int o = ((ry + 1) * B.BW + rx + 1) * (NN + 1) + k;
      const T v = __ldcg(r + g);
      X.sU[o] = v;
      if constexpr (!std::is_same<T, TP>::value) su[o] = TP(v);
    }
    __syncthreads();
    rzb += pc_cells<T, N, TP>(C, G, B, P, X);
    __syncthreads();
  }
  T rzsum = T(0);
  if (!reduce_all(X, rzb, rzsum)) return false;
  T ucrc = T(0);
  if (!pc_coarse<TP, T>(G, P, X, ucrc)) return false;
  rz = rzsum + ucrc;
  return true;
}

// The CG iterations proper (PCG when P is non-null), from r (residual of the current y) with
// rr = r.r, rhob = b.b (the stopping rule is on r.r) and, with a preconditioner, z = M^-1 r
// already applied and rz = r.z.  The stopping rule is on the true residual: when the
// recursive residual meets the tolerance, one more tile pass computes b - Ahat y; if that
// misses the tolerance, CG restarts from it.  Returns the iteration count; raises flags.
template <typename T, int N, typename TP = T>
__device__ __forceinline__ int cg_iterate(const Ops2D<T, N>& C, const Geom& G, const CgVectors<T>& V,
                                          const PrecondArgs<TP>* P, const RhsSource<T>& Bsrc, SolveCtx<T>& X,
                                          T& rr, T rz, T rhob, double tol2, int maxit, int fixed_iters, int& flags,
                                          int max_restarts = kMaxRestarts, double floor2 = 0.0, T* ay = nullptr) {
  constexpr int NN = N * N;
  const int ntiles = G.tilesX * G.tilesY;
  const size_t ndof = (size_t)G.Nx * G.Ny * NN;
  const size_t stride = (size_t)X.vsize * blockDim.x;
  int it = 0, restarts = 0;
  double rr_prev = -1.0;  // true residual at the previous verification
  T beta = T(0);
  int cur = 0;
  bool first = true;  // p = z (no previous direction)
  const bool spec = P && P->kind == kPrecondSpectral;
  if (!P) rz = rr;
  while (true) {
    if (fixed_iters > 0) {
      if (it >= fixed_iters) break;
    } else if (double(rr) <= tol2 * double(rhob)) {
      if (max_restarts == 0) break;  // loose inner solves: the recursive residual suffices
      // Verify on the true residual r = b - Ahat y: accept it below the tolerance, or once it
      // stagnates below the float64 rounding floor of the iterate y (floor2 * y.y, see
      // CgArgs::floor2), where no float64 iterate can do better.
      T rt = T(0), yt = T(0);
      for (int t = X.vrank; t < ntiles; t += X.vsize) {
        solve_apply<T, N>(
            C, G, t, X, [&](size_t g, int, bool) { return __ldcg(V.y + g); }, [&](size_t g) { return __ldcg(V.y + g); },
            [&](size_t g, int k, T yv, T qv) {
              const T r = rhs_at<T, N>(C, Bsrc, g, k) - qv;
              __stcg(V.r + g, r);
              if (ay) __stcg(ay + g, qv);
              rt = fma(r, r, rt);
              yt = fma(yv, yv, yt);
            });
      }
      T rr_true = T(0), yy = T(0);
      if (!reduce_all2(X, rt, yt, rr_true, yy)) {
        flags |= kFlagTimeout;
        return it;
      }
      rr = rr_true;
      if (double(rr_true) <= tol2 * double(rhob)) break;
      // stagnation at the rounding floor: below it, and less than a factor 4 below the previous
      // check's true residual
      if (double(rr_true) <= floor2 * double(yy) && rr_prev >= 0.0 && double(rr_true) > 0.25 * rr_prev) break;
      rr_prev = double(rr_true);
      if (restarts >= max_restarts) {
        flags |= kFlagNoconv;
        break;
      }
      ++restarts;
      if (P) {
        if (!pc_apply<T, N, TP>(C, G, *P, V.r, X, rz)) {
          flags |= kFlagTimeout;
          return it;
        }
      } else {
        rz = rr;
      }
      first = true;
      continue;
    }
    if (rr == T(0)) break;
    if (it >= maxit) {
      flags |= kFlagNoconv;
      break;
    }
    T* pin = cur ? V.p1 : V.p0;
    T* pout = cur ? V.p0 : V.p1;
    // Phase A: p = z + beta p_old (halo recomputed locally), q = Ahat p, p.q.
    T pq = T(0);
    for (int t = X.vrank; t < ntiles; t += X.vsize) {
      solve_apply<T, N>(
          C, G, t, X,
          [&](size_t g, int k, bool interior) {
            const T zv = spec ? T(__ldcg(P->z + g))
                         : P  ? fma(C.sw[k], T(__ldcg(P->uc + unsigned(g) / NN)), T(__ldcg(P->z + g)))
                              : __ldcg(V.r + g);
            const T pv = first ? zv : fma(beta, __ldcg(pin + g), zv);
            if (interior) __stcg(pout + g, pv);
            return pv;
          },
          [&](size_t g) { return __ldcg(pout + g); },  // written above, by this block
          [&](size_t g, int, T pv, T qv) {
            __stcg(V.q + g, qv);
            pq = fma(pv, qv, pq);
          });
    }
    T pqs = T(0);
    if (!reduce_all(X, pq, pqs)) {
      flags |= kFlagTimeout;
      return it;
    }
    if (!(pqs > T(0))) {
      // In parity mode (a fixed iteration count) CG may run past exact convergence on tiny
      // systems, where p.q is rounding noise (zero or negative): stop there.  Anything else
      // (a non-positive p.q in a tolerance-stopped solve, or NaN) is a breakdown.
      if (!(fixed_iters > 0 && pqs <= T(0))) flags |= kFlagBreakdown;
      break;
    }
    const T alpha = rz / pqs;
    // Phase B: y += alpha p, r -= alpha q, r.r (and the cell part of the preconditioner).
    T rrb = T(0), rzb = T(0);
    if (!P || spec) {
      struct Pqyr {
        T p, q, y, r;
      };
      strided_pass<2>(
          (size_t)X.vrank * blockDim.x + threadIdx.x, ndof, stride,
          [&](size_t i) { return Pqyr{__ldcg(pout + i), __ldcg(V.q + i), __ldcg(V.y + i), __ldcg(V.r + i)}; },
          [&](size_t i, const Pqyr& v) {
            const T yv = fma(alpha, v.p, v.y);
            const T rv = fma(-alpha, v.q, v.r);
            __stcg(V.y + i, yv);
            __stcg(V.r + i, rv);
            rrb = fma(rv, rv, rrb);
          });
    } else {
      for (int t = X.vrank; t < ntiles; t += X.vsize) {
        const TileBox B = make_box(G, t);
        const int nin = B.TYe * B.TXe * NN;
        for (int i = threadIdx.x; i < nin; i += blockDim.x) {
          const int c = i / NN, k = i - (i / NN) * NN;
          const int ry = quot(c, B.mTXe), rx = c - ry * B.TXe;
          const size_t g = ((size_t)(B.ty0 + ry) * G.Nx + (B.tx0 + rx)) * NN + k;
          const T pv = __ldcg(pout + g), qv = __ldcg(V.q + g);
          const T yv = fma(alpha, pv, __ldcg(V.y + g));
          const T rv = fma(-alpha, qv, __ldcg(V.r + g));
          __stcg(V.y + g, yv);
          __stcg(V.r + g, rv);
          rrb = fma(rv, rv, rrb);
          const int o = ((ry + 1) * B.BW + rx + 1) * (NN + 1) + k;
          X.sU[o] = rv;
          if constexpr (!std::is_same<T, TP>::value) pc_stage<T, TP>(X)[o] = TP(rv);
        }
        __syncthreads();
        rzb += pc_cells<T, N, TP>(C, G, B, *P, X);
        __syncthreads();
      }
    }
    T rnew = T(0), rzjs = T(0);
    if (!reduce_all2(X, rrb, rzb, rnew, rzjs)) {
      flags |= kFlagTimeout;
      return it;
    }
    T rznew = rnew;
    if (fixed_iters == 0 && double(rnew) <= tol2 * double(rhob)) {
      // converged by the recursive residual: the next pass verifies the true residual and, on
      // a restart, preconditions that one, so this residual needs no preconditioning
      rr = rnew;
      cur ^= 1;
      first = false;
      ++it;
      continue;
    }
    if (spec) {
      if (!pc_spectral<TP, N, T>(G, *P, V.r, X, rznew)) {
        flags |= kFlagTimeout;
        return it;
      }
    } else if (P) {
      T ucrc = T(0);
      if (!pc_coarse<TP, T>(G, *P, X, ucrc)) {
        flags |= kFlagTimeout;
        return it;
      }
      rznew = rzjs + ucrc;
    }
    beta = rznew / rz;
    rz = rznew;
    rr = rnew;
    cur ^= 1;
    first = false;
    ++it;
  }
  return it;
}

// The solve proper with the spectral preconditioner in fixed point: M^-1 = Ahat^+ makes the first CG
// step length 1 up to rounding, so the iteration is y <- y + Ahat^+ r with the true residual
// r = b - Ahat y after every step -- the stopping rule of cg_iterate, without the second operator
// application, the dot products and the vector updates that find a step length of 1.  y starts in
// V.p0 and ends in V.y; r, rr, mag (its largest magnitude word) belong to it.  Whatever rr says, the
// pass that evaluates the true residual runs at least once: it also leaves the operator product of y
// in ay and the sums that take the W-mean out.  Returns the number of preconditioner applications;
// raises flags.
template <int N>
__device__ __forceinline__ int fx_spectral_iterate(const Ops2D<double, N>& C, const Geom& G, const CgVectors<double>& V,
                                                   const PrecondArgs<double>& P, const RhsSource<double>& Bsrc,
                                                   SolveCtx<double>& X, double& rr, double rhob, unsigned mag,
                                                   double tol2, int maxit, int& flags, double floor2, double sumW,
                                                   double* ay, SolveStatus* st) {
  __shared__ unsigned s_or[3];
  const int ntiles = G.tilesX * G.tilesY;
  const size_t ndof = (size_t)G.Nx * G.Ny * N * N;
  double *yin = V.p0, *yout = V.y;
  double yy = 0.0, sy = 0.0, rr_prev = -1.0;
  int it = 0;
  bool fresh = false;  // rr is the residual that the pass below evaluated
  while (true) {
    const bool met = rr <= tol2 * rhob;
    if (X.vrank == 0 && threadIdx.x == 0 && it < kRefineHistory) {
      st->hist_rr[it] = rr / rhob;
      st->hist_it[it] = 1;
      st->hist_len = it + 1;
    }
    if (fresh) {
      if (met || rr == 0.0) break;
      // stagnation at the float64 rounding floor of y (see CgArgs::floor2)
      if (rr <= floor2 * yy && rr_prev >= 0.0 && rr > 0.25 * rr_prev) break;
      rr_prev = rr;
      if (it >= maxit || it > kMaxRestarts) {
        flags |= kFlagNoconv;
        break;
      }
    }
    const bool step = !met && it < maxit;  // (maxit = 0: y0 is evaluated alone)
    const int er = int(mag >> 20);
    if (step) {
      // a finite non-zero rr bounds the largest residual by 2^+-537: every scale below is a normal number
      if (!(rr <= 1.7976931348623157e308)) {
        flags |= kFlagBreakdown;
        break;
      }
      fx_rows_fwd<N>(G, P, V.r, er, X, s_or);
      bool ok = solve_barrier(X);
      if (ok) {
        fx_cols<N>(G, P, X, s_or);
        ok = solve_barrier(X);
      }
      if (ok) {
        fx_rows_inv<N>(G, P, X, s_or);
        ok = solve_barrier(X);
      }
      if (!ok) {
        flags |= kFlagTimeout;
        return it;
      }
      ++it;
    }
    double rt = 0.0, yt = 0.0, st_ = 0.0;
    mag = 0;
    for (int t = X.vrank; t < ntiles; t += X.vsize) {
      solve_apply<double, N>(
          C, G, t, X,
          [&](size_t g, int k, bool interior) {
            double y = __ldcg(yin + g);
            if (step) y += __ldcg(P.z + g);
            if (interior) {
              __stcg(yout + g, y);
              yt = fma(y, y, yt);
              st_ = fma(C.sw[k], y, st_);
            }
            return y;
          },
          [](size_t) { return 0.0; },
          [&](size_t g, int k, double, double q) {
            const double r = rhs_at<double, N>(C, Bsrc, g, k) - q;
            __stcg(V.r + g, r);
            if (ay) __stcg(ay + g, q);
            rt = fma(r, r, rt);
            mag = max(mag, fx_mag(r));
          });
    }
    double v[3] = {rt, yt, st_}, o[3];
    if (!reduce_sums<3>(X, v, o, &mag)) {
      flags |= kFlagTimeout;
      return it;
    }
    rr = o[0];
    yy = o[1];
    sy = o[2];
    fresh = true;
    double* const t = yin;
    yin = yout;
    yout = t;
  }
  // the W-mean of psi = y / sqrt(W) comes out (y -= m sqrt(W), as project_mean); the transforms drop
  // the constant, so what is left is usually below the rounding of y and the pass is skipped
  const double m = sy / sumW;
  const bool project = m * m * sumW > ldexp(yy, -108);
  if (yin != V.y || project) {
    strided_pass<4>((size_t)X.vrank * blockDim.x + threadIdx.x, ndof, (size_t)X.vsize * blockDim.x,
                    [&](size_t i) { return __ldcg(yin + i); },
                    [&](size_t i, double y) { __stcg(V.y + i, project ? fma(-m, C.sw[unsigned(i) % (N * N)], y) : y); });
    if (!solve_barrier(X)) flags |= kFlagTimeout;
  }
  return it;
}

// Removes the W-mean of psi = y / sqrt(W) from y (y -= m sqrt(W)): a preconditioner other
// than W^-1 moves the iterates along the constants, the kernel of A.
template <typename T, int N>
__device__ __forceinline__ bool project_mean(const Ops2D<T, N>& C, const Geom& G, T* y, double sumW,
                                             SolveCtx<T>& X) {
  constexpr int NN = N * N;
  const size_t ndof = (size_t)G.Nx * G.Ny * NN;
  const size_t stride = (size_t)X.vsize * blockDim.x;
  const size_t first = (size_t)X.vrank * blockDim.x + threadIdx.x;
  T s = T(0);
  strided_pass<4>(first, ndof, stride, [&](size_t i) { return __ldcg(y + i); },
                  [&](size_t i, T v) { s = fma(C.sw[unsigned(i) % NN], v, s); });
  T m = T(0);
  if (!reduce_all(X, s, m)) return false;
  m = m / T(sumW);
  strided_pass<4>(first, ndof, stride, [&](size_t i) { return __ldcg(y + i); },
                  [&](size_t i, T v) { __stcg(y + i, fma(-m, C.sw[unsigned(i) % NN], v)); });
  return solve_barrier(X);
}

template <typename T, typename TP = T>
struct CgArgs {
  const double* omega;  // b = sqrt(W) (omega - mean_W omega) ...
  const T* rhs;         // ... or b = rhs (scaled space) when non-null
  const double* xa;     // initial guess y0 = ca xa + cb xb (null terms dropped), times
  const double* xb;     // sqrt(W) when x_unscaled
  double ca, cb;
  int x_unscaled;
  // Recycled operator products (the stepper's extrapolated guesses): with axa non-null, Ahat y0
  // = ca axa + cb axb (scaled space, x_unscaled == 0) replaces the setup's operator application,
  // and with ay non-null the solve stores Ahat y of its final iterate there (from the verifying
  // true-residual pass that ends every tolerance-stopped solve).
  const T* axa;
  const T* axb;
  T* ay;
  CgVectors<T> v;
  int precond;          // kPrecondJacobi (W^-1: plain CG on the scaled system), kPrecondTwoLevel or kPrecondSpectral
  PrecondArgs<TP> pc;   // (TP = float: the preconditioner applied in float32)
  double* psi_out;      // if non-null: psi = y / sqrt(W) at the end
  T* part;              // 8 * gridDim.x
  SyncState* sync;
  SolveStatus* status;
  double tol2;
  // The float64 rounding floor of the residual, per unit y.y: rounding y to float64 and
  // evaluating b - Ahat y in float64 leave a residual of up to about 2 u lambda_max |y|
  // (u = 2^-53, lambda_max bounded by the row sums of |Ahat|), so floor2 = (2^-52 lambda)^2;
  // a solve whose true residual stagnates below floor2 y.y stops there, even above tol2 b.b.
  double floor2;
  int maxit, fixed_iters;
  double sumW;
  int cluster;          // launched as one thread-block cluster (cluster barriers)
  int keep_mean;        // homogeneous Dirichlet: A is definite, b = sqrt(W) omega (no mean removed)
  FxScale ks;           // factors of the fixed-point operator
};

// Dynamic shared memory of the persistent solves: [Bt (with the preconditioner)] then one
// region used both for the tile staging and for two DFT lines.
__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

template <typename T, int N>
__host__ __device__ constexpr size_t cg_tile_values(int TY, int TX) {
  return (size_t)(TY + 2) * (TX + 2) * (N * N + 1 + 4 * N);
}

// Bytes of the tile staging of a solve: float32 (and, in 8-byte values, double-float) operator
// applications use cg_tile_values, float64 ones the fixed-point pass; the two-level
// preconditioner's cell part stages a box of values with, in float64, a float32 copy beside it.
template <typename T, int N>
__host__ __device__ constexpr size_t cg_tile_bytes(int TY, int TX) {
  if (sizeof(T) == 4) return cg_tile_values<T, N>(TY, TX) * sizeof(T);
  const size_t a = fx_apply_bytes<N>(TY, TX), b = (size_t)(TY + 2) * (TX + 2) * (N * N + 1) * 12;
  return a > b ? a : b;
}

// Bytes of the DFT line buffers of a preconditioner (kind: PrecondArgs): two lines for the
// two-level coarse solve, N lines (2N for a length that is not a power of two) for the spectral
// one; pow2: both cell counts are powers of two.
template <typename T, int N>
__host__ __device__ constexpr size_t pc_line_bytes(int kind, int Lmax, bool pow2) {
  return kind == kPrecondTwoLevel   ? 2 * (size_t)Lmax * sizeof(Cplx<T>)
         : kind == kPrecondSpectral ? (pow2 ? 1 : 2) * (size_t)N * Lmax * sizeof(Cplx<T>)
                                    : 0;
}

template <typename T, int N>
__host__ __device__ constexpr size_t cg_smem_bytes(int TY, int TX, int Lmax, int kind, bool pow2) {
  return (kind == kPrecondTwoLevel ? align16(sizeof(T) * N * N * N * N) : 0) +
         align16(cg_tile_bytes<T, N>(TY, TX) > pc_line_bytes<T, N>(kind, Lmax, pow2)
                     ? cg_tile_bytes<T, N>(TY, TX)
                     : pc_line_bytes<T, N>(kind, Lmax, pow2));
}

// Lays out the solve context over dynamic shared memory starting at base (bytes).
template <typename T, int N, typename TB = T>
__device__ __forceinline__ void init_ctx(SolveCtx<T>& X, unsigned char* base, const Geom& G, const TB* Bt_global,
                                         bool pc, int Lmax) {
  constexpr int NN = N * N;
  unsigned char* p = base;
  if (pc) {
    TB* Bs = reinterpret_cast<TB*>(p);  // Bt in the preconditioner's precision TB (<= T)
    for (int i = threadIdx.x; i < NN * NN; i += blockDim.x) Bs[i] = Bt_global[i];
    X.Bs = reinterpret_cast<const T*>(Bs);
    p += align16(sizeof(T) * NN * NN);
  } else {
    X.Bs = nullptr;
  }
  const int boxc = (G.TY + 2) * (G.TX + 2);
  X.sU = reinterpret_cast<T*>(p);
  X.tXR = X.sU + boxc * (NN + 1);
  X.tXL = X.tXR + boxc * N;
  X.tYR = X.tXL + boxc * N;
  X.tYL = X.tYR + boxc * N;
  X.line0 = reinterpret_cast<Cplx<T>*>(p);
  X.line1 = X.line0 + Lmax;
  X.cluster = 0;
  X.kdf = nullptr;
  X.wU = X.wXR = X.wXL = X.wYR = X.wYL = nullptr;
  __syncthreads();
}

// Whether a float64 solve takes the fixed-point spectral path: the spectral preconditioner with its
// fixed-point tables (power-of-two cell counts), run to a tolerance.
__host__ __device__ __forceinline__ bool fx_spectral_solve(const PrecondArgs<double>& P, int precond, int fixed_iters) {
  return precond == kPrecondSpectral && P.fVx && fixed_iters == 0;
}

// The whole Poisson solve on the (virtual) grid of X (context laid out by init_ctx).  Fxs: the
// fixed-point spectral path (fx_spectral_solve), else CG.
template <typename T, int N, typename TP = T, bool Fxs = false>
__device__ __forceinline__ void cg_solve(const Ops2D<T, N>& C, const Geom& G, const CgArgs<T, TP>& A,
                                         SolveCtx<T>& X) {
  constexpr int NN = N * N;
  const bool pc = A.precond != kPrecondJacobi;
  X.sync = A.sync;
  X.part = A.part;
  X.phase = 0;
  X.ks = A.ks;
  X.tbase = read_ticket<T>(A.sync);  // before the first barrier: no block has drawn yet
  const int ntiles = G.tilesX * G.tilesY;
  const size_t ndof = (size_t)G.Nx * G.Ny * NN;
  const size_t stride = (size_t)X.vsize * blockDim.x;
  int flags = 0, it = 0;
  T rr = T(0), rhob = T(0), rz = T(0);

  // the fixed-point spectral path starts from y0 in p0
  T* const y0v = Fxs ? A.v.p0 : A.v.y;
  unsigned mag = 0;
  auto reduce_rr = [&](T a, T b) {
    T v[2] = {a, b}, o[2];
    if (!reduce_sums<2>(X, v, o, Fxs ? &mag : nullptr)) return false;
    rr = o[0];
    rhob = o[1];
    return true;
  };

  // P0: W-mean of omega, in two passes (the second removes the rounding left by the first,
  // so that b carries no rounding-sized component along the kernel of A).
  T wbar = T(0);
  if (A.rhs == nullptr && !A.keep_mean) {
    for (int pass = 0; pass < 2; ++pass) {
      T s = T(0);
      const size_t first = (size_t)X.vrank * blockDim.x + threadIdx.x;
      auto ld = [&](size_t i) { return T(A.omega[i]); };
      if (pass == 0)  // (the float64 pipe bounds these passes: no subtraction of 0)
        strided_pass<4>(first, ndof, stride, ld, [&](size_t i, T v) { s = fma(C.wq[unsigned(i) % NN], v, s); });
      else
        strided_pass<4>(first, ndof, stride, ld, [&](size_t i, T v) { s = fma(C.wq[unsigned(i) % NN], v - wbar, s); });
      T m = T(0);
      if (!reduce_all(X, s, m)) {
        flags |= kFlagTimeout;
        goto finish;
      }
      wbar += m / T(A.sumW);
    }
  }
  // P1: y0, b, r0 = b - Ahat y0, rr0 = r0.r0, rhob = b.b.
  if (A.axa) {  // Ahat y0 from the recycled products: a pointwise pass
    T rrb = T(0), bbb = T(0);
    const RhsSource<T> src{A.omega, A.rhs, wbar};
    for (size_t g = (size_t)X.vrank * blockDim.x + threadIdx.x; g < ndof; g += stride) {
      const int k = int(unsigned(g) % NN);
      T y0 = T(0), ax = T(0);
      if (A.xa) {
        y0 = T(A.ca) * T(A.xa[g]);
        ax = T(A.ca) * __ldcg(A.axa + g);
      }
      if (A.xb) {
        const T xb = T(A.xb[g]), axb = __ldcg(A.axb + g);
        if (A.cb == -1.0 && A.xa) {  // the stepper's 2 psi^k - psi^{k-1}: one rounding
          y0 = fma(T(A.ca), T(A.xa[g]), -xb);
          ax = fma(T(A.ca), __ldcg(A.axa + g), -axb);
        } else {
          y0 = fma(T(A.cb), xb, y0);
          ax = fma(T(A.cb), axb, ax);
        }
      }
      __stcg(y0v + g, y0);
      const T b = rhs_at<T, N>(C, src, g, k);
      const T r = b - ax;
      __stcg(A.v.r + g, r);
      rrb = fma(r, r, rrb);
      if constexpr (Fxs) mag = max(mag, fx_mag(r));
      bbb = fma(b, b, bbb);
    }
    if (!reduce_rr(rrb, bbb)) {
      flags |= kFlagTimeout;
      goto finish;
    }
  } else {
    T rrb = T(0), bbb = T(0);
    for (int t = X.vrank; t < ntiles; t += X.vsize) {
      solve_apply<T, N>(
          C, G, t, X,
          [&](size_t g, int k, bool interior) {
            double v = 0.0;
            if (A.xa) v = A.ca * A.xa[g];
            if (A.xb) v = fma(A.cb, A.xb[g], v);
            T tv = A.x_unscaled ? T(v) * C.sw[k] : T(v);
            if (interior) __stcg(y0v + g, tv);
            return tv;
          },
          [](size_t) { return T(0); },
          [&](size_t g, int k, T, T qv) {
            const T b = rhs_at<T, N>(C, RhsSource<T>{A.omega, A.rhs, wbar}, g, k);
            const T r = b - qv;
            __stcg(A.v.r + g, r);
            rrb = fma(r, r, rrb);
            if constexpr (Fxs) mag = max(mag, fx_mag(r));
            bbb = fma(b, b, bbb);
          });
    }
    if (!reduce_rr(rrb, bbb)) {
      flags |= kFlagTimeout;
      goto finish;
    }
  }
  if (rhob == T(0)) {
    for (size_t i = (size_t)X.vrank * blockDim.x + threadIdx.x; i < ndof; i += stride) __stcg(A.v.y + i, T(0));
    rr = T(0);
  } else if constexpr (Fxs) {
    it = fx_spectral_iterate<N>(C, G, A.v, A.pc, RhsSource<T>{A.omega, A.rhs, wbar}, X, rr, rhob, mag, A.tol2,
                                A.maxit, flags, A.floor2, A.sumW, A.ay, A.status);
  } else {
    if (pc && !pc_apply<T, N, TP>(C, G, A.pc, A.v.r, X, rz)) {
      flags |= kFlagTimeout;
      goto finish;
    }
    it = cg_iterate<T, N, TP>(C, G, A.v, pc ? &A.pc : nullptr, RhsSource<T>{A.omega, A.rhs, wbar}, X, rr, rz, rhob,
                              A.tol2, A.maxit, A.fixed_iters, flags, kMaxRestarts, A.floor2, A.ay);
    if (pc && !(flags & kFlagTimeout) && !project_mean<T, N>(C, G, A.v.y, A.sumW, X)) flags |= kFlagTimeout;
  }
finish:
  if (A.psi_out && !(flags & kFlagTimeout)) {
    strided_pass<4>((size_t)X.vrank * blockDim.x + threadIdx.x, ndof, stride,
                    [&](size_t i) { return __ldcg(A.v.y + i); },
                    [&](size_t i, T v) { A.psi_out[i] = double(v * C.isw[unsigned(i) % NN]); });
  }
  if (X.vrank == 0 && threadIdx.x == 0) {
    SolveStatus* st = A.status;
    st->total_iters += it;
    st->last_iters = it;
    st->max_iters = max(st->max_iters, it);
    st->last_flags = flags;
    st->flags |= flags;
    st->nsolves += 1;
    st->last_sweeps = Fxs ? it : 0;
    st->last_rho = double(rr);
    st->last_rhob = double(rhob);
  }
}

// Two blocks per SM and up to 128 registers a thread: the fixed-point operator and the spectral
// transforms hold a line's or a wave number's n values in registers (blocks of 384 and 512 threads with
// 80 and 64 registers are no faster: 1024^2 cells, n = 5 4148 / 4102 / 4153 us per solve, 32^2, n = 3
// 65 / 76 / 83).
template <typename T, int N, typename TP = T, bool Fxs = false>
__global__ void __launch_bounds__(kThreads, 2) cg_kernel(const __grid_constant__ Ops2D<T, N> C, const Geom G,
                                                        const __grid_constant__ CgArgs<T, TP> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T red[112];
  __shared__ BarrierState bs;
  if (threadIdx.x == 0) bs = BarrierState{0, 0};
  const Ops2D<T, N>& Cs = stage_table(C, smem_raw);
  SolveCtx<T> X;
  init_ctx<T, N, TP>(X, smem_raw + table_bytes<Ops2D<T, N>>(), G, A.pc.Bt, A.precond == 1, max(G.Nx, G.Ny));
  X.red = red;
  X.bs = &bs;
  X.vrank = blockIdx.x;
  X.vsize = gridDim.x;
  X.cluster = A.cluster;
  cg_solve<T, N, TP, Fxs>(Cs, G, A, X);
}

// =========================================================================================
// Mixed precision Poisson solve (iterative refinement, all on the device):
//   y  <- y0;  r = b - Ahat y  in float64
//   while r.r > tol^2 b.b:  solve Ahat e = r in float32 by CG from e = 0 to the relative
//                           tolerance tol_in;  y += e (float64);  r = b - Ahat y (float64)
// The float64 residual is the true residual of the float64 iterate, so the outer stopping
// rule needs no further check.
// =========================================================================================
struct MixedArgs {
  const double* omega;
  const double* xa;
  const double* xb;
  double ca, cb;
  int x_unscaled;
  const double* axa;   // recycled operator products, as in CgArgs
  const double* axb;
  double* ay;
  double* y;           // float64 solution (scaled space)
  double* psi_out;     // if non-null: psi = y / sqrt(W) at the end
  float* rf;           // float32 copy of the float64 residual (inner right-hand side)
  CgVectors<float> v;  // inner solve: y = e, r, p0, p1, q
  int precond;         // kPrecondJacobi, kPrecondTwoLevel or kPrecondSpectral (inner float32 solve)
  PrecondArgs<float> pc;
  double* partd;       // 8 * gridDim.x
  float* partf;        // 8 * gridDim.x
  SyncState* sync;
  SolveStatus* status;
  double tol2, tol_in2;
  double floor2;       // the float64 rounding floor per unit y.y (see CgArgs::floor2)
  int max_sweeps, maxit_in;
  double sumW;
  int cluster;         // launched as one thread-block cluster (cluster barriers)
  // the inner solve's operator apply (see solve_apply): 0 float32, 1 double-float, 2 float32
  // until a refinement sweep after the second reduces the residual by less than a factor 100
  // (too inexact on this problem's smoothest modes), double-float from then on
  int precise_apply;
  int keep_mean;       // homogeneous Dirichlet: b = sqrt(W) omega (no mean removed)
  FxScale ks;          // factors of the fixed-point operator (float64 residuals)
  bool half;           // the residuals' tiles are half the solve's (launch_mixed)
};

// The operator tables a mixed solve stages in shared memory: float64 (residuals), float32
// (inner solve) and the double-float CG operator (compensated apply).
template <int N>
__host__ __device__ constexpr size_t mixed_ops_bytes() {
  return table_bytes<Ops2D<double, N>>() + table_bytes<Ops2D<float, N>>() + table_bytes<OpsK<df, N>>();
}

// The tiles of the float64 residuals: the solve's, or (half) half of them.
__host__ __device__ inline Geom residual_geom(Geom G, bool half) {
  if (half) {
    if (G.TX >= G.TY)
      G.TX = (G.TX + 1) / 2;
    else
      G.TY = (G.TY + 1) / 2;
    G.tilesX = (G.Nx + G.TX - 1) / G.TX;
    G.tilesY = (G.Ny + G.TY - 1) / G.TY;
  }
  return G;
}

template <int N>
inline size_t mixed_smem_bytes(const Geom& G, int Lmax, int kind, bool pow2, bool half) {
  const int TY = G.TY, TX = G.TX;
  const Geom R = residual_geom(G, half);
  size_t t = fx_apply_bytes<N>(R.TY, R.TX);
  const size_t w = cg_tile_values<df, N>(TY, TX) * 8, l = pc_line_bytes<float, N>(kind, Lmax, pow2);
  t = t > w ? t : w;
  return (kind == kPrecondTwoLevel ? align16(sizeof(float) * N * N * N * N) : 0) + align16(t > l ? t : l);
}

// One float64 residual pass: r = b - Ahat y (y staged with halo; pass 0: y = y0), rf =
// float(r), inner residual = rf, e = 0.  Accumulates this block's r.r and b.b.
template <int N>
__device__ __forceinline__ void mixed_residual(const Ops2D<double, N>& Cd, const Geom& G, const MixedArgs& A,
                                               double wbar, bool from_x0, SolveCtx<double>& X, double& rr,
                                               double& bb, double& yy) {
  constexpr int NN = N * N;
  if (from_x0 && A.axa) {  // Ahat y0 from the recycled products: a pointwise pass
    const size_t ndof = (size_t)G.Nx * G.Ny * NN;
    for (size_t g = (size_t)X.vrank * blockDim.x + threadIdx.x; g < ndof; g += (size_t)X.vsize * blockDim.x) {
      const int k = int(unsigned(g) % NN);
      double y0 = 0.0, ax = 0.0;
      if (A.xa) {
        y0 = A.ca * A.xa[g];
        ax = A.ca * __ldcg(A.axa + g);
      }
      if (A.xb) {
        y0 = fma(A.cb, A.xb[g], y0);
        ax = fma(A.cb, __ldcg(A.axb + g), ax);
      }
      __stcg(A.y + g, y0);
      if (A.ay) __stcg(A.ay + g, ax);
      const double b = Cd.sw[k] * (A.omega[g] - wbar);
      const double r = b - ax;
      const float r32 = float(r);
      __stcg(A.rf + g, r32);
      __stcg(A.v.r + g, r32);
      __stcg(A.v.y + g, 0.0f);
      rr = fma(r, r, rr);
      bb = fma(b, b, bb);
      yy = fma(y0, y0, yy);
    }
    return;
  }
  const int ntiles = G.tilesX * G.tilesY;
  for (int t = X.vrank; t < ntiles; t += X.vsize) {
    solve_apply<double, N>(
        Cd, G, t, X,
        [&](size_t g, int k, bool interior) {
          if (!from_x0) return __ldcg(A.y + g);
          double v = 0.0;
          if (A.xa) v = A.ca * A.xa[g];
          if (A.xb) v = fma(A.cb, A.xb[g], v);
          if (A.x_unscaled) v *= Cd.sw[k];
          if (interior) __stcg(A.y + g, v);
          return v;
        },
        [&](size_t g) { return __ldcg(A.y + g); },
        [&](size_t g, int k, double yv, double qv) {
          const double b = Cd.sw[k] * (A.omega[g] - wbar);
          const double r = b - qv;
          if (A.ay) __stcg(A.ay + g, qv);
          const float r32 = float(r);
          __stcg(A.rf + g, r32);
          __stcg(A.v.r + g, r32);
          __stcg(A.v.y + g, 0.0f);
          rr = fma(r, r, rr);
          bb = fma(b, b, bb);
          yy = fma(yv, yv, yy);
        });
  }
}

// The whole mixed-precision solve on the (virtual) grid of Xf / Xd (float context with the
// staged block matrix, double context over the same region; see mixed_cg_kernel).
template <int N>
__device__ __forceinline__ void mixed_solve(const Ops2D<double, N>& Cd, const Ops2D<float, N>& Cf,
                                            const OpsK<df, N>& Ck, const Geom& G, const MixedArgs& A,
                                            SolveCtx<float>& Xf, SolveCtx<double>& Xd) {
  constexpr int NN = N * N;
  const bool pc = A.precond != kPrecondJacobi;
  // the double-float apply stages its tiles in the float64 buffers
  Xf.wU = reinterpret_cast<df*>(Xd.sU);
  Xf.wXR = reinterpret_cast<df*>(Xd.tXR);
  Xf.wXL = reinterpret_cast<df*>(Xd.tXL);
  Xf.wYR = reinterpret_cast<df*>(Xd.tYR);
  Xf.wYL = reinterpret_cast<df*>(Xd.tYL);
  Xf.kdf = A.precise_apply == 1 ? &Ck : nullptr;
  Xf.sync = A.sync;
  Xf.part = A.partf;
  Xf.phase = 0;
  Xd.sync = A.sync;
  Xd.part = A.partd;
  Xd.phase = 0;
  Xd.ks = A.ks;
  Xf.tbase = Xd.tbase = read_ticket<float>(A.sync);  // before the first barrier
  const size_t ndof = (size_t)G.Nx * G.Ny * NN;
  const size_t stride = (size_t)Xd.vsize * blockDim.x;
  int flags = 0, sweeps = 0;
  long long inner = 0;
  double rr = 0.0, bb = 0.0, wbar = 0.0, rr_prev = -1.0;
  for (int mp = 0; mp < (A.keep_mean ? 0 : 2); ++mp) {  // two-pass W-mean, as in cg_kernel
    double s = 0.0;
    strided_pass<4>((size_t)Xd.vrank * blockDim.x + threadIdx.x, ndof, stride,
                    [&](size_t i) { return A.omega[i]; },
                    [&](size_t i, double v) { s = fma(Cd.wq[unsigned(i) % NN], v - wbar, s); });
    double m = 0.0;
    if (!reduce_all(Xd, s, m)) {
      flags |= kFlagTimeout;
      goto finish;
    }
    wbar += m / A.sumW;
  }
  for (int pass = 0;; ++pass) {
    // float64 residual of the current iterate (pass 0: of the initial guess)
    double yy = 0.0;
    {
      double r2 = 0.0, b2 = 0.0, y2 = 0.0;
      mixed_residual<N>(Cd, residual_geom(G, A.half), A, wbar, pass == 0, Xd, r2, b2, y2);
      if (!reduce_all3(Xd, r2, b2, y2, rr, bb, yy)) {
        flags |= kFlagTimeout;
        goto finish;
      }
    }
    if (bb == 0.0) {
      for (size_t i = (size_t)Xd.vrank * blockDim.x + threadIdx.x; i < ndof; i += stride) __stcg(A.y + i, 0.0);
      rr = 0.0;
      break;
    }
    if (Xd.vrank == 0 && threadIdx.x == 0 && pass < kRefineHistory) {
      A.status->hist_rr[pass] = rr / bb;
      A.status->hist_len = pass + 1;
    }
    if (rr <= A.tol2 * bb) break;
    // stagnation at the float64 rounding floor of y (see CgArgs::floor2): below it, and less
    // than a factor 4 below the previous sweep's residual
    if (rr <= A.floor2 * yy && rr_prev >= 0.0 && rr > 0.25 * rr_prev) break;
    // adaptive apply: a sweep after the second that gained less than a factor 100 in the
    // residual norm (1e-4 in r.r) switches the inner solves to the double-float apply (the
    // first sweep from a poor guess is limited by the float32 rounding of its large correction
    // instead)
    if (A.precise_apply == 2 && !Xf.kdf && pass >= 2 && rr > 1e-4 * rr_prev) Xf.kdf = &Ck;
    rr_prev = rr;
    if (sweeps >= A.max_sweeps) {
      flags |= kFlagNoconv;
      break;
    }
    // float32 inner (P)CG from e = 0 on the residual equation, to the relative tolerance
    // tol_in -- or to what is left to reach the outer tolerance (with a factor 1/2 of
    // margin), if that is looser: the last sweep then does only the iterations it needs
    const double tol_eff2 = fmax(A.tol_in2, 0.25 * A.tol2 * bb / rr);
    float rho_in = float(rr);
    const float rhob_in = rho_in;
    float rz_in = rho_in;
    if (pc && !pc_apply<float, N>(Cf, G, A.pc, A.v.r, Xf, rz_in)) {
      flags |= kFlagTimeout;
      goto finish;
    }
    int fin = 0;
    const int it_in = cg_iterate<float, N>(Cf, G, A.v, pc ? &A.pc : nullptr, RhsSource<float>{nullptr, A.rf, 0.0f},
                                           Xf, rho_in, rz_in, rhob_in, tol_eff2, A.maxit_in, 0, fin, 0);
    inner += it_in;
    if (Xd.vrank == 0 && threadIdx.x == 0 && pass < kRefineHistory) A.status->hist_it[pass] = it_in;
    if (fin & kFlagTimeout) {
      flags |= kFlagTimeout;
      goto finish;
    }
    // y += e
    struct Ye {
      double y;
      float e;
    };
    strided_pass<4>((size_t)Xd.vrank * blockDim.x + threadIdx.x, ndof, stride,
                    [&](size_t i) { return Ye{__ldcg(A.y + i), __ldcg(A.v.y + i)}; },
                    [&](size_t i, const Ye& v) { __stcg(A.y + i, v.y + double(v.e)); });
    if (!solve_barrier(Xd)) {
      flags |= kFlagTimeout;
      goto finish;
    }
    ++sweeps;
  }
  if (pc && !(flags & kFlagTimeout) && !project_mean<double, N>(Cd, G, A.y, A.sumW, Xd)) flags |= kFlagTimeout;
finish:
  if (A.psi_out && !(flags & kFlagTimeout)) {
    strided_pass<4>((size_t)Xd.vrank * blockDim.x + threadIdx.x, ndof, stride,
                    [&](size_t i) { return __ldcg(A.y + i); },
                    [&](size_t i, double v) { A.psi_out[i] = v * Cd.isw[unsigned(i) % NN]; });
  }
  if (Xd.vrank == 0 && threadIdx.x == 0) {
    SolveStatus* st = A.status;
    const int it = int(inner);
    st->total_iters += it;
    st->last_iters = it;
    st->max_iters = max(st->max_iters, it);
    st->last_flags = flags;
    st->flags |= flags;
    st->nsolves += 1;
    st->last_sweeps = sweeps;
    st->last_rho = rr;
    st->last_rhob = bb;
  }
}

template <int N, int MinB = 4>
__global__ void __launch_bounds__(kThreads, MinB) mixed_cg_kernel(const __grid_constant__ Ops2D<double, N> Cd,
                                                           const __grid_constant__ Ops2D<float, N> Cf,
                                                           const __grid_constant__ OpsK<df, N> Ck, const Geom G,
                                                           const __grid_constant__ MixedArgs A) {
  constexpr int NN = N * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double redd[112];
  __shared__ float redf[128];
  __shared__ BarrierState bs;
  if (threadIdx.x == 0) bs = BarrierState{0, 0};
  const bool pc = A.precond == kPrecondTwoLevel;  // the cell blocks are staged
  const int Lmax = max(G.Nx, G.Ny);
  const Ops2D<double, N>& Cds = stage_table(Cd, smem_raw);
  const Ops2D<float, N>& Cfs = stage_table(Cf, smem_raw + table_bytes<Ops2D<double, N>>());
  const OpsK<df, N>& Cks =
      stage_table(Ck, smem_raw + table_bytes<Ops2D<double, N>>() + table_bytes<Ops2D<float, N>>());
  unsigned char* smem = smem_raw + mixed_ops_bytes<N>();
  SolveCtx<float> Xf;
  init_ctx<float, N>(Xf, smem, G, A.pc.Bt, pc, Lmax);
  Xf.red = redf;
  Xf.bs = &bs;
  Xf.vrank = blockIdx.x;
  Xf.vsize = gridDim.x;
  SolveCtx<double> Xd;
  init_ctx<double, N>(Xd, smem + (pc ? align16(sizeof(float) * NN * NN) : 0), G, (const double*)nullptr, false, Lmax);
  Xd.red = redd;
  Xd.bs = &bs;
  Xd.vrank = blockIdx.x;
  Xd.vsize = gridDim.x;
  Xf.cluster = Xd.cluster = A.cluster;
  mixed_solve<N>(Cds, Cfs, Cks, G, A, Xf, Xd);
}

// =========================================================================================
// Batched persistent step: many independent simulations (different grids, n, viscosities)
// advance in one cooperative launch.  The blocks are split into groups; each group is a
// virtual grid (its own barrier, block ranks and partial sums) that runs whole AB3 steps --
// the RHS tile pass, the Poisson solve, the rotation of the state rings -- for the
// simulations queued on it, one after the other.  Groups run concurrently.
// =========================================================================================
struct BatchSim {
  int n, precision, precond;       // precision: 0 float64, else mixed
  int precise_apply;               // mixed: the inner solve applies Ahat in double-float
  int keep_mean;                   // homogeneous Dirichlet grid: no mean removed from omega
  Geom Gr, Gc;                     // tiles of the RHS and of the solve
  const void* ops_d;               // device copy of Ops2D<double, n>
  const void* ops_f;               // device copy of Ops2D<float, n>
  const void* ops_rhs;             // device copy of FxRhs<n> (fixed-point RHS)
  const void* ops_k;               // device copy of OpsK<df, n> (double-float CG operator)
  double* omega[2];
  double* psi[3];                  // sqrt(W) psi
  double* apsi[3];                 // Ahat psi of each slot, valid where apsi_ok (see dg_sim)
  int apsi_ok[3];
  double* R[4];                    // right-hand-side history
  int oc, p0, p1, p2, r1, r2, r3, rfree;  // ring indices, advanced by the kernel
  long long step;
  long long limit;                 // no batched step once step == limit (0: no limit)
  double D, dt, tol2, tol_in2, floor2;
  int maxit, max_sweeps, fixed_iters;
  double sumW;
  FxScale ks;
  // float64 solve
  double *r, *p0v, *p1v, *q, *part;
  // mixed solve
  float *rf, *fr, *fe, *fp0, *fp1, *fq, *partf;
  SolveStatus* status;
  PrecondArgs<double> pc;
  PrecondArgs<float> pcf;
};

struct BatchGroup {
  int first_block, nblocks;  // blocks [first_block, first_block + nblocks)
  int first, count;          // simulations order[first .. first + count)
  SyncState* sync;
};

struct BatchArgs {
  BatchSim* sims;
  const int* order;
  const BatchGroup* groups;
  int ngroups;
  int nsteps;
  int* error;                // first error flag of any group
};

// The arguments of a batched pass live in shared memory: as local variables of these functions they
// held the registers that the passes need (a stand-alone kernel reads them from the constant bank).
template <int N>
__device__ __noinline__ void batch_rhs(const BatchSim& S, const FxRhs<N>& F, int oc, int p0, int r1, int r2, int rfree,
                                       int vrank, int vsize, unsigned char* smem) {
  __shared__ RhsArgs A;
  __shared__ Geom G;
  if (threadIdx.x == 0) {
    RhsArgs a{};
    a.psi = S.psi[p0];
    a.omega_in = S.omega[oc];
    a.omega_base = S.omega[oc];
    a.omega_out = S.omega[oc ^ 1];
    a.R_out = S.R[rfree];
    a.hist[0] = S.R[r1];
    a.hist[1] = S.R[r2];
    a.c_new = 23.0 / 12.0;
    a.c_hist[0] = -16.0 / 12.0;
    a.c_hist[1] = 5.0 / 12.0;
    a.nhist = 2;
    a.dt = S.dt;
    a.visc = S.D;
    a.psi_scaled = 1;
    A = a;
    G = S.Gr;
  }
  __syncthreads();
  const int nt = G.tilesX * G.tilesY;
  const Ops2D<double, N>& C = *static_cast<const Ops2D<double, N>*>(S.ops_d);
  if (G.bc)
    for (int t = vrank; t < nt; t += vsize) rhs_tile<N, true>(F, C, G, A, t, smem);
  else
    for (int t = vrank; t < nt; t += vsize) rhs_tile<N, false>(F, C, G, A, t, smem);
}

template <int N, bool Fxs>
__device__ __noinline__ void batch_solve(const Ops2D<double, N>& C, const Geom& G, const CgArgs<double>& A,
                                         unsigned char* smem, double* red, BarrierState* bs, int vrank, int vsize) {
  SolveCtx<double> X;
  init_ctx<double, N>(X, smem, G, A.pc.Bt, A.precond == kPrecondTwoLevel, max(G.Nx, G.Ny));
  X.red = red;
  X.bs = bs;
  X.vrank = vrank;
  X.vsize = vsize;
  cg_solve<double, N, double, Fxs>(C, G, A, X);
}

template <int N>
__device__ __noinline__ void batch_mixed(const Ops2D<double, N>& Cd, const Ops2D<float, N>& Cf, const OpsK<df, N>& Ck,
                                         const Geom& G, const MixedArgs& A, unsigned char* smem, double* redd,
                                         float* redf, BarrierState* bs, int vrank, int vsize) {
  const bool pc = A.precond == kPrecondTwoLevel;  // the cell blocks are staged
  const int Lmax = max(G.Nx, G.Ny);
  SolveCtx<float> Xf;
  init_ctx<float, N>(Xf, smem, G, A.pc.Bt, pc, Lmax);
  Xf.red = redf;
  Xf.bs = bs;
  Xf.vrank = vrank;
  Xf.vsize = vsize;
  SolveCtx<double> Xd;
  init_ctx<double, N>(Xd, smem + (pc ? align16(sizeof(float) * N * N * N * N) : 0), G, (const double*)nullptr, false, Lmax);
  Xd.red = redd;
  Xd.bs = bs;
  Xd.vrank = vrank;
  Xd.vsize = vsize;
  mixed_solve<N>(Cd, Cf, Ck, G, A, Xf, Xd);
}

// One AB3 step of simulation S on a group.  Returns false after a barrier timeout.
// Shared-memory tables of a batched step: the float64 operators (the fixed-point tables during
// the RHS pass), float32, double-float CG operator.
template <int N>
__host__ __device__ constexpr size_t batch_ops_bytes() {
  static_assert(sizeof(FxRhs<N>) <= sizeof(Ops2D<double, N>), "table sizes");
  return table_bytes<Ops2D<double, N>>() + table_bytes<Ops2D<float, N>>() + table_bytes<OpsK<df, N>>();
}

template <int N>
__device__ __forceinline__ bool batch_step_body(BatchSim* Sp, const BatchGroup& grp, int vrank, unsigned char* smem_all,
                                           double* redd, float* redf, BarrierState* bs) {
  __shared__ CgArgs<double> s_cg;
  __shared__ MixedArgs s_mixed;
  __shared__ Geom s_g;
  const BatchSim& S = *Sp;
  // a simulation that has reached its step limit sits the step out (every block of the
  // group reads the same step index: it was written before the group's last barrier)
  if (S.limit > 0 && __ldcg(&Sp->step) >= S.limit) return true;
  const int oc = __ldcg(&Sp->oc), p0 = __ldcg(&Sp->p0), p1 = __ldcg(&Sp->p1), p2 = __ldcg(&Sp->p2);
  const int r1 = __ldcg(&Sp->r1), r2 = __ldcg(&Sp->r2), r3 = __ldcg(&Sp->r3), rfree = __ldcg(&Sp->rfree);
  // this simulation's operator tables, staged in shared memory (the previous step's last
  // barrier has synchronised the block)
  unsigned char* smem = smem_all + batch_ops_bytes<N>();
  const FxRhs<N>& Fr = stage_table(*static_cast<const FxRhs<N>*>(S.ops_rhs), smem_all);
  batch_rhs<N>(S, Fr, oc, p0, r1, r2, rfree, vrank, grp.nblocks, smem);
  if (!grid_barrier(grp.sync, bs, grp.nblocks)) return false;
  // the solve's tables (the barrier has synchronised the block: the RHS table is no longer read)
  const Ops2D<double, N>& Cd = stage_table(*static_cast<const Ops2D<double, N>*>(S.ops_d), smem_all);
  // the initial residual from the kept operator products (as in the single-simulation stepper)
  const bool rec = S.fixed_iters == 0 && __ldcg(&Sp->apsi_ok[p0]) && __ldcg(&Sp->apsi_ok[p1]);
  const bool fxs = fx_spectral_solve(S.pc, S.precond, S.fixed_iters);
  if (S.precision == 0) {
    CgArgs<double> A{};
    A.omega = S.omega[oc ^ 1];
    A.xa = S.psi[p0];
    A.xb = S.psi[p1];
    A.ca = 2.0;
    A.cb = -1.0;
    if (rec) {
      A.axa = S.apsi[p0];
      A.axb = S.apsi[p1];
    }
    if (S.fixed_iters == 0) A.ay = S.apsi[p2];
    A.v = CgVectors<double>{S.psi[p2], S.r, S.p0v, S.p1v, S.q};
    A.precond = S.precond;
    A.pc = S.pc;
    A.part = S.part;
    A.sync = grp.sync;
    A.status = S.status;
    A.tol2 = S.tol2;
    A.floor2 = S.floor2;
    A.keep_mean = S.keep_mean;
    A.maxit = S.fixed_iters > 0 ? max(S.maxit, S.fixed_iters) : S.maxit;
    A.fixed_iters = S.fixed_iters;
    A.sumW = S.sumW;
    A.ks = S.ks;
    if (threadIdx.x == 0) {
      s_cg = A;
      s_g = S.Gc;
    }
    __syncthreads();
    if (fxs)
      batch_solve<N, true>(Cd, s_g, s_cg, smem, redd, bs, vrank, grp.nblocks);
    else
      batch_solve<N, false>(Cd, s_g, s_cg, smem, redd, bs, vrank, grp.nblocks);
  } else {
    MixedArgs A{};
    A.omega = S.omega[oc ^ 1];
    A.xa = S.psi[p0];
    A.xb = S.psi[p1];
    A.ca = 2.0;
    A.cb = -1.0;
    if (rec) {
      A.axa = S.apsi[p0];
      A.axb = S.apsi[p1];
    }
    if (S.fixed_iters == 0) A.ay = S.apsi[p2];
    A.y = S.psi[p2];
    A.rf = S.rf;
    A.v = CgVectors<float>{S.fe, S.fr, S.fp0, S.fp1, S.fq};
    A.precond = S.precond;
    A.pc = S.pcf;
    A.partd = S.part;
    A.partf = S.partf;
    A.sync = grp.sync;
    A.status = S.status;
    A.tol2 = S.tol2;
    A.floor2 = S.floor2;
    A.keep_mean = S.keep_mean;
    A.tol_in2 = S.tol_in2;
    A.max_sweeps = S.max_sweeps;
    A.maxit_in = S.maxit;
    A.sumW = S.sumW;
    A.ks = S.ks;
    A.precise_apply = S.precise_apply;
    const Ops2D<float, N>& Cf =
        stage_table(*static_cast<const Ops2D<float, N>*>(S.ops_f), smem_all + table_bytes<Ops2D<double, N>>());
    const OpsK<df, N>& Ck = stage_table(*static_cast<const OpsK<df, N>*>(S.ops_k),
                                        smem_all + table_bytes<Ops2D<double, N>>() + table_bytes<Ops2D<float, N>>());
    if (threadIdx.x == 0) {
      s_mixed = A;
      s_g = S.Gc;
    }
    __syncthreads();
    batch_mixed<N>(Cd, Cf, Ck, s_g, s_mixed, smem, redd, redf, bs, vrank, grp.nblocks);
  }
  // every block has finished the solve before the rings move
  if (!grid_barrier(grp.sync, bs, grp.nblocks)) return false;
  if (vrank == 0 && threadIdx.x == 0) {
    Sp->apsi_ok[p2] = S.fixed_iters == 0 ? 1 : 0;
    Sp->oc = oc ^ 1;
    Sp->p0 = p2;
    Sp->p1 = p0;
    Sp->p2 = p1;
    Sp->r1 = rfree;
    Sp->r2 = r1;
    Sp->r3 = r2;
    Sp->rfree = r3;
    Sp->step = S.step + 1;
    __threadfence();
  }
  return grid_barrier(grp.sync, bs, grp.nblocks);
}



// =========================================================================================
// Invariants: partial sums of W omega, W psi omega, W omega^2 per block, then one block
// adds the partials in a fixed order.
// =========================================================================================
template <int N>
struct NodeWeights {
  double w[N * N];    // W_ab
  double sw[N * N];   // sqrt(W_ab)
  double isw[N * N];  // 1 / sqrt(W_ab)
};

template <int N>
__global__ void __launch_bounds__(kThreads) invariants_partial_kernel(const __grid_constant__ NodeWeights<N> W,
                                                                     const double* __restrict__ psi,
                                                                     const double* __restrict__ omega,
                                                                     size_t ndof, int psi_scaled,
                                                                     double* __restrict__ part) {
  constexpr int NN = N * N;
  __shared__ double red[32];
  double v = 0.0, e = 0.0, o = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndof; i += (size_t)gridDim.x * blockDim.x) {
    const int k = int(unsigned(i) % NN);
    const double w = omega[i];
    const double p = psi_scaled ? psi[i] * W.isw[k] : psi[i];
    const double ww = W.w[k] * w;
    v += ww;
    e = fma(ww, p, e);
    o = fma(ww, w, o);
  }
  v = block_sum(v, red);
  if (threadIdx.x == 0) part[3 * blockIdx.x] = v;
  e = block_sum(e, red);
  if (threadIdx.x == 0) part[3 * blockIdx.x + 1] = e;
  o = block_sum(o, red);
  if (threadIdx.x == 0) part[3 * blockIdx.x + 2] = o;
}


// ---- small elementwise kernels ----------------------------------------------------------

// y[i] = x[i] * s[i % NN]   (psi <-> sqrt(W) psi)
template <int N>
__global__ void scale_nodes_kernel(const __grid_constant__ NodeWeights<N> W, const double* __restrict__ x,
                                   double* __restrict__ y, size_t ndof, int inverse) {
  constexpr int NN = N * N;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndof; i += (size_t)gridDim.x * blockDim.x) {
    const int k = int(unsigned(i) % NN);
    y[i] = x[i] * (inverse ? W.isw[k] : W.sw[k]);
  }
}


}  // namespace dgk
