// Fixed-point arithmetic on the integer pipe for the float64 operators.
//
// What bounds the float64 kernels here is the float64 pipe: measured 1.9 fused multiply-adds
// per clock and SM, against 50-64 32 x 32 -> 64-bit integer multiply-adds.  A tile's linear
// operators and products therefore run on 64-bit fixed-point numbers that share one power of
// two per field and tile:
//
//   value u = X 2^e,  |X| <= 2^60 for staged fields (7 bits more than a float64 significand,
//   counted from the tile's largest value), |X| <= 2^61 for results,
//   X = h 2^30 + l  with a signed 32-bit h and |l| <= 2^29, stored as the pair (h, l).
//
// A coefficient c = C 2^-60 2^e' is split the same way; a dot product sums the partial
// products C_h X_h (weight 2^60) and C_h X_l + C_l X_h (weight 2^30) in two 64-bit
// accumulators -- three integer multiply-adds per term, no rounding inside the sum -- and is
// rounded once at the end (fx_round: half away from zero, so that f(-x) = -f(x) exactly).
// The dropped C_l X_l contribute at most 2^-2 units per term.  With rows scaled so that
// sum |c_j| <= 1, a result of n + 2 terms is off by at most 1 + (n + 2) / 4 units of 2^-60 of
// (largest input x row sum), where a float64 evaluation commits up to (n + 2) 2^-53 of it.
//
// Bounds that keep the accumulators within 63 bits: |X| <= 2^61, row sum |C| <= 2^60, at most
// 7 terms: |acc1| <= 2^30 2^31, |acc0| <= 7 2^29 2^31 + 2^30 2^29 < 2^63.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace dgk {

struct fx {
  int h, l;
};

struct Cfx {
  fx re, im;
};

struct FxAcc {
  long long a1 = 0, a0 = 0;
};

__host__ __device__ __forceinline__ void fx_mac(FxAcc& s, fx c, fx x) {
  s.a1 += (long long)c.h * x.h;
  s.a0 += (long long)c.h * x.l;
  s.a0 += (long long)c.l * x.h;
}

// a1 + a0 / 2^30, rounded half away from zero.
__host__ __device__ __forceinline__ long long fx_round(FxAcc s) {
  return s.a1 + ((s.a0 + (1ll << 29) + (s.a0 >> 63)) >> 30);
}

// The stored form of a result, |y| <= 2^61.
__host__ __device__ __forceinline__ fx fx_split(long long y) {
  const long long t = y + (1ll << 29);
  return fx{int(t >> 30), int(unsigned(t) & 0x3fffffffu) - (1 << 29)};
}

__host__ __device__ __forceinline__ long long fx_join(fx v) { return ((long long)v.h << 30) + v.l; }

__host__ __device__ __forceinline__ fx fx_neg(fx v) { return fx{-v.h, -v.l}; }
__host__ __device__ __forceinline__ fx fx_and(fx v, int mask) { return fx{v.h & mask, v.l & mask}; }

// (a b - c d) / 2^60, rounded.  |a|, |c| <= 2^60, |b|, |d| <= 2^60.
__host__ __device__ __forceinline__ long long fx_prod_diff(fx a, fx b, fx c, fx d) {
  FxAcc s;
  fx_mac(s, a, b);
  fx_mac(s, fx_neg(c), d);
  return fx_round(s);
}

// float64 (bit pattern, finite) to units of 2^(emax - 1082), emax >= 1 the biased exponent of the
// tile's largest value: |X| < 2^60.  Bits below the unit are cut off (toward zero).
__host__ __device__ __forceinline__ long long fx_from_bits(unsigned hi, unsigned lo, int emax) {
  const int eb = int((hi >> 20) & 0x7ffu);
  unsigned long long m = (unsigned long long)((hi & 0xfffffu) | (eb ? 0x100000u : 0u)) << 32 | lo;
  const int d = emax - (eb ? eb : 1);
  m = (m << 7) >> (d < 63 ? d : 63);
  const long long x = (long long)m;
  return int(hi) < 0 ? -x : x;
}

// y 2^e as a float64, rounded to nearest (halves away from zero); the result is a normal number.
__host__ __device__ __forceinline__ double fx_to_double(long long y, int e = 0) {
  const long long s = y >> 63;
  unsigned long long v = (unsigned long long)((y ^ s) - s);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)v);
#else
  const int lz = v ? __builtin_clzll(v) : 64;
#endif
  if (v == 0) return 0.0;
  v = (v << lz);
  // the leading one adds to the exponent field, and a carry out of the rounding does too
  const unsigned long long r = (v >> 11) + ((v >> 10) & 1u);
  const unsigned long long bits = ((unsigned long long)(1085 - lz + e) << 52) + r + ((unsigned long long)s << 63);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double d;
  __builtin_memcpy(&d, &bits, 8);
  return d;
#endif
}

// 2^k as a float64, -1022 <= k <= 1023.
__host__ __device__ __forceinline__ double fx_pow2(int k) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((1023 + k) << 20, 0);
#else
  const unsigned long long bits = (unsigned long long)(1023 + k) << 52;
  double d;
  __builtin_memcpy(&d, &bits, 8);
  return d;
#endif
}

// A 1D operator (Op1D) on the reference cell in fixed point: coefficients times 2^(60 - e), so that
// every row's sum of magnitudes (the traces' own sums included) is below 2^60; the trace vectors r
// times 2^(60 - er) and s, sf times 2^(60 - es), the lifts a, af times 2^er and d times 2^es in
// return.  Mf, af, sf: the first cell of a line at a Dirichlet boundary.  The tables are functions
// of n alone (dg_fixed_tables.cuh) and are compiled in: their entries become immediate operands of
// the multiply-adds (as kernel parameters, the compiler kept a line's 90 words in registers across
// its loop and spilled them).
template <int N>
struct FxTable {
  int e, er, es;
  fx M[N][N];
  fx a[N], r[N], d[N], s[N];
  fx Mf[N][N];
  fx af[N], sf[N];
};

template <int N>
__device__ constexpr FxTable<N> fx_deriv();  // h d/dx with central fluxes
template <int N>
__device__ constexpr FxTable<N> fx_stiff();  // h^2 W^-1/2 A1 W^-1/2
template <int N>
__device__ constexpr FxTable<N> fx_lap();    // h^2 W^-1 A1

// One line of a 1D operator: y_i = sum_j M_ij u_j + a_i (r . u+) + d_i (s . u-).  own, right and
// left point at the first node of the line in the own cell and its neighbours, nodes `st` apart.
// out(i, y) receives the results.
template <int N, class Out>
__device__ __forceinline__ void fx_line_traced(const fx (&M)[N][N], const fx (&a)[N], const fx (&d)[N], const fx (&u)[N],
                                               fx tr, fx tl, Out&& out) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    FxAcc s;
    fx_mac(s, a[i], tr);
    fx_mac(s, d[i], tl);
#pragma unroll
    for (int j = 0; j < N; ++j) fx_mac(s, M[i][j], u[j]);
    out(i, fx_round(s));
  }
}

template <int N>
__device__ __forceinline__ fx fx_trace(const fx (&r)[N], const fx* u, int st) {
  FxAcc s;
#pragma unroll
  for (int j = 0; j < N; ++j) fx_mac(s, r[j], u[j * st]);
  return fx_split(fx_round(s));
}

template <int N>
__device__ __forceinline__ void fx_load(fx (&u)[N], const fx* p, int st) {
#pragma unroll
  for (int j = 0; j < N; ++j) u[j] = p[j * st];
}

// One line of a 1D operator: own points at the first node of the line, nodes `st` apart, the
// neighbour cells `dc` apart.
template <int N, class Out>
__device__ __forceinline__ void fx_line(const FxTable<N>& O, const fx* own, int st, int dc, Out&& out) {
  fx u[N];
  fx_load<N>(u, own, st);
  fx_line_traced<N>(O.M, O.a, O.d, u, fx_trace<N>(O.r, own + dc, st), fx_trace<N>(O.s, own - dc, st), out);
}

// The central derivative of a cell at a Dirichlet boundary: the flux on a boundary face is 0, as if
// the ghost cell had the negated trace of the boundary cell on that face.  first / last: the cell
// lies at the lower / upper end of its line.
template <int N, class Out>
__device__ __forceinline__ void fx_line_bounded(const FxTable<N>& O, const fx* own, int st, int dc, bool first,
                                                bool last, Out&& out) {
  fx u[N];
  fx_load<N>(u, own, st);
  const fx tr = last ? fx_neg(fx_trace<N>(O.s, own, st)) : fx_trace<N>(O.r, own + dc, st);
  const fx tl = first ? fx_neg(fx_trace<N>(O.r, own, st)) : fx_trace<N>(O.s, own - dc, st);
  fx_line_traced<N>(O.M, O.a, O.d, u, tr, tl, out);
}

// One line of an LDG operator on a Dirichlet grid (zeros outside).  pos: the cell's index along the
// line: the first cell has its own block and lift, the second sees the first through its own trace
// vector.
template <int N, class Out>
__device__ __forceinline__ void fx_ldg_bounded(const FxTable<N>& O, const fx* own, int st, int dc, int pos, Out&& out) {
  fx u[N];
  fx_load<N>(u, own, st);
  const fx tr = fx_trace<N>(O.r, own + dc, st);
  const fx tl = pos == 1 ? fx_trace<N>(O.sf, own - dc, st) : fx_trace<N>(O.s, own - dc, st);
  if (pos == 0)
    fx_line_traced<N>(O.Mf, O.af, O.d, u, tr, tl, out);
  else
    fx_line_traced<N>(O.M, O.a, O.d, u, tr, tl, out);
}

// The exponent word that orders values by magnitude for a tile's maximum: the high word without
// its sign (0 only for zeros; a value below 2^-1042 counts as the smallest non-zero word).
__device__ __forceinline__ unsigned fx_mag(double v) {
  const unsigned hi = unsigned(__double2hiint(v)) & 0x7fffffffu;
  return hi ? hi : (__double2loint(v) ? 1u : 0u);
}

}  // namespace dgk
