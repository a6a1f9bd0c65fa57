// Operator kernels on Kuhn meshes that form each row of A x in one thread, from
// the lattice neighbours of its dof: no scatter, no dof maps, no zero-fill, and
// the Chebyshev update of the row in the same launch.
//
// Every Kuhn tet is a path of three axis-parallel edges and its geometric factor
// is c M (one c = kappa h / w per tet, see Level), which is diagonal in the
// directions of that path: the bilinear form of Section 2, Eq. 4 on a tet is c
// times the integral of (du/dx)^2 + (du/dy)^2 + (du/dz)^2, each axis taken along
// the tet's own edge of that axis.
//
// P1 (any coefficient): du/da is the difference along that edge, so A is the
// graph Laplacian of the axis edges with the weight of an edge the sum of c over
// its (up to six) tets: seven entries per row.
//
// P2 with one coefficient on the level: the rows are eight constant stencils of
// small integers times 8 c, one per parity class of the dof lattice.
//
// x is read as 0 on and outside the boundary.  An interior row only couples to
// points of tets that exist, so edges of the domain need no special case.
#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>
#include <utility>

#include "fe_fixed.cuh"
#include "fe_internal.cuh"
#include "fe_kuhn.h"

namespace {

using namespace fe_fixed;

inline int ceil_div(long long a, int b) { return (int)((a + b - 1) / b); }

// What a kernel does with its row y_i of A x.
enum Epilogue { EPI_APPLY = 0, EPI_CHEB = 1, EPI_RESIDUAL = 2 };

template <typename T>
struct Rows {
  const T* x;     // the operator's input (also the iterate that a Chebyshev step updates)
  T* out;         // APPLY: y; CHEB: the new iterate (another vector than x); RESIDUAL: b - y
  const T* b;     // CHEB, RESIDUAL: right-hand side
  const T* din;   // CHEB: the previous direction (null: c1 = 0)
  T* dout;        // CHEB: the new direction (null: not stored)
  const T* dinv;  // CHEB on P1 with a coefficient per cell: inverse diagonal
  T c1, c2;
  T wd[8];        // CHEB with one coefficient: c2 / diagonal per parity code (P1: wd[0])
};

// The vectors that a row needs besides y, loaded before the row is formed.
template <int EPI, typename T>
struct RowIn {
  T b = T(0), d = T(0), x = T(0);
  __device__ __forceinline__ RowIn() {}
  __device__ __forceinline__ RowIn(const Rows<T>& R, int i) {
    if constexpr (EPI != EPI_APPLY) b = __ldg(R.b + i);
    if constexpr (EPI == EPI_CHEB) {
      if (R.din) d = R.din[i];
      x = __ldg(R.x + i);
    }
  }
};

__device__ __forceinline__ double fma_t(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// By the exponent field (a comparison would go to the FP64 pipe).
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7FF00000) == 0x7FF00000; }
__device__ __forceinline__ bool not_finite(float v) { return (__float_as_int(v) & 0x7F800000) == 0x7F800000; }

// Row y_i = s v; residual: b - y; Chebyshev: d = c1 d + w (b - y), x += d with w = c2 / A_ii.
// FP64 operations are scarce (2 per clock and SM), so the scaling of y and the
// diagonal are folded: 4 of them per row with a previous direction.
template <int EPI, typename T>
__device__ __forceinline__ void finish_row(const Rows<T>& R, const RowIn<EPI, T>& in, int i, T v, T s, T w) {
  if constexpr (EPI == EPI_APPLY) {
    R.out[i] = v * s;
  } else if constexpr (EPI == EPI_RESIDUAL) {
    R.out[i] = fma_t(-v, s, in.b);
  } else {
    const T r = fma_t(-v, s, in.b);
    const T dn = R.din ? fma_t(w, r, R.c1 * in.d) : w * r;
    if (R.dout) R.dout[i] = dn;
    R.out[i] = in.x + dn;
  }
}
// A Dirichlet row: y = x.
template <int EPI, typename T>
__device__ __forceinline__ void identity_row(const Rows<T>& R, int i) {
  const RowIn<EPI, T> in(R, i);
  finish_row<EPI>(R, in, i, R.x[i], T(1), R.c2);
}

// ------------------------------------------------------------------- P1 ---
// One thread per vertex: y = D x - sum over the six axis edges of w x, with D
// the diagonal and w the weight of the edge (stored at its lower end; CONST:
// one coefficient, w = 6 c and D = 36 c).  FP64 issues 2 operations per clock
// and SM, so the row is kept at 7 of them (differences would take 12): bound by
// the FP64 pipe with a coefficient per edge, else by memory.
constexpr int kP1Block = 256;

// The row from sixteenths of the values (a call, so that its operations are not issued with every row: 112^3 V-cycle 374
// against 253 us).
template <typename T>
__device__ __noinline__ T p1_sixteenth(T xi, T xl, T xr, T yl, T yr, T zl, T zr) {
  const T q = T(0.0625);
  return fma_t(6 * q, xi, -(((q * xl + q * xr) + (q * yl + q * yr)) + (q * zl + q * zr)));
}

template <typename T, bool CONST, int EPI>
__global__ void __launch_bounds__(kP1Block) k_flux1(int N, int n, const T* __restrict__ w, T c, Rows<T> R) {
  const int i = blockIdx.x * kP1Block + threadIdx.x;
  if (i >= n) return;
  const int n1 = N + 1, sz = n1 * n1;
  const int X = i % n1, q = i / n1, Y = q % n1, Z = q / n1;
  if (X == 0 || Y == 0 || Z == 0 || X == N || Y == N || Z == N) {
    identity_row<EPI>(R, i);
    return;
  }
  const RowIn<EPI, T> in(R, i);
  const T* __restrict__ x = R.x;
  const T xi = x[i];
  // a neighbour on the boundary counts as 0
  const T xl = X > 1 ? x[i - 1] : T(0), xr = X < N - 1 ? x[i + 1] : T(0);
  const T yl = Y > 1 ? x[i - n1] : T(0), yr = Y < N - 1 ? x[i + n1] : T(0);
  const T zl = Z > 1 ? x[i - sz] : T(0), zr = Z < N - 1 ? x[i + sz] : T(0);
  if constexpr (CONST) {
    T v = fma_t(T(6), xi, -(((xl + xr) + (yl + yr)) + (zl + zr))), unit = c;
    if (not_finite(v)) {  // values close to the end of the range
      v = p1_sixteenth(xi, xl, xr, yl, yr, zl, zr);
      unit *= T(16);
    }
    finish_row<EPI>(R, in, i, v, unit, R.wd[0]);
  } else {
    const T* wx = w;
    const T* wy = w + n;
    const T* wz = w + 2 * (size_t)n;
    T y = w[3 * (size_t)n + i] * xi;
    y = fma_t(-wx[i - 1], xl, y);
    y = fma_t(-wx[i], xr, y);
    y = fma_t(-wy[i - n1], yl, y);
    y = fma_t(-wy[i], yr, y);
    y = fma_t(-wz[i - sz], zl, y);
    y = fma_t(-wz[i], zr, y);
    finish_row<EPI>(R, in, i, y, T(1), EPI == EPI_CHEB ? R.c2 * R.dinv[i] : T(0));
  }
}

// Edge weights from the coefficients c of the cells: the edge of axis a that
// starts at vertex v belongs to a ring of six tets; ring tet f is Kuhn type
// ring_type of the cube at v + ring_b(f) e_b + ring_c(f) e_c (b < c the other axes).
__host__ __device__ constexpr int ring_type(int axis, int f) {
  constexpr int t[3][6] = {{0, 1, 2, 5, 3, 4}, {2, 3, 0, 4, 1, 5}, {4, 5, 1, 2, 0, 3}};
  return t[axis][f];
}
__host__ __device__ constexpr int ring_b(int f) { return f >= 2 && f <= 4 ? -1 : 0; }  // offset along b
__host__ __device__ constexpr int ring_c(int f) { return f >= 3 ? -1 : 0; }            // offset along c

__global__ void k_edge_weights(int N, int n, const double* __restrict__ geo22, double* __restrict__ w64,
                               float* __restrict__ w32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int n1 = N + 1;
  const int p[3] = {i % n1, (i / n1) % n1, i / (n1 * n1)};
  // weight of the edge of `axis` starting at vertex v
  auto weight = [&](int axis, int vx, int vy, int vz) {
    const int v[3] = {vx, vy, vz};
    if (v[axis] < 0 || v[axis] >= N) return 0.0;
    const int b = axis == 0 ? 1 : 0, c = axis == 2 ? 1 : 2;
    double s = 0.0;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      int q[3];
      q[axis] = v[axis];
      q[b] = v[b] + ring_b(f);
      q[c] = v[c] + ring_c(f);
      if (q[b] < 0 || q[b] >= N || q[c] < 0 || q[c] >= N) continue;
      s += geo22[6 * (q[0] + (size_t)N * (q[1] + (size_t)N * q[2])) + ring_type(axis, f)];
    }
    return s;
  };
  const double wx = weight(0, p[0], p[1], p[2]), wy = weight(1, p[0], p[1], p[2]), wz = weight(2, p[0], p[1], p[2]);
  const double dg = wx + wy + wz + weight(0, p[0] - 1, p[1], p[2]) + weight(1, p[0], p[1] - 1, p[2]) +
                    weight(2, p[0], p[1], p[2] - 1);
  const size_t m = n;
  w64[i] = wx;
  w64[m + i] = wy;
  w64[2 * m + i] = wz;
  w64[3 * m + i] = dg;
  w32[i] = (float)wx;
  w32[m + i] = (float)wy;
  w32[2 * m + i] = (float)wz;
  w32[3 * m + i] = (float)dg;
}

// ------------------------------------------- P2, one coefficient: stencils ---
// With one c on the level the rows of A are eight constant stencils of 19 to 51
// small integers times 8 c, one per parity
// class of the dof lattice; 23 entries per row on average, all in 58 lattice
// values around a vertex cell.  A block stages the values of TX x TY x KZ
// vertex cells and one layer around them in shared memory (asynchronous copies,
// all in flight at once) and each thread forms the eight rows of a cell.
//
// FP64: the staged values become two 30-bit integers hi 2^30 + lo of the tile's
// common scale (its largest exponent), a value and its mirror image (every
// stencil is symmetric) are added in 32 bits, the coefficient times that sum in
// 64 bits: every sum is exact (rows of |K| / 8 sum to at most 216 < 2^8), and a
// row is rounded once, by one int64 -> FP64 conversion and one multiplication.
// The FP64 pipe (2 operations per clock and SM) would need 23 operations per row,
// the element-by-element form on the FP32 pipes 453 instructions per dof, this
// form 233.  What the integers cut off a value is below 2^-59 of the tile's scale
// 2^E.  They form the rows whose |A| |x| is large enough that less than 2^-47 of
// it is lost (row_kept).  The others, where values of very different size meet, and
// the rows of tiles whose scale is near the ends of the FP64 range are formed
// separately, each from a scale of its own: a thread marks them, the block stages the
// tile once more, and its warps take 32 cells of one stencil in turn.  P2 64^3: 26.7
// us without such rows, as before they were looked for (128^3: 169 against 166, the
// headline solve 4.19 ms both), 33 with a single value in a vector of zeros, 119 to
// 132 where most rows of most tiles are such rows (values of 2^-60 .. 1 in every
// tile, exp(-200 r^2)); 24^3: 10.4, 23 and 39 us.  In FP64 the same rows took 185 us
// (64^3) and 48 (24^3), in windows of the next lower bits of the whole tile 120 and 74.
template <typename V>
struct RowSum;
template <>
struct RowSum<float> {
  static constexpr double unit = 8.0;  // sums of |k| / 8 leave FP32's range no sooner than the sums of an element
  float s = 0.0f;
  template <typename... A>
  __device__ __forceinline__ void add(int k, A... v) {
    s = __fmaf_rn((float)k * 0.125f, (v + ...), s);
  }
};
template <>
struct RowSum<double> {
  static constexpr double unit = 1.0;
  double s = 0.0;
  template <typename... A>
  __device__ __forceinline__ void add(int k, A... v) {
    s = __fma_rn((double)k, (v + ...), s);
  }
};
template <>
struct RowSum<Pair32> : PairSum {
  // |hi|, |lo| < 216 * 2^30: the sum as one int64, or in units of 64 where hi is large
  __device__ __forceinline__ bool fits() const { return (unsigned long long)(hi + (1ll << 32)) < (1ull << 33); }
  __device__ __forceinline__ double value(bool fits) const {
    return (double)(fits ? (long long)((unsigned long long)hi << 30) + lo
                         : (long long)((unsigned long long)hi << 24) + (lo >> 6));
  }
};

// The row of the lattice point of parity code CODE in units of 8 c; at(x, y, z):
// the value at that offset from the vertex of its cell, components in [-2, 2].
template <int CODE, typename V, typename At>
__device__ __forceinline__ RowSum<V> stencil_row(At at) {
  constexpr int X = CODE & 1, Y = (CODE >> 1) & 1, Z = CODE >> 2;
  RowSum<V> r;
  auto p = [&](int x, int y, int z) -> V { return at(X + x, Y + y, Z + z); };
  auto s = [&](int x, int y, int z) -> V { return p(x, y, z) + p(-x, -y, -z); };
  if constexpr (CODE == 0) {  // a vertex
    r.add(54, p(0, 0, 0));
    r.add(-14, s(1, 0, 0), s(0, 1, 0), s(0, 0, 1));
    r.add(3, s(2, 0, 0), s(0, 2, 0), s(0, 0, 2));
    r.add(-3, s(1, 1, 1), s(1, 1, 0), s(1, 0, 1), s(0, 1, 1));
    r.add(2, s(1, -1, 0), s(1, 0, -1), s(0, 1, -1));
    r.add(1, s(2, 1, 1), s(1, 2, 1), s(1, 1, 2), s(2, 1, 0), s(2, 0, 1), s(1, 2, 0), s(0, 2, 1), s(1, 0, 2),
          s(0, 1, 2), s(1, 1, -1), s(1, -1, 1), s(-1, 1, 1));
  } else if constexpr (CODE == 7) {  // on the cube's main diagonal
    r.add(48, p(0, 0, 0));
    r.add(-4, s(1, 0, 0), s(0, 1, 0), s(0, 0, 1), s(1, -1, 0), s(1, 0, -1), s(0, 1, -1));
    r.add(-3, s(1, 1, 1));
    r.add(1, s(1, 1, -1), s(1, -1, 1), s(-1, 1, 1));
  } else if constexpr (X + Y + Z == 1) {  // on an axis edge a
    auto t = [&](int a, int b, int c) -> V {
      if constexpr (CODE == 1) return s(a, b, c);
      if constexpr (CODE == 2) return s(b, a, c);
      if constexpr (CODE == 4) return s(b, c, a);
    };
    r.add(56, p(0, 0, 0));
    r.add(-14, t(1, 0, 0));
    r.add(-6, t(0, 1, 0), t(0, 0, 1));
    r.add(-4, t(0, 1, -1));
    r.add(4, t(1, 1, 1));
    r.add(-2, t(1, 1, 2), t(1, 2, 1));
    r.add(1, t(1, 0, 2), t(1, 2, 0));
  } else {  // on a face diagonal, n normal to the face
    auto t = [&](int a, int b, int n) -> V {
      if constexpr (CODE == 3) return s(a, b, n);
      if constexpr (CODE == 5) return s(a, n, b);
      if constexpr (CODE == 6) return s(n, a, b);
    };
    r.add(48, p(0, 0, 0));
    r.add(-6, t(1, 0, 0), t(0, 1, 0), t(1, 0, 1), t(0, 1, 1));
    r.add(-4, t(0, 0, 1));
    r.add(4, t(1, 1, 1));
    r.add(-3, t(1, 1, 0));
    r.add(2, t(1, -1, 0));
    r.add(1, t(1, 1, 2));
  }
  return r;
}

// f(code) for the eight parity codes as constants
template <typename F>
__device__ __forceinline__ void for_codes(F&& f) {
  f(std::integral_constant<int, 0>{});
  f(std::integral_constant<int, 1>{});
  f(std::integral_constant<int, 2>{});
  f(std::integral_constant<int, 3>{});
  f(std::integral_constant<int, 4>{});
  f(std::integral_constant<int, 5>{});
  f(std::integral_constant<int, 6>{});
  f(std::integral_constant<int, 7>{});
}

// The coefficient (in units of 8 c) of the lattice point at offset (ox, oy, oz)
// from the vertex of a cell in the row of the cell's point of parity code CODE:
// the integer element matrices of the tets that hold both, summed.
__host__ __device__ constexpr int stencil_coef(int code, int ox, int oy, int oz) {
  const int p[3] = {code & 1, (code >> 1) & 1, code >> 2}, o[3] = {ox, oy, oz};
  int sum = 0;
  for (int cube = 0; cube < 8; ++cube) {
    int a[3] = {0, 0, 0}, b[3] = {0, 0, 0};  // both points in the cube's lattice [0, 2]^3
    bool in = true;
    for (int d = 0; d < 3; ++d) {
      const int c = (cube >> d & 1) ? -2 : 0;
      a[d] = p[d] - c;
      b[d] = o[d] - c;
      in = in && a[d] <= 2 && b[d] >= 0 && b[d] <= 2;
    }
    if (!in) continue;
    const int la = a[0] + 3 * a[1] + 9 * a[2], lb = b[0] + 3 * b[1] + 9 * b[2];
    for (int t = 0; t < 6; ++t) {
      int i = -1, j = -1;
      for (int n = 0; n < 10; ++n) {
        if (cube_local(2, t, n) == la) i = n;
        if (cube_local(2, t, n) == lb) j = n;
      }
      if (i >= 0 && j >= 0) sum += fe_kuhn::kuhn_p2_k(i, j);
    }
  }
  return sum / 2;
}
// the eight coefficients of one offset, packed for a compile-time test that any is not zero
__host__ __device__ constexpr bool stencil_uses(int ox, int oy, int oz) {
  for (int code = 0; code < 8; ++code)
    if (stencil_coef(code, ox, oy, oz) != 0) return true;
  return false;
}
static_assert(stencil_coef(0, 0, 0, 0) == 54 && stencil_coef(3, 1, 1, 0) == 48 &&
                  stencil_coef(1, 1, 0, 0) == 56 && stencil_coef(7, 1, 1, 1) == 48 &&
                  stencil_coef(0, 2, 1, 1) == 1 && stencil_coef(3, 0, 0, -1) == 4,
              "P2 Kuhn stencils");

// All eight rows of a cell, one lattice value at a time: each is loaded once and
// goes into every row that couples to it.
template <int I, typename V, typename At>
__device__ __forceinline__ void stencil_point(RowSum<V> (&r)[8], At& at) {
  constexpr int x = I % 5 - 2, y = I / 5 % 5 - 2, z = I / 25 - 2;
  if constexpr (stencil_uses(x, y, z)) {
    const V v = at(x, y, z);
    auto one = [&](auto code_) {
      constexpr int code = decltype(code_)::value;
      constexpr int k = stencil_coef(code, x, y, z);
      if constexpr (k != 0) r[code].add(k, v);
    };
    one(std::integral_constant<int, 0>{});
    one(std::integral_constant<int, 1>{});
    one(std::integral_constant<int, 2>{});
    one(std::integral_constant<int, 3>{});
    one(std::integral_constant<int, 4>{});
    one(std::integral_constant<int, 5>{});
    one(std::integral_constant<int, 6>{});
    one(std::integral_constant<int, 7>{});
  }
}
// The cell's own points, whose coefficients (the diagonals among them) are the
// largest, come last, so that few sums are rounded at their size.
template <typename V, typename At, int... I>
__device__ __forceinline__ void stencil_rows(RowSum<V> (&r)[8], At at, std::integer_sequence<int, I...>) {
  constexpr auto own = [](int i) { return i % 5 - 2 >> 1 == 0 && (i / 5 % 5 - 2) >> 1 == 0 && (i / 25 - 2) >> 1 == 0; };
  auto point = [&](auto i, auto want) {
    if constexpr (own(decltype(i)::value) == decltype(want)::value) stencil_point<decltype(i)::value>(r, at);
  };
  (point(std::integral_constant<int, I>{}, std::false_type{}), ...);
  (point(std::integral_constant<int, I>{}, std::true_type{}), ...);
}

// The same stencils as lists, for the rows with a scale of their own: few as a rule, and eight stencils unrolled a
// second time would be fetched for each of them (FP64 64^3: 372 us).
template <int CODE, int I>
constexpr int kCoef = stencil_coef(CODE, I % 5 - 2, I / 5 % 5 - 2, I / 25 - 2);
struct StencilList {
  int n, sum, k[51], point[51];  // points, sum of |k|; coefficients, offsets as (x + 2) + 5 (y + 2) + 25 (z + 2)
};
template <int CODE, int... I>
constexpr StencilList stencil_list(std::integer_sequence<int, I...>) {
  StencilList L{};
  auto point = [&L](int k, int i) {
    if (k == 0) return;
    L.sum += k < 0 ? -k : k;
    L.k[L.n] = k;
    L.point[L.n++] = i;
  };
  (point(kCoef<CODE, I>, I), ...);
  return L;
}
template <int CODE>
constexpr StencilList kList = stencil_list<CODE>(std::make_integer_sequence<int, 125>{});

// Whether less than 2^-47 of a row's |A| |x| is cut off (at most the sum of |k| times 2^-59 of the scale): its own value
// is at least 2^-kOwnBits of the scale, or the sum of |k| |x| over it and its six axis neighbours is large enough.  The
// second test keeps the rows beside the corners of a smooth field, 2^-11.4 of the largest value in a tile of 16 x 4 x 4
// cells at a corner of the domain.
constexpr int kOwnBits = 10;
template <int CODE, typename At>
__device__ __forceinline__ bool row_kept(At at, int own) {
  constexpr int X = CODE & 1, Y = CODE >> 1 & 1, Z = CODE >> 2, sum = kList<CODE>.sum;
  constexpr int k = stencil_coef(CODE, X, Y, Z), kx = -stencil_coef(CODE, X - 1, Y, Z),
                ky = -stencil_coef(CODE, X, Y - 1, Z), kz = -stencil_coef(CODE, X, Y, Z - 1);
  static_assert(sum <= 216 && sum <= k << (12 - kOwnBits), "own value");
  static_assert(kx > 0 && ky > 0 && kz > 0, "axis neighbours");
  auto two = [&](int x, int y, int z) {
    return (abs(at(X + x, Y + y, Z + z).hi) >> 9) + (abs(at(X - x, Y - y, Z - z).hi) >> 9);
  };
  // 2^E: hi = 2^29
  return k * (own >> 9) + kx * two(1, 0, 0) + ky * two(0, 1, 0) + kz * two(0, 0, 1) >= sum << 8;
}

constexpr int kListStride = 56;
template <int TX_, int TY_, int KZ_, int THREADS_, int BLOCKS_>
struct TileShape {  // BLOCKS: resident blocks per SM that the registers are limited for
  static constexpr int blocks = BLOCKS_;
  static constexpr int TX = TX_, TY = TY_, KZ = KZ_, threads = THREADS_;
  static constexpr int W = TX + 2, H = TY + 2, D = KZ + 2, cells = W * H * D, own = TX * TY * KZ;
  template <typename T>
  static constexpr size_t smem() {
    return (size_t)cells * 8 * sizeof(T) + (sizeof(T) == 8 ? own + 4 * 8 * kListStride : 0);
  }
};

struct Lattice2 {  // the P2 numbering per parity code px + 2 py + 4 pz: first dof and strides of its class
  int N, off[8], sy[8], sz[8];
};

// The lists with the points' places in a staged tile, relative to the cell's: the number of points, the sum of |k|,
// then from entry 4 on place * 256 + (k & 255), the last point again with k = 0 up to whole groups of four.
struct TileLists {
  int p[8 * kListStride];
};
template <typename S, int... CODE>
constexpr TileLists tile_lists(std::integer_sequence<int, CODE...>) {
  TileLists L{};
  auto list = [&L](int* p, const StencilList& a) {
    p[0] = (a.n + 3) / 4 * 4;
    p[1] = a.sum;
    for (int i = 0; i < p[0]; ++i) {
      const int q = i < a.n ? i : a.n - 1;
      const int x = a.point[q] % 5 - 2, y = a.point[q] / 5 % 5 - 2, z = a.point[q] / 25 - 2;
      const int cls = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
      p[4 + i] = (cls * S::cells + (x >> 1) + S::W * ((y >> 1) + S::H * (z >> 1))) * 256 + (i < a.n ? a.k[q] & 255 : 0);
    }
  };
  (list(L.p + CODE * kListStride, kList<CODE>), ...);
  return L;
}
template <typename S>
__device__ const TileLists d_lists = tile_lists<S>(std::make_integer_sequence<int, 8>{});

// f(k, x) for the points of list p (in shared memory) of the staged cell.
template <typename V, typename F>
__device__ __forceinline__ void for_list(const int* p, const V* cell, F&& f) {
  const int4* a4 = reinterpret_cast<const int4*>(p + 4);
  const int n4 = p[0] / 4;
#pragma unroll 2
  for (int q = 0; q < n4; ++q) {
    const int4 a = a4[q];
    const V v0 = cell[a.x >> 8], v1 = cell[a.y >> 8], v2 = cell[a.z >> 8], v3 = cell[a.w >> 8];
    f((int)(signed char)a.x, v0);
    f((int)(signed char)a.y, v1);
    f((int)(signed char)a.z, v2);
    f((int)(signed char)a.w, v3);
  }
}

// The largest biased exponent of the values in the row of list p at the staged cell.
__device__ __forceinline__ int list_exponent(const int* p, const double* cell) {
  int er = 0;
  for_list(p, cell, [&](int, double v) { er = max(er, (__double2hiint(v) >> 20) & 0x7FF); });
  return er;
}
// The row in units of u, from the scale er of its own largest value (subnormal values count as 0); scale: of the matrix.
// With a value that is not finite, the FP64 sum.
__device__ __forceinline__ double listed_row(const int* p, const double* cell, int er, double scale, double& u) {
  u = scale;
  if (er == 0x7FF) {
    double s = 0.0;
    for_list(p, cell, [&](int k, double v) { s += k != 0 ? (double)k * v : 0.0; });
    return s;
  }
  if (er == 0) return 0.0;
  RowSum<Pair32> r;
  for_list(p, cell, [&](int k, double v) { r.add((__double2hiint(v) >> 20) & 0x7FF ? k : 0, fixed_pair(v, er)); });
  const bool fits = r.fits();
  const int ex = er - 1023 - kTop + (fits ? 0 : 6);  // the integers' unit
  if (er <= 300 || er >= 1900) {                     // (2^ex can lie outside the FP64 range)
    u = 1.0;
    return r.value(fits) * scale * pow2(ex / 2) * pow2(ex - ex / 2);
  }
  u = __hiloint2double(__double2hiint(scale) + ex * (1 << 20), __double2loint(scale));
  return r.value(fits);
}

template <typename T, int EPI, typename S>
__global__ void __launch_bounds__(S::threads, S::blocks)
    k_stencil2(const __grid_constant__ Lattice2 G, double scale, const __grid_constant__ Rows<T> R, int nb,
               const int* __restrict__ bnd) {
  constexpr bool FIX = sizeof(T) == 8;
  using V = typename std::conditional<FIX, Pair32, float>::type;
  static_assert(sizeof(V) == sizeof(T), "staged in place");
  static_assert(S::own % S::threads == 0 && S::own / S::threads <= 4, "a thread's rows in one word");
  extern __shared__ __align__(16) unsigned char smem[];
  T* raw = reinterpret_cast<T*>(smem);  // [8][cells]
  V* xs = reinterpret_cast<V*>(smem);
  int* lists = reinterpret_cast<int*>(smem + (size_t)S::cells * 8 * sizeof(T));  // [8][kListStride]
  unsigned char* marks = reinterpret_cast<unsigned char*>(lists + 8 * kListStride);  // [own]
  __shared__ int s_max, s_bad;
  const int tid = threadIdx.x, N = G.N;
  const int ntx = (N + S::TX - 1) / S::TX, nty = (N + S::TY - 1) / S::TY;
  const int i0 = (blockIdx.x % ntx) * S::TX, j0 = (blockIdx.x / ntx) % nty * S::TY, k0 = blockIdx.x / (ntx * nty) * S::KZ;
  if constexpr (FIX) {
    if (tid == 0) {
      s_max = 0;
      s_bad = 0;
    }
  }
  // the values of staged cell s: f(code, dof, whether it is interior)
  auto for_points = [&](int s, auto&& f) {
    const int ci = i0 - 1 + s % S::W, cj = j0 - 1 + (s / S::W) % S::H, ck = k0 - 1 + s / (S::W * S::H);
    // even coordinates are interior for 0 < c < N, odd ones for 0 <= c < N
    const bool below = ci < N && cj < N && ck < N;
    const bool xe = ci > 0, xo = ci >= 0, ye = cj > 0 && below, yo = cj >= 0 && below, ze = ck > 0, zo = ck >= 0;
#pragma unroll
    for (int code = 0; code < 8; ++code)
      f(code, G.off[code] + ci + G.sy[code] * cj + G.sz[code] * ck,
        (code & 1 ? xo : xe) && (code & 2 ? yo : ye) && (code & 4 ? zo : ze));
  };
  auto stage = [&] {
    for (int s = tid; s < S::cells; s += S::threads)
      for_points(s, [&](int code, int i, bool in) {
        cp_async_or_zero<sizeof(T)>(raw + code * S::cells + s, R.x + (in ? i : 0), in);
      });
    cp_async_commit();
  };
  stage();
  for (int i = blockIdx.x * S::threads + tid; i < nb; i += gridDim.x * S::threads) {  // Dirichlet rows: identity
    identity_row<EPI>(R, bnd[i]);
  }
  cp_async_wait_all();
  __syncthreads();
  int E = 0;
  bool bad = false;
  if constexpr (FIX) {
    int emax = 0, nf = 0;
    for (int s = tid; s < S::cells; s += S::threads) {
      int e = 0;
#pragma unroll
      for (int code = 0; code < 8; ++code)
        e = max(e, (int)(((unsigned int)__double2hiint(raw[code * S::cells + s]) >> 20) & 0x7FFu));
      if (e == 0x7FF) {  // values that are not finite are staged as 0
        nf = 1;
        e = 0;
#pragma unroll 1
        for (int code = 0; code < 8; ++code) {
          const int ev = (int)(((unsigned int)__double2hiint(raw[code * S::cells + s]) >> 20) & 0x7FFu);
          if (ev != 0x7FF) e = max(e, ev);
        }
      }
      emax = max(emax, e);
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    nf = __any_sync(0xffffffffu, nf);
    if ((tid & 31) == 0) {
      if (emax > 0) atomicMax(&s_max, emax);
      if (nf) atomicOr(&s_bad, 1);
    }
    __syncthreads();
    E = s_max;
    bad = s_bad != 0;
    for (int s = tid; s < S::cells; s += S::threads)
#pragma unroll
      for (int code = 0; code < 8; ++code) {
        const double v = raw[code * S::cells + s];
        xs[code * S::cells + s] = fixed_pair(v, max(E, 64));
      }
    __syncthreads();
  }
  // rows in units of s1 (FIX: scale 2^(E - 1023 - kTop)), where that and every row lie well inside the FP64 range
  const bool ranged = !FIX || (E > 300 && E < 1900);
  const double s1 = FIX && ranged ? scale * pow2(E - 1023 - kTop) : scale, s64 = 64.0 * s1;
  // |hi| of a row's own value below which it is tested: none in a tile of zeros
  const int low_own = E == 0 ? 0 : ranged ? 1 << (29 - kOwnBits) : INT_MAX;
  unsigned int low = 0u;  // this thread's rows that need a scale of their own: bit 8 (its cell) + code
#pragma unroll 1
  for (int c = tid, k = 0; c < S::own; c += S::threads, k += 8) {
    const int a = c % S::TX, b = (c / S::TX) % S::TY, e = c / (S::TX * S::TY);
    const int vi = i0 + a, vj = j0 + b, vk = k0 + e;
    if (vi >= N || vj >= N || vk >= N) continue;
    const V* base = xs + (a + 1 + S::W * (b + 1 + S::H * (e + 1)));
    auto at = [&](int x, int y, int z) -> V {
      return base[((x & 1) | ((y & 1) << 1) | ((z & 1) << 2)) * S::cells + (x >> 1) +
                  S::W * ((y >> 1) + S::H * (z >> 1))];
    };
    RowSum<V> rs[8];
    RowIn<EPI, T> ins[8];  // FP32: every row's vectors in flight before the rows are formed
    if constexpr (!FIX && EPI != EPI_APPLY) {
#pragma unroll
      for (int code = 0; code < 8; ++code)
        if (((code & 1) || vi > 0) && ((code & 2) || vj > 0) && ((code & 4) || vk > 0))
          ins[code] = RowIn<EPI, T>(R, G.off[code] + vi + G.sy[code] * vj + G.sz[code] * vk);
    }
    if constexpr (!FIX) stencil_rows(rs, at, std::make_integer_sequence<int, 125>{});
    // rows on the boundary; by one mask in FP64 only (two Chebyshev steps at 64^3 81.4 us against 81.9; FP32 application
    // at 128^3 49.2 against 47.2 without it)
    const unsigned int edge = (vi == 0 ? 0x55u : 0u) | (vj == 0 ? 0x33u : 0u) | (vk == 0 ? 0x0Fu : 0u);
    auto row = [&](auto code_) {
      constexpr int code = decltype(code_)::value;
      if (FIX ? (edge >> code & 1) != 0
              : !((code & 1) || vi > 0) || !((code & 2) || vj > 0) || !((code & 4) || vk > 0))
        return;
      const int i = G.off[code] + vi + G.sy[code] * vj + G.sz[code] * vk;
      if constexpr (FIX) {
        auto left = [&] {
          const int own = abs(at(code & 1, code >> 1 & 1, code >> 2).hi);
          if (own >= low_own || (ranged && row_kept<code>(at, own))) return false;
          low |= 1u << (k + code);
          return true;
        };
        // a residual's row is tested first, the others once formed (64^3: 36.4 against 39.4 us; two Chebyshev steps 81.4
        // against 84.4, an application 29.9 against 30.4)
        if constexpr (EPI == EPI_RESIDUAL)
          if (left()) return;
        const RowIn<EPI, T> in(R, i);
        const RowSum<V> r = stencil_row<code, V>(at);
        if constexpr (EPI != EPI_RESIDUAL)
          if (left()) return;
        const bool fits = r.fits();
        finish_row<EPI>(R, in, i, r.value(fits), fits ? s1 : s64, R.wd[code]);
      } else {
        finish_row<EPI>(R, ins[code], i, rs[code].s, (float)(scale * RowSum<V>::unit), R.wd[code]);
      }
    };
    for_codes(row);
  }
  if constexpr (FIX) {
    // The warps take 32 cells' rows of one stencil in turn: f(turn, code, cell, whether the row is marked).
    auto for_rows = [&](auto&& f) {
#pragma unroll 1
      for (int t = tid / 32, turn = 0; t < S::own / 4; t += S::threads / 32, ++turn) {
        const int code = t & 7, c = (t >> 3) * 32 + tid % 32;
        f(turn, code, c, (marks[c] >> code & 1) != 0);
      }
    };
    auto place = [&](int c) { return c % S::TX + 1 + S::W * ((c / S::TX) % S::TY + 1 + S::H * (c / (S::TX * S::TY) + 1)); };
    auto put = [&](int code, int c, double v, double u) {
      const int i = G.off[code] + i0 + c % S::TX + G.sy[code] * (j0 + (c / S::TX) % S::TY) +
                    G.sz[code] * (k0 + c / (S::TX * S::TY));
      finish_row<EPI>(R, RowIn<EPI, T>(R, i), i, v, u, R.wd[code]);
    };
    const int marking = __syncthreads_count(low != 0u);
    if (marking > 0 || bad) {
      for (int c = tid; c < S::own; c += S::threads, low >>= 8) marks[c] = (unsigned char)low;
      for (int q = tid; q < 8 * kListStride; q += S::threads) lists[q] = d_lists<S>.p[q];
      __syncthreads();
      // first, unless they are many, the exact test of what is cut off, on the values staged already: it keeps the rows
      // where nodal planes of a smooth field meet (64^3: 31 us against 36)
      const bool test = ranged && marking <= S::threads / 4;
      unsigned int scaled = 0u, check = 0u;  // this thread's turns left: rows with a scale of their own; all others of a
                                             // tile with values that are not finite, for the rows that couple to one
      for_rows([&](int turn, int code, int c, bool marked) {
        if (!marked) {
          if (bad) check |= 1u << turn;
          return;
        }
        const int* list = lists + code * kListStride;
        RowSum<Pair32> r;
        int w = 0;
        if (test)
          for_list(list, xs + place(c), [&](int k, Pair32 v) {
            r.add(k, v);
            w += abs(k) * (abs(v.hi) >> 9);
          });
        if (!test || w < list[1] << 8) {
          scaled |= 1u << turn;
          return;
        }
        if (bad) check |= 1u << turn;
        const bool fits = r.fits();
        put(code, c, r.value(fits), fits ? s1 : s64);
      });
      if (__syncthreads_or((int)(scaled | check))) {
        stage();
        cp_async_wait_all();
        __syncthreads();
        for_rows([&](int turn, int code, int c, bool) {
          if (!((scaled | check) >> turn & 1)) return;
          const int vi = i0 + c % S::TX, vj = j0 + (c / S::TX) % S::TY, vk = k0 + c / (S::TX * S::TY);
          if (vi >= N || vj >= N || vk >= N || !((code & 1) || vi > 0) || !((code & 2) || vj > 0) ||
              !((code & 4) || vk > 0))
            return;
          const int* list = lists + code * kListStride;
          const int er = list_exponent(list, raw + place(c));
          if (!(scaled >> turn & 1) && er != 0x7FF) return;
          double u;
          const double v = listed_row(list, raw + place(c), er, scale, u);
          put(code, c, v, u);
        });
      }
    }
  }
}

// Small levels: one thread per dof (a block row per parity class, so that its
// threads share one stencil) reads its 19 to 51 values from the caches and sums
// them in the vectors' own arithmetic.  A level of a few thousand cells is bound by
// the latency of its one launch, and this form has no staging, no scale and no
// barrier: P2 16^3 in FP64 is 36 k rows of 23 operations, 1.3 us of the FP64 pipe.
constexpr int kDirectBlock = 128;

template <typename T, int EPI>
__global__ void __launch_bounds__(kDirectBlock)
    k_stencil2_direct(Lattice2 G, double scale, Rows<T> R, int nb, const int* __restrict__ bnd) {
  const int N = G.N, tid = blockIdx.x * kDirectBlock + threadIdx.x;
  const int stride = gridDim.x * gridDim.y * kDirectBlock;
  for (int i = tid + blockIdx.y * gridDim.x * kDirectBlock; i < nb; i += stride) {  // Dirichlet rows: identity
    identity_row<EPI>(R, bnd[i]);
  }
  const int vi = tid % N, vj = (tid / N) % N, vk = tid / (N * N);
  if (vk >= N) return;
  auto row = [&](auto code_) {
    constexpr int code = decltype(code_)::value;
    if (!((code & 1) || vi > 0) || !((code & 2) || vj > 0) || !((code & 4) || vk > 0)) return;
    auto at = [&](int x, int y, int z) -> T {
      // coarse coordinate v + floor(o / 2) of the point's class; interior for 0 < 2 v + o < 2 N
      const int px = 2 * vi + x, py = 2 * vj + y, pz = 2 * vk + z;
      const bool in = px > 0 && px < 2 * N && py > 0 && py < 2 * N && pz > 0 && pz < 2 * N;
      const int c = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
      return in ? __ldg(R.x + G.off[c] + (px >> 1) + G.sy[c] * (py >> 1) + G.sz[c] * (pz >> 1)) : T(0);
    };
    const int i = G.off[code] + vi + G.sy[code] * vj + G.sz[code] * vk;
    const RowIn<EPI, T> in(R, i);
    RowSum<T> r = stencil_row<code, T>(at);
    T unit = (T)(scale * RowSum<T>::unit);
    if (not_finite(r.s)) {  // values close to the end of the range
      r = stencil_row<code, T>([&](int x, int y, int z) { return at(x, y, z) * T(0.00390625); });
      unit *= T(256);
    }
    finish_row<EPI>(R, in, i, r.s, unit, R.wd[code]);
  };
  switch (blockIdx.y) {
    case 0: row(std::integral_constant<int, 0>{}); break;
    case 1: row(std::integral_constant<int, 1>{}); break;
    case 2: row(std::integral_constant<int, 2>{}); break;
    case 3: row(std::integral_constant<int, 3>{}); break;
    case 4: row(std::integral_constant<int, 4>{}); break;
    case 5: row(std::integral_constant<int, 5>{}); break;
    case 6: row(std::integral_constant<int, 6>{}); break;
    default: row(std::integral_constant<int, 7>{}); break;
  }
}

// FP64: 43 KB, five blocks per SM, on levels whose tiles are few, where the whole
// grid is one or two rounds of blocks (two Chebyshev steps at 32^3 30.8 us against
// 35.0 with the larger tile, 64^3 80.6 against 84.6, 80^3 166.9 against 167.5); above,
// 71 KB and less of the values staged twice (96^3 267 against 254, 128^3 568 against
// 547; applications are within 2% of each other).  FP32: rows of 32 cells, so that
// a warp's shared-memory accesses fall into distinct banks (rows of 16: 58 against
// 48 us at 128^3).
using Tile64Few = TileShape<16, 4, 4, 128, 5>;
using Tile64Many = TileShape<16, 8, 4, 256, 3>;
using Tile32 = TileShape<32, 4, 8, 256, 3>;
constexpr int kTileFewMax = 96;  // cubes per axis
// The direct kernel: an application at 16^3 6.2 us against 12.3 with the larger tile, two steps 14.4 against 34.8; its
// operations grow with the level, the tiles' latency does not (24^3 10.6 against 10.3, steps 24.8 against 30.7, with the
// smaller tile).
constexpr int kDirectMax = 16;

Lattice2 lattice_of(const Level& L) {
  Lattice2 G{};
  G.N = L.N;
  for (int code = 0; code < 8; ++code) {
    const int c = code == 3 ? 4 : code == 4 ? 3 : code;
    G.off[code] = L.num.off[c];
    G.sy[code] = L.num.sx[c];
    G.sz[code] = L.num.sx[c] * L.num.sy[c];
  }
  return G;
}

template <int EPI, typename T, typename S>
void launch_tiles(const Level& L, double scale, const Rows<T>& R, cudaStream_t s) {
  const int grid = ceil_div(L.N, S::TX) * ceil_div(L.N, S::TY) * ceil_div(L.N, S::KZ);
  k_stencil2<T, EPI, S><<<grid, S::threads, S::template smem<T>(), s>>>(lattice_of(L), scale, R, L.nb, L.bnd);
}

template <int EPI, typename T>
void launch_stencil(const Level& L, const Rows<T>& R, cudaStream_t s) {
  const double scale = 8.0 * (L.kappa0 / (120.0 * L.N));
  if (L.N <= kDirectMax)
    k_stencil2_direct<T, EPI><<<dim3(ceil_div((long long)L.Q, kDirectBlock), 8), kDirectBlock, 0, s>>>(
        lattice_of(L), scale, R, L.nb, L.bnd);
  else if constexpr (sizeof(T) == 4)
    launch_tiles<EPI, T, Tile32>(L, scale, R, s);
  else if (L.N <= kTileFewMax)
    launch_tiles<EPI, T, Tile64Few>(L, scale, R, s);
  else
    launch_tiles<EPI, T, Tile64Many>(L, scale, R, s);
  LAUNCH_CHECK();
}

// The shared-memory limit of a kernel is a property of the device's context and
// has one value per kernel, so setting it again for another hierarchy is harmless.
template <typename T, int EPI, typename S>
void set_smem() {
  CUDA_CHECK(cudaFuncSetAttribute((const void*)k_stencil2<T, EPI, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)S::template smem<T>()));
}
template <int EPI>
void set_smems() {
  set_smem<double, EPI, Tile64Few>();
  set_smem<double, EPI, Tile64Many>();
  set_smem<float, EPI, Tile32>();
}

template <int EPI, typename T>
void launch(const Level& L, const Rows<T>& R, cudaStream_t s) {
  constexpr bool F64 = sizeof(T) == 8;
  if (L.deg == 1) {
    const int grid = ceil_div(L.n, kP1Block);
    const T* w = nullptr;
    if constexpr (F64)
      w = L.fw64;
    else
      w = L.fw32;
    if (L.flux == FLUX_CONST)
      k_flux1<T, true, EPI><<<grid, kP1Block, 0, s>>>(L.N, L.n, nullptr, (T)(L.kappa0 / L.N), R);
    else
      k_flux1<T, false, EPI><<<grid, kP1Block, 0, s>>>(L.N, L.n, w, T(0), R);
    LAUNCH_CHECK();
    return;
  }
  launch_stencil<EPI, T>(L, R, s);
}

}  // namespace

// Data of the flux form of a level whose L.flux launch_uniform_geometry has set.
void launch_flux_setup(Level& L, cudaStream_t s) {
  if (L.flux == FLUX_NONE) return;
  if (L.deg == 2) {
    set_smems<EPI_APPLY>();
    set_smems<EPI_CHEB>();
    set_smems<EPI_RESIDUAL>();
  } else if (L.flux == FLUX_VAR) {
    L.fw64.alloc((size_t)4 * L.n);
    L.fw32.alloc((size_t)4 * L.n);
    k_edge_weights<<<ceil_div(L.n, 128), 128, 0, s>>>(L.N, L.n, L.geo64.p + (size_t)5 * L.Cs, L.fw64, L.fw32);
    LAUNCH_CHECK();
  }
}

template <typename T>
void launch_flux_apply(const Level& L, const T* x, T* y, cudaStream_t s) {
  Rows<T> R{};
  R.x = x;
  R.out = y;
  launch<EPI_APPLY>(L, R, s);
}
template void launch_flux_apply<double>(const Level&, const double*, double*, cudaStream_t);
template void launch_flux_apply<float>(const Level&, const float*, float*, cudaStream_t);

template <typename T>
void launch_flux_residual(const Level& L, const T* b, const T* x, T* r, cudaStream_t s) {
  Rows<T> R{};
  R.x = x;
  R.b = b;
  R.out = r;
  launch<EPI_RESIDUAL>(L, R, s);
}
template void launch_flux_residual<double>(const Level&, const double*, const double*, double*, cudaStream_t);
template void launch_flux_residual<float>(const Level&, const float*, const float*, float*, cudaStream_t);

template <typename T>
void launch_flux_cheb(const Level& L, const T* b, const T* x, T* xout, const T* din, T* dout, double c1, double c2,
                      cudaStream_t s) {
  Rows<T> R{};
  R.x = x;
  R.out = xout;
  R.b = b;
  R.din = c1 != 0.0 ? din : nullptr;
  R.dout = dout;
  if constexpr (sizeof(T) == 8)
    R.dinv = L.dinv64;
  else
    R.dinv = L.dinv32;
  R.c1 = (T)c1;
  R.c2 = (T)c2;
  const double k = L.kappa0 / L.N;
  const int diag[8] = {54, 56, 56, 48, 56, 48, 48, 48};
  for (int code = 0; code < 8; ++code)
    R.wd[code] = (T)(L.deg == 1 ? c2 / (6.0 * k) : c2 * (120.0 / 8.0) / (diag[code] * k));
  launch<EPI_CHEB>(L, R, s);
}
template void launch_flux_cheb<double>(const Level&, const double*, const double*, double*, const double*, double*,
                                       double, double, cudaStream_t);
template void launch_flux_cheb<float>(const Level&, const float*, const float*, float*, const float*, float*, double,
                                      double, cudaStream_t);
