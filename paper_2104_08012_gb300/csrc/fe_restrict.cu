// P2 restriction rc = P^T (b - y) between nested Kuhn meshes with zero
// boundary rows (paper Section 3: the multigrid transfers), each fine value staged
// once per tile.
//
// A coarse basis function is evaluated at the fine nodes of its support: with
// fine coordinates counted from four times the coarse vertex, the eight coarse
// dofs of a vertex cell take 275 weights (multiples of 1/8, pro_w8) on the window
// [-3, 3]^3, 4.3 per fine dof.  The table-driven form (k_restrict) gathers every
// one of them from L2 with its index arithmetic.  Here a block stages the
// residual of TX x TY x KZ coarse cells and one layer below them in shared
// memory, split by the fine coordinates modulo 4 so that a warp's accesses are
// contiguous, and the weights are immediate operands.  Two threads serve a cell:
// one the vertex row (125 weights), one the seven others (150).  At 128^3 -> 64^3
// the gathers took 215 us, staging b and y through registers 131 us, and with the
// residual left by the operator one vector staged by asynchronous copies 48 us
// (its bytes: 11 us).
// FP64: 275 operations per coarse cell on the FP64 pipe (2 per clock and SM), 16 us
// at 64^3 -> 32^3, and 30 us measured against 43 for the gathers where the operator
// has left the residual.  Staging b - y costs 2.4 more operations per fine dof (59
// us), so there the gathers stay; exact integer sums of 30-bit halves took 31 us.
#include <utility>

#include "fe_internal.cuh"
#include "fe_kuhn.h"

namespace {

template <int TX_, int TY_, int KZ_, int BLOCKS_>
struct RestrictTile {
  static constexpr int TX = TX_, TY = TY_, KZ = KZ_, blocks = BLOCKS_;
  static constexpr int W = TX + 1, H = TY + 1, D = KZ + 1, own = TX * TY * KZ, threads = 2 * own;
  // entries per residue class, padded to 8 modulo 16: the two classes that neighbouring fine cells alternate between
  // start half the banks apart
  static constexpr int S = (W * H * D + 7) / 16 * 16 + 8;
  static_assert(S >= W * H * D && own % 32 == 0, "tile");
  template <typename T>
  static constexpr size_t smem() {
    return (size_t)64 * S * sizeof(T);
  }
};

struct Classes {
  int N, off[8], sy[8], sz[8];  // cubes per axis; per parity code px + 2 py + 4 pz: first dof, strides
};

// 8 times the value of the coarse basis function of the cell's dof of parity code
// CODE at the fine point (x, y, z) of the window.
__host__ __device__ constexpr int restrict_w8(int code, int x, int y, int z) {
  const int f[3] = {x, y, z};
  int o[3] = {0, 0, 0}, n[3] = {0, 0, 0};
  for (int d = 0; d < 3; ++d) {
    const int c = f[d] < 0 ? -1 : 0;  // the coarse cube that holds the point
    o[d] = f[d] - 4 * c;
    n[d] = (code >> d & 1) - 2 * c;
    if (n[d] > 2) return 0;
  }
  return fe_kuhn::pro_w8(o[0], o[1], o[2], n[0], n[1], n[2]);
}

template <int FIRST, int LAST>
__host__ __device__ constexpr bool any_w8(int x, int y, int z) {
  for (int code = FIRST; code <= LAST; ++code)
    if (restrict_w8(code, x, y, z) != 0) return true;
  return false;
}

// the window point I (x fastest) and its weights in the rows FIRST .. LAST: add(row, 8 w, v) as constants
template <int FIRST, int LAST, int I, typename At, typename Add>
__device__ __forceinline__ void window_point(At& at, Add& add) {
  constexpr int x = I % 7 - 3, y = I / 7 % 7 - 3, z = I / 49 - 3;
  if constexpr (any_w8<FIRST, LAST>(x, y, z)) {
    const auto v = at(x, y, z);
    auto one = [&](auto code_) {
      constexpr int code = decltype(code_)::value;
      if constexpr (code >= FIRST && code <= LAST) {
        constexpr int w = restrict_w8(code, x, y, z);
        if constexpr (w != 0) add(code, w, v);
      }
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
template <int FIRST, int LAST, typename At, typename Add, int... I>
__device__ __forceinline__ void window_points(At& at, Add& add, std::integer_sequence<int, I...>) {
  (window_point<FIRST, LAST, I>(at, add), ...);
}
template <int FIRST, int LAST, typename At, typename Add>
__device__ __forceinline__ void window(At at, Add add) {
  window_points<FIRST, LAST>(at, add, std::make_integer_sequence<int, 343>{});
}

// Rows FIRST .. LAST of a cell, put(row, value).
template <int FIRST, int LAST, typename At, typename Put>
__device__ __forceinline__ void restrict_rows(At at, Put put) {
  using T = decltype(at(0, 0, 0));
  T r[8] = {};
  window<FIRST, LAST>(at, [&](int code, int w, T v) { r[code] += (T)w * v; });  // (fused to one operation)
#pragma unroll
  for (int code = FIRST; code <= LAST; ++code) put(code, T(0.125) * r[code]);
}

template <typename T, typename S>
__global__ void __launch_bounds__(S::threads, S::blocks)
    k_restrict2(Classes F, Classes C, const T* __restrict__ b, const T* __restrict__ y, T* __restrict__ rc, int nb,
                const int* __restrict__ bnd) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* v = reinterpret_cast<T*>(smem);  // [zm][ym][xm][S]: fine coordinates modulo 4, then coarse cells
  const int tid = threadIdx.x, N = C.N;
  const int ntx = (N + S::TX - 1) / S::TX, nty = (N + S::TY - 1) / S::TY;
  const int i0 = (blockIdx.x % ntx) * S::TX, j0 = (blockIdx.x / ntx) % nty * S::TY, k0 = blockIdx.x / (ntx * nty) * S::KZ;
  for (int i = blockIdx.x * S::threads + tid; i < nb; i += gridDim.x * S::threads) rc[bnd[i]] = T(0);
  // fine cells (two per coarse cell and axis) of the coarse cells i0 - 1 .. i0 + TX - 1, x fastest
  constexpr int FW = 2 * S::W, FH = 2 * S::H, FD = 2 * S::D;
  for (int s = tid; s < FW * FH * FD; s += S::threads) {
    const int a = s % FW, bb = (s / FW) % FH, c = s / (FW * FH);
    const int ci = 2 * i0 - 2 + a, cj = 2 * j0 - 2 + bb, ck = 2 * k0 - 2 + c;
    const bool in = ci >= 0 && cj >= 0 && ck >= 0;
    T* at = v + a / 2 + S::W * (bb / 2 + S::H * (c / 2)) + S::S * (2 * (a & 1) + 8 * (bb & 1) + 32 * (c & 1));
#pragma unroll
    for (int code = 0; code < 8; ++code) {
      const int px = code & 1, py = code >> 1 & 1, pz = code >> 2;
      const int i = F.off[code] + ci + F.sy[code] * cj + F.sz[code] * ck;
      const bool ok = in && ci + px <= F.N && cj + py <= F.N && ck + pz <= F.N;
      T* to = at + S::S * (px + 4 * py + 16 * pz);
      if (!y)  // one vector: every copy in flight at once
        cp_async_or_zero<sizeof(T)>(to, b + (ok ? i : 0), ok);
      else
        *to = ok ? __ldg(b + i) - __ldg(y + i) : T(0);
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  const int c = tid % S::own;
  const int a = c % S::TX, bb = (c / S::TX) % S::TY, e = c / (S::TX * S::TY);
  const int vi = i0 + a, vj = j0 + bb, vk = k0 + e;
  if (vi >= N || vj >= N || vk >= N) return;
  const T* base = v + a + 1 + S::W * (bb + 1 + S::H * (e + 1));
  auto at = [&](int x, int yy, int z) -> T {
    return base[S::S * ((x & 3) + 4 * (yy & 3) + 16 * (z & 3)) + (x >> 2) + S::W * ((yy >> 2) + S::H * (z >> 2))];
  };
  auto put = [&](int code, T r) {
    if (((code & 1) || vi > 0) && ((code & 2) || vj > 0) && ((code & 4) || vk > 0))
      rc[C.off[code] + vi + C.sy[code] * vj + C.sz[code] * vk] = r;
  };
  if (tid < S::own)  // (whole warps)
    restrict_rows<0, 0>(at, put);
  else
    restrict_rows<1, 7>(at, put);
}

// 113 KB: two blocks of 512 threads per SM (whole mixed-precision P2 128^3 solves: 11.06 ms; smaller tiles 11.3 to
// 12.1, the values of their extra layers)
template <typename T>
using Tile = RestrictTile<16, 4, 4, sizeof(T) == 4 ? 2 : 1>;

Classes classes_of(const Level& L) {
  Classes c{};
  c.N = L.N;
  for (int code = 0; code < 8; ++code) {
    const int k = code == 3 ? 4 : code == 4 ? 3 : code;
    c.off[code] = L.num.off[k];
    c.sy[code] = L.num.sx[k];
    c.sz[code] = L.num.sx[k] * L.num.sy[k];
  }
  return c;
}

}  // namespace

template <typename T>
void launch_restrict_p2(const Level& F, const Level& Cc, const T* b, const T* y, T* rc, cudaStream_t s) {
  using S = Tile<T>;
  const int grid = (Cc.N + S::TX - 1) / S::TX * ((Cc.N + S::TY - 1) / S::TY) * ((Cc.N + S::KZ - 1) / S::KZ);
  k_restrict2<T, S><<<grid, S::threads, S::template smem<T>(), s>>>(classes_of(F), classes_of(Cc), b, y, rc, Cc.nb,
                                                                    Cc.bnd);
  LAUNCH_CHECK();
}
template void launch_restrict_p2<double>(const Level&, const Level&, const double*, const double*, double*,
                                         cudaStream_t);
template void launch_restrict_p2<float>(const Level&, const Level&, const float*, const float*, float*, cudaStream_t);

// The kernel's shared-memory limit (one value per kernel, see fe_flux.cu).
template <typename T>
static void set_smem() {
  CUDA_CHECK(cudaFuncSetAttribute((const void*)k_restrict2<T, Tile<T>>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Tile<T>::template smem<T>()));
}
void restrict_p2_prepare() {
  set_smem<double>();
  set_smem<float>();
}
