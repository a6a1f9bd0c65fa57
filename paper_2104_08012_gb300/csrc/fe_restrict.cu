// FP32 P2 restriction rc = P^T (b - y) between nested Kuhn meshes with zero
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
// FP64 keeps the table-driven form: its 4.3 + 2.4 (residuals of the extra layer)
// operations per fine dof bind it to the FP64 pipe (64^3: 60 against 45 us).
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
  static constexpr size_t smem = (size_t)64 * S * sizeof(float);
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

// the window point I (x fastest) into the rows FIRST .. LAST
template <int FIRST, int LAST, int I, typename At>
__device__ __forceinline__ void window_point(float (&r)[8], At& at) {
  constexpr int x = I % 7 - 3, y = I / 7 % 7 - 3, z = I / 49 - 3;
  if constexpr (any_w8<FIRST, LAST>(x, y, z)) {
    const float v = at(x, y, z);
    auto one = [&](auto code_) {
      constexpr int code = decltype(code_)::value;
      if constexpr (code >= FIRST && code <= LAST) {
        constexpr int w = restrict_w8(code, x, y, z);
        if constexpr (w != 0) r[code] = __fmaf_rn((float)w, v, r[code]);
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
template <int FIRST, int LAST, typename At, int... I>
__device__ __forceinline__ void window(float (&r)[8], At at, std::integer_sequence<int, I...>) {
  (window_point<FIRST, LAST, I>(r, at), ...);
}

template <typename S>
__global__ void __launch_bounds__(S::threads, S::blocks)
    k_restrict2(Classes F, Classes C, const float* __restrict__ b, const float* __restrict__ y, float* __restrict__ rc,
                int nb, const int* __restrict__ bnd) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* v = reinterpret_cast<float*>(smem);  // [zm][ym][xm][S]: fine coordinates modulo 4, then coarse cells
  const int tid = threadIdx.x, N = C.N;
  const int ntx = (N + S::TX - 1) / S::TX, nty = (N + S::TY - 1) / S::TY;
  const int i0 = (blockIdx.x % ntx) * S::TX, j0 = (blockIdx.x / ntx) % nty * S::TY, k0 = blockIdx.x / (ntx * nty) * S::KZ;
  for (int i = blockIdx.x * S::threads + tid; i < nb; i += gridDim.x * S::threads) rc[bnd[i]] = 0.0f;
  // fine cells (two per coarse cell and axis) of the coarse cells i0 - 1 .. i0 + TX - 1, x fastest
  constexpr int FW = 2 * S::W, FH = 2 * S::H, FD = 2 * S::D;
  for (int s = tid; s < FW * FH * FD; s += S::threads) {
    const int a = s % FW, bb = (s / FW) % FH, c = s / (FW * FH);
    const int ci = 2 * i0 - 2 + a, cj = 2 * j0 - 2 + bb, ck = 2 * k0 - 2 + c;
    const bool in = ci >= 0 && cj >= 0 && ck >= 0;
    float* at = v + a / 2 + S::W * (bb / 2 + S::H * (c / 2)) + S::S * (2 * (a & 1) + 8 * (bb & 1) + 32 * (c & 1));
#pragma unroll
    for (int code = 0; code < 8; ++code) {
      const int px = code & 1, py = code >> 1 & 1, pz = code >> 2;
      const int i = F.off[code] + ci + F.sy[code] * cj + F.sz[code] * ck;
      const bool ok = in && ci + px <= F.N && cj + py <= F.N && ck + pz <= F.N;
      float* to = at + S::S * (px + 4 * py + 16 * pz);
      if (!y)  // one vector: every copy in flight at once
        cp_async_or_zero<4>(to, b + (ok ? i : 0), ok);
      else
        *to = ok ? __ldg(b + i) - __ldg(y + i) : 0.0f;
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  const int c = tid % S::own;
  const int a = c % S::TX, bb = (c / S::TX) % S::TY, e = c / (S::TX * S::TY);
  const int vi = i0 + a, vj = j0 + bb, vk = k0 + e;
  if (vi >= N || vj >= N || vk >= N) return;
  const float* base = v + a + 1 + S::W * (bb + 1 + S::H * (e + 1));
  auto at = [&](int x, int yy, int z) -> float {
    return base[S::S * ((x & 3) + 4 * (yy & 3) + 16 * (z & 3)) + (x >> 2) + S::W * ((yy >> 2) + S::H * (z >> 2))];
  };
  float r[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  auto put = [&](int code) {
    if (((code & 1) || vi > 0) && ((code & 2) || vj > 0) && ((code & 4) || vk > 0))
      rc[C.off[code] + vi + C.sy[code] * vj + C.sz[code] * vk] = 0.125f * r[code];
  };
  if (tid < S::own) {  // (whole warps)
    window<0, 0>(r, at, std::make_integer_sequence<int, 343>{});
    put(0);
  } else {
    window<1, 7>(r, at, std::make_integer_sequence<int, 343>{});
#pragma unroll
    for (int code = 1; code < 8; ++code) put(code);
  }
}

// 113 KB: two blocks of 512 threads per SM (whole mixed-precision P2 128^3 solves: 11.06 ms; smaller tiles 11.3 to
// 12.1, the values of their extra layers)
using Tile = RestrictTile<16, 4, 4, 2>;

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

void launch_restrict_p2(const Level& F, const Level& Cc, const float* b, const float* y, float* rc, cudaStream_t s) {
  using S = Tile;
  const int grid = (Cc.N + S::TX - 1) / S::TX * ((Cc.N + S::TY - 1) / S::TY) * ((Cc.N + S::KZ - 1) / S::KZ);
  k_restrict2<S><<<grid, S::threads, S::smem, s>>>(classes_of(F), classes_of(Cc), b, y, rc, Cc.nb, Cc.bnd);
  LAUNCH_CHECK();
}

// The kernel's shared-memory limit (one value per kernel, see fe_flux.cu).
void restrict_p2_prepare() {
  CUDA_CHECK(cudaFuncSetAttribute((const void*)k_restrict2<Tile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Tile::smem));
}
