// P3 operator on Kuhn tets (the paper's degree; the bilinear form of Section 2,
// Eq. 4) by the integer element matrix K of fe_p3.cuh: A_K = 48 c K, one c per tet.
//
// FP64: a tet's 20 dofs become two 30-bit integers of the tet's own scale (its
// largest exponent), each of the 362 products takes one 32 x 32 + 64-bit
// multiply-add per word, so K x is exact, and a row is rounded by one int64 ->
// FP64 conversion and one multiplication with 48 c times the scale.  The same
// element through the gradient at the P2 nodes in float pairs (fe_p3.cuh) takes
// 7.1 k instructions per tet at 8 warps per SM, this form about 1.6 k: P3 8^3,
// 32^3 and 40^3 19.4, 74 and 123 us -> 14.7, 43 and 73 us (3 blocks of 128 threads
// per SM; 2: 49 us at 32^3, 4: 47 with spills).  FP32 keeps the gradient form: with
// 362 multiply-adds instead of its 677 operations it took the same 18.5 us, bound
// by the gathers and the atomics.
#include <algorithm>
#include <utility>

#include "fe_fixed.cuh"
#include "fe_internal.cuh"
#include "fe_p3.cuh"

namespace {

using namespace fe_fixed;
constexpr int kBlock = 128;

template <int K>
__device__ __forceinline__ void term(PairSum& r, Pair32 v) {
  if constexpr (K != 0) r.add(K, v);
}
template <int I, int... J>
__device__ __forceinline__ PairSum row(const Pair32 (&u)[20], std::integer_sequence<int, J...>) {
  PairSum r;
  (term<fe_p3::kKuhnP3.k[I][J]>(r, u[J]), ...);
  return r;
}
template <typename Emit, int... I>
__device__ __forceinline__ void rows(const Pair32 (&u)[20], Emit&& emit, std::integer_sequence<int, I...>) {
  (emit(I, row<I>(u, std::make_integer_sequence<int, 20>{})), ...);
}

__global__ void __launch_bounds__(kBlock, 3)
    k_apply_p3_int(int C, int Cs, const int* __restrict__ map, const double* __restrict__ c161280,
                   const double* __restrict__ x, double* __restrict__ y, int nb, const int* __restrict__ bnd) {
  const int tid = blockIdx.x * kBlock + threadIdx.x, stride = gridDim.x * kBlock;
  for (int i = tid; i < nb; i += stride) y[bnd[i]] = x[bnd[i]];  // Dirichlet rows: identity
  for (int c = tid; c < C; c += stride) {
    int idx[20];
    double xv[20];
#pragma unroll
    for (int j = 0; j < 20; ++j) idx[j] = __ldg(map + (size_t)j * Cs + c);
#pragma unroll
    for (int j = 0; j < 20; ++j) xv[j] = idx[j] >= 0 ? __ldg(x + idx[j]) : 0.0;
    int E = 0;
#pragma unroll
    for (int j = 0; j < 20; ++j) E = max(E, (int)(((unsigned int)__double2hiint(xv[j]) >> 20) & 0x7FFu));
    double s1, s2 = 1.0;
    const bool tiny = E < 200;  // (and subnormal) dofs: by 2^600 up before and down after
    if (tiny) {
#pragma unroll
      for (int j = 0; j < 20; ++j) xv[j] *= pow2(600);
      E = 0;
#pragma unroll
      for (int j = 0; j < 20; ++j) E = max(E, (int)(((unsigned int)__double2hiint(xv[j]) >> 20) & 0x7FFu));
      if (E == 0) continue;  // every dof is zero
      s2 = pow2(-600);
    }
    Pair32 u[20];
#pragma unroll
    for (int j = 0; j < 20; ++j) u[j] = fixed_pair(xv[j], E);
    // rows |hi|, |lo| < 15768 * 2^30 < 2^44, as one int64 in units of 2^12
    s1 = 48.0 * __ldg(c161280 + c) * pow2(E - 1023 - kTop + 12);
    if (E == 0x7FF) s1 = __longlong_as_double(0x7ff8000000000000ll);  // a dof is not finite
    rows(
        u,
        [&](int j, const PairSum& r) {
          double v = (double)((long long)((unsigned long long)r.hi << 18) + (r.lo >> 12)) * s1;
          if (tiny) v *= s2;
          if (idx[j] >= 0) atomicAdd(y + idx[j], v);
        },
        std::make_integer_sequence<int, 20>{});
  }
}

}  // namespace

void launch_apply64_p3(const Level& L, const double* x, double* y, cudaStream_t s, bool y_zero) {
  if (!y_zero) CUDA_CHECK(cudaMemsetAsync(y, 0, sizeof(double) * (size_t)L.n, s));
  static int g = 0;
  if (!g) g = resident_grid(k_apply_p3_int, kBlock, 1 << 30);
  const int grid = std::max(1, std::min(g, (std::max(L.C, L.nb) + kBlock - 1) / kBlock));
  k_apply_p3_int<<<grid, kBlock, 0, s>>>(L.C, L.Cs, L.map, L.geo64.p + (size_t)5 * L.Cs, x, y, L.nb, L.bnd);
  LAUNCH_CHECK();
}
