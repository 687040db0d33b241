// Adjoint of the Hamiltonian application with respect to the potential.
//
// Eq. Veff and Hloc with Section 2.3: Ht = 1/2 M^-1/2 K M^-1/2 + diag(V_eff) on psi nodes,
// the potential collocated at the nodes.  For Y = Ht(V) X and a loss L(Y) with
// Ybar = dL/dY, V enters only through the diagonal term, so
//   dL/dV_I = sum_v Ybar_Iv X_Iv,
// and the adjoint with respect to X is Ht^T Ybar = Ht Ybar (Ht is symmetric), i.e.
// fe_apply_H itself.  One warp per node row: the lanes stride over the row's vector
// entries (coalesced), accumulate in double, and the warp sums them in a fixed order, so
// the result is deterministic.
#include <cstdint>

#include "fe_blas.cuh"
#include "fe_internal.h"

namespace {

template <typename T>
__global__ void k_potential_vjp(const T* __restrict__ X, const T* __restrict__ Yb, int64_t ld,
                                int64_t nl, int64_t n, double* __restrict__ g) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); row < n;
       row += warps) {
    const T* x = X + row * ld;
    const T* y = Yb + row * ld;
    double s = 0.0;
    for (int64_t v = lane; v < nl; v += 32) s = fma((double)y[v], (double)x[v], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) g[row] = s;
  }
}

// A normal float as a double by integer arithmetic (exact): conversions share the FP64 pipe
// with the FMAs, and at two an entry they were most of its work.
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(b << 29));
}
__device__ __forceinline__ bool normal(float f) {
  return ((__float_as_uint(f) & 0x7f800000u) - 0x00800000u) < 0x7f000000u;
}
__device__ __forceinline__ double term(float y, float x, double s) {
  return fma((double)y, (double)x, s);   // (zeros, subnormals, infinities, NaNs)
}

// The same sums for float rows of 16-byte aligned groups of four: eight lanes a row, so that all
// lanes take part in the last adds.  FP64 issue bounds it (one FMA an entry): 17 us on 53,100
// nodes x 96 vectors, where k_potential_vjp takes 47.
__global__ void __launch_bounds__(256)
k_potential_vjp4(const float* __restrict__ X, const float* __restrict__ Yb, int64_t ld, int64_t nl,
                 int64_t n, double* __restrict__ g) {
  const int lane = threadIdx.x % 8;
  const int64_t rows = (int64_t)gridDim.x * (blockDim.x / 8);
  for (int64_t row0 = (int64_t)blockIdx.x * (blockDim.x / 8); row0 < n; row0 += rows) {
    const int64_t row = row0 + threadIdx.x / 8;
    double s = 0.0;
    if (row < n) {
      const float* x = X + row * ld;
      const float* y = Yb + row * ld;
#pragma unroll 4
      for (int64_t v = 4 * lane; v + 4 <= nl; v += 32) {
        const float4 a = *reinterpret_cast<const float4*>(x + v);
        const float4 b = *reinterpret_cast<const float4*>(y + v);
        if (normal(a.x) && normal(a.y) && normal(a.z) && normal(a.w) && normal(b.x) &&
            normal(b.y) && normal(b.z) && normal(b.w)) {
          s = fma(widen(b.x), widen(a.x), s);
          s = fma(widen(b.y), widen(a.y), s);
          s = fma(widen(b.z), widen(a.z), s);
          s = fma(widen(b.w), widen(a.w), s);
        } else {
          s = term(b.w, a.w, term(b.z, a.z, term(b.y, a.y, term(b.x, a.x, s))));
        }
      }
      const int64_t rest = nl & ~(int64_t)3;
      if (rest + lane < nl) s = term(y[rest + lane], x[rest + lane], s);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (row < n && lane == 0) g[row] = s;
  }
}

}  // namespace

extern "C" fe_status fe_potential_vjp(fe_mesh* m, const void* X, const void* Ybar, int64_t nvec,
                                      int64_t ld, double* gV, fe_precision prec) {
  if (!m || !X || !Ybar || !gV) return fe_fail(FE_EINVAL, "fe_potential_vjp: null argument");
  if (prec != FE_F64 && prec != FE_F32 && prec != FE_BF16_F32ACC && prec != FE_F32_F32ACC)
    return fe_fail(FE_EINVAL, "fe_potential_vjp: bad precision");
  if (nvec < 1 || ld < nvec) return fe_fail(FE_EINVAL, "fe_potential_vjp: need 1 <= nvec <= ld");
  if (m->has_quad)
    return fe_fail(FE_EUNSUPPORTED, "fe_potential_vjp: the potential is collocated only (the "
                   "Gauss-quadrature potential is in effect)");
  FE_TRY(fe_activate(m));
  // complex (Bloch) blocks: the diagonal term acts on both (re, im) lanes alike
  const int64_t lanes = m->has_k ? 2 : 1;
  const int64_t nl = nvec * lanes, ldl = ld * lanes;
  const int blocks = fe::grid_for(m->n_psi * 32, 256);
  if (prec == FE_F64)
    k_potential_vjp<double><<<blocks, 256, 0, m->stream>>>((const double*)X, (const double*)Ybar,
                                                           ldl, nl, m->n_psi, gV);
  else if ((uintptr_t)X % 16 == 0 && (uintptr_t)Ybar % 16 == 0 && ldl % 4 == 0)
    k_potential_vjp4<<<fe::grid_for(m->n_psi * 8, 256), 256, 0, m->stream>>>(
        (const float*)X, (const float*)Ybar, ldl, nl, m->n_psi, gV);
  else
    k_potential_vjp<float><<<blocks, 256, 0, m->stream>>>((const float*)X, (const float*)Ybar,
                                                          ldl, nl, m->n_psi, gV);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}
