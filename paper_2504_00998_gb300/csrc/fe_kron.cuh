// Matrix-free application of the finite-element stiffness of Section 2.3 on the uniform
// tensor-product slab mesh to one double vector, without scratch memory (where the cell-by-cell
// form's scratch cannot be had; blocks of vectors run in fe_sweep.cuh), and the coefficient
// tables and helpers that it shares with the tensor-core operator (fe_kron_tc.cu).
//
// For a uniform hexahedral mesh the assembled stiffness K_IJ = int grad N_I . grad N_J is a
// sum of Kronecker products of the exactly integrated 1D element matrices,
//   K = ax K1 (x) M1 (x) M1 + ay M1 (x) K1 (x) M1 + az M1 (x) M1 (x) K1,
// (ax = hy hz / (2 hx), ...).
//
// Work decomposition: one CTA owns the nodes of an xy block of B x B cells (half-open) and a
// range of z layers.  It sweeps the z planes in order.  Each plane (with a p-node periodic halo
// in x and y) is staged into shared memory with cp.async one plane ahead; the plane is
// contracted in y then in x (cell by cell, the shared boundary node taking the previous cell's
// last row), and the two in-plane results are accumulated into the p+1 output planes of the
// current z layer held in registers.  A layer's first p planes are final once its top plane
// is processed; the top plane's sum carries into the next layer.  No scatter, no atomics: every
// output node is written once by the thread that owns it, so results are bitwise reproducible.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fe_internal.h"

namespace fe {

// Device copy of the coefficient tables.  Rows have a stride of 8 entries, 16-byte aligned,
// so that the compiler can fetch four coefficients per constant load.
constexpr int KCS = 8;

template <typename T>
struct KronCoefT {
  alignas(16) T AyM[FE_MAXN1][KCS];
  alignas(16) T AyK[FE_MAXN1][KCS];
  alignas(16) T AxM[FE_MAXN1][KCS];
  alignas(16) T AxK[FE_MAXN1][KCS];
  // z tables with the plane's input scale folded in: AzKs[j][k] = AzK[j][k] zin / sqrt(mz_k),
  // mz_k the z mass factor of an interior plane with local index k (k = 0 and k = p: a plane
  // shared by two cells); a face plane multiplies its inputs by face_fix first
  alignas(16) T AzKs[FE_MAXN1][KCS];
  alignas(16) T AzMs[FE_MAXN1][KCS];
  T sig[FE_MAXN1];
  // 1/sqrt and sqrt of the z mass factor of a plane by local index (index 0: a plane shared
  // by two cells; *_face: the bottom or top face), so that no plane pays a division
  T rsq[FE_MAXN1], sq[FE_MAXN1];
  T rsq_face, sq_face, face_fix;
  T zout, izout;
  int mass_scale;
};

template <typename T>
inline KronCoefT<T> convert_coef(const KronCoef& c) {
  KronCoefT<T> o = {};
  double rsq[FE_MAXN1];
  for (int i = 0; i < FE_MAXN1; ++i) {
    const double mz = i == 0 ? 2.0 * c.wz[0] : c.wz[i];
    rsq[i] = c.mass_scale ? (mz > 0.0 ? 1.0 / std::sqrt(mz) : 0.0) : 1.0;
  }
  int p = 0;   // degree: the last local index with a nonzero GLL weight
  for (int i = 1; i < FE_MAXN1; ++i)
    if (c.wz[i] > 0.0) p = i;
  for (int i = 0; i < FE_MAXN1; ++i) {
    for (int j = 0; j < FE_MAXN1; ++j) {
      o.AyM[i][j] = (T)c.AyM[i][j];
      o.AyK[i][j] = (T)c.AyK[i][j];
      o.AxM[i][j] = (T)c.AxM[i][j];
      o.AxK[i][j] = (T)c.AxK[i][j];
      const double sz = c.zin * rsq[(j == p) ? 0 : j];
      o.AzKs[i][j] = (T)(c.AzK[i][j] * sz);
      o.AzMs[i][j] = (T)(c.AzM[i][j] * sz);
    }
    o.sig[i] = (T)c.sig[i];
    const double mz = i == 0 ? 2.0 * c.wz[0] : c.wz[i];
    o.rsq[i] = mz > 0.0 ? (T)(1.0 / std::sqrt(mz)) : T(0);
    o.sq[i] = (T)std::sqrt(mz > 0.0 ? mz : 0.0);
  }
  o.rsq_face = c.wz[0] > 0.0 ? (T)(1.0 / std::sqrt(c.wz[0])) : T(0);
  o.sq_face = (T)std::sqrt(c.wz[0] > 0.0 ? c.wz[0] : 0.0);
  o.face_fix = c.mass_scale ? (T)std::sqrt(2.0) : T(1);
  o.zout = (T)c.zout;
  o.izout = (T)(1.0 / c.zout);
  o.mass_scale = c.mass_scale;
  return o;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem, int nbytes_valid) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  if constexpr (BYTES == 16) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(nbytes_valid));
  } else if constexpr (BYTES == 8) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(nbytes_valid));
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(nbytes_valid));
  }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ int pmod(int a, int n) {
  int r = a % n;
  return r < 0 ? r + n : r;
}

// cells per block side for each p: about ten nodes per side
template <int P>
struct KronBlock {
  static constexpr int B = P == 1 ? 8 : P == 2 ? 5 : P == 3 ? 3 : 2;
};

// compile-time tile shape; threads: enough for one output node and one y-phase item each
template <int P_>
struct KronTile {
  static constexpr int P = P_, B = KronBlock<P>::B, BN = B * P, BH = BN + P + 1;
  static constexpr int NZI = BN * BN;                    // output nodes
  static constexpr int NST = BH * BH;                    // staged nodes per plane
  static constexpr int NYI = BH * B, NXI = BN * B;       // y- and x-phase items (cell segments)
  static constexpr int NTHR = ((NZI > NYI ? NZI : NYI) + 31) / 32 * 32;
  static constexpr int SPT = (NST + NTHR - 1) / NTHR;    // staged nodes per thread
  // stage slots: plane gz + 2 is staged while other threads may still read plane gz after the
  // plane's last barrier, so three slots keep those reads race-free
  static constexpr int NSB = 3;
  // row strides of the in-plane intermediates, odd so that the x phase's column-wise accesses
  // (consecutive threads on consecutive rows) fall in distinct banks
  static constexpr int ARS = BH | 1, WRS = BN | 1;
  static constexpr size_t SMEM = sizeof(double) * (NSB * (size_t)NST + 2 * (size_t)BN * ARS + 2 * (size_t)BN * WRS);
  static_assert(NTHR <= 512 && NXI <= NTHR, "one item a thread in every phase");
};

// y = K x on the phi nodes; block b: xy block b % (nbx nby) (x fastest), z segment b / (nbx nby)
template <class TL>
__global__ void __launch_bounds__(TL::NTHR)
kron_kernel(const KronCoefT<double> cf, const KronGeom g, const double* __restrict__ x,
            double* __restrict__ y) {
  constexpr int P = TL::P, BN = TL::BN, BH = TL::BH, NTHR = TL::NTHR, NST = TL::NST, SPT = TL::SPT;
  constexpr int ARS = TL::ARS, WRS = TL::WRS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* stage0 = reinterpret_cast<double*>(smem_raw);   // [NSB][BH][BH]
  double* A = stage0 + TL::NSB * NST;                     // [BN][ARS]
  double* Bs = A + BN * ARS;
  double* W1 = Bs + BN * ARS;                             // [BN][WRS]
  double* W2 = W1 + BN * WRS;

  const int tid = threadIdx.x, nxy = g.nbx * g.nby, zsi = blockIdx.x / nxy, bxy = blockIdx.x - zsi * nxy;
  const int x0 = (bxy % g.nbx) * BN, y0 = (bxy / g.nbx) * BN;
  const int c0 = zsi * g.zseg, c1 = min(c0 + g.zseg, g.nz);
  const int cb = c0 > 0 ? c0 - 1 : 0;
  const int gbeg = cb * P, gend = c1 * P;
  const int64_t plane_nodes = (int64_t)g.NX * g.NY;

  // staging offsets within a plane (per thread, once)
  int64_t s_off[SPT];
#pragma unroll
  for (int i = 0; i < SPT; ++i) {
    const int e = tid + i * NTHR, ec = e < NST ? e : 0;
    s_off[i] = pmod(x0 - P + ec % BH, g.NX) + (int64_t)g.NX * pmod(y0 - P + ec / BH, g.NY);
  }
  auto stage_plane = [&](int gz) {
    double* dst = stage0 + (gz - gbeg) % TL::NSB * NST;
    const double* src = x + gz * plane_nodes;
#pragma unroll
    for (int i = 0; i < SPT; ++i) {
      const int e = tid + i * NTHR;
      if (e < NST) cp_async<8>(dst + e, src + s_off[i], 8);
    }
  };

  // the thread's output node
  const int ox = tid % BN, oy = tid / BN;
  const bool own = tid < TL::NZI && x0 + ox < g.NX && y0 + oy < g.NY;
  const int ow = tid < TL::NZI ? oy * WRS + ox : 0;
  double* out = y + (x0 + ox) + (int64_t)g.NX * (y0 + oy);
  double acc[P + 1];
#pragma unroll
  for (int j = 0; j <= P; ++j) acc[j] = 0.0;
  // planes this segment writes
  auto write_plane = [&](int gz, int j) {
    if (own && ((gz >= c0 * P && gz < c1 * P) || (gz == g.nz * P && c1 == g.nz))) out[gz * plane_nodes] = acc[j];
  };
  // z contraction of the in-plane results of the plane with local index K (compile time, so
  // every coefficient is an immediate operand) into the layer accumulators
  auto plane_z = [&](auto kc, double a, double b) {
    constexpr int K = decltype(kc)::value;
    if constexpr (K <= P) {
#pragma unroll
      for (int j = 0; j <= P; ++j) {
        acc[j] = __fma_rn(cf.AzKs[j][K], a, acc[j]);
        acc[j] = __fma_rn(cf.AzMs[j][K], b, acc[j]);
      }
    }
  };
  auto dispatch_z = [&](int k, double a, double b) {
    switch (k) {
      case 0: plane_z(std::integral_constant<int, 0>{}, a, b); break;
      case 1: plane_z(std::integral_constant<int, 1>{}, a, b); break;
      case 2: plane_z(std::integral_constant<int, 2>{}, a, b); break;
      case 3: plane_z(std::integral_constant<int, 3>{}, a, b); break;
      case 4: plane_z(std::integral_constant<int, 4>{}, a, b); break;
      case 5: plane_z(std::integral_constant<int, 5>{}, a, b); break;
      case 6: plane_z(std::integral_constant<int, 6>{}, a, b); break;
      default: break;
    }
  };

  const int yh = tid % BH, yc = tid / BH * P;   // y-phase item: halo column, first row of the cell
  const int xr = tid % BN, xc = tid / BN * P;   // x-phase item: row, first node of the cell

  stage_plane(gbeg);
  cp_commit();
  int c = cb;
  for (int gz = gbeg; gz <= gend; ++gz) {
    const int k = gz - c * P;
    if (gz < gend) {
      stage_plane(gz + 1);
      cp_commit();
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const double* st = stage0 + (gz - gbeg) % TL::NSB * NST;
    // phase Y: a = AyM u, b = AyK u along y for every halo x
    if (tid < TL::NYI) {
      double u[P + 1], prv[P];
#pragma unroll
      for (int kk = 0; kk <= P; ++kk) u[kk] = st[(yc + P + kk) * BH + yh];
#pragma unroll
      for (int kk = 0; kk < P; ++kk) prv[kk] = st[(yc + kk) * BH + yh];
#pragma unroll
      for (int j = 0; j < P; ++j) {
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int kk = 0; kk <= P; ++kk) {
          a = __fma_rn(cf.AyM[j][kk], u[kk], a);
          b = __fma_rn(cf.AyK[j][kk], u[kk], b);
        }
        if (j == 0) {
#pragma unroll
          for (int kk = 0; kk < P; ++kk) {
            a = __fma_rn(cf.AyM[P][kk], prv[kk], a);
            b = __fma_rn(cf.AyK[P][kk], prv[kk], b);
          }
          a = __fma_rn(cf.AyM[P][P], u[0], a);
          b = __fma_rn(cf.AyK[P][P], u[0], b);
        }
        A[(yc + j) * ARS + yh] = a;
        Bs[(yc + j) * ARS + yh] = b;
      }
    }
    __syncthreads();
    // phase X: W1 = AxM a, W2 = AxK a + AxM b along x for every owned y
    if (tid < TL::NXI) {
      const double* ar = A + xr * ARS + xc;
      const double* br = Bs + xr * ARS + xc;
      double ao[P + 1], bo[P + 1];
#pragma unroll
      for (int kk = 0; kk <= P; ++kk) {
        ao[kk] = ar[P + kk];
        bo[kk] = br[P + kk];
      }
#pragma unroll
      for (int j = 0; j < P; ++j) {
        double u = 0.0, v = 0.0;
#pragma unroll
        for (int kk = 0; kk <= P; ++kk) {
          u = __fma_rn(cf.AxM[j][kk], ao[kk], u);
          v = __fma_rn(cf.AxK[j][kk], ao[kk], v);
          v = __fma_rn(cf.AxM[j][kk], bo[kk], v);
        }
        if (j == 0) {
#pragma unroll
          for (int kk = 0; kk < P; ++kk) {
            u = __fma_rn(cf.AxM[P][kk], ar[kk], u);
            v = __fma_rn(cf.AxK[P][kk], ar[kk], v);
            v = __fma_rn(cf.AxM[P][kk], br[kk], v);
          }
          u = __fma_rn(cf.AxM[P][P], ao[0], u);
          v = __fma_rn(cf.AxK[P][P], ao[0], v);
          v = __fma_rn(cf.AxM[P][P], bo[0], v);
        }
        W1[xr * WRS + xc + j] = u;
        W2[xr * WRS + xc + j] = v;
      }
    }
    __syncthreads();
    const double w1 = W1[ow], w2 = W2[ow];
    dispatch_z(k, w1, w2);
    if (k == P) {
      // the layer is complete: its first P planes are final; the top plane's sum becomes the
      // bottom accumulator of the next layer
#pragma unroll
      for (int j = 0; j < P; ++j) write_plane(c * P + j, j);
      acc[0] = acc[P];
#pragma unroll
      for (int j = 1; j <= P; ++j) acc[j] = 0.0;
      ++c;
      if (c < c1) dispatch_z(0, w1, w2);
    }
  }
  // the last processed plane (gend = c1 P) is final only if it is the top face
  write_plane(gend, 0);
}

// Dynamic shared memory limit, and the largest shared-memory carveout so that the residency
// of these kernels is set by registers and their own shared memory, not by the L1 split.
template <typename K>
inline fe_status kron_func_setup(K kern, size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fe_fail(FE_ECUDA, "kernel attributes: %s", cudaGetErrorString(e));
  }
  return FE_OK;
}

inline int device_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 152;
  }
  return sms;
}

// z segments are halved while the grid has fewer than four CTAs an SM
template <class TL>
fe_status kron_launch(const KronCoef& cf, KronGeom g, const double* x, double* y, cudaStream_t st) {
  const int nx = g.NX / g.p, ny = g.NY / g.p;
  g.bx = g.by = TL::B;
  g.nbx = (nx + TL::B - 1) / TL::B;
  g.nby = (ny + TL::B - 1) / TL::B;
  const int64_t base = (int64_t)g.nbx * g.nby, want = 4 * (int64_t)device_sms();
  g.zseg = g.nz;
  while (g.zseg > 2 && base * ((g.nz + g.zseg - 1) / g.zseg) < want) g.zseg = (g.zseg + 1) / 2;
  const int64_t total = base * ((g.nz + g.zseg - 1) / g.zseg);
  if (total > 0x7fffffffLL) return fe_fail(FE_EINVAL, "grid too large");
  FE_TRY(kron_func_setup(kron_kernel<TL>, TL::SMEM));
  kron_kernel<TL><<<(unsigned)total, TL::NTHR, TL::SMEM, st>>>(convert_coef<double>(cf), g, x, y);
  fe_count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fe_fail(FE_ECUDA, "kron kernel launch: %s", cudaGetErrorString(e));
  return FE_OK;
}

}  // namespace fe
