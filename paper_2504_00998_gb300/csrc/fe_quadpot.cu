// Potential term integrated by Gauss quadrature: the consistent (cell-matrix) form of the
// potential in the discretised Kohn-Sham operator of Section 2.3,
//   V_IJ = int N_I V_eff N_J dx = sum_cells sum_q w_q |J| V_e(x_q) N_I(x_q) N_J(x_q),
// with V_eff given at the (p+1)^3 Gauss-Legendre points of every cell.  Each cell's matrix
// is V_e = B^T diag(W_e) B with B = B1 (x) B1 (x) B1 the interpolation from the cell's GLL
// nodes to its Gauss points, so it is applied without being stored: per cell and vector,
// three line contractions to the Gauss points, the pointwise weight W_e = w |J| V_e, and
// three transposed contractions back (6 (p+1)^4 FMAs instead of (p+1)^6 for a stored
// matrix, and no matrix traffic).  The scaled operator adds
//   Y += alpha M^-1/2 V M^-1/2 X
// to the output of the sum-factorised kinetic operator (which then runs with a zero
// collocated potential and only the Chebyshev shift on its diagonal).
//
// Assembly is deterministic: the cells are processed in colour passes such that no two cells
// of one pass share a node (parity of cx, cy, cz; a third x (y) class holds the last cell when
// nx (ny) is odd, since the periodic wrap joins it to cell 0), and a cell that meets itself
// across the periodic wrap (nx or ny = 1) folds its two copies of a node before writing.
#include <cmath>
#include <vector>

#include <type_traits>

#include "fe_blas.cuh"
#include "fe_gll_tables.h"
#include "fe_internal.h"

namespace {

template <typename T>
struct QuadLanes;
template <>
struct QuadLanes<float> {
  static constexpr int v = 32;   // vector lanes per CTA
  using V16 = float4;            // one 16-byte access
};
template <>
struct QuadLanes<double> {
  static constexpr int v = 16;
  using V16 = double2;
};

// thread layout of one cell: a thread per 16-byte lane group of a line (N1^2 lines per
// direction), rounded up to whole warps
template <typename T, int P>
struct QuadShape {
  static constexpr int N1 = P + 1, NN = N1 * N1 * N1;
  static constexpr int VC = QuadLanes<T>::v;
  static constexpr int VW = 16 / (int)sizeof(T);   // lanes per 16-byte access
  static constexpr int G = VC / VW;                // lane groups per node
  static constexpr int LINES = N1 * N1 * G;
  static constexpr int NT = (LINES + 31) / 32 * 32;
  static constexpr int RES = 896 / NT < 16 ? 896 / NT : 16;   // 28 warps an SM: 72 registers
};

struct QuadPass {
  int nx, ny, NX, NY, gz_lo, gz_hi;
  int ox, oy, oz;         // colour class per direction (2: the last cell of an odd row)
  int cntx, cnty, cntz;   // cells of the class per direction
  int foldx, foldy;       // a single cell along x (y): local nodes 0 and p coincide
};

__device__ __forceinline__ int class_cell(int t, int cls, int n) {
  return cls == 2 ? n - 1 : 2 * t + cls;
}

// lanes of one 16-byte access; float lanes in pairs, so that an FMA instruction takes two
__device__ __forceinline__ unsigned long long pack(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack(unsigned long long r) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(r));
  return f;
}
template <typename T>
struct Lanes;
template <>
struct Lanes<float> {
  unsigned long long a, b;
  static __device__ __forceinline__ Lanes of(const float4& f) { return {pack(f.x, f.y), pack(f.z, f.w)}; }
  __device__ __forceinline__ float4 v16() const {
    const float2 x = unpack(a), y = unpack(b);
    return make_float4(x.x, x.y, y.x, y.y);
  }
};
template <>
struct Lanes<double> {
  double a, b;
  static __device__ __forceinline__ Lanes of(const double2& f) { return {f.x, f.y}; }
  __device__ __forceinline__ double2 v16() const { return make_double2(a, b); }
};
using LF = Lanes<float>;
using LD = Lanes<double>;
__device__ __forceinline__ unsigned long long fma2(unsigned long long x, unsigned long long y,
                                                   unsigned long long z) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long x, unsigned long long y) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long x, unsigned long long y) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ LF lfma(float c, const LF& x, const LF& y) {
  const unsigned long long s = pack(c, c);
  return {fma2(s, x.a, y.a), fma2(s, x.b, y.b)};
}
__device__ __forceinline__ LF lmul(float c, const LF& x) {
  const unsigned long long s = pack(c, c);
  return {mul2(s, x.a), mul2(s, x.b)};
}
__device__ __forceinline__ LF ladd(const LF& x, const LF& y) { return {add2(x.a, y.a), add2(x.b, y.b)}; }
__device__ __forceinline__ LF lsub(const LF& x, const LF& y) { return lfma(-1.f, y, x); }
__device__ __forceinline__ LD lfma(double c, const LD& x, const LD& y) { return {fma(c, x.a, y.a), fma(c, x.b, y.b)}; }
__device__ __forceinline__ LD lmul(double c, const LD& x) { return {c * x.a, c * x.b}; }
__device__ __forceinline__ LD ladd(const LD& x, const LD& y) { return {x.a + y.a, x.b + y.b}; }
__device__ __forceinline__ LD lsub(const LD& x, const LD& y) { return {x.a - y.a, x.b - y.b}; }
__device__ __forceinline__ float4 vzero(float) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 vzero(double) { return make_double2(0.0, 0.0); }
// keep the first k lanes (k < lanes of the access), zero the rest
__device__ __forceinline__ float4 vkeep(float4 x, int k) {
  if (k < 4) x.w = 0.f;
  if (k < 3) x.z = 0.f;
  if (k < 2) x.y = 0.f;
  return x;
}
__device__ __forceinline__ double2 vkeep(double2 x, int k) {
  if (k < 2) x.y = 0.0;
  return x;
}
__device__ __forceinline__ void vstore_first(float* p, const float4& x, int k) {
  p[0] = x.x;
  if (k > 1) p[1] = x.y;
  if (k > 2) p[2] = x.z;
}
__device__ __forceinline__ void vstore_first(double* p, const double2& x, int) { p[0] = x.x; }

// Lines.  The interpolation table commutes with the mirror image of the cell, B[p-q][p-e] = B[q][e],
// so a line contraction is split into the even parts u_k + u_{p-k} and the odd ones u_k - u_{p-k}:
// (p + 1)^2 / 2 FMAs and 2 (p + 1) sums for (p + 1)^2 FMAs, and half the constants.
// Coefficient (j, k) of the even (odd = 0) or odd part; TR: of the transposed table.
template <int P, bool TR>
__device__ __forceinline__ constexpr double quad_c(int odd, int j, int k) {
  const double a = TR ? fe::gauss_b<P>(k, j) : fe::gauss_b<P>(j, k);
  if (k == P - k) return a;
  const double b = TR ? fe::gauss_b<P>(P - k, j) : fe::gauss_b<P>(j, P - k);
  return odd ? 0.5 * (a - b) : 0.5 * (a + b);
}
template <typename T, int P>
struct Parts {
  static constexpr int E = (P + 2) / 2, O = (P + 1) / 2;
  Lanes<T> e[E], o[O];
  __device__ __forceinline__ void split(const Lanes<T> (&u)[P + 1]) {
#pragma unroll
    for (int k = 0; k < O; ++k) {
      e[k] = ladd(u[k], u[P - k]);
      o[k] = lsub(u[k], u[P - k]);
    }
    if constexpr (E > O) e[O] = u[O];
  }
  // parts of output q
  template <bool TR>
  __device__ __forceinline__ Lanes<T> even(int q) const {
    Lanes<T> s = lmul((T)quad_c<P, TR>(0, q, 0), e[0]);
#pragma unroll
    for (int k = 1; k < E; ++k) s = lfma((T)quad_c<P, TR>(0, q, k), e[k], s);
    return s;
  }
  template <bool TR>
  __device__ __forceinline__ Lanes<T> odd(int q) const {
    Lanes<T> s = lmul((T)quad_c<P, TR>(1, q, 0), o[0]);
#pragma unroll
    for (int k = 1; k < O; ++k) s = lfma((T)quad_c<P, TR>(1, q, k), o[k], s);
    return s;
  }
};

// u <- B u (TR: B^T u)
template <typename T, int P, bool TR>
__device__ __forceinline__ void line(Lanes<T> (&u)[P + 1]) {
  Parts<T, P> s;
  s.split(u);
#pragma unroll
  for (int q = 0; q < Parts<T, P>::E; ++q) {
    const Lanes<T> ev = s.template even<TR>(q);
    if (q < Parts<T, P>::O) {
      const Lanes<T> od = s.template odd<TR>(q);
      u[q] = ladd(ev, od);
      u[P - q] = lsub(ev, od);
    } else {
      u[q] = ev;
    }
  }
}
// u <- B^T diag(w) B u, w[q * stride] the weight of point q
template <typename T, int P>
__device__ __forceinline__ void line_weighted(Lanes<T> (&u)[P + 1], const T* __restrict__ w, int stride) {
  using S = Parts<T, P>;
  S s;
  s.split(u);
  Lanes<T> e[S::E], o[S::O];
#pragma unroll
  for (int q = 0; q < S::E; ++q) {
    Lanes<T> g = s.template even<false>(q), d;
    if (q < S::O) {
      const Lanes<T> od = s.template odd<false>(q);
      const Lanes<T> lo = lmul(w[q * stride], ladd(g, od)), hi = lmul(w[(P - q) * stride], lsub(g, od));
      g = ladd(lo, hi);
      d = lsub(lo, hi);
    } else {
      g = lmul(w[q * stride], g);
    }
#pragma unroll
    for (int k = 0; k < S::E; ++k) {
      const T c = (T)quad_c<P, true>(0, k, q);
      e[k] = q ? lfma(c, g, e[k]) : lmul(c, g);
    }
    if (q < S::O) {
#pragma unroll
      for (int k = 0; k < S::O; ++k) {
        const T c = (T)quad_c<P, true>(1, k, q);
        o[k] = q ? lfma(c, d, o[k]) : lmul(c, d);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < S::O; ++k) {
    u[k] = ladd(e[k], o[k]);
    u[P - k] = lsub(e[k], o[k]);
  }
  if constexpr (S::E > S::O) u[S::O] = e[S::O];
}

// the calling thread's line of the cell block in shared memory ([node][lane], 16-byte groups)
template <typename T, int P, int D>
struct LineAt {
  using S = QuadShape<T, P>;
  using V = typename QuadLanes<T>::V16;
  static constexpr int STRIDE = D == 0 ? 1 : D == 1 ? S::N1 : S::N1 * S::N1;
  V* at;
  int base;
  // (a, b): the two other local indices
  __device__ __forceinline__ LineAt(T* buf, int a, int b, int grp)
      : at(reinterpret_cast<V*>(buf)),
        base(D == 0 ? (b * S::N1 + a) * S::N1 : D == 1 ? b * S::N1 * S::N1 + a : b * S::N1 + a) {
    at += base * S::G + grp;
  }
  __device__ __forceinline__ void load(Lanes<T> (&u)[P + 1]) const {
#pragma unroll
    for (int e = 0; e <= P; ++e) u[e] = Lanes<T>::of(at[e * STRIDE * S::G]);
  }
  __device__ __forceinline__ void store(const Lanes<T> (&u)[P + 1]) const {
#pragma unroll
    for (int e = 0; e <= P; ++e) at[e * STRIDE * S::G] = u[e].v16();
  }
};

// Y += alpha M^-1/2 V M^-1/2 X on the cells of one colour; a CTA takes one cell and VC lanes.
// What bounds it: memory latency, two trips a CTA (X at the start, Y at the end) with 27 warps an
// SM to cover them, at 4.6 TB/s of its algorithmic bytes on 16 x 16 x 16 cells p = 5, 256 float
// vectors: 74 us a colour pass, where dense lines, unpaired float FMAs, a shared round trip
// between the two z contractions and a node table that the X loads waited for took 83.  The
// z contraction, the weights and the transposed contraction are one step in registers, and
// every thread rewrites its own lines only: one buffer, four barriers.  A filter of degree 8 on
// that slab, kinetic part included: 9.75 -> 9.14 ms.
template <typename T, int P, bool PREFETCH>
__global__ void __launch_bounds__(QuadShape<T, P>::NT, QuadShape<T, P>::RES)
k_quad_apply(const QuadPass g, const T* __restrict__ X, T* __restrict__ Y, int64_t ld, int64_t nvec,
             const T* __restrict__ W, const T* __restrict__ rsq, T alpha) {
  using S = QuadShape<T, P>;
  using V = typename QuadLanes<T>::V16;
  using L = Lanes<T>;
  constexpr int N1 = S::N1, NN = S::NN, VC = S::VC, VW = S::VW, G = S::G, NT = S::NT;
  constexpr int SLOTS = NN * G;                      // 16-byte slots of the cell block
  constexpr int IT = (SLOTS + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  T* Ws = buf + NN * VC;                             // w |J| V at the Gauss points

  int t = blockIdx.x;
  const int tx = t % g.cntx;
  t /= g.cntx;
  const int ty = t % g.cnty, tz = t / g.cnty;
  const int cx = class_cell(tx, g.ox, g.nx), cy = class_cell(ty, g.oy, g.ny);
  const int cz = 2 * tz + g.oz;
  const int64_t cell = ((int64_t)cz * g.ny + cy) * g.nx + cx;
  const int64_t v0 = (int64_t)blockIdx.y * VC;
  const int64_t plane = (int64_t)g.NX * g.NY;
  const int tid = threadIdx.x;

  for (int e = tid; e < NN; e += NT) Ws[e] = W[cell * NN + e];
  const int grp = tid % G, ab = tid / G;
  const int la = ab % N1, lb = ab / N1;     // (j, k) of the thread's x line
  const int64_t vv = v0 + (int64_t)grp * VW;
  const int64_t left = nvec - vv;           // lanes of the group that are vectors
  const bool act = tid < S::LINES;
  // first node of the row of nodes j, k (-1 outside the stored planes), and the x index of node i
  auto row_of = [&](int j, int k) {
    const int gz = cz * P + k;
    int gy = cy * P + j;
    gy -= gy >= g.NY ? g.NY : 0;
    return gz >= g.gz_lo && gz <= g.gz_hi ? (gz - g.gz_lo) * plane + (int64_t)gy * g.NX : (int64_t)-1;
  };
  auto x_of = [&](int i) {
    const int gx = cx * P + i;
    return i == P && gx >= g.NX ? gx - g.NX : gx;
  };
  const int64_t row = act ? row_of(la, lb) : -1;
  const bool on = row >= 0 && left > 0;
  // x lines straight from global memory: u = M^-1/2 X on the line's nodes (every load of
  // the thread in flight before the first use; zero on Dirichlet faces and past the last
  // vector; a row holds ld >= the group's end, so the whole group is in bounds), then the
  // forward x contraction.  A thread reads and writes its own lines only, so one buffer does.
  // The Y lines, needed at the end, are asked for now where they are not in L2 anyway.
  L u[N1];
  if (act) {
    V in[N1];
    T r[N1];
#pragma unroll
    for (int e = 0; e < N1; ++e) {
      in[e] = vzero(T(0));
      r[e] = T(0);
      if (on) {
        const int64_t n = row + x_of(e);
        in[e] = *reinterpret_cast<const V*>(X + n * ld + vv);
        r[e] = rsq[n];
        if (PREFETCH && grp == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(Y + n * ld + vv));
      }
    }
#pragma unroll
    for (int e = 0; e < N1; ++e) {
      if (left < VW) in[e] = vkeep(in[e], left > 0 ? (int)left : 0);
      u[e] = lmul(r[e], L::of(in[e]));
    }
    line<T, P, false>(u);
    LineAt<T, P, 0>(buf, la, lb, grp).store(u);
  }
  __syncthreads();
  if (act) {
    const LineAt<T, P, 1> at(buf, la, lb, grp);
    at.load(u);
    line<T, P, false>(u);
    at.store(u);
  }
  __syncthreads();
  if (act) {
    const LineAt<T, P, 2> at(buf, la, lb, grp);
    at.load(u);
    line_weighted<T, P>(u, Ws + at.base, N1 * N1);
    at.store(u);
  }
  __syncthreads();
  if (act) {
    const LineAt<T, P, 1> at(buf, la, lb, grp);
    at.load(u);
    line<T, P, true>(u);
    at.store(u);
  }
  __syncthreads();
  if (!g.foldy) {
    // transposed x contraction in registers and Y += alpha M^-1/2 (.) along the line; a
    // single cell along x (foldx) adds its two copies of node 0 before writing it once
    if (act) {
      LineAt<T, P, 0>(buf, la, lb, grp).load(u);
      line<T, P, true>(u);
      if (g.foldx) u[0] = ladd(u[P], u[0]);
      if (!on) return;
      V yv[N1];
      T r[N1];
#pragma unroll
      for (int e = 0; e < N1; ++e) {
        const int64_t n = row + x_of(e);
        yv[e] = vzero(T(0));
        r[e] = rsq[n];
        if (!(g.foldx && e == P)) yv[e] = *reinterpret_cast<const V*>(Y + n * ld + vv);
      }
#pragma unroll
      for (int e = 0; e < N1; ++e) {
        if (g.foldx && e == P) continue;
        const V o = lfma(alpha * r[e], u[e], L::of(yv[e])).v16();
        T* yp = Y + (row + x_of(e)) * ld + vv;
        if (left >= VW)
          *reinterpret_cast<V*>(yp) = o;
        else
          vstore_first(yp, o, (int)left);
      }
    }
    return;
  }
  // a single cell along y: the two copies of each j = 0 node are in different x lines, so
  // the block goes back to the nodes in shared memory and is folded there
  if (act) {
    const LineAt<T, P, 0> at(buf, la, lb, grp);
    at.load(u);
    line<T, P, true>(u);
    at.store(u);
  }
  __syncthreads();
  V* A = reinterpret_cast<V*>(buf);
  if (g.foldx) {
    for (int idx = tid; idx < N1 * N1 * G; idx += NT) {
      const int gg = idx % G, r = idx / G;   // r = (k, j)
      const L x = L::of(A[(r * N1) * G + gg]), y = L::of(A[(r * N1 + P) * G + gg]);
      A[(r * N1) * G + gg] = ladd(x, y).v16();
    }
    __syncthreads();
  }
  for (int idx = tid; idx < N1 * N1 * G; idx += NT) {
    const int gg = idx % G, r = idx / G;
    const int i = r % N1, k = r / N1;
    const L x = L::of(A[(k * N1 * N1 + i) * G + gg]), y = L::of(A[(k * N1 * N1 + P * N1 + i) * G + gg]);
    A[(k * N1 * N1 + i) * G + gg] = ladd(x, y).v16();
  }
  __syncthreads();
  // Y += alpha M^-1/2 (V u): all loads of Y first, then the updates
  {
    V yv[IT];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int sl = tid + it * NT;
      yv[it] = vzero(T(0));
      if (sl < SLOTS) {
        const int e = sl / G, ww = (sl % G) * VW;
        const int64_t nr = row_of((e / N1) % N1, e / (N1 * N1));
        if (nr >= 0 && v0 + ww < nvec)
          yv[it] = *reinterpret_cast<const V*>(Y + (nr + x_of(e % N1)) * ld + v0 + ww);
      }
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int sl = tid + it * NT;
      if (sl >= SLOTS) continue;
      const int e = sl / G, ww = (sl % G) * VW;
      const int i = e % N1, j = (e / N1) % N1;
      if ((g.foldx && i == P) || j == P) continue;
      const int64_t nr = row_of(j, e / (N1 * N1)), n = nr + x_of(i);
      if (nr < 0 || v0 + ww >= nvec) continue;
      const V o = lfma(alpha * rsq[n], L::of(A[sl]), L::of(yv[it])).v16();
      T* yp = Y + n * ld + v0 + ww;
      const int64_t rem = nvec - (v0 + ww);
      if (rem >= VW)
        *reinterpret_cast<V*>(yp) = o;
      else
        vstore_first(yp, o, (int)rem);
    }
  }
}

template <typename T, int P>
size_t quad_smem() {
  using S = QuadShape<T, P>;
  return sizeof(T) * ((size_t)S::NN * S::VC + S::NN);
}

template <typename T, int P>
fe_status quad_apply_p(fe_mesh* m, const T* X, T* Y, int64_t ld, int64_t nvec, const T* W,
                       const T* rsq, T alpha) {
  using S = QuadShape<T, P>;
  constexpr int VC = S::VC;
  const size_t smem = quad_smem<T, P>();
  // Y's lines are asked for at the start where the block exceeds L2 (524 MB: 1164 -> 1114 us an
  // H X); smaller blocks only pay for the instructions (94 MB: 247 -> 256 us, 71 MB: 207 -> 211).
  int l2 = 0;
  if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, m->device) != cudaSuccess) cudaGetLastError();
  const bool beyond = (double)m->n_psi * (double)ld * sizeof(T) > (double)l2;
  auto kern = beyond ? k_quad_apply<T, P, true> : k_quad_apply<T, P, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fe_fail(FE_ECUDA, "quadrature potential: %s", cudaGetErrorString(e));
  }
  if (((uintptr_t)X) % 16 || ((uintptr_t)Y) % 16 || (ld * (int64_t)sizeof(T)) % 16)
    return fe_fail(FE_EINVAL, "quadrature potential: blocks need 16-byte aligned rows");
  const int64_t nchunk = (nvec + VC - 1) / VC;
  if (nchunk > 65535) return fe_fail(FE_EINVAL, "quadrature potential: too many vectors");
  // colour classes per direction: {class, cells}
  auto classes = [](int n, bool periodic, int* cls, int* cnt) {
    if (!periodic) {
      cls[0] = 0; cnt[0] = (n + 1) / 2;
      cls[1] = 1; cnt[1] = n / 2;
      return 2;
    }
    if (n == 1) { cls[0] = 0; cnt[0] = 1; return 1; }
    if (n % 2 == 0) {
      cls[0] = 0; cnt[0] = n / 2;
      cls[1] = 1; cnt[1] = n / 2;
      return 2;
    }
    cls[0] = 0; cnt[0] = (n - 1) / 2;
    cls[1] = 1; cnt[1] = (n - 1) / 2;
    cls[2] = 2; cnt[2] = 1;
    return 3;
  };
  int clx[3], cnx[3], cly[3], cny[3], clz[3], cnz[3];
  const int ncx = classes(m->nx, true, clx, cnx);
  const int ncy = classes(m->ny, true, cly, cny);
  const int ncz = classes(m->nz, false, clz, cnz);
  QuadPass g;
  g.nx = m->nx; g.ny = m->ny; g.NX = m->NX; g.NY = m->NY;
  g.gz_lo = m->gz_lo; g.gz_hi = m->gz_hi;
  g.foldx = m->nx == 1; g.foldy = m->ny == 1;
  for (int a = 0; a < ncz; ++a)
    for (int b = 0; b < ncy; ++b)
      for (int c = 0; c < ncx; ++c) {
        const int64_t cells = (int64_t)cnx[c] * cny[b] * cnz[a];
        if (cells == 0) continue;
        if (cells > 0x7fffffffLL) return fe_fail(FE_EINVAL, "quadrature potential: mesh too large");
        g.ox = clx[c]; g.oy = cly[b]; g.oz = clz[a];
        g.cntx = cnx[c]; g.cnty = cny[b]; g.cntz = cnz[a];
        kern<<<dim3((unsigned)cells, (unsigned)nchunk), S::NT, smem, m->stream>>>(
            g, X, Y, ld, nvec, W, rsq, alpha);
        fe_count_launch();
      }
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

template <typename T>
fe_status quad_apply_t(fe_mesh* m, const T* X, T* Y, int64_t ld, int64_t nvec, const T* W,
                       const T* rsq, T alpha) {
  switch (m->p) {
    case 1: return quad_apply_p<T, 1>(m, X, Y, ld, nvec, W, rsq, alpha);
    case 2: return quad_apply_p<T, 2>(m, X, Y, ld, nvec, W, rsq, alpha);
    case 3: return quad_apply_p<T, 3>(m, X, Y, ld, nvec, W, rsq, alpha);
    case 4: return quad_apply_p<T, 4>(m, X, Y, ld, nvec, W, rsq, alpha);
    case 5: return quad_apply_p<T, 5>(m, X, Y, ld, nvec, W, rsq, alpha);
    case 6: return quad_apply_p<T, 6>(m, X, Y, ld, nvec, W, rsq, alpha);
    default: return fe_fail(FE_EUNSUPPORTED, "p = %d", m->p);
  }
}

// n-point Gauss-Legendre rule on [-1, 1]: Newton's method on P_n from the Chebyshev-like
// first guesses cos(pi (i + 3/4) / (n + 1/2)), P_n and P_n' from the three-term recurrence;
// weights 2 / ((1 - x^2) P_n'(x)^2).  Ascending order.
void gauss_legendre(int n, double* x, double* w) {
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[n - 1 - i] = z;
    w[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

static_assert(FE_MAXN1 == 7, "the weight kernel takes seven Gauss weights");

// W[e][q] = w_a w_b w_c |J| Vq[e][q], q = a + nq (b + nq c); float copy alongside
__global__ void k_quad_weights(const double* __restrict__ Vq, int64_t n, int nq, double detJ,
                               double w0, double w1, double w2, double w3, double w4, double w5,
                               double w6, double* __restrict__ W, float* __restrict__ Wf) {
  const double wq[7] = {w0, w1, w2, w3, w4, w5, w6};
  const int nn = nq * nq * nq;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(i % nn);
    const int a = q % nq, b = (q / nq) % nq, c = q / (nq * nq);
    const double v = wq[a] * wq[b] * wq[c] * detJ * Vq[i];
    W[i] = v;
    Wf[i] = (float)v;
  }
}

// M^-1/2 at psi nodes from the lumped mass at phi nodes
__global__ void k_psi_rsq(const double* __restrict__ mass, int64_t off, int64_t n,
                          double* __restrict__ r, float* __restrict__ rf) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double s = 1.0 / sqrt(mass[i + off]);
    r[i] = s;
    rf[i] = (float)s;
  }
}

__global__ void k_zero2(double* __restrict__ a, float* __restrict__ b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    a[i] = 0.0;
    b[i] = 0.0f;
  }
}

struct InterpB {
  double B[FE_MAXN1][FE_MAXN1];
};

// f at every cell's Gauss points from its nodal values on phi nodes
__global__ void k_interp_quad(const InterpB cb, const double* __restrict__ f, int p, int nx,
                              int ny, int NX, int NY, int64_t ncells, double* __restrict__ out) {
  const int n1 = p + 1, nn = n1 * n1 * n1;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ncells * nn;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cell = i / nn;
    const int q = (int)(i % nn);
    const int a = q % n1, b = (q / n1) % n1, c = q / (n1 * n1);
    const int cx = (int)(cell % nx), cy = (int)((cell / nx) % ny);
    const int cz = (int)(cell / ((int64_t)nx * ny));
    double s = 0.0;
    for (int k = 0; k < n1; ++k) {
      const int64_t gz = (int64_t)cz * p + k;
      double sy = 0.0;
      for (int j = 0; j < n1; ++j) {
        int gy = cy * p + j;
        gy -= gy >= NY ? NY : 0;
        const double* row = f + (gz * NY + gy) * NX;
        double sx = 0.0;
        for (int l = 0; l < n1; ++l) {
          int gx = cx * p + l;
          gx -= gx >= NX ? NX : 0;
          sx = fma(cb.B[a][l], row[gx], sx);
        }
        sy = fma(cb.B[b][j], sx, sy);
      }
      s = fma(cb.B[c][k], sy, s);
    }
    out[i] = s;
  }
}

}  // namespace

void fe_quad_setup_basis(fe_mesh* m) {
  const int n1 = m->p + 1;
  double x[FE_MAXN1], w[FE_MAXN1];
  gauss_legendre(n1, x, w);
  for (int q = 0; q < FE_MAXN1; ++q) {
    m->wq[q] = q < n1 ? w[q] : 0.0;
    for (int i = 0; i < FE_MAXN1; ++i) {
      double l = 0.0;
      if (q < n1 && i < n1) {
        l = 1.0;
        for (int j = 0; j < n1; ++j)
          if (j != i) l *= (x[q] - m->xi[j]) / (m->xi[i] - m->xi[j]);
      }
      m->Bq[q][i] = l;
    }
  }
}

void fe_quad_free(fe_mesh* m) {
  cudaFree(m->d_qW);
  cudaFree(m->d_qW_f);
  cudaFree(m->d_rsq);
  cudaFree(m->d_rsq_f);
  m->d_qW = nullptr;
  m->d_qW_f = nullptr;
  m->d_rsq = nullptr;
  m->d_rsq_f = nullptr;
  m->has_quad = false;
}

fe_status fe_quad_apply(fe_mesh* m, const void* X, void* Y, int64_t nvec, int64_t ld,
                        double alpha, bool dbl) {
  if (!m->has_quad) return FE_OK;
  if (dbl)
    return quad_apply_t<double>(m, (const double*)X, (double*)Y, ld, nvec, m->d_qW, m->d_rsq,
                                alpha);
  return quad_apply_t<float>(m, (const float*)X, (float*)Y, ld, nvec, m->d_qW_f, m->d_rsq_f,
                             (float)alpha);
}

extern "C" fe_status fe_set_potential_quad(fe_mesh* m, const double* vq) {
  if (!m || !vq) return fe_fail(FE_EINVAL, "fe_set_potential_quad: null argument");
  if (m->p > 6) return fe_fail(FE_EUNSUPPORTED, "fe_set_potential_quad: p = %d", m->p);
  FE_TRY(fe_activate(m));
  const int n1 = m->p + 1;
  const int64_t nq = m->n_cells * (int64_t)n1 * n1 * n1;
  if (!m->d_veff) {
    if (cudaMalloc(&m->d_veff, m->n_psi * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&m->d_veff_f, m->n_psi * sizeof(float)) != cudaSuccess) {
      cudaGetLastError();
      return fe_fail(FE_ENOMEM, "potential allocation failed");
    }
  }
  if (!m->d_qW) {
    if (cudaMalloc(&m->d_qW, nq * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&m->d_qW_f, nq * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&m->d_rsq, m->n_psi * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&m->d_rsq_f, m->n_psi * sizeof(float)) != cudaSuccess) {
      cudaGetLastError();
      fe_quad_free(m);
      return fe_fail(FE_ENOMEM, "quadrature potential allocation failed");
    }
  }
  cudaStream_t st = m->stream;
  // the collocated potential is zero: the kinetic kernel keeps only the Chebyshev shift
  k_zero2<<<fe::grid_for(m->n_psi), 256, 0, st>>>(m->d_veff, m->d_veff_f, m->n_psi);
  fe_count_launch();
  const double* w = m->wq;
  k_quad_weights<<<fe::grid_for(nq), 256, 0, st>>>(vq, nq, n1, m->J, w[0], w[1], w[2], w[3],
                                                   w[4], w[5], w[6], m->d_qW, m->d_qW_f);
  fe_count_launch();
  k_psi_rsq<<<fe::grid_for(m->n_psi), 256, 0, st>>>(
      m->d_mass, (int64_t)m->gz_lo * m->NX * m->NY, m->n_psi, m->d_rsq, m->d_rsq_f);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  m->has_potential = true;
  m->has_quad = true;
  return FE_OK;
}

extern "C" fe_status fe_interp_quad(fe_mesh* m, const double* f_phi, double* out) {
  if (!m || !f_phi || !out) return fe_fail(FE_EINVAL, "fe_interp_quad: null argument");
  FE_TRY(fe_activate(m));
  InterpB cb;
  for (int q = 0; q < FE_MAXN1; ++q)
    for (int i = 0; i < FE_MAXN1; ++i) cb.B[q][i] = m->Bq[q][i];
  const int n1 = m->p + 1;
  const int64_t total = m->n_cells * (int64_t)n1 * n1 * n1;
  k_interp_quad<<<fe::grid_for(total), 256, 0, m->stream>>>(cb, f_phi, m->p, m->nx, m->ny, m->NX,
                                                           m->NY, m->n_cells, out);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}
