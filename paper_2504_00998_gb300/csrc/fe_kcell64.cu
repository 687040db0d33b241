// Single-vector stiffness product y = K x in double for the Poisson residuals and the CG of
// Section 2.3, cell by cell like the float one (fe_kcell.cu): strips of cells along x, three
// line contractions a cell into the discontinuous node grid, then per-node sums of the cell
// copies, lower cells first (bitwise repeatable).
//
// FP64 issue bounds it (this GPU starts a double FMA of a warp every sixteen cycles an SM), so
// the arithmetic is kept short.  With the GLL weights W taken out, K1 = W K', and the exact
// mass is M1 = W P with P = 1 - s q^T: it differs from the GLL rule in the L_p . L_p product
// only (q_k = w_k P_p(x_k), s_j = p (p + 1) / (2 (2 p + 1)) P_p(x_j)), so a mass line costs a dot
// product and an update, and it has no halo.  Even p: 168 double operations a line triple where
// dense mass lines take 252 (at p = 5).  Odd p: the mirror parts below, 120 operations.  A product
// on the 16 x 16 x 48-cell p = 5 slab (1.54 M nodes) takes 129 + 16 us (160 + 16 without the
// mirror parts; 333 in the scratch-free sweep kernel, with its halo columns, segment overlap and
// idle lanes).
#include <cstdint>

#include "fe_internal.h"
#include "fe_kcell.cuh"

namespace {

using fe_kc::CellStrip;

struct Cell64 {
  double Kx[FE_MAXN1][FE_MAXN1], Ky[FE_MAXN1][FE_MAXN1], Kz[FE_MAXN1][FE_MAXN1];   // scale * W^-1 K1
  double q[FE_MAXN1], s[FE_MAXN1], w[FE_MAXN1];
};

Cell64 cell64(const fe_mesh* m) {
  Cell64 c = {};
  const int p = m->p;
  const double ax = m->h[1] * m->h[2] / (2.0 * m->h[0]), ay = m->h[0] * m->h[2] / (2.0 * m->h[1]),
               az = m->h[0] * m->h[1] / (2.0 * m->h[2]);
  for (int j = 0; j <= p; ++j) {
    // P_p(x_j) by the Legendre recurrence
    double p0 = 1.0, p1 = m->xi[j];
    for (int k = 2; k <= p; ++k) {
      const double p2 = ((2.0 * k - 1.0) * m->xi[j] * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    c.w[j] = m->w[j];
    c.q[j] = m->w[j] * p1;
    c.s[j] = p * (p + 1.0) / (2.0 * (2.0 * p + 1.0)) * p1;
    for (int k = 0; k <= p; ++k) {
      const double v = m->K1[j][k] / m->w[j];
      c.Kx[j][k] = ax * v;
      c.Ky[j][k] = ay * v;
      c.Kz[j][k] = az * v;
    }
  }
  return c;
}

template <int P>
__global__ void __launch_bounds__(CellStrip<P>::NTHR)
k_cell64_apply(const Cell64 cf, const double* __restrict__ x, double* __restrict__ ycell, int nx,
               int ny, int NX, int NY) {
  using S = CellStrip<P>;
  constexpr int N1 = S::N1, CX = S::CX, UW = S::UW;
  __shared__ double U[S::U_FLOATS];
  __shared__ double A[S::A_FLOATS];
  __shared__ double B[S::A_FLOATS];
  const int tid = threadIdx.x, cx0 = blockIdx.x * CX, cy = blockIdx.y, cz = blockIdx.z;
  for (int e = tid; e < S::U_FLOATS; e += S::NTHR) U[e] = x[fe_kc::strip_node<P>(e, cx0, cy, cz, NX, NY)];
  __syncthreads();
  const bool active = tid < S::LINES;
  // y lines: A = P u, B = Ky u
  if (active) {
    const int lx = tid % N1, c = (tid / N1) % CX, lz = tid / (N1 * CX);
    double in[N1], d = 0.0;
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      in[k] = U[(lz * N1 + k) * UW + c * P + lx];
      d = fma(cf.q[k], in[k], d);
    }
#pragma unroll
    for (int j = 0; j < N1; ++j) {
      double b = 0.0;
#pragma unroll
      for (int k = 0; k < N1; ++k) b = fma(cf.Ky[j][k], in[k], b);
      const int o = ((lz * N1 + j) * CX + c) * N1 + lx;
      A[o] = fma(-cf.s[j], d, in[j]);
      B[o] = b;
    }
  }
  __syncthreads();
  // x lines, in place: A <- P a, B <- Kx a + P b
  if (active) {
    const int c = tid % CX, ly = (tid / CX) % N1, lz = tid / (CX * N1);
    const int base = ((lz * N1 + ly) * CX + c) * N1;
    double a[N1], b[N1], d = 0.0, e = 0.0;
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      a[k] = A[base + k];
      b[k] = B[base + k];
      d = fma(cf.q[k], a[k], d);
      e = fma(cf.q[k], b[k], e);
    }
#pragma unroll
    for (int j = 0; j < N1; ++j) {
      double v = fma(-cf.s[j], e, b[j]);
#pragma unroll
      for (int k = 0; k < N1; ++k) v = fma(cf.Kx[j][k], a[k], v);
      A[base + j] = fma(-cf.s[j], d, a[j]);
      B[base + j] = v;
    }
  }
  __syncthreads();
  // z lines: y_e = W (x) W (x) W (Kz A + P B), to the discontinuous grid
  if (active) {
    const int lx = tid % N1, c = (tid / N1) % CX, ly = tid / (N1 * CX);
    const int cx = cx0 + c;
    if (cx < nx) {
      double u[N1], v[N1], e = 0.0;
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        const int o = ((k * N1 + ly) * CX + c) * N1 + lx;
        u[k] = A[o];
        v[k] = B[o];
        e = fma(cf.q[k], v[k], e);
      }
      double wl = 0.0, wy = 0.0;
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        wl = k == lx ? cf.w[k] : wl;
        wy = k == ly ? cf.w[k] : wy;
      }
      const double wxy = wl * wy;
      const int64_t dnx = (int64_t)nx * N1, dny = (int64_t)ny * N1;
      double* out = ycell + ((int64_t)cz * N1 * dny + (int64_t)cy * N1 + ly) * dnx + (int64_t)cx * N1 + lx;
#pragma unroll
      for (int j = 0; j < N1; ++j) {
        double r = fma(-cf.s[j], e, v[j]);
#pragma unroll
        for (int k = 0; k < N1; ++k) r = fma(cf.Kz[j][k], u[k], r);
        out[j * dny * dnx] = wxy * cf.w[j] * r;
      }
    }
  }
}

// ---- odd p: mirror parts ------------------------------------------------------------------------
// K' commutes with the mirror image of a cell and q, s are odd, so a line of p + 1 values is
// kept as its (p + 1) / 2 even parts u_k + u_{p-k} (at k) and its odd ones u_k - u_{p-k} (at p - k):
// a stiffness line then takes half the operations and a mass line too.  In the three directions
// the parts are taken and put back once: a thread of the y and the z pass has the four mirror
// images of a line.  (Even p has a middle line without an image, which would leave those threads
// a third idle: 5 x 5 lines are 9 quadruples.)
template <int P>
struct Mirror {
  static constexpr int N1 = P + 1, H = N1 / 2;
  static constexpr int CX = P == 1 ? 64 : P == 3 ? 16 : 7;   // cells a block: two whole warps
  static constexpr int QUADS = CX * H * H, NTHR = (QUADS + 31) / 32 * 32;
  static constexpr int NODES = CX * N1 * N1 * N1, ROWS = CX * N1 * N1;
  static_assert(P % 2 == 1, "no middle node");
};

constexpr int MAXH = FE_MAXN1 / 2;
struct Mirror64 {
  double Kx[2][MAXH][MAXH], Ky[2][MAXH][MAXH], Kz[2][MAXH][MAXH];   // even, odd parts
  double q[MAXH], s[MAXH], w[MAXH];
};

Mirror64 mirror64(const Cell64& c, int p) {
  Mirror64 t = {};
  for (int j = 0; j < (p + 1) / 2; ++j) {
    t.q[j] = 2.0 * c.q[j];
    t.s[j] = c.s[j];
    t.w[j] = c.w[j];
    for (int k = 0; k < (p + 1) / 2; ++k)
      for (int o = 0; o < 2; ++o) {
        t.Kx[o][j][k] = o ? c.Kx[j][k] - c.Kx[j][p - k] : c.Kx[j][k] + c.Kx[j][p - k];
        t.Ky[o][j][k] = o ? c.Ky[j][k] - c.Ky[j][p - k] : c.Ky[j][k] + c.Ky[j][p - k];
        t.Kz[o][j][k] = o ? c.Kz[j][k] - c.Kz[j][p - k] : c.Kz[j][k] + c.Kz[j][p - k];
      }
  }
  return t;
}

// out += K in
template <int P>
__device__ __forceinline__ void mirror_k(const double (&K)[2][MAXH][MAXH], const double (&in)[P + 1],
                                         double (&out)[P + 1]) {
#pragma unroll
  for (int j = 0; j < (P + 1) / 2; ++j)
#pragma unroll
    for (int k = 0; k < (P + 1) / 2; ++k) {
      out[j] = fma(K[0][j][k], in[k], out[j]);
      out[P - j] = fma(K[1][j][k], in[P - k], out[P - j]);
    }
}
// the mass of in, in place: the odd parts only
template <int P>
__device__ __forceinline__ void mirror_mass(const Mirror64& cf, double (&in)[P + 1]) {
  double d = 0.0;
#pragma unroll
  for (int k = 0; k < (P + 1) / 2; ++k) d = fma(cf.q[k], in[P - k], d);
#pragma unroll
  for (int k = 0; k < (P + 1) / 2; ++k) in[P - k] = fma(-cf.s[k], d, in[P - k]);
}

template <int P>
__global__ void __launch_bounds__(Mirror<P>::NTHR)
k_cell64_mirror(const Mirror64 cf, const double* __restrict__ x, double* __restrict__ ycell, int nx,
                int ny, int cells, int NX, int NY) {
  using M = Mirror<P>;
  constexpr int N1 = M::N1, CX = M::CX, H = M::H, NT = M::NTHR;
  __shared__ double A[M::NODES];   // [lz][ly][cell][lx]: the nodes, then A
  __shared__ double B[M::NODES];
  __shared__ int at[3][CX];        // the cells' indices (the last cell again past the end)
  const int tid = threadIdx.x, first = blockIdx.x * CX;
  for (int c = tid; c < CX; c += NT) {
    const int id = min(first + c, cells - 1), row = id / nx;
    at[0][c] = id - row * nx;
    at[2][c] = row / ny;
    at[1][c] = row - at[2][c] * ny;
  }
  __syncthreads();
#pragma unroll 8
  for (int e = tid; e < M::NODES; e += NT) {
    const int lx = e % N1, c = (e / N1) % CX, ly = (e / (N1 * CX)) % N1, lz = e / (N1 * CX * N1);
    int gx = at[0][c] * P + lx, gy = at[1][c] * P + ly;
    gx -= gx >= NX ? NX : 0;
    gy -= gy >= NY ? NY : 0;
    A[e] = x[((int64_t)(at[2][c] * P + lz) * NY + gy) * NX + gx];
  }
  __syncthreads();
  const int k0 = tid % H, cell = (tid / H) % CX, k1 = tid / (H * CX);
  // y lines, the mirror images in x and z: to parts in three directions (eight times the
  // parts), then A = P u, B = Ky u
  if (tid < M::QUADS) {
    double* a = A + cell * N1;
    double* b = B + cell * N1;
    double in[4][N1];   // 2 (odd in z) + (odd in x)
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      const double* lo = a + (k1 * N1 + k) * CX * N1;
      const double* hi = a + ((P - k1) * N1 + k) * CX * N1;
      const double e0 = lo[k0] + lo[P - k0], o0 = lo[k0] - lo[P - k0];
      const double e1 = hi[k0] + hi[P - k0], o1 = hi[k0] - hi[P - k0];
      in[0][k] = e0 + e1;
      in[1][k] = o0 + o1;
      in[2][k] = e0 - e1;
      in[3][k] = o0 - o1;
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int o = (l & 2 ? P - k1 : k1) * N1 * CX * N1 + (l & 1 ? P - k0 : k0);
      double u[N1], v[N1];
#pragma unroll
      for (int k = 0; k < H; ++k) {
        u[k] = in[l][k] + in[l][P - k];
        u[P - k] = in[l][k] - in[l][P - k];
        v[k] = v[P - k] = 0.0;
      }
      mirror_k<P>(cf.Ky, u, v);
      mirror_mass<P>(cf, u);
#pragma unroll
      for (int j = 0; j < N1; ++j) {
        a[o + j * CX * N1] = u[j];
        b[o + j * CX * N1] = v[j];
      }
    }
  }
  __syncthreads();
  // x lines, in place: A <- P a, B <- Kx a + P b
  for (int r = tid; r < M::ROWS; r += NT) {
    double a[N1], b[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      a[k] = A[r * N1 + k];
      b[k] = B[r * N1 + k];
    }
    mirror_mass<P>(cf, b);
    mirror_k<P>(cf.Kx, a, b);
    mirror_mass<P>(cf, a);
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      A[r * N1 + k] = a[k];
      B[r * N1 + k] = b[k];
    }
  }
  __syncthreads();
  // z lines, the mirror images in x and y: y_e = W (x) W (x) W (Kz A + P B), back to nodal
  // values, to the discontinuous grid
  if (tid < M::QUADS && first + cell < cells) {
    double r[4][N1];   // 2 (odd in y) + (odd in x)
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int o = ((l & 2 ? P - k1 : k1) * CX + cell) * N1 + (l & 1 ? P - k0 : k0);
      double u[N1], v[N1];
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        u[k] = A[o + k * N1 * CX * N1];
        v[k] = B[o + k * N1 * CX * N1];
      }
      mirror_mass<P>(cf, v);
      mirror_k<P>(cf.Kz, u, v);
#pragma unroll
      for (int k = 0; k < H; ++k) {
        r[l][k] = v[k] + v[P - k];
        r[l][P - k] = v[k] - v[P - k];
      }
    }
    double w0 = 0.0, w1 = 0.0;
#pragma unroll
    for (int k = 0; k < H; ++k) {
      w0 = k == k0 ? cf.w[k] : w0;
      w1 = k == k1 ? cf.w[k] : w1;
    }
    const double wxy = 0.125 * (w0 * w1);
    const int64_t dnx = (int64_t)nx * N1, dny = (int64_t)ny * N1;
    double* out = ycell + ((int64_t)at[2][cell] * N1 * dny + (int64_t)at[1][cell] * N1) * dnx +
                  (int64_t)at[0][cell] * N1;
#pragma unroll
    for (int j = 0; j < N1; ++j) {
      const double w = wxy * cf.w[j < H ? j : P - j];
      const double e0 = r[0][j] + r[1][j], e1 = r[0][j] - r[1][j];
      const double o0 = r[2][j] + r[3][j], o1 = r[2][j] - r[3][j];
      double* lo = out + (j * dny + k1) * dnx;
      double* hi = out + (j * dny + P - k1) * dnx;
      lo[k0] = w * (e0 + o0);
      lo[P - k0] = w * (e1 + o1);
      hi[k0] = w * (e0 - o0);
      hi[P - k0] = w * (e1 - o1);
    }
  }
}

// y at node (gx, gy, gz): the sum of its one to eight copies, lower cells first
template <int P>
__global__ void __launch_bounds__(256)
k_cell64_gather(const double* __restrict__ ycell, double* __restrict__ y, int nx, int ny, int nz,
                int NX, int NY) {
  constexpr int N1 = P + 1;
  const int gx = blockIdx.x * 32 + threadIdx.x, gy = blockIdx.y * 8 + threadIdx.y;
  if (gx >= NX || gy >= NY) return;
  int dx[2], dy[2];
  const int nxc = fe_kc::cell_copies_periodic<P>(gx, nx, dx);
  const int nyc = fe_kc::cell_copies_periodic<P>(gy, ny, dy);
  const int64_t dnx = (int64_t)nx * N1, dny = (int64_t)ny * N1;
  for (int gz = blockIdx.z; gz <= nz * P; gz += gridDim.z) {
    const int c = gz / P, l = gz - c * P;
    int dz[2], nzc = 0;
    if (l == 0 && c > 0) dz[nzc++] = (c - 1) * N1 + P;
    if (c < nz) dz[nzc++] = c * N1 + l;
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      if (a >= nzc) break;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if (b >= nyc) break;
        const double* row = ycell + ((int64_t)dz[a] * dny + dy[b]) * dnx;
#pragma unroll
        for (int e = 0; e < 2; ++e)
          if (e < nxc) s += row[dx[e]];
      }
    }
    y[((int64_t)gz * NY + gy) * NX + gx] = s;
  }
}

template <int P>
fe_status run(fe_mesh* m, const double* x, double* y, double* yc) {
  using S = CellStrip<P>;
  const Cell64 cf = cell64(m);
  if constexpr (P % 2) {
    using M = Mirror<P>;
    const int cells = m->nx * m->ny * m->nz;
    k_cell64_mirror<P><<<(cells + M::CX - 1) / M::CX, M::NTHR, 0, m->stream>>>(
        mirror64(cf, P), x, yc, m->nx, m->ny, cells, m->NX, m->NY);
  } else {
    k_cell64_apply<P><<<dim3((m->nx + S::CX - 1) / S::CX, m->ny, m->nz), S::NTHR, 0, m->stream>>>(
        cf, x, yc, m->nx, m->ny, m->NX, m->NY);
  }
  fe_count_launch();
  k_cell64_gather<P><<<dim3((m->NX + 31) / 32, (m->NY + 7) / 8, m->NZ < 65535 ? m->NZ : 65535),
                       dim3(32, 8), 0, m->stream>>>(yc, y, m->nx, m->ny, m->nz, m->NX, m->NY);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

}  // namespace

fe_status fe_kcell64_reserve(fe_mesh* m, double** ws) {
  *ws = nullptr;
  const size_t bytes = 2 * fe_kcell_scratch_bytes(m);   // (p + 1)^3 doubles a cell
  if (m->ws_bytes[WS_KCELL64] < bytes) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    FE_CUDA(cudaStreamIsCapturing(m->stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) return FE_OK;
  }
  void* w = nullptr;
  const fe_status st = fe_ws(m, WS_KCELL64, bytes, &w);
  if (st == FE_ENOMEM) return FE_OK;
  FE_TRY(st);
  *ws = static_cast<double*>(w);
  return FE_OK;
}

namespace {

// Whether a product enqueued now has the scratch to itself.  Products on one stream follow one
// another, and the library's own stream follows the caller's; but after fe_mesh_set_stream the
// former stream's products may still be running, and a graph that the caller captures may be
// replayed on any stream.
fe_status scratch_ours(fe_mesh* m, bool* ours) {
  const cudaStream_t user = (cudaStream_t)m->desc.stream;
  *ours = !m->kcell64_pending || m->kcell64_user == user;
  if (*ours && m->stream != m->aux_stream) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    FE_CUDA(cudaStreamIsCapturing(m->stream, &cs));
    *ours = cs == cudaStreamCaptureStatusNone;
  }
  if (*ours) {
    m->kcell64_pending = true;
    m->kcell64_user = user;
  }
  return FE_OK;
}

}  // namespace

// y = K x; *done is false (nothing enqueued) when the scratch is neither there nor to be had now,
// when another stream or a captured graph may use it at the same time, or when the grid would be
// too large: the caller then takes the sweep kernel, which needs no scratch
fe_status fe_kcell_apply_f64(fe_mesh* m, const double* x, double* y, bool* done) {
  *done = false;
  if (m->ny > 65535 || m->nz > 65535) return FE_OK;
  bool ours = false;
  FE_TRY(scratch_ours(m, &ours));
  if (!ours) return FE_OK;
  double* yc = nullptr;
  FE_TRY(fe_kcell64_reserve(m, &yc));
  if (!yc) return FE_OK;
  *done = true;
  switch (m->p) {
    case 1: return run<1>(m, x, y, yc);
    case 2: return run<2>(m, x, y, yc);
    case 3: return run<3>(m, x, y, yc);
    case 4: return run<4>(m, x, y, yc);
    case 5: return run<5>(m, x, y, yc);
    default: return run<6>(m, x, y, yc);
  }
}
