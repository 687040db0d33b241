// Single-vector stiffness product y = K x in double for the Poisson residuals and the CG of
// Section 2.3, cell by cell like the float one (fe_kcell.cu): strips of cells along x, three
// line contractions a cell into the discontinuous node grid, then per-node sums of the cell
// copies, lower cells first (bitwise repeatable).
//
// FP64 issue bounds it (this GPU starts a double FMA of a warp every sixteen cycles an SM), so
// the arithmetic is kept short.  With the GLL weights W taken out, K1 = W K', and the exact
// mass is M1 = W P with P = 1 - s q^T: it differs from the GLL rule in the L_p . L_p product
// only (q_k = w_k P_p(x_k), s_j = p (p + 1) / (2 (2 p + 1)) P_p(x_j)), so a mass line costs a dot
// product and an update.  A cell product is then 168 double operations a line triple (at p = 5)
// where dense mass lines take 252, and it has no halo: 160 + 16 us a product on the
// 16 x 16 x 48-cell p = 5 slab (1.54 M nodes, 48 operations a node, 0.87 of the FP64 rate that a
// DGEMM reaches), where the sweep kernel, with its halo columns, segment overlap and idle
// lanes, takes 377 us.
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
  k_cell64_apply<P><<<dim3((m->nx + S::CX - 1) / S::CX, m->ny, m->nz), S::NTHR, 0, m->stream>>>(
      cf, x, yc, m->nx, m->ny, m->NX, m->NY);
  fe_count_launch();
  k_cell64_gather<P><<<dim3((m->NX + 31) / 32, (m->NY + 7) / 8, m->NZ < 65535 ? m->NZ : 65535),
                       dim3(32, 8), 0, m->stream>>>(yc, y, m->nx, m->ny, m->nz, m->NX, m->NY);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

}  // namespace

// y = K x; *done is false (nothing enqueued) when the scratch of (p + 1)^3 doubles a cell is
// neither there nor to be had now (a capturing stream, no memory) or the grid would be too
// large: the caller then takes the sweep kernel, which needs no scratch
fe_status fe_kcell_apply_f64(fe_mesh* m, const double* x, double* y, bool* done) {
  *done = false;
  if (m->ny > 65535 || m->nz > 65535) return FE_OK;
  const size_t bytes = 2 * fe_kcell_scratch_bytes(m);
  if (m->ws_bytes[WS_KCELL] < bytes) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    FE_CUDA(cudaStreamIsCapturing(m->stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) return FE_OK;
  }
  void* w = nullptr;
  const fe_status st = fe_ws(m, WS_KCELL, bytes, &w);
  if (st == FE_ENOMEM) return FE_OK;
  FE_TRY(st);
  double* yc = static_cast<double*>(w);
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
