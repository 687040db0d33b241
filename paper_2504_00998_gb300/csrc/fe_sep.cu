// Poisson solve by a separable preconditioner (Section 2.3: K phi = c on the slab mesh).
//
// On the uniform tensor-product mesh K = ax K1 (x) M1 (x) M1 + ay M1 (x) K1 (x) M1 +
// az M1 (x) M1 (x) K1, also when whole z planes are constrained (CEF, CPD): the free planes
// only shorten the z chain.  With the generalised eigenvectors of each direction,
// K1 V = M1 V diag(lambda), V^T M1 V = 1, the inverse is
//   K^-1 = V diag(1 / (ax lx + ay ly + az lz)) V^T,   V = Vx (x) Vy (x) Vz
// (the fast diagonalisation of Lynch, Rice and Thomas, Numer. Math. 6, 1964): six small dense
// products along the axes.  They run in float as the preconditioner of a CG in double: every
// iteration takes the residual down by about 1e5 (the float rounding of the transforms), so
// the double stopping test is met after two or three iterations, where the iteration with
// the plane and mode coarse spaces takes hundreds.  A local bias region (L-CPD) constrains
// part of some planes; those planes then stay in the z chain as if free, the preconditioned
// residual is masked, and the CG takes about twenty iterations, whatever the mesh size.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fe_blas.cuh"
#include "fe_sep.cuh"

namespace {

// ---- generalised eigenproblem of one chain (host, once per mesh and constraint set) ----------
using Mat = std::vector<double>;   // row-major n x n

// Eigenpairs of the symmetric matrix A (destroyed): ascending order is not needed.  Q holds
// the eigenvectors as rows.  Householder tridiagonalisation, then the implicit QR iteration
// with Wilkinson's shift (Golub and Van Loan, Matrix Computations, 8.3), its rotations
// applied to rows so that every inner loop runs over contiguous memory.
bool symmetric_eigen(Mat& A, int n, std::vector<double>& d, Mat& Q) {
  std::vector<double> e(n, 0.0), beta(n, 0.0), v(n), w(n);
  Mat H((size_t)n * n, 0.0);   // row k: the Householder vector of column k
  d.assign(n, 0.0);
  for (int k = 0; k + 2 < n; ++k) {
    double nrm = 0.0;
    for (int i = k + 1; i < n; ++i) { v[i] = A[(size_t)k * n + i]; nrm += v[i] * v[i]; }
    nrm = std::sqrt(nrm);
    e[k] = 0.0;
    if (nrm == 0.0) continue;
    const double alpha = v[k + 1] > 0.0 ? -nrm : nrm;
    e[k] = alpha;
    v[k + 1] -= alpha;
    double vv = 0.0;
    for (int i = k + 1; i < n; ++i) vv += v[i] * v[i];
    beta[k] = vv > 0.0 ? 2.0 / vv : 0.0;
    double vw = 0.0;
    for (int i = k + 1; i < n; ++i) {
      const double* row = &A[(size_t)i * n];
      double s = 0.0;
      for (int j = k + 1; j < n; ++j) s += row[j] * v[j];
      w[i] = beta[k] * s;
      vw += w[i] * v[i];
    }
    const double c = 0.5 * beta[k] * vw;
    for (int i = k + 1; i < n; ++i) w[i] -= c * v[i];
    for (int i = k + 1; i < n; ++i) {
      double* row = &A[(size_t)i * n];
      const double vi = v[i], wi = w[i];
      for (int j = k + 1; j < n; ++j) row[j] -= vi * w[j] + wi * v[j];
    }
    for (int i = k + 1; i < n; ++i) H[(size_t)k * n + i] = v[i];
  }
  if (n > 1) e[n - 2] = A[(size_t)(n - 2) * n + n - 1];
  for (int i = 0; i < n; ++i) d[i] = A[(size_t)i * n + i];
  // rows of Q: (H_0 H_1 ...)^T, built from the last reflector on: Q <- Q (1 - beta v v^T)
  Q.assign((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i) Q[(size_t)i * n + i] = 1.0;
  for (int k = n - 3; k >= 0; --k) {
    if (beta[k] == 0.0) continue;
    const double* h = &H[(size_t)k * n];
    for (int i = k + 1; i < n; ++i) {
      double* row = &Q[(size_t)i * n];
      double s = 0.0;
      for (int j = k + 1; j < n; ++j) s += row[j] * h[j];
      s *= beta[k];
      for (int j = k + 1; j < n; ++j) row[j] -= s * h[j];
    }
  }
  int hi = n - 1, guard = 60 * n + 60;
  while (hi > 0) {
    const double tiny = 2.3e-16 * (std::fabs(d[hi]) + std::fabs(d[hi - 1]));
    if (std::fabs(e[hi - 1]) <= tiny) { e[hi - 1] = 0.0; --hi; continue; }
    int lo = hi - 1;
    while (lo > 0 && std::fabs(e[lo - 1]) > 2.3e-16 * (std::fabs(d[lo]) + std::fabs(d[lo - 1]))) --lo;
    if (--guard < 0) return false;
    const double del = 0.5 * (d[hi - 1] - d[hi]), eh = e[hi - 1];
    const double mu = d[hi] - eh * eh / (del + (del >= 0.0 ? 1.0 : -1.0) * std::hypot(del, eh));
    double x = d[lo] - mu, y = e[lo];
    for (int k = lo; k < hi; ++k) {
      const double r = std::hypot(x, y);
      const double c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? -y / r : 0.0;
      if (k > lo) e[k - 1] = r;
      const double dk = d[k], d1 = d[k + 1], ek = e[k];
      d[k] = c * c * dk - 2.0 * c * s * ek + s * s * d1;
      d[k + 1] = s * s * dk + 2.0 * c * s * ek + c * c * d1;
      e[k] = c * s * (dk - d1) + (c * c - s * s) * ek;
      if (k + 1 < hi) { x = e[k]; y = -s * e[k + 1]; e[k + 1] *= c; }
      double* q0 = &Q[(size_t)k * n];
      double* q1 = q0 + n;
      for (int j = 0; j < n; ++j) {
        const double a = q0[j], b = q1[j];
        q0[j] = c * a - s * b;
        q1[j] = s * a + c * b;
      }
    }
  }
  return true;
}

// K u = lambda M u for symmetric K and positive definite M: rows of V with V M V^T = 1
bool generalised_eigen(const Mat& K, const Mat& M, int n, std::vector<double>& lam, Mat& V) {
  Mat L(M);   // lower Cholesky factor, row by row
  for (int i = 0; i < n; ++i)
    for (int j = 0; j <= i; ++j) {
      double s = L[(size_t)i * n + j];
      const double *a = &L[(size_t)i * n], *b = &L[(size_t)j * n];
      for (int k = 0; k < j; ++k) s -= a[k] * b[k];
      if (i == j) {
        if (!(s > 0.0)) return false;
        L[(size_t)i * n + i] = std::sqrt(s);
      } else {
        L[(size_t)i * n + j] = s / L[(size_t)j * n + j];
      }
    }
  // C = L^-1 K L^-T: forward substitution on the rows of K, then on the rows of the transpose
  auto forward = [&](Mat& B) {   // B <- L^-1 B
    for (int i = 0; i < n; ++i) {
      double* bi = &B[(size_t)i * n];
      for (int k = 0; k < i; ++k) {
        const double l = L[(size_t)i * n + k];
        if (l == 0.0) continue;
        const double* bk = &B[(size_t)k * n];
        for (int j = 0; j < n; ++j) bi[j] -= l * bk[j];
      }
      const double r = 1.0 / L[(size_t)i * n + i];
      for (int j = 0; j < n; ++j) bi[j] *= r;
    }
  };
  Mat C(K);
  forward(C);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < i; ++j) std::swap(C[(size_t)i * n + j], C[(size_t)j * n + i]);
  forward(C);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < i; ++j) {
      const double s = 0.5 * (C[(size_t)i * n + j] + C[(size_t)j * n + i]);
      C[(size_t)i * n + j] = C[(size_t)j * n + i] = s;
    }
  if (!symmetric_eigen(C, n, lam, V)) return false;
  // rows of V: u = L^-T q, by back substitution
  for (int a = 0; a < n; ++a) {
    double* u = &V[(size_t)a * n];
    for (int i = n - 1; i >= 0; --i) {
      u[i] /= L[(size_t)i * n + i];
      const double x = u[i];
      const double* l = &L[(size_t)i * n];
      for (int k = 0; k < i; ++k) u[k] -= l[k] * x;
    }
  }
  return true;
}

// The chain's assembled 1D matrices on the nodes [lo, hi) of nc cells (periodic: all nc p
// nodes).  A chain that is its own mirror image splits into its even and odd parts, which
// quarters the work.
bool chain_eigen(const fe_mesh* m, int nc, bool periodic, int lo, int hi,
                 std::vector<double>& lam, Mat& V) {
  const int p = m->p, n = hi - lo, all = periodic ? nc * p : nc * p + 1;
  Mat K((size_t)n * n, 0.0), M((size_t)n * n, 0.0);
  for (int c = 0; c < nc; ++c)
    for (int i = 0; i <= p; ++i)
      for (int j = 0; j <= p; ++j) {
        const int a = (c * p + i) % all - lo, b = (c * p + j) % all - lo;
        if (a < 0 || a >= n || b < 0 || b >= n) continue;
        K[(size_t)a * n + b] += m->K1[i][j];
        M[(size_t)a * n + b] += m->M1[i][j];
      }
  auto mirror = [&](int i) { return periodic ? (n - i) % n : n - 1 - i; };
  bool symmetric = true;
  for (int i = 0; i < n && symmetric; ++i)
    for (int j = 0; j < n && symmetric; ++j) {
      const size_t a = (size_t)i * n + j, b = (size_t)mirror(i) * n + mirror(j);
      symmetric = std::fabs(K[a] - K[b]) <= 1e-11 * std::fabs(m->K1[0][0]) * p &&
                  std::fabs(M[a] - M[b]) <= 1e-13;
    }
  if (!symmetric) return generalised_eigen(K, M, n, lam, V);
  lam.clear();
  V.assign((size_t)n * n, 0.0);
  for (int part = 0; part < 2; ++part) {
    std::vector<int> rep;   // one node of each mirrored pair (and, even part, the fixed ones)
    for (int i = 0; i < n; ++i)
      if (i < mirror(i) || (part == 0 && i == mirror(i))) rep.push_back(i);
    const int nr = (int)rep.size();
    if (nr == 0) continue;
    Mat Kr((size_t)nr * nr), Mr((size_t)nr * nr);
    const double sg = part == 0 ? 1.0 : -1.0, h = std::sqrt(0.5);
    for (int a = 0; a < nr; ++a)
      for (int b = 0; b < nr; ++b) {
        const int i = rep[a], j = rep[b], mi = mirror(i), mj = mirror(j);
        const double ca = mi == i ? 1.0 : h, cb = mj == j ? 1.0 : h;
        auto red = [&](const Mat& A) {
          double s = A[(size_t)i * n + j];
          if (mj != j) s += sg * A[(size_t)i * n + mj];
          if (mi != i) s += sg * A[(size_t)mi * n + j];
          if (mi != i && mj != j) s += A[(size_t)mi * n + mj];
          return ca * cb * s;
        };
        Kr[(size_t)a * nr + b] = red(K);
        Mr[(size_t)a * nr + b] = red(M);
      }
    std::vector<double> lr;
    Mat Vr;
    if (!generalised_eigen(Kr, Mr, nr, lr, Vr)) return false;
    for (int e = 0; e < nr; ++e) {
      double* u = &V[lam.size() * (size_t)n];
      for (int a = 0; a < nr; ++a) {
        const int i = rep[a], mi = mirror(i);
        const double x = Vr[(size_t)e * nr + a];
        if (mi == i) {
          u[i] = x;
        } else {
          u[i] = h * x;
          u[mi] = sg * h * x;
        }
      }
      lam.push_back(lr[e]);
    }
  }
  return true;
}

// ---- reductions -----------------------------------------------------------------------------------
// FP64 adds are slow here (sixteen cycles a warp and SM), so a block's sum is one warp's work:
// each lane adds its share of the threads' terms in order, then a shuffle tree.  The total is
// valid in thread 0.  blockDim.x is 256.
__device__ __forceinline__ double block_total(double v) {
  __shared__ double s[256];
  s[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s[threadIdx.x + 32 * w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  __syncthreads();
  return t;
}
// Whether this block is the last of `blocks` to get here (every block's partials are then
// visible); it finishes the sum, and the ticket is ready for the next launch.
__device__ __forceinline__ bool last_block(unsigned int* ticket, unsigned int blocks) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1u) == blocks - 1;
    if (last) {
      *ticket = 0;
      __threadfence();
    }
  }
  __syncthreads();
  return last;
}
__device__ __forceinline__ double sum_partials(const double* part, int n) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) v += __ldcg(part + i);
  return block_total(v);
}

// scalars of the iteration: r.z, alpha, beta, |r|^2, and the tickets of the three reductions
struct Scalars {
  double rz, alpha, beta, rr;
  unsigned int ticket[3];
};

// ---- transforms -----------------------------------------------------------------------------
// Device tables of the plan (floats): V [node][mode] and its transpose for every direction
// and the eigenvalues with their mesh scale.
struct Tables {
  const float *Vx, *VxT, *Vy, *VyT, *Vz, *VzT, *lx, *ly, *lz;
};

struct Gemm {
  const float* W;        // the small matrix, row-major [K][M] (left) or [K][N] (right)
  const float* in;       // left: [batch][K][N]; right: [M][K]
  float* out;            // left: [batch][M][N]; right: [M][N]
  int M, N, K;
  int64_t in_batch, out_batch;
  // spectral scaling (left products of the z direction): rows are z modes, a column is
  // b NX + a; the part of eigenvalue zero, the constant's, is dropped
  const float *lx, *ly, *lz;
  int NX;
  // double ends of the x products
  const double* in_d;
  double* out_d;
  const unsigned char* mask;
  const double *r, *q;   // dot products r.z (and q.z unless null) of the written values
  double* part;          // [2][blocks]
  Scalars* s;
  int first;             // the first iteration: no direction to keep
};

enum { LEFT = 0, LEFT_SCALE = 1, RIGHT_IN = 2, RIGHT_OUT = 3 };   // (LEFT_SCALE: z products only)

constexpr int GT = 256, BK = 16;

// One 16 TM x 16 TN tile per block of 256 threads, TM x TN results a thread.  The products
// are 60 to 360 wide along every dimension, 0.25 to 0.75 GFLOP each on the benchmark slab and
// read from L2, so they are bound by FFMA issue and shared-memory reads (TM + TN words for
// TM TN FMAs); the tile follows the matrix size (tile_for) because padding to 64 or 96 costs
// more than the smaller tile does.
template <int TM, int TN, int MODE>
__global__ void __launch_bounds__(GT) k_sep_gemm(const Gemm g) {
  constexpr int BM = 16 * TM, BN = 16 * TN;
  constexpr bool RIGHT = MODE == RIGHT_IN || MODE == RIGHT_OUT;
  __shared__ float As[BK][BM + 1];
  __shared__ float Bs[BK][BN];
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  // right products: many row tiles, taken along x
  const int m0 = (RIGHT ? blockIdx.x : blockIdx.y) * BM;
  const int n0 = (RIGHT ? blockIdx.y : blockIdx.x) * BN;
  const float* in = RIGHT ? g.in : g.in + (int64_t)blockIdx.z * g.in_batch;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  float ra[TM], rb[TN];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if constexpr (RIGHT) {
        const int k = k0 + tx, r = m0 + ty + 16 * i;
        const int64_t at = (int64_t)r * g.K + k;
        const bool in_range = k < g.K && r < g.M;
        if constexpr (MODE == RIGHT_IN) ra[i] = in_range ? (float)g.in_d[at] : 0.f;
        else ra[i] = in_range ? in[at] : 0.f;
      } else {
        const int k = k0 + ty, m = m0 + tx + 16 * i;
        ra[i] = (k < g.K && m < g.M) ? g.W[(int64_t)k * g.M + m] : 0.f;
      }
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int k = k0 + ty, n = n0 + tx + 16 * j;
      const float* src = RIGHT ? g.W : in;
      rb[j] = (k < g.K && n < g.N) ? src[(int64_t)k * g.N + n] : 0.f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < g.K; k0 += BK) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if constexpr (RIGHT) As[tx][ty + 16 * i] = ra[i];
      else As[ty][tx + 16 * i] = ra[i];
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) Bs[ty][tx + 16 * j] = rb[j];
    __syncthreads();
    if (k0 + BK < g.K) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = __fmaf_rn(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  double rz = 0.0, qz = 0.0;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int mm = m0 + ty + 16 * i;
    if (mm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int nn = n0 + tx + 16 * j;
      if (nn >= g.N) continue;
      const int64_t at = (int64_t)mm * g.N + nn;
      if constexpr (MODE == RIGHT_OUT) {
        const double z = g.mask[at] ? 0.0 : (double)acc[i][j];
        g.out_d[at] = z;
        rz += g.r[at] * z;
        if (g.q) qz += g.q[at] * z;
      } else {
        g.out[(RIGHT ? 0 : (int64_t)blockIdx.z * g.out_batch) + at] = acc[i][j];
      }
    }
  }
  if constexpr (MODE == RIGHT_OUT) {
    // r.z and q.z; the last block takes the direction's beta = -alpha_old (q.z) / (r.z)_old
    // (the flexible form: the float preconditioner is symmetric to rounding only)
    const int nb = gridDim.x * gridDim.y, at = blockIdx.y * gridDim.x + blockIdx.x;
    rz = block_total(rz);
    qz = block_total(qz);
    if (t == 0) {
      g.part[at] = rz;
      g.part[nb + at] = qz;
    }
    if (last_block(&g.s->ticket[0], nb)) {
      rz = sum_partials(g.part, nb);
      qz = g.first ? 0.0 : sum_partials(g.part + nb, nb);
      if (t == 0) {
        Scalars* s = g.s;
        const double old = s->rz;
        s->beta = g.first || old == 0.0 ? 0.0 : -s->alpha * qz / old;
        s->rz = rz;
      }
    }
  }
}

// The z products (LEFT, LEFT_SCALE) at a larger tile: 64 x 128 a block, 4 x 8 results a thread
// read as three 16-byte words for 32 FMAs (nine words for 20 in k_sep_gemm).  M is the length
// of the z chain and N a whole plane: on the benchmark slab 237 to 241 x 6400, 200 blocks,
// 37 us a product against 43 (means of the two; the 5 x 4 tile of k_sep_gemm).
template <int MODE>
__global__ void __launch_bounds__(GT) k_sep_gemm_z(const Gemm g) {
  constexpr int BM = 64, BN = 128;
  __shared__ __align__(16) float As[BK][BM];
  __shared__ __align__(16) float Bs[BK][BN];
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  float acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  float ra[4], rb[8];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + t / 64 + 4 * i, m = m0 + t % 64;
      ra[i] = (k < g.K && m < g.M) ? g.W[(int64_t)k * g.M + m] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + t / 128 + 2 * i, n = n0 + t % 128;
      rb[i] = (k < g.K && n < g.N) ? g.in[(int64_t)k * g.N + n] : 0.f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < g.K; k0 += BK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) As[t / 64 + 4 * i][t % 64] = ra[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) Bs[t / 128 + 2 * i][t % 128] = rb[i];
    __syncthreads();
    if (k0 + BK < g.K) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][4 * ty]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k][4 * tx]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[k][64 + 4 * tx]);
      const float av[4] = {a.x, a.y, a.z, a.w};
      const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = __fmaf_rn(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int mm = m0 + 4 * ty + i;
    if (mm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int nn = n0 + (j < 4 ? 4 * tx + j : 60 + 4 * tx + j);
      if (nn >= g.N) continue;
      float v = acc[i][j];
      if constexpr (MODE == LEFT_SCALE) {
        const int bb = nn / g.NX, aa = nn - bb * g.NX;
        const float l = g.lz[mm] + (g.ly[bb] + g.lx[aa]);
        v = l > 0.f ? v / l : 0.f;
      }
      g.out[(int64_t)mm * g.N + nn] = v;
    }
  }
}

// 4, 5 or 6 results a thread along a dimension of n: the least padding, the larger tile on a tie
int tile_for(int64_t n) {
  int best = 4;
  int64_t waste = -1;
  for (int t : {6, 5, 4}) {
    const int64_t w = (n + 16 * t - 1) / (16 * t) * (16 * t);
    if (waste < 0 || w < waste) { waste = w; best = t; }
  }
  return best;
}

dim3 grid_of(bool right, int tm, int tn, const Gemm& g, int batch) {
  const unsigned bm = (unsigned)((g.M + 16 * tm - 1) / (16 * tm));
  const unsigned bn = (unsigned)((g.N + 16 * tn - 1) / (16 * tn));
  return right ? dim3(bm, bn, 1) : dim3(bn, bm, (unsigned)batch);
}

template <int MODE>
fe_status gemm(const Gemm& g, int batch, cudaStream_t st) {
  constexpr bool RIGHT = MODE == RIGHT_IN || MODE == RIGHT_OUT;
  const int tm = tile_for(g.M), tn = tile_for(g.N);
  const dim3 grid = grid_of(RIGHT, tm, tn, g, batch);
#define FE_SEP_CASE(a, b) \
  if (tm == a && tn == b) k_sep_gemm<a, b, MODE><<<grid, GT, 0, st>>>(g);
  FE_SEP_CASE(4, 4) FE_SEP_CASE(4, 5) FE_SEP_CASE(4, 6) FE_SEP_CASE(5, 4) FE_SEP_CASE(5, 5)
  FE_SEP_CASE(5, 6) FE_SEP_CASE(6, 4) FE_SEP_CASE(6, 5) FE_SEP_CASE(6, 6)
#undef FE_SEP_CASE
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

template <int MODE>
fe_status gemm_z(const Gemm& g, cudaStream_t st) {
  k_sep_gemm_z<MODE><<<dim3((g.N + 127) / 128, (g.M + 63) / 64), GT, 0, st>>>(g);
  fe_count_launch();
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}

// blocks of the last x product (its dot-product partials)
int out_blocks(int rows, int NX) {
  const int tm = tile_for(rows), tn = tile_for(NX);
  return ((rows + 16 * tm - 1) / (16 * tm)) * ((NX + 16 * tn - 1) / (16 * tn));
}

// ---- vector steps ------------------------------------------------------------------------------
// blocks of the vector steps (four an SM)
constexpr int VEC_BLOCKS = 608;

// p = z + beta p (p = z in the first iteration)
__global__ void __launch_bounds__(256)
k_sep_direction(double* __restrict__ p, const double* __restrict__ z, int64_t n, const Scalars* s,
                int first) {
  const int64_t step = (int64_t)gridDim.x * 256;
  if (first) {
    for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < n; i += step) p[i] = z[i];
    return;
  }
  const double beta = s->beta;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < n; i += step)
    p[i] = fma(beta, p[i], z[i]);
}

// p.q; the last block takes alpha = r.z / p.q, or zero when that is no step: a residual outside
// the floats' range makes z zero or not finite, and nothing of it must reach phi
__global__ void __launch_bounds__(256)
k_sep_dot(const double* __restrict__ p, const double* __restrict__ q, int64_t n,
          double* __restrict__ part, Scalars* s) {
  double v = 0.0;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
    v = fma(p[i], q[i], v);
  v = block_total(v);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
  if (last_block(&s->ticket[1], gridDim.x)) {
    const double pq = sum_partials(part, gridDim.x);
    if (threadIdx.x == 0) {
      const double a = s->rz / pq;
      s->alpha = isfinite(a) && isfinite(pq) ? a : 0.0;
    }
  }
}

// phi += alpha p, r -= alpha q on free nodes (p is zero elsewhere), nothing for alpha = 0; |r|^2
__global__ void __launch_bounds__(256)
k_sep_update(double* __restrict__ phi, double* __restrict__ r, const double* __restrict__ p,
             const double* __restrict__ q, const unsigned char* __restrict__ mask, int64_t n,
             double* __restrict__ part, Scalars* s) {
  const double alpha = s->alpha;
  double v = 0.0;
#pragma unroll 4
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    double x = mask[i] ? 0.0 : r[i];
    if (alpha != 0.0) {
      phi[i] = fma(alpha, p[i], phi[i]);
      if (!mask[i]) x = fma(-alpha, q[i], x);
      r[i] = x;
    }
    v = fma(x, x, v);
  }
  v = block_total(v);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
  if (last_block(&s->ticket[2], gridDim.x)) {
    const double rr = sum_partials(part, gridDim.x);
    if (threadIdx.x == 0) s->rr = rr;
  }
}

// the largest chain the host eigensolver takes: about 9 n^3 flops after the mirror split
constexpr int MAX_CHAIN = 512;

}  // namespace

namespace fe_sep {

bool supported(const fe_mesh* m) {
  return m->NX <= MAX_CHAIN && m->NY <= MAX_CHAIN && m->NZ <= MAX_CHAIN &&
         (int64_t)m->NZ * m->NY <= 65535 * 64;
}

size_t part_doubles(const fe_mesh* m) {
  // (tiles are at least 64 wide, and the z chain at most NZ planes long)
  const size_t rows = (size_t)m->NZ * m->NY;
  return 2 * ((rows + 63) / 64) * (((size_t)m->NX + 63) / 64) + VEC_BLOCKS + sizeof(Scalars) / sizeof(double);
}

fe_status plan(fe_mesh* m, const double* cnt, bool constant_null) {
  m->sep_state = 2;
  // the planes with free nodes, one run; without a fully constrained plane (and without the
  // constant null space that the CEF load is projected against) the separable operator
  // would be singular where K on the free nodes is not
  int lo = 0, hi = m->NZ;
  while (lo < hi && cnt[lo] < 0.5) ++lo;
  while (hi > lo && cnt[hi - 1] < 0.5) --hi;
  if (hi - lo < 1) return FE_OK;
  for (int k = lo; k < hi; ++k)
    if (cnt[k] < 0.5) return FE_OK;
  if (!constant_null && hi - lo == m->NZ) return FE_OK;
  const int n[3] = {m->NX, m->NY, hi - lo};
  const double scale[3] = {m->h[1] * m->h[2] / (2.0 * m->h[0]), m->h[0] * m->h[2] / (2.0 * m->h[1]),
                           m->h[0] * m->h[1] / (2.0 * m->h[2])};
  std::vector<float> host;
  std::vector<float> lam_f[3];
  for (int d = 0; d < 3; ++d) {
    std::vector<double> lam;
    Mat V;
    if (!chain_eigen(m, d == 0 ? m->nx : d == 1 ? m->ny : m->nz, d < 2, d < 2 ? 0 : lo,
                     d < 2 ? n[d] : hi, lam, V))
      return FE_OK;
    const size_t nn = (size_t)n[d] * n[d], at = host.size();
    host.resize(at + 2 * nn);
    for (int a = 0; a < n[d]; ++a)
      for (int i = 0; i < n[d]; ++i) {
        host[at + (size_t)i * n[d] + a] = (float)V[(size_t)a * n[d] + i];   // V [node][mode]
        host[at + nn + (size_t)a * n[d] + i] = (float)V[(size_t)a * n[d] + i];
      }
    // The constant is an eigenvector of every chain without a constrained end, and its
    // eigenvalue zero comes out at rounding level: set to zero, the sum over the directions is zero
    // for the constant alone, however different the cell lengths (a threshold on the sum
    // dropped the slow modes along cells 80 times longer than wide).
    if (d < 2 || constant_null) *std::min_element(lam.begin(), lam.end()) = 0.0;
    for (double l : lam) lam_f[d].push_back((float)(scale[d] * l));
  }
  for (int d = 0; d < 3; ++d) host.insert(host.end(), lam_f[d].begin(), lam_f[d].end());
  void* w = nullptr;
  FE_TRY(fe_ws(m, WS_SEP, sizeof(float) * host.size(), &w));
  FE_CUDA(cudaMemcpyAsync(w, host.data(), sizeof(float) * host.size(), cudaMemcpyHostToDevice,
                          m->stream));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  m->sep_lo = lo;
  m->sep_hi = hi;
  m->sep_state = 1;
  return FE_OK;
}

fe_status solve(fe_mesh* m, const Buf& b, double tol2, int maxit, double* rr, int* iters,
                bool* lost) {
  const int NX = m->NX, NY = m->NY, nz = m->sep_hi - m->sep_lo;
  const int64_t plane = (int64_t)NX * NY, n = m->n_phi, off = m->sep_lo * plane;
  cudaStream_t st = m->stream;
  Tables t;
  const float* w = static_cast<const float*>(m->ws[WS_SEP]);
  t.Vx = w;
  t.VxT = t.Vx + (size_t)NX * NX;
  t.Vy = t.VxT + (size_t)NX * NX;
  t.VyT = t.Vy + (size_t)NY * NY;
  t.Vz = t.VyT + (size_t)NY * NY;
  t.VzT = t.Vz + (size_t)nz * nz;
  t.lx = t.VzT + (size_t)nz * nz;
  t.ly = t.lx + NX;
  t.lz = t.ly + NY;
  const int rows = nz * NY, np = out_blocks(rows, NX);
  double* part_z = b.part;
  double* part = part_z + 2 * (size_t)np;
  Scalars* s = reinterpret_cast<Scalars*>(part + VEC_BLOCKS);
  FE_CUDA(cudaMemsetAsync(s, 0, sizeof(Scalars), st));
  // the constrained planes' entries of z and p stay zero
  FE_CUDA(cudaMemsetAsync(b.z, 0, sizeof(double) * n, st));
  const double rr0 = *rr;
  double best = rr0;
  int since = 0;
  *iters = 0;
  *lost = false;
  for (int it = 0; it < maxit && *rr > tol2; ++it) {
    // z = V diag(1 / lambda) V^T r
    Gemm g = {};
    g.W = t.Vx; g.in_d = b.r + off; g.out = b.ta; g.M = rows; g.N = NX; g.K = NX;
    FE_TRY(gemm<RIGHT_IN>(g, 1, st));
    g = {};
    g.W = t.Vy; g.in = b.ta; g.out = b.tb; g.M = NY; g.N = NX; g.K = NY;
    g.in_batch = g.out_batch = plane;
    FE_TRY(gemm<LEFT>(g, nz, st));
    g = {};
    g.W = t.Vz; g.in = b.tb; g.out = b.ta; g.M = nz; g.N = (int)plane; g.K = nz;
    g.lx = t.lx; g.ly = t.ly; g.lz = t.lz; g.NX = NX;
    FE_TRY(gemm_z<LEFT_SCALE>(g, st));
    g = {};
    g.W = t.VzT; g.in = b.ta; g.out = b.tb; g.M = nz; g.N = (int)plane; g.K = nz;
    FE_TRY(gemm_z<LEFT>(g, st));
    g = {};
    g.W = t.VyT; g.in = b.tb; g.out = b.ta; g.M = NY; g.N = NX; g.K = NY;
    g.in_batch = g.out_batch = plane;
    FE_TRY(gemm<LEFT>(g, nz, st));
    g = {};
    g.W = t.VxT; g.in = b.ta; g.out_d = b.z + off; g.M = rows; g.N = NX; g.K = NX;
    g.mask = b.mask + off; g.r = b.r + off; g.q = it > 0 ? b.q + off : nullptr; g.part = part_z;
    g.s = s; g.first = it == 0;
    FE_TRY(gemm<RIGHT_OUT>(g, 1, st));
    k_sep_direction<<<VEC_BLOCKS, 256, 0, st>>>(b.p, b.z, n, s, it == 0);
    fe_count_launch();
    FE_TRY(fe_poisson_apply_K(m, b.p, b.q));
    k_sep_dot<<<VEC_BLOCKS, 256, 0, st>>>(b.p, b.q, n, part, s);
    fe_count_launch();
    k_sep_update<<<VEC_BLOCKS, 256, 0, st>>>(b.phi, b.r, b.p, b.q, b.mask, n, part, s);
    fe_count_launch();
    FE_CUDA(cudaGetLastError());
    Scalars h;
    FE_CUDA(cudaMemcpyAsync(&h, s, sizeof h, cudaMemcpyDeviceToHost, st));
    FE_CUDA(cudaStreamSynchronize(st));
    *rr = h.rr;
    *iters = it + 1;
    // no progress over thirty iterations, or no step at all: hand the solve back
    if (*rr < 0.25 * best) { best = *rr; since = 0; } else { ++since; }
    if (h.alpha == 0.0 || since >= 30) { *lost = true; break; }
  }
  return FE_OK;
}

}  // namespace fe_sep
