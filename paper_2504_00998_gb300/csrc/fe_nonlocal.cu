// Nonlocal pseudopotential term with synthetic projectors (Eq. V_nloc).
//
// (V_nloc psi)(x) = sum_a sum_beta p^a_beta(x - R_a) D^a_beta int p^a_beta(y - R_a) psi(y) dy
// with one s and three p channels per atom: g(d) = exp(-|d|^2 / (2 s_a^2)),
// p_s = g, p_x = (d_x / s_a) g, p_y = (d_y / s_a) g, p_z = (d_z / s_a) g, summed over the
// periodic x/y images and cut at |d| <= rc.  With the lumped quadrature <N_I, p> ~ M_II p(x_I)
// the scaled operator is Ht_nloc = M^1/2 P D P^T M^1/2 (Section 2.3's H u = eps M u).
//
// Layout: the nonzeros of Pt = M^1/2 P are kept atom-major (entry e: psi node, atom, four
// channel values) for the projection C[a][beta][v] = sum_e Pt[e][beta] X[node_e][v], and
// node-major (the entries of each touched psi node) for the output-stationary update
// Y[node][v] += alpha sum_{e at node} sum_beta Pt[e][beta] D[a_e][beta] C[a_e][beta][v]: every
// output entry is written by one thread, no atomics.
#include <algorithm>
#include <cmath>
#include <unordered_map>
#include <vector>

#include "fe_internal.h"

namespace {

constexpr int NCHAN = 4;

// 16-byte groups of vectors (rows are 16-byte aligned and a multiple of 16 bytes long, so a
// group that holds a vector lies inside its row)
template <typename T>
struct NlGroup;
template <>
struct NlGroup<float> {
  using V = float4;
  static constexpr int W = 4;
  static __device__ __forceinline__ float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ float4 fma(float a, const float4& x, const float4& y) {
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
  }
  static __device__ __forceinline__ float4 add_xor(float4 x, int o) {
    x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
    x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
    x.z += __shfl_xor_sync(0xffffffffu, x.z, o);
    x.w += __shfl_xor_sync(0xffffffffu, x.w, o);
    return x;
  }
};
template <>
struct NlGroup<double> {
  using V = double2;
  static constexpr int W = 2;
  static __device__ __forceinline__ double2 zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ double2 fma(double a, const double2& x, const double2& y) {
    return make_double2(::fma(a, x.x, y.x), ::fma(a, x.y, y.y));
  }
  static __device__ __forceinline__ double2 add_xor(double2 x, int o) {
    x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
    x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
    return x;
  }
};

constexpr int PROJ_GROUPS = 8, PROJ_SLOTS = 32;   // vector groups and entry slots of a block
constexpr int PROJ_THREADS = PROJ_GROUPS * PROJ_SLOTS;

// C[a][beta][v] = D[a][beta] sum_e Pt[e][beta] X[node_e][v] for one atom and a tile of vector
// groups (rows of C are ldc long, a multiple of a group).  An atom has a thousand entries
// and there are few atoms, so its entries are spread over 32 slots of a block, four loads in
// flight each, and the slots summed in a fixed order: with one thread walking all entries of
// a vector the launch took 300 us (64 atoms, 128 float vectors, 190,400 nodes, p = 5), bound by
// the latency of its loads; now 24 us.  (The coefficients D are applied here, once an atom,
// instead of at every node.)  Grid: atoms in x, tiles in y and, past its 65,535, in z.
template <typename T>
__global__ void __launch_bounds__(PROJ_THREADS)
k_nl_project(const T* __restrict__ X, int64_t ld, int64_t nvec, const int* __restrict__ atom_ptr,
             const int* __restrict__ ent_node, const T* __restrict__ ent_val,
             const T* __restrict__ Dv, T* __restrict__ C, int64_t ldc) {
  using G = NlGroup<T>;
  using V = typename G::V;
  __shared__ V red[PROJ_THREADS / 32][PROJ_GROUPS][NCHAN];
  const int a = blockIdx.x, g = threadIdx.x % PROJ_GROUPS, slot = threadIdx.x / PROJ_GROUPS;
  const int64_t tile = blockIdx.y + (int64_t)blockIdx.z * gridDim.y;
  const int64_t v = (tile * PROJ_GROUPS + g) * G::W;
  if (tile * PROJ_GROUPS * G::W >= nvec) return;
  const bool in = v < nvec;
  const int e1 = atom_ptr[a + 1];
  V c[NCHAN];
#pragma unroll
  for (int b = 0; b < NCHAN; ++b) c[b] = G::zero();
#pragma unroll 4
  for (int e = atom_ptr[a] + slot; e < e1; e += PROJ_SLOTS) {
    V x = G::zero();
    if (in) x = *reinterpret_cast<const V*>(X + (int64_t)ent_node[e] * ld + v);
#pragma unroll
    for (int b = 0; b < NCHAN; ++b) c[b] = G::fma(ent_val[(int64_t)NCHAN * e + b], x, c[b]);
  }
#pragma unroll
  for (int b = 0; b < NCHAN; ++b) {
    c[b] = G::add_xor(c[b], 8);
    c[b] = G::add_xor(c[b], 16);
    if ((threadIdx.x & 31) < PROJ_GROUPS) red[threadIdx.x / 32][g][b] = c[b];
  }
  __syncthreads();
  if (threadIdx.x < PROJ_GROUPS * NCHAN) {
    const int b = threadIdx.x / PROJ_GROUPS;
    V t = red[0][g][b];
#pragma unroll
    for (int w = 1; w < PROJ_THREADS / 32; ++w) t = G::fma(T(1), red[w][g][b], t);
    // (a group past the last vector lies in the padding of C's row, or beyond it)
    if (in)
      *reinterpret_cast<V*>(C + ((int64_t)a * NCHAN + b) * ldc + v) =
          G::fma(Dv[NCHAN * a + b], t, G::zero());
  }
}

// Y[node][v] += alpha sum_e sum_beta Pt[e][beta] C[a_e][beta][v]: one thread per touched node
// and vector group (35 us with a warp per node and scalar lanes, 21 us so, on the same slab:
// half of it the update of Y itself)
template <typename T>
__global__ void __launch_bounds__(256)
k_nl_apply(T* __restrict__ Y, int64_t ld, int64_t nvec, int64_t ntouched,
           const int* __restrict__ tn_node, const int* __restrict__ tn_ptr,
           const int* __restrict__ tn_ent, const int* __restrict__ ent_atom,
           const T* __restrict__ ent_val, const T* __restrict__ C, int64_t ldc, T alpha) {
  using G = NlGroup<T>;
  using V = typename G::V;
  const uint32_t ng = (uint32_t)(ldc / G::W);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ntouched * ng;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = i / ng, v = (i - t * ng) * G::W;
    T* yp = Y + (int64_t)tn_node[t] * ld + v;
    V y = *reinterpret_cast<const V*>(yp), acc = G::zero();
    for (int k = tn_ptr[t]; k < tn_ptr[t + 1]; ++k) {
      const int e = tn_ent[k];
      const T* Ca = C + (int64_t)ent_atom[e] * NCHAN * ldc + v;
#pragma unroll
      for (int b = 0; b < NCHAN; ++b)
        acc = G::fma(ent_val[(int64_t)NCHAN * e + b], *reinterpret_cast<const V*>(Ca + b * ldc), acc);
    }
    y = G::fma(alpha, acc, y);
    if (v + G::W <= nvec) {
      *reinterpret_cast<V*>(yp) = y;
    } else {
      const T* o = reinterpret_cast<const T*>(&y);
      for (int64_t j = 0; v + j < nvec; ++j) yp[j] = o[j];
    }
  }
}

template <typename T>
T* dev_copy(const std::vector<T>& h, fe_status* st) {
  T* d = nullptr;
  if (h.empty()) return nullptr;
  if (cudaMalloc(&d, sizeof(T) * h.size()) != cudaSuccess ||
      cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    if (d) cudaFree(d);
    *st = fe_fail(FE_ENOMEM, "nonlocal tables of %zu bytes", sizeof(T) * h.size());
    return nullptr;
  }
  return d;
}

}  // namespace

void fe_nonlocal_free(fe_mesh* m) {
  void* ptrs[] = {m->nl.atom_ptr, m->nl.ent_node, m->nl.ent_atom, m->nl.ent_val, m->nl.ent_val_f,
                  m->nl.D, m->nl.D_f, m->nl.tn_node, m->nl.tn_ptr, m->nl.tn_ent};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  m->nl = FeNonlocal{};
}

extern "C" fe_status fe_set_nonlocal(fe_mesh* m, int natoms, const double* R, const double* sigma,
                                     const double* D, double rc) {
  if (!m) return fe_fail(FE_EINVAL, "fe_set_nonlocal: null mesh");
  if (natoms < 0) return fe_fail(FE_EINVAL, "fe_set_nonlocal: natoms < 0");
  FE_TRY(fe_activate(m));
  FE_CUDA(cudaStreamSynchronize(m->stream));
  fe_nonlocal_free(m);
  if (natoms == 0) return FE_OK;
  if (!R || !sigma || !D) return fe_fail(FE_EINVAL, "fe_set_nonlocal: null array");
  if (!(rc > 0.0)) return fe_fail(FE_EINVAL, "fe_set_nonlocal: need rc > 0");
  for (int a = 0; a < natoms; ++a)
    if (!(sigma[a] > 0.0)) return fe_fail(FE_EINVAL, "fe_set_nonlocal: atom %d: sigma <= 0", a);
  const int p = m->p;
  const double Lx = m->desc.L[0], Ly = m->desc.L[1];
  auto coord = [&](int g, int d) { return (g / p) * m->h[d] + (m->xi[g % p] + 1.0) * 0.5 * m->h[d]; };
  auto mass1 = [&](int g, bool periodic, int gmax) {
    const int l = g % p;
    if (l) return m->w[l];
    if (periodic) return 2.0 * m->w[0];
    return (g == 0 || g == gmax) ? m->w[0] : 2.0 * m->w[0];
  };
  const int gzmax = m->nz * p;
  std::vector<int> atom_ptr(natoms + 1, 0), ent_node, ent_atom;
  std::vector<double> ent_val;
  for (int a = 0; a < natoms; ++a) {
    const double s = sigma[a];
    std::unordered_map<int64_t, int> at;   // psi node -> entry of this atom
    // unwrapped x / y node indices around the atom: each (node, periodic image) pair within
    // rc appears once, the image being (g - wrapped g) / N periods away
    const double cx = R[3 * a], cy = R[3 * a + 1], cz = R[3 * a + 2];
    const int x0 = (int)std::floor((cx - rc) / m->h[0]) * p, x1 = ((int)std::floor((cx + rc) / m->h[0]) + 1) * p;
    const int y0 = (int)std::floor((cy - rc) / m->h[1]) * p, y1 = ((int)std::floor((cy + rc) / m->h[1]) + 1) * p;
    const int z0 = std::max((int)std::floor((cz - rc) / m->h[2]) * p, m->gz_lo);
    const int z1 = std::min(((int)std::floor((cz + rc) / m->h[2]) + 1) * p, m->gz_lo + m->NZs - 1);
    for (int gz = z0; gz <= z1; ++gz) {
      const double dz = coord(gz, 2) - cz;
      for (int gy = y0; gy <= y1; ++gy) {
        const int wy = ((gy % m->NY) + m->NY) % m->NY;
        const double dy = (double)((gy - wy) / m->NY) * Ly + coord(wy, 1) - cy;
        for (int gx = x0; gx <= x1; ++gx) {
          const int wx = ((gx % m->NX) + m->NX) % m->NX;
          const double dx = (double)((gx - wx) / m->NX) * Lx + coord(wx, 0) - cx;
          const double r2 = dx * dx + dy * dy + dz * dz;
          if (r2 > rc * rc) continue;
          const int64_t node = (int64_t)(gz - m->gz_lo) * m->NX * m->NY + (int64_t)wy * m->NX + wx;
          const double g = std::exp(-r2 / (2.0 * s * s));
          const double sm = std::sqrt(m->J * mass1(wx, true, 0) * mass1(wy, true, 0) * mass1(gz, false, gzmax));
          int e;
          auto it = at.find(node);
          if (it == at.end()) {
            e = (int)ent_node.size();
            at.emplace(node, e);
            ent_node.push_back((int)node);
            ent_atom.push_back(a);
            ent_val.insert(ent_val.end(), 4, 0.0);
          } else {
            e = it->second;
          }
          ent_val[4 * e + 0] += sm * g;
          ent_val[4 * e + 1] += sm * dx / s * g;
          ent_val[4 * e + 2] += sm * dy / s * g;
          ent_val[4 * e + 3] += sm * dz / s * g;
        }
      }
    }
    atom_ptr[a + 1] = (int)ent_node.size();
  }
  // node-major lists
  const int nnz = (int)ent_node.size();
  std::vector<int> order(nnz);
  for (int e = 0; e < nnz; ++e) order[e] = e;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return ent_node[x] < ent_node[y]; });
  std::vector<int> tn_node, tn_ptr(1, 0);
  for (int k = 0; k < nnz; ++k) {
    if (tn_node.empty() || tn_node.back() != ent_node[order[k]]) {
      if (!tn_node.empty()) tn_ptr.push_back(k);
      tn_node.push_back(ent_node[order[k]]);
    }
  }
  tn_ptr.push_back(nnz);
  if (tn_node.empty()) tn_ptr.assign(1, 0);
  std::vector<double> Dv(D, D + 4 * (size_t)natoms);
  std::vector<float> ent_val_f(ent_val.begin(), ent_val.end()), D_f(Dv.begin(), Dv.end());
  fe_status st = FE_OK;
  FeNonlocal nl{};
  nl.natoms = natoms;
  nl.nnz = nnz;
  nl.ntouched = (int)tn_node.size();
  nl.atom_ptr = dev_copy(atom_ptr, &st);
  nl.ent_node = dev_copy(ent_node, &st);
  nl.ent_atom = dev_copy(ent_atom, &st);
  nl.ent_val = dev_copy(ent_val, &st);
  nl.ent_val_f = dev_copy(ent_val_f, &st);
  nl.D = dev_copy(Dv, &st);
  nl.D_f = dev_copy(D_f, &st);
  nl.tn_node = dev_copy(tn_node, &st);
  nl.tn_ptr = dev_copy(tn_ptr, &st);
  nl.tn_ent = dev_copy(order, &st);
  m->nl = nl;
  if (st != FE_OK) {
    fe_nonlocal_free(m);
    return st;
  }
  return FE_OK;
}

// Y += alpha Ht_nloc X (float or double blocks; the bf16 tensor-core path uses float blocks)
fe_status fe_nonlocal_apply(fe_mesh* m, const void* X, void* Y, int64_t nvec, int64_t ld,
                            double alpha, bool dbl) {
  const FeNonlocal& nl = m->nl;
  if (nl.natoms == 0 || nl.nnz == 0) return FE_OK;
  cudaStream_t st = m->stream;
  const size_t eb = dbl ? 8 : 4;
  const int64_t w = dbl ? 2 : 4, ldc = (nvec + w - 1) / w * w, ng = ldc / w;
  void* c;
  FE_TRY(fe_ws(m, WS_NL, eb * NCHAN * (size_t)nl.natoms * ldc + 64, &c));
  const int64_t tiles = (ng + PROJ_GROUPS - 1) / PROJ_GROUPS;
  const int64_t ty = std::min<int64_t>(tiles, 65535), tz = (tiles + ty - 1) / ty;
  if (tz > 65535) return fe_fail(FE_EINVAL, "nonlocal term: too many vectors");
  const dim3 pg(nl.natoms, (unsigned)ty, (unsigned)tz);
  const int ab = (int)std::min<int64_t>(((int64_t)nl.ntouched * ng + 255) / 256, 152 * 32);
  auto run = [&](auto zero, const auto* val, const auto* D) {
    using T = decltype(zero);
    k_nl_project<T><<<pg, PROJ_THREADS, 0, st>>>((const T*)X, ld, nvec, nl.atom_ptr, nl.ent_node, val,
                                                 D, (T*)c, ldc);
    fe_count_launch();
    k_nl_apply<T><<<ab, 256, 0, st>>>((T*)Y, ld, nvec, nl.ntouched, nl.tn_node, nl.tn_ptr, nl.tn_ent,
                                      nl.ent_atom, val, (const T*)c, ldc, (T)alpha);
    fe_count_launch();
  };
  if (dbl) run(0.0, (const double*)nl.ent_val, (const double*)nl.D);
  else run(0.f, (const float*)nl.ent_val_f, (const float*)nl.D_f);
  FE_CUDA(cudaGetLastError());
  return FE_OK;
}
