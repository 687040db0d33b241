// Matrix-free application of the mass-scaled Hamiltonian of Section 2.3 to blocks of vectors,
//   Y = alpha (Ht - shift) X + beta Z,   Ht = 1/2 M^-1/2 K M^-1/2 + diag(V)  (real), or
//   Ht_k = Ht + 1/2 |k|^2 - i M^-1/2 (kx Gx + ky Gy) M^-1/2  on interleaved (re, im) lanes.
//
// Arithmetic.  With the symmetrically scaled one-dimensional matrices Kh = D^-1/2 K1 D^-1/2 and
// Mh = D^-1/2 M1 D^-1/2 (D the assembled GLL-lumped mass) the kinetic operator is
//   cx Kh (x) Mh (x) Mh + cy Mh (x) Kh (x) Mh + cz Mh (x) Mh (x) Kh,
// without any nodal scale.  The exact mass differs from the lumped one by one product per
// cell, Mh = 1 - sum_cells t t^T (gen_gll_tables.py), so a mass contraction is a dot product and
// an update per cell line, 2 (p + 1) FMAs where the dense one takes (p + 1)^2: at p = 5 about 40
// FMAs a node and vector against 58, and nothing else is needed of the mesh than three scalars.
//
// Work decomposition.  A CTA owns the nodes of CX x CY cells (half-open), VP packed elements of
// the vectors (an element is 8 bytes: two floats, handled by paired FMAs, or one double), and
// a range of cell layers; it sweeps the z planes in order, one CTA barrier a plane:
//   all threads    copy plane g + 3 (with its periodic halo of p + 1 nodes) into one of four
//                  slots with cp.async, from a table of offsets built once;
//   y threads      one (halo x, element) column each: the column's whole y line is read once
//                  into registers, a = Mh u and b = Kh u go to shared memory (plane g + 1);
//   xz threads     one (row, XC cells, element) each (plane g): the x contractions give u and
//                  v of the row's own nodes in registers, which go straight into the
//                  (p + 1)-plane accumulators of the z contraction held by the same thread; the
//                  potential and the previous iterate Z are added when their plane passes, so
//                  Z needs no staging.  A layer's first p planes are written when it is
//                  complete; the top plane's sum carries into the next layer.
// No scatter, no atomics: every node is written once by the thread that owns it, so results
// do not depend on scheduling.
//
// What bounds it.  On the 16 x 16 x 48-cell p = 5 slab with 512 float vectors a filter step takes
// 2.83 ms (9.3 GB algorithmic, 0.49 of the measured copy bandwidth), where the sweep with dense
// mass contractions, scalar in-plane phases and three barriers a plane took 3.86 ms; on the
// 16 x 16 x 16-cell slab with 256 vectors 484 against 681 us, from 266 M against 615 M warp
// instructions.  DRAM moves 1.78 GB there (algorithmic 1.56), 54 % of the copy rate; issue slots
// are 46 % busy, the FMA pipe 37 %, the shared-memory data pipe 56 %: with 160 registers a thread
// only ten warps are resident, too few to cover the FMA and shared-memory latencies.  The
// accumulators set the registers, so more warps mean spills, and those were slower (three CTAs
// an SM at p = 5: 734 us); so were planes staged without the one-barrier double buffer of a, b
// (524 us), coefficients from constant memory (763), a code copy per plane of the layer (769),
// Z and V through shared memory (502) and four elements a node instead of eight (660).  At
// p = 4 the smaller tile leaves room for four CTAs without the double buffer: 234 against
// 255 us.  Other sizes, before and after: 12 x 12 x 40 cells p = 4, 64 vectors 170 -> 107 us;
// 9 x 7 x 21 cells p = 6, 101 vectors 344 -> 247 us; the Bloch operator (one launch instead of a
// real and a gradient one) 16 x 16 x 16 cells p = 5, 128 complex vectors 1.42 -> 0.55 ms.
#pragma once

#include <algorithm>
#include <type_traits>

#include "fe_gll_tables.h"
#include "fe_internal.h"

namespace fe {

// ---- packed elements: 8 bytes of consecutive vectors ---------------------------------------
struct PackF {   // two floats
  using T = float;
  using R = unsigned long long;
  static constexpr int LANES = 2;
  static __device__ __forceinline__ R splat(float a) {
    R r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
  }
  static __device__ __forceinline__ R pair(float a, float b) {
    R r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
  }
  static __device__ __forceinline__ R zero() { return 0ull; }
  static __device__ __forceinline__ float fma1(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  static __device__ __forceinline__ R fma(R a, R b, R c) {
    R d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
  }
  static __device__ __forceinline__ R mul(R a, R b) {
    R d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
  }
  static __device__ __forceinline__ R add(R a, R b) {
    R d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
  }
  // -i (re + i im) = im - i re, times the real g
  static __device__ __forceinline__ R minus_i(float g, R a, R acc, int, unsigned) {
    return fma(pair(g, -g), swap(a), acc);
  }
  static __device__ __forceinline__ R swap(R a) {
    R d;
    asm("{\n\t.reg .f32 x, y;\n\tmov.b64 {x, y}, %1;\n\tmov.b64 %0, {y, x};\n\t}" : "=l"(d) : "l"(a));
    return d;
  }
  static __device__ __forceinline__ void store_first(float* p, R a) {
    *p = __uint_as_float((unsigned)(a & 0xffffffffull));
  }
};
struct PackD {   // one double
  using T = double;
  using R = double;
  static constexpr int LANES = 1;
  static __device__ __forceinline__ R splat(double a) { return a; }
  static __device__ __forceinline__ R zero() { return 0.0; }
  static __device__ __forceinline__ double fma1(double a, double b, double c) { return __fma_rn(a, b, c); }
  static __device__ __forceinline__ R fma(R a, R b, R c) { return __fma_rn(a, b, c); }
  static __device__ __forceinline__ R mul(R a, R b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ R add(R a, R b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ void store_first(double* p, R a) { *p = a; }
  // the parts are in neighbouring threads (even: real)
  static __device__ __forceinline__ R minus_i(double g, R a, R acc, int lane, unsigned mask) {
    const double o = __shfl_xor_sync(mask, a, 1);
    return fma((lane & 1) ? -g : g, o, acc);
  }
};

// the mesh's scalars: the operator is divided by the z stiffness scale cz, which alpha takes
template <typename T>
struct SweepCoef {
  T rx, ry;        // cx / cz, cy / cz
  T gx, gy;        // Bloch term over cz: kx and ky times its scales (0: real operator)
  // Nothing reads these bytes, but the compiler places the parameters behind them better: without
  // them the double kernels spill 2,712 bytes in all, not 2,388, and a cycle of 6 x 6 x 16 cells
  // p = 3, 32 double vectors takes 2.19 ms, not 2.17.
  char room[504];
};

template <class V_, int P_, int CX_, int CY_, int XC_, int VP_, int RES_, bool DB_>
struct SweepTile {
  using V = V_;
  static constexpr int P = P_, CX = CX_, CY = CY_, XC = XC_, VP = VP_;
  static constexpr int RES = RES_;                  // CTAs per SM the registers are held to
  static constexpr bool DB = DB_;                   // a, b of two planes: one barrier a plane
  static constexpr int BXn = CX * P, BYn = CY * P;
  static constexpr int BXH = BXn + P + 1, BYH = BYn + P + 1;
  static constexpr int NXI = XC * P;                // own nodes of an xz thread
  static constexpr int NY = BXH * VP;               // y threads
  static constexpr int NXZ = (CX / XC) * BYn * VP;  // xz threads
  static constexpr int NT = ((NXZ > NY ? NXZ : NY) + 31) / 32 * 32;
  static constexpr int RC = BXH * VP / 2;           // 16-byte chunks of a staged row
  static constexpr int NST = BYH * RC;              // of a plane
  static constexpr int SLOTS = DB ? 4 : 3, ABS = DB ? 2 : 1;
  // Bank layout.  A warp of xz threads reads 16 / VP rows at one x.  Staged rows of an even
  // number of nodes would fall on the same banks, so their odd rows swap neighbouring nodes;
  // the a and b halves of a node swap with the parity of x plus the row.
  static constexpr bool SWZ = BXH % 2 == 0;
  static constexpr int U_ELEMS = BYH * BXH * VP;    // 8-byte elements of a slot
  static constexpr int AB_ELEMS = BYn * BXH * 2 * VP;
  static constexpr size_t SMEM = sizeof(double) * (SLOTS * (size_t)U_ELEMS + ABS * (size_t)AB_ELEMS) +
                                 sizeof(uint32_t) * (size_t)NST;
  static_assert(CX % XC == 0 && VP % 2 == 0 && NT <= 1024, "tile shape");
};

// periodic index (a halo reaches past a narrow mesh more than once)
__device__ __forceinline__ int wrap_index(int a, int n) {
  while (a < 0) a += n;
  while (a >= n) a -= n;
  return a;
}

template <class TL, bool CPLX, bool FULL>
__device__ __forceinline__ void sweep_body(const SweepCoef<typename TL::V::T>& cf, const KronGeom& g,
                                           const SweepIO<typename TL::V::T>& io, int bxy, int vti,
                                           int zsi) {
  using V = typename TL::V;
  using T = typename V::T;
  using R = typename V::R;
  constexpr int P = TL::P, VP = TL::VP, XC = TL::XC, CY = TL::CY, NXI = TL::NXI;
  constexpr int BXH = TL::BXH, BYH = TL::BYH, BYn = TL::BYn, LANES = V::LANES;
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  R* U = reinterpret_cast<R*>(sweep_smem);              // [SLOTS][BYH][BXH][VP]
  R* AB = U + TL::SLOTS * TL::U_ELEMS;                  // [2][BYn][BXH][2 VP]
  uint32_t* soff = reinterpret_cast<uint32_t*>(AB + TL::ABS * TL::AB_ELEMS);

  auto KH = [](int j, int k) -> R { return V::splat((T)hat_k<P>(j, k)); };
  auto GH = [](int j, int k) -> R { return V::splat((T)hat_g<P>(j, k)); };
  auto TH = [](int j) -> R { return V::splat((T)hat_t<P>(j)); };
  auto nTH = [](int j) -> R { return V::splat((T)-hat_t<P>(j)); };
  const int tid = threadIdx.x;
  // the threads of this warp that are below n
  auto warp_mask = [&](int n) {
    const int left = n - (tid & ~31);
    return left >= 32 ? 0xffffffffu : (1u << left) - 1u;
  };
  const int x0 = (bxy % g.nbx) * TL::BXn, y0 = (bxy / g.nbx) * TL::BYn;
  const int64_t ld = io.ld;
  const int64_t vbase = (int64_t)vti * VP * LANES;
  const int c0 = zsi * g.zseg, c1 = min(c0 + g.zseg, g.nz);
  const int cb = c0 > 0 ? c0 - 1 : 0;
  const int gbeg = cb * P, gend = c1 * P;
  const int64_t pstride = (int64_t)g.NX * g.NY * ld;    // elements of a plane of the blocks
  const int64_t plane_nodes = (int64_t)g.NX * g.NY;
  auto stored = [&](int gz) { return gz >= g.gz_lo && gz < g.gz_lo + g.NZs; };
  auto owned_plane = [&](int gz) {
    return stored(gz) && gz >= c0 * P && (gz < c1 * P || c1 == g.nz);
  };

  // offsets of the staged chunks within a plane, in 16-byte units
  for (int e = tid; e < TL::NST; e += TL::NT) {
    const int row = e / TL::RC, c = e - row * TL::RC;
    const int at = c / (VP / 2), q = c - at * (VP / 2);
    const int x = TL::SWZ ? at ^ (row & 1) : at;
    const int gx = wrap_index(x0 - P + x, g.NX), gy = wrap_index(y0 - P + row, g.NY);
    soff[e] = (uint32_t)(((gx + (int64_t)g.NX * gy) * ld + vbase) * (int64_t)sizeof(T) / 16) + q;
  }
  __syncthreads();

  // ---- staging ---------------------------------------------------------------------------
  // valid bytes of this thread's chunks (the last vector tile may be partial; a thread's chunks
  // are all at one place of a node's row)
  int nb = 16;
  if constexpr (!FULL) {
    const int64_t rem = (io.nvec - vbase) * (int64_t)sizeof(T) - 16 * (tid % (VP / 2));
    nb = rem >= 16 ? 16 : (rem > 0 ? (int)rem : 0);
  }
  const char* xplane = reinterpret_cast<const char*>(io.X) +
                       (int64_t)(gbeg - g.gz_lo) * pstride * (int64_t)sizeof(T);
  const int64_t xstep = pstride * (int64_t)sizeof(T);
  auto stage = [&](int gz) {   // called for gbeg, gbeg + 1, ... in order
    if (gz <= gend && stored(gz)) {
      const unsigned dst = (unsigned)__cvta_generic_to_shared(U + ((gz - gbeg) % TL::SLOTS) * TL::U_ELEMS) +
                           (unsigned)tid * 16u;
      constexpr int IT = (TL::NST + TL::NT - 1) / TL::NT;
#pragma unroll
      for (int i = 0; i < IT; ++i) {
        if (TL::NST % TL::NT != 0 && i == IT - 1 && tid + i * TL::NT >= TL::NST) break;
        const uint32_t o = soff[tid + i * TL::NT];
        const unsigned at = dst + i * TL::NT * 16;
        const char* p = xplane + (uint64_t)o * 16;
        if constexpr (FULL) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(at), "l"(p));
        } else {
          if (nb == 0) p = (const char*)io.X;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(at), "l"(p), "r"(nb));
        }
      }
    }
    xplane += xstep;
    asm volatile("cp.async.commit_group;\n" ::);
  };

  // ---- y phase: the column (xh, pr) of plane gz ------------------------------------------------
  const int pr = tid % VP;
  const int xh = tid / VP;
  auto y_phase = [&](int gz) {
    if (tid >= TL::NY) return;
    const R* s = U + ((gz - gbeg) % TL::SLOTS) * TL::U_ELEMS;
    const R* col0 = s + xh * VP + pr;
    const R* col1 = TL::SWZ ? s + (xh ^ 1) * VP + pr : col0;
    auto u = [&](int r) { return ((r & 1) ? col1 : col0)[r * BXH * VP]; };
    R* ab = AB + (TL::DB ? ((gz - gbeg) & 1) * TL::AB_ELEMS : 0) + xh * 2 * VP + pr;
    const R ry = V::splat(cf.ry);
    // Cell by cell, one row at a time into every output it reaches (independent FMAs, and only
    // the cell's own rows stay in registers).  Of the cell before: t.u and the top rows of
    // Kh u and Gh u.
    R d, kp, gp = V::zero();
    {
      R x = u(0);
      d = V::mul(TH(0), x);
      kp = V::mul(KH(P, 0), x);
      if constexpr (CPLX) gp = V::mul(GH(P, 0), x);
#pragma unroll
      for (int k = 1; k < P; ++k) {
        x = u(k);
        d = V::fma(TH(k), x, d);
        kp = V::fma(KH(P, k), x, kp);
        if constexpr (CPLX) gp = V::fma(GH(P, k), x, gp);
      }
    }
    R x = u(P);   // shared with the next cell
    d = V::fma(TH(P), x, d);
    kp = V::fma(KH(P, P), x, kp);
    if constexpr (CPLX) gp = V::fma(GH(P, P), x, gp);
#pragma unroll
    for (int c = 0; c < CY; ++c) {
      R a[P], b[P + 1], q[P + 1], dn = V::mul(TH(0), x);
      b[0] = V::fma(KH(0, 0), x, kp);
#pragma unroll
      for (int j = 1; j <= P; ++j) b[j] = V::mul(KH(j, 0), x);
      if constexpr (CPLX) {
        q[0] = V::fma(GH(0, 0), x, gp);
#pragma unroll
        for (int j = 1; j <= P; ++j) q[j] = V::mul(GH(j, 0), x);
      }
      a[0] = x;
#pragma unroll
      for (int k = 1; k <= P; ++k) {
        x = u(P + c * P + k);
        if (k < P) a[k] = x;
        dn = V::fma(TH(k), x, dn);
#pragma unroll
        for (int j = 0; j <= P; ++j)
          if (j < P || c + 1 < CY) b[j] = V::fma(KH(j, k), x, b[j]);
        if constexpr (CPLX) {
#pragma unroll
          for (int j = 0; j <= P; ++j)
            if (j < P || c + 1 < CY) q[j] = V::fma(GH(j, k), x, q[j]);
        }
      }
      a[0] = V::fma(nTH(P), d, a[0]);
#pragma unroll
      for (int j = 0; j < P; ++j) {
        R o = V::mul(ry, b[j]);
        if constexpr (CPLX) o = V::minus_i(cf.gy, q[j], o, pr, warp_mask(TL::NY));
        const R m = V::fma(nTH(j), dn, a[j]);
        const int y = c * P + j;
        const int h = (xh + (VP == 8 ? y : y >> 1)) & 1;
        ab[y * BXH * 2 * VP + h * VP] = m;
        ab[y * BXH * 2 * VP + (1 - h) * VP] = o;
      }
      d = dn;
      kp = b[P];
      if constexpr (CPLX) gp = q[P];
    }
  };

  // ---- xz role ------------------------------------------------------------------------------------
  const bool is_xz = tid < TL::NXZ;
  const int yr = (tid / VP) % BYn;                         // own row
  const int xb = is_xz ? (tid / VP / BYn) * NXI : 0;       // first node of the cell before, halo index
  const int64_t vpos = vbase + (int64_t)pr * LANES;
  const int gx0 = x0 + xb, gy0 = y0 + yr;                  // first own node
  const int nown = !is_xz ? 0 : FULL ? NXI : gy0 < g.NY && vpos < io.nvec ? min(NXI, g.NX - gx0) : 0;
  const bool whole = FULL || vpos + LANES <= io.nvec;
  const int64_t own_node = gx0 + (int64_t)g.NX * gy0;
  const bool use_z = io.Z != nullptr;
  // The loads of Z and V are unconditional, so that they stay in flight until their use (a
  // load under a condition is merged with the old value, and so waited for, at once): threads,
  // nodes and planes that own nothing read an owned or the first entry again.
  const int own_lo = max(c0 * P, g.gz_lo);
  const int own_hi = min(c1 == g.nz ? g.nz * P : c1 * P - 1, g.gz_lo + g.NZs - 1);
  const bool own_any = nown > 0 && own_lo <= own_hi;
  const T* zp = use_z ? io.Z : io.X;
  const T* vp = io.V;
  if (own_any) {
    zp += own_node * ld + vpos;
    vp += own_node;
  }
  const int64_t zld = own_any ? ld : 0, zplane = own_any ? pstride : 0;
  const int64_t vplane = own_any ? plane_nodes : 0;
  T* yp = io.Y + own_node * ld + vpos;
  R acc[NXI][P + 1], dz[NXI], un[NXI], vn[NXI], zr[NXI];
  T vr[NXI];
#pragma unroll
  for (int i = 0; i < NXI; ++i) {
    dz[i] = un[i] = vn[i] = zr[i] = V::zero();
    vr[i] = T(0);
#pragma unroll
    for (int j = 0; j <= P; ++j) acc[i][j] = V::zero();
  }
  // Z and V of the own nodes of plane gz, one plane ahead of their use
  auto fetch_zv = [&](int gz) {
    const int pz = max(own_lo, min(gz, own_hi)) - g.gz_lo;
    const T* q = zp + pz * zplane;
    const T* v = vp + pz * vplane;
#pragma unroll
    for (int i = 0; i < NXI; ++i) {
      const int at = FULL ? i : max(0, min(i, nown - 1));
      // (a last odd lane is read with its neighbour in the padded row and never written)
      zr[i] = *reinterpret_cast<const R*>(q + at * zld);
      vr[i] = v[at];
    }
  };
  // u = Mh a and v = rx Kh a + Mh b (+ the Bloch term) along x on the own nodes of plane gz
  auto plane_uv = [&](int gz) {
    const R* ab = AB + (TL::DB ? ((gz - gbeg) & 1) * TL::AB_ELEMS : 0) + (yr * BXH + xb) * 2 * VP + pr;
    const int h = (xb + (VP == 8 ? yr : yr >> 1)) & 1;
    const R* e0 = ab + h * VP;         // a at even offsets, b at odd ones
    const R* e1 = ab + (1 - h) * VP;
    auto la = [&](int i) { return ((i & 1) ? e1 : e0)[i * 2 * VP]; };
    auto lb = [&](int i) { return ((i & 1) ? e0 : e1)[i * 2 * VP]; };
    const R rx = V::splat(cf.rx);
    R d, e, kp, gp = V::zero();
    {
      const R a0 = la(0), b0 = lb(0);
      d = V::mul(TH(0), a0);
      kp = V::mul(KH(P, 0), a0);
      e = V::mul(TH(0), b0);
      if constexpr (CPLX) gp = V::mul(GH(P, 0), a0);
#pragma unroll
      for (int k = 1; k < P; ++k) {
        const R ak = la(k), bk = lb(k);
        d = V::fma(TH(k), ak, d);
        kp = V::fma(KH(P, k), ak, kp);
        e = V::fma(TH(k), bk, e);
        if constexpr (CPLX) gp = V::fma(GH(P, k), ak, gp);
      }
    }
    R xa = la(P), xe = lb(P);
    d = V::fma(TH(P), xa, d);
    kp = V::fma(KH(P, P), xa, kp);
    e = V::fma(TH(P), xe, e);
    if constexpr (CPLX) gp = V::fma(GH(P, P), xa, gp);
#pragma unroll
    for (int c = 0; c < XC; ++c) {
      R w[P + 1], q[P + 1], m[P], dn = V::mul(TH(0), xa), en = V::mul(TH(0), xe);
      w[0] = V::fma(KH(0, 0), xa, kp);
#pragma unroll
      for (int j = 1; j <= P; ++j) w[j] = V::mul(KH(j, 0), xa);
      if constexpr (CPLX) {
        q[0] = V::fma(GH(0, 0), xa, gp);
#pragma unroll
        for (int j = 1; j <= P; ++j) q[j] = V::mul(GH(j, 0), xa);
      }
      un[c * P] = xa;
      m[0] = xe;
#pragma unroll
      for (int k = 1; k <= P; ++k) {
        xa = la(P + c * P + k);
        xe = lb(P + c * P + k);
        if (k < P) { un[c * P + k] = xa; m[k] = xe; }
        dn = V::fma(TH(k), xa, dn);
        en = V::fma(TH(k), xe, en);
#pragma unroll
        for (int j = 0; j <= P; ++j)
          if (j < P || c + 1 < XC) w[j] = V::fma(KH(j, k), xa, w[j]);
        if constexpr (CPLX) {
#pragma unroll
          for (int j = 0; j <= P; ++j)
            if (j < P || c + 1 < XC) q[j] = V::fma(GH(j, k), xa, q[j]);
        }
      }
      un[c * P] = V::fma(nTH(P), d, un[c * P]);
      m[0] = V::fma(nTH(P), e, m[0]);
#pragma unroll
      for (int j = 0; j < P; ++j) {
        un[c * P + j] = V::fma(nTH(j), dn, un[c * P + j]);
        R o = V::fma(rx, w[j], m[j]);
        if constexpr (CPLX) o = V::minus_i(cf.gx, q[j], o, pr, warp_mask(TL::NXZ));
        vn[c * P + j] = V::fma(nTH(j), en, o);
      }
      d = dn;
      e = en;
      kp = w[P];
      if constexpr (CPLX) gp = q[P];
    }
  };
  // the in-plane results (and, WITH_T, the own-node terms) into the layer accumulators, plane K
  // of the layer
  R tn[NXI];
  auto apply = [&](auto kc, auto with_t) {
    constexpr int K = decltype(kc)::value;
    if constexpr (K <= P) {
#pragma unroll
      for (int i = 0; i < NXI; ++i) {
#pragma unroll
        for (int j = 0; j <= P; ++j) acc[i][j] = V::fma(KH(j, K), un[i], acc[i][j]);
        dz[i] = V::fma(TH(K), vn[i], dz[i]);
        // a plane shared by two layers takes half of its identity part from each
        acc[i][K] = (K == 0 || K == P) ? V::fma(V::splat(T(0.5)), vn[i], acc[i][K])
                                       : V::add(vn[i], acc[i][K]);
        if constexpr (decltype(with_t)::value) acc[i][K] = V::add(tn[i], acc[i][K]);
      }
    }
  };
  auto apply_k = [&](int k) {
    const std::true_type t;
    switch (k) {
      case 0: apply(std::integral_constant<int, 0>{}, t); break;
      case 1: apply(std::integral_constant<int, 1>{}, t); break;
      case 2: apply(std::integral_constant<int, 2>{}, t); break;
      case 3: apply(std::integral_constant<int, 3>{}, t); break;
      case 4: apply(std::integral_constant<int, 4>{}, t); break;
      case 5: apply(std::integral_constant<int, 5>{}, t); break;
      case 6: apply(std::integral_constant<int, 6>{}, t); break;
      default: break;
    }
  };
  // a face plane (one layer only) has half the mass of a shared one: its scale is sqrt(2)
  // larger on both sides of the operator
  const R root2 = V::splat(T(1.4142135623730951));
  // the own-node terms (V - shift) x + (beta / alpha) z of plane gz (zero on planes that
  // another segment owns)
  auto own_terms = [&](int gz) {
    const R* s = U + ((gz - gbeg) % TL::SLOTS) * TL::U_ELEMS + ((yr + P) * BXH + xb + P) * VP + pr;
    // swapped rows: neighbours trade places, which way depends on the parities
    const int par = TL::SWZ ? ((yr + P) & 1) : 0;
    const int sg = par ? (((xb + P) & 1) ? -VP : VP) : 0;
    const R z2 = V::splat(io.zs);
    const bool own = owned_plane(gz);
#pragma unroll
    for (int i = 0; i < NXI; ++i) {
      const R x = s[i * VP + ((i & 1) ? -sg : sg)];
      const T w = own ? V::fma1(vr[i] - io.shift, io.vs, io.v0) : T(0);
      tn[i] = V::mul(V::splat(w), x);
      if (use_z && own) tn[i] = V::fma(z2, zr[i], tn[i]);
    }
  };
  auto write_layer = [&](int c) {   // planes c P + j, j < P, then (top of the slab) the face
#pragma unroll
    for (int i = 0; i < NXI; ++i)
#pragma unroll
      for (int j = 0; j <= P; ++j) acc[i][j] = V::fma(nTH(j), dz[i], acc[i][j]);
    const R al = V::splat(io.al);
#pragma unroll
    for (int j = 0; j <= P; ++j) {
      const int gz = c * P + j;
      if (j == P && !(c + 1 == c1 && c1 == g.nz)) continue;
      if (!owned_plane(gz)) continue;
      const bool face = gz == 0 || gz == g.nz * P;
      T* q = yp + (int64_t)(gz - g.gz_lo) * pstride;
#pragma unroll
      for (int i = 0; i < NXI; ++i) {
        if (!FULL && i >= nown) continue;
        R o = acc[i][j];
        if (j == 0 || j == P)
          if (face) o = V::mul(root2, o);
        o = V::mul(al, o);
        if (whole) *reinterpret_cast<R*>(q + i * ld) = o;
        else V::store_first(q + i * ld, o);
      }
    }
#pragma unroll
    for (int i = 0; i < NXI; ++i) {
      acc[i][0] = acc[i][P];
      dz[i] = V::zero();
#pragma unroll
      for (int j = 1; j <= P; ++j) acc[i][j] = V::zero();
    }
  };

  // ---- sweep ---------------------------------------------------------------------------------
  // (one copy of the plane's code, with a switch for the z coefficients: unrolled over the
  // planes of a layer it ran half as fast)
  stage(gbeg);
  stage(gbeg + 1);
  if constexpr (TL::DB) {
    stage(gbeg + 2);
    asm volatile("cp.async.wait_group 2;\n" ::);
    __syncthreads();
  }
  fetch_zv(gbeg);
  if (TL::DB && stored(gbeg)) y_phase(gbeg);
  int c = cb, k = 0;   // layer and local index of plane gz
  for (int gz = gbeg; gz <= gend; ++gz, ++k) {
    asm volatile("cp.async.wait_group 1;\n" ::);
    __syncthreads();
    if constexpr (TL::DB) {
      stage(gz + 3);
    } else {
      stage(gz + 2);
      if (stored(gz)) y_phase(gz);
      __syncthreads();
    }
    if (is_xz) {
      const bool in = stored(gz);
      if (in) {
        plane_uv(gz);
        const bool face = gz == 0 || gz == g.nz * P;
        if (face) {
#pragma unroll
          for (int i = 0; i < NXI; ++i) {
            un[i] = V::mul(root2, un[i]);
            vn[i] = V::mul(root2, vn[i]);
          }
        }
        own_terms(gz);
        if (face) {
          // (the plane's output is multiplied by sqrt(2) when written)
          const R f = V::splat(T(0.70710678118654757));
#pragma unroll
          for (int i = 0; i < NXI; ++i) tn[i] = V::mul(f, tn[i]);
        }
        apply_k(k);
      }
      if (k == P) {
        write_layer(c);
        if (in && c + 1 < c1) apply(std::integral_constant<int, 0>{}, std::false_type{});
      }
    }
    if (k == P) { ++c; k = 0; }
    if (gz < gend) {
      fetch_zv(gz + 1);
      if (TL::DB && stored(gz + 1)) y_phase(gz + 1);
    }
  }
}

// ---- kernels -------------------------------------------------------------------------------------
// 1D grid, vector tile fastest: the CTAs that read the neighbouring parts of a node's rows run
// side by side, then neighbouring xy blocks, which share halos in L2.
template <class TL, bool CPLX, bool FULL>
__global__ void __launch_bounds__(TL::NT, TL::RES)
sweep_kernel(const SweepCoef<typename TL::V::T> cf, const KronGeom g,
             const SweepIO<typename TL::V::T> io, int nvt) {
  const int b = blockIdx.x, nxy = g.nbx * g.nby, r = b / nvt;
  sweep_body<TL, CPLX, FULL>(cf, g, io, r % nxy, b % nvt, r / nxy);
}

// instance of item b in the concatenated grids (ascending first-CTA offsets)
template <typename T>
__device__ __forceinline__ int sweep_instance(const KronInst<T>* inst, int n, int64_t b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].cta0 <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}
template <class TL, bool FULL>
__device__ __forceinline__ void sweep_item(const SweepCoef<typename TL::V::T>& cf,
                                           const KronInst<typename TL::V::T>* inst, int n, int64_t b) {
  const int i = sweep_instance(inst, n, b);
  const KronGeom g = inst[i].g;
  const SweepIO<typename TL::V::T> io = inst[i].io;
  const int64_t local = b - inst[i].cta0, nvt = inst[i].nvt, r = local / nvt;
  const int nxy = g.nbx * g.nby;
  sweep_body<TL, false, FULL>(cf, g, io, (int)(r % nxy), (int)(local % nvt), (int)(r / nxy));
}

// Batched form: many independent meshes that share p and the cell size in one launch, their
// CTA grids concatenated.
template <class TL, bool FULL>
__global__ void __launch_bounds__(TL::NT, TL::RES)
sweep_batch_kernel(const SweepCoef<typename TL::V::T> cf,
                   const KronInst<typename TL::V::T>* __restrict__ inst, int ninst) {
  sweep_item<TL, FULL>(cf, inst, ninst, blockIdx.x);
}

// Persistent batched form: resident CTAs take the items of that grid from a device counter,
// which balances slabs of uneven height.
template <class TL, bool FULL>
__global__ void __launch_bounds__(TL::NT, TL::RES)
sweep_batch_persist_kernel(const SweepCoef<typename TL::V::T> cf,
                           const KronInst<typename TL::V::T>* __restrict__ inst, int ninst,
                           int64_t total, unsigned long long* __restrict__ counter) {
  __shared__ long long s_item;
  for (;;) {
    __syncthreads();   // every thread is done with the previous item's shared memory
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(counter, 1ull);
    __syncthreads();
    const int64_t b = s_item;
    if (b >= total) break;
    sweep_item<TL, FULL>(cf, inst, ninst, b);
  }
}

// ---- tiles and launches -----------------------------------------------------------------------
// Cells of a CTA per degree: about ten nodes a side, so that the y threads, the xz threads and
// the staged halo stay in proportion, and the accumulators (XC P (p + 1) packed values) within
// the registers of two to four CTAs an SM; a, b of two planes (one barrier a plane) except
// where their shared memory would cost a CTA.
template <class V, int P, int VP>
struct SweepTileFor;
#define FE_SWEEP_TILE(p, cx, cy, xc, vp, res, db)     \
  template <class V>                                  \
  struct SweepTileFor<V, p, vp> {                     \
    using type = SweepTile<V, p, cx, cy, xc, vp, res, db>; \
  };
FE_SWEEP_TILE(1, 8, 8, 4, 8, 4, false)
FE_SWEEP_TILE(1, 8, 8, 4, 4, 4, false)
FE_SWEEP_TILE(2, 4, 4, 2, 8, 4, false)
FE_SWEEP_TILE(2, 4, 4, 2, 4, 4, false)
FE_SWEEP_TILE(3, 3, 3, 1, 8, 2, true)
FE_SWEEP_TILE(3, 3, 3, 1, 4, 4, true)
FE_SWEEP_TILE(4, 2, 2, 1, 8, 4, false)
FE_SWEEP_TILE(4, 2, 2, 1, 4, 4, true)
FE_SWEEP_TILE(5, 2, 2, 1, 8, 2, true)
FE_SWEEP_TILE(5, 2, 2, 1, 4, 3, true)
FE_SWEEP_TILE(6, 2, 2, 1, 4, 2, true)
#undef FE_SWEEP_TILE

// packed elements of a tile: eight, or four where the block has no more (and at p = 6, whose
// accumulators and planes would leave one CTA an SM)
template <class V>
inline int sweep_vp(int p, int64_t nvec) {
  return p == 6 || nvec <= 4 * V::LANES ? 4 : 8;
}

template <class V, class F>
auto sweep_tile(int p, int vp, F&& f) {
#define FE_SWEEP_CASE(pp) \
  case pp: return vp == 4 ? f(typename SweepTileFor<V, pp, 4>::type{}) : f(typename SweepTileFor<V, pp, 8>::type{});
  switch (p) {
    FE_SWEEP_CASE(1) FE_SWEEP_CASE(2) FE_SWEEP_CASE(3) FE_SWEEP_CASE(4) FE_SWEEP_CASE(5)
    default: return f(typename SweepTileFor<V, 6, 4>::type{});
  }
#undef FE_SWEEP_CASE
}

inline int sweep_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
    cudaGetLastError();
    sms = 152;
  }
  return sms;
}

// Layers of a z segment.  A segment works through the layer below it again, so segments cost a
// layer each and are worth it only where the grid would leave SMs idle: the length with the
// least (layers + 1) x CTAs an SM.  A float CTA alone on an SM runs about 1.5 times as fast as
// its share of a full one; double ones only share the FP64 pipe.
template <typename T>
inline int sweep_zseg(int64_t base, int nz) {
  const int64_t sms = sweep_sms();
  const double alone = sizeof(T) == 8 ? 1.0 : 1.5;
  int best = nz;
  double cost = 1e300;
  for (int s = 1; s <= nz;) {
    const int z = (nz + s - 1) / s, segs = (nz + z - 1) / z;
    const double per = std::max(alone, (double)((base * segs + sms - 1) / sms));
    const double t = (z + (segs > 1 ? 1 : 0)) * per;
    if (t < cost * (1.0 - 1e-9)) { cost = t; best = z; }
    if (z == 1) break;
    s = (int)(((int64_t)nz + z - 2) / (z - 1));   // the next shorter segment: 2 sqrt(nz) lengths, not nz
  }
  return best;
}

template <class TL>
void sweep_fill(KronGeom& g) {
  g.bx = TL::CX;
  g.by = TL::CY;
  g.nbx = (g.NX / g.p + TL::CX - 1) / TL::CX;
  g.nby = (g.NY / g.p + TL::CY - 1) / TL::CY;
}

template <class TL>
int64_t sweep_vtiles(int64_t nvec) {
  return (nvec + TL::VP * TL::V::LANES - 1) / (TL::VP * TL::V::LANES);
}

// whole xy blocks and vector tiles: no ownership or ragged-vector test anywhere in the sweep
template <class TL>
bool sweep_full(const KronGeom& g, int64_t nvec) {
  return g.NX % TL::BXn == 0 && g.NY % TL::BYn == 0 && nvec % (TL::VP * TL::V::LANES) == 0;
}

template <typename T>
SweepCoef<T> sweep_coef(const KronCoef& cf, double bgx, double bgy) {
  // the kinetic scales K / (2 J) and the Bloch scales G / J over cz = az / (2 J)
  SweepCoef<T> c;
  const double cz = cf.az * cf.zin * cf.zout;
  c.rx = (T)(cf.ax / cf.az);
  c.ry = (T)(cf.ay / cf.az);
  c.gx = (T)(bgx * cf.zin * cf.zin / cz);
  c.gy = (T)(bgy * cf.zin * cf.zin / cz);
  return c;
}

// The kinetic energy that the tables, rounded to T, give the constant function (0 exactly):
// the Rayleigh quotient of one direction's matrix.
template <typename T, int P>
constexpr double sweep_null_shift() {
  double q = 0.0, n = 0.0;
  for (int j = 0; j <= P; ++j) {
    for (int k = 0; k <= P; ++k) q += hat_n<P>(j) * (double)(T)hat_k<P>(j, k) * hat_n<P>(k);
    if (j < P) n += hat_n<P>(j) * hat_n<P>(j);
  }
  return sizeof(T) == 8 ? 0.0 : q / n;
}

// Scalars of Y = alpha (Ht - shift) X + beta Z.  The launch takes al = alpha cz, and what
// multiplies it is chosen against the rounded al.  A filter step's shift is tens of Hartree and
// its states a few, so in float a relative rounding of any factor on it (the shift itself, vs,
// al) would move the whole spectrum by up to 4e-6 Ha, the same way in every step: v0 holds, to
// double accuracy, what the rounded product vs (V - shift) leaves of the shift, and the null
// shift of the rounded tables.
template <typename T>
void sweep_scalars(const KronCoef& cf, int p, double alpha, double beta, double shift,
                   SweepIO<T>* io) {
  const double k = cf.zin * cf.zout, cz = cf.az * k;
  double null1 = 0.0;
  switch (p) {
    case 1: { constexpr double d = sweep_null_shift<T, 1>(); null1 = d; break; }
    case 2: { constexpr double d = sweep_null_shift<T, 2>(); null1 = d; break; }
    case 3: { constexpr double d = sweep_null_shift<T, 3>(); null1 = d; break; }
    case 4: { constexpr double d = sweep_null_shift<T, 4>(); null1 = d; break; }
    case 5: { constexpr double d = sweep_null_shift<T, 5>(); null1 = d; break; }
    default: { constexpr double d = sweep_null_shift<T, 6>(); null1 = d; break; }
  }
  io->al = (T)(alpha * cz);
  const double al = (double)io->al;
  io->zs = al != 0.0 ? (T)(beta / al) : T(0);
  io->vs = al != 0.0 ? (T)(alpha / al) : T(0);
  io->shift = (T)shift;
  const double c = shift + null1 * (cf.ax + cf.ay + cf.az) * k;
  io->v0 = al != 0.0 ? (T)((double)io->vs * (double)io->shift - alpha / al * c) : T(0);
  if (beta == 0.0) io->Z = nullptr;
}

template <typename K>
inline fe_status sweep_setup(K kern, size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fe_fail(FE_ECUDA, "kernel attributes: %s", cudaGetErrorString(e));
  }
  return FE_OK;
}

// what every block of a launch has to satisfy (the entry points check the alignment)
template <typename T>
inline fe_status sweep_check(const KronGeom& g, const SweepIO<T>& io) {
  if (!io.V) return fe_fail(FE_EINVAL, "operator: no potential");
  if (io.al == T(0)) return fe_fail(FE_EINVAL, "operator: alpha is zero");
  if ((uint64_t)g.NX * g.NY * io.ld * sizeof(T) / 16 >= (1ull << 32))
    return fe_fail(FE_EINVAL, "operator: a z plane of the block exceeds 64 GB");
  return FE_OK;
}

template <class V>
fe_status sweep_run(const KronCoef& cf, double bgx, double bgy, const KronGeom& g0,
                    const SweepIO<typename V::T>& io, cudaStream_t st) {
  using T = typename V::T;
  FE_TRY(sweep_check(g0, io));
  const SweepCoef<T> c = sweep_coef<T>(cf, bgx, bgy);
  const bool cplx = bgx != 0.0 || bgy != 0.0;
  if (cplx && io.nvec % 2 != 0)
    return fe_fail(FE_EINVAL, "complex operator needs interleaved (re, im) lane pairs");
  return sweep_tile<V>(g0.p, sweep_vp<V>(g0.p, io.nvec), [&](auto tile) -> fe_status {
    using TL = decltype(tile);
    KronGeom g = g0;
    sweep_fill<TL>(g);
    const int64_t nvt = sweep_vtiles<TL>(io.nvec), base = (int64_t)g.nbx * g.nby * nvt;
    g.zseg = sweep_zseg<T>(base, g.nz);
    const int64_t total = base * ((g.nz + g.zseg - 1) / g.zseg);
    if (total > 0x7fffffffLL) return fe_fail(FE_EINVAL, "grid too large");
    const bool full = sweep_full<TL>(g, io.nvec);
    auto kern = cplx ? (full ? sweep_kernel<TL, true, true> : sweep_kernel<TL, true, false>)
                     : (full ? sweep_kernel<TL, false, true> : sweep_kernel<TL, false, false>);
    FE_TRY(sweep_setup(kern, TL::SMEM));
    kern<<<(unsigned)total, TL::NT, TL::SMEM, st>>>(c, g, io, (int)nvt);
    fe_count_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fe_fail(FE_ECUDA, "operator launch: %s", cudaGetErrorString(e));
    return FE_OK;
  });
}

// widest block of a batch: its tile serves every instance
template <typename T>
int64_t sweep_widest(const KronInst<T>* inst, int n) {
  int64_t w = 1;
  for (int i = 0; i < n; ++i) w = std::max(w, inst[i].io.nvec);
  return w;
}

// Batched plan: tile fields, z segmentation (the requested length, or the rule above over the
// whole batch and its tallest slab), vector tiles and first CTAs; the total CTA count.
template <class V>
int64_t sweep_batch_plan(int p, KronInst<typename V::T>* inst, int n, int zseg_req) {
  return sweep_tile<V>(p, sweep_vp<V>(p, sweep_widest(inst, n)), [&](auto tile) -> int64_t {
    using TL = decltype(tile);
    int nzmax = 1;
    int64_t base = 0;
    for (int i = 0; i < n; ++i) {
      KronGeom& g = inst[i].g;
      sweep_fill<TL>(g);
      inst[i].nvt = sweep_vtiles<TL>(inst[i].io.nvec);
      inst[i].full = sweep_full<TL>(g, inst[i].io.nvec);
      nzmax = std::max(nzmax, g.nz);
      base += (int64_t)g.nbx * g.nby * inst[i].nvt;
    }
    const int zseg = zseg_req > 0 ? std::min(zseg_req, nzmax) : sweep_zseg<typename V::T>(base, nzmax);
    int64_t cta = 0;
    for (int i = 0; i < n; ++i) {
      KronGeom& g = inst[i].g;
      g.zseg = zseg;
      inst[i].cta0 = cta;
      cta += (int64_t)g.nbx * g.nby * inst[i].nvt * ((g.nz + zseg - 1) / zseg);
    }
    return cta;
  });
}

// One operator application over the device copy of the instances (widest: their widest block,
// as the plan saw it; full: of every instance); counter: one device word for the persistent form, or nullptr.
template <class V>
fe_status sweep_batch_run(const KronCoef& cf, int p, int64_t widest, bool full,
                          const KronInst<typename V::T>* d_inst, int n, int64_t total, cudaStream_t st,
                          unsigned long long* counter) {
  if (total < 1 || total > 0x7fffffffLL)
    return fe_fail(FE_EINVAL, "batched grid of %lld CTAs", (long long)total);
  const SweepCoef<typename V::T> c = sweep_coef<typename V::T>(cf, 0.0, 0.0);
  return sweep_tile<V>(p, sweep_vp<V>(p, widest), [&](auto tile) -> fe_status {
    using TL = decltype(tile);
    if (counter) {
      auto kern = full ? sweep_batch_persist_kernel<TL, true> : sweep_batch_persist_kernel<TL, false>;
      FE_TRY(sweep_setup(kern, TL::SMEM));
      int per_sm = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TL::NT, TL::SMEM) != cudaSuccess ||
          per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
      }
      const int64_t grid = std::min<int64_t>(total, (int64_t)per_sm * sweep_sms());
      if (cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st) != cudaSuccess) {
        cudaGetLastError();
        return fe_fail(FE_ECUDA, "batched operator: counter reset failed");
      }
      kern<<<(unsigned)grid, TL::NT, TL::SMEM, st>>>(c, d_inst, n, total, counter);
    } else {
      auto kern = full ? sweep_batch_kernel<TL, true> : sweep_batch_kernel<TL, false>;
      FE_TRY(sweep_setup(kern, TL::SMEM));
      kern<<<(unsigned)total, TL::NT, TL::SMEM, st>>>(c, d_inst, n);
    }
    fe_count_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fe_fail(FE_ECUDA, "batched operator launch: %s", cudaGetErrorString(e));
    return FE_OK;
  });
}

}  // namespace fe
