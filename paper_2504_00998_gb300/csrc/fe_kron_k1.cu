// Instantiations of the scratch-free stiffness product (one double vector).
#include "fe_kron.cuh"

namespace fe {

fe_status kron_k1(const KronCoef& cf, const KronGeom& g, const double* x, double* y, cudaStream_t st) {
  switch (g.p) {
    case 1: return kron_launch<KronTile<1>>(cf, g, x, y, st);
    case 2: return kron_launch<KronTile<2>>(cf, g, x, y, st);
    case 3: return kron_launch<KronTile<3>>(cf, g, x, y, st);
    case 4: return kron_launch<KronTile<4>>(cf, g, x, y, st);
    case 5: return kron_launch<KronTile<5>>(cf, g, x, y, st);
    case 6: return kron_launch<KronTile<6>>(cf, g, x, y, st);
    default: return fe_fail(FE_EUNSUPPORTED, "p = %d", g.p);
  }
}

}  // namespace fe
