// Instantiations of the Hamiltonian sweep kernel: float blocks.
#include "fe_sweep.cuh"

namespace fe {

fe_status sweep_f32(const KronCoef& cf, double bgx, double bgy, const KronGeom& g,
                    const SweepIO<float>& io, cudaStream_t st) {
  return sweep_run<PackF>(cf, bgx, bgy, g, io, st);
}

void sweep_scalars_f32(const KronCoef& cf, int p, double alpha, double beta, double shift,
                       SweepIO<float>* io) {
  sweep_scalars<float>(cf, p, alpha, beta, shift, io);
}

}  // namespace fe
