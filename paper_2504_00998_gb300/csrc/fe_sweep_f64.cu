// Instantiations of the Hamiltonian sweep kernel: double blocks.
#include "fe_sweep.cuh"

namespace fe {

fe_status sweep_f64(const KronCoef& cf, double bgx, double bgy, const KronGeom& g,
                    const SweepIO<double>& io, cudaStream_t st) {
  return sweep_run<PackD>(cf, bgx, bgy, g, io, st);
}

void sweep_scalars_f64(const KronCoef& cf, int p, double alpha, double beta, double shift,
                       SweepIO<double>* io) {
  sweep_scalars<double>(cf, p, alpha, beta, shift, io);
}

}  // namespace fe
