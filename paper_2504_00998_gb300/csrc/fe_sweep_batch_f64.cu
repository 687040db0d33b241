// Instantiations of the batched Hamiltonian sweep kernels: double blocks.
#include "fe_sweep.cuh"

namespace fe {

int64_t sweep_batch_plan_f64(int p, KronInst<double>* inst, int n, int zseg_req) {
  return sweep_batch_plan<PackD>(p, inst, n, zseg_req);
}

fe_status sweep_batch_f64(const KronCoef& cf, int p, int64_t widest, bool full,
                          const KronInst<double>* d_inst, int n, int64_t total, cudaStream_t st, unsigned long long* counter) {
  return sweep_batch_run<PackD>(cf, p, widest, full, d_inst, n, total, st, counter);
}

}  // namespace fe
