// Instantiations of the batched Hamiltonian sweep kernels: float blocks.
#include "fe_sweep.cuh"

namespace fe {

int64_t sweep_batch_plan_f32(int p, KronInst<float>* inst, int n, int zseg_req) {
  return sweep_batch_plan<PackF>(p, inst, n, zseg_req);
}

fe_status sweep_batch_f32(const KronCoef& cf, int p, int64_t widest, bool full,
                          const KronInst<float>* d_inst, int n, int64_t total, cudaStream_t st, unsigned long long* counter) {
  return sweep_batch_run<PackF>(cf, p, widest, full, d_inst, n, total, st, counter);
}

}  // namespace fe
