// Final synthesis reduction for float (FP32 contractions: contract_tile.cuh, contract_direct.cuh).
#include "contract.cuh"

namespace s2dw {

template <>
void launch_syn_reduce<float>(const ReduceJobs& jobs, int njobs, int Lmax, cudaStream_t st) {
  if (njobs <= 0) return;
  dim3 grid((Lmax + 127) / 128, Lmax, njobs), block(128);
  launch_after(k_syn_reduce<float>, grid, block, 0, st, jobs);
}

int contract_rows_per_thread(bool fp64) { return fp64 ? 2 : 4; }

}  // namespace s2dw
