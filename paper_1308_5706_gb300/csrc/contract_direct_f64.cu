// Instantiations of the direct contraction (contract_direct.cuh) for double.
#include "contract_direct.cuh"

namespace s2dw {

template void launch_contract_direct<double>(int, bool, int, const DirTasks<double>&, const DirTasks<double>&, const CallPtrs&,
                                        cudaStream_t);

// shared-memory caps (once per device, under the caller's lock)
cudaError_t contract_direct_prepare_f64() { return dir_attrs<double>(); }

}  // namespace s2dw
