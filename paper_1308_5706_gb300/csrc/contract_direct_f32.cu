// Instantiations of the direct contraction (contract_direct.cuh) for float.
#include "contract_direct.cuh"

namespace s2dw {

template void launch_contract_direct<float>(int, bool, int, const DirTasks<float>&, const DirTasks<float>&, const CallPtrs&,
                                        cudaStream_t);

// shared-memory caps (once per device, under the caller's lock)
cudaError_t contract_direct_prepare_f32() { return dir_attrs<float>(); }

}  // namespace s2dw
