// Instantiations and launchers of the FP32 contraction of large band-limits
// (contract_tile.cuh), and the per-call packing of f_lm into its layout.
#include "contract_tile.cuh"

namespace s2dw {

// fP[b][l][re, im][c] = f_{l, 32 b + c} for 32 b + c <= l < L, else 0 (Lrf rows
// per block).  Grid (ceil(Lrmax / 8), max blocks, jobs); 8 rows l per CTA.
__global__ void __launch_bounds__(256) k_fpack(const ContractDesc<float>* __restrict__ descs, CallPtrs ptrs) {
  begin_after();
  const int job = blockIdx.z, b = blockIdx.y;
  const ContractDesc<float>* D = descs + job;
  const int L = D->L, Lrf = D->Lrf;
  if (!D->fP || 32 * b >= L) return;  // (a plan of the direct contraction reads f itself)
  const int l = blockIdx.x * 8 + (threadIdx.x >> 5), c = threadIdx.x & 31;
  if (l >= Lrf) return;
  const int m = 32 * b + c;
  const float2* __restrict__ f = reinterpret_cast<const float2*>(ptrs.f[job]);
  const float2 v = (l < L && m <= l) ? f[l * l + l + m] : make_float2(0.f, 0.f);
  float* dst = const_cast<float*>(reinterpret_cast<const float*>(D->fP)) + ((size_t)b * Lrf + l) * 64;
  dst[c] = v.x;
  dst[32 + c] = v.y;
}

void launch_fpack(const ContractDesc<float>* descs, int njobs, int nbmax, int Lrmax, const CallPtrs& ptrs,
                  cudaStream_t st) {
  if (njobs <= 0 || nbmax <= 0) return;
  dim3 grid((Lrmax + 7) / 8, nbmax, njobs);
  launch_after(k_fpack, grid, 256, 0, st, descs, ptrs);
}

bool tile_both_halves(int N) { return N <= 6; }

namespace {

// f(kernel geometry) for N orders and nslot slots
template <typename F>
void tile_pick(int N, int nslot, F&& f) {
  if (nslot == 1) {
    f(std::integral_constant<int, 1>(), std::integral_constant<int, 1>());
    return;
  }
  constexpr std::integral_constant<int, 2> two{};
  switch (N) {
    case 1: f(std::integral_constant<int, 1>(), two); break;
    case 2: f(std::integral_constant<int, 2>(), two); break;
    case 3: f(std::integral_constant<int, 3>(), two); break;
    case 4: f(std::integral_constant<int, 4>(), two); break;
    case 5: f(std::integral_constant<int, 5>(), two); break;
    case 6: f(std::integral_constant<int, 6>(), two); break;
    case 7: f(std::integral_constant<int, 7>(), two); break;
    case 8: f(std::integral_constant<int, 8>(), two); break;
    default: break;
  }
}

}  // namespace

void launch_contract_tile(int N, int nslot, bool syn, const ContractDesc<float>* descs, const CTask* tasks, int ntasks,
                          cudaStream_t st, long long limit) {
  if (ntasks <= 0) return;
  tile_pick(N, nslot, [&](auto n, auto s) {
    constexpr int NN = decltype(n)::value, NS = decltype(s)::value, H = NN <= 6 ? 2 : 1;
    if (syn)
      launch_after(k_contract_tile<NN, NS, true, H>, ntasks, 256, TileGeom<NN, NS, true, H>::SMEM, st, descs, tasks, limit);
    else
      launch_after(k_contract_tile<NN, NS, false, H>, ntasks, 256, TileGeom<NN, NS, false, H>::SMEM, st, descs, tasks, limit);
  });
}

// Shared-memory caps of every instantiation (once per device, under the caller's lock).
cudaError_t contract_tile_prepare() {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i <= 8; ++i)
    tile_pick(i == 0 ? 1 : i, i == 0 ? 1 : 2, [&](auto n, auto s) {
      constexpr int NN = decltype(n)::value, NS = decltype(s)::value, H = NN <= 6 ? 2 : 1;
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_contract_tile<NN, NS, true, H>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)TileGeom<NN, NS, true, H>::SMEM);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_contract_tile<NN, NS, false, H>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)TileGeom<NN, NS, false, H>::SMEM);
    });
  return e;
}

cudaError_t pair_timeouts(int* count) {
  cudaError_t e = cudaMemcpyFromSymbol(count, g_pair_timeouts, sizeof(int));
  if (e != cudaSuccess) return e;
  const int zero = 0;
  return cudaMemcpyToSymbol(g_pair_timeouts, &zero, sizeof(int));
}

}  // namespace s2dw
