// Internal descriptors shared by the plan, the launchers and the kernels.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace s2dw {

constexpr int MAXS = 66;   // wavelet scales (<= 64) plus headroom
constexpr int MAXB = 64;   // transforms per batched launch
constexpr int TILE = 32;   // contraction tile edge (m' and m)
constexpr int LCH = 8;     // l-chunk of the synthesis in-tile reduction
constexpr long long kWaitLimit = 2000000000LL;  // cycles of a bounded wait: about one second at the maximum SM clock

// One l-segment on which the scale held by each of the two accumulator
// slots is constant (slot s holds the scale j with j % 2 == s, or -1).
struct LSeg {
  int lo, hi;
  int j[2];
};

// Launch of a kernel that begins with begin_after(): its launch overlaps the end
// of the kernel before it in the stream (under capture: a programmatic edge).
// Measured, plain launches -> this, analysis / synthesis, us: L = 32, N = 3 21 / 32 ->
// 14 / 24; L = 128, N = 5 50 / 60 -> 40 / 47; L = 361, N = 4 141 / 157 -> 128 / 140;
// L = 1024, N = 5 1105 / 1338 -> 1083 / 1314.  No kernel asks for its successor
// earlier (griddepcontrol.launch_dependents at its start): the waiting CTAs
// then shared the SMs' resources and filled them unevenly, L = 128 46 / 50, L =
// 1024 1169 / 1384.
template <typename... P, typename... A>
inline void launch_after(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// Static, per-plan description of one contraction pass (wavelet scales with
// N orders, or the scaling function with N = 1), device resident.
template <typename T>
struct ContractDesc {
  const T* delta;    // Delta table (padded eighth domain; FP64 plans)
  // contract_direct.cuh and (FP32 plans) contract_tile.cuh:
  const T* dpair;      // Delta pair table of the plan's shared table
  const T* RSp;        // [nb][Lr][nslot][(N+1)/2][32]: R rows per 32-block of m', l outermost
  const cx<T>* fP;     // [nb][Lrf][re, im][32] (as floats): f_lm per 32-block of m (zero for m > l), packed per call
  int Lr, Lrf;         // l rows of RSp and fP (>= L + 7: a stage may read seven l past the last)
  const T* RS;       // [L][nslot][(N+1)/2][Lp]: Delta^l_{m',n_k} kappa^j(l) |s_{l,n_k}|, n_k >= 0
  cx<T>* P;          // synthesis partials [nbr][L][Lp32]
  int L, Lp, Lp32, nbr;
  int nseg;
  int N, nslot, eta_odd;   // eta_odd: N even -> eta = i
  // gamma factors [k N + g]: analysis conj(eta) i^{n_k} e^{i n_k gamma_g},
  // synthesis eta (2 pi/N) i^{-n_k} e^{-i n_k gamma_g} (direct FP32 contraction)
  cx<T> cga[64], cgs[64];
  int Lj[MAXS];            // per scale band-limit (support hi + 1)
  cx<T>* Y[MAXS];          // per scale cube [N][Lj][Lj] (analysis out / synthesis in)
  LSeg seg[2 * MAXS + 2];
  int jlo[MAXS], jhi[MAXS];  // per scale first and last l with a nonzero kernel (empty: jhi < jlo)
};

// l rows of padding after the tables the FP32 contraction streams (the
// pair table's last run, the R rows and f values of each block): a pipeline
// stage of up to eight l may read seven l past a tile's last l; the values
// read there never enter the sums.
constexpr int kPairPadL = 8;

// Pair table of reach Lmax (a multiple of 32): pairs ordered by q, then p;
// the run of pair (p, q) holds Lmax - 32 q blocks of 32 x 32 entries.
// Entry of its first block (l = 32 q):
//   1024 * (Lmax q (q+1)/2 - 32 (q-1) q (q+1)/3 + p (Lmax - 32 q)).
__host__ __device__ __forceinline__ long long pair_run_base(int p, int q, int Lmax) {
  const long long Q = q;
  return 1024LL * ((long long)Lmax * Q * (Q + 1) / 2 - 32LL * (Q - 1) * Q * (Q + 1) / 3 + (long long)p * (Lmax - 32 * Q));
}
// entries of the whole table (+ one stage of read-ahead past the last run)
__host__ __device__ __forceinline__ long long pair_table_entries(int Lmax) {
  return pair_run_base(0, Lmax / 32, Lmax) + kPairPadL * 1024;
}

// One task of the FP32 contractions: a tile of the block pair p <= q (half 0: m'
// in block p, m in q; half 1: the other way round), or both tiles
// (tile_both_halves), over l in [lstart, lend].  j, j2: scales of the two slots
// (-1: none); the direct analysis takes one scale, j, held in R slot `slot`.
// 16 bytes: a batch of 64 transforms has some 1e5 tasks, built and copied to
// the device when its plan set is first used.
struct CTask {
  uint8_t prob, p, q, half;
  int8_t j, j2, slot, pad;
  int16_t lstart, lend, Lmax, pad2;  // Lmax: reach of the pair table
  __host__ __device__ __forceinline__ long long dbase() const {  // pair-table entry of lstart
    return pair_run_base(p, q, Lmax) + 1024LL * (lstart - 32 * q);
  }
};
static_assert(sizeof(CTask) == 16 && MAXB <= 256 && MAXS <= 127, "task fields");

struct TileTask {
  int prob;    // index into the descriptor array of the launch
  int bmp;     // m' block
  int bm;      // m block
  int lstart;  // first l of the tile (max(32 bmp, 32 bm))
  int lend;    // last l with a nonzero contribution
};

// Per-call pointers, passed by value to the kernels.
struct CallPtrs {
  const void* f[MAXB];   // analysis input f_lm
  void* out[MAXB];       // synthesis output f_lm
  void* W[MAXB];         // wavelet coefficients
  void* Wphi[MAXB];      // scaling coefficients
};

enum CztKind {
  CZT_BETA_ANA = 0,
  CZT_ALPHA_ANA = 1,
  CZT_ALPHA_SYN = 2,
  CZT_BETA_SYN = 3,
  CZT_ALPHA_ANA_DIRECT = 4,  // small-band scales, direct sums
  CZT_ALPHA_SYN_DIRECT = 5,
  CZT_BETA_ANA_FFT = 6,      // beta sums as one FFT of length 4L (L a power of two)
  CZT_BETA_SYN_FFT = 7,
  CZT_ALPHA_ANA_SEG = 8,     // segmented chirp-z (bands small next to L)
  CZT_ALPHA_SYN_SEG = 9,
  CZT_BETA_MW_DFT = 10,      // MW grid, synthesis: torus coefficients from the L beta samples
  CZT_BETA_RS_FFT = 11,      // MW grid, synthesis: those coefficients evaluated on the DH beta grid
  CZT_BETA_RS = 12,          //   (single FFT, or chirp-z for non-power-of-two L)
  CZT_BETA_ANA_DCT = 13,     // beta sums as half-length transforms (L a power of two, L >= 16)
  CZT_BETA_SYN_DCT = 14,
  CZT_BETA_RS_DCT = 15,      //   (MW grid, synthesis: evaluation on the DH beta grid)
  SG_KIND_BETA_ANA = 16,     // split matrix products on the tensor cores (FP32 plans)
  SG_KIND_BETA_SYN = 17,
  SG_KIND_ALPHA_ANA = 18,
  SG_KIND_ALPHA_SYN = 19,
  SG_KIND_BETA_RS = 20       //   (MW grid, synthesis: evaluation on the DH beta grid)
};
// Or-ed into an alpha chirp-z kind: the list may hold segments with an odd row
// count N nb (MW grid), whose last row pair has one row.
constexpr int CZT_ODD_ROWS = 0x100;
// shared memory of the segmented chirp-z kernels: two buffers of M' (+ padding)
// for each of the 4096 / M' row pairs of a CTA
template <typename T>
constexpr size_t alpha_seg_smem() { return 2 * (size_t)(4096 + 4096 / 16) * 2 * sizeof(T); }
constexpr int kDirectMaxLj = 32;     // synthesis: direct alpha sums for L_j <= 32
constexpr int kDirectMaxLjAna = 32;  // analysis: direct (matrix-product) alpha sums for L_j <= 32
// tile of the direct analysis kernel: samples per CTA, rows per pass, fewest rows per CTA
constexpr int kAgCols = 128, kAgRows = 64, kAgMinRows = 16;
template <typename T>  // B tile + A tile
constexpr size_t alpha_ana_direct_smem() {
  return (size_t)(2 * kDirectMaxLjAna - 1) * (kAgCols + kAgRows) * sizeof(T);
}
// row pairs (complex transforms) per CTA of the alpha chirp-z kernels: one
// (FP32 measured 9% faster at three CTAs per SM than two transforms per CTA
// sharing their table loads at two CTAs per SM; FP64 buffers allow one)
__host__ __device__ constexpr int alpha_czt_nt(bool fp64) { return (void)fp64, 1; }
// adjacent columns per CTA of the single-FFT beta kernels (FP32: a 16-byte pair)
__host__ __device__ constexpr int beta_fft_nt(bool fp64) { return fp64 ? 1 : 2; }
// adjacent columns per CTA of the chirp-z beta kernels for transforms of
// length 2^logM: FP32 a 16-byte pair up to 2^12, one at 2^13 (so that a CTA's
// buffers stay at 2 x 4352 complex); FP64 one
__host__ __device__ constexpr int beta_czt_cols(int logM, bool fp64) { return (fp64 || logM >= 13) ? 1 : 2; }
inline int direct_rows_syn(bool fp64) { return fp64 ? 4 : 8; }  // 32-byte line per alpha sample

// One segment of a chirp-z launch: all columns / row pairs of one scale of
// one transform.
template <typename T>
struct CztSeg {
  int start;      // first CTA index of this segment
  int items;
  int job;        // index into CallPtrs
  int L, Lj, N, logM;
  int64_t woff;   // element offset of this scale in W (or 0 for Wphi)
  int is_phi;     // 1: W pointer is CallPtrs::Wphi
  cx<T>* buf_in;  // plan workspace input (X / Y buffers)
  cx<T>* buf_out; // plan workspace output
  const cx<T>* H; // bit-reversed chirp kernel spectrum, scaled by 1/M
  const cx<T>* tw;
  const cx<T>* pre;
  const cx<T>* post;
  T scale;
  int P, nsegs;   // segmented chirp-z: samples per segment, segments
  int tabP, tabK, tabD;  // split products: basis tiles and stages of the table, first data stage of the launch
  int nb;         // beta samples per gamma sample (rows of X, V and W per g): 2L, or L on the MW grid
};

// Direct alpha sums on the tensor cores (FP32 plans, scales with L_j <= 32;
// alpha_tc.cu).  Basis tables: one per scale and direction, built per plan.
size_t alpha_tc_table_floats(int L, int Lj, bool syn);
struct TcBasis {
  float* out;
  int L;
  short Lj, syn;
};
cudaError_t alpha_tc_build_tables(const TcBasis* tables, int n, cudaStream_t st);  // n <= 2 MAXS
int alpha_tc_items(int L, int rows, int njobs, bool syn, int& P);  // CTAs; P: rows per CTA
void launch_alpha_tc(bool syn, const CztSeg<float>* segs, int nseg, int total_items, const CallPtrs& ptrs,
                     cudaStream_t st, long long limit = kWaitLimit);
cudaError_t alpha_tc_prepare();
cudaError_t alpha_tc_timeouts(int* count);  // reads and resets the device count
cudaError_t alpha_tc_wait_probe(long long limit, cudaStream_t st);  // a wait that runs out

// Beta and alpha sums as split FP16 matrix products on the tensor cores
// (split_gemm.cu).  Modes 0 beta analysis, 1 beta synthesis, 2 alpha analysis, 3
// alpha synthesis; basis tables per grid, laid out per stage of 32 terms.
constexpr int kSgDataBytes = 4 * 16 * 512 + 512;  // one data stage of 128 rows: operand images, inverse row scales
struct SgTable {
  int sets, tiles, stages;
  size_t bytes;
};
struct SgDims {
  int data_tiles, basis_tiles, stages;
};
SgTable sg_table(int mode, int L);
SgDims sg_dims(int mode, int L, int Lj, int N, int nb);
float sg_out_scale(int mode, int L);
size_t sg_build_scratch(int L);  // double2
cudaError_t sg_build_tables(void* const* out, double2* scratch, const double* qw, int L, bool mw, cudaStream_t st);
void launch_split_gemm(int mode, const CztSeg<float>* segs, int nseg, int total, int stages, const CallPtrs& ptrs,
                       cudaStream_t st, long long limit = kWaitLimit);
// Whether the products are the faster form.  beta: the chirp-z (other L than
// powers of two) costs two FFTs of M >= 4L per column: 20.5 against 20 us at L =
// 100, N = 3, 30 against 21 at L = 200; the half-length transforms of
// power-of-two L one of 2L: 230 against 243 us at L = 1024, N = 5, 2807 against
// 2144 at L = 2048, N = 8.
inline bool sg_beta_faster(int L, bool pow2) { return pow2 ? L >= 2048 : L > 112; }
// alpha, band L_j on a grid of band-limit L: a row costs L L_j terms here, a
// chirp-z `fft_cost` = (FFTs) x (length) x log2(length) (two FFTs of M, or S + 1
// of M' segmented).  Per row at L = 1024, N = 5: 16 ps per term against 0.1 ps
// per unit of that cost; below L = 128 the two launches cost more than they save
// (L = 64, N = 3 18 against 10.5 us, L = 128, N = 5 21 against 27).  Lines at 4 / 6.5 /
// 9 / 13 times the cost, analysis and synthesis of the whole call, us: where 9
// moves segmented scales, L = 1024, N = 5 2452 / 2400 / 2364 / 2526, L = 1500, N = 3
// 4741 / 4705 / 4652 / 4655; where it moves a full chirp-z, L = 900, N = 3 1383 /
// 1357 / 1415 / 1414.
inline bool sg_alpha_faster(int L, int Lj, double fft_cost, bool segmented) {
  return L >= 128 && (double)L * Lj < (segmented ? 9.0 : 6.5) * fft_cost;
}
cudaError_t split_gemm_prepare();
cudaError_t split_gemm_timeouts(int* count);  // reads and resets the device count

// Per-job parameters of the batched final synthesis reduction.
struct ReduceJobs {
  const void* dw[MAXB];
  const void* dp[MAXB];
  void* out[MAXB];
  int L[MAXB];
  int lend[MAXB];
  int Lphi[MAXB];
  int tmp[MAXB];  // rows m' per block of synthesis partials
  int halves[MAXB];  // 1: blocks are halves of 32-row tiles (direct FP64 contraction)
  int sht[MAXB];  // 1: forward spherical harmonic transform (factor 1/(2 pi), see s2dw_sht_forward)
};

template <typename T>
void launch_contract(int N, int nslot, bool syn, const ContractDesc<T>* descs, const TileTask* tiles,
                     int ntiles, const CallPtrs& ptrs, cudaStream_t st);
// FP32 contraction of large band-limits and its tables (contract_tile.cu)
bool tile_both_halves(int N);  // a CTA computes both tiles of a block pair
// CTA-shape values of s2dw_plan_choices (FP32 plans), see there
constexpr int kPairShapePair = 0, kPairShapeTile = 1, kPairShapeTile2 = 2;
inline bool pair_shapes_offered(int N) { return N <= 5; }
void launch_contract_tile(int N, int nslot, bool syn, const ContractDesc<float>* descs, const CTask* tasks, int ntasks,
                          cudaStream_t st, long long limit = kWaitLimit);
void launch_fpack(const ContractDesc<float>* descs, int njobs, int nbmax, int Lrmax, const CallPtrs& ptrs,
                  cudaStream_t st);
template <typename T>
cudaError_t launch_pair_table(T* out, const double* d64, int Lmax, cudaStream_t st);
template <typename T>
cudaError_t launch_rtable_pair(T* RSp, const double* d64, const double* kap, const double* sabs,
                               const int* slotj, int L, int Lr, int N, int nslot, int kapL, cudaStream_t st);
// Contraction of small and middle band-limits (contract_direct.cuh): one launch
// over the tiles of the plans' wavelet scales (N orders) and of their scaling
// parts.  rt: rows per thread of the analysis (1, 2 or 4).
template <typename T>
struct DirTasks {
  const ContractDesc<T>* descs;
  const CTask* tasks;
  int n;
};
template <typename T>
void launch_contract_direct(int N, bool syn, int rt, const DirTasks<T>& w, const DirTasks<T>& p, const CallPtrs& ptrs,
                            cudaStream_t st);
extern template void launch_contract_direct<float>(int, bool, int, const DirTasks<float>&, const DirTasks<float>&,
                                                   const CallPtrs&, cudaStream_t);
extern template void launch_contract_direct<double>(int, bool, int, const DirTasks<double>&, const DirTasks<double>&,
                                                    const CallPtrs&, cudaStream_t);
// FP32 band-limits up to this run it (both directions of a plan), above the tile
// kernel (contract_tile.cuh), whose CTAs are fewer and longer but read Delta and
// the R rows once for two scales.  Contraction per call, direct against tile,
// analysis / synthesis, us:
//   L      N = 1             N = 3             N = 5              N = 8
//   320    27 / 20, 44 / 34  31 / 37, 55 / 45  36 / 60, 63 / 60   40 / 77, 51 / 48
//   384    42 / 27, 53 / 41  57 / 48, 61 / 52  77 / 83, 73 / 69   67 / 106, 57 / 54
//   448    56 / 39, 59 / 47  76 / 59, 69 / 58  104 / 111, 81 / 77 105 / 138, 63 / 75
//   512    74 / 53, 64 / 55  91 / 75, 73 / 64  132 / 155, 90 / 84 138 / 190, 81 / 100
// and at the small end direct against one CTA per tile pair: L = 32, N = 3 8 / 13,
// 34 / 38; L = 128, N = 5 15 / 17, 62 / 77; L = 256, N = 5 28 / 40, 85 / 106.
constexpr int contract_direct_max_l(int N) { return N <= 2 ? 448 : (N <= 4 ? 384 : (N <= 6 ? 320 : 288)); }
// FP64 (pair table of its own, 152 MB at 384): eighth-domain kernel with its
// scaling launch -> direct, us: L = 32, N = 3 112 / 121 -> 13 / 25; L = 100, N = 3
// 239 / 256 -> 37 / 45; L = 256, N = 1 280 / 351 -> 127 / 125, N = 3 500 / 545 ->
// 195 / 220, N = 8 1212 / 1192 -> 299 / 427; L = 384, N = 5 1048 / 1108 -> 638 /
// 725.  At L = 512 it would still gain (N = 3 1102 / 1195 -> 1044 / 1129, N = 8 2318 /
// 2257 -> 1831 / 1989: 1 and 4% of a call), but its 358 MB of table cost a new plan
// 0.3 ms, more than two calls gain at N = 3.
constexpr int kContractDirectMaxL64 = 384;
cudaError_t contract_direct_prepare_f32();
cudaError_t contract_direct_prepare_f64();
cudaError_t contract_tile_prepare();
cudaError_t pair_timeouts(int* count);  // reads and resets the device count
template <typename T>
void launch_czt(int kind, const CztSeg<T>* segs, int nseg, int total_items, int maxlogM,
                const CallPtrs& ptrs, cudaStream_t st, int uniform_logM);
template <typename T>
void launch_syn_reduce(const ReduceJobs& jobs, int njobs, int Lmax, cudaStream_t st);

template <> void launch_contract<double>(int, int, bool, const ContractDesc<double>*, const TileTask*, int,
                                         const CallPtrs&, cudaStream_t);
template <> void launch_czt<float>(int, const CztSeg<float>*, int, int, int, const CallPtrs&, cudaStream_t, int);
template <> void launch_czt<double>(int, const CztSeg<double>*, int, int, int, const CallPtrs&, cudaStream_t, int);
template <> void launch_syn_reduce<float>(const ReduceJobs&, int, int, cudaStream_t);
template <> void launch_syn_reduce<double>(const ReduceJobs&, int, int, cudaStream_t);
cudaError_t czt_prepare_f32(int maxlogM);
cudaError_t czt_prepare_f64(int maxlogM);
int contract_rows_per_thread(bool fp64);
constexpr int kDeltaPad = 64;     // spare entries after a Delta table (row-segment copies)
constexpr int kDeltaFront = 512;  // zero entries before it: the contraction's unguarded row
                                  // copies start up to 324 entries early (small l)

}  // namespace s2dw
