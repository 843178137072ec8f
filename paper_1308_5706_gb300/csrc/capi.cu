// C ABI: plans, the shared Delta table, launch lists, analysis and synthesis.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/s2dw.h"
#include "internal.h"
#include "plan_kernels.h"
#include "steer.h"

using namespace s2dw;

namespace {

inline int round_up(int x, int a) { return (x + a - 1) / a * a; }
inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

struct CudaFail {
  cudaError_t err;
};
inline void ck(cudaError_t e) {
  if (e != cudaSuccess) throw CudaFail{e};
}

// Segmented chirp-z choice for a band Lj on a grid of band L whose chirp-z
// length is 2^logM: the length M' = 2^logMs (512 <= M' <= min(M/2, 4096)) and
// S = ceil(n / P) segments of P = M' - 2 Lj + 2 samples (n = 2L - 1) that
// minimise the FFT work (S + 1) M' log2 M', used where that is below 0.85 of
// the two FFTs of length M of one convolution (else S = 0).
void seg_choice(int L, int Lj, int logM, int& logMs, int& P, int& S) {
  const int n = 2 * L - 1;
  double best = 0.85 * 2.0 * (double)(1 << logM) * logM;
  logMs = P = S = 0;
  for (int lm = 9; lm <= std::min(logM - 1, 12); ++lm) {
    const int Mp = 1 << lm, p = Mp - 2 * Lj + 2;
    if (p <= 0) continue;
    const int s = (n + p - 1) / p;
    if (s > 64) continue;
    const double c = (double)(s + 1) * Mp * lm;
    if (c < best) {
      best = c;
      logMs = lm;
      P = p;
      S = s;
    }
  }
}

// J_max = ceil(log_lam L) by an integer loop (Sec. 2.2); -1 when it exceeds
// kJmaxCap (lambda so close to 1 that the loop would not end in reasonable
// time; such a plan would exceed the 64-scale limit anyway unless J0 were huge).
constexpr int kJmaxCap = 1 << 20;
int jmax_of(int L, double lam) {
  int J = 0;
  double p = 1.0;
  while (p < L) {
    p *= lam;
    if (++J > kJmaxCap) return -1;
  }
  return J;
}

// Gauss-Legendre nodes/weights on [-1, 1] (Newton iteration on P_Q).
void gauss_legendre(int Q, std::vector<double>& x, std::vector<double>& w) {
  x.assign(Q, 0.0);
  w.assign(Q, 0.0);
  const double pi = 3.14159265358979323846;
  for (int i = 0; i < Q; ++i) {
    double z = std::cos(pi * (i + 0.75) / (Q + 0.5));
    double dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= Q; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = Q * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// Library-wide non-blocking stream for set-up copies and frees, and the
// device's stream-ordered memory pool configured to keep freed memory cached:
// creating and destroying plans then never synchronises the whole device
// (plain cudaFree / cudaMemcpy on the legacy stream would drain every stream
// of a serving process).
std::mutex g_setup_mu;
cudaStream_t g_setup_stream[64] = {};
// Freed blocks that the pool keeps: up to 16 GiB beside what is in use.  The pool's
// threshold counts what is in use as well, so it moves with the live tables and
// workspaces: at a fixed 16 GiB the Delta tables of L = 2048 alone (17.4 GB) were above
// it, and every plan mapped and unmapped its workspace (1 ms per GB each; create
// + destroy, L = 723, N = 6 2.46 -> 1.14 ms, L = 2048, N = 8 12.7 -> 2.75).
constexpr uint64_t kPoolCache = 16ull << 30;
uint64_t g_pool_live[64] = {};  // bytes of live tables and workspaces
void pool_live(int dev, int64_t delta) {
  if (dev < 0 || dev >= 64) return;
  std::lock_guard<std::mutex> lk(g_setup_mu);
  g_pool_live[dev] += (uint64_t)delta;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t thr = kPoolCache + g_pool_live[dev];
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
}

// Kernel attributes (shared-memory limits sized for every plan, L <= 2048)
// are set once per device and precision under a lock, so that creating a plan
// in one host thread never changes an attribute of a kernel that another
// thread is launching.
std::mutex g_prep_mu;
void kernels_prepare(bool fp64, bool pair) {
  int dev = 0;
  ck(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) throw CudaFail{cudaErrorInvalidDevice};
  static unsigned long long done_czt[2] = {0, 0}, done_pair = 0;
  const unsigned long long bit = 1ull << dev;
  std::lock_guard<std::mutex> lk(g_prep_mu);
  if (!(done_czt[fp64 ? 1 : 0] & bit)) {
    ck(fp64 ? czt_prepare_f64(13) : czt_prepare_f32(13));
    if (fp64) ck(contract_direct_prepare_f64());
    done_czt[fp64 ? 1 : 0] |= bit;
  }
  if (pair && !(done_pair & bit)) {
    ck(contract_tile_prepare());
    ck(contract_direct_prepare_f32());
    ck(split_gemm_prepare());
    done_pair |= bit;
  }
}
cudaStream_t setup_stream() {
  int dev = 0;
  ck(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_setup_mu);
  if (dev < 0 || dev >= 64) throw CudaFail{cudaErrorInvalidDevice};
  if (!g_setup_stream[dev]) {
    ck(cudaStreamCreateWithFlags(&g_setup_stream[dev], cudaStreamNonBlocking));
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
      uint64_t thr = kPoolCache + g_pool_live[dev];
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
  }
  return g_setup_stream[dev];
}
template <typename P>
void amalloc(P** p, size_t bytes, cudaStream_t st) {
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(p), bytes, st);
  if (e == cudaErrorMemoryAllocation) {  // once more without the cached blocks
    cudaGetLastError();
    int dev = 0;
    cudaMemPool_t pool;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocAsync(reinterpret_cast<void**>(p), bytes, st);
  }
  ck(e);
}
inline void afree(void* p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
}

// ---------------------------------------------------------------------------
// Process-wide Delta tables, reference counted (one per band-limit reach).
// ---------------------------------------------------------------------------
struct DeltaTab {
  int Lmax;
  int device;
  double* d64;  // entry 0 of the table (kDeltaFront zero entries precede it)
  int refs;
  size_t bytes;
  double* raw64 = nullptr;  // the allocations
  float* pair32 = nullptr;  // pair table of the FP32 contraction (built for the first FP32 plan)
  double* pair64 = nullptr; // that of the direct FP64 contraction, l < min(Lmax, kContractDirectMaxL64)
};
std::mutex g_mu;
std::vector<DeltaTab*> g_tabs;

DeltaTab* delta_acquire(int L, cudaStream_t st) {
  int dev = 0;
  ck(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_mu);
  DeltaTab* best = nullptr;
  for (DeltaTab* t : g_tabs)
    if (t->device == dev && t->Lmax >= L && (!best || t->Lmax < best->Lmax)) best = t;
  if (best) {
    best->refs++;
    return best;
  }
  // Size classes (multiples of 64 up to 256, then of 256) keep the number of
  // distinct tables small when plans of many band-limits come and go.  Slab l
  // does not depend on Lmax, so the slabs of the largest existing table are
  // copied and only the new ones are computed.
  const int Lmax = L <= 256 ? round_up(L, 64) : round_up(L, 256);
  DeltaTab* donor = nullptr;
  for (DeltaTab* u : g_tabs)
    if (u->device == dev && u->Lmax < Lmax && (!donor || u->Lmax > donor->Lmax)) donor = u;
  const int l_first = donor ? donor->Lmax : 0;
  const int64_t entries = delta_table_entries(Lmax) + 64;  // + read-ahead pad
  DeltaTab* t = new DeltaTab{Lmax, dev, nullptr, 1, 0};
  double* em = nullptr;
  int* ee = nullptr;
  try {
    // kDeltaPad spare entries: the contraction copies 16-byte chunks of row
    // segments that may run past the last row of the last slab
    amalloc(&t->raw64, (kDeltaFront + entries + kDeltaPad) * sizeof(double), st);
    ck(cudaMemsetAsync(t->raw64, 0, kDeltaFront * sizeof(double), st));
    t->d64 = t->raw64 + kDeltaFront;
    t->bytes = entries * sizeof(double);
    const int64_t kept = delta_slab_offset(l_first);
    if (donor) ck(cudaMemcpyAsync(t->d64, donor->d64, kept * sizeof(double), cudaMemcpyDeviceToDevice, st));
    ck(cudaMemsetAsync(t->d64 + kept, 0, (entries + kDeltaPad - kept) * sizeof(double), st));
    const size_t ne = (size_t)Lmax * (Lmax + 1) / 2;
    amalloc(&em, ne * sizeof(double), st);
    amalloc(&ee, ne * sizeof(int), st);
    ck(launch_delta_build(t->d64, nullptr, em, ee, Lmax, l_first, st));
    afree(em, st);
    afree(ee, st);
    ck(cudaStreamSynchronize(st));
  } catch (...) {
    cudaStreamSynchronize(st);
    afree(em, st);
    afree(ee, st);
    afree(t->raw64, st);
    delete t;
    throw;
  }
  g_tabs.push_back(t);
  pool_live(dev, (int64_t)t->bytes);
  return t;
}

// The FP32 pair table of a shared table (built from its FP64 slabs on first need).
void delta_pair_ensure(DeltaTab* t, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (t->pair32) return;
  float* pt = nullptr;
  amalloc(&pt, (size_t)pair_table_entries(t->Lmax) * sizeof(float), st);
  cudaError_t e = launch_pair_table<float>(pt, t->d64, t->Lmax, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    afree(pt, st);
    throw CudaFail{e};
  }
  t->pair32 = pt;
  const size_t bytes = (size_t)pair_table_entries(t->Lmax) * sizeof(float);
  t->bytes += bytes;
  pool_live(t->device, (int64_t)bytes);
}

// The FP64 pair table of the direct contraction (small band-limits only).
int pair64_reach(const DeltaTab* t) { return std::min(t->Lmax, kContractDirectMaxL64); }
void delta_pair64_ensure(DeltaTab* t, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (t->pair64) return;
  double* pt = nullptr;
  const size_t bytes = (size_t)pair_table_entries(pair64_reach(t)) * sizeof(double);
  amalloc(&pt, bytes, st);
  cudaError_t e = launch_pair_table<double>(pt, t->d64, pair64_reach(t), st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    afree(pt, st);
    throw CudaFail{e};
  }
  t->pair64 = pt;
  t->bytes += bytes;
  pool_live(t->device, (int64_t)bytes);
}

void delta_release(DeltaTab* t) {
  if (!t) return;
  std::lock_guard<std::mutex> lk(g_mu);
  if (--t->refs == 0) {
    cudaStream_t st = setup_stream();
    afree(t->raw64, st);
    afree(t->pair32, st);
    afree(t->pair64, st);
    pool_live(t->device, -(int64_t)t->bytes);
    g_tabs.erase(std::remove(g_tabs.begin(), g_tabs.end(), t), g_tabs.end());
    delete t;
  }
}

// Device-resident launch lists for a set of jobs (one plan = one job).
struct Lists {
  void* mem = nullptr;
  void* desc_w = nullptr;     // ContractDesc<T>[njobs]
  void* desc_phi = nullptr;   // ContractDesc<T>[njobs]
  // FP64: (N, (tiles, count))
  std::vector<std::pair<int, std::pair<void*, int>>> tiles_w;
  void* tiles_phi = nullptr;
  int ntiles_phi = 0;
  // FP32 contraction, direct and tile kernel: per N the analysis and synthesis
  // tasks of the wavelet scales; *_phi (N = 1): those of the scaling parts (the
  // direct ones are launched with the first direct group)
  struct FpGroup {
    int N = 1, rt = 4;
    void* task[2] = {nullptr, nullptr};  // analysis, synthesis
    int n[2] = {0, 0};
  };
  std::vector<FpGroup> dir_w, tile_w;
  FpGroup dir_phi, tile_phi;
  static constexpr int NK = 21;  // chirp-z 0..3, direct alpha 4..5, single-FFT beta 6..7, segmented alpha 8..9,
                                 // MW-grid synthesis beta 10..12, half-length beta 13..15, split products 16..20
  void* segs[NK] = {};
  int nseg[NK] = {};
  int items[NK] = {};
  int stages[NK] = {};  // data stages of the split products
  int ulogM[NK] = {};  // the segments' common transform length log2 (0: lengths differ)
  // half-length beta kinds (13..15): the segments ordered by transform length,
  // one launch per length {first segment, segments, items, log2 length}, so
  // that each launch runs the kernel compiled for its length
  std::vector<std::array<int, 4>> dct_parts[3];
  int maxlogM = 0;
  int Lmax = 0;
  int odd = 0;  // CZT_ODD_ROWS when a plan of the list samples the MW grid
  int njobs = 0, nbmax = 0, Lrmax = 0;  // f packing of the FP32 contraction (jobs, 32-blocks, rows)
  ~Lists() {
    if (mem) {
      try {
        afree(mem, setup_stream());
      } catch (...) {
      }
    }
  }
};

}  // namespace

struct s2dw_plan_s {
  int L = 0, N = 0, J0 = 0, J = 0, nscale = 0;
  unsigned flags = 0;
  double lam = 0;
  bool fp64 = false;
  int E = 4, TMP = 32;
  std::vector<int> lo, hi, Lj;
  int lend_w = -1, L0 = 0, lphi = 0, Lphi = 1;
  int logM = 0, M = 0;
  int device = 0;
  DeltaTab* tab = nullptr;
  std::vector<double> psi_host, phi_host;
  bool sht = false;                 // companion plan of the spherical harmonic transforms
  s2dw_plan_s* sht_child = nullptr; // created on the first s2dw_sht_* call
  cudaStream_t pst = nullptr;       // private non-blocking stream (set-up, frees)
  cudaEvent_t last_use = nullptr;   // recorded after every call using the plan
  void* ws = nullptr;
  size_t ws_bytes = 0;
  // workspace views
  void* RS = nullptr;
  void* RSphi = nullptr;
  std::vector<void*> Y, X;  // [nscale + 1], last = scaling part
  std::vector<int> Ycols;   // band-limit of each buffer (Lj, last = Lphi)
  void* P = nullptr;
  void* Pphi = nullptr;
  int nbr = 0, nbr_phi = 0, Lp = 0, Lp32 = 0, Lphip = 0, Lphip32 = 0;
  // Tables of one sampling grid (band-limit Lg: 2Lg beta, 2Lg-1 alpha samples).
  struct GridTables {
    int L = 0, logM = 0, M = 0;
    int nb = 0;              // beta samples: 2L (DH), or L (MW grid)
    void* tw = nullptr;
    void* chirp_a = nullptr;
    void* pre_b = nullptr;
    void* post_b = nullptr;
    void* preS_b = nullptr;
    void* postS_b = nullptr;
    void* root_a = nullptr;  // e^{2 pi i t/(2Lg-1)}
    void* pre_mw = nullptr;  // MW beta chirp e^{i pi (m'^2 + m')/(2Lg-1)}, |m'| < Lg
    void* bfft = nullptr;    // e^{i pi m'/(4Lg)} (|m'| < Lg), then q_b (b < 2Lg): single-FFT beta
    void* tw2 = nullptr;     // FFT twiddles of length 2Lg (half-length beta)
    void* Hs = nullptr;      // 4 x M spectra
    // FP32 plans: basis tables of the split products (beta analysis, beta
    // synthesis, alpha analysis, alpha synthesis, MW: beta evaluation on the
    // DH grid), where some launch uses them
    void* sg[5] = {};
    bool sg_beta[2] = {false, false};  // the beta sums of a direction run as products
  };
  bool multires = false;       // every scale on the grid of its own band-limit
  bool mw = false;             // L beta samples per grid (McEwen-Wiaux), not 2L
  std::vector<GridTables> gt;  // one set per distinct grid band-limit
  std::vector<int> grid_of;    // [nscale + 1]: set of scale j (last: scaling part)
  std::vector<int64_t> woff;   // [nscale + 1]: element offset of scale j in W (last: total)
  // segmented chirp-z of scale j (S == 0: one convolution of the grid's length M)
  struct SegTables {
    int logM = 0, P = 0, S = 0;
    void* tw = nullptr;  // twiddles of length 2^logM
    void* Ha = nullptr;  // S analysis spectra of length 2^logM
    void* Hs = nullptr;  // S synthesis spectra
  };
  std::vector<SegTables> seg;  // [nscale + 1]
  // launch methods (s2dw_plan_choices / s2dw_plan_tune): beta_mode[dir] 0 = one
  // FFT of length 4L, 1 = half-length transforms on the grids where they are
  // faster (power-of-two L >= 128; synthesis up to 1024);
  // alpha_mode[dir][j] 0 = direct sums (L_j <= 32), 1 = chirp-z of the grid's
  // length, 2 = segmented chirp-z (where its tables exist), 3 = split products
  // (where alpha_sg: FP32 plans, the scales on which they are faster; their
  // default); dir 0 = analysis
  int beta_mode[2] = {1, 1};
  std::vector<int> alpha_mode[2];
  std::vector<char> alpha_sg[2];
  void* sg_data = nullptr;  // operand images of the product launch under way
  // [nscale + 1]: tensor-core basis images of the direct alpha sums (FP32 plans)
  std::vector<void*> tc_ana, tc_syn;
  // FP32 plans: R rows and packed f of the FP32 contraction
  void* RSp = nullptr;
  void* RSphi_p = nullptr;
  void* fP = nullptr;
  int Lr = 0, Lrphi = 0, Lrf = 0;
  // host copies of the static descriptors (device copies live in `own`)
  std::vector<unsigned char> desc_w_host, desc_phi_host;
  std::vector<TileTask> tiles_w_host, tiles_phi_host;  // FP64 plans
  bool direct_w = false, direct_phi = false;  // the direct contraction (else FP32: the tile kernel, FP64: k_contract)
  int pair_shape = kPairShapePair;  // FP32: last value of s2dw_plan_choices (selects nothing)
  Lists own;
  // stage timing (s2dw_profile): one set of events per call, up to kProfCalls
  static constexpr int kProfCalls = 256;
  bool prof = false;
  static constexpr int kEvAna = 7, kEvSyn = 8;  // events per call (stages + 1)
  std::vector<cudaEvent_t> ev_ana, ev_syn;      // kProfCalls x kEvAna, kProfCalls x kEvSyn
  int nana = 0, nsyn = 0;
  ~s2dw_plan_s() {
    for (auto e : ev_ana)
      if (e) cudaEventDestroy(e);
    for (auto e : ev_syn)
      if (e) cudaEventDestroy(e);
    delete sht_child;
    if (last_use) {
      cudaEventSynchronize(last_use);  // only this plan's work, not the device
      cudaEventDestroy(last_use);
    }
    if (ws) {
      cudaFreeAsync(ws, pst);
      pool_live(device, -(int64_t)ws_bytes);
    }
    own.mem = nullptr;
    if (own_mem) cudaFreeAsync(own_mem, pst);
    if (pst) cudaStreamDestroy(pst);  // releases after the queued frees
    delta_release(tab);
  }
  void* own_mem = nullptr;
};

namespace {

// Launch lists of the plan sets seen by the batched entry points.  At most
// kBatchCacheMax entries: beyond that the least recently used one is freed
// once its last launch has completed, unless it was used while its stream was
// being captured into a CUDA graph (the graph keeps reading it, so it lives
// until one of its plans is destroyed).
struct BatchEnt {
  Lists* ls = nullptr;
  uint64_t tick = 0;
  cudaEvent_t done = nullptr;  // recorded after the entry's latest launches
  bool pinned = false;
};
constexpr size_t kBatchCacheMax = 64;
std::mutex g_batch_mu;
std::map<std::vector<s2dw_plan_t>, BatchEnt> g_batch_cache;
uint64_t g_batch_tick = 0;

void free_batch_ent(BatchEnt& e) {
  if (e.done) {
    cudaEventSynchronize(e.done);  // only this entry's launches
    cudaEventDestroy(e.done);
  }
  delete e.ls;
}

void drop_batches_with(s2dw_plan_t p) {
  std::lock_guard<std::mutex> lk(g_batch_mu);
  for (auto it = g_batch_cache.begin(); it != g_batch_cache.end();) {
    if (std::find(it->first.begin(), it->first.end(), p) != it->first.end()) {
      free_batch_ent(it->second);
      it = g_batch_cache.erase(it);
    } else {
      ++it;
    }
  }
}

void evict_batches() {  // g_batch_mu held; called before an insertion
  while (g_batch_cache.size() >= kBatchCacheMax) {  // room for one more
    auto victim = g_batch_cache.end();
    for (auto it = g_batch_cache.begin(); it != g_batch_cache.end(); ++it)
      if (!it->second.pinned && (victim == g_batch_cache.end() || it->second.tick < victim->second.tick))
        victim = it;
    if (victim == g_batch_cache.end()) return;
    free_batch_ent(victim->second);
    g_batch_cache.erase(victim);
  }
}

// Gamma factors [k N + g], n_k = -(N-1) + 2k, gamma_g = pi g / N, eta = 1 (N
// odd) or i: analysis conj(eta) i^{n_k} e^{i n_k gamma_g} (Eq. (28)), synthesis
// eta (2 pi/N) i^{-n_k} e^{-i n_k gamma_g} (Eq. (39)).
template <typename T>
void gamma_factors(int N, cx<T>* ana, cx<T>* syn) {
  const double pi = 3.14159265358979323846;
  for (int k = 0; k < N; ++k)
    for (int g = 0; g < N; ++g) {
      const int n = -(N - 1) + 2 * k;
      // n g pi / N + n pi/2 - (N even) pi/2 in units of pi/(2N), reduced exactly
      const int u = (((2 * n * g + n * N - (N % 2 == 0 ? N : 0)) % (4 * N)) + 4 * N) % (4 * N);
      const double c = std::cos(pi * u / (2 * N)), s = std::sin(pi * u / (2 * N)), sc = 2.0 * pi / N;
      ana[k * N + g] = mkc<T>((T)c, (T)s);
      syn[k * N + g] = mkc<T>((T)(c * sc), (T)(-s * sc));
    }
}

template <typename T>
void fill_desc(s2dw_plan_s* p, ContractDesc<T>& dw, ContractDesc<T>& dp, const T* delta) {
  std::memset(&dw, 0, sizeof(dw));
  std::memset(&dp, 0, sizeof(dp));
  dw.delta = delta;
  const T* pairs = sizeof(T) == 4 ? reinterpret_cast<const T*>(p->tab->pair32) : reinterpret_cast<const T*>(p->tab->pair64);
  dw.dpair = pairs;
  dw.RSp = reinterpret_cast<const T*>(p->RSp);
  dw.fP = reinterpret_cast<const cx<T>*>(p->fP);
  dw.Lr = p->Lr;
  dw.Lrf = p->Lrf;
  dw.RS = reinterpret_cast<const T*>(p->RS);
  dw.P = reinterpret_cast<cx<T>*>(p->P);
  dw.L = p->L;
  dw.Lp = p->Lp;
  dw.Lp32 = p->Lp32;
  dw.nbr = p->nbr;
  dw.N = p->N;
  dw.nslot = 2;
  dw.eta_odd = (p->N % 2 == 0) ? 1 : 0;
  gamma_factors<T>(p->N, dw.cga, dw.cgs);
  gamma_factors<T>(1, dp.cga, dp.cgs);
  for (int j = 0; j < MAXS; ++j) {
    dw.jlo[j] = dp.jlo[j] = 0;
    dw.jhi[j] = dp.jhi[j] = -1;
  }
  dp.jhi[0] = p->Lphi - 1;
  for (int j = 0; j < p->nscale; ++j) {
    if (p->hi[j] >= 0) {
      dw.jlo[j] = p->lo[j];
      dw.jhi[j] = p->hi[j];
    }
    dw.Lj[j] = p->Lj[j];
    dw.Y[j] = reinterpret_cast<cx<T>*>(p->Y[j]);
  }
  // l-segments with constant slot occupancy, covering [0, L-1]
  int ns = 0;
  int prev0 = -2, prev1 = -2;
  for (int l = 0; l < p->L; ++l) {
    int s0 = -1, s1 = -1;
    for (int j = 0; j < p->nscale; ++j) {
      if (p->Lj[j] == 0 || l < p->lo[j] || l > p->hi[j]) continue;
      if (j % 2 == 0) s0 = j;
      else s1 = j;
    }
    if (s0 != prev0 || s1 != prev1) {
      dw.seg[ns].lo = l;
      dw.seg[ns].hi = l;
      dw.seg[ns].j[0] = s0;
      dw.seg[ns].j[1] = s1;
      ++ns;
      prev0 = s0;
      prev1 = s1;
    } else {
      dw.seg[ns - 1].hi = l;
    }
  }
  dw.nseg = ns;
  // scaling part: one N = 1 "scale" with kernel Phi on [0, lphi]
  dp.delta = delta;
  dp.dpair = pairs;
  dp.RSp = reinterpret_cast<const T*>(p->RSphi_p);
  dp.fP = reinterpret_cast<const cx<T>*>(p->fP);
  dp.Lr = p->Lrphi;
  dp.Lrf = p->Lrf;
  dp.RS = reinterpret_cast<const T*>(p->RSphi);
  dp.P = reinterpret_cast<cx<T>*>(p->Pphi);
  dp.L = p->Lphi;
  dp.Lp = p->Lphip;
  dp.Lp32 = p->Lphip32;
  dp.nbr = p->nbr_phi;
  dp.N = 1;
  dp.nslot = 1;
  dp.eta_odd = 0;
  dp.Lj[0] = p->Lphi;
  dp.Y[0] = reinterpret_cast<cx<T>*>(p->Y[p->nscale]);
  dp.seg[0].lo = 0;
  dp.seg[0].hi = p->Lphi - 1;
  dp.seg[0].j[0] = 0;
  dp.seg[0].j[1] = -1;
  dp.nseg = 1;
}

void build_tiles(int Lband, int lend, int TMP, int prob, std::vector<TileTask>& out) {
  if (Lband <= 0 || lend < 0) return;
  const int nbp = (Lband + TMP - 1) / TMP, nbm = (Lband + TILE - 1) / TILE;
  for (int bp = 0; bp < nbp; ++bp)
    for (int bm = 0; bm < nbm; ++bm) {
      const int ls = std::max(bp * TMP, bm * TILE);
      if (ls > lend) continue;
      out.push_back(TileTask{prob, bp, bm, ls, lend});
    }
}

CTask make_task(int prob, int p, int q, int half, int lstart, int lend, int j, int j2, int slot, int table_Lmax) {
  CTask t;
  std::memset(&t, 0, sizeof(t));
  t.prob = (uint8_t)prob, t.p = (uint8_t)p, t.q = (uint8_t)q, t.half = (uint8_t)half;
  t.j = (int8_t)j, t.j2 = (int8_t)j2, t.slot = (int8_t)slot;
  t.lstart = (int16_t)lstart, t.lend = (int16_t)lend, t.Lmax = (int16_t)table_Lmax;
  return t;
}

// Tasks of the contraction of large band-limits (contract_tile.cuh): per block
// pair (and tile, where a CTA computes one), the analysis by pairs of adjacent
// scales 2i, 2i + 1 (one per slot) over the union of their l ranges, the
// synthesis by l ranges on which each slot holds one scale (an l-segment
// where a slot is empty joins its neighbour).
template <typename T>
void build_tile_tasks(const ContractDesc<T>& d, int prob, int Lband, int lend, int table_Lmax,
                      std::vector<CTask>& ana, std::vector<CTask>& syn) {
  if (Lband <= 0 || lend < 0) return;
  struct Range { int lo, hi, j, j2; };
  std::vector<Range> ra, rs;
  for (int j = 0; j < MAXS; j += d.nslot) {
    const int j2 = d.nslot == 2 ? j + 1 : -1;
    const bool a = d.jhi[j] >= d.jlo[j], b = j2 >= 0 && j2 < MAXS && d.jhi[j2] >= d.jlo[j2];
    if (!a && !b) continue;
    ra.push_back({a && b ? std::min(d.jlo[j], d.jlo[j2]) : (a ? d.jlo[j] : d.jlo[j2]),
                  a && b ? std::max(d.jhi[j], d.jhi[j2]) : (a ? d.jhi[j] : d.jhi[j2]), a ? j : -1, b ? j2 : -1});
  }
  for (int i = 0; i < d.nseg; ++i) {
    const LSeg& g = d.seg[i];
    const int n2 = d.nslot == 2 ? g.j[1] : -1;
    auto fits = [](int cur, int next) { return cur == next || cur < 0 || next < 0; };
    if (!rs.empty() && fits(rs.back().j, g.j[0]) && fits(rs.back().j2, n2)) {
      rs.back().hi = g.hi;
      rs.back().j = std::max(rs.back().j, g.j[0]);
      rs.back().j2 = std::max(rs.back().j2, n2);
    } else {
      rs.push_back({g.lo, g.hi, g.j[0], n2});
    }
  }
  const int nb = (Lband + 31) / 32;
  const bool both = tile_both_halves(d.N);
  for (int q = 0; q < nb; ++q)
    for (int p = 0; p <= q; ++p) {
      for (int half = 0; half <= (both || p == q ? 0 : 1); ++half)
        for (int dir = 0; dir < 2; ++dir)
          for (const Range& r : dir ? rs : ra) {
            const int a = std::max(r.lo, 32 * q), b = std::min(r.hi, lend);
            if (a <= b) (dir ? syn : ana).push_back(make_task(prob, p, q, half, a, b, r.j, r.j2, 0, table_Lmax));
          }
    }
}

// longest first (a counting sort on the length of the l range)
void sort_tasks(std::vector<CTask>& v) {
  int maxlen = 0;
  for (const CTask& t : v) maxlen = std::max(maxlen, t.lend - t.lstart);
  std::vector<size_t> at(maxlen + 2, 0);
  for (const CTask& t : v) ++at[maxlen - (t.lend - t.lstart) + 1];
  for (int i = 0; i <= maxlen; ++i) at[i + 1] += at[i];
  std::vector<CTask> sorted(v.size());
  for (const CTask& t : v) sorted[at[maxlen - (t.lend - t.lstart)]++] = t;
  v.swap(sorted);
}

// Direct contraction tasks of one plan's wavelet scales or scaling part (d:
// its descriptor, band Lband, last l lend): every tile, for the analysis once
// per scale over the scale's l (its [lo, hi] from the l-segments), for the
// synthesis once per l-segment.
template <typename T>
void build_direct_tasks(const ContractDesc<T>& d, int prob, int Lband, int lend, int table_Lmax,
                        std::vector<CTask>& ana, std::vector<CTask>& syn) {
  if (Lband <= 0 || lend < 0) return;
  const int nb = (Lband + 31) / 32;
  for (int q = 0; q < nb; ++q)
    for (int p = 0; p <= q; ++p) {
      for (int half = 0; half <= (p == q ? 0 : 1); ++half) {
        auto add = [&](std::vector<CTask>& v, int a, int b, int j, int j2, int slot) {
          a = std::max(a, 32 * q);
          b = std::min(b, lend);
          if (a <= b) v.push_back(make_task(prob, p, q, half, a, b, j, j2, slot, table_Lmax));
        };
        for (int j = 0; j < MAXS; ++j)
          if (d.jhi[j] >= d.jlo[j]) add(ana, d.jlo[j], d.jhi[j], j, -1, j % 2);
        for (int i = 0; i < d.nseg; ++i) add(syn, d.seg[i].lo, d.seg[i].hi, d.seg[i].j[0], d.seg[i].j[1], 0);
      }
    }
}

// Analysis rows per thread and synthesis l ranges of a direct launch, from the
// number of tasks over all its plans (neither enters the arithmetic).
// Analysis: rt rows per thread, so 32 / (8 rt) CTAs of 8 warps per task (8 CTAs
// of 4 warps at rt = 1): fewer rows per thread while the tasks alone would
// leave SMs idle (a thread's R loads serve its rt rows).  Synthesis: pieces of
// a multiple of 16 l, about four CTAs per SM over the launch.  FP64 (rt is not
// used): pieces of a multiple of 4 l, two CTAs each; with N > 2 two CTAs per SM,
// because each repeats the gamma step of its rows (four / one piece per SM, us:
// L = 256, N = 1 125 / 152, N = 3 256 / 220, N = 8 682 / 427).
int direct_split(std::vector<CTask>& ana, std::vector<CTask>& syn, int sms, bool fp64, int N) {
  const long long n = (long long)ana.size();
  long long total = 0;
  for (const CTask& t : syn) total += t.lend - t.lstart + 1;
  const long long want = (fp64 && N > 2 ? 1LL : 4LL) * sms;
  const int ls = round_up((int)std::min<long long>(std::max<long long>((total + want - 1) / want, 1), 4096), fp64 ? 4 : 16);
  std::vector<CTask> cut;
  for (const CTask& t : syn)
    for (int l = t.lstart; l <= t.lend; l += ls) {
      CTask u = t;
      u.lstart = (int16_t)l;
      u.lend = (int16_t)std::min((int)t.lend, l + ls - 1);
      cut.push_back(u);
    }
  syn.swap(cut);
  sort_tasks(ana);
  sort_tasks(syn);
  return n >= 2 * sms ? 4 : (n >= sms / 2 ? 2 : 1);
}

void sort_tiles(std::vector<TileTask>& t) {
  std::stable_sort(t.begin(), t.end(), [](const TileTask& a, const TileTask& b) {
    return (a.lend - a.lstart) > (b.lend - b.lstart);
  });
}

template <typename T>
void build_segs(s2dw_plan_s* p, int job, int njobs, int kind, std::vector<CztSeg<T>>& out, int& start, int& stages) {
  // kinds 4 / 5 collect the alpha segments of scales with Lj <= kDirectMaxLjAna
  // (analysis) or kDirectMaxLj (synthesis),
  // kinds 6 / 7 the beta segments of plans whose FFT length M is 4L
  // kinds 8 / 9 the alpha segments of scales with a segmented chirp-z;
  // kinds 10..12 (MW grid only) the synthesis-side resampling of V from the L
  // MW beta samples to the DH beta grid (torus coefficients, then their
  // evaluation on the DH grid by the analysis beta kernels)
  if ((kind == CZT_BETA_MW_DFT || kind == CZT_BETA_RS_FFT || kind == CZT_BETA_RS || kind == CZT_BETA_RS_DCT ||
       kind == SG_KIND_BETA_RS) &&
      !p->mw)
    return;
  const int base_kind = (kind == CZT_ALPHA_ANA_DIRECT || kind == CZT_ALPHA_ANA_SEG || kind == SG_KIND_ALPHA_ANA)
                            ? CZT_ALPHA_ANA
                        : (kind == CZT_ALPHA_SYN_DIRECT || kind == CZT_ALPHA_SYN_SEG || kind == SG_KIND_ALPHA_SYN)
                            ? CZT_ALPHA_SYN
                        : (kind == SG_KIND_BETA_ANA || kind == SG_KIND_BETA_RS) ? CZT_BETA_ANA
                        : kind == SG_KIND_BETA_SYN                              ? CZT_BETA_SYN
                        : (kind == CZT_BETA_ANA_FFT || kind == CZT_BETA_RS_FFT || kind == CZT_BETA_RS ||
                           kind == CZT_BETA_MW_DFT || kind == CZT_BETA_ANA_DCT || kind == CZT_BETA_RS_DCT)
                            ? CZT_BETA_ANA
                        : (kind == CZT_BETA_SYN_FFT || kind == CZT_BETA_SYN_DCT) ? CZT_BETA_SYN
                                                                                  : kind;
  const bool sg_list = kind >= SG_KIND_BETA_ANA && kind <= SG_KIND_BETA_RS;
  if (sg_list && sizeof(T) != sizeof(float)) return;
  const bool rs_list =
      kind == CZT_BETA_RS_FFT || kind == CZT_BETA_RS || kind == CZT_BETA_RS_DCT || kind == SG_KIND_BETA_RS;
  const bool dct_list = kind == CZT_BETA_ANA_DCT || kind == CZT_BETA_SYN_DCT || kind == CZT_BETA_RS_DCT;
  const bool direct_list = kind == CZT_ALPHA_ANA_DIRECT || kind == CZT_ALPHA_SYN_DIRECT;
  const bool seg_list = kind == CZT_ALPHA_ANA_SEG || kind == CZT_ALPHA_SYN_SEG;
  size_t sg_used = 0;  // data stages of this plan so far
  const bool fft_list = kind == CZT_BETA_ANA_FFT || kind == CZT_BETA_SYN_FFT || kind == CZT_BETA_RS_FFT;
  for (int j = 0; j <= p->nscale; ++j) {
    const bool phi = (j == p->nscale);
    const int Nj = phi ? 1 : p->N;
    const int Lj = p->Ycols[j];
    const s2dw_plan_s::GridTables& G = p->gt[p->grid_of[j]];
    const int L = G.L, n = 2 * L - 1;  // this scale's sampling grid
    // the analysis beta step of an MW plan evaluates at the MW samples (chirp-z only);
    // the DH-grid beta kernels (FFT for power-of-two L) serve DH plans and the MW resampling
    const bool mw_ana_beta = p->mw && base_kind == CZT_BETA_ANA && !rs_list && kind != CZT_BETA_MW_DFT;
    // power-of-two L: half-length transforms (L >= 16) or one FFT of length 4L (L = 8); else chirp-z
    const bool beta_pow2 = (4 * L == G.M) && !mw_ana_beta;
    const int bdir = base_kind == CZT_BETA_SYN ? 1 : 0;
    // mode 1: the half-length transforms on the grids where they measured
    // faster than the length-4L FFT (GB300, N = 3): L >= 128 in the analysis,
    // 128 <= L <= 1024 in the synthesis
    const bool dct_faster = bdir == 0 ? L >= 128 : (L >= 128 && L <= 1024);
    const bool beta_dct = beta_pow2 && L >= 16 && p->beta_mode[bdir] == 1 && dct_faster;
    const bool beta_fft = beta_pow2 && !beta_dct;
    const bool is_beta = base_kind == CZT_BETA_ANA || base_kind == CZT_BETA_SYN;
    if (is_beta && kind != CZT_BETA_MW_DFT) {
      // split products on the grids where they are faster, in mode 1 (the default)
      const bool sg = p->beta_mode[bdir] == 1 && (rs_list ? G.sg[4] != nullptr : G.sg_beta[bdir]);
      if (sg != sg_list) continue;
      if (!sg && (beta_fft != fft_list || beta_dct != dct_list)) continue;
    }
    const cx<T>* Hs = reinterpret_cast<const cx<T>*>(G.Hs);
    CztSeg<T> s;
    std::memset(&s, 0, sizeof(s));
    s.job = job;
    s.L = L;
    s.Lj = Lj;
    s.N = Nj;
    s.logM = G.logM;
    s.woff = phi ? 0 : p->woff[j];
    s.is_phi = phi ? 1 : 0;
    s.tw = reinterpret_cast<const cx<T>*>(G.tw);
    s.scale = (T)(2.0 * 3.14159265358979323846 / n);
    s.nb = G.nb;
    const bool is_alpha = base_kind == CZT_ALPHA_ANA || base_kind == CZT_ALPHA_SYN;
    const int amode = is_alpha ? p->alpha_mode[base_kind == CZT_ALPHA_SYN ? 1 : 0][j] : -1;
    const bool direct = is_alpha && amode == 0;
    if (direct != direct_list) continue;
    if (is_alpha && !direct && ((amode == 3) != sg_list || (amode == 2) != seg_list)) continue;
    switch (base_kind) {
      case CZT_BETA_ANA:
        s.P = beta_czt_cols(G.logM, sizeof(T) == 8);  // columns per CTA of the chirp-z beta kernels
        s.items = Nj * ((Lj + s.P - 1) / s.P);
        s.buf_in = reinterpret_cast<cx<T>*>(p->Y[j]);
        s.buf_out = reinterpret_cast<cx<T>*>(p->X[j]);
        s.H = Hs + 0 * (size_t)G.M;
        s.pre = reinterpret_cast<const cx<T>*>(G.pre_b);
        s.post = reinterpret_cast<const cx<T>*>(G.post_b);
        if (kind == CZT_BETA_MW_DFT) {  // V [g][b < L][m] -> torus coefficients [g][m][p]
          s.buf_in = reinterpret_cast<cx<T>*>(p->X[j]);
          s.buf_out = reinterpret_cast<cx<T>*>(p->Y[j]);
          s.H = Hs + 2 * (size_t)G.M;   // the alpha synthesis kernel e^{+i pi u^2/n}
          s.pre = reinterpret_cast<const cx<T>*>(G.chirp_a);
          s.post = reinterpret_cast<const cx<T>*>(G.pre_mw);
        } else if (rs_list) {           // coefficients -> the 2L DH samples
          s.nb = 2 * L;
        } else if (p->mw) {             // analysis: the L MW samples beta_b = (2b+1) pi / n
          s.H = Hs + 1 * (size_t)G.M;   // the alpha analysis kernel e^{-i pi u^2/n}
          s.pre = reinterpret_cast<const cx<T>*>(G.pre_mw);
          s.post = reinterpret_cast<const cx<T>*>(G.chirp_a);
        }
        break;
      case CZT_ALPHA_ANA:
        s.items = ((Nj * G.nb + 1) / 2 + alpha_czt_nt(sizeof(T) == 8) - 1) / alpha_czt_nt(sizeof(T) == 8);
        s.buf_in = reinterpret_cast<cx<T>*>(p->X[j]);
        s.H = Hs + 1 * (size_t)G.M;
        s.pre = reinterpret_cast<const cx<T>*>(G.chirp_a);
        s.post = reinterpret_cast<const cx<T>*>(G.chirp_a);
        break;
      case CZT_ALPHA_SYN:
        s.items = ((Nj * G.nb + 1) / 2 + alpha_czt_nt(sizeof(T) == 8) - 1) / alpha_czt_nt(sizeof(T) == 8);
        s.buf_out = reinterpret_cast<cx<T>*>(p->X[j]);
        s.H = Hs + 2 * (size_t)G.M;
        s.pre = reinterpret_cast<const cx<T>*>(G.chirp_a);
        s.post = reinterpret_cast<const cx<T>*>(G.chirp_a);
        break;
      case CZT_BETA_SYN:
        s.P = beta_czt_cols(G.logM, sizeof(T) == 8);  // columns per CTA of the chirp-z beta kernels
        s.items = Nj * ((Lj + s.P - 1) / s.P);
        s.nb = 2 * L;  // DH quadrature (an MW plan resamples V to the DH grid first)
        s.buf_in = reinterpret_cast<cx<T>*>(p->X[j]);
        s.buf_out = reinterpret_cast<cx<T>*>(p->Y[j]);
        s.H = Hs + 3 * (size_t)G.M;
        s.pre = reinterpret_cast<const cx<T>*>(G.preS_b);
        s.post = reinterpret_cast<const cx<T>*>(G.postS_b);
        break;
    }
    if (fft_list) {
      const int ntb = beta_fft_nt(sizeof(T) == 8);
      s.items = Nj * ((Lj + ntb - 1) / ntb);
      s.pre = reinterpret_cast<const cx<T>*>(G.bfft);
      s.post = reinterpret_cast<const cx<T>*>(G.bfft) + (2 * L - 1);
    }
    if (dct_list) {
      const int cols = 4096 / (2 * L);  // transforms of length 2L per CTA
      s.items = Nj * ((Lj + cols - 1) / cols);
      s.tw = reinterpret_cast<const cx<T>*>(G.tw2);
      s.pre = reinterpret_cast<const cx<T>*>(G.bfft);
      s.post = reinterpret_cast<const cx<T>*>(G.bfft) + (2 * L - 1);
    }
    if (seg_list) {
      const auto& sgt = p->seg[j];
      const int groups = 1 << (12 - sgt.logM);  // row pairs per CTA (one per group of M'/16 threads)
      s.items = ((Nj * G.nb + 1) / 2 + groups - 1) / groups;
      s.logM = sgt.logM;
      s.tw = reinterpret_cast<const cx<T>*>(sgt.tw);
      s.H = reinterpret_cast<const cx<T>*>(base_kind == CZT_ALPHA_ANA ? sgt.Ha : sgt.Hs);
      s.P = sgt.P;
      s.nsegs = sgt.S;
    }
    if (direct) {
      const bool syn = base_kind == CZT_ALPHA_SYN;
      if (sizeof(T) == sizeof(float)) {  // tensor cores: the plan's basis image of this scale
        s.items = alpha_tc_items(L, Nj * G.nb, njobs, syn, s.P);
        s.H = reinterpret_cast<const cx<T>*>(syn ? p->tc_syn[j] : p->tc_ana[j]);
      } else if (!syn) {
        const int tiles = (L + kAgCols - 1) / kAgCols, rows = Nj * G.nb;
        s.P = 512;  // rows per CTA: fewer while a scale has less than a CTA per SM
        while (s.P > kAgMinRows && tiles * ((rows + s.P - 1) / s.P) < 152) s.P /= 2;
        s.items = tiles * ((rows + s.P - 1) / s.P);
      } else {
        s.items = (Nj * G.nb + direct_rows_syn(sizeof(T) == 8) - 1) / direct_rows_syn(sizeof(T) == 8);
      }
      s.pre = reinterpret_cast<const cx<T>*>(G.root_a);
    }
    if constexpr (sizeof(T) == sizeof(float)) {
      if (sg_list) {
        const int k = kind - SG_KIND_BETA_ANA, mode = k == 4 ? 0 : k;
        const SgDims d = sg_dims(mode, L, Lj, Nj, s.nb);
        const SgTable t = sg_table(mode, L);
        s.items = d.data_tiles * d.basis_tiles;
        s.P = d.basis_tiles;
        s.nsegs = d.stages;
        s.tabP = t.tiles;
        s.tabK = t.stages;
        s.H = reinterpret_cast<const cx<T>*>(G.sg[k]);
        s.scale = sg_out_scale(mode, L);
        s.tabD = stages;
        // this plan's images of the launch: one buffer, its segments in turn
        s.pre = reinterpret_cast<const cx<T>*>(reinterpret_cast<const char*>(p->sg_data) + sg_used * kSgDataBytes);
        stages += d.data_tiles * d.stages;
        sg_used += (size_t)d.data_tiles * d.stages;
      }
    }
    if (s.items <= 0) continue;
    s.start = start;
    start += s.items;
    out.push_back(s);
  }
}

// Build the device launch lists for a set of plans (same precision).
template <typename T>
Lists* build_lists(const std::vector<s2dw_plan_t>& plans) {
  // FP64 plans: eighth-domain tiles; FP32 plans: the tile kernel or, for small
  // and middle band-limits, the direct one, each with its own tasks
  using Task = TileTask;
  const int nj = (int)plans.size();
  std::vector<ContractDesc<T>> dw(nj), dp(nj);
  std::map<int, std::vector<Task>> tw_byN;
  std::vector<Task> tphi;
  struct FpTasks {  // direct and tile contractions: analysis and synthesis tasks
    std::vector<CTask> task[2];
    int rt = 4;
    size_t off[2] = {0, 0};
  };
  std::map<int, FpTasks> dir_byN, tile_byN;
  FpTasks dir_phi, tile_phi;
  std::vector<CztSeg<T>> segs[Lists::NK];
  int start[Lists::NK] = {}, stages[Lists::NK] = {};
  Lists* ls = new Lists();
  ls->njobs = nj;
  for (int i = 0; i < nj; ++i) {
    s2dw_plan_s* p = plans[i];
    std::memcpy(&dw[i], p->desc_w_host.data(), sizeof(ContractDesc<T>));
    std::memcpy(&dp[i], p->desc_phi_host.data(), sizeof(ContractDesc<T>));
    const int reach = sizeof(T) == sizeof(float) ? p->tab->Lmax : pair64_reach(p->tab);
    auto add = [&](FpTasks& w, const ContractDesc<T>& d, bool direct, int Lband, int lend) {
      if (direct) build_direct_tasks<T>(d, i, Lband, lend, reach, w.task[0], w.task[1]);
      else build_tile_tasks<T>(d, i, Lband, lend, reach, w.task[0], w.task[1]);
    };
    if (sizeof(T) == sizeof(float) || p->direct_w)
      add((p->direct_w ? dir_byN : tile_byN)[p->N], dw[i], p->direct_w, p->L0, p->lend_w);
    if (sizeof(T) == sizeof(float) || p->direct_phi)
      add(p->direct_phi ? dir_phi : tile_phi, dp[i], p->direct_phi, p->Lphi, p->lphi);
    for (Task t : p->tiles_w_host) {  // (FP64 plans)
      t.prob = i;
      tw_byN[p->N].push_back(t);
    }
    for (Task t : p->tiles_phi_host) {
      t.prob = i;
      tphi.push_back(t);
    }
    for (int k = 0; k < Lists::NK; ++k) build_segs<T>(p, i, (int)plans.size(), k, segs[k], start[k], stages[k]);
    ls->maxlogM = std::max(ls->maxlogM, p->logM);
    ls->Lmax = std::max(ls->Lmax, p->L);
    if (p->fP) {  // packed f: plans that run the tile contraction
      ls->nbmax = std::max(ls->nbmax, (p->L + 31) / 32);
      ls->Lrmax = std::max(ls->Lrmax, p->Lrf);
    }
    if (p->mw) ls->odd = CZT_ODD_ROWS;
  }
  for (int k = CZT_BETA_ANA_DCT; k <= CZT_BETA_RS_DCT; ++k) {
    std::stable_sort(segs[k].begin(), segs[k].end(),
                     [](const CztSeg<T>& a, const CztSeg<T>& b) { return a.logM < b.logM; });
    auto& parts = ls->dct_parts[k - CZT_BETA_ANA_DCT];
    int first = 0, st = 0;
    for (int i = 0; i <= (int)segs[k].size(); ++i) {
      if (i == (int)segs[k].size() || (i > first && segs[k][i].logM != segs[k][first].logM)) {
        if (i > first) parts.push_back({first, i - first, st, segs[k][first].logM});
        if (i == (int)segs[k].size()) break;
        first = i;
        st = 0;
      }
      segs[k][i].start = st;  // CTA indices restart in every part
      st += segs[k][i].items;
    }
  }
  for (int k = 0; k < Lists::NK; ++k) {
    int u = segs[k].empty() ? 0 : segs[k][0].logM;
    for (const CztSeg<T>& sg : segs[k])
      if (sg.logM != u) u = 0;
    ls->ulogM[k] = u;
  }
  for (auto& kv : tw_byN) sort_tiles(kv.second);
  sort_tiles(tphi);
  int sms = 152;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  }
  std::vector<FpTasks*> fp;
  for (auto& kv : dir_byN) {
    fp.push_back(&kv.second);
    kv.second.rt = direct_split(kv.second.task[0], kv.second.task[1], sms, sizeof(T) == 8, kv.first);
  }
  fp.push_back(&dir_phi);
  dir_phi.rt = direct_split(dir_phi.task[0], dir_phi.task[1], sms, sizeof(T) == 8, 1);
  const size_t ndir = fp.size();
  for (auto& kv : tile_byN) fp.push_back(&kv.second);
  fp.push_back(&tile_phi);
  for (size_t i = ndir; i < fp.size(); ++i) {
    sort_tasks(fp[i]->task[0]);
    sort_tasks(fp[i]->task[1]);
  }
  // one allocation for everything
  size_t off = 0;
  const size_t o_dw = off;
  off = align256(off + nj * sizeof(ContractDesc<T>));
  const size_t o_dp = off;
  off = align256(off + nj * sizeof(ContractDesc<T>));
  std::vector<size_t> o_tw;
  for (auto& kv : tw_byN) {
    o_tw.push_back(off);
    off = align256(off + kv.second.size() * sizeof(Task));
  }
  const size_t o_tp = off;
  off = align256(off + tphi.size() * sizeof(Task));
  for (FpTasks* b : fp)
    for (int d = 0; d < 2; ++d) {
      b->off[d] = off;
      off = align256(off + b->task[d].size() * sizeof(CTask));
    }
  size_t o_sg[Lists::NK];
  for (int k = 0; k < Lists::NK; ++k) {
    o_sg[k] = off;
    off = align256(off + segs[k].size() * sizeof(CztSeg<T>));
  }
  std::vector<unsigned char> host(off, 0);
  std::memcpy(host.data() + o_dw, dw.data(), nj * sizeof(ContractDesc<T>));
  std::memcpy(host.data() + o_dp, dp.data(), nj * sizeof(ContractDesc<T>));
  int q = 0;
  for (auto& kv : tw_byN) {
    std::memcpy(host.data() + o_tw[q], kv.second.data(), kv.second.size() * sizeof(Task));
    ++q;
  }
  if (!tphi.empty()) std::memcpy(host.data() + o_tp, tphi.data(), tphi.size() * sizeof(Task));
  for (FpTasks* b : fp)
    for (int d = 0; d < 2; ++d)
      if (!b->task[d].empty()) std::memcpy(host.data() + b->off[d], b->task[d].data(), b->task[d].size() * sizeof(CTask));
  for (int k = 0; k < Lists::NK; ++k)
    if (!segs[k].empty()) std::memcpy(host.data() + o_sg[k], segs[k].data(), segs[k].size() * sizeof(CztSeg<T>));
  try {
    cudaStream_t st = setup_stream();
    amalloc(&ls->mem, off, st);
    ck(cudaMemcpyAsync(ls->mem, host.data(), off, cudaMemcpyHostToDevice, st));
    ck(cudaStreamSynchronize(st));  // host staging buffer is local
  } catch (...) {
    delete ls;
    throw;
  }
  char* base = reinterpret_cast<char*>(ls->mem);
  ls->desc_w = base + o_dw;
  ls->desc_phi = base + o_dp;
  q = 0;
  for (auto& kv : tw_byN) {
    ls->tiles_w.push_back({kv.first, {base + o_tw[q], (int)kv.second.size()}});
    ++q;
  }
  ls->tiles_phi = base + o_tp;
  ls->ntiles_phi = (int)tphi.size();
  auto group = [&](int N, const FpTasks& b) {
    Lists::FpGroup g;
    g.N = N;
    g.rt = b.rt;
    for (int d = 0; d < 2; ++d) {
      g.task[d] = base + b.off[d];
      g.n[d] = (int)b.task[d].size();
    }
    return g;
  };
  for (auto& kv : dir_byN) ls->dir_w.push_back(group(kv.first, kv.second));
  for (auto& kv : tile_byN) ls->tile_w.push_back(group(kv.first, kv.second));
  ls->dir_phi = group(1, dir_phi);
  ls->tile_phi = group(1, tile_phi);
  for (int k = 0; k < Lists::NK; ++k) {
    ls->segs[k] = base + o_sg[k];
    ls->nseg[k] = (int)segs[k].size();
    ls->items[k] = start[k];
    ls->stages[k] = stages[k];
  }
  return ls;
}

inline void rec(cudaEvent_t* ev, int i, cudaStream_t st) {
  if (ev) cudaEventRecord(ev[i], st);
}

// True while `st` is being captured into a CUDA graph.  The library's own
// events (last use, stage timing) are not recorded then: a captured record
// would tie the plan's events to the caller's graph (and cannot be waited
// on), so keeping a plan alive while a graph that captured it may still run
// is the caller's responsibility, as for the buffers it passed.
inline bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}
inline void mark_use(s2dw_plan_t p, cudaStream_t st) {
  if (!capturing(st)) cudaEventRecord(p->last_use, st);
}

// Direct contraction launches of one direction (the scaling parts ride
// with the first group); the number of launches.
int direct_groups(const Lists& ls) { return (int)ls.dir_w.size() + (ls.dir_w.empty() && ls.dir_phi.n[0] > 0 ? 1 : 0); }
template <typename T>
void run_direct(const Lists& ls, bool syn, const ContractDesc<T>* dw, const ContractDesc<T>* dp,
                const CallPtrs& ptrs, cudaStream_t st) {
  const int d = syn ? 1 : 0;
  const DirTasks<T> phi{dp, reinterpret_cast<const CTask*>(ls.dir_phi.task[d]), ls.dir_phi.n[d]};
  DirTasks<T> none = phi;
  none.n = 0;
  bool first = true;
  for (const auto& g : ls.dir_w) {
    launch_contract_direct<T>(g.N, syn, g.rt, DirTasks<T>{dw, reinterpret_cast<const CTask*>(g.task[d]), g.n[d]},
                           first ? phi : none, ptrs, st);
    first = false;
  }
  if (first) launch_contract_direct<T>(1, syn, ls.dir_phi.rt, DirTasks<T>{dw, nullptr, 0}, phi, ptrs, st);
}

// Analysis stages: [contraction + gamma | scaling contraction | beta | alpha chirp-z full-band | segmented
// | alpha direct].
// the half-length beta launches of a kind, one per transform length
template <typename T>
void launch_dct_parts(const Lists& ls, int kind, const CallPtrs& ptrs, cudaStream_t st) {
  const CztSeg<T>* segs = reinterpret_cast<const CztSeg<T>*>(ls.segs[kind]);
  for (const auto& pt : ls.dct_parts[kind - CZT_BETA_ANA_DCT])
    launch_czt<T>(kind, segs + pt[0], pt[1], pt[2], ls.maxlogM, ptrs, st, pt[3]);
}

// split matrix products of a kind (FP32 plans)
template <typename T>
void launch_products(const Lists& ls, int kind, const CallPtrs& ptrs, cudaStream_t st, long long limit = kWaitLimit) {
  if constexpr (sizeof(T) == sizeof(float))
    launch_split_gemm(kind == SG_KIND_BETA_RS ? 0 : kind - SG_KIND_BETA_ANA, reinterpret_cast<const CztSeg<T>*>(ls.segs[kind]),
                      ls.nseg[kind], ls.items[kind], ls.stages[kind], ptrs, st, limit);
}

template <typename T>
void run_analysis(const Lists& ls, const CallPtrs& ptrs, cudaStream_t st, cudaEvent_t* ev = nullptr) {
  const ContractDesc<T>* dw = reinterpret_cast<const ContractDesc<T>*>(ls.desc_w);
  const ContractDesc<T>* dp = reinterpret_cast<const ContractDesc<T>*>(ls.desc_phi);
  rec(ev, 0, st);
  if constexpr (sizeof(T) == sizeof(float)) {
    launch_fpack(dw, ls.njobs, ls.nbmax, ls.Lrmax, ptrs, st);
  }
  run_direct<T>(ls, false, dw, dp, ptrs, st);
  if constexpr (sizeof(T) == sizeof(float)) {
    for (auto& g : ls.tile_w)
      launch_contract_tile(g.N, 2, false, dw, reinterpret_cast<const CTask*>(g.task[0]), g.n[0], st);
    rec(ev, 1, st);
    launch_contract_tile(1, 1, false, dp, reinterpret_cast<const CTask*>(ls.tile_phi.task[0]), ls.tile_phi.n[0], st);
  } else {
    for (auto& t : ls.tiles_w)
      launch_contract<T>(t.first, 2, false, dw, reinterpret_cast<const TileTask*>(t.second.first), t.second.second,
                         ptrs, st);
    rec(ev, 1, st);
    launch_contract<T>(1, 1, false, dp, reinterpret_cast<const TileTask*>(ls.tiles_phi), ls.ntiles_phi, ptrs, st);
  }
  rec(ev, 2, st);
  launch_czt<T>(CZT_BETA_ANA, reinterpret_cast<const CztSeg<T>*>(ls.segs[0]), ls.nseg[0], ls.items[0], ls.maxlogM,
                ptrs, st, ls.ulogM[0]);
  launch_czt<T>(CZT_BETA_ANA_FFT, reinterpret_cast<const CztSeg<T>*>(ls.segs[6]), ls.nseg[6], ls.items[6],
                ls.maxlogM, ptrs, st, ls.ulogM[6]);
  launch_dct_parts<T>(ls, CZT_BETA_ANA_DCT, ptrs, st);
  launch_products<T>(ls, SG_KIND_BETA_ANA, ptrs, st);
  rec(ev, 3, st);
  launch_products<T>(ls, SG_KIND_ALPHA_ANA, ptrs, st);
  launch_czt<T>(CZT_ALPHA_ANA | ls.odd, reinterpret_cast<const CztSeg<T>*>(ls.segs[1]), ls.nseg[1], ls.items[1],
                ls.maxlogM, ptrs, st, ls.ulogM[1]);
  rec(ev, 4, st);
  launch_czt<T>(CZT_ALPHA_ANA_SEG | ls.odd, reinterpret_cast<const CztSeg<T>*>(ls.segs[8]), ls.nseg[8], ls.items[8],
                ls.maxlogM, ptrs, st, ls.ulogM[8]);
  rec(ev, 5, st);
  launch_czt<T>(CZT_ALPHA_ANA_DIRECT, reinterpret_cast<const CztSeg<T>*>(ls.segs[4]), ls.nseg[4], ls.items[4],
                ls.maxlogM, ptrs, st, ls.ulogM[4]);
  rec(ev, 6, st);
}

// Synthesis stages: [alpha direct | alpha chirp-z full-band | segmented | beta | contraction | scaling
// contraction | reduction].
template <typename T>
void run_synthesis(const Lists& ls, const CallPtrs& ptrs, const ReduceJobs& rj, int njobs, cudaStream_t st,
                   cudaEvent_t* ev = nullptr) {
  const ContractDesc<T>* dw = reinterpret_cast<const ContractDesc<T>*>(ls.desc_w);
  const ContractDesc<T>* dp = reinterpret_cast<const ContractDesc<T>*>(ls.desc_phi);
  rec(ev, 0, st);
  launch_czt<T>(CZT_ALPHA_SYN_DIRECT, reinterpret_cast<const CztSeg<T>*>(ls.segs[5]), ls.nseg[5], ls.items[5],
                ls.maxlogM, ptrs, st, ls.ulogM[5]);
  rec(ev, 1, st);
  launch_products<T>(ls, SG_KIND_ALPHA_SYN, ptrs, st);
  launch_czt<T>(CZT_ALPHA_SYN, reinterpret_cast<const CztSeg<T>*>(ls.segs[2]), ls.nseg[2], ls.items[2], ls.maxlogM,
                ptrs, st, ls.ulogM[2]);
  rec(ev, 2, st);
  launch_czt<T>(CZT_ALPHA_SYN_SEG | ls.odd, reinterpret_cast<const CztSeg<T>*>(ls.segs[9]), ls.nseg[9], ls.items[9],
                ls.maxlogM, ptrs, st, ls.ulogM[9]);
  rec(ev, 3, st);
  // MW grid: V from its L beta samples to the DH grid (torus coefficients, then the DH samples)
  launch_czt<T>(CZT_BETA_MW_DFT, reinterpret_cast<const CztSeg<T>*>(ls.segs[10]), ls.nseg[10], ls.items[10],
                ls.maxlogM, ptrs, st, ls.ulogM[10]);
  launch_czt<T>(CZT_BETA_RS_FFT, reinterpret_cast<const CztSeg<T>*>(ls.segs[11]), ls.nseg[11], ls.items[11],
                ls.maxlogM, ptrs, st, ls.ulogM[11]);
  launch_dct_parts<T>(ls, CZT_BETA_RS_DCT, ptrs, st);
  launch_products<T>(ls, SG_KIND_BETA_RS, ptrs, st);
  launch_czt<T>(CZT_BETA_RS, reinterpret_cast<const CztSeg<T>*>(ls.segs[12]), ls.nseg[12], ls.items[12],
                ls.maxlogM, ptrs, st, ls.ulogM[12]);
  launch_czt<T>(CZT_BETA_SYN, reinterpret_cast<const CztSeg<T>*>(ls.segs[3]), ls.nseg[3], ls.items[3], ls.maxlogM,
                ptrs, st, ls.ulogM[3]);
  launch_czt<T>(CZT_BETA_SYN_FFT, reinterpret_cast<const CztSeg<T>*>(ls.segs[7]), ls.nseg[7], ls.items[7],
                ls.maxlogM, ptrs, st, ls.ulogM[7]);
  launch_dct_parts<T>(ls, CZT_BETA_SYN_DCT, ptrs, st);
  launch_products<T>(ls, SG_KIND_BETA_SYN, ptrs, st);
  rec(ev, 4, st);
  run_direct<T>(ls, true, dw, dp, ptrs, st);
  if constexpr (sizeof(T) == sizeof(float)) {
    for (auto& g : ls.tile_w)
      launch_contract_tile(g.N, 2, true, dw, reinterpret_cast<const CTask*>(g.task[1]), g.n[1], st);
    rec(ev, 5, st);
    launch_contract_tile(1, 1, true, dp, reinterpret_cast<const CTask*>(ls.tile_phi.task[1]), ls.tile_phi.n[1], st);
  } else {
    for (auto& t : ls.tiles_w)
      launch_contract<T>(t.first, 2, true, dw, reinterpret_cast<const TileTask*>(t.second.first), t.second.second,
                         ptrs, st);
    rec(ev, 5, st);
    launch_contract<T>(1, 1, true, dp, reinterpret_cast<const TileTask*>(ls.tiles_phi), ls.ntiles_phi, ptrs, st);
  }
  rec(ev, 6, st);
  launch_syn_reduce<T>(rj, njobs, ls.Lmax, st);
  rec(ev, 7, st);
}

// (Re)builds the plan's own launch lists from its current methods; the
// previous lists are freed once the plan's private stream is idle.
template <typename T>
void own_lists_build(s2dw_plan_s* p) {
  Lists* ls = build_lists<T>(std::vector<s2dw_plan_t>{p});
  if (p->own_mem) cudaFreeAsync(p->own_mem, p->pst);
  // move into the plan (the plan frees the list memory at destruction)
  p->own_mem = ls->mem;
  p->own.mem = nullptr;
  ls->mem = nullptr;
  p->own.desc_w = ls->desc_w;
  p->own.desc_phi = ls->desc_phi;
  p->own.tiles_w = ls->tiles_w;
  p->own.tiles_phi = ls->tiles_phi;
  p->own.ntiles_phi = ls->ntiles_phi;
  p->own.dir_w = ls->dir_w;
  p->own.tile_w = ls->tile_w;
  p->own.dir_phi = ls->dir_phi;
  p->own.tile_phi = ls->tile_phi;
  for (int k = 0; k < Lists::NK; ++k) {
    p->own.segs[k] = ls->segs[k];
    p->own.nseg[k] = ls->nseg[k];
    p->own.items[k] = ls->items[k];
    p->own.stages[k] = ls->stages[k];
    p->own.ulogM[k] = ls->ulogM[k];
  }
  for (int k = 0; k < 3; ++k) p->own.dct_parts[k] = ls->dct_parts[k];
  p->own.maxlogM = ls->maxlogM;
  p->own.Lmax = ls->Lmax;
  p->own.odd = ls->odd;
  p->own.njobs = ls->njobs;
  p->own.nbmax = ls->nbmax;
  p->own.Lrmax = ls->Lrmax;
  delete ls;
}

// Byte offsets of a plan's workspace.
struct PlanLayout {
  size_t RS, RSphi, RSp, RSphi_p, fP, P, Pphi, images = 0, bytes = 0;  // images: operand images, in P
  std::vector<size_t> Y, X, ta, ts;
  struct GridOff { size_t tw, ca, pb, qb, pS, qS, root, bf, H, pm, tw2; };
  std::vector<GridOff> grid;
  struct SegOff { size_t tw, Ha, Hs; };
  std::vector<SegOff> seg;
  std::vector<std::array<size_t, 5>> sg;
};

// Workspace layout and launch methods of a plan whose bands and grids are set.
// bound: bands are upper bounds (s2dw_plan_bytes), so every table and buffer that
// bands up to kBandSlack below them could need (kappa underflows within 4e-4 of
// its support's end).
constexpr int kBandSlack = 5;
template <typename T>
PlanLayout plan_layout(s2dw_plan_s* p, bool bound) {
  const int L = p->L, N = p->N;
  PlanLayout o;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = align256(off + bytes);
    return at;
  };
  const bool dir64 = sizeof(T) == sizeof(double) && p->direct_w;
  const bool pairc = sizeof(T) == sizeof(float);  // FP32 contraction (pair table)
  const int NH = (N + 1) / 2;
  p->Lr = L + kPairPadL;  // read-ahead rows of the tile contraction
  p->Lrphi = p->Lphi + kPairPadL;
  p->Lrf = L + kPairPadL;
  const int nbw = (L + 31) / 32, nbp = (p->Lphi + 31) / 32;
  const bool pairt = pairc || dir64;  // R rows in the pair layout
  o.RS = pairt ? take(0) : take((size_t)L * 2 * NH * p->Lp * sizeof(T));
  o.RSphi = pairt ? take(0) : take((size_t)p->Lphi * p->Lphip * sizeof(T));
  o.RSp = pairt ? take((size_t)nbw * p->Lr * 2 * NH * 32 * sizeof(T)) : take(0);
  o.RSphi_p = pairt ? take((size_t)nbp * p->Lrphi * 32 * sizeof(T)) : take(0);
  const bool packf = pairc && !(p->direct_w && p->direct_phi);  // the direct contraction reads f itself
  o.fP = packf ? take((size_t)nbw * p->Lrf * 32 * sizeof(cx<T>)) : take(0);
  o.Y.resize(p->nscale + 1);
  o.X.resize(p->nscale + 1);
  for (int j = 0; j <= p->nscale; ++j) {
    const int Nj = (j == p->nscale) ? 1 : N;
    const int Lj = p->Ycols[j];
    o.Y[j] = take((size_t)Nj * Lj * Lj * sizeof(cx<T>));
    o.X[j] = take((size_t)Nj * 2 * p->gt[p->grid_of[j]].L * Lj * sizeof(cx<T>));
  }
  o.Pphi = take((size_t)p->nbr_phi * p->Lphi * p->Lphip32 * sizeof(cx<T>));
  // per grid: twiddles, chirps, roots, beta phases and weights, spectra
  auto& go = o.grid;
  go.resize(p->gt.size());
  // sets of tables of a grid (bound: scales whose bounds share a grid may have their own)
  auto sets = [&](size_t g) {
    return bound && p->multires ? (int)std::count(p->grid_of.begin(), p->grid_of.end(), (int)g) : 1;
  };
  for (size_t g = 0; g < p->gt.size(); ++g)
    for (int k = 0; k < sets(g); ++k) {
      const int Lg = p->gt[g].L, ng = 2 * Lg - 1, Mg = p->gt[g].M;
      go[g].tw = take((size_t)Mg * sizeof(cx<T>));
      go[g].ca = take((size_t)ng * sizeof(cx<T>));
      go[g].pb = take((size_t)(2 * Lg - 1) * sizeof(cx<T>));
      go[g].qb = take((size_t)2 * Lg * sizeof(cx<T>));
      go[g].pS = take((size_t)2 * Lg * sizeof(cx<T>));
      go[g].qS = take((size_t)(2 * Lg - 1) * sizeof(cx<T>));
      go[g].root = take((size_t)ng * sizeof(cx<T>));
      go[g].bf = take((size_t)(4 * Lg - 1) * sizeof(cx<T>));
      go[g].H = take((size_t)4 * Mg * sizeof(cx<T>));
      go[g].pm = take((size_t)ng * sizeof(cx<T>));
      go[g].tw2 = take((size_t)twiddle_entries(p->gt[g].logM - 1) * sizeof(cx<T>));
    }
  // segmented chirp-z tables of the scales that use it (chirp-z bands only)
  p->seg.assign(p->nscale + 1, s2dw_plan_s::SegTables());
  auto& so = o.seg;
  so.resize(p->nscale + 1);
  for (int j = 0; j <= p->nscale; ++j) {
    const auto& G = p->gt[p->grid_of[j]];
    const int Lj = p->Ycols[j];
    if (Lj <= kDirectMaxLj) continue;  // direct sums
    auto& sgt = p->seg[j];
    if (bound) {  // any choice: twiddles and two times S M' <= 1.7 M log2 M / 9 entries
      take((size_t)8 * G.M * sizeof(cx<T>));
      continue;
    }
    seg_choice(G.L, Lj, G.logM, sgt.logM, sgt.P, sgt.S);
    if (sgt.S == 0) continue;
    const size_t Ms = (size_t)1 << sgt.logM;
    so[j].tw = take((size_t)twiddle_entries(sgt.logM) * sizeof(cx<T>));
    so[j].Ha = take((size_t)sgt.S * Ms * sizeof(cx<T>));
    so[j].Hs = take((size_t)sgt.S * Ms * sizeof(cx<T>));
  }
  // default launch methods: direct sums for L_j <= 32, split products where they are
  // faster, segmented chirp-z where it was chosen above, else the grid's chirp-z
  for (int d = 0; d < 2; ++d) {
    p->alpha_mode[d].assign(p->nscale + 1, 1);
    p->alpha_sg[d].assign(p->nscale + 1, 0);
    for (int j = 0; j <= p->nscale; ++j) {
      const int Lj = p->Ycols[j];
      if (Lj <= (d == 0 ? kDirectMaxLjAna : kDirectMaxLj)) p->alpha_mode[d][j] = 0;
      else if (p->seg[j].S > 0) p->alpha_mode[d][j] = 2;
      const auto& G = p->gt[p->grid_of[j]];
      // (bound: for any band up to kBandSlack below)
      for (int b = Lj; pairc && p->alpha_mode[d][j] != 0 && b >= Lj - (bound ? kBandSlack : 0); --b) {
        int lm, P, S;
        seg_choice(G.L, b, G.logM, lm, P, S);
        const double cost = S > 0 ? (double)(S + 1) * ((size_t)1 << lm) * lm : 2.0 * G.M * G.logM;
        if (sg_alpha_faster(G.L, b, cost, S > 0)) p->alpha_sg[d][j] = 1;
      }
      if (p->alpha_sg[d][j]) p->alpha_mode[d][j] = 3;
    }
  }
  // basis tables of the split products
  auto& o_sg = o.sg;
  o_sg.resize(p->gt.size());
  for (size_t g = 0; g < p->gt.size(); ++g) {
    auto& G = p->gt[g];
    o_sg[g].fill(SIZE_MAX);
    if (!pairc) continue;
    // (the bound of a scale's own grid may be a power of two where the grid is none)
    const bool pow2 = !(bound && p->multires) && 4 * G.L == G.M;
    // (an MW analysis evaluates at the MW samples, whatever L)
    G.sg_beta[0] = sg_beta_faster(G.L, pow2 && !p->mw);
    G.sg_beta[1] = sg_beta_faster(G.L, pow2);
    bool need[5] = {G.sg_beta[0], G.sg_beta[1], false, false, p->mw && sg_beta_faster(G.L, pow2)};
    for (int j = 0; j <= p->nscale; ++j)
      if (p->grid_of[j] == (int)g)
        for (int d = 0; d < 2; ++d) need[2 + d] = need[2 + d] || p->alpha_sg[d][j];
    for (int k = 0; k < 5; ++k)
      if (need[k]) o_sg[g][k] = take(sets(g) * sg_table(k == 4 ? 0 : k, G.L).bytes);
  }
  // operand images of one product launch (shared by the five kinds), in the
  // buffer of the synthesis partials: the contraction that writes those comes
  // after every product launch of its call
  size_t& sgd_bytes = o.images;
  if (pairc) {
    size_t most = 0;
    for (int k = 0; k < 5; ++k) {
      size_t n = 0;
      for (int j = 0; j <= p->nscale; ++j) {
        const auto& G = p->gt[p->grid_of[j]];
        const bool used = k < 2 ? G.sg_beta[k] : (k < 4 ? p->alpha_sg[k - 2][j] != 0 : o_sg[p->grid_of[j]][4] != SIZE_MAX);
        if (!used) continue;
        const SgDims d = sg_dims(k == 4 ? 0 : k, G.L, p->Ycols[j], j == p->nscale ? 1 : N, G.nb);
        n += (size_t)d.data_tiles * d.stages;
      }
      most = std::max(most, n);
    }
    sgd_bytes = most * kSgDataBytes;
  }
  o.P = take(std::max((size_t)p->nbr * L * p->Lp32 * sizeof(cx<T>), sgd_bytes));
  // tensor-core basis images of the direct alpha sums (FP32 plans)
  auto &o_ta = o.ta, &o_ts = o.ts;
  o_ta.assign(p->nscale + 1, SIZE_MAX);
  o_ts.assign(p->nscale + 1, SIZE_MAX);
  if (sizeof(T) == sizeof(float)) {
    for (int j = 0; j <= p->nscale; ++j) {
      int Lj = p->Ycols[j];
      const int Lg = p->gt[p->grid_of[j]].L;
      if (Lj <= 0) continue;
      if (bound && Lj <= kDirectMaxLj + kBandSlack) Lj = std::min(Lj, kDirectMaxLj);
      if (Lj <= kDirectMaxLjAna) o_ta[j] = take(alpha_tc_table_floats(Lg, Lj, false) * sizeof(float));
      if (Lj <= kDirectMaxLj) o_ts[j] = take(alpha_tc_table_floats(Lg, Lj, true) * sizeof(float));
    }
  }
  o.bytes = off;
  return o;
}

template <typename T>
void plan_build_typed(s2dw_plan_s* p, const double* kap_d, const double* phi_d, const double* sabs_d,
                      const double* q_d, cudaStream_t st) {
  const int L = p->L, N = p->N;
  const bool dir64 = sizeof(T) == sizeof(double) && p->direct_w;
  const bool pairc = sizeof(T) == sizeof(float);  // FP32 contraction (pair table)
  const bool pairt = pairc || dir64;              // R rows in the pair layout
  const bool packf = pairc && !(p->direct_w && p->direct_phi);
  const PlanLayout o = plan_layout<T>(p, false);
  const size_t off = o.bytes;
  p->ws_bytes = off;
  amalloc(&p->ws, off, st);
  pool_live(p->device, (int64_t)off);
  char* b = reinterpret_cast<char*>(p->ws);
  p->RS = pairt ? nullptr : b + o.RS;
  p->RSphi = pairt ? nullptr : b + o.RSphi;
  p->RSp = pairt ? b + o.RSp : nullptr;
  p->RSphi_p = pairt ? b + o.RSphi_p : nullptr;
  p->fP = packf ? b + o.fP : nullptr;
  p->Y.resize(p->nscale + 1);
  p->X.resize(p->nscale + 1);
  for (int j = 0; j <= p->nscale; ++j) {
    p->Y[j] = b + o.Y[j];
    p->X[j] = b + o.X[j];
  }
  p->P = b + o.P;
  p->Pphi = b + o.Pphi;
  for (size_t g = 0; g < p->gt.size(); ++g) {
    auto& G = p->gt[g];
    G.tw = b + o.grid[g].tw;
    G.chirp_a = b + o.grid[g].ca;
    G.pre_b = b + o.grid[g].pb;
    G.post_b = b + o.grid[g].qb;
    G.preS_b = b + o.grid[g].pS;
    G.postS_b = b + o.grid[g].qS;
    G.root_a = b + o.grid[g].root;
    G.bfft = b + o.grid[g].bf;
    G.Hs = b + o.grid[g].H;
    G.pre_mw = b + o.grid[g].pm;
    G.tw2 = b + o.grid[g].tw2;
    for (int k = 0; k < 5; ++k) G.sg[k] = o.sg[g][k] != SIZE_MAX ? b + o.sg[g][k] : nullptr;
  }
  for (int j = 0; j <= p->nscale; ++j) {
    auto& sgt = p->seg[j];
    if (sgt.S == 0) continue;
    sgt.tw = b + o.seg[j].tw;
    sgt.Ha = b + o.seg[j].Ha;
    sgt.Hs = b + o.seg[j].Hs;
  }
  p->sg_data = o.images > 0 ? p->P : nullptr;
  p->tc_ana.assign(p->nscale + 1, nullptr);
  p->tc_syn.assign(p->nscale + 1, nullptr);
  std::vector<TcBasis> tcb;
  for (int j = 0; j <= p->nscale; ++j) {
    const int Lj = p->Ycols[j], Lg = p->gt[p->grid_of[j]].L;
    for (int d = 0; d < 2; ++d) {
      const size_t at = d ? o.ts[j] : o.ta[j];
      if (at == SIZE_MAX) continue;
      (d ? p->tc_syn : p->tc_ana)[j] = b + at;
      tcb.push_back(TcBasis{reinterpret_cast<float*>(b + at), Lg, (short)Lj, (short)d});
    }
  }
  if (!tcb.empty()) {  // (the last part of the workspace)
    char* first = reinterpret_cast<char*>(tcb[0].out);
    ck(cudaMemsetAsync(first, 0, b + off - first, st));  // image pads
    ck(alpha_tc_build_tables(tcb.data(), (int)tcb.size(), st));
  }

  // ---- R tables ----
  std::vector<int> slot_w((size_t)L * 2, -1), slot_p(p->Lphi, 0);
  for (int l = 0; l < L; ++l)
    for (int j = 0; j < p->nscale; ++j)
      if (p->Lj[j] > 0 && l >= p->lo[j] && l <= p->hi[j]) slot_w[(size_t)l * 2 + (j % 2)] = j;
  int* slot_d = nullptr;
  amalloc(&slot_d, (slot_w.size() + slot_p.size()) * sizeof(int), st);
  ck(cudaMemcpyAsync(slot_d, slot_w.data(), slot_w.size() * sizeof(int), cudaMemcpyHostToDevice, st));
  ck(cudaMemcpyAsync(slot_d + slot_w.size(), slot_p.data(), slot_p.size() * sizeof(int), cudaMemcpyHostToDevice,
                     st));
  if (pairt) {
    ck(launch_rtable_pair<T>(reinterpret_cast<T*>(p->RSp), p->tab->d64, kap_d, sabs_d, slot_d, L, p->Lr, N, 2, L, st));
    ck(launch_rtable_pair<T>(reinterpret_cast<T*>(p->RSphi_p), p->tab->d64, phi_d, nullptr, slot_d + slot_w.size(),
                             p->Lphi, p->Lrphi, 1, 1, L, st));
  } else {
    ck(launch_rtable<T>(reinterpret_cast<T*>(p->RS), p->tab->d64, kap_d, sabs_d, slot_d, L, p->Lp, N, 2, L, st));
    ck(launch_rtable<T>(reinterpret_cast<T*>(p->RSphi), p->tab->d64, phi_d, nullptr, slot_d + slot_w.size(),
                        p->Lphi, p->Lphip, 1, 1, L, st));
  }
  // ---- chirp tables of every grid (float64, then the working precision) ----
  double2* t64 = nullptr;
  double* qg = nullptr;
  {
    size_t need = 0;
    for (const auto& G : p->gt) {
      const size_t Lg = G.L, ng = 2 * Lg - 1;
      need = std::max(need, (size_t)G.M + ng + (2 * Lg - 1) + 2 * Lg + 2 * Lg + (2 * Lg - 1) + ng + (4 * Lg - 1) +
                                4 * (size_t)G.M);
      need = std::max(need, sg_build_scratch(G.L));  // roots of the split products' basis
    }
    amalloc(&t64, need * sizeof(double2), st);
    amalloc(&qg, (size_t)2 * p->gt.back().L * sizeof(double), st);
  }
  for (auto& G : p->gt) {
    const int Lg = G.L, ng = 2 * Lg - 1, Mg = G.M;
    double2* tw64 = t64;
    double2* ca64 = tw64 + Mg;
    double2* pb64 = ca64 + ng;
    double2* qb64 = pb64 + (2 * Lg - 1);
    double2* pS64 = qb64 + 2 * Lg;
    double2* qS64 = pS64 + 2 * Lg;
    double2* rt64 = qS64 + (2 * Lg - 1);
    double2* bf64 = rt64 + ng;
    double2* H64 = bf64 + (4 * Lg - 1);
    const double* q_g = q_d;  // the plan's own grid reuses its weights
    if (Lg != L) {
      ck(launch_dh_weights(qg, Lg, st));
      q_g = qg;
    }
    ck(launch_chirp_build64(tw64, ca64, pb64, qb64, pS64, qS64, rt64, bf64, H64, q_g, Lg, G.logM, st));
    auto put = [&](void* dst, const double2* src, int64_t cnt) {
      if (sizeof(T) == sizeof(double))
        ck(cudaMemcpyAsync(dst, src, (size_t)cnt * sizeof(double2), cudaMemcpyDeviceToDevice, st));
      else
        ck(launch_to_prec<float>(reinterpret_cast<float2*>(dst), src, cnt, st));
    };
    put(G.tw, tw64, Mg);
    put(G.chirp_a, ca64, ng);
    put(G.pre_b, pb64, 2 * Lg - 1);
    put(G.post_b, qb64, 2 * Lg);
    put(G.preS_b, pS64, 2 * Lg);
    put(G.postS_b, qS64, 2 * Lg - 1);
    put(G.root_a, rt64, ng);
    put(G.bfft, bf64, 4 * Lg - 1);
    put(G.Hs, H64, (int64_t)4 * Mg);
    ck(launch_mw_pre64(tw64, Lg, st));  // reuse the scratch: the grid's tables are converted above
    put(G.pre_mw, tw64, ng);
    ck(launch_twiddles64(tw64, G.logM - 1, st));  // length 2Lg (half-length beta transforms)
    put(G.tw2, tw64, twiddle_entries(G.logM - 1));
    ck(sg_build_tables(G.sg, tw64, q_g, Lg, p->mw, st));  // (its roots in the same scratch)
  }
  {
    size_t need = 0;
    for (const auto& sgt : p->seg)
      if (sgt.S)
        need = std::max(need, (size_t)twiddle_entries(sgt.logM) + 2 * (size_t)sgt.S * ((size_t)1 << sgt.logM));
    double2* s64 = nullptr;
    if (need) amalloc(&s64, need * sizeof(double2), st);
    for (int j = 0; j <= p->nscale; ++j) {
      const auto& sgt = p->seg[j];
      if (sgt.S == 0) continue;
      const auto& G = p->gt[p->grid_of[j]];
      const int64_t Ms = (int64_t)1 << sgt.logM, ntw = twiddle_entries(sgt.logM);
      double2* tw64 = s64;
      double2* ha64 = tw64 + ntw;
      double2* hs64 = ha64 + sgt.S * Ms;
      ck(launch_seg_build64(tw64, ha64, hs64, G.L, p->Ycols[j], sgt.logM, sgt.P, sgt.S, st));
      auto put = [&](void* dst, const double2* src, int64_t cnt) {
        if (sizeof(T) == sizeof(double))
          ck(cudaMemcpyAsync(dst, src, (size_t)cnt * sizeof(double2), cudaMemcpyDeviceToDevice, st));
        else
          ck(launch_to_prec<float>(reinterpret_cast<float2*>(dst), src, cnt, st));
      };
      put(sgt.tw, tw64, ntw);
      put(sgt.Ha, ha64, sgt.S * Ms);
      put(sgt.Hs, hs64, sgt.S * Ms);
    }
    afree(s64, st);
  }
  afree(qg, st);
  afree(t64, st);
  afree(slot_d, st);
  ck(cudaStreamSynchronize(st));  // slot_w / slot_p host vectors are local

  // ---- descriptors, tiles, launch lists ----
  if (pairc) {
    delta_pair_ensure(p->tab, st);
    kernels_prepare(false, true);
  } else if (dir64) {
    delta_pair64_ensure(p->tab, st);
  }
  ContractDesc<T> dw, dp;
  // (FP32 plans read the pair table only)
  const T* delta = sizeof(T) == sizeof(double) ? reinterpret_cast<const T*>(p->tab->d64) : nullptr;
  fill_desc<T>(p, dw, dp, delta);
  p->desc_w_host.assign(reinterpret_cast<unsigned char*>(&dw), reinterpret_cast<unsigned char*>(&dw) + sizeof(dw));
  p->desc_phi_host.assign(reinterpret_cast<unsigned char*>(&dp), reinterpret_cast<unsigned char*>(&dp) + sizeof(dp));
  if (pairc) {
    // the reported value of the last choice; it no longer selects a kernel
    {
      int dev = 0, sms = 0;
      ck(cudaGetDevice(&dev));
      ck(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      const long long nbk = (p->L0 + 31) / 32, npairs = nbk * (nbk + 1) / 2;
      if (!pair_shapes_offered(N) || npairs < 3LL * sms) p->pair_shape = kPairShapeTile;
      else p->pair_shape = N >= 4 ? kPairShapePair : kPairShapeTile2;
    }
  } else if (!dir64) {
    build_tiles(p->L0, p->lend_w, p->TMP, 0, p->tiles_w_host);
    build_tiles(p->Lphi, p->lphi, p->TMP, 0, p->tiles_phi_host);
    sort_tiles(p->tiles_w_host);
    sort_tiles(p->tiles_phi_host);
  }
  own_lists_build<T>(p);
  // the cap covers every plan size (M <= 8192 for L <= 2048), so plans of
  // different sizes can share a batched launch
  kernels_prepare(sizeof(T) == sizeof(double), false);
}

// Sizes, kernels and grids that follow from the bands (p->Lj, L0, lphi).
void plan_shape(s2dw_plan_s* p) {
  const int L = p->L, N = p->N;
  const unsigned flags = p->flags;
  p->Lphi = p->lphi + 1;
  p->Ycols = p->Lj;
  p->Ycols.push_back(p->Lphi);
  p->Lp = round_up(L, 32);  // R-table row pitch: whole 32-row tiles are staged
  p->Lp32 = round_up(L, 32);
  p->Lphip = round_up(p->Lphi, 32);
  p->Lphip32 = round_up(p->Lphi, 32);
  if (p->fp64) {
    p->direct_w = p->direct_phi = L <= kContractDirectMaxL64;
  } else {
    p->direct_w = p->L0 <= contract_direct_max_l(N);
    p->direct_phi = p->Lphi <= contract_direct_max_l(1);
  }
  // blocks of partials: TMP rows each; the direct contraction writes whole 32-row tiles
  const int rows = p->direct_w ? 32 : p->TMP, rows_phi = p->direct_phi ? 32 : p->TMP;
  p->nbr = (p->L0 + rows - 1) / rows * (rows / p->TMP);
  p->nbr_phi = (p->Lphi + rows_phi - 1) / rows_phi * (rows_phi / p->TMP);
  // sampling grid of every scale (last: the scaling part): the full grid of
  // band-limit L, or with S2DW_MULTIRES the grid of the scale's own
  // band-limit (1 + the last l with a nonzero kernel)
  p->multires = (flags & S2DW_MULTIRES) != 0;
  p->mw = (flags & S2DW_MW) != 0;
  if (p->mw && p->multires) throw CudaFail{cudaErrorInvalidValue};
  std::vector<int> Lg(p->nscale + 1);
  for (int j = 0; j < p->nscale; ++j) Lg[j] = p->multires ? std::max(1, p->Lj[j]) : L;
  Lg[p->nscale] = p->multires ? p->Lphi : L;
  std::vector<int> uniq(Lg);
  std::sort(uniq.begin(), uniq.end());
  uniq.erase(std::unique(uniq.begin(), uniq.end()), uniq.end());
  p->gt.resize(uniq.size());
  p->logM = 0;
  for (size_t g = 0; g < uniq.size(); ++g) {
    auto& G = p->gt[g];
    G.L = uniq[g];
    G.logM = 5;  // the radix-16 convolution engine needs M >= 32
    while ((1 << G.logM) < 4 * G.L - 2) ++G.logM;
    G.M = 1 << G.logM;
    G.nb = p->mw ? G.L : 2 * G.L;
    p->logM = std::max(p->logM, G.logM);
  }
  p->M = 1 << p->logM;
  p->grid_of.resize(p->nscale + 1);
  for (int j = 0; j <= p->nscale; ++j)
    p->grid_of[j] = (int)(std::lower_bound(uniq.begin(), uniq.end(), Lg[j]) - uniq.begin());
  p->woff.resize(p->nscale + 1);
  int64_t wacc = 0;
  for (int j = 0; j < p->nscale; ++j) {
    p->woff[j] = wacc;
    wacc += (int64_t)N * p->gt[p->grid_of[j]].nb * (2 * Lg[j] - 1);
  }
  p->woff[p->nscale] = wacc;
}

// sht_mode: the companion plan of s2dw_sht_*: no wavelet scales, N = 1 and
// Phi_l = sqrt((2l+1)/(4 pi)) for every l < L, so that its scaling part is
// the spherical harmonic transform pair on the DH sphere grid.
int plan_create(s2dw_plan_t* out, int L, int N, double lam, int J0, unsigned flags, bool sht_mode = false) {
  if (sht_mode) {
    N = 1;
    lam = 2.0;
    J0 = jmax_of(L, lam);
  }
  const int Jm = jmax_of(L, lam);
  if (J0 < 0 || J0 > Jm) return S2DW_EINVAL;
  const int J = Jm - J0;
  if (J + 1 > 64) return S2DW_ENOTSUP;
  s2dw_plan_s* p = new s2dw_plan_s();
  p->L = L;
  p->N = N;
  p->J0 = J0;
  p->J = J;
  p->nscale = J + 1;
  p->flags = flags | S2DW_REAL_SIGNAL;
  p->lam = lam;
  p->fp64 = (flags & S2DW_FP64) != 0;
  p->E = contract_rows_per_thread(p->fp64);
  p->TMP = 8 * p->E;
  cudaStream_t st = nullptr;
  double *kap = nullptr, *phi = nullptr, *sabs = nullptr, *q = nullptr, *gl = nullptr;
  double2* psi = nullptr;
  int rc = S2DW_OK;
  try {
    ck(cudaGetDevice(&p->device));
    setup_stream();  // configures the caching memory pool once per device
    ck(cudaStreamCreateWithFlags(&p->pst, cudaStreamNonBlocking));
    ck(cudaEventCreateWithFlags(&p->last_use, cudaEventDisableTiming));
    st = p->pst;
    std::vector<double> glx, glw;
    const int Q = 16, PAN = 32;
    gauss_legendre(Q, glx, glw);
    amalloc(&gl, (2 * Q + 1) * sizeof(double), st);  // nodes, weights, the kappa normalisation
    ck(cudaMemcpyAsync(gl, glx.data(), Q * sizeof(double), cudaMemcpyHostToDevice, st));
    ck(cudaMemcpyAsync(gl + Q, glw.data(), Q * sizeof(double), cudaMemcpyHostToDevice, st));
    amalloc(&kap, (size_t)(J + 1) * L * sizeof(double), st);
    amalloc(&phi, (size_t)L * sizeof(double), st);
    amalloc(&sabs, (size_t)L * N * sizeof(double), st);
    amalloc(&psi, (size_t)(J + 1) * L * N * sizeof(double2), st);
    amalloc(&q, (size_t)2 * L * sizeof(double), st);
    ck(launch_kernel_values(kap, phi, sabs, psi, q, L, N, J, lam, gl, gl + Q, Q, PAN, gl + 2 * Q, st));
    std::vector<double> kap_h((size_t)(J + 1) * L);
    p->phi_host.resize(L);
    p->psi_host.resize((size_t)(J + 1) * L * N * 2);
    ck(cudaMemcpyAsync(kap_h.data(), kap, kap_h.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    ck(cudaMemcpyAsync(p->phi_host.data(), phi, L * sizeof(double), cudaMemcpyDeviceToHost, st));
    ck(cudaMemcpyAsync(p->psi_host.data(), psi, p->psi_host.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    ck(cudaStreamSynchronize(st));
    if (sht_mode) {
      for (int l = 0; l < L; ++l) p->phi_host[l] = std::sqrt((2.0 * l + 1.0) / (4.0 * 3.14159265358979323846));
      ck(cudaMemcpyAsync(phi, p->phi_host.data(), L * sizeof(double), cudaMemcpyHostToDevice, st));
      ck(cudaStreamSynchronize(st));
      p->nscale = 0;
      p->sht = true;
    }
    // supports where kappa^j(l) > 0 and their overlaps
    p->lo.assign(p->nscale, -1);
    p->hi.assign(p->nscale, -1);
    p->Lj.assign(p->nscale, 0);
    std::vector<int> count(L, 0);
    for (int j = 0; j < p->nscale; ++j)
      for (int l = 0; l < L; ++l)
        if (kap_h[(size_t)j * L + l] > 0.0) {
          if (p->lo[j] < 0) p->lo[j] = l;
          p->hi[j] = l;
          count[l]++;
        }
    for (int l = 0; l < L; ++l)
      if (count[l] > 2) throw CudaFail{cudaErrorInvalidValue};
    for (int j = 0; j < p->nscale; ++j) {
      if (p->hi[j] >= 0) p->Lj[j] = p->hi[j] + 1;
      if (j >= 2 && p->hi[j] >= 0 && p->lo[j - 2] >= 0 && p->lo[j - 2] <= p->hi[j])
        throw CudaFail{cudaErrorInvalidValue};
      p->lend_w = std::max(p->lend_w, p->hi[j]);
      p->L0 = std::max(p->L0, p->Lj[j]);
    }
    p->lphi = 0;
    for (int l = 0; l < L; ++l)
      if (p->phi_host[l] > 0.0) p->lphi = l;
    plan_shape(p);
    p->tab = delta_acquire(L, st);
    if (p->fp64) plan_build_typed<double>(p, kap, phi, sabs, q, st);
    else plan_build_typed<float>(p, kap, phi, sabs, q, st);
    ck(cudaStreamSynchronize(st));
  } catch (const CudaFail& e) {
    rc = (e.err == cudaErrorMemoryAllocation) ? S2DW_ENOMEM
         : (e.err == cudaErrorInvalidValue) ? S2DW_EINVAL
                                             : S2DW_ECUDA;
  } catch (const std::bad_alloc&) {
    rc = S2DW_ENOMEM;
  } catch (...) {
    rc = S2DW_ECUDA;
  }
  if (st) {
    afree(gl, st);
    afree(kap, st);
    afree(phi, st);
    afree(sabs, st);
    afree(psi, st);
    afree(q, st);
  }
  if (rc != S2DW_OK) {
    cudaGetLastError();
    delete p;
    return rc;
  }
  *out = p;
  return S2DW_OK;
}

int plan_args(int L, int N, double lambda, int J0, unsigned flags) {
  const unsigned prec = flags & (S2DW_FP64 | S2DW_MIXED);
  if (prec != S2DW_FP64 && prec != S2DW_MIXED) return S2DW_EINVAL;
  if (flags & ~(unsigned)(S2DW_FP64 | S2DW_MIXED | S2DW_REAL_SIGNAL | S2DW_MULTIRES | S2DW_MW)) return S2DW_EINVAL;
  if ((flags & S2DW_MW) && (flags & S2DW_MULTIRES)) return S2DW_EINVAL;
  // invalid requests (no transform exists) before limits of this build
  if (L < 2 || N < 1 || N > L) return S2DW_EINVAL;
  if (!(lambda > 1.0) || !std::isfinite(lambda)) return S2DW_EINVAL;
  const int jm = jmax_of(L, lambda);
  if (jm < 0) return S2DW_ENOTSUP;  // over a million scales
  if (J0 < 0 || J0 > jm) return S2DW_EINVAL;
  if (L > 2048 || N > 8) return S2DW_ENOTSUP;
  return S2DW_OK;
}

int err_of(cudaError_t e) {
  if (e == cudaSuccess) return S2DW_OK;
  if (e == cudaErrorMemoryAllocation) return S2DW_ENOMEM;
  return S2DW_ECUDA;
}

}  // namespace

// ===========================================================================
// C ABI
// ===========================================================================
extern "C" {

const char* s2dw_strerror(int status) {
  switch (status) {
    case S2DW_OK: return "ok";
    case S2DW_EINVAL: return "invalid argument";
    case S2DW_ENOMEM: return "device allocation failed";
    case S2DW_ECUDA: return "CUDA call or kernel launch failed";
    case S2DW_ETIMEOUT: return "bounded device wait ran out";
    case S2DW_EBUSY: return "resource busy";
    case S2DW_ENOTSUP: return "not supported by this build";
    default: return "unknown status";
  }
}

int s2dw_plan(s2dw_plan_t* out, int L, int N, double lambda, int J0, unsigned flags) {
  if (!out) return S2DW_EINVAL;
  *out = nullptr;
  if (int rc = plan_args(L, N, lambda, J0, flags); rc != S2DW_OK) return rc;
  try {
    return plan_create(out, L, N, lambda, J0, flags);
  } catch (...) {
    return S2DW_ECUDA;
  }
}

int s2dw_plan_bytes(int L, int N, double lambda, int J0, unsigned flags, int64_t* bytes) {
  if (!bytes) return S2DW_EINVAL;
  if (int rc = plan_args(L, N, lambda, J0, flags); rc != S2DW_OK) return rc;
  try {
    s2dw_plan_s p;
    p.L = L, p.N = N, p.J0 = J0, p.lam = lambda, p.flags = flags | S2DW_REAL_SIGNAL;
    p.J = jmax_of(L, lambda) - J0;
    p.nscale = p.J + 1;
    if (p.nscale > 64) return S2DW_ENOTSUP;
    p.fp64 = (flags & S2DW_FP64) != 0;
    p.E = contract_rows_per_thread(p.fp64);
    p.TMP = 8 * p.E;
    // kappa^j is supported in L lambda^-(j+1) < l < L lambda^(1-j), Phi in l < L lambda^-J
    // (one more where the power is rounded)
    auto band = [&](int e) { return (int)std::min<double>(L, std::floor(L * std::pow(lambda, e)) + 2); };
    p.lo.assign(p.nscale, -1);
    p.hi.assign(p.nscale, -1);
    p.Lj.assign(p.nscale, 0);
    for (int j = 0; j < p.nscale; ++j) {
      p.Lj[j] = band(1 - j);
      p.L0 = std::max(p.L0, p.Lj[j]);
    }
    p.lphi = band(-p.J) - 1;
    plan_shape(&p);
    *bytes = (int64_t)(p.fp64 ? plan_layout<double>(&p, true).bytes : plan_layout<float>(&p, true).bytes);
  } catch (...) {
    return S2DW_ENOMEM;
  }
  return S2DW_OK;
}

int s2dw_plan_destroy(s2dw_plan_t plan) {
  if (!plan) return S2DW_OK;
  drop_batches_with(plan);
  delete plan;  // waits for the plan's last recorded call, frees stream-ordered
  return err_of(cudaGetLastError());
}

int s2dw_query(s2dw_plan_t p, int* J, int64_t* w_elems_per_scale, int64_t* wphi_elems, int64_t* workspace_bytes,
               int64_t* total_device_bytes) {
  if (!p) return S2DW_EINVAL;
  const int64_t L = p->L, n = 2 * L - 1;
  const int64_t wps = p->multires ? 0 : (int64_t)p->N * p->gt[0].nb * n;
  const auto& Gp = p->gt[p->grid_of[p->nscale]];
  const int64_t Lp = Gp.L, wph = (int64_t)Gp.nb * (2 * Lp - 1);
  const int64_t el = p->fp64 ? 8 : 4;
  if (J) *J = p->J;
  if (w_elems_per_scale) *w_elems_per_scale = wps;
  if (wphi_elems) *wphi_elems = wph;
  if (workspace_bytes) *workspace_bytes = (int64_t)p->ws_bytes;
  if (total_device_bytes)
    *total_device_bytes = (int64_t)p->ws_bytes + (p->woff[p->nscale] + wph) * el + L * L * 2 * el;
  return S2DW_OK;
}

int s2dw_steer(s2dw_plan_t p, const void* W, const double* gammas, int ngamma, void* out, void* stream) {
  if (!p || !W || !gammas || !out || ngamma < 1 || ngamma > kSteerMaxGamma) return S2DW_EINVAL;
  const int N = p->N;
  SteerWeights sw;
  std::memset(&sw, 0, sizeof(sw));
  for (int t = 0; t < ngamma; ++t)
    for (int g = 0; g < N; ++g) {
      const double x = gammas[t] - 3.14159265358979323846 * g / N;
      double z = 0.0;
      for (int k = 0; k < N; ++k) z += std::cos((-(N - 1) + 2 * k) * x);
      sw.w[t][g] = z / N;
    }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const size_t el = p->fp64 ? sizeof(double) : sizeof(float);
  cudaError_t e = cudaSuccess;
  if (!p->multires) {
    const int64_t per_scale = (int64_t)p->gt[0].nb * (2 * p->L - 1);
    e = p->fp64 ? launch_steer<double>(W, out, sw, p->nscale, N, ngamma, per_scale, st)
                : launch_steer<float>(W, out, sw, p->nscale, N, ngamma, per_scale, st);
  } else {
    // scales of different grids: out holds [ngamma][2Lg][2Lg-1] per scale, in order
    for (int j = 0; j < p->nscale && e == cudaSuccess; ++j) {
      const int64_t Lg = p->gt[p->grid_of[j]].L, per_scale = 2 * Lg * (2 * Lg - 1);
      const char* Wj = reinterpret_cast<const char*>(W) + (size_t)p->woff[j] * el;
      char* Oj = reinterpret_cast<char*>(out) + (size_t)(p->woff[j] / N) * ngamma * el;
      e = p->fp64 ? launch_steer<double>(Wj, Oj, sw, 1, N, ngamma, per_scale, st)
                  : launch_steer<float>(Wj, Oj, sw, 1, N, ngamma, per_scale, st);
    }
  }
  return err_of(e);
}

namespace {
int sht_child(s2dw_plan_t p, s2dw_plan_t* c) {
  if (!p->sht_child) {
    const int rc = plan_create(&p->sht_child, p->L, 1, 2.0, 0, p->fp64 ? S2DW_FP64 : S2DW_MIXED, true);
    if (rc != S2DW_OK) {
      p->sht_child = nullptr;
      return rc;
    }
  }
  *c = p->sht_child;
  return S2DW_OK;
}
}  // namespace

int s2dw_sht_inverse(s2dw_plan_t p, const void* flm, void* fpix, void* stream) {
  if (!p || !flm || !fpix) return S2DW_EINVAL;
  s2dw_plan_t c = nullptr;
  const int rc = sht_child(p, &c);
  if (rc != S2DW_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ptrs.f[0] = flm;
  ptrs.Wphi[0] = fpix;
  if (c->fp64) run_analysis<double>(c->own, ptrs, st);
  else run_analysis<float>(c->own, ptrs, st);
  mark_use(c, st);
  return err_of(cudaGetLastError());
}

int s2dw_sht_forward(s2dw_plan_t p, const void* fpix, void* flm, void* stream) {
  if (!p || !flm || !fpix) return S2DW_EINVAL;
  s2dw_plan_t c = nullptr;
  const int rc = sht_child(p, &c);
  if (rc != S2DW_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ptrs.Wphi[0] = const_cast<void*>(fpix);
  ReduceJobs rj;
  std::memset(&rj, 0, sizeof(rj));
  rj.dw[0] = c->own.desc_w;
  rj.dp[0] = c->own.desc_phi;
  rj.out[0] = flm;
  rj.L[0] = c->L;
  rj.tmp[0] = c->TMP;
  rj.halves[0] = c->fp64 && c->direct_w ? 1 : 0;
  rj.lend[0] = c->lend_w;
  rj.Lphi[0] = c->Lphi;
  rj.sht[0] = 1;
  if (c->fp64) run_synthesis<double>(c->own, ptrs, rj, 1, st);
  else run_synthesis<float>(c->own, ptrs, rj, 1, st);
  mark_use(c, st);
  return err_of(cudaGetLastError());
}

int s2dw_scale_grid(s2dw_plan_t p, int j, int* Lgrid, int64_t* offset, int64_t* elems) {
  if (!p || j < 0 || j > p->nscale) return S2DW_EINVAL;
  const int64_t Lg = p->gt[p->grid_of[j]].L, nb = p->gt[p->grid_of[j]].nb;
  const int64_t per = (j == p->nscale ? 1 : p->N) * nb * (2 * Lg - 1);
  if (Lgrid) *Lgrid = (int)Lg;
  if (offset) *offset = (j == p->nscale) ? 0 : p->woff[j];
  if (elems) *elems = per;
  return S2DW_OK;
}

int s2dw_alpha_method(s2dw_plan_t p, int j, int dir, int* method, int* fft_len, int* segments, int* seg_len) {
  if (!p || j < 0 || j > p->nscale || dir < 0 || dir > 1) return S2DW_EINVAL;
  const auto& G = p->gt[p->grid_of[j]];
  const auto& sgt = p->seg[j];
  int m = p->alpha_mode[dir][j], len = G.M, ns = 1, sl = 2 * G.L - 1;
  if (m == 3) m = sgt.S > 0 ? 2 : 1;  // products: the transform in their place
  if (m == 0) {
    len = ns = sl = 0;
  } else if (m == 2) {
    len = 1 << sgt.logM;
    ns = sgt.S;
    sl = sgt.P;
  }
  if (method) *method = m;
  if (fft_len) *fft_len = len;
  if (segments) *segments = ns;
  if (seg_len) *seg_len = sl;
  return S2DW_OK;
}

// ---- launch methods and the autotuner -------------------------------------
static int choices_count(s2dw_plan_t p) { return 3 + 2 * (p->nscale + 1); }

// Whether method v is available for choice idx of the plan (layout of s2dw_plan_choices).
static bool choice_valid(s2dw_plan_t p, int idx, int v) {
  if (idx < 2) return v == 0 || v == 1;  // grids without half-length transforms keep the FFT
  if (idx == choices_count(p) - 1) {  // accepted for saved choices (FP32 plans with N <= 5 have three values)
    if (p->fp64) return v == 0;
    return pair_shapes_offered(p->N) ? (v >= kPairShapePair && v <= kPairShapeTile2) : v == kPairShapeTile;
  }
  const int j = (idx - 2) / 2, d = (idx - 2) % 2;
  const int Lj = p->Ycols[j];
  if (v == 0) return Lj <= (d == 0 ? kDirectMaxLjAna : kDirectMaxLj);  // direct kernels sized for L_j <= 32
  if (v == 1) return true;
  if (v == 2) return p->seg[j].S > 0;  // segment tables built at plan creation
  if (v == 3) return p->alpha_sg[d][j] != 0;  // basis tables built at plan creation
  return false;
}

static void choices_get(s2dw_plan_t p, int* c) {
  c[0] = p->beta_mode[0];
  c[1] = p->beta_mode[1];
  for (int j = 0; j <= p->nscale; ++j) {
    c[2 + 2 * j] = p->alpha_mode[0][j];
    c[3 + 2 * j] = p->alpha_mode[1][j];
  }
  c[choices_count(p) - 1] = p->fp64 ? 0 : p->pair_shape;
}

static void choices_put(s2dw_plan_t p, const int* c) {
  p->beta_mode[0] = c[0];
  p->beta_mode[1] = c[1];
  for (int j = 0; j <= p->nscale; ++j) {
    p->alpha_mode[0][j] = c[2 + 2 * j];
    p->alpha_mode[1][j] = c[3 + 2 * j];
  }
  if (!p->fp64) p->pair_shape = c[choices_count(p) - 1];
  drop_batches_with(p);
  if (p->fp64) own_lists_build<double>(p);
  else own_lists_build<float>(p);
}

int s2dw_plan_choices(s2dw_plan_t p, int* choices, int* n) {
  if (!p || !n) return S2DW_EINVAL;
  const int need = choices_count(p);
  if (!choices) {
    *n = need;
    return S2DW_OK;
  }
  if (*n < need) {
    *n = need;
    return S2DW_EINVAL;
  }
  choices_get(p, choices);
  *n = need;
  return S2DW_OK;
}

int s2dw_plan_set_choices(s2dw_plan_t p, const int* choices, int n) {
  if (!p || !choices || n != choices_count(p)) return S2DW_EINVAL;
  for (int i = 0; i < n; ++i)
    if (!choice_valid(p, i, choices[i])) return S2DW_EINVAL;
  try {
    ck(cudaEventSynchronize(p->last_use));  // this plan's calls so far (the lists are replaced)
    choices_put(p, choices);
    ck(cudaStreamSynchronize(p->pst));
  } catch (const CudaFail& e) {
    return err_of(e.err);
  } catch (...) {
    return S2DW_ECUDA;
  }
  return S2DW_OK;
}

int s2dw_plan_tune(s2dw_plan_t p, int reps, int* choices, int* n) {
  if (!p || reps < 1 || reps > 64 || (choices && !n)) return S2DW_EINVAL;
  const int nc = choices_count(p);
  if (choices && *n < nc) {
    *n = nc;
    return S2DW_EINVAL;
  }
  cudaStream_t st = p->pst;
  const size_t el = p->fp64 ? 8 : 4;
  int64_t wphi = 0;
  s2dw_query(p, nullptr, nullptr, &wphi, nullptr, nullptr);
  const size_t fbytes = (size_t)p->L * p->L * 2 * el;
  const size_t wbytes = ((size_t)p->woff[p->nscale] + (size_t)wphi) * el;
  void *f = nullptr, *fr = nullptr, *W = nullptr;
  constexpr int A = s2dw_plan_s::kEvAna, S = s2dw_plan_s::kEvSyn;
  cudaEvent_t ev[A + S] = {};
  std::vector<int> cur(nc), best(nc);
  try {
    ck(cudaEventSynchronize(p->last_use));
    amalloc(&f, fbytes, st);
    amalloc(&fr, fbytes, st);
    amalloc(&W, wbytes, st);
    // nonzero inputs: the analysis then writes W of the same kind for the synthesis
    if (p->fp64) ck(launch_fill_noise<double>(reinterpret_cast<double*>(f), (int64_t)(fbytes / 8), 0x5eedu, st));
    else ck(launch_fill_noise<float>(reinterpret_cast<float*>(f), (int64_t)(fbytes / 4), 0x5eedu, st));
    ck(cudaMemsetAsync(W, 0, wbytes, st));
    for (auto& e : ev) ck(cudaEventCreate(&e));
    CallPtrs ptrs;
    std::memset(&ptrs, 0, sizeof(ptrs));
    ptrs.f[0] = f;
    ptrs.out[0] = fr;
    ptrs.W[0] = W;
    ptrs.Wphi[0] = reinterpret_cast<char*>(W) + (size_t)p->woff[p->nscale] * el;
    // milliseconds of the beta launch and of the alpha launches of each
    // direction, the minimum over `reps` round trips
    auto measure = [&](double (&ms)[5]) {
      for (double& v : ms) v = 1e30;
      for (int r = 0; r < reps; ++r) {
        ReduceJobs rj;
        std::memset(&rj, 0, sizeof(rj));
        rj.dw[0] = p->own.desc_w;
        rj.dp[0] = p->own.desc_phi;
        rj.out[0] = fr;
        rj.L[0] = p->L;
        rj.tmp[0] = p->TMP;
        rj.halves[0] = p->fp64 && p->direct_w ? 1 : 0;
        rj.lend[0] = p->lend_w;
        rj.Lphi[0] = p->Lphi;
        if (p->fp64) {
          run_analysis<double>(p->own, ptrs, st, ev);
          run_synthesis<double>(p->own, ptrs, rj, 1, st, ev + A);
        } else {
          run_analysis<float>(p->own, ptrs, st, ev);
          run_synthesis<float>(p->own, ptrs, rj, 1, st, ev + A);
        }
        ck(cudaGetLastError());
        ck(cudaEventSynchronize(ev[A + S - 1]));
        float t[6] = {};
        ck(cudaEventElapsedTime(&t[0], ev[2], ev[3]));          // analysis beta
        ck(cudaEventElapsedTime(&t[1], ev[A + 3], ev[A + 4]));  // synthesis beta
        ck(cudaEventElapsedTime(&t[2], ev[3], ev[6]));          // analysis alpha (all launches)
        ck(cudaEventElapsedTime(&t[3], ev[A + 0], ev[A + 3]));  // synthesis alpha
        ck(cudaEventElapsedTime(&t[4], ev[0], ev[2]));          // analysis contractions
        ck(cudaEventElapsedTime(&t[5], ev[A + 4], ev[A + 6]));  // synthesis contractions
        t[4] += t[5];
        for (int i = 0; i < 5; ++i) ms[i] = std::min(ms[i], (double)t[i]);
      }
    };
    // the choices now in place beat the incumbent's time base[i] on stage i:
    // 3 % faster in a first measurement and again in a second one (the
    // incumbent re-measured between them), so that noise does not switch methods
    auto better = [&](double (&ms)[5], int i, double (&base)[5]) {
      measure(ms);
      if (!(ms[i] < 0.97 * base[i])) return false;
      std::vector<int> trial(nc);
      choices_get(p, trial.data());
      choices_put(p, cur.data());
      double again[5];
      measure(again);
      base[i] = std::min(base[i], again[i]);
      choices_put(p, trial.data());
      double ms2[5];
      measure(ms2);
      for (int k = 0; k < 5; ++k) ms[k] = std::min(ms[k], ms2[k]);
      return ms[i] < 0.97 * base[i];
    };
    choices_get(p, cur.data());
    double base[5];
    choices_put(p, cur.data());
    measure(base);  // warms up as well
    measure(base);
    // coordinate descent: the beta method of each direction, then each
    // scale's alpha method (largest band first) against its direction's total
    for (int d = 0; d < 2; ++d) {
      for (int v = 0; v < 2; ++v) {
        if (v == cur[d] || !choice_valid(p, d, v)) continue;
        std::vector<int> trial(cur);
        trial[d] = v;
        choices_put(p, trial.data());
        double ms[5];
        if (better(ms, d, base)) {
          cur = trial;
          base[d] = ms[d];
        }
      }
    }
    choices_put(p, cur.data());
    measure(base);
    std::vector<int> order(p->nscale + 1);
    for (int j = 0; j <= p->nscale; ++j) order[j] = j;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return p->Ycols[a] > p->Ycols[b]; });
    for (int d = 0; d < 2; ++d)
      for (int j : order) {
        const int idx = 2 + 2 * j + d;
        for (int v = 0; v < 4; ++v) {
          if (v == cur[idx] || !choice_valid(p, idx, v) || p->Ycols[j] <= 0) continue;
          std::vector<int> trial(cur);
          trial[idx] = v;
          choices_put(p, trial.data());
          double ms[5];
          if (better(ms, 2 + d, base)) {
            cur = trial;
            base[2 + d] = ms[2 + d];
          }
        }
      }
    choices_put(p, cur.data());
    ck(cudaStreamSynchronize(st));
  } catch (const CudaFail& e) {
    cudaStreamSynchronize(st);
    for (auto& e2 : ev) if (e2) cudaEventDestroy(e2);
    afree(f, st);
    afree(fr, st);
    afree(W, st);
    return err_of(e.err);
  } catch (...) {
    cudaStreamSynchronize(st);
    for (auto& e2 : ev) if (e2) cudaEventDestroy(e2);
    afree(f, st);
    afree(fr, st);
    afree(W, st);
    return S2DW_ECUDA;
  }
  for (auto& e : ev) cudaEventDestroy(e);
  afree(f, st);
  afree(fr, st);
  afree(W, st);
  cudaStreamSynchronize(st);
  if (choices) {
    choices_get(p, choices);
    *n = nc;
  }
  return S2DW_OK;
}

int s2dw_wait_timeouts(int* count) {
  if (!count) return S2DW_EINVAL;
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return err_of(e);
  e = alpha_tc_timeouts(count);
  if (e != cudaSuccess) return err_of(e);
  int pc = 0;
  e = pair_timeouts(&pc);
  if (e != cudaSuccess) return err_of(e);
  *count += pc;
  e = split_gemm_timeouts(&pc);
  if (e != cudaSuccess) return err_of(e);
  *count += pc;
  return *count > 0 ? S2DW_ETIMEOUT : S2DW_OK;
}

int s2dw_wait_probe(long long limit_cycles, void* stream) {
  const long long lim = std::min(std::max(limit_cycles, 1000LL), 2000000000LL);
  return err_of(alpha_tc_wait_probe(lim, reinterpret_cast<cudaStream_t>(stream)));
}

int s2dw_plan_wait_probe(s2dw_plan_t p, long long limit_cycles, void* stream) {
  if (!p) return S2DW_EINVAL;
  if (p->fp64) return S2DW_ENOTSUP;
  const long long lim = std::min(std::max(limit_cycles, 0LL), kWaitLimit);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int64_t wphi = 0;
  s2dw_query(p, nullptr, nullptr, &wphi, nullptr, nullptr);
  const size_t wbytes = ((size_t)p->woff[p->nscale] + (size_t)wphi) * sizeof(float);
  void* W = nullptr;  // scratch: the alpha sums' W and W^Phi
  if (cudaError_t e = cudaMallocAsync(&W, wbytes, st); e != cudaSuccess) return err_of(e);
  cudaMemsetAsync(W, 0, wbytes, st);
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ptrs.W[0] = W;
  ptrs.Wphi[0] = reinterpret_cast<float*>(W) + p->woff[p->nscale];
  const Lists& ls = p->own;
  const ContractDesc<float>* dw = reinterpret_cast<const ContractDesc<float>*>(ls.desc_w);
  const ContractDesc<float>* dp = reinterpret_cast<const ContractDesc<float>*>(ls.desc_phi);
  auto contract = [&](bool syn) {
    for (auto& g : ls.tile_w)
      launch_contract_tile(g.N, 2, syn, dw, reinterpret_cast<const CTask*>(g.task[syn]), g.n[syn], st, lim);
    launch_contract_tile(1, 1, syn, dp, reinterpret_cast<const CTask*>(ls.tile_phi.task[syn]), ls.tile_phi.n[syn], st, lim);
  };
  auto direct = [&](bool syn) {
    const int k = syn ? CZT_ALPHA_SYN_DIRECT : CZT_ALPHA_ANA_DIRECT;
    launch_alpha_tc(syn, reinterpret_cast<const CztSeg<float>*>(ls.segs[k]), ls.nseg[k], ls.items[k], ptrs, st, lim);
  };
  contract(false);
  launch_products<float>(ls, SG_KIND_BETA_ANA, ptrs, st, lim);
  launch_products<float>(ls, SG_KIND_ALPHA_ANA, ptrs, st, lim);
  direct(false);
  direct(true);
  launch_products<float>(ls, SG_KIND_ALPHA_SYN, ptrs, st, lim);
  launch_products<float>(ls, SG_KIND_BETA_RS, ptrs, st, lim);
  launch_products<float>(ls, SG_KIND_BETA_SYN, ptrs, st, lim);
  contract(true);
  cudaFreeAsync(W, st);
  mark_use(p, st);
  return err_of(cudaGetLastError());
}

int s2dw_launch_counts(s2dw_plan_t p, int* analysis, int* synthesis) {
  if (!p) return S2DW_EINVAL;
  const Lists& ls = p->own;
  int contract = (ls.ntiles_phi > 0 ? 1 : 0) + direct_groups(ls) + (ls.tile_phi.n[0] > 0 ? 1 : 0);
  for (auto& g : ls.tile_w) contract += g.n[0] > 0 ? 1 : 0;
  for (auto& t : ls.tiles_w) contract += t.second.second > 0 ? 1 : 0;
  auto has = [&](int k) {
    if (k >= CZT_BETA_ANA_DCT && k <= CZT_BETA_RS_DCT) return (int)ls.dct_parts[k - CZT_BETA_ANA_DCT].size();
    return ls.items[k] > 0 ? 1 : 0;
  };
  const int fpack = (!p->fp64 && ls.njobs > 0 && ls.nbmax > 0) ? 1 : 0;  // f packing of the FP32 contraction
  if (analysis) *analysis = fpack + contract + has(0) + has(1) + has(4) + has(6) + has(8) + has(13) + 2 * (has(16) + has(18));
  if (synthesis)
    *synthesis = contract + has(2) + has(3) + has(5) + has(7) + has(9) + has(10) + has(11) + has(12) + has(14) +
                 has(15) + 2 * (has(17) + has(19) + has(20)) + 1;
  return S2DW_OK;
}

int s2dw_kernels(s2dw_plan_t p, double* psi, double* phi) {
  if (!p) return S2DW_EINVAL;
  if (psi) std::memcpy(psi, p->psi_host.data(), p->psi_host.size() * sizeof(double));
  if (phi) std::memcpy(phi, p->phi_host.data(), p->phi_host.size() * sizeof(double));
  return S2DW_OK;
}

int s2dw_analysis(s2dw_plan_t p, const void* flm, void* W, void* Wphi, void* stream) {
  if (!p || !flm || !W || !Wphi) return S2DW_EINVAL;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ptrs.f[0] = flm;
  ptrs.W[0] = W;
  ptrs.Wphi[0] = Wphi;
  cudaEvent_t* ev = nullptr;
  if (p->prof && p->nana < s2dw_plan_s::kProfCalls && !capturing(st))
    ev = p->ev_ana.data() + s2dw_plan_s::kEvAna * (p->nana++);
  if (p->fp64) run_analysis<double>(p->own, ptrs, st, ev);
  else run_analysis<float>(p->own, ptrs, st, ev);
  mark_use(p, st);
  return err_of(cudaGetLastError());
}

int s2dw_synthesis(s2dw_plan_t p, const void* W, const void* Wphi, void* flm, void* stream) {
  if (!p || !flm || !W || !Wphi) return S2DW_EINVAL;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ptrs.out[0] = flm;
  ptrs.W[0] = const_cast<void*>(W);
  ptrs.Wphi[0] = const_cast<void*>(Wphi);
  ReduceJobs rj;
  std::memset(&rj, 0, sizeof(rj));
  rj.dw[0] = p->own.desc_w;
  rj.dp[0] = p->own.desc_phi;
  rj.out[0] = flm;
  rj.L[0] = p->L;
  rj.tmp[0] = p->TMP;
  rj.halves[0] = p->fp64 && p->direct_w ? 1 : 0;
  rj.lend[0] = p->lend_w;
  rj.Lphi[0] = p->Lphi;
  cudaEvent_t* ev = nullptr;
  if (p->prof && p->nsyn < s2dw_plan_s::kProfCalls && !capturing(st))
    ev = p->ev_syn.data() + s2dw_plan_s::kEvSyn * (p->nsyn++);
  if (p->fp64) run_synthesis<double>(p->own, ptrs, rj, 1, st, ev);
  else run_synthesis<float>(p->own, ptrs, rj, 1, st, ev);
  mark_use(p, st);
  return err_of(cudaGetLastError());
}

int s2dw_profile(s2dw_plan_t p, int enable) {
  if (!p) return S2DW_EINVAL;
  if (enable && p->ev_ana.empty()) {
    p->ev_ana.assign(s2dw_plan_s::kEvAna * s2dw_plan_s::kProfCalls, nullptr);
    p->ev_syn.assign(s2dw_plan_s::kEvSyn * s2dw_plan_s::kProfCalls, nullptr);
    for (auto& e : p->ev_ana)
      if (cudaEventCreate(&e) != cudaSuccess) return S2DW_ECUDA;
    for (auto& e : p->ev_syn)
      if (cudaEventCreate(&e) != cudaSuccess) return S2DW_ECUDA;
  }
  p->prof = enable != 0;
  p->nana = 0;
  p->nsyn = 0;
  return S2DW_OK;
}

int s2dw_profile_read(s2dw_plan_t p, double* ms, int* ncalls) {
  if (!p || !ms) return S2DW_EINVAL;
  constexpr int A = s2dw_plan_s::kEvAna, S = s2dw_plan_s::kEvSyn;
  for (int i = 0; i < A + S - 2; ++i) ms[i] = 0.0;
  if (ncalls) ncalls[0] = ncalls[1] = 0;
  if (p->ev_ana.empty()) return S2DW_OK;
  cudaError_t e = cudaSuccess;
  int na = 0, ns = 0;
  for (int c = 0; c < p->nana; ++c) {
    cudaEvent_t* ev = p->ev_ana.data() + A * c;
    if ((e = cudaEventSynchronize(ev[A - 1])) != cudaSuccess) return err_of(e);
    for (int i = 0; i < A - 1; ++i) {
      float t = 0.f;
      if ((e = cudaEventElapsedTime(&t, ev[i], ev[i + 1])) != cudaSuccess) return err_of(e);
      ms[i] += t;
    }
    ++na;
  }
  for (int c = 0; c < p->nsyn; ++c) {
    cudaEvent_t* ev = p->ev_syn.data() + S * c;
    if ((e = cudaEventSynchronize(ev[S - 1])) != cudaSuccess) return err_of(e);
    for (int i = 0; i < S - 1; ++i) {
      float t = 0.f;
      if ((e = cudaEventElapsedTime(&t, ev[i], ev[i + 1])) != cudaSuccess) return err_of(e);
      ms[A - 1 + i] += t;
    }
    ++ns;
  }
  if (ncalls) {
    ncalls[0] = na;
    ncalls[1] = ns;
  }
  return S2DW_OK;
}

// Looks up (or builds) the launch lists of a plan set; g_batch_mu must be held
// by the caller until the launches using the entry are queued and recorded.
static int batch_lists(const s2dw_plan_t* plans, int njobs, BatchEnt** out, bool* fp64) {
  if (!plans || njobs < 1 || njobs > MAXB) return S2DW_EINVAL;
  std::vector<s2dw_plan_t> key(plans, plans + njobs);
  for (int i = 0; i < njobs; ++i) {
    if (!key[i]) return S2DW_EINVAL;
    for (int k = 0; k < i; ++k)
      if (key[k] == key[i]) return S2DW_EINVAL;
    if (key[i]->fp64 != key[0]->fp64) return S2DW_ENOTSUP;
  }
  *fp64 = key[0]->fp64;
  auto it = g_batch_cache.find(key);
  if (it == g_batch_cache.end()) {
    evict_batches();
    BatchEnt e;
    try {
      e.ls = *fp64 ? build_lists<double>(key) : build_lists<float>(key);
    } catch (const CudaFail& err) {
      return err_of(err.err);
    } catch (...) {
      return S2DW_ENOMEM;
    }
    if (cudaEventCreateWithFlags(&e.done, cudaEventDisableTiming) != cudaSuccess) {
      delete e.ls;
      return S2DW_ECUDA;
    }
    it = g_batch_cache.emplace(key, e).first;
  }
  it->second.tick = ++g_batch_tick;
  *out = &it->second;
  return S2DW_OK;
}

static void batch_used(BatchEnt* e, cudaStream_t st) {
  if (capturing(st)) e->pinned = true;
  else cudaEventRecord(e->done, st);
}

int s2dw_analysis_batch(const s2dw_plan_t* plans, const void* const* flm, void* const* W, void* const* Wphi,
                        int njobs, void* stream) {
  if (!flm || !W || !Wphi) return S2DW_EINVAL;
  std::lock_guard<std::mutex> lk(g_batch_mu);
  BatchEnt* be = nullptr;
  bool fp64 = false;
  int rc = batch_lists(plans, njobs, &be, &fp64);
  if (rc != S2DW_OK) return rc;
  const Lists* ls = be->ls;
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  for (int i = 0; i < njobs; ++i) {
    if (!flm[i] || !W[i] || !Wphi[i]) return S2DW_EINVAL;
    ptrs.f[i] = flm[i];
    ptrs.W[i] = W[i];
    ptrs.Wphi[i] = Wphi[i];
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (fp64) run_analysis<double>(*ls, ptrs, st);
  else run_analysis<float>(*ls, ptrs, st);
  batch_used(be, st);
  for (int i = 0; i < njobs; ++i) mark_use(plans[i], st);
  return err_of(cudaGetLastError());
}

int s2dw_synthesis_batch(const s2dw_plan_t* plans, const void* const* W, const void* const* Wphi, void* const* flm,
                         int njobs, void* stream) {
  if (!flm || !W || !Wphi) return S2DW_EINVAL;
  std::lock_guard<std::mutex> lk(g_batch_mu);
  BatchEnt* be = nullptr;
  bool fp64 = false;
  int rc = batch_lists(plans, njobs, &be, &fp64);
  if (rc != S2DW_OK) return rc;
  const Lists* ls = be->ls;
  CallPtrs ptrs;
  std::memset(&ptrs, 0, sizeof(ptrs));
  ReduceJobs rj;
  std::memset(&rj, 0, sizeof(rj));
  const size_t dsz = fp64 ? sizeof(ContractDesc<double>) : sizeof(ContractDesc<float>);
  for (int i = 0; i < njobs; ++i) {
    if (!flm[i] || !W[i] || !Wphi[i]) return S2DW_EINVAL;
    ptrs.out[i] = flm[i];
    ptrs.W[i] = const_cast<void*>(W[i]);
    ptrs.Wphi[i] = const_cast<void*>(Wphi[i]);
    rj.dw[i] = reinterpret_cast<const char*>(ls->desc_w) + i * dsz;
    rj.dp[i] = reinterpret_cast<const char*>(ls->desc_phi) + i * dsz;
    rj.out[i] = flm[i];
    rj.L[i] = plans[i]->L;
    rj.tmp[i] = plans[i]->TMP;
    rj.halves[i] = plans[i]->fp64 && plans[i]->direct_w ? 1 : 0;
    rj.lend[i] = plans[i]->lend_w;
    rj.Lphi[i] = plans[i]->Lphi;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (fp64) run_synthesis<double>(*ls, ptrs, rj, njobs, st);
  else run_synthesis<float>(*ls, ptrs, rj, njobs, st);
  batch_used(be, st);
  for (int i = 0; i < njobs; ++i) mark_use(plans[i], st);
  return err_of(cudaGetLastError());
}

int s2dw_scale_support(s2dw_plan_t p, int j, int* lo, int* hi) {
  if (!p || j < 0 || j > p->nscale) return S2DW_EINVAL;
  if (j == p->nscale) {
    if (lo) *lo = 0;
    if (hi) *hi = p->lphi;
  } else {
    if (lo) *lo = p->lo[j];
    if (hi) *hi = p->hi[j];
  }
  return S2DW_OK;
}

int s2dw_delta_slab(s2dw_plan_t p, int l, double* host_out) {
  if (!p || !host_out || l < 0 || l >= p->L) return S2DW_EINVAL;
  const int64_t sz = delta_slab_size(l);
  std::vector<double> slab(sz);
  cudaError_t e = cudaMemcpy(slab.data(), p->tab->d64 + delta_slab_offset(l), sz * sizeof(double),
                             cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return err_of(e);
  for (int mp = 0; mp <= l; ++mp)
    for (int m = 0; m <= l; ++m) {
      double v;
      if (m >= 4 * (mp >> 2)) v = slab[delta_entry(l, mp, m)];
      else v = (((mp - m) & 1) ? -1.0 : 1.0) * slab[delta_entry(l, m, mp)];
      host_out[(size_t)mp * (l + 1) + m] = v;
    }
  return S2DW_OK;
}

int s2dw_stage(s2dw_plan_t p, int stage, int j, void* host_out, int64_t* nbytes) {
  if (!p || j < 0 || j > p->nscale || stage < 0 || stage > 1) return S2DW_EINVAL;
  const int Nj = (j == p->nscale) ? 1 : p->N;
  const int Lj = p->Ycols[j];
  const int64_t el = p->fp64 ? 16 : 8;
  const int64_t Lg = p->gt[p->grid_of[j]].L;  // the scale's beta grid
  const int64_t bytes = (stage == 0 ? (int64_t)Nj * Lj * Lj : (int64_t)Nj * 2 * Lg * Lj) * el;
  if (nbytes) *nbytes = bytes;
  if (!host_out) return S2DW_OK;
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return err_of(e);
  e = cudaMemcpy(host_out, stage == 0 ? p->Y[j] : p->X[j], bytes, cudaMemcpyDeviceToHost);
  return err_of(e);
}

}  // extern "C"
