// Direct alpha sums of the small-band scales on the tensor cores (FP32 plans).
//
// Analysis (Eq. (30)), per row (g, b) of X_g[b][m] (m < L_j, complex, stored
// as 2 L_j floats x_k = (Re X_0, Im X_0, Re X_1, ...)):
//   W[row][a] = Re X_0 + 2 sum_{m>=1} Re(X_m e^{i m alpha_a}) = sum_k x_k B[a][k],
//   B[a][2m] = c_m cos(m alpha_a), B[a][2m+1] = -c_m sin(m alpha_a), c_0 = 1, c_m = 2,
// a matrix product with K = 2 L_j <= 64.  Tile: D[a (128)][row (128)] =
// B[a][k] x[row][k]^T in TMEM, so that a warp's TMEM load gives 32
// consecutive samples a of each row and every store is one 128-byte line.
// Synthesis (Eq. (37)): V[row][m] = (2 pi/n) sum_{a<n} W[row][a] e^{-i m alpha_a},
// the product D[row (128)][j (2 L_j, padded)] = W[row][a] C[j][a]^T with
// C[2m][a] = (2 pi/n) cos(m alpha_a), C[2m+1][a] = -(2 pi/n) sin(m alpha_a),
// K = n streamed from HBM in chunks of 32 samples.
//
// FP32 accuracy from TF32 MMAs by the three-product split of tc.cuh.  The
// basis operands are built once per plan, already split and laid out as the
// shared-memory images the MMAs read (tc::img_off), and copied with cp.async;
// the X and W operands are split by the threads on their way to shared memory.
#include "czt.cuh"
#include "tc.cuh"

namespace s2dw {

__device__ int g_tc_timeouts;  // bounded waits that gave up (read and reset by the host)

namespace {

constexpr int kTcA = 128;       // analysis: samples a per tile (MMA M)
constexpr int kTcRows = 128;    // analysis: rows per tile (MMA N)
constexpr int kAnaProd = 8;     // analysis: producer warps
constexpr int kAnaEpi = 8;      // analysis: epilogue warps
// analysis: a CTA takes 2048 rows of a scale, halved down to one row tile while
// the scale has fewer CTAs than this over the jobs of the launch (a launch
// holds about five scales; a CTA starts with its 64 KB basis image).  1024 rows
// always -> at least 40 / 64 / 160 CTAs, us: L = 128, N = 5 32 -> 11 / 11 / 11;
// L = 361, N = 4 27 -> 15 / 15 / 19; L = 512, N = 3 34 -> 29 / 33 / 39; L = 1024,
// N = 5 125 -> 123 / 123 / 126; L = 2048, N = 8 707 -> 678 / 677 / 663.
constexpr int kTcAnaCtas = 40;
constexpr int kTcAnaThreads = (kAnaProd + kAnaEpi) * 32;
constexpr int kTcM = 128;       // synthesis: rows per CTA (MMA M)
constexpr int kTcKc = 32;       // synthesis: samples per K chunk
constexpr int kSynStages = 3;   // synthesis: shared-memory ring stages

// The shared-memory and TMEM budgets below hold for K8 <= 64 and NP <= 64.
static_assert(kDirectMaxLjAna <= 32 && kDirectMaxLj <= 32, "tensor-core direct alpha sums sized for L_j <= 32");

__host__ __device__ constexpr int ana_k8(int Lj) { return (2 * Lj + 7) & ~7; }
__host__ __device__ constexpr int syn_npad(int Lj) { return 2 * Lj <= 16 ? 16 : (2 * Lj + 15) & ~15; }

__device__ __forceinline__ void cp16(float* sdst, const float* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(sdst)), "l"(gsrc) : "memory");
}

// smem bytes of the analysis kernel for K8 = 64: basis image (hi, lo) and two
// stages of the row image (hi, lo)
constexpr size_t ana_tc_smem() { return (size_t)(2 + 4) * tc::img_floats(kTcRows, 64) * sizeof(float); }
// smem bytes of the synthesis kernel for Npad = 64: three ring stages of
// (W image, basis image) x (hi, lo)
constexpr size_t syn_tc_smem() {
  return (size_t)kSynStages * 2 * (tc::img_floats(kTcM, kTcKc) + tc::img_floats(64, kTcKc)) * sizeof(float);
}

// Analysis, warp-specialised (one CTA of 128 samples x up to 2048 rows per SM):
//   warps 0-7   producers: rows of X (registers, two row tiles ahead) split
//               into the row image of stage i % 2; arrive on full[stage];
//               thread 0 then waits full[stage] and tempty[stage], issues the
//               MMAs and commits to empty[stage] and tfull[stage] (a warp of its
//               own would cap the registers at 96: spills)
//   warps 8-15  epilogue: wait tfull[stage], read the sums (TMEM lanes =
//               samples, half the rows per warp), arrive on tempty[stage] and
//               store, every store one 128-byte run of a row of W
// What bounds it: the stores of W.  With every warp staging, then storing (one
// barrier per row tile) the store path idled while X was staged and the warps
// queued for it afterwards; the roles keep both going.  Measured (scales of band
// <= 32, with the rows per CTA of kTcAnaCtas, us, before -> now): L = 128, N = 5 31
// -> 11, L = 361, N = 4 26 -> 15, L = 1024, N = 5 (503 MB of W) 144 -> 123, L = 2048,
// N = 8 784 -> 678.
// Every wait is bounded and a timeout in any role stops all of them.
// PROBE: waits of wait_limit cycles (s2dw_plan_wait_probe); a run-time limit in the
// kernels themselves costs them 1%.
template <bool PROBE>
__global__ void __launch_bounds__(kTcAnaThreads, 1) k_alpha_ana_tc(const CztSeg<float>* __restrict__ segs,
                                                                   int nseg, CallPtrs ptrs, long long wait_limit) {
  begin_after();
  const long long limit = PROBE ? wait_limit : tc::kWaitCycles;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar[8];  // full[2], empty[2], tfull[2], tempty[2]
  __shared__ uint32_t tbase;
  __shared__ volatile int fail;
  __shared__ int issued;  // last row tile whose MMAs were issued, -1: none
  const CztSeg<float> sg = segs[czt_find_seg<float>(segs, nseg)];
  const int item = blockIdx.x - sg.start;
  const int Lj = sg.Lj, n = 2 * sg.L - 1, K8 = ana_k8(Lj);
  const int ntile = (n + kTcA - 1) / kTcA;
  const int ta = item % ntile, a0 = ta * kTcA;
  const int nrows = sg.N * sg.nb, rbeg = (item / ntile) * sg.P, rend = min(nrows, rbeg + sg.P);
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  float* __restrict__ Wb = reinterpret_cast<float*>(sg.is_phi ? ptrs.Wphi[sg.job] : ptrs.W[sg.job]) + sg.woff;
  if (Lj <= 0) {  // empty scale: W = 0
    for (int r = rbeg; r < rend; ++r)
      for (int c = t; c < kTcA; c += blockDim.x)
        if (a0 + c < n) Wb[(size_t)r * n + a0 + c] = 0.f;
    return;
  }
  const int img = tc::img_floats(kTcRows, K8);  // = img_floats(kTcA, K8)
  float* Ahi = reinterpret_cast<float*>(smem_raw);
  float* Alo = Ahi + img;
  float* Bimg = Alo + img;  // [stage][hi, lo][img]
  auto full = [&](int b) { return tc::smem_u32(&bar[b]); };
  auto empty = [&](int b) { return tc::smem_u32(&bar[2 + b]); };
  auto tfull = [&](int b) { return tc::smem_u32(&bar[4 + b]); };
  auto tempty = [&](int b) { return tc::smem_u32(&bar[6 + b]); };
  if (t == 0) {
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(full(b), kAnaProd * 32);
      tc::mbar_init(empty(b), 1);
      tc::mbar_init(tfull(b), 1);
      tc::mbar_init(tempty(b), kAnaEpi);
    }
    fail = 0;
  }
  // TMEM: the sums of stage s at column 128 s
  if (w == 0) tc::tmem_alloc(&tbase, 2 * kTcRows);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tbase;
  const int ntr = (rend - rbeg + kTcRows - 1) / kTcRows;  // row tiles of this CTA
  if (w < kAnaProd) {
    // basis image of this sample tile (built per plan, already split)
    const float* src = reinterpret_cast<const float*>(sg.H) + (size_t)ta * 2 * img;
    for (int i = 4 * t; i < 2 * img; i += 4 * kAnaProd * 32) cp16(Ahi + i, src + i);
    asm volatile("cp.async.commit_group;" ::: "memory");
    // thread t holds X_m, m = t % KP, of rows rl0 + q RS of a row tile (KP = K8 / 2
    // rounded up to a power of two, RS = 256 / KP >= 8 rows), so the image
    // offset is linear in q and a warp reads consecutive m of a row
    const int lk = K8 <= 8 ? 2 : (K8 <= 16 ? 3 : (K8 <= 32 ? 4 : 5));
    const int m = t & ((1 << lk) - 1), rl0 = t >> lk, RS = (kAnaProd * 32) >> lk, NQ = kTcRows / RS;
    const bool kin = m < Lj, kst = 2 * m < K8;
    const int o0 = kst ? tc::img_off(rl0, 2 * m, K8) : 0, oq = (RS / 8) * (K8 / 4) * tc::kLboF;
    const float2* __restrict__ X = sg.buf_in;
    const size_t rsk = (size_t)RS * Lj;  // values between the rows q and q + 1 of a thread
    auto load = [&](int i, float2 (&xr)[16]) {  // NQ <= 16
      const int r = rbeg + i * kTcRows + rl0;
      const float2* p = X + (size_t)r * Lj + m;
      const int qn = kin ? (rend - r + RS - 1) / RS : 0;  // rows r + q RS < rend exist
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        if (q < NQ) xr[q] = q < qn ? __ldg(p) : make_float2(0.f, 0.f);
        p += rsk;
      }
    };
    int last = -1;  // thread 0: last row tile whose MMAs were issued
    auto issue = [&](int i) {
      const int s = i & 1;
      if (!tc::mbar_wait(full(s), (uint32_t)(i >> 1) & 1u, limit) ||
          (i >= 2 && !tc::mbar_wait(tempty(s), (uint32_t)((i >> 1) - 1) & 1u, limit))) {
        fail = 1;
        return;
      }
      tc::fence_after();
      // D = (A_hi B_lo + A_lo B_hi) + A_hi B_hi, cross terms first
      const uint32_t idesc = tc::idesc_tf32(kTcA, kTcRows), d = tmem + (uint32_t)(s * kTcRows);
      const uint64_t kstep = (uint64_t)(tc::img_kstep_bytes(1) >> 4);  // start-address field per K-step
      const uint64_t aH = tc::smem_desc(tc::smem_u32(Ahi), K8), aL = tc::smem_desc(tc::smem_u32(Alo), K8);
      const uint64_t bH = tc::smem_desc(tc::smem_u32(Bimg + (size_t)s * 2 * img), K8);
      const uint64_t bL = tc::smem_desc(tc::smem_u32(Bimg + (size_t)s * 2 * img + img), K8);
      for (int k = 0; k < K8 / 8; ++k) {
        const uint64_t o = kstep * k;
        tc::mma_tf32(d, aH + o, bL + o, idesc, k > 0);
        tc::mma_tf32(d, aL + o, bH + o, idesc, 1);
      }
      for (int k = 0; k < K8 / 8; ++k) {
        const uint64_t o = kstep * k;
        tc::mma_tf32(d, aH + o, bH + o, idesc, 1);
      }
      tc::mma_commit(empty(s));
      tc::mma_commit(tfull(s));
      last = i;
    };
    auto step = [&](int i, float2 (&xr)[16]) -> bool {
      const int s = i & 1;
      if (fail) return false;
      if (i >= 2 && !tc::mbar_wait(empty(s), (uint32_t)((i >> 1) - 1) & 1u, limit)) {
        fail = 1;
        return false;
      }
      float* hi = Bimg + (size_t)s * 2 * img + o0;
      float* lo = hi + img;
      if (kst) {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          if (q < NQ) {
            float2 h, l;
            tc::split_tf32(xr[q].x, h.x, l.x);
            tc::split_tf32(xr[q].y, h.y, l.y);
            *reinterpret_cast<float2*>(hi + q * oq) = h;
            *reinterpret_cast<float2*>(lo + q * oq) = l;
          }
        }
      }
      if (i + 2 < ntr) load(i + 2, xr);
      if (i == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
      tc::fence_async_smem();
      tc::mbar_arrive(full(s));
      if (t == 0) issue(i);
      return true;
    };
    float2 xa[16], xb[16];
    load(0, xa);
    if (ntr > 1) load(1, xb);
    for (int i = 0; i < ntr; i += 2) {
      if (!step(i, xa)) break;
      if (i + 1 < ntr && !step(i + 1, xb)) break;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (t == 0) issued = last;
  } else {
    // samples a0 + 32 (w % 4) + lane, rows 64 h .. 64 h + 63 of a tile
    const int a = a0 + 32 * (w & 3) + lane, cg = 64 * ((w - kAnaProd) >> 2);
    for (int i = 0; i < ntr; ++i) {
      const int s = i & 1;
      const bool got = !fail && tc::mbar_wait(tfull(s), (uint32_t)(i >> 1) & 1u, limit);
      if (!__all_sync(0xffffffffu, got)) {  // warp-uniform: the TMEM loads below are warp-collective
        fail = 1;
        break;
      }
      tc::fence_after();
      const uint32_t te = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(s * kTcRows + cg);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[32];
        tc::tmem_ld32(te + 32 * h, v);
        if (h == 1) {
          tc::fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(tempty(s));
        }
        // row j at q + j n: the pointer advances by one row per store, and a
        // full group of 32 rows (all but the last tile) needs no row test
        const int r0 = rbeg + i * kTcRows + cg + 32 * h, jn = rend - r0;
        if (a < n && jn > 0) {
          float* q = Wb + (size_t)r0 * n + a;
          if (jn >= 32) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              __stcs(q, v[j]);  // written once: streaming
              q += n;
            }
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              if (j < jn) __stcs(q, v[j]);
              q += n;
            }
          }
        }
      }
    }
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  if (w == 0) {
    // after a give-up, whichever role's it was: a bounded wait for the MMAs in flight before TMEM is released
    if (t == 0 && fail) {
      if (issued >= 0) tc::mbar_wait(tfull(issued & 1), (uint32_t)(issued >> 1) & 1u, tc::kWaitCycles);
      atomicAdd(&g_tc_timeouts, 1);
    }
    __syncwarp();
    tc::tmem_free(tmem, 2 * kTcRows);
  }
}

// Synthesis, warp-specialised (one CTA of 128 rows per SM):
//   warps 0-7   producers: W chunk c (registers, two chunks ahead) split into
//               the A image of ring stage c % 3, the basis chunk copied into
//               its B image (cp.async, one chunk ahead); arrive on full[stage]
//   warp  16    MMA issuer (one thread): waits full[stage] and tempty[buffer],
//               12 MMAs into TMEM buffer c % 2, commits to empty[stage] and
//               tfull[buffer]
//   warps 8-15  accumulators: wait tfull[buffer], add the chunk's sums (TMEM
//               lanes = rows, half the columns per warp, one TMEM wait per
//               chunk) to FP32 registers, arrive on tempty[buffer]; finally
//               write V
// No CTA-wide barrier inside the K loop; every wait is bounded and a timeout
// in any role stops all of them.
constexpr int kSynProd = 8;                          // producer warps
constexpr int kSynAcc = 8;                            // accumulator warps
constexpr int kSynThreads = (kSynProd + kSynAcc + 1) * 32;  // + the MMA warp

template <bool PROBE>
__global__ void __launch_bounds__(kSynThreads, 1) k_alpha_syn_tc(const CztSeg<float>* __restrict__ segs, int nseg,
                                                                 CallPtrs ptrs, long long wait_limit) {
  begin_after();
  const long long limit = PROBE ? wait_limit : tc::kWaitCycles;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar[2 * kSynStages + 4];  // full[S], empty[S], tfull[2], tempty[2]
  __shared__ uint32_t tbase;
  __shared__ volatile int fail;
  __shared__ int issued;  // last chunk whose MMAs were issued, -1: none
  const CztSeg<float> sg = segs[czt_find_seg<float>(segs, nseg)];
  const int item = blockIdx.x - sg.start;
  const int Lj = sg.Lj, n = 2 * sg.L - 1, NP = syn_npad(Lj);
  const int nrows = sg.N * sg.nb, r0 = item * kTcM, nr = min(kTcM, nrows - r0);
  const int nchunk = (n + kTcKc - 1) / kTcKc;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const float* __restrict__ Wb =
      reinterpret_cast<const float*>(sg.is_phi ? ptrs.Wphi[sg.job] : ptrs.W[sg.job]) + sg.woff + (size_t)r0 * n;
  cx<float>* __restrict__ V = sg.buf_out + (size_t)r0 * Lj;
  if (Lj <= 0) return;
  const int imgA = tc::img_floats(kTcM, kTcKc), imgB = tc::img_floats(NP, kTcKc);
  const int stage = 2 * (imgA + imgB);  // floats: A hi, A lo, B hi, B lo
  float* base = reinterpret_cast<float*>(smem_raw);
  // TMEM buffer b (chunk parity): the chunk's sums at column NP b
  const int ncols = 2 * NP <= 32 ? 32 : (2 * NP <= 64 ? 64 : 128);
  auto full = [&](int i) { return tc::smem_u32(&bar[i]); };
  auto empty = [&](int i) { return tc::smem_u32(&bar[kSynStages + i]); };
  auto tfull = [&](int b) { return tc::smem_u32(&bar[2 * kSynStages + b]); };
  auto tempty = [&](int b) { return tc::smem_u32(&bar[2 * kSynStages + 2 + b]); };
  if (t == 0) {
    for (int i = 0; i < kSynStages; ++i) {
      tc::mbar_init(full(i), kSynProd * 32);
      tc::mbar_init(empty(i), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(tfull(b), 1);
      tc::mbar_init(tempty(b), kSynAcc * 32);
    }
    fail = 0;
  }
  if (w == kSynProd) tc::tmem_alloc(&tbase, ncols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tbase;
  int last = -1;  // MMA thread: last chunk whose MMAs were issued
  if (w < kSynProd) {
    // ---- producers: rows w + 8 q (q < 16), samples 32 c + lane ----
    const float* __restrict__ basis = reinterpret_cast<const float*>(sg.H);  // [chunk][B hi, B lo]
    // row w + 8 q at wrow + 8 q n; rows w + 8 q < nr exist (q < nq)
    const float* __restrict__ wrow = Wb + (size_t)w * n + lane;
    const size_t n8 = (size_t)8 * n;
    const int nq = (nr - w + 7) >> 3;
    auto load = [&](int c, float (&x)[16]) {
      const bool ain = kTcKc * c + lane < n;
      const float* __restrict__ p = wrow + kTcKc * c;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        x[q] = (ain && q < nq) ? __ldcs(p) : 0.f;  // read once: streaming
        p += n8;
      }
    };
    auto fetch_basis = [&](int c) {  // basis chunk c into the B images of stage c % S
      float* Bhi = base + (size_t)(c % kSynStages) * stage + 2 * imgA;
      const float* src = basis + (size_t)c * 2 * imgB;
      for (int i = 4 * t; i < 2 * imgB; i += 4 * kSynProd * 32) cp16(Bhi + i, src + i);
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // W registers two chunks ahead in a ring of three buffers used by name
    // (the loop is unrolled by three), so no copy waits on loads in flight
    auto step = [&](int c, float (&use)[16], float (&fill)[16]) -> bool {
      if (fail) return false;
      const int st = c % kSynStages;
      if (c + 2 < nchunk) load(c + 2, fill);
      if (c + 1 < nchunk) {
        const int c1 = c + 1;
        if (c1 >= kSynStages &&
            !tc::mbar_wait(empty(c1 % kSynStages), (c1 / kSynStages - 1) & 1, limit)) {
          fail = 1;
          return false;
        }
        fetch_basis(c1);  // stage of chunk c + 1 is free: its previous chunk's MMAs completed
      }
      float* Ahi = base + (size_t)st * stage;
      float* Alo = Ahi + imgA;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int o = tc::img_off(w + 8 * q, lane, kTcKc);
        float h, l;
        tc::split_tf32(use[q], h, l);
        Ahi[o] = h;
        Alo[o] = l;
      }
      if (c + 1 < nchunk)
        asm volatile("cp.async.wait_group 1;" ::: "memory");  // basis chunk c landed (c + 1 may be in flight)
      else
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      tc::fence_async_smem();
      tc::mbar_arrive(full(st));
      return true;
    };
    float b0[16], b1[16], b2[16];
    load(0, b0);
    if (nchunk > 1) load(1, b1);
    fetch_basis(0);
    for (int c = 0; c < nchunk; c += 3) {
      if (!step(c, b0, b2)) break;
      if (c + 1 < nchunk && !step(c + 1, b1, b0)) break;
      if (c + 2 < nchunk && !step(c + 2, b2, b1)) break;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (w < kSynProd + kSynAcc) {
    // ---- accumulators: TMEM lanes 32 (w % 4) .. = rows, columns HC h .. + HC of both
    //      halves (h = 0, 1; HC = NP / 2 = 8, 16, 24 or 32) ----
    const int lrow = 32 * (w & 3), h = (w - kSynProd) >> 2, HC = NP / 2;
    float acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
    bool ok = true;
    for (int c = 0; c < nchunk; ++c) {
      const int b = c & 1;
      const bool got = !fail && tc::mbar_wait(tfull(b), (c >> 1) & 1, limit);
      if (!__all_sync(0xffffffffu, got)) {  // warp-uniform: the TMEM loads below are warp-collective
        fail = 1;
        ok = false;
        break;
      }
      tc::fence_after();
      const uint32_t ta = tmem + ((uint32_t)lrow << 16) + (uint32_t)(NP * b + HC * h);
      if (HC == 32) {
        float v[32];
        tc::tmem_ld32(ta, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] += v[j];
      } else if (HC == 16) {
        float va[8], vb[8];
        tc::tmem_ld8x2(ta, ta + 8, va, vb);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          acc[j] += va[j];
          acc[8 + j] += vb[j];
        }
      } else {
#pragma unroll
        for (int g = 0; g < 3; ++g) {
          if (8 * g < HC) {
            float v[8];
            tc::tmem_ld8(ta + 8 * g, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[8 * g + j] += v[j];
          }
        }
      }
      tc::fence_before();
      tc::mbar_arrive(tempty(b));
    }
    const int r = lrow + lane;
    if (ok && r < nr) {
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const int m = (HC * h + j) >> 1;
        if (j < HC && m < Lj) V[(size_t)r * Lj + m] = mkc<float>(acc[j], acc[j + 1]);
      }
    }
  } else if (lane == 0) {
    // ---- MMA issuer ----
    const uint32_t idesc = tc::idesc_tf32(kTcM, NP);
    const uint64_t kstep = (uint64_t)(tc::img_kstep_bytes(1) >> 4);
    for (int c = 0; c < nchunk; ++c) {
      if (fail) break;
      const int st = c % kSynStages, b = c & 1;
      if (!tc::mbar_wait(full(st), (c / kSynStages) & 1, limit) ||
          (c >= 2 && !tc::mbar_wait(tempty(b), ((c >> 1) - 1) & 1, limit))) {
        fail = 1;
        break;
      }
      tc::fence_after();
      const uint32_t aH = tc::smem_u32(base + (size_t)st * stage), aL = aH + imgA * 4, bH = aL + imgA * 4,
                     bL = bH + imgB * 4;
      const uint32_t dm = tmem + (uint32_t)(NP * b);
      const uint64_t dAH = tc::smem_desc(aH, kTcKc), dAL = tc::smem_desc(aL, kTcKc);
      const uint64_t dBH = tc::smem_desc(bH, kTcKc), dBL = tc::smem_desc(bL, kTcKc);
#pragma unroll
      for (int k = 0; k < kTcKc / 8; ++k) {  // cross terms first, then hi*hi
        const uint64_t o = kstep * k;
        tc::mma_tf32(dm, dAH + o, dBL + o, idesc, k > 0);
        tc::mma_tf32(dm, dAL + o, dBH + o, idesc, 1);
      }
#pragma unroll
      for (int k = 0; k < kTcKc / 8; ++k) {
        const uint64_t o = kstep * k;
        tc::mma_tf32(dm, dAH + o, dBH + o, idesc, 1);
      }
      tc::mma_commit(empty(st));
      tc::mma_commit(tfull(b));
      last = c;
    }
    issued = last;
  }
  __syncwarp();
  tc::fence_before();
  __syncthreads();
  if (w == kSynProd) {
    // after a give-up, whichever role's it was: a bounded wait for the MMAs in flight before TMEM is released
    if (lane == 0 && fail) {
      if (issued >= 0) tc::mbar_wait(tfull(issued & 1), (issued >> 1) & 1, tc::kWaitCycles);
      atomicAdd(&g_tc_timeouts, 1);
    }
    __syncwarp();
    tc::tmem_free(tmem, ncols);
  }
}

// Basis images.  Analysis: [tile][hi, lo][img_floats(128, K8)], sample a =
// 128 tile + r, column k.  Synthesis: [chunk][hi, lo][img_floats(NP, 32)],
// row j, sample a = 32 chunk + k.  Values from the exact angle
// 2 pi ((m a) mod n) / n in FP64, then split.
__device__ __forceinline__ void put_split(float* hi, float* lo, int o, double v) {
  const float h = tc::to_tf32((float)v);
  hi[o] = h;
  lo[o] = tc::to_tf32((float)(v - (double)h));
}

struct TcBasisJobs {
  TcBasis t[2 * MAXS];
};
// blockIdx.y: table
__global__ void __launch_bounds__(256) k_tc_basis(TcBasisJobs jobs) {
  const TcBasis& b = jobs.t[blockIdx.y];
  const int n = 2 * b.L - 1, Lj = b.Lj, RC = b.syn ? syn_npad(Lj) : kTcA, KC = b.syn ? kTcKc : ana_k8(Lj);
  const int img = tc::img_floats(RC, KC), ntile = (n + (b.syn ? kTcKc : kTcA) - 1) / (b.syn ? kTcKc : kTcA);
  const long long total = (long long)ntile * RC * KC;
  for (long long idx = blockIdx.x * 256ll + threadIdx.x; idx < total; idx += gridDim.x * 256ll) {
    const int tile = (int)(idx / (RC * KC)), r = (int)(idx / KC % RC), k = (int)(idx % KC);
    const int a = b.syn ? tile * kTcKc + k : tile * kTcA + r, q = b.syn ? r : k, m = q >> 1;
    double v = 0.0;
    if (a < n && q < 2 * Lj) {
      const long long u = ((long long)m * a) % n;
      double sn, cs;
      sincospi(2.0 * (double)u / (double)n, &sn, &cs);
      const double c = b.syn ? 2.0 * 3.14159265358979323846 / n : (m == 0 ? 1.0 : 2.0);
      v = (q & 1) ? -c * sn : c * cs;
    }
    float* hi = b.out + (size_t)tile * 2 * img;
    put_split(hi, hi + img, tc::img_off(r, k, KC), v);
  }
}

// One warp waits, bounded, on an mbarrier that nothing arrives on: the
// failure path of every bounded wait above (give up, count it), on demand.
__global__ void k_wait_probe(long long limit) {
  __shared__ __align__(8) uint64_t mbar;
  const uint32_t mb = tc::smem_u32(&mbar);
  if (threadIdx.x == 0) tc::mbar_init(mb, 1);
  __syncwarp();
  const bool ok = tc::mbar_wait(mb, 0, limit);
  if (!__any_sync(0xffffffffu, ok) && threadIdx.x == 0) atomicAdd(&g_tc_timeouts, 1);
}

}  // namespace

cudaError_t alpha_tc_wait_probe(long long limit, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(limit);
  return cudaGetLastError();
}

size_t alpha_tc_table_floats(int L, int Lj, bool syn) {
  if (Lj <= 0) return 0;
  const int n = 2 * L - 1;
  if (!syn) return (size_t)((n + kTcA - 1) / kTcA) * 2 * tc::img_floats(kTcA, ana_k8(Lj));
  return (size_t)((n + kTcKc - 1) / kTcKc) * 2 * tc::img_floats(syn_npad(Lj), kTcKc);
}

// All basis tables of a plan in one launch (a memset and a launch each: 28 in a
// plan of L = 32; their pads are zeroed by the caller).
cudaError_t alpha_tc_build_tables(const TcBasis* tables, int n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  TcBasisJobs jobs;
  for (int i = 0; i < n; ++i) jobs.t[i] = tables[i];
  k_tc_basis<<<dim3(128, n), 256, 0, st>>>(jobs);
  return cudaGetLastError();
}

int alpha_tc_items(int L, int rows, int njobs, bool syn, int& P) {
  P = kTcRows;
  if (syn) return (rows + kTcM - 1) / kTcM;
  const int tiles = (2 * L - 1 + kTcA - 1) / kTcA;
  for (P = 2048; P > kTcRows && (long long)njobs * tiles * ((rows + P - 1) / P) < kTcAnaCtas; P /= 2) {}
  return tiles * ((rows + P - 1) / P);
}

void launch_alpha_tc(bool syn, const CztSeg<float>* segs, int nseg, int total_items, const CallPtrs& ptrs,
                     cudaStream_t st, long long limit) {
  if (total_items <= 0) return;
  const bool probe = limit != kWaitLimit;
  if (syn)
    launch_after(probe ? k_alpha_syn_tc<true> : k_alpha_syn_tc<false>, total_items, kSynThreads, syn_tc_smem(), st, segs, nseg, ptrs, limit);
  else
    launch_after(probe ? k_alpha_ana_tc<true> : k_alpha_ana_tc<false>, total_items, kTcAnaThreads, ana_tc_smem(), st, segs, nseg, ptrs, limit);
}

cudaError_t alpha_tc_prepare() {
  for (auto k : {k_alpha_ana_tc<false>, k_alpha_ana_tc<true>})
    if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ana_tc_smem()); e != cudaSuccess)
      return e;
  for (auto k : {k_alpha_syn_tc<false>, k_alpha_syn_tc<true>})
    if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)syn_tc_smem()); e != cudaSuccess)
      return e;
  return cudaSuccess;
}

cudaError_t alpha_tc_timeouts(int* count) {
  int zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(count, g_tc_timeouts, sizeof(int));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_tc_timeouts, &zero, sizeof(int));
}

}  // namespace s2dw
