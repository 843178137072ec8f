// Beta and alpha sums as matrix products on the tensor cores (FP32 plans;
// Eqs. (29)-(30), (37), (40)): dense cosine / sine transforms of any length.
//
// Folding by symmetry halves each product and splits it in two:
//   beta, analysis (column m, sigma = (-1)^{m+N-1}; cos for sigma = 1, else i sin):
//     E_b = sum over even m', O_b = sum over odd m' of c_{m'} Yhat_{m'} trig(m' beta_b),
//     X_b = E + O, X_{2L-1-b} = sigma (E - O)          (b < L, c_0 = 1, else 2);
//   beta, synthesis: s, d = V_b +- V_{2L-1-b},
//     Vhat_{m'} = c_{m'} sum_{b<L} q_b (s or d) trig(m' beta_b), even and odd m' apart;
//   alpha, analysis: W_a = C + S, W_{n-a} = C - S, C = sum_m c_m Re X_m cos(m alpha_a),
//     S = -sum_m c_m Im X_m sin(m alpha_a)               (a < L, n = 2L - 1);
//   alpha, synthesis: s, d = W_a +- W_{n-a},
//     Re V_m = (2 pi/n) sum_{a<L} s cos(m alpha_a), Im V_m = -(2 pi/n) sum d sin(m alpha_a).
// Each is a pair of real products of a 128-row data operand with a constant
// basis; one FFT per column or row (two where the length is no power of two)
// costs 15 to 60 FP32 instructions per value on the FP32 pipes, the products
// run on pipes 50 times as fast.
//
// FP32 accuracy from FP16 products: x = hi + lo with hi = x rounded to FP16 (11
// bits) and lo = x - hi rounded to FP16, so that x is held to 2^-23 (an FP32
// value to 2^-24), and x y = hi hi + hi lo + lo hi up to 2^-21, 2^-23.7 in the
// mean square: single terms are worse than FP32 products, sums of whole calls
// are closer to 64 bits than the transforms' were (3.3e-7 -> 2.4e-7 at L = 723,
// 2.6e-7 -> 2.0e-7 at L = 361), as few roundings follow one another.  Range: the
// basis is scaled by a power of two per table; the data by a power of two per row
// and stage (32 values of each of the two products), chosen from their maximum;
// in the beta synthesis per tile and stage, whose 64 columns m come out of one
// alpha sum per row b with errors relative to its largest (a column 2^-16 below
// its neighbours still keeps 24 bits).  The tensor cores' FP32 accumulation
// truncates, so a stage's sums (cross products first) leave TMEM after its 32
// terms and are added, with both scales taken back, in FP32 registers with
// rounding to nearest: any input whose partial sums are finite works.
//
// Two kernels.  k_sg_convert folds, scales and splits the data once, a CTA per
// tile of 128 rows and stage, into the operand images the products read (in
// shared memory, then one bulk store); splitting inside the product kernel
// instead was repeated for every basis tile and took 2.5 us per stage.
// k_split_gemm: one persistent CTA per SM walks 128 x 128 output tiles (both
// products: 256 accumulator columns, double-buffered in TMEM):
//   warp 0      one thread: bulk copies of the data and basis images of a stage
//               into a ring of three;
//   warp 1      one thread: the MMAs and their commits;
//   warps 2-9   accumulators: 128 registers of sums per thread; the epilogue
//               overlaps the next tile's first stages.
// Images: no-swizzle K-major core matrices of 8 rows x 16 bytes (padding them
// apart for conflict-free stores in the conversion made the products no faster
// and the traffic larger).
// What bounds it (L = 1000, N = 5, analysis beta, 248 us where the chirp-z took
// 417): conversion 35 us; the products 133 us, 0.85 us per stage, near what
// shared memory allows (it feeds each MMA 128 bytes per cycle and takes the
// images at the same time: 164 KB per stage, 1280 cycles); the stores of X 80
// us, half-filled sectors as a tile holds the columns of one parity.  The alpha
// analysis spills 8 bytes per thread, the alpha synthesis 4.
// Measured (GB300, us, analysis / synthesis, before -> now).  beta: L = 361, N =
// 4, lambda = 3 72 / 64 -> 31 / 33, L = 723, N = 6 337 / 320 -> 152 / 184, L = 1900,
// N = 4 1834 / 1756 -> 948 / 1050, L = 2048, N = 8 2807 / 2991 -> 2188 / 2330, MW
// grid L = 511, N = 3 91 / 280 -> 39 / 179; alpha of all scales above 32: L = 256,
// N = 5 57 / 55 -> 29 / 27, L = 512, N = 3 102 / 98 -> 66 / 64, L = 723, N = 6 361 /
// 411 -> 283 / 309, L = 1024, N = 5 512 / 540 -> 401 / 495.
// Every wait is bounded; a CTA that gives up stops all roles, and once they have
// met waits for its MMAs and copies in flight (bounded), counts the event and
// frees its TMEM.
#include <cuda_fp16.h>

#include "czt.cuh"
#include "tc.cuh"

namespace s2dw {

__device__ int g_sg_timeouts;  // bounded waits that gave up (read and reset by the host)

namespace {

constexpr int kSgK = 32;                      // terms of each product per stage
constexpr int kLbo = 128, kSbo = 512;         // bytes between core matrices along K, between 8-row groups
constexpr int kImg = 16 * kSbo;               // one 128 x 32 FP16 image
constexpr int kHalf = 4 * kImg;               // operand of a stage: products 0, 1 x (hi, lo)
constexpr int kSgStages = 3;
constexpr int kScaleB = 128 * 4;              // the rows' inverse scales of a stage
constexpr int kData = kHalf + kScaleB;        // a data stage in global memory: images, inverse scales
constexpr int kSgAcc = 8;                     // accumulator warps (two per TMEM lane quadrant)
constexpr int kSgThreads = 32 * (2 + kSgAcc);
constexpr int kSgScales = 6;                  // stages of row scales kept: three in the ring, two in TMEM, one spare
constexpr size_t kSgSmem = (size_t)kSgStages * 2 * kHalf + (size_t)kSgScales * kScaleB;
static_assert(kSgDataBytes == kData, "bytes of a data stage");
constexpr int kCvWarps = 8;                   // warps of the conversion kernel
constexpr float kSgAnaScale = 8192.f;         // scale of the analysis bases (values up to 2), a power of two
constexpr float kSgAlphaSynScale = 16384.f;   // of the alpha synthesis basis (values up to 1)

enum SgMode { SG_BETA_ANA = 0, SG_BETA_SYN = 1, SG_ALPHA_ANA = 2, SG_ALPHA_SYN = 3 };

__device__ __forceinline__ int sg_off(int r, int k) {
  return (r >> 3) * kSbo + (k >> 3) * kLbo + (r & 7) * 16 + (k & 7) * 2;
}
__device__ __forceinline__ uint64_t sg_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kLbo >> 4) << 16) | ((uint64_t)(kSbo >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}
// Wait bounded in time; false once any role of the CTA has given up.  Polls
// without suspending: the roles hand each stage on several times, and waking
// from a suspended wait costs more than the poll's issue slots.
__device__ __forceinline__ bool sg_poll(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool sg_wait(uint32_t mbar, uint32_t parity, volatile int* fail, long long limit) {
  if (sg_poll(mbar, parity)) return true;
  const long long t0 = clock64();
  while (!sg_poll(mbar, parity)) {
    if (*fail) return false;
    if (clock64() - t0 > limit) {
      *fail = 1;
      return false;
    }
  }
  return true;
}

// 2^(14 - e) for a row maximum in [2^e, 2^(e+1)), as a float (1 for 0, Inf and
// NaN), and its inverse; clamped so that both stay normal (the inverse times the
// basis scale, 2^-23 at least, is then 2^-136 at least: exact)
__device__ __forceinline__ float sg_scale(uint32_t maxbits, float& inv) {
  const int e = (int)(maxbits >> 23);  // biased exponent; the sign bit is clear
  if (maxbits == 0u || e == 255) {
    inv = 1.f;
    return 1.f;
  }
  const int s = min(127 + 14 - (e - 127), 240);  // biased exponent of the scale
  inv = __uint_as_float((uint32_t)(254 - s) << 23);
  return __uint_as_float((uint32_t)s << 23);
}
__device__ __forceinline__ uint32_t absmax(uint32_t m, float x) { return max(m, __float_as_uint(x) & 0x7fffffffu); }

// the pair (a, b) scaled and split, stored at byte o of the images hi, hi + kImg
__device__ __forceinline__ void put2(unsigned char* img, int o, float a, float b, float s) {
  a *= s;
  b *= s;
  const __half2 h = __floats2half2_rn(a, b);
  const float2 hf = __half22float2(h);
  *reinterpret_cast<__half2*>(img + o) = h;
  *reinterpret_cast<__half2*>(img + kImg + o) = __floats2half2_rn(a - hf.x, b - hf.y);
}

struct SgTile {  // one output tile
  const CztSeg<float>* sg;
  int rt, nt, nk;      // data tile, basis tile, stages
  int g, par, mt;      // beta: gamma sample, parity of m, tile of 64 columns m
  int r0, rows;        // alpha: first row of 128, rows of the segment
  bool minus;          // beta: sigma = -1
};

template <int MODE>
__device__ __forceinline__ SgTile sg_data_tile(const CztSeg<float>& sg, int rt) {
  SgTile t;
  t.sg = &sg;
  t.rt = rt;
  t.nt = 0;
  t.nk = sg.nsegs;
  if (MODE == SG_BETA_ANA || MODE == SG_BETA_SYN) {
    const int tpp = ((sg.Lj + 1) / 2 + 63) / 64;
    t.g = rt / (2 * tpp);
    t.par = (rt / tpp) & 1;
    t.mt = rt % tpp;
    t.minus = (t.par + sg.N - 1) & 1;
    t.r0 = t.rows = 0;
  } else {
    t.r0 = rt * 128;
    t.rows = sg.N * sg.nb;
    t.g = t.par = t.mt = 0;
    t.minus = false;
  }
  return t;
}
// basis tiles of a data tile are consecutive: the CTAs that share its images run together
template <int MODE>
__device__ __forceinline__ SgTile sg_tile(const CztSeg<float>* __restrict__ segs, int nseg, int tile) {
  const CztSeg<float>& sg = segs[czt_find_seg<float>(segs, nseg, tile)];
  const int i = tile - sg.start;
  SgTile t = sg_data_tile<MODE>(sg, i / sg.P);
  t.nt = i % sg.P;
  return t;
}

// 1-D bulk copy global -> shared, completion on the mbarrier
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, int bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"((uint32_t)bytes), "r"(mbar)
               : "memory");
}

// Folds, scales and splits one stage (32 terms of both products) of one tile of
// 128 data rows.  blockIdx.x: data stage of the launch (stages of a tile
// consecutive, tiles of a segment consecutive).
template <int MODE>
__global__ void __launch_bounds__(32 * kCvWarps)
k_sg_convert(const CztSeg<float>* __restrict__ segs, int nseg, CallPtrs ptrs) {
  begin_after();
  extern __shared__ __align__(128) unsigned char sg_smem[];
  unsigned char* img = sg_smem;
  float* sinv = reinterpret_cast<float*>(sg_smem + kHalf);
  __shared__ uint32_t smax;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  int lo = 0, hi = nseg - 1;  // segment by first data stage (tabD)
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segs[mid].tabD <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const CztSeg<float>& sg = segs[lo];
  const int i0 = blockIdx.x - sg.tabD, c = i0 % sg.nsegs, rt = i0 / sg.nsegs;
  const SgTile T = sg_data_tile<MODE>(sg, rt);
  const int Lj = sg.Lj, L = sg.L, n = 2 * L - 1;
  // 1 / (scale of the basis): the sums are scaled back by it stage by stage, with
  // the row's own scale (kept to the end it brought sums above 2^104 to Inf)
  const float unbasis = MODE == SG_ALPHA_SYN ? 1.f / kSgAlphaSynScale : sg.scale;
  const int hl = lane >> 4, tl = lane & 15;  // half-warp, position in it
  if constexpr (MODE == SG_BETA_SYN) {
    // lanes: 32 of the tile's 64 columns; a task is one half of the columns and
    // four b (and their reflections); one scale for the stage
    if (t == 0) smax = 0;
    __syncthreads();
    float2 v[2][8];
    uint32_t mx = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int task = w + kCvWarps * i, m = 2 * (64 * T.mt + 32 * (task & 1) + lane) + T.par;
      const float2* V = sg.buf_in + (size_t)T.g * sg.nb * Lj + m;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int b = kSgK * c + 4 * (task >> 1) + u;
        const bool in = m < Lj && b < L;
        const float2 x = in ? V[(size_t)b * Lj] : make_float2(0.f, 0.f);
        const float2 y = in ? V[(size_t)(2 * L - 1 - b) * Lj] : make_float2(0.f, 0.f);
        v[i][u] = make_float2(x.x + y.x, x.y + y.y);
        v[i][4 + u] = make_float2(x.x - y.x, x.y - y.y);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int u = 0; u < 8; ++u) mx = absmax(absmax(mx, v[i][u].x), v[i][u].y);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) atomicMax(&smax, mx);
    __syncthreads();
    float inv;
    const float s = sg_scale(smax, inv);
    if (t < 128) sinv[t] = inv * unbasis;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int task = w + kCvWarps * i;
      const int r = 2 * (32 * (task & 1) + lane), o = sg_off(r, 4 * (task >> 1));
#pragma unroll
      for (int p = 0; p < 2; ++p) {  // products: sums, differences
        const float2* x = &v[i][4 * p];
        unsigned char* q = img + 2 * p * kImg + o;
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // rows (m, Re), (m, Im); sigma = -1: -2i sum q V sin
          float y[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) y[u] = (T.minus ? (e == 0 ? x[u].y : -x[u].x) : (e == 0 ? x[u].x : x[u].y)) * s;
          const __half2 h0 = __floats2half2_rn(y[0], y[1]), h1 = __floats2half2_rn(y[2], y[3]);
          const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
          const __half2 l0 = __floats2half2_rn(y[0] - f0.x, y[1] - f0.y), l1 = __floats2half2_rn(y[2] - f1.x, y[3] - f1.y);
          *reinterpret_cast<uint2*>(q + 16 * e) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
          *reinterpret_cast<uint2*>(q + kImg + 16 * e) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
        }
      }
    }
  } else {
    // half-warps: beta, analysis: columns i and i + 2 of the tile's 64 (rows 2 i,
    // 2 i + 1 of the image: Re, Im); alpha: rows r and r + 4.  A lane holds the
    // terms tl and tl + 16 of the stage (positions 2 tl, 2 tl + 1 of the images;
    // the basis is laid out alike).
    constexpr int NIT = (MODE == SG_BETA_ANA ? 32 : 64) / kCvWarps;
    constexpr int NV = MODE == SG_BETA_ANA ? 8 : 4;
    const float* Wb = nullptr;
    if (MODE == SG_ALPHA_SYN)
      Wb = reinterpret_cast<const float*>(sg.is_phi ? ptrs.Wphi[sg.job] : ptrs.W[sg.job]) + sg.woff + (size_t)T.r0 * n;
    auto row_of = [&](int i) {  // column i (beta) or row (alpha) of this half-warp's item
      const int it = w + kCvWarps * i;
      return MODE == SG_BETA_ANA ? (it >> 1) * 4 + (it & 1) + 2 * hl : (it >> 2) * 8 + (it & 3) + 4 * hl;
    };
    float v[NIT][NV];
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
      const int r = row_of(i);
      float(&x)[NV] = v[i];
      if constexpr (MODE == SG_BETA_ANA) {
        const int m = 2 * (64 * T.mt + r) + T.par;
        const float2* Y = sg.buf_in + ((size_t)T.g * Lj + m) * Lj;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int mp = 2 * (kSgK * c + tl + 16 * u);  // even m', then odd
          float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
          if (m < Lj && mp < Lj) {
            if ((Lj & 1) == 0) q = *reinterpret_cast<const float4*>(Y + mp);
            else {
              const float2 a = Y[mp], b = mp + 1 < Lj ? Y[mp + 1] : make_float2(0.f, 0.f);
              q = make_float4(a.x, a.y, b.x, b.y);
            }
          }
          x[4 * u] = q.x, x[4 * u + 1] = q.y, x[4 * u + 2] = q.z, x[4 * u + 3] = q.w;
        }
      } else if constexpr (MODE == SG_ALPHA_ANA) {
        const float2* X = sg.buf_in + (size_t)(T.r0 + r) * Lj;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int m = kSgK * c + tl + 16 * u;
          const float2 q = (T.r0 + r < T.rows && m < Lj) ? __ldcs(X + m) : make_float2(0.f, 0.f);
          x[2 * u] = q.x, x[2 * u + 1] = q.y;
        }
      } else {
        const float* W = Wb + (size_t)r * n;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int a = kSgK * c + tl + 16 * u;
          const bool in = T.r0 + r < T.rows && a < L;
          const float p = in ? __ldcs(W + a) : 0.f, q = (in && a > 0) ? __ldcs(W + n - a) : 0.f;
          x[2 * u] = p + q, x[2 * u + 1] = p - q;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
      float(&x)[NV] = v[i];
      uint32_t mx = 0;
#pragma unroll
      for (int e = 0; e < NV; ++e) mx = absmax(mx, x[e]);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float inv;
      const float s = sg_scale(mx, inv);
      const int r = row_of(i);
      if constexpr (MODE == SG_BETA_ANA) {
        // x: even (Re, Im), odd (Re, Im) of term tl, then of tl + 16; sigma = -1: 2i sum Y sin
        const int o = sg_off(2 * r, 2 * tl);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const float a0 = x[2 * p], a1 = x[2 * p + 1], b0 = x[4 + 2 * p], b1 = x[5 + 2 * p];
          put2(img + 2 * p * kImg, o, T.minus ? -a1 : a0, T.minus ? -b1 : b0, s);
          put2(img + 2 * p * kImg, o + 16, T.minus ? a0 : a1, T.minus ? b0 : b1, s);
        }
        if (tl < 2) sinv[2 * r + tl] = inv * unbasis;
      } else {
        const int o = sg_off(r, 2 * tl);
        put2(img, o, x[0], x[2], s);
        put2(img + 2 * kImg, o, x[1], x[3], s);
        if (tl == 0) sinv[r] = inv * unbasis;
      }
    }
  }
  tc::fence_async_smem();
  __syncthreads();
  if (t == 0) {
    unsigned char* dst = const_cast<unsigned char*>(reinterpret_cast<const unsigned char*>(sg.pre)) + (size_t)i0 * kData;
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(tc::smem_u32(sg_smem)),
                 "r"((uint32_t)kData)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
}

template <int MODE>
__global__ void __launch_bounds__(kSgThreads, 1)
k_split_gemm(const CztSeg<float>* __restrict__ segs, int nseg, int total, CallPtrs ptrs, long long wait_limit) {
  begin_after();
  // (as a constant here, or the register allocation costs the kernel 2%: L = 723, N = 6 309 against 316 us;
  // that of the alpha analysis has room for it and spills less, 305 -> 283)
  const long long limit = MODE == SG_ALPHA_SYN ? kWaitLimit : wait_limit;
  extern __shared__ __align__(128) unsigned char sg_smem[];
  const float* scales = reinterpret_cast<const float*>(sg_smem + (size_t)kSgStages * 2 * kHalf);
  __shared__ __align__(8) uint64_t bar[2 * kSgStages + 4];  // full[S], empty[S], tfull[2], tempty[2]
  __shared__ uint32_t tbase;
  __shared__ int s_fail, s_loaded, s_issued;  // a role gave up; stages whose copies, whose products were issued
  volatile int* fail = &s_fail;
  constexpr bool DATA_A = MODE == SG_BETA_ANA || MODE == SG_BETA_SYN;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const uint32_t bar0 = tc::smem_u32(&bar[0]);
  auto bfull = [&](int s) { return bar0 + 8u * s; };
  auto bempty = [&](int s) { return bar0 + 8u * (kSgStages + s); };
  auto btfull = [&](int b) { return bar0 + 8u * (2 * kSgStages + b); };
  auto btempty = [&](int b) { return bar0 + 8u * (2 * kSgStages + 2 + b); };
  if (t == 0) {
    for (int s = 0; s < kSgStages; ++s) {
      tc::mbar_init(bfull(s), 1);
      tc::mbar_init(bempty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(btfull(b), 1);
      tc::mbar_init(btempty(b), kSgAcc);
    }
    s_fail = 0;
  }
  if (w == 1) tc::tmem_alloc(&tbase, 512);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tbase;

  if (w == 0) {
    if (lane == 0) {
      int gc = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
        const SgTile T = sg_tile<MODE>(segs, nseg, tile);
        const size_t set = DATA_A ? (size_t)(T.minus ? 1 : 0) * T.sg->tabP : 0;
        const unsigned char* bas = reinterpret_cast<const unsigned char*>(T.sg->H) + ((set + T.nt) * T.sg->tabK) * (size_t)kHalf;
        const unsigned char* dat = reinterpret_cast<const unsigned char*>(T.sg->pre) + (size_t)T.rt * T.nk * kData;
        for (int c = 0; c < T.nk; ++c, ++gc) {
          const int s = gc % kSgStages;
          if (gc >= kSgStages && !sg_wait(bempty(s), (uint32_t)(gc / kSgStages - 1) & 1u, fail, limit)) {
            ok = false;
            break;
          }
          const uint32_t mb = bfull(s), dst = tc::smem_u32(sg_smem + (size_t)s * 2 * kHalf);
          const uint32_t dsc = tc::smem_u32(scales) + (uint32_t)((gc % kSgScales) * kScaleB);
          asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(mb),
                       "r"((uint32_t)(kData + kHalf))
                       : "memory");
          bulk_g2s(dst, dat + (size_t)c * kData, kHalf, mb);
          bulk_g2s(dst + kHalf, bas + (size_t)c * kHalf, kHalf, mb);
          bulk_g2s(dsc, dat + (size_t)c * kData + kHalf, kScaleB, mb);
        }
      }
      s_loaded = gc;
    }
    __syncwarp();
  } else if (w == 1) {
    if (lane == 0) {
      const uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);  // FP16 x FP16 -> FP32, 128 x 128
      int gc = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
        const int nk = sg_tile<MODE>(segs, nseg, tile).nk;
        for (int c = 0; c < nk; ++c, ++gc) {
          const int s = gc % kSgStages, b = gc & 1;
          if (!sg_wait(bfull(s), (uint32_t)(gc / kSgStages) & 1u, fail, limit) ||
              (gc >= 2 && !sg_wait(btempty(b), (uint32_t)(gc / 2 - 1) & 1u, fail, limit))) {
            ok = false;
            break;
          }
          tc::fence_after();
          const uint32_t dat = tc::smem_u32(sg_smem + (size_t)s * 2 * kHalf), bas = dat + kHalf;
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const uint32_t d = tmem + (uint32_t)(b * 256 + p * 128);
            const uint64_t a0 = sg_desc((DATA_A ? dat : bas) + 2 * p * kImg), b0 = sg_desc((DATA_A ? bas : dat) + 2 * p * kImg);
            constexpr uint64_t lo = kImg >> 4, ks = (2 * kLbo) >> 4;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              mma_f16(d, a0 + k * ks, b0 + lo + k * ks, idesc, k > 0);
              mma_f16(d, a0 + lo + k * ks, b0 + k * ks, idesc, 1);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) mma_f16(d, a0 + k * ks, b0 + k * ks, idesc, 1);
          }
          tc::mma_commit(bempty(s));
          tc::mma_commit(btfull(b));
        }
      }
      s_issued = gc;
    }
    __syncwarp();
  } else {
    // TMEM lanes 32 (w % 4) + lane, columns 64 h .. 64 h + 63 of both products
    const int h = (w - 2) >> 2, ml = 32 * (w & 3) + lane;
    const uint32_t tq = tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)(64 * h);
    int gc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
      const SgTile T = sg_tile<MODE>(segs, nseg, tile);
      float acc[2][64];
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int j = 0; j < 64; ++j) acc[p][j] = 0.f;
      for (int c = 0; c < T.nk; ++c) {
        const int b = gc & 1;
        const float* sc = scales + (gc % kSgScales) * (kScaleB / 4);
        // one decision per warp: the TMEM loads and the barrier below are warp-collective
        if (!__all_sync(0xffffffffu, sg_wait(btfull(b), (uint32_t)(gc / 2) & 1u, fail, limit))) {
          *fail = 1;
          ok = false;
          break;
        }
        tc::fence_after();
        const float rs = DATA_A ? sc[ml] : 0.f;
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float x[16];
            tc::tmem_ld16(tq + (uint32_t)(b * 256 + p * 128 + 16 * q), x);
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
              const float4 s4 = DATA_A ? make_float4(rs, rs, rs, rs) : *reinterpret_cast<const float4*>(sc + 64 * h + 16 * q + j);
              float* a = &acc[p][16 * q + j];
              a[0] = __fmaf_rn(x[j], s4.x, a[0]);
              a[1] = __fmaf_rn(x[j + 1], s4.y, a[1]);
              a[2] = __fmaf_rn(x[j + 2], s4.z, a[2]);
              a[3] = __fmaf_rn(x[j + 3], s4.w, a[3]);
            }
          }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(btempty(b));
        ++gc;
      }
      if (!ok) break;
      const CztSeg<float>& sg = *T.sg;
      const int Lj = sg.Lj, L = sg.L, n = 2 * L - 1;
      if constexpr (MODE == SG_BETA_ANA) {
        const int m = 2 * (64 * T.mt + (ml >> 1)) + T.par, b0 = 128 * T.nt + 64 * h, jn = min(64, L - b0);
        const bool reflect = sg.nb == 2 * L;
        if (m < Lj) {
          float* X = reinterpret_cast<float*>(sg.buf_out + (size_t)T.g * sg.nb * Lj + m) + (ml & 1);
          const float so = T.minus ? -1.f : 1.f;
          const size_t rl = 2 * (size_t)Lj;
          float* up = X + (size_t)b0 * rl;
          float* dn = X + (size_t)(2 * L - 1 - b0) * rl;
          // an odd row count N nb (MW grid) pairs the last row with row N nb of
          // the buffer in the alpha analysis: zero it
          if (T.nt == 0 && h == 0 && T.g == sg.N - 1 && ((sg.N * sg.nb) & 1)) X[(size_t)sg.nb * rl] = 0.f;
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            if (j < jn) {
              *up = acc[0][j] + acc[1][j];
              if (reflect) *dn = (acc[0][j] - acc[1][j]) * so;
            }
            up += rl;
            dn -= rl;
          }
        }
      } else if constexpr (MODE == SG_BETA_SYN) {
        const int m = 2 * (64 * T.mt + (ml >> 1)) + T.par, i0 = 128 * T.nt + 64 * h;
        if (m < Lj) {
          float* V = reinterpret_cast<float*>(sg.buf_out + (size_t)T.g * Lj * Lj + m) + (ml & 1);
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            // product 0 (sums): even m' with cos, odd with sin; product 1 the others
            const int m0 = 2 * (i0 + j) + (T.minus ? 1 : 0), m1 = 2 * (i0 + j) + (T.minus ? 0 : 1);
            if (m0 < Lj) V[(size_t)m0 * 2 * Lj] = acc[0][j];
            if (m1 < Lj) V[(size_t)m1 * 2 * Lj] = acc[1][j];
          }
        }
      } else if constexpr (MODE == SG_ALPHA_ANA) {
        const int a = 128 * T.nt + ml, r = T.r0 + 64 * h, jn = min(64, T.rows - r);
        if (a < L && jn > 0) {
          float* W = reinterpret_cast<float*>(sg.is_phi ? ptrs.Wphi[sg.job] : ptrs.W[sg.job]) + sg.woff + (size_t)r * n;
          float *up = W + a, *dn = W + (a > 0 ? n - a : 0);
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            if (j < jn) {
              const float c = acc[0][j], s = acc[1][j];
              if (a > 0) __stcs(dn, c - s);
              __stcs(up, c + s);
            }
            up += n;
            dn += n;
          }
        }
      } else {
        const int m = 128 * T.nt + ml, r = T.r0 + 64 * h, jn = min(64, T.rows - r);
        if (m < Lj && jn > 0) {
          float2* V = sg.buf_out + (size_t)r * Lj + m;
          const float os = sg.scale;  // 2 pi / n
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            if (j < jn) *V = make_float2(acc[0][j] * os, acc[1][j] * os);
            V += Lj;
          }
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (w == 1) {
    // After a give-up, whichever role's it was (every role has left its loop): the
    // copies and products in flight, in bounded waits, before TMEM goes
    if (lane == 0 && s_fail) {
      for (int g = max(0, s_loaded - kSgStages); g < s_loaded; ++g)
        tc::mbar_wait(bfull(g % kSgStages), (uint32_t)(g / kSgStages) & 1u, tc::kWaitCycles);
      if (s_issued > 0) tc::mbar_wait(btfull((s_issued - 1) & 1), (uint32_t)((s_issued - 1) / 2) & 1u, tc::kWaitCycles);
      atomicAdd(&g_sg_timeouts, 1);
    }
    __syncwarp();
    tc::tmem_free(tmem, 512);
  }
}

// Basis images of a grid, all its tables in one launch (a launch per table, with
// FP64 arithmetic and 2-byte stores per element, took 63 us of a new plan at L =
// 723 and 425 at L = 2048; now with the roots 25 and 152).
// Roots: trig values of the three periods, split once per root instead of once
// per element: {cos hi, cos lo, sin hi, sin lo} of 2^14 e^{2 pi i u / period}, the
// scaled coefficient 2 of the analyses (1 only where the angle is 0) and 1 of the
// alpha synthesis; FP64 values for the beta synthesis, whose terms carry q_b.
struct SgRoots {
  double2* beta64;                 // 8 L
  uint2 *beta, *beta_mw, *alpha;   // 8 L, 2 (2L - 1), 2L - 1
  int n[3];
};
__device__ __forceinline__ uint32_t sg_split(double v) {  // hi | lo << 16
  const __half hi = __double2half(v);
  const __half lo = __double2half(v - (double)__half2float(hi));
  return (uint32_t)__half_as_ushort(hi) | ((uint32_t)__half_as_ushort(lo) << 16);
}
__global__ void __launch_bounds__(256) k_sg_roots(SgRoots t) {
  int u = blockIdx.x * 256 + threadIdx.x, k = 0;
  while (k < 3 && u >= t.n[k]) u -= t.n[k++];
  if (k == 3) return;
  double s, c;
  sincospi(2.0 * u / t.n[k], &s, &c);
  (k == 0 ? t.beta : (k == 1 ? t.beta_mw : t.alpha))[u] =
      make_uint2(sg_split(c * kSgAlphaSynScale), sg_split(s * kSgAlphaSynScale));
  if (k == 0) t.beta64[u] = make_double2(c, s);
}

struct SgBuild {  // one table of the launch
  unsigned char* out;
  int mode, mw, tiles, stages, first;  // first block
};
struct SgBuilds {
  SgBuild t[5];
  int n;
};
// A thread writes 16 bytes of both images: eight positions k of one row r of (set,
// tile, stage, product).  Term of position k: 2 t + u holds term t + 16 u of the
// stage; the synthesis of beta keeps its terms in order (four b per store).
__global__ void __launch_bounds__(256) k_sg_basis(SgBuilds b, SgRoots roots, const double* __restrict__ qw, int L, double syn_scale) {
  int job = 0;
  while (job + 1 < b.n && (int)blockIdx.x >= b.t[job + 1].first) ++job;
  const SgBuild& t = b.t[job];
  const int idx = (blockIdx.x - t.first) * 256 + threadIdx.x;
  const int r = idx & 127, kc = (idx >> 7) & 3, p = (idx >> 9) & 1, st = idx >> 10;  // st: (set * tiles + tile) * stages + stage
  const int c = st % t.stages, tile = (st / t.stages) % t.tiles, set = st / (t.stages * t.tiles);
  const int row = 128 * tile + r, mode = t.mode, period = roots.n[t.mw ? 1 : (mode >= SG_ALPHA_ANA ? 2 : 0)];
  const uint2* __restrict__ tab = t.mw ? roots.beta_mw : (mode >= SG_ALPHA_ANA ? roots.alpha : roots.beta);
  uint32_t w[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 8 * kc + i, term = kSgK * c + (mode == SG_BETA_SYN ? k : (k >> 1) + 16 * (k & 1));
    w[i] = 0;
    if (mode == SG_BETA_ANA) {  // row: b, term: i of m' = 2 i + p; set 1: sin
      const int mp = 2 * term + p;
      if (row < L && mp < L) {
        const uint2 e = tab[mp * (2 * row + 1) % period];
        w[i] = mp == 0 ? (set ? 0u : sg_split(kSgAnaScale)) : (set ? e.y : e.x);
      }
    } else if (mode == SG_BETA_SYN) {  // row: i of m', term: b; product 0: even m' (cos) or odd (sin)
      const int mp = 2 * row + (p ^ set);
      if (term < L && mp < L) {
        const double2 e = roots.beta64[mp * (2 * term + 1) % period];
        w[i] = sg_split((mp == 0 ? 1.0 : 2.0) * qw[term] * (set ? e.y : e.x) * syn_scale);
      }
    } else {  // alpha, analysis: row a, term m; synthesis: row m, term a; product 1: -sin
      if (row < L && term < L) {
        const uint2 e = tab[term * row % period];
        w[i] = p ? e.y ^ 0x80008000u : (mode == SG_ALPHA_ANA && term == 0 ? sg_split(kSgAnaScale) : e.x);
      }
    }
  }
  unsigned char* q = t.out + (size_t)st * kHalf + (size_t)(2 * p) * kImg + sg_off(r, 8 * kc);
  uint4 hi, lo;
  uint32_t* h = &hi.x;
  uint32_t* l = &lo.x;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
    l[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
  }
  *reinterpret_cast<uint4*>(q) = hi;
  *reinterpret_cast<uint4*>(q + kImg) = lo;
}

// power of two that brings the synthesis beta basis, |2 q_b| < 4 / L, up to 2^14
double beta_syn_scale(int L) {
  double s = 4096.0;
  for (int x = L; x > 1; x >>= 1) s *= 2.0;
  return s;
}

int sg_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

}  // namespace

// Table of mode `mode` for grids of band-limit L: basis tiles and stages
// (a scale of band L_j uses a prefix of the tiles or of the stages).
SgTable sg_table(int mode, int L) {
  const int half = (L + 1) / 2;
  SgTable t;
  switch (mode) {
    case SG_BETA_ANA: t = {2, (L + 127) / 128, (half + kSgK - 1) / kSgK}; break;
    case SG_BETA_SYN: t = {2, (half + 127) / 128, (L + kSgK - 1) / kSgK}; break;
    default: t = {1, (L + 127) / 128, (L + kSgK - 1) / kSgK}; break;
  }
  t.bytes = (size_t)t.sets * t.tiles * t.stages * kHalf;
  return t;
}
// scale of a segment: the inverse of the basis scale (a power of two); alpha
// synthesis: Eq. (37)'s 2 pi / n
float sg_out_scale(int mode, int L) {
  if (mode == SG_BETA_SYN) return (float)(1.0 / beta_syn_scale(L));
  if (mode == SG_ALPHA_SYN) return (float)(2.0 * 3.14159265358979323846 / (2 * L - 1));
  return 1.f / kSgAnaScale;
}
// tiles of one segment: prod of data tiles and basis tiles (P), stages
SgDims sg_dims(int mode, int L, int Lj, int N, int nb) {
  SgDims d{0, 0, 0};
  if (Lj <= 0) return d;
  const int half = (Lj + 1) / 2, cols = N * 2 * ((half + 63) / 64), rows = (N * nb + 127) / 128;
  switch (mode) {
    case SG_BETA_ANA: d = {cols, (L + 127) / 128, (half + kSgK - 1) / kSgK}; break;
    case SG_BETA_SYN: d = {cols, (half + 127) / 128, (L + kSgK - 1) / kSgK}; break;
    case SG_ALPHA_ANA: d = {rows, (L + 127) / 128, (Lj + kSgK - 1) / kSgK}; break;
    default: d = {rows, (Lj + 127) / 128, (L + kSgK - 1) / kSgK}; break;
  }
  return d;
}

// scratch of the build, double2
size_t sg_build_scratch(int L) { return 16 * (size_t)L; }
// Tables out[k] (null: not wanted) of a grid of band-limit L, k the modes and 4: mode 0
// on the DH samples of an MW grid, whose own mode 0 evaluates at the MW samples.
// qw: quadrature weights q_b.
cudaError_t sg_build_tables(void* const* out, double2* scratch, const double* qw, int L, bool mw, cudaStream_t st) {
  SgRoots r;
  r.n[0] = 8 * L, r.n[1] = 2 * (2 * L - 1), r.n[2] = 2 * L - 1;
  r.beta64 = scratch;
  r.beta = reinterpret_cast<uint2*>(scratch + r.n[0]);
  r.beta_mw = r.beta + r.n[0];
  r.alpha = r.beta_mw + r.n[1];
  SgBuilds b;
  b.n = 0;
  int blocks = 0;
  for (int k = 0; k < 5; ++k) {
    if (!out[k]) continue;
    const int mode = k == 4 ? 0 : k;
    const SgTable t = sg_table(mode, L);
    b.t[b.n++] = SgBuild{reinterpret_cast<unsigned char*>(out[k]), mode, mw && k == 0, t.tiles, t.stages, blocks};
    blocks += t.sets * t.tiles * t.stages * 4;
  }
  if (blocks == 0) return cudaSuccess;
  k_sg_roots<<<(r.n[0] + r.n[1] + r.n[2] + 255) / 256, 256, 0, st>>>(r);
  k_sg_basis<<<blocks, 256, 0, st>>>(b, r, qw, L, beta_syn_scale(L));
  return cudaGetLastError();
}

namespace {
template <int MODE>
void sg_launch(const CztSeg<float>* segs, int nseg, int total, int stages, const CallPtrs& ptrs, cudaStream_t st,
               long long limit) {
  launch_after(k_sg_convert<MODE>, stages, 32 * kCvWarps, kData, st, segs, nseg, ptrs);
  launch_after(k_split_gemm<MODE>, std::min(total, sg_sms()), kSgThreads, kSgSmem, st, segs, nseg, total, ptrs, limit);
}
template <int MODE>
cudaError_t sg_attr() {
  return cudaFuncSetAttribute(k_split_gemm<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSgSmem);
}
}  // namespace

// total: output tiles, stages: data stages of the launch (two launches); limit:
// cycles of the products' bounded waits
void launch_split_gemm(int mode, const CztSeg<float>* segs, int nseg, int total, int stages, const CallPtrs& ptrs,
                       cudaStream_t st, long long limit) {
  if (total <= 0) return;
  switch (mode) {
    case SG_BETA_ANA: sg_launch<SG_BETA_ANA>(segs, nseg, total, stages, ptrs, st, limit); break;
    case SG_BETA_SYN: sg_launch<SG_BETA_SYN>(segs, nseg, total, stages, ptrs, st, limit); break;
    case SG_ALPHA_ANA: sg_launch<SG_ALPHA_ANA>(segs, nseg, total, stages, ptrs, st, limit); break;
    default: sg_launch<SG_ALPHA_SYN>(segs, nseg, total, stages, ptrs, st, limit); break;
  }
}

cudaError_t split_gemm_prepare() {
  for (auto f : {sg_attr<SG_BETA_ANA>, sg_attr<SG_BETA_SYN>, sg_attr<SG_ALPHA_ANA>, sg_attr<SG_ALPHA_SYN>})
    if (cudaError_t e = f(); e != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t split_gemm_timeouts(int* count) {
  cudaError_t e = cudaMemcpyFromSymbol(count, g_sg_timeouts, sizeof(int));
  if (e != cudaSuccess) return e;
  const int zero = 0;
  return cudaMemcpyToSymbol(g_sg_timeouts, &zero, sizeof(int));
}

}  // namespace s2dw
