// FP32 l-contraction for large band-limits (Sec. 3.2 Eq. (27); Sec. 3.3
// Eqs. (34), (32)), on pairs of 32-wide blocks p <= q:
//   analysis  G^j_{m'mk} = sum_{l in supp j} Delta^l_{m'm} f_lm R^j_{l m' k},
//             then the gamma step (Eq. (28)) as an epilogue into Y^j_g[m][m'];
//   synthesis partial_l(m) = sum_{m' in tile} Delta^l_{m'm} sum_{j,k} R^j_{l m' k} H^j_{m'mk},
//             H from Vhat by the gamma quadrature (Eq. (39)) as a prologue.
//
// Data.  The pair table stores, for l = 32q .. Lmax-1 one after the other, the
// block D_l[r][c] = Delta^l_{32p+r, 32q+c}: one 4 KB run per l.  It serves tile
// A (m' in p, m in q) and, read transposed with the sign (-1)^{m'-m} (applied
// once, to G or H), tile B (m' in q, m in p), so Delta is read from HBM once.
// R rows and f values are runs too (RSp[b][l][slot][n_k >= 0][32],
// fP[b][l][re, im][32]); a pipeline stage of eight l is five 1-D bulk copies
// issued by one thread into a ring of four stages.
//
// What bounds it: the FP32 pipe (per l and element of a tile a product with f
// and one multiply-add per slot and order n_k >= 0) against shared-memory
// reads, which return 128 bytes per cycle and SM whatever the broadcast.  A
// thread that owns 4 rows x 1 column reads 30 words per l for 14 packed FMA
// pairs of work; one that owns 2 rows x 8 columns reads 44 for 56.  Sixteen
// elements fit in 255 registers only because a warp handles the l of one
// parity (N = 5 and 6 spill 12 to 24 bytes per thread all the same): the sums
// over even and odd l of an order pair +-n are separate banks (R_{l m' -n} =
// (-1)^{l+m'} R_{l m' n}), and here the two banks live in different warps, which
// exchange halves through shared memory at the end (analysis) or fold H for
// their parity at the start (synthesis).
// Task: in the analysis two adjacent scales (one per slot) over the union of
// their l ranges, so that no accumulator changes scale on the way; in the
// synthesis an l range on which each slot holds one scale.  Where only one of
// the two is active, only its half of the sums runs.
//
// Threads: 256.  HALVES = 2 (at most six accumulated orders per element, N <=
// 6): tiles A and B of the pair, two warps per tile and parity, 16 elements per
// thread.  HALVES = 1 (N > 6): one tile per CTA, four warps per parity, 8
// elements.  Analysis: 2 rows x 8 (4) columns, tile A pairing columns for the
// packed arithmetic, tile B rows (the contiguous direction of the stored
// block).  Synthesis: 4 rows x 4 (2) columns, pairing rows: its sums over m'
// then leave half as many values to add across lanes per l (2 x 8 with its
// sixteen-value butterfly: 0.455 ms at L = 1024, N = 5, 4 x 4: 0.415 ms).
// Lanes are placed so that the 8 or 16 lanes of a wide read's phase cover 128
// consecutive bytes; in the analysis of tile A at 8 columns a thread's two
// groups of four are 16 apart and the odd row groups take them in the other
// order.
//
// Measured (GB300, ms per call, analysis / synthesis; before: one tile pair per
// 512-thread CTA, 4 x 1 elements per thread, cp.async ring): L = 1024, N = 5
// 0.401 / 0.394 -> 0.307 / 0.380, N = 3 0.341 / 0.353 -> 0.239 / 0.279, N = 1
// 0.245 / 0.283 -> 0.205 / 0.221; L = 723, N = 6 0.229 / 0.240 -> 0.148 / 0.165;
// L = 2048, N = 8 4.26 / 4.89 -> 2.92 / 3.49.  At N = 5 the FP32 pipe is 48%
// (41%) busy, DRAM at 3.3 (2.7) TB/s; the copies alone take 0.19 (0.15) ms and
// the sums without copies 0.27 ms: two warps per scheduler leave fixed
// latencies exposed, more do not fit beside the accumulators.
//
// Every wait is bounded (about a second): a CTA that gives up issues no more
// copies, runs through what is left, waits for its own copies and counts the event
// for s2dw_wait_timeouts.
#pragma once

#include <type_traits>

#include "contract.cuh"
#include "tc.cuh"

namespace s2dw {

__device__ int g_pair_timeouts;  // bounded waits that gave up (read and reset by the host)

constexpr int kTileKL = 8;  // l per pipeline stage (tables are padded for it: kPairPadL)
static_assert(kTileKL <= kPairPadL, "tables are padded for a stage past the last l");

template <int N, int NSLOT, bool SYN, int HALVES>
struct TileGeom {
  static constexpr int NH = (N + 1) / 2;
  static constexpr int K = NSLOT * NH;            // accumulated orders per element
  static constexpr int KL = kTileKL, STAGES = 4, LAG = 2;  // a slot is refilled LAG stages after its read
  static constexpr int RROW = K * 32;             // floats of one l of one R block
  static constexpr int D_F = KL * 1024, R_F = KL * RROW, F_F = SYN ? 0 : KL * 64;
  static constexpr int R_OFF = D_F, F_OFF = R_OFF + HALVES * R_F;
  static constexpr int SIZE = F_OFF + HALVES * F_F;  // floats per stage
  static constexpr int NEL = HALVES == 2 ? 16 : 8;  // elements per thread
  static constexpr int NWA = 32 / NEL;            // warps of a tile per parity
  // synthesis, tile A: partial sums of its warps, [2 buffers][2 parities][4 l][NWA][32]
  static constexpr size_t RED_BYTES = SYN ? (size_t)2 * 2 * (KL / 2) * NWA * 32 * sizeof(float2) : 0;
  // synthesis: staged Vhat rows, [tile][2 buffers][32][33]
  static constexpr size_t STG_BYTES = SYN ? (size_t)HALVES * 2 * 32 * 33 * sizeof(float2) : 0;
  static constexpr size_t SMEM = (size_t)STAGES * SIZE * 4 + RED_BYTES + STG_BYTES;
  static_assert(SMEM <= 232448, "227 KB per CTA");
  static_assert(SYN || (size_t)NEL / 2 * K * 256 * sizeof(float2) <= (size_t)STAGES * SIZE * 4, "exchange fits in the ring");
};

// Non-blocking test of the phase of parity `par`.
__device__ __forceinline__ bool mbar_ready(uint32_t mbar, uint32_t par) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(par)
      : "memory");
  return ok != 0;
}
// Blocking wait (try_wait, system-dependent suspension) for the phase of
// parity `par`; false once *abort is set (by this or another thread) or after
// `limit` cycles, which sets it.
__device__ __noinline__ bool pair_wait_slow(uint32_t mbar, uint32_t par, volatile int* abort, long long limit) {
  const long long t0 = clock64();
  for (;;) {
    if (*abort) return false;
    if (clock64() - t0 >= limit) {
      *abort = 1;
      return false;
    }
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(par)
        : "memory");
    if (ok) return true;
  }
}
__device__ __forceinline__ bool pair_wait(uint32_t mbar, uint32_t par, volatile int* abort, long long limit) {
  return mbar_ready(mbar, par) || pair_wait_slow(mbar, par, abort, limit);
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes) {
  asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(mbar), "r"(bytes)
               : "memory");
}
// 1-D bulk copy global -> shared, completion on the mbarrier (16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}

// source addresses of the next stage, kept in shared memory (registers are
// short, and re-reading the descriptor would cost a global load per stage)
struct TileSrc {
  uint64_t d, r[2], f[2];
};

// a task's fields, unpacked
struct TileJob {
  int p, q, half, lstart, lend, j, j2;
  long long dbase;
};

struct TileCtx {
  const ContractDesc<float>* D;
  TileJob tk;
  float* ring;
  float2* red;
  float2* stg;
  const float2* cg;      // gamma factors in shared memory
  TileSrc* src;
  uint32_t ring_s, full_s, empty_s;
  volatile int* abort;
  long long limit;       // cycles of a bounded wait
  int lo[2], hi[2];      // l range of each slot's scale (empty: hi < lo)
};

// Ring of one CTA: thread 0 fills stage i into slot i % STAGES by bulk copies.
template <typename G, bool SYN, int HALVES>
struct TileRing {
  const TileCtx& x;
  int issued = 0;
  bool live = true;  // none of this thread's waits for a stage has given up
  __device__ __forceinline__ explicit TileRing(const TileCtx& c) : x(c) {}
  __device__ __forceinline__ void issue() {
    const uint32_t slot = (uint32_t)issued % G::STAGES, mb = x.full_s + 8u * slot;
    const uint32_t so = x.ring_s + slot * (uint32_t)(G::SIZE * 4);
    volatile TileSrc* q = x.src;
    mbar_expect(mb, (uint32_t)(G::SIZE * 4));
    const uint64_t d = q->d;
    bulk_load(so, reinterpret_cast<const void*>(d), G::D_F * 4, mb);
    q->d = d + G::D_F * 4;
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      const uint64_t r = q->r[h];
      bulk_load(so + (G::R_OFF + h * G::R_F) * 4, reinterpret_cast<const void*>(r), G::R_F * 4, mb);
      q->r[h] = r + G::R_F * 4;
      if (!SYN) {
        const uint64_t f = q->f[h];
        bulk_load(so + (G::F_OFF + h * G::F_F) * 4, reinterpret_cast<const void*>(f), G::F_F * 4, mb);
        q->f[h] = f + G::F_F * 4;
      }
    }
    ++issued;
  }
  // thread 0: the first stages (isb: the tile of a one-tile CTA)
  __device__ __forceinline__ void start(int nst, bool isb) {
    const ContractDesc<float>* D = x.D;
    x.src->d = reinterpret_cast<uint64_t>(D->dpair + x.tk.dbase);
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      const bool hb = HALVES == 2 ? h == 1 : isb;
      x.src->r[h] = reinterpret_cast<uint64_t>(D->RSp + ((size_t)(hb ? x.tk.q : x.tk.p) * D->Lr + x.tk.lstart) * G::RROW);
      if (!SYN)
        x.src->f[h] = reinterpret_cast<uint64_t>(reinterpret_cast<const float*>(D->fP) +
                                                 ((size_t)(hb ? x.tk.p : x.tk.q) * D->Lrf + x.tk.lstart) * 64);
    }
    for (int i = 0; i < min(nst, G::STAGES); ++i) issue();
  }
  // Data of stage i.  A wait that gave up changes nothing in the control flow (the
  // sums that follow shuffle over the whole warp, and stay in bounds whatever the
  // ring holds); the CTA's results are lost and counted.
  __device__ __forceinline__ const float* wait(int i) {
    const uint32_t slot = (uint32_t)i % G::STAGES;
    if (!pair_wait(x.full_s + 8u * slot, ((uint32_t)i / G::STAGES) & 1u, x.abort, x.limit)) live = false;
    return x.ring + slot * G::SIZE;
  }
  // This warp has read stage i; thread 0 refills the slot read LAG stages ago.  Not
  // after a give-up: the slot's last copy may be in flight, and its barrier takes
  // one arrival per phase.
  __device__ __forceinline__ void release(int i, int nst) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) tc::mbar_arrive(x.empty_s + 8u * ((uint32_t)i % G::STAGES));
    const int r = i - G::LAG;
    if (threadIdx.x == 0 && live && r >= 0 && r + G::STAGES < nst &&
        pair_wait(x.empty_s + 8u * ((uint32_t)r % G::STAGES), ((uint32_t)r / G::STAGES) & 1u, x.abort, x.limit))
      issue();
  }
  // once every warp has left its loop: a CTA that gave up, whichever warp's wait it
  // was, waits for its own copies before it may leave, and is counted
  __device__ __forceinline__ void finish() {
    __syncthreads();
    if (threadIdx.x == 0 && *x.abort) {
      for (int i = max(0, issued - G::STAGES); i < issued; ++i)
        tc::mbar_wait(x.full_s + 8u * ((uint32_t)i % G::STAGES), ((uint32_t)i / G::STAGES) & 1u, tc::kWaitCycles);
      atomicAdd(&g_pair_timeouts, 1);
    }
  }
};

// f(mask of the slots active at l)
template <int NSLOT, typename F>
__device__ __forceinline__ void tile_dispatch(const TileCtx& x, int l, F&& f) {
  int mask = 0;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s)
    if (l >= x.lo[s] && l <= x.hi[s]) mask |= 1 << s;
  if (mask == (1 << NSLOT) - 1) f(std::integral_constant<int, (1 << NSLOT) - 1>());
  else if (mask == 0) f(std::integral_constant<int, 0>());
  else if constexpr (NSLOT > 1) {
    if (mask == 1) f(std::integral_constant<int, 1>());
    else f(std::integral_constant<int, 2>());
  }
}

template <int N, int NSLOT, int CC, int HALVES, bool ISB>
__device__ __forceinline__ void tile_ana_body(const TileCtx& x) {
  using G = TileGeom<N, NSLOT, false, HALVES>;
  constexpr int NH = G::NH, K = G::K, KL = G::KL, E = CC, FULL = (1 << NSLOT) - 1;
  const ContractDesc<float>* __restrict__ D = x.D;
  const TileJob& tk = x.tk;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, par = w >> 2;
  const int w2 = HALVES == 2 ? (w & 1) : (w & 3);
  // tile A: lane = column group + NCG * row group; tile B: lane = row group + 16 * column group
  constexpr int NCG = CC == 8 ? 4 : 8;
  const int rgl = ISB ? (lane & 15) : lane / NCG, cgl = ISB ? (lane >> 4) : lane % NCG;
  const int r0 = ISB ? 2 * rgl : 2 * (w2 * (32 / NCG) + rgl);  // this thread's rows r0, r0 + 1 of its block
  // first column of its group g of four (tile A), or of all its columns (tile B)
  auto colg = [&](int g) { return ISB ? CC * (2 * w2 + cgl) + 4 * g : 4 * cgl + (CC == 8 ? 16 * ((g ^ rgl) & 1) : 0); };
  const int mp0 = 32 * (ISB ? tk.q : tk.p) + r0, cb = ISB ? tk.p : tk.q;
  const bool idle = ISB && tk.p == tk.q;  // a diagonal block has one tile
  const int l_start = tk.lstart, l_end = tk.lend;
  const int nst = (l_end - l_start + KL) / KL;
  const int hh = HALVES == 2 && ISB ? 1 : 0;
  TileRing<G, false, HALVES> ring(x);
  if (tid == 0) ring.start(nst, ISB);

  // element pairs e, orders k (slot s, n_k >= 0 index h: k = s NH + h).  Tile A:
  // e = 2 (column pair) + row, the pair being two columns; tile B: e = column,
  // the pair being the two rows.
  float2 ax[E][K], ay[E][K];
#pragma unroll
  for (int e = 0; e < E; ++e)
#pragma unroll
    for (int k = 0; k < K; ++k) ax[e][k] = ay[e][k] = make_float2(0.f, 0.f);

  // one l at position li of the stage; M: active slots (bit s)
  auto one = [&](const float* S, int li, auto mm) {
    constexpr int M = decltype(mm)::value;
    if constexpr (M == 0) return;
    const float* Dl = S + li * 1024;
    const float* Rl = S + G::R_OFF + hh * G::R_F + li * G::RROW + r0;
    float2 R[K];  // rows r0, r0 + 1
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((M >> (k / NH)) & 1) R[k] = *reinterpret_cast<const float2*>(Rl + k * 32);
#pragma unroll
    for (int g = 0; g < CC / 4; ++g) {  // four columns at a time
      const int c0 = colg(g);
      const float* fl = S + G::F_OFF + hh * G::F_F + li * 64 + c0;
      const float4 fa = *reinterpret_cast<const float4*>(fl), fb = *reinterpret_cast<const float4*>(fl + 32);
      if constexpr (!ISB) {
        const float2 fx2[2] = {make_float2(fa.x, fa.y), make_float2(fa.z, fa.w)};
        const float2 fy2[2] = {make_float2(fb.x, fb.y), make_float2(fb.z, fb.w)};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float4 d4 = *reinterpret_cast<const float4*>(Dl + (r0 + r) * 32 + c0);
          const float2 d[2] = {make_float2(d4.x, d4.y), make_float2(d4.z, d4.w)};
          const float2 tx[2] = {__fmul2_rn(d[0], fx2[0]), __fmul2_rn(d[1], fx2[1])};
          const float2 ty[2] = {__fmul2_rn(d[0], fy2[0]), __fmul2_rn(d[1], fy2[1])};
#pragma unroll
          for (int k = 0; k < K; ++k) {
            if (!((M >> (k / NH)) & 1)) continue;
            const float rs = r == 0 ? R[k].x : R[k].y;
            const float2 rv = make_float2(rs, rs);
#pragma unroll
            for (int cp = 0; cp < 2; ++cp) {
              const int e = 2 * (2 * g + cp) + r;
              ax[e][k] = __ffma2_rn(tx[cp], rv, ax[e][k]);
              ay[e][k] = __ffma2_rn(ty[cp], rv, ay[e][k]);
            }
          }
        }
      } else {
        const float fx[4] = {fa.x, fa.y, fa.z, fa.w}, fy[4] = {fb.x, fb.y, fb.z, fb.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int e = 4 * g + c;
          const float2 d = *reinterpret_cast<const float2*>(Dl + (c0 + c) * 32 + r0);
          const float2 tx = __fmul2_rn(d, make_float2(fx[c], fx[c])), ty = __fmul2_rn(d, make_float2(fy[c], fy[c]));
#pragma unroll
          for (int k = 0; k < K; ++k) {
            if (!((M >> (k / NH)) & 1)) continue;
            ax[e][k] = __ffma2_rn(tx, R[k], ax[e][k]);
            ay[e][k] = __ffma2_rn(ty, R[k], ay[e][k]);
          }
        }
      }
    }
  };
  // every slot active on [fa, fb]
  int fa = l_start, fb = l_end;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) fa = max(fa, x.lo[s]), fb = min(fb, x.hi[s]);

  for (int i = 0; i < nst; ++i) {
    const int l0 = l_start + KL * i;
    const float* S = ring.wait(i);
    if (!idle) {
      if (l0 >= fa && l0 + KL - 1 <= fb) {
#pragma unroll 1
        for (int ii = 0; ii < KL / 2; ++ii) one(S, 2 * ii + par, std::integral_constant<int, FULL>());
      } else {
#pragma unroll 1
        for (int ii = 0; ii < KL / 2; ++ii) {
          const int l = l0 + 2 * ii + par;
          if (l > l_end) break;
          tile_dispatch<NSLOT>(x, l, [&](auto mm) { one(S, 2 * ii + par, mm); });
        }
      }
    }
    ring.release(i, nst);
  }
  ring.finish();
  // Exchange: the threads of parity 0 finish the element pairs e < E/2, those
  // of parity 1 the others; each hands over its sums of the rest.
  constexpr int EH = E / 2;
  float2* ex = reinterpret_cast<float2*>(x.ring);
  if (!idle) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int e = 0; e < EH; ++e) {
        ex[((k * EH + e) * 2) * 256 + tid] = par == 0 ? ax[EH + e][k] : ax[e][k];
        ex[((k * EH + e) * 2 + 1) * 256 + tid] = par == 0 ? ay[EH + e][k] : ay[e][k];
      }
  }
  __syncthreads();
  if (idle) return;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int e = 0; e < EH; ++e) {
      const float2 ox = ex[((k * EH + e) * 2) * 256 + (tid ^ 128)], oy = ex[((k * EH + e) * 2 + 1) * 256 + (tid ^ 128)];
      // bank of lstart's parity into [e], the other into [EH + e]
      const float2 mx = par == 0 ? ax[e][k] : ax[EH + e][k], my = par == 0 ? ay[e][k] : ay[EH + e][k];
      ax[e][k] = par == 0 ? mx : ox, ay[e][k] = par == 0 ? my : oy;
      ax[EH + e][k] = par == 0 ? ox : mx, ay[EH + e][k] = par == 0 ? oy : my;
    }
  // this thread's columns u, each with the rows mp0, mp0 + 1
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int j = s == 0 ? tk.j : tk.j2;
    if (j < 0) continue;
    const int Lj = D->Lj[j];
    float2* __restrict__ Y = D->Y[j];
#pragma unroll
    for (int u = 0; u < CC / 2; ++u) {
      const int c = par * (CC / 2) + u, mp = mp0, m = 32 * cb + colg(c >> 2) + (c & 3);
      if (m >= Lj || mp >= Lj) continue;
      float2 y[2][N];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int e = ISB ? u : 2 * (u >> 1) + r;
        const bool up = ISB ? r == 1 : (u & 1);
        float2 b0[NH], b1[NH];
#pragma unroll
        for (int q = 0; q < NH; ++q) {
          const int k = s * NH + q;
          b0[q] = up ? make_float2(ax[e][k].y, ay[e][k].y) : make_float2(ax[e][k].x, ay[e][k].x);
          b1[q] = up ? make_float2(ax[EH + e][k].y, ay[EH + e][k].y) : make_float2(ax[EH + e][k].x, ay[EH + e][k].x);
        }
        // m and m' have the parities of u and r (CC/2 is even, mp0 and the column groups too)
        gamma_ana<N, float>(b0, b1, ((r + l_start + N - 1) & 1) == 0, x.cg, y[r]);
        const float fs = (ISB && ((r + u) & 1)) ? -1.f : 1.f;
#pragma unroll
        for (int g = 0; g < N; ++g) y[r][g] = cscale<float>(cmul_ipow<float>(y[r][g], (-m) & 3), fs);
      }
#pragma unroll
      for (int g = 0; g < N; ++g) {
        float2* dst = Y + ((size_t)g * Lj + m) * Lj + mp;
        if ((Lj & 1) == 0) {  // mp even: 16-byte aligned, and mp + 1 < Lj
          *reinterpret_cast<float4*>(dst) = make_float4(y[0][g].x, y[0][g].y, y[1][g].x, y[1][g].y);
        } else {
          dst[0] = y[0][g];
          if (mp + 1 < Lj) dst[1] = y[1][g];
        }
      }
    }
  }
}

// v[i] of this lane and of the lane `m` away, HALF values kept: the upper ones where `up`
template <int HALF>
__device__ __forceinline__ void fold_lanes(float* v, bool up, int m) {
#pragma unroll
  for (int i = 0; i < HALF; ++i) v[i] = (up ? v[i + HALF] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + HALF], m);
}

template <int N, int NSLOT, int C, int HALVES, bool ISB>
__device__ __forceinline__ void tile_syn_body(const TileCtx& x) {
  using G = TileGeom<N, NSLOT, true, HALVES>;
  constexpr int NH = G::NH, K = G::K, KL = G::KL, E = 2 * C, FULL = (1 << NSLOT) - 1;
  const ContractDesc<float>* __restrict__ D = x.D;
  const TileJob& tk = x.tk;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, par = w >> 2;
  const int w2 = HALVES == 2 ? (w & 1) : (w & 3);
  constexpr int NCG = 32 / C;  // tile A: lane = column group + NCG * row group; tile B: lane = row group + 8 * column group
  const int r0 = ISB ? 4 * (lane & 7) : 4 * (w2 * C + lane / NCG);  // rows r0 .. r0 + 3, columns c0 .. c0 + C - 1
  const int c0 = ISB ? C * (4 * w2 + (lane >> 3)) : C * (lane % NCG);
  const int rb = ISB ? tk.q : tk.p, cb = ISB ? tk.p : tk.q;
  const int mp0 = 32 * rb + r0, m0 = 32 * cb + c0;
  const bool idle = ISB && tk.p == tk.q;  // a diagonal block has one tile
  const int l_start = tk.lstart, l_end = tk.lend;
  const int nst = (l_end - l_start + KL) / KL;
  const int hh = HALVES == 2 && ISB ? 1 : 0;
  TileRing<G, true, HALVES> ring(x);
  if (tid == 0) ring.start(nst, ISB);
  const int Lp32 = D->Lp32;
  float2* __restrict__ P = D->P + ((size_t)rb * D->L + l_start) * Lp32 + 32 * cb;

  // H of the element pairs e = 2 c + r/2 (rows 2 rp, 2 rp + 1 of column c) for
  // this warp's parity of l (gamma adjoint).  The tile's Vhat is staged row by
  // row, one gamma sample at a time (loading each thread's 4 x C elements
  // straight from global memory touched 8 lines per load: 13 us per task), the
  // next sample's rows in flight meanwhile.
  constexpr int TW = G::NWA * 2, PITCH = 33;  // warps of this tile
  const int gi = HALVES == 2 ? par * 2 + w2 : w;
  float2* stg = x.stg + (HALVES == 2 && ISB ? 2 * 32 * PITCH : 0);
  float2 ax[E][K], ay[E][K];
  const bool ub = ((l_start + par + N - 1) & 1) == 0;  // "plus" for even m'
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int j = s == 0 ? tk.j : tk.j2;
    const int Lj = (j >= 0 && !idle) ? D->Lj[j] : 0;
    const float2* __restrict__ V = j >= 0 ? D->Y[j] : nullptr;
    float2 h[4 * C][NH];
#pragma unroll
    for (int i = 0; i < 4 * C; ++i)
#pragma unroll
      for (int q = 0; q < NH; ++q) h[i][q] = make_float2(0.f, 0.f);
    if (Lj > 0) {  // (the same for every warp of the tile)
      float2 nx[32 / TW];
      auto fetch = [&](int g) {
#pragma unroll
        for (int i = 0; i < 32 / TW; ++i) {
          const int mp = 32 * rb + gi * (32 / TW) + i, m = 32 * cb + lane;
          nx[i] = (mp < Lj && m < Lj) ? V[((size_t)g * Lj + mp) * Lj + m] : make_float2(0.f, 0.f);
        }
      };
      fetch(0);
#pragma unroll 1
      for (int g = 0; g < N; ++g) {
        float2* sb = stg + ((s * N + g) & 1) * 32 * PITCH;
#pragma unroll
        for (int i = 0; i < 32 / TW; ++i) sb[(gi * (32 / TW) + i) * PITCH + lane] = nx[i];
        if (g + 1 < N) fetch(g + 1);
        asm volatile("bar.sync %0, %1;" ::"n"(ISB ? 4 : 3), "n"(32 * TW) : "memory");
#pragma unroll
        for (int c = 0; c < C; ++c) {
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            // i^m: c0 is a multiple of C (m = c modulo 4 at C = 4, modulo 2 at C = 2)
            float2 u = cmul_ipow<float>(sb[(r0 + r) * PITCH + c0 + c], c & 3);
            if (C == 2 && (c0 & 2)) u = make_float2(-u.x, -u.y);
            gamma_syn_add<N, float>(h[4 * c + r], cscale<float>(u, (ISB && ((r + c) & 1)) ? -1.f : 1.f), ub == ((r & 1) == 0), x.cg,
                             g);
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int rp = 0; rp < 2; ++rp)
#pragma unroll
        for (int q = 0; q < NH; ++q) {
          const float2 u0 = h[4 * c + 2 * rp][q], u1 = h[4 * c + 2 * rp + 1][q];
          ax[2 * c + rp][s * NH + q] = make_float2(u0.x, u1.x);
          ay[2 * c + rp][s * NH + q] = make_float2(u0.y, u1.y);
        }
  }

  // one l at position li of the stage; M: active slots (bit s)
  auto one = [&](const float* S, int li, auto mm, float2* redl, int l) {
    constexpr int M = decltype(mm)::value;
    const float* Dl = S + li * 1024;
    const float* Rl = S + G::R_OFF + hh * G::R_F + li * G::RROW + r0;
    float v[2 * C];  // column c: (v[2c], v[2c + 1])
#pragma unroll
    for (int i = 0; i < 2 * C; ++i) v[i] = 0.f;
    float db[C][4];  // tile B: the columns' Delta
    if constexpr (ISB) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const float4 d4 = *reinterpret_cast<const float4*>(Dl + (c0 + c) * 32 + r0);
        db[c][0] = d4.x, db[c][1] = d4.y, db[c][2] = d4.z, db[c][3] = d4.w;
      }
    }
#pragma unroll
    for (int rp = 0; rp < 2; ++rp) {
      float2 R[K];
#pragma unroll
      for (int k = 0; k < K; ++k)
        if ((M >> (k / NH)) & 1) R[k] = *reinterpret_cast<const float2*>(Rl + k * 32 + 2 * rp);
      float da[2][C];
      if constexpr (!ISB) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          if constexpr (C == 4) {
            const float4 d4 = *reinterpret_cast<const float4*>(Dl + (r0 + 2 * rp + r) * 32 + c0);
            da[r][0] = d4.x, da[r][1] = d4.y, da[r][C > 2 ? 2 : 0] = d4.z, da[r][C > 2 ? 3 : 0] = d4.w;
          } else {
            const float2 d2 = *reinterpret_cast<const float2*>(Dl + (r0 + 2 * rp + r) * 32 + c0);
            da[r][0] = d2.x, da[r][1] = d2.y;
          }
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        float2 sx = make_float2(0.f, 0.f), sy = sx;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if (!((M >> (k / NH)) & 1)) continue;
          sx = __ffma2_rn(ax[2 * c + rp][k], R[k], sx);
          sy = __ffma2_rn(ay[2 * c + rp][k], R[k], sy);
        }
        const float d0 = ISB ? db[c][2 * rp] : da[0][c], d1 = ISB ? db[c][2 * rp + 1] : da[1][c];
        v[2 * c] = __fmaf_rn(d1, sx.y, __fmaf_rn(d0, sx.x, v[2 * c]));
        v[2 * c + 1] = __fmaf_rn(d1, sy.y, __fmaf_rn(d0, sy.x, v[2 * c + 1]));
      }
    }
    if constexpr (!ISB) {
      // over the row groups (lane bits above the column groups): half the columns per step
      int col = c0;
      if constexpr (C == 4) {
        fold_lanes<4>(v, lane & 16, 16);
        fold_lanes<2>(v, lane & 8, 8);
        col += ((lane & 16) ? 2 : 0) + ((lane & 8) ? 1 : 0);
      } else {
        fold_lanes<2>(v, lane & 16, 16);
        col += (lane & 16) ? 1 : 0;
      }
      redl[w2 * 32 + col] = make_float2(v[0], v[1]);
    } else {
      // over the eight row groups (lane bits 0..2)
      float* Pr = reinterpret_cast<float*>(P + (size_t)(l - l_start) * Lp32 + c0);
      if constexpr (C == 4) {
        fold_lanes<4>(v, lane & 4, 4);
        fold_lanes<2>(v, lane & 2, 2);
        fold_lanes<1>(v, lane & 1, 1);
        Pr[lane & 7] = v[0];
      } else {
        fold_lanes<2>(v, lane & 4, 4);
        fold_lanes<1>(v, lane & 2, 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if (!(lane & 1)) Pr[(lane & 7) >> 1] = v[0];
      }
    }
  };
  // every slot active on [fa, fb]
  int fa = l_start, fb = l_end;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) fa = max(fa, x.lo[s]), fb = min(fb, x.hi[s]);

  for (int i = 0; i < nst; ++i) {
    const int l0 = l_start + KL * i;
    float2* redb = x.red + (size_t)(((i & 1) * 2 + par) * (KL / 2)) * G::NWA * 32;
    const float* S = ring.wait(i);
    if (!idle) {
      if (l0 >= fa && l0 + KL - 1 <= fb) {
#pragma unroll 1
        for (int ii = 0; ii < KL / 2; ++ii)
          one(S, 2 * ii + par, std::integral_constant<int, FULL>(), redb + ii * G::NWA * 32, l0 + 2 * ii + par);
      } else {
#pragma unroll 1
        for (int ii = 0; ii < KL / 2; ++ii) {
          const int l = l0 + 2 * ii + par;
          if (l > l_end) break;
          tile_dispatch<NSLOT>(x, l, [&](auto mm) { one(S, 2 * ii + par, mm, redb + ii * G::NWA * 32, l); });
        }
      }
    }
    ring.release(i, nst);
    if constexpr (!ISB) {
      // the partial sums of tile A's warps of this parity
      asm volatile("bar.sync %0, %1;" ::"r"(1 + par), "n"(32 * G::NWA) : "memory");
#pragma unroll
      for (int ii = w2; ii < KL / 2; ii += G::NWA) {
        const int l = l0 + 2 * ii + par;
        if (l <= l_end) {
          float2 sum = redb[ii * G::NWA * 32 + lane];
#pragma unroll
          for (int k = 1; k < G::NWA; ++k) {
            const float2 u = redb[(ii * G::NWA + k) * 32 + lane];
            sum.x += u.x;
            sum.y += u.y;
          }
          P[(size_t)(l - l_start) * Lp32 + lane] = sum;
        }
      }
    }
  }
  ring.finish();
}

template <int N, int NSLOT, bool SYN, int HALVES>
__global__ void __launch_bounds__(256, 1)
k_contract_tile(const ContractDesc<float>* __restrict__ descs, const CTask* __restrict__ tasks, long long limit) {
  begin_after();
  using G = TileGeom<N, NSLOT, SYN, HALVES>;
  extern __shared__ __align__(128) unsigned char tile_smem[];
  __shared__ __align__(8) uint64_t full[G::STAGES], empty[G::STAGES];
  __shared__ float2 cg[64];
  __shared__ TileSrc src;
  __shared__ int s_abort;
  TileCtx x;
  const CTask tk = tasks[blockIdx.x];
  x.tk = TileJob{tk.p, tk.q, tk.half, tk.lstart, tk.lend, tk.j, tk.j2, tk.dbase()};
  x.D = descs + tk.prob;
  x.ring = reinterpret_cast<float*>(tile_smem);
  x.red = reinterpret_cast<float2*>(tile_smem + (size_t)G::STAGES * G::SIZE * 4);
  x.stg = reinterpret_cast<float2*>(tile_smem + (size_t)G::STAGES * G::SIZE * 4 + G::RED_BYTES);
  x.cg = cg;
  x.src = &src;
  x.ring_s = tc::smem_u32(x.ring);
  x.full_s = tc::smem_u32(&full[0]);
  x.empty_s = tc::smem_u32(&empty[0]);
  x.abort = &s_abort;
  x.limit = limit;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int j = s == 0 ? x.tk.j : x.tk.j2;
    x.lo[s] = j >= 0 ? x.D->jlo[j] : 0;
    x.hi[s] = j >= 0 ? x.D->jhi[j] : -1;
  }
  if (threadIdx.x < N * N) cg[threadIdx.x] = SYN ? x.D->cgs[threadIdx.x] : x.D->cga[threadIdx.x];
  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < G::STAGES; ++s) {
      tc::mbar_init(x.full_s + 8 * s, 1);
      tc::mbar_init(x.empty_s + 8 * s, 8);
    }
  }
  __syncthreads();
  const bool isb = HALVES == 2 ? ((threadIdx.x >> 6) & 1) : x.tk.half == 1;
  if constexpr (SYN) {
    constexpr int C = HALVES == 2 ? 4 : 2;
    if (!isb) tile_syn_body<N, NSLOT, C, HALVES, false>(x);
    else tile_syn_body<N, NSLOT, C, HALVES, true>(x);
  } else {
    constexpr int CC = HALVES == 2 ? 8 : 4;
    if (!isb) tile_ana_body<N, NSLOT, CC, HALVES, false>(x);
    else tile_ana_body<N, NSLOT, CC, HALVES, true>(x);
  }
}

}  // namespace s2dw
