// l-contraction for small and middle band-limits (Sec. 3.2 Eq. (27);
// Sec. 3.3 Eqs. (34), (32)): the sums of contract_tile.cuh, organised for
// latency instead of for one long stream per CTA.
//
// What bounds it.  At small L a whole contraction is a few microseconds of FP32
// work; a ring kernel with one CTA per 32 x 32 tile (pair)
// walks its l one stage after the other, at L = 128 on 16 of 152 SMs for 128
// dependent steps.  Here
//   analysis: a task is one scale of one tile over that scale's own l range, so
//     the scales run side by side and the gamma step runs once, at the end; a
//     thread owns RT rows x 1 column and keeps its accumulators; a task is cut
//     into 32 / (RT warps) CTAs, RT chosen so that the launch fills the SMs
//     (RT does not enter the arithmetic);
//   synthesis: a tile's l range is cut at the changes of scale and further (the
//     sums over m' of different l are independent), each CTA loading the H
//     values of its own range once.
// Delta goes from the pair table straight to registers, the next l group in
// flight while the current one is summed; the R rows and f values of 16 l are
// staged in shared memory by cp.async, double-buffered, one barrier per 16 l.
// Lanes run along the second index of the stored block D_l[r][c] =
// Delta^l_{32p+r, 32q+c} in both tiles of a pair, so every Delta load is one
// 128-byte line: tile A (m' in p, m in q) has lanes along m, tile B
// (m' in q, m in p; Delta_{m'm} = (-1)^{m'-m} Delta_{mm'}) lanes along m'.
// The scaling part's tiles (N = 1, one slot) ride in the same launch.
//
// FP64.  The FP64 pipes bound it (two multiply-adds per cycle and SM: a warp's
// multiply-add holds its quarter of the SM for 64 cycles, so loads, registers
// and barriers hide behind them), and what counts is that every SM has the same
// number of them: the analysis always runs one row per thread, the synthesis
// takes half tiles (kDirSynSub).
#pragma once

#include "contract.cuh"

namespace s2dw {

namespace {

template <typename T>
constexpr int kDirLC = sizeof(T) == 4 ? 16 : 8;  // l per shared-memory stage

// CTAs per synthesis task, each 32 / kDirSynSub rows of the stored block
template <typename T>
constexpr int kDirSynSub = sizeof(T) == 4 ? 1 : 2;

// f(integral_constant<0>) .. f(integral_constant<K - 1>), unrolled
template <int K, typename F>
__device__ __forceinline__ void dir_unroll(F&& f) {
  if constexpr (K > 0) {
    dir_unroll<K - 1>(f);
    f(std::integral_constant<int, K - 1>());
  }
}

// one complex value, or zero where !ok
__device__ __forceinline__ void cp_async_c(float2* smem, const float2* gmem, bool ok) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_c(double2* smem, const double2* gmem, bool ok) {
  cp_async16(smem, gmem, ok ? 16 : 0);
}

template <typename T, int RT>
__device__ __forceinline__ void lds_rows(const T* p, T (&r)[RT]) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int e = 0; e < RT; ++e) r[e] = p[e];  // (16-byte loads where RT is even)
  } else if constexpr (RT == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    r[0] = v.x, r[1] = v.y, r[2] = v.z, r[3] = v.w;
  } else if constexpr (RT == 2) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    r[0] = v.x, r[1] = v.y;
  } else {
    r[0] = *p;
  }
}

// One scale of one tile: G^j over l in [lstart, lend], then the gamma step.
// nslot: slots of the R rows (the scale's values sit in slot tk.slot).
template <typename T, int N, int RT, int NW, bool ISB>
__device__ __forceinline__ void dir_ana_tile(const ContractDesc<T>* __restrict__ D, int nslot, const CTask& tk, int sub,
                                             const cx<T>* __restrict__ f, cx<T>* cg, T* Rs0, cx<T>* fs0) {
  constexpr int NH = (N + 1) / 2, ZH = N & 1, NP = N / 2, RW = NH * 32, LC = kDirLC<T>;
  constexpr int EPC = 16 / (int)sizeof(T);  // values per 16-byte copy
  constexpr int NTH = 32 * NW, U = RT == 4 ? 4 : 8;  // (LC = 8 at FP64: static shared memory)
  static_assert(LC % U == 0 && U % 2 == 0, "the parity of a position is its l's relative to lstart");
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int rw = (sub * NW + w) * RT;  // first row of the stored block
  const int l_start = tk.lstart, l_end = tk.lend, rrow = nslot * RW;
  const T* __restrict__ dp = D->dpair + tk.dbase() + rw * 32 + lane;
  const T* __restrict__ Rg = D->RSp + ((size_t)(ISB ? tk.q : tk.p) * D->Lr + l_start) * rrow + tk.slot * RW;
  const int mb = 32 * (ISB ? tk.p : tk.q);  // m block of f
  const int Lj = D->Lj[tk.j];
  cx<T>* __restrict__ Y = D->Y[tk.j];
  for (int i = t; i < N * N; i += NTH) cg[i] = D->cga[i];

  auto stage = [&](int ch) {  // R rows and f of l_start + 16 ch .., zero past l_end
    T* Rs = Rs0 + (ch & 1) * LC * RW;
    cx<T>* fs = fs0 + (ch & 1) * LC * 32;
    const int l0 = l_start + ch * LC;
    const T* src = Rg + (size_t)ch * LC * rrow;
    for (int i = t; i < LC * (RW / EPC); i += NTH) {
      const int r = i / (RW / EPC), c = EPC * (i % (RW / EPC));
      const bool ok = l0 + r <= l_end;
      cp_async16(Rs + r * RW + c, src + (ok ? (size_t)r * rrow + c : 0), ok ? 16 : 0);
    }
    for (int i = t; i < LC * 32; i += NTH) {
      const int l = l0 + (i >> 5), m = mb + (i & 31);
      const bool ok = m <= l && l <= l_end;
      cp_async_c(fs + i, f + (ok ? (size_t)l * l + l + m : 0), ok);
    }
    cp_async_commit();
  };

  T ax[RT][N], ay[RT][N];
#pragma unroll
  for (int e = 0; e < RT; ++e)
#pragma unroll
    for (int k = 0; k < N; ++k) ax[e][k] = ay[e][k] = T(0);

  T dn[U][RT], dc[U][RT] = {};  // Delta of the next and the current group
  auto fetch = [&](int l) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < RT; ++e) dn[u][e] = l + u <= l_end ? __ldg(dp + (size_t)(l - l_start + u) * 1024 + e * 32) : T(0);
  };
  auto compute = [&](const T* Rl, const cx<T>* fl, auto uu) {
    constexpr int u = decltype(uu)::value, BQ = (u & 1) * NP;
    T tx[RT], ty[RT];
    if constexpr (!ISB) {
      const cx<T> fv = fl[lane];
#pragma unroll
      for (int e = 0; e < RT; ++e) tx[e] = mul_rn(dc[u][e], fv.x), ty[e] = mul_rn(dc[u][e], fv.y);
    } else {
#pragma unroll
      for (int e = 0; e < RT; ++e) {
        const cx<T> fv = fl[rw + e];
        tx[e] = mul_rn(dc[u][e], fv.x), ty[e] = mul_rn(dc[u][e], fv.y);
      }
    }
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      const int q = (ZH && h == 0) ? 2 * NP : BQ + h - ZH;
      T r[RT];
      if constexpr (!ISB) {
        lds_rows<T, RT>(Rl + h * 32 + rw, r);
      } else {
        const T r0 = Rl[h * 32 + lane];
#pragma unroll
        for (int e = 0; e < RT; ++e) r[e] = r0;
      }
#pragma unroll
      for (int e = 0; e < RT; ++e) {
        ax[e][q] = fma_rn(tx[e], r[e], ax[e][q]);
        ay[e][q] = fma_rn(ty[e], r[e], ay[e][q]);
      }
    }
  };

  stage(0);
  fetch(l_start);
  const int nch = (l_end - l_start) / LC + 1;
  for (int ch = 0; ch < nch; ++ch) {
    cp_async_wait<0>();
    __syncthreads();  // this chunk's rows visible, the previous buffer free
    if (ch + 1 < nch) stage(ch + 1);
    const T* Rs = Rs0 + (ch & 1) * LC * RW;
    const cx<T>* fs = fs0 + (ch & 1) * LC * 32;
#pragma unroll 1
    for (int gi = 0; gi < LC; gi += U) {
      const int l0 = l_start + ch * LC + gi;
      if (l0 > l_end) break;
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < RT; ++e) dc[u][e] = dn[u][e];
      fetch(l0 + U);
      dir_unroll<U>([&](auto uu) { compute(Rs + (gi + decltype(uu)::value) * RW, fs + (gi + decltype(uu)::value) * 32, uu); });
    }
  }

  // gamma step (Eq. (28)) from the sums over the l of lstart's parity and of the other
#pragma unroll
  for (int e = 0; e < RT; ++e) {
    const int mp = ISB ? 32 * tk.q + lane : 32 * tk.p + rw + e;
    const int m = ISB ? 32 * tk.p + rw + e : 32 * tk.q + lane;
    if (mp >= Lj || m >= Lj) continue;
    cx<T> b0[NH], b1[NH], y[N];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      const int q0 = (ZH && h == 0) ? 2 * NP : h - ZH, q1 = (ZH && h == 0) ? -1 : NP + h - ZH;
      b0[h] = mkc<T>(ax[e][q0], ay[e][q0]);
      b1[h] = q1 < 0 ? mkc<T>(0, 0) : mkc<T>(ax[e][q1 < 0 ? 0 : q1], ay[e][q1 < 0 ? 0 : q1]);
    }
    gamma_ana<N, T>(b0, b1, ((mp + l_start + N - 1) & 1) == 0, cg, y);
    const T fs = (ISB && ((mp + m) & 1)) ? T(-1) : T(1);
#pragma unroll
    for (int g = 0; g < N; ++g)
      Y[((size_t)g * Lj + m) * Lj + mp] = cscale<T>(cmul_ipow<T>(y[g], (-m) & 3), fs);
  }
}

template <typename T, int N, int RT, int NW>
__global__ void __launch_bounds__(32 * NW)
k_contract_dir_ana(const ContractDesc<T>* __restrict__ dw, const CTask* __restrict__ tw, int nw,
                   const ContractDesc<T>* __restrict__ dphi, const CTask* __restrict__ tp, CallPtrs ptrs) {
  begin_after();
  constexpr int SUB = 32 / (RT * NW), RW = ((N + 1) / 2) * 32;
  __shared__ cx<T> cg[64];
  __shared__ __align__(16) T Rs[2 * kDirLC<T> * RW];
  __shared__ __align__(16) cx<T> fs[2 * kDirLC<T> * 32];
  const int i = blockIdx.x / SUB, sub = blockIdx.x % SUB;
  if (i < nw) {
    const CTask tk = tw[i];
    const cx<T>* f = reinterpret_cast<const cx<T>*>(ptrs.f[tk.prob]);
    if (tk.half == 0) dir_ana_tile<T, N, RT, NW, false>(dw + tk.prob, 2, tk, sub, f, cg, Rs, fs);
    else dir_ana_tile<T, N, RT, NW, true>(dw + tk.prob, 2, tk, sub, f, cg, Rs, fs);
  } else {
    const CTask tk = tp[i - nw];
    const cx<T>* f = reinterpret_cast<const cx<T>*>(ptrs.f[tk.prob]);
    if (tk.half == 0) dir_ana_tile<T, 1, RT, NW, false>(dphi + tk.prob, 1, tk, sub, f, cg, Rs, fs);
    else dir_ana_tile<T, 1, RT, NW, true>(dphi + tk.prob, 1, tk, sub, f, cg, Rs, fs);
  }
}

// Synthesis of one tile over l in [lstart, lend], a range on which the two
// slots hold constant scales (tk.j, tk.j2; -1: empty).  8 warps x 4 rows of the
// stored block.  Tile A sums its rows m' in the thread, then over the warps in
// shared memory; tile B's rows m' are the lanes: a butterfly that halves the
// values with the lanes leaves one column part per four lanes.  FP64: 4 rows of
// two slots do not fit the registers at N > 5 and the gamma adjoint alone is as
// long as 5 (N = 3) to 14 (N = 8) l, so a task is two CTAs of 2 rows per warp,
// each with its own block of partials (tile B: its own columns of the first).
template <typename T, int N, int NSLOT, bool ISB>
__device__ __forceinline__ void dir_syn_tile(const ContractDesc<T>* __restrict__ D, const CTask& tk, int sub, cx<T>* cg,
                                             T* Rs0, cx<T>* red) {
  constexpr int NH = (N + 1) / 2, ZH = N & 1, NP = N / 2, RROW = NSLOT * NH * 32, LC = kDirLC<T>;
  constexpr int SUB = kDirSynSub<T>, RT = 4 / SUB, EPC = 16 / (int)sizeof(T), NTH = 256, U = 4;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31, rw = (sub * 8 + w) * RT;
  const int l_start = tk.lstart, l_end = tk.lend;
  const int rb = ISB ? tk.q : tk.p, cb = ISB ? tk.p : tk.q, L = D->L, Lp32 = D->Lp32;
  const T* __restrict__ dp = D->dpair + tk.dbase() + rw * 32 + lane;
  const T* __restrict__ Rg = D->RSp + ((size_t)rb * D->Lr + l_start) * RROW;
  cx<T>* __restrict__ P = D->P + ((size_t)(rb * SUB + (ISB ? 0 : sub)) * L + l_start) * Lp32 + 32 * cb;

  auto stage = [&](int ch) {
    T* Rs = Rs0 + (ch & 1) * LC * RROW;
    const int nl = l_end - l_start - ch * LC + 1;
    const T* src = Rg + (size_t)ch * LC * RROW;
    for (int i = t; i < LC * (RROW / EPC); i += NTH) {
      const bool ok = i / (RROW / EPC) < nl;
      cp_async16(Rs + EPC * i, src + (ok ? EPC * i : 0), ok ? 16 : 0);
    }
    cp_async_commit();
  };
  T dn[U][RT], dc[U][RT] = {};
  auto fetch = [&](int l) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < RT; ++e) dn[u][e] = l + u <= l_end ? __ldg(dp + (size_t)(l - l_start + u) * 1024 + e * 32) : T(0);
  };
  stage(0);
  fetch(l_start);
  for (int i = t; i < N * N; i += NTH) cg[i] = D->cgs[i];
  __syncthreads();

  // gamma adjoint (Eq. (39)) of both slots, folded into the parity banks
  T hx[RT][NSLOT][N], hy[RT][NSLOT][N];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int j = s == 0 ? tk.j : tk.j2;
    const int Lj = j >= 0 ? D->Lj[j] : 0;
    const cx<T>* __restrict__ V = j >= 0 ? D->Y[j] : nullptr;
#pragma unroll
    for (int e = 0; e < RT; ++e) {
      const int mp = ISB ? 32 * tk.q + lane : 32 * tk.p + rw + e;
      const int m = ISB ? 32 * tk.p + rw + e : 32 * tk.q + lane;
      cx<T> h0[NH], h1[NH];  // banks of lstart's parity and of the other
#pragma unroll
      for (int h = 0; h < NH; ++h) h0[h] = h1[h] = mkc<T>(0, 0);
      if (mp < Lj && m < Lj) {
        cx<T> vg[N];
#pragma unroll
        for (int g = 0; g < N; ++g) vg[g] = V[((size_t)g * Lj + mp) * Lj + m];
        const T fs = (ISB && ((mp + m) & 1)) ? T(-1) : T(1);
        const bool plus = ((mp + l_start + N - 1) & 1) == 0;
#pragma unroll
        for (int g = 0; g < N; ++g) {
          const cx<T> v = cscale<T>(cmul_ipow<T>(vg[g], m & 3), fs);
          gamma_syn_add<N, T>(h0, v, plus, cg, g);
          gamma_syn_add<N, T>(h1, v, !plus, cg, g);
        }
      }
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const int q0 = (ZH && h == 0) ? 2 * NP : h - ZH;
        hx[e][s][q0] = h0[h].x, hy[e][s][q0] = h0[h].y;
        if (!(ZH && h == 0)) hx[e][s][q0 + NP] = h1[h].x, hy[e][s][q0 + NP] = h1[h].y;
      }
    }
  }
  auto compute = [&](const T* Rl, int li, int l, auto uu) {
    constexpr int u = decltype(uu)::value, BQ = (u & 1) * NP;
    T px[RT], py[RT];
#pragma unroll
    for (int e = 0; e < RT; ++e) px[e] = py[e] = T(0);
#pragma unroll
    for (int s = 0; s < NSLOT; ++s)
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const int q = (ZH && h == 0) ? 2 * NP : BQ + h - ZH;
        T r[RT];
        if constexpr (!ISB) {
          lds_rows<T, RT>(Rl + (s * NH + h) * 32 + rw, r);
        } else {
          const T r0 = Rl[(s * NH + h) * 32 + lane];
#pragma unroll
          for (int e = 0; e < RT; ++e) r[e] = r0;
        }
#pragma unroll
        for (int e = 0; e < RT; ++e) {
          px[e] = fma_rn(hx[e][s][q], r[e], px[e]);
          py[e] = fma_rn(hy[e][s][q], r[e], py[e]);
        }
      }
    if constexpr (!ISB) {
      cx<T> v = mkc<T>(mul_rn(dc[u][0], px[0]), mul_rn(dc[u][0], py[0]));
#pragma unroll
      for (int e = 1; e < RT; ++e) v.x = fma_rn(dc[u][e], px[e], v.x), v.y = fma_rn(dc[u][e], py[e], v.y);
      red[(li * 8 + w) * 32 + lane] = v;
    } else {
      T v[2 * RT];
#pragma unroll
      for (int e = 0; e < RT; ++e) v[2 * e] = mul_rn(dc[u][e], px[e]), v[2 * e + 1] = mul_rn(dc[u][e], py[e]);
      // halve the values with the lanes, then add the lanes left with the same value
      int off = 16;
#pragma unroll
      for (int c = RT; c >= 1; c >>= 1, off >>= 1) {
        const bool hi = lane & off;
#pragma unroll
        for (int i = 0; i < RT; ++i)
          if (i < c) v[i] = (hi ? v[i + c] : v[i]) + __shfl_xor_sync(0xffffffffu, hi ? v[i] : v[i + c], off);
      }
#pragma unroll
      for (int o = 16 / (2 * RT); o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
      constexpr int LPV = 32 / (2 * RT);  // lanes per value
      if (lane % LPV == 0 && l <= l_end) reinterpret_cast<T*>(P + (size_t)(l - l_start) * Lp32 + rw)[lane / LPV] = v[0];
    }
  };

  const int nch = (l_end - l_start) / LC + 1;
  for (int ch = 0; ch < nch; ++ch) {
    cp_async_wait<0>();
    __syncthreads();
    if (ch + 1 < nch) stage(ch + 1);
    const T* Rs = Rs0 + (ch & 1) * LC * RROW;
    const int lc0 = l_start + ch * LC;
#pragma unroll 1
    for (int gi = 0; gi < LC; gi += U) {
      const int l0 = lc0 + gi;
      if (l0 > l_end) break;
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < RT; ++e) dc[u][e] = dn[u][e];
      fetch(l0 + U);
      dir_unroll<U>([&](auto uu) {
        constexpr int u = decltype(uu)::value;
        compute(Rs + (gi + u) * RROW, gi + u, l0 + u, uu);
      });
    }
    if constexpr (!ISB) {
      __syncthreads();
      const int nl = min(LC, l_end - lc0 + 1);
      for (int i = w; i < nl; i += 8) {
        cx<T> sum = red[i * 256 + lane];
#pragma unroll
        for (int r2 = 1; r2 < 8; ++r2) {
          const cx<T> v = red[i * 256 + r2 * 32 + lane];
          sum.x += v.x;
          sum.y += v.y;
        }
        P[(size_t)(lc0 - l_start + i) * Lp32 + lane] = sum;
      }
    }
  }
}

template <typename T, int N>
constexpr size_t dir_syn_smem() {
  return (size_t)2 * kDirLC<T> * 2 * ((N + 1) / 2) * 32 * sizeof(T) + (size_t)kDirLC<T> * 8 * 32 * sizeof(cx<T>);
}

template <typename T, int N>
__global__ void __launch_bounds__(256)
k_contract_dir_syn(const ContractDesc<T>* __restrict__ dw, const CTask* __restrict__ tw, int nw,
                   const ContractDesc<T>* __restrict__ dphi, const CTask* __restrict__ tp) {
  begin_after();
  extern __shared__ __align__(16) unsigned char dir_smem[];
  __shared__ cx<T> cg[64];
  cx<T>* red = reinterpret_cast<cx<T>*>(dir_smem);
  T* Rs = reinterpret_cast<T*>(dir_smem + (size_t)kDirLC<T> * 8 * 32 * sizeof(cx<T>));
  const int i = blockIdx.x / kDirSynSub<T>, sub = blockIdx.x % kDirSynSub<T>;
  if (i < nw) {
    const CTask tk = tw[i];
    if (tk.half == 0) dir_syn_tile<T, N, 2, false>(dw + tk.prob, tk, sub, cg, Rs, red);
    else dir_syn_tile<T, N, 2, true>(dw + tk.prob, tk, sub, cg, Rs, red);
  } else {
    const CTask tk = tp[i - nw];
    if (tk.half == 0) dir_syn_tile<T, 1, 1, false>(dphi + tk.prob, tk, sub, cg, Rs, red);
    else dir_syn_tile<T, 1, 1, true>(dphi + tk.prob, tk, sub, cg, Rs, red);
  }
}

template <typename T, int N>
void dir_launch(bool syn, int rt, const DirTasks<T>& w, const DirTasks<T>& p, const CallPtrs& ptrs, cudaStream_t st) {
  const int n = w.n + p.n;
  const ContractDesc<T>* dw = w.descs;
  const ContractDesc<T>* dp = p.descs;
  if (syn) launch_after(k_contract_dir_syn<T, N>, kDirSynSub<T> * n, 256, dir_syn_smem<T, N>(), st, dw, w.tasks, w.n, dp, p.tasks);
  else if constexpr (sizeof(T) == 8) launch_after(k_contract_dir_ana<T, N, 1, 4>, 8 * n, 128, 0, st, dw, w.tasks, w.n, dp, p.tasks, ptrs);
  else if (rt == 4) launch_after(k_contract_dir_ana<T, N, 4, 8>, n, 256, 0, st, dw, w.tasks, w.n, dp, p.tasks, ptrs);
  else if (rt == 2) launch_after(k_contract_dir_ana<T, N, 2, 8>, 2 * n, 256, 0, st, dw, w.tasks, w.n, dp, p.tasks, ptrs);
  else launch_after(k_contract_dir_ana<T, N, 1, 4>, 8 * n, 128, 0, st, dw, w.tasks, w.n, dp, p.tasks, ptrs);
}

template <typename T, int N>
cudaError_t dir_attr() {
  return cudaFuncSetAttribute(k_contract_dir_syn<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)dir_syn_smem<T, N>());
}

template <typename T>
cudaError_t dir_attrs() {
  cudaError_t (*fns[])() = {dir_attr<T, 1>, dir_attr<T, 2>, dir_attr<T, 3>, dir_attr<T, 4>,
                            dir_attr<T, 5>, dir_attr<T, 6>, dir_attr<T, 7>, dir_attr<T, 8>};
  for (auto f : fns)
    if (cudaError_t e = f(); e != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace

// One launch over the tasks of w (N orders, two slots) and p (scaling parts).
template <typename T>
void launch_contract_direct(int N, bool syn, int rt, const DirTasks<T>& w, const DirTasks<T>& p, const CallPtrs& ptrs,
                            cudaStream_t st) {
  if (w.n + p.n <= 0) return;
  switch (N) {
    case 1: dir_launch<T, 1>(syn, rt, w, p, ptrs, st); break;
    case 2: dir_launch<T, 2>(syn, rt, w, p, ptrs, st); break;
    case 3: dir_launch<T, 3>(syn, rt, w, p, ptrs, st); break;
    case 4: dir_launch<T, 4>(syn, rt, w, p, ptrs, st); break;
    case 5: dir_launch<T, 5>(syn, rt, w, p, ptrs, st); break;
    case 6: dir_launch<T, 6>(syn, rt, w, p, ptrs, st); break;
    case 7: dir_launch<T, 7>(syn, rt, w, p, ptrs, st); break;
    case 8: dir_launch<T, 8>(syn, rt, w, p, ptrs, st); break;
    default: break;
  }
}

}  // namespace s2dw
