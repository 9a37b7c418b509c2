// step_blk.cuh -- the FP32 S-ADI step (Sec. 3, eq. "ADI scheme equivalent")
// for FFT lengths N' = 256 .. 2048 (blk_path) on the block-wide register FFT
// of blkfft.cuh.  The four kernels of step_reg.cuh, with one row, column half
// or column per T = 32 .. 256 threads:
//   kb_rows_r2c    row of the increment d^n -> half spectrum along x
//   kb_cols_conv   x frequency: y FFT (even / odd half) x symbol, inverse
//   kb_rows_solve  inverse real FFT, C += conv(d^n), B^n, then the x sweep
//                  (Algorithm 1), or B^n alone (dense-inverse form)
//   kb_cols_solve  y sweep (Algorithm 1) + compensated leapfrog
//
// Between the row and the column kernels the data changes direction twice:
// the spectrum is stored by x frequency (S[k * lds + row]) and the x sweep's
// result by column (W[k * ld + row]), so that each column kernel reads one
// contiguous vector.  A single row would then move 8- or 4-byte pieces a
// column apart; groups of V = 8 rows, in one block (R = 8) or in a cluster of
// V / R, are therefore exchanged through (distributed) shared memory: row c of
// the group gathers frequencies (columns) c L/V .. of all V rows and moves runs
// of V rows, 64 or 32 bytes.  This replaces the two transpose passes of the shared-memory
// engine's y sweep and its 8-byte column gathers.
//
// Measured (GB300): N = 2047 dense, four instances, row FFT, convolution and
// B^n 80 + 192 + 264 -> 75 + 175 + 170 us against the 64-elements-per-lane
// kernels this replaces there; steps of the other lengths at blk_path.  Longer
// transforms keep the shared-memory engine (reg_path_supported).  What bounds
// the kernels is the latency of the table loads and barriers at 16 to 32 warps
// per SM.
#pragma once
#include <cuda_runtime.h>

#include "bf16split.cuh"
#include "blkfft.cuh"
#include "border.cuh"
#include "sadi_internal.h"

namespace sadi {
namespace blk {

using bf::BlkFFT;
using rf::static_for;

constexpr int kCluster = 8;   // V

// g(u) in full FP32 precision; the general form out of line
static __device__ __noinline__ float g_general_b(float u, float c1, float c3, float cs) {
  return (c1 + c3 * u * u) * u + cs * sinf(u);
}
__device__ __forceinline__ float g_of_b(const RegInst& I, float u) {
  if (I.gkind == 1) return -u * u * u;
  if (I.gkind == 2) return -sinf(u);
  if (I.gkind == 3) return g_general_b(u, I.gc1, I.gc3, I.gcs);
  return 0.f;
}

// Loads of streamed data (read once) that leave L1 to the twiddle, symbol and
// spectral tables, which every block of the SM reads again.
__device__ __forceinline__ float2 ld_stream(const float2* p) {
  float2 v;
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_stream(const float* p) {
  float v;
  asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// ---- cluster exchange ---------------------------------------------------------
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ void st_peer(unsigned a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_peer(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// Tables of blkfft.cuh (RegInst::tw1).
template <int LOGL>
__device__ __forceinline__ const float2* btw1(const RegInst& I) { return I.tw1 + BlkFFT<LOGL>::L; }
template <int LOGL>
__device__ __forceinline__ const float2* btw1h(const RegInst& I) { return I.tw1 + 2 * BlkFFT<LOGL>::L; }
template <int LOGL>
__device__ __forceinline__ const float2* btw2(const RegInst& I) { return I.tw1 + 3 * BlkFFT<LOGL>::L; }

// Barrier of the T threads of a row (rl: the row's place in its block).
template <int T>
__device__ __forceinline__ void row_sync(int rl) {
  if constexpr (T == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + rl), "n"(T) : "memory");
}

template <int LOGL>
struct Cfg {
  using F = BlkFFT<LOGL>;
  static constexpr int V = kCluster;
  // rows per block: short rows share one, which needs fewer or no distributed
  // exchanges (us per step, 1 / 16 instances at 1, 2, 4, 8 rows a block: GS N =
  // 511 32 / 238, 32 / 231, 31 / 219, 29 / 201; N = 1023 64 / 840, 62 / 817, 62 /
  // 774 (4); at N = 2047 four rows measured slower than one, 246 against 224)
  static constexpr int R = LOGL <= 9 ? 8 : LOGL == 10 ? 4 : 1;
  static constexpr int CL = V / R;                   // blocks per cluster
  static constexpr int SEG = F::L / V;               // frequencies (columns) per block of the exchange
  static constexpr int QS = F::E / V;                // registers q per segment: t + T q lies in segment q / QS
  static_assert(SEG % F::T == 0 && QS * V == F::E, "whole register groups per segment");
  // row pitches of the exchange buffers: a half-warp (8-byte) or a warp
  // (4-byte) reading V rows x 16/V (32/V) neighbours finds distinct banks
  static constexpr int P2 = SEG + 16 / V, P1 = SEG + 32 / V;
  // transform buffer and exchange buffers share the space
  static constexpr int ELEMS = F::BUF > V * P2 ? F::BUF : V * P2;
  static_assert(V * P1 <= 2 * ELEMS, "the float exchange buffer fits too");
  static constexpr size_t bytes = (size_t)R * ELEMS * sizeof(float2);
  static constexpr size_t bytes_conv = (size_t)(F::BUF + (LOGL <= 10 ? F::BUF : F::L)) * sizeof(float2);
  // resident blocks promised to the compiler (its register budget): 64
  // registers a thread for the row FFT and, at N' = 512 and 2048, the dense
  // B^n kernel (seven N = 511 instances: 18 us, 21 at 85 registers), 128 for
  // the sweeps
  static constexpr int kM = 256 / F::T;   // rows for each 256 threads
  static constexpr int per(int rows) { return rows / R > 0 ? rows / R : 1; }
  static constexpr int kR2cBlocks = per(4 * kM);
  static constexpr int kDenseBlocks = per(LOGL == 11 || LOGL == 9 ? 4 * kM : 2 * kM);
  static constexpr int kGsBlocks = per(2 * kM);
  static constexpr int kColsBlocks = per(2 * kM);
  // the two convolution kernels: both halves in one block up to N' = 1024
  // (29 us at 4 blocks a SM, 30 at 5, 31 at 6 for three N = 1023 instances),
  // one after the other above
  static constexpr bool kConvSplit = LOGL <= 10;
  // what runs at this length (launch_step_reg): the dense form's row kernels, the
  // GS sweeps, and border ranks above kBorderInline among them (below N' = 1024
  // those take dense sweeps, dir_mode)
  static constexpr bool kDense = LOGL != 10, kGS = LOGL <= 10, kBorder = LOGL == 10;
  static constexpr int kConvBlocks = LOGL == 10 ? 4 : LOGL == 9 ? 6 : LOGL == 8 ? 12 : 2 * kM;
};

// Exchange between the V rows of a cluster: the barrier over all of them
// (release / acquire: it orders a block's own reads before its peers' writes to
// the same buffer, and the peers' writes before its reads) and the address of p
// (in the calling row's buffer) in the buffer of row `to`.
template <int LOGL>
struct Exchange {
  using C = Cfg<LOGL>;
  __device__ static __forceinline__ void sync() {
    if constexpr (C::CL == 1) __syncthreads();
    else cluster_sync();
  }
  template <typename P>
  __device__ static __forceinline__ unsigned at(const P* p, int rl, int to) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p) + (unsigned)((to % C::R - rl) * (int)(C::ELEMS * sizeof(float2)));
    if constexpr (C::CL == 1) return a;
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(to / C::R));
    return r;
  }
  template <typename T>
  __device__ static __forceinline__ void put(unsigned a, T v) {
    if constexpr (C::CL > 1) st_peer(a, v);
    else if constexpr (sizeof(T) == 8) asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
    else asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
  }
};

__device__ __forceinline__ void pdl_wait_prerequisites() { pdl_entry(); }

// ---------------------------------------------------------------------------
template <int LOGL>
__global__ void __launch_bounds__(Cfg<LOGL>::R * BlkFFT<LOGL>::T, Cfg<LOGL>::kR2cBlocks)
kb_rows_r2c(const __grid_constant__ RegBatch B) {
  using F = BlkFFT<LOGL>;
  using C = Cfg<LOGL>;
  using X = Exchange<LOGL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // row rl of the block, thread t of the row
  const int rl = C::R == 1 ? 0 : threadIdx.x / F::T, t = C::R == 1 ? threadIdx.x : threadIdx.x % F::T;
  float2* sm = reinterpret_cast<float2*>(smem_raw) + rl * C::ELEMS;
  const RegInst& I = B.in[blockIdx.y];
  const int N = I.N;
  const int row = blockIdx.x * C::R + rl, rank = row % C::V, row0 = row - rank;
  if (row0 >= N) return;   // the whole cluster
  const bool valid = row < N;
  auto sync = [rl] { C::R == 1 ? __syncthreads() : row_sync<F::T>(rl); };
  pdl_wait_prerequisites();
  // z[n] = d[2n] + i d[2n+1], zero from n = N'/2 on (2n < N <= N'); an even
  // offset in a 128-byte aligned row: 8-byte loads, row padding beyond N - 1
  const float* ur = I.u_d + (size_t)(valid ? row : 0) * I.ld;
  float2 x[F::E];
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    float2 v = make_float2(0.f, 0.f);
    if constexpr (q < F::E / 2) {
      const int n = t + F::T * q;
      if (valid && 2 * n < N) v = ld_stream(reinterpret_cast<const float2*>(ur + 2 * n));
      if (2 * n + 1 >= N) v.y = 0.f;
    }
    x[q] = v;
  });
  F::fwd(x, sm, t, btw1<LOGL>(I), false, btw2<LOGL>(I), sync);
  static_for<0, F::E>([&](auto qc) { sm[t + F::T * decltype(qc)::value] = x[decltype(qc)::value]; });
  sync();
  // X[k] = (Z[k] + conj Z[-k]) / 2 + w^k (Z[k] - conj Z[-k]) / (2 i); slot 0 = X[0] + i X[N']
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int k = t + F::T * q;
    const float2 Z = x[q], Zc = cconj(sm[(F::L - k) & (F::L - 1)]);
    const float2 Ev = cscale(cadd(Z, Zc), 0.5f);
    const float2 Ov = cscale(cmul_mi(csub(Z, Zc)), 0.5f);
    x[q] = (q == 0 && t == 0) ? make_float2(Ev.x + Ov.x, Ev.x - Ov.x) : cadd(Ev, cmul(__ldg(&I.tw[k]), Ov));
  });
  X::sync();   // every row of the cluster has read its buffer
  static_for<0, C::V>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    const unsigned dst = X::at(sm + rank * C::P2 + t, rl, c);
    static_for<0, C::QS>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      X::put(dst + (unsigned)(F::T * j * sizeof(float2)), x[c * C::QS + j]);
    });
  });
  X::sync();   // the rows' segments have arrived
  const int vv = t % C::V, s0 = t / C::V;
  if (row0 + vv >= N) return;
  float2* col = I.S + (size_t)(rank * C::SEG + s0) * I.lds + row0 + vv;
  const float2* src = sm + vv * C::P2 + s0;
#pragma unroll 4
  for (int i = 0; i < F::E; ++i) col[(size_t)(F::T / C::V * i) * I.lds] = src[F::T / C::V * i];
}

// ---------------------------------------------------------------------------
// Block: x frequency kx = blockIdx.x (0 .. N'); threads 0 .. T-1 the even y
// frequencies 2 m, T .. 2T-1 the odd ones 2 m + 1.  Frequencies 0 and N' are
// the real and the imaginary part of slot 0: two blocks, each reading and
// writing its own halves of the slot's elements.
template <int LOGL>
__global__ void __launch_bounds__(2 * BlkFFT<LOGL>::T, Cfg<LOGL>::kConvBlocks)
kb_cols_conv(const __grid_constant__ RegBatch B) {
  using F = BlkFFT<LOGL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const RegInst& I = B.in[blockIdx.y];
  const int N = I.N, kx = blockIdx.x;
  const int h = threadIdx.x / F::T, t = threadIdx.x % F::T;
  float2* const sm0 = reinterpret_cast<float2*>(smem_raw);
  float2* const sm = sm0 + h * F::BUF;
  auto sync = [h] { asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "n"(F::T) : "memory"); };
  float2* col = I.S + (size_t)(kx == F::L ? 0 : kx) * I.lds;
  pdl_wait_prerequisites();
  float2 x[F::E];
  if (kx == 0 || kx == F::L) {
    const float* c1 = reinterpret_cast<const float*>(col) + (kx == 0 ? 0 : 1);
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int j = t + F::T * q;
      x[q] = make_float2(j < N ? c1[2 * j] : 0.f, 0.f);
    });
  } else {
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int j = t + F::T * q;
      x[q] = j < N ? col[j] : make_float2(0.f, 0.f);
    });
  }
  // odd half: frequencies m + 1/2 of the length-L transform
  const float2* tw1 = h ? btw1h<LOGL>(I) : btw1<LOGL>(I);
  F::fwd(x, sm, t, tw1, h, btw2<LOGL>(I), sync);
  // the symbol at y frequency 2 m + h, stored for 0 .. N' (it is even)
  const float* lam = I.sym + (size_t)kx * (F::L + 1);
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int k2 = 2 * (t + F::T * q) + h;
    x[q] = cscale(x[q], __ldg(&lam[q < F::E / 2 ? k2 : 2 * F::L - k2]));
  });
  F::inv(x, sm, t, tw1, h, btw2<LOGL>(I), sync);
  // even + odd half: the odd threads hand over the rows of
  // q < E/2, the even threads the others, and each finishes its own rows
  constexpr int HE = F::E / 2;
  static_for<0, HE>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    sm[t + F::T * q] = h ? x[q] : x[q + HE];
  });
  __syncthreads();
  const float2* other = sm0 + (h ^ 1) * F::BUF + t;
  static_for<0, HE>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int j = t + F::T * (h ? q + HE : q);
    const float2 y = cadd(h ? x[q + HE] : x[q], other[F::T * q]);
    if (j < N) {
      if (kx == 0) reinterpret_cast<float*>(col + j)[0] = y.x;
      else if (kx == F::L) reinterpret_cast<float*>(col + j)[1] = y.x;
      else col[j] = y;
    }
  });
}

// The same with one half after the other on T threads, at N' = 2048: the even
// half's result waits in shared memory (each thread its own elements), and the
// odd half reads the column again (from L2).  Independent blocks with their full
// registers overlap loads, transforms and stores (N = 2047 39 -> 37 us); below,
// the split kernel's smaller blocks do that too (N = 1023 15.9 us, 16.3 so).
template <int LOGL>
__global__ void __launch_bounds__(BlkFFT<LOGL>::T, Cfg<LOGL>::kConvBlocks)
kb_cols_conv_seq(const __grid_constant__ RegBatch B) {
  using F = BlkFFT<LOGL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const RegInst& I = B.in[blockIdx.y];
  const int N = I.N, kx = blockIdx.x, t = threadIdx.x;
  float2* const sm = reinterpret_cast<float2*>(smem_raw);
  float2* const keep = sm + F::BUF + t;
  auto sync = [] { __syncthreads(); };
  float2* col = I.S + (size_t)(kx == F::L ? 0 : kx) * I.lds;
  pdl_wait_prerequisites();
  float2 x[F::E];
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    if (kx == 0 || kx == F::L) {
      const float* c1 = reinterpret_cast<const float*>(col) + (kx == 0 ? 0 : 1);
      static_for<0, F::E>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const int j = t + F::T * q;
        x[q] = make_float2(j < N ? c1[2 * j] : 0.f, 0.f);
      });
    } else {
      static_for<0, F::E>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const int j = t + F::T * q;
        x[q] = j < N ? col[j] : make_float2(0.f, 0.f);
      });
    }
    const float2* tw1 = h ? btw1h<LOGL>(I) : btw1<LOGL>(I);
    F::fwd(x, sm, t, tw1, h, btw2<LOGL>(I), sync);
    const float* lam = I.sym + (size_t)kx * (F::L + 1);
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int k2 = 2 * (t + F::T * q) + h;
      x[q] = cscale(x[q], __ldg(&lam[q < F::E / 2 ? k2 : 2 * F::L - k2]));
    });
    F::inv(x, sm, t, tw1, h, btw2<LOGL>(I), sync);
    if (h == 0) static_for<0, F::E>([&](auto qc) { keep[F::T * decltype(qc)::value] = x[decltype(qc)::value]; });
  }
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int j = t + F::T * q;
    const float2 y = cadd(keep[F::T * q], x[q]);
    if (j < N) {
      if (kx == 0) reinterpret_cast<float*>(col + j)[0] = y.x;
      else if (kx == F::L) reinterpret_cast<float*>(col + j)[1] = y.x;
      else col[j] = y;
    }
  });
}

// ---------------------------------------------------------------------------
// Algorithm 1 on the bordered matrix: x = v' + i J v' (natural) -> vhat (its
// factors Q and Q^H are the half-frequency shift of the first pair), then
// y[q] = (H^-1 v)[k], k = t + T q: Re vhat[k] + Im vhat[N'-1-k] + the border
// correction sum_p G[k, p] ybot[p], ybot[p] = Re vhat[N+p] + Im vhat[r-1-p];
// for r > kBorderInline ybot of vector vec is stored for border.cuh.
template <int LOGL, typename Sync>
__device__ __forceinline__ void gs_solve(float2* x, float* y, float2* sm, int t, int vec, const RegInst& I, Sync sync) {
  using F = BlkFFT<LOGL>;
  // skew-circulant factor lambda_s, then circulant factor lambda_c.  Rolled:
  // one forward and one inverse transform body in the kernel.
#pragma unroll 1
  for (int round = 0; round < 2; ++round) {
    const float2* lam = round == 0 ? I.lam_s : I.lam_c;
    const float2* tw1 = round == 0 ? btw1h<LOGL>(I) : btw1<LOGL>(I);
    F::fwd(x, sm, t, tw1, round == 0, btw2<LOGL>(I), sync);
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      x[q] = cmul(x[q], __ldg(&lam[t + F::T * q]));
    });
    F::inv(x, sm, t, tw1, round == 0, btw2<LOGL>(I), sync);
  }
  static_for<0, F::E>([&](auto qc) { sm[t + F::T * decltype(qc)::value] = x[decltype(qc)::value]; });
  sync();
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    y[q] = x[q].x + sm[F::L - 1 - (t + F::T * q)].y;
  });
  const int N = I.N, r = I.r;
  if constexpr (Cfg<LOGL>::kBorder) {
    if (r > kBorderInline) {
      float* yb = ybot_of(I, F::L);
      if (vec < N)
        for (int p = t; p < r; p += F::T) yb[(size_t)p * I.ld + vec] = sm[N + p].x + sm[r - 1 - p].y;
      return;
    }
  }
#pragma unroll 1
  for (int p = 0; p < r; ++p) {
    const float yb = sm[N + p].x + sm[r - 1 - p].y;
    const float* Gp = I.G + (size_t)p * N;
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int k = t + F::T * q;
      if (k < N) y[q] += __ldg(Gp + k) * yb;
    });
  }
}

// ---------------------------------------------------------------------------
// DENSE: the dense-inverse form stops after B^n, which it writes to W (FP32)
// and, split into BF16 pairs, to Bh / Bl (the first sweep GEMM's A operand).
// Else W receives the x sweep by columns, W[k * ld + row].
template <int LOGL, bool DENSE>
__global__ void __launch_bounds__(Cfg<LOGL>::R * BlkFFT<LOGL>::T, DENSE ? Cfg<LOGL>::kDenseBlocks : Cfg<LOGL>::kGsBlocks)
kb_rows_solve(const __grid_constant__ RegBatch B) {
  using F = BlkFFT<LOGL>;
  using C = Cfg<LOGL>;
  using X = Exchange<LOGL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // row rl of the block, thread t of the row
  const int rl = C::R == 1 ? 0 : threadIdx.x / F::T, t = C::R == 1 ? threadIdx.x : threadIdx.x % F::T;
  float2* sm = reinterpret_cast<float2*>(smem_raw) + rl * C::ELEMS;
  const RegInst& I = B.in[blockIdx.y];
  const int N = I.N;
  const int row = blockIdx.x * C::R + rl, rank = row % C::V, row0 = row - rank;
  if (row0 >= N) return;   // the whole cluster
  const bool valid = row < N;
  const size_t rbase = (size_t)(valid ? row : 0) * I.ld;
  auto sync = [rl] { C::R == 1 ? __syncthreads() : row_sync<F::T>(rl); };
  if constexpr (C::CL > 1) cluster_arrive_relaxed();   // peers may be written once every block runs
  // the rows the B^n epilogue reads into L2 under the convolution's tail
  // (written in the previous step; a prefetch cannot make a load see older data)
  if (valid) {
    for (int c0 = 32 * t; c0 < N; c0 += 32 * F::T) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(I.C_hi + rbase + c0));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(I.C_lo + rbase + c0));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(I.u_hi + rbase + c0));
    }
  }
  pdl_wait_prerequisites();
  if constexpr (DENSE) {
    // zero the sweep GEMM's counters for the GEMM that follows
    if (row == 0 && I.dep)
      for (int i = t; i < I.ndep; i += F::T) I.dep[i] = 0;
  }
  float2 x[F::E];
  {
    // frequencies rank L/V .. of the cluster's V rows, handed to their rows
    const int vv = t % C::V, s0 = t / C::V;
    const bool ok = row0 + vv < N;
    const float2* col = I.S + (size_t)(rank * C::SEG + s0) * I.lds + row0 + (ok ? vv : 0);
    static_for<0, F::E>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      x[i] = ok ? ld_stream(col + (size_t)(F::T / C::V * i) * I.lds) : make_float2(0.f, 0.f);
    });
    if constexpr (C::CL > 1) cluster_wait();
    const unsigned dst = X::at(sm + rank * C::SEG + s0, rl, vv);
    static_for<0, F::E>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      X::put(dst + (unsigned)(F::T / C::V * i * sizeof(float2)), x[i]);
    });
  }
  X::sync();
  // half spectrum X[k] -> Z[k] = E + i O, the spectrum of z[n] = x[2n] + i x[2n+1]
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int k = t + F::T * q;
    const float2 Xk = sm[k], Xc = cconj(sm[(F::L - k) & (F::L - 1)]);
    const float2 Ev = cscale(cadd(Xk, Xc), 0.5f);
    const float2 Ov = cscale(cmulc(csub(Xk, Xc), __ldg(&I.tw[k])), 0.5f);
    x[q] = (q == 0 && t == 0) ? make_float2(0.5f * (Xk.x + Xk.y), 0.5f * (Xk.x - Xk.y)) : cadd(Ev, cmul_pi(Ov));
  });
  sync();
  F::inv(x, sm, t, btw1<LOGL>(I), false, btw2<LOGL>(I), sync);
  // x[q], q < E/2, now holds the convolution at 2n, 2n + 1, n = t + T q.
  // Wave step: B = C + tau^2 (g(u) + f), n = 0: tau phi2 + (C + tau^2 (g + f))/2,
  // with C <- C + conv; diffusion: B = C + conv/2 + tau (g(u~) + f) - d,
  // u~ = u + d/2.  The equation is uniform over the launch.
  const float tau = I.tau, tau2 = I.tau2;
  auto bn = [&](auto diff_c) {
    constexpr bool DIFF = decltype(diff_c)::value;
    constexpr int HE = F::E / 2, GR = HE < 8 ? HE : 8;   // loads in flight per array
    static_for<0, HE / GR>([&](auto gc) {
      constexpr int q0 = decltype(gc)::value * GR;
      float2 ch[GR], cl[GR], uv[GR];
      [[maybe_unused]] float2 dv[GR];
      static_for<0, GR>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const int e = 2 * (t + F::T * (q0 + j));
        const bool ok = valid && e < N;
        const size_t at = ok ? rbase + e : 0;
        const float2 z = make_float2(0.f, 0.f);
        ch[j] = ok ? ld_stream(reinterpret_cast<const float2*>(I.C_hi + at)) : z;
        cl[j] = ok ? ld_stream(reinterpret_cast<const float2*>(I.C_lo + at)) : z;
        uv[j] = ok ? ld_stream(reinterpret_cast<const float2*>(I.u_hi + at)) : z;
        if constexpr (DIFF) dv[j] = (ok && !I.first) ? ld_stream(reinterpret_cast<const float2*>(I.u_d + at)) : z;
      });
      static_for<0, GR>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const int e0 = 2 * (t + F::T * (q0 + j));
        float b[2] = {0.f, 0.f}, cn[2] = {0.f, 0.f}, cln[2] = {0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = e0 + e;
          if (valid && i < N) {
            // C <- C + conv (two-sum into the double-float pair)
            const float hi = e ? ch[j].y : ch[j].x, lo = e ? cl[j].y : cl[j].x;
            const float cx = e ? x[q0 + j].y : x[q0 + j].x;
            const float s = hi + cx;
            const float bb = s - hi;
            const float err = (hi - (s - bb)) + (cx - bb);
            const float l2 = lo + err;
            const float c = s + l2;
            cn[e] = c;
            cln[e] = l2 - (c - s);
            const float u = e ? uv[j].y : uv[j].x;
            if constexpr (!DIFF) {
              float gs = g_of_b(I, u);
              if (I.F) gs += I.fsc * I.F[(size_t)row * I.ldF + i];
              const float gg = tau2 * gs;
              b[e] = I.first ? tau * I.phi2[rbase + i] + 0.5f * (c + gg) : c + gg;
            } else {
              const float d = e ? dv[j].y : dv[j].x;
              float gs = g_of_b(I, u + 0.5f * d);
              if (I.F) gs += I.fsc * I.F[(size_t)row * I.ldF + i];
              b[e] = (c + 0.5f * cx) + tau2 * gs - d;
            }
          }
        }
        // 8-byte stores, or the single element at N - 1 (the padding is never written)
        if (valid && e0 + 1 < N) {
          *reinterpret_cast<float2*>(I.C_hi + rbase + e0) = make_float2(cn[0], cn[1]);
          *reinterpret_cast<float2*>(I.C_lo + rbase + e0) = make_float2(cln[0], cln[1]);
        } else if (valid && e0 < N) {
          I.C_hi[rbase + e0] = cn[0];
          I.C_lo[rbase + e0] = cln[0];
        }
        if constexpr (DENSE) {
          // B^n to W and its BF16 pairs (at e0 + 1 = N, the zero padding of
          // the pairs, the split of 0 is stored)
          if (valid && e0 < N) {
            float* wr = I.W + rbase;
            if (e0 + 1 < N) *reinterpret_cast<float2*>(wr + e0) = make_float2(b[0], b[1]);
            else wr[e0] = b[0];
            if (I.Bh) {
              unsigned hi, lo;
              split_bf16x2(b[0], b[1], &hi, &lo);
              *reinterpret_cast<unsigned*>(I.Bh + (size_t)row * I.ldp + e0) = hi;
              *reinterpret_cast<unsigned*>(I.Bl + (size_t)row * I.ldp + e0) = lo;
            }
          }
        } else {
          sm[t + F::T * (q0 + j)] = make_float2(b[0], b[1]);
        }
      });
    });
  };
  if (I.eq == 1) bn(std::integral_constant<bool, true>{});
  else bn(std::integral_constant<bool, false>{});
  if constexpr (DENSE) {
    return;
  } else {
    sync();
    // B' + i J B'
    const float* bf = reinterpret_cast<const float*>(sm);
    static_for<0, F::E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int k = t + F::T * q;
      x[q] = make_float2(bf[k], bf[F::L - 1 - k]);
    });
    sync();
    float y[F::E];
    gs_solve<LOGL>(x, y, sm, t, row, I, sync);
    X::sync();   // every row of the cluster has read its buffer
    float* smf = reinterpret_cast<float*>(sm);
    static_for<0, C::V>([&](auto cc) {
      constexpr int c = decltype(cc)::value;
      const unsigned dst = X::at(smf + rank * C::P1 + t, rl, c);
      static_for<0, C::QS>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        X::put(dst + (unsigned)(F::T * j * sizeof(float)), y[c * C::QS + j]);
      });
    });
    X::sync();
    const int vv = t % C::V, s0 = t / C::V;
    if (row0 + vv >= N) return;
    const float* src = smf + vv * C::P1 + s0;
#pragma unroll 4
    for (int i = 0; i < F::E; ++i) {
      const int k = rank * C::SEG + s0 + F::T / C::V * i;
      if (k < N) I.W[(size_t)k * I.ld + row0 + vv] = src[F::T / C::V * i];
    }
  }
}

// ---------------------------------------------------------------------------
// Column i of W (row i of the array by columns): uhat = H^-1 W, then, on the
// rows handed out over the cluster's V columns, the compensated leapfrog
// d^{n+1} = d^n + uhat (d^1 = uhat), u^{n+1} = u^n + d^{n+1}, u = u_hi + u_lo.
template <int LOGL>
__global__ void __launch_bounds__(Cfg<LOGL>::R * BlkFFT<LOGL>::T, Cfg<LOGL>::kColsBlocks)
kb_cols_solve(const __grid_constant__ RegBatch B) {
  using F = BlkFFT<LOGL>;
  using C = Cfg<LOGL>;
  using X = Exchange<LOGL>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // row rl of the block, thread t of the row
  const int rl = C::R == 1 ? 0 : threadIdx.x / F::T, t = C::R == 1 ? threadIdx.x : threadIdx.x % F::T;
  float2* sm = reinterpret_cast<float2*>(smem_raw) + rl * C::ELEMS;
  float* smf = reinterpret_cast<float*>(sm);
  const RegInst& I = B.in[blockIdx.y];
  const int N = I.N;
  const int i = blockIdx.x * C::R + rl, rank = i % C::V, i0 = i - rank;
  if (i0 >= N) return;   // the whole cluster
  const bool valid = i < N;
  auto sync = [rl] { C::R == 1 ? __syncthreads() : row_sync<F::T>(rl); };
  pdl_wait_prerequisites();
  const float* w = I.W + (size_t)(valid ? i : 0) * I.ld;
  float2 x[F::E];
  static_for<0, F::E>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int k = t + F::T * q, k2 = F::L - 1 - k;
    x[q] = make_float2((valid && k < N) ? w[k] : 0.f, (valid && k2 < N) ? w[k2] : 0.f);
  });
  float y[F::E];
  gs_solve<LOGL>(x, y, sm, t, i, I, sync);
  X::sync();   // every row of the cluster has read its buffer
  static_for<0, C::V>([&](auto cc) {
    constexpr int c = decltype(cc)::value;
    const unsigned dst = X::at(smf + rank * C::P1 + t, rl, c);
    static_for<0, C::QS>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      X::put(dst + (unsigned)(F::T * j * sizeof(float)), y[c * C::QS + j]);
    });
  });
  X::sync();
  const int vv = t % C::V, s0 = t / C::V;
  if (i0 + vv >= N) return;
  const float* src = smf + vv * C::P1 + s0;
  if constexpr (C::kBorder) {
    if (I.r > kBorderInline) {
      // uhat short of its border correction, by rows, for border.cuh
      float* U = reinterpret_cast<float*>(I.S);
#pragma unroll 4
      for (int e = 0; e < F::E; ++e) {
        const int j = rank * C::SEG + s0 + F::T / C::V * e;
        if (j < N) U[(size_t)j * I.ld + i0 + vv] = src[F::T / C::V * e];
      }
      return;
    }
  }
  const int first = I.first;
#pragma unroll 1
  for (int g = 0; g < F::E; g += 8) {
    float hi[8], lo[8], dd[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int j = rank * C::SEG + s0 + F::T / C::V * (g + e);
      const size_t at = (size_t)j * I.ld + i0 + vv;
      hi[e] = j < N ? ld_stream(I.u_hi + at) : 0.f;
      lo[e] = j < N ? ld_stream(I.u_lo + at) : 0.f;
      dd[e] = (j < N && !first) ? ld_stream(I.u_d + at) : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int j = rank * C::SEG + s0 + F::T / C::V * (g + e);
      if (j >= N) continue;
      const size_t at = (size_t)j * I.ld + i0 + vv;
      const float d = dd[e] + src[F::T / C::V * (g + e)];
      const float s = hi[e] + d;
      const float bb = s - hi[e];
      const float err = (hi[e] - (s - bb)) + (d - bb);
      const float l2 = lo[e] + err;
      const float h2 = s + l2;
      I.u_hi[at] = h2;
      I.u_lo[at] = l2 - (h2 - s);
      I.u_d[at] = d;
    }
  }
}

template <int LOGL>
cudaError_t launch_blk_conv(const RegBatch& b, cudaStream_t st) {
  using F = BlkFFT<LOGL>;
  using C = Cfg<LOGL>;
  static LaunchCache attr_done[kLauncherDevices];
  const int dev = device_slot();
  if (dev < 0) return cudaErrorInvalidDevice;
  auto go = [&](auto kernel, int threads) {
    if (!attr_done[dev].load(std::memory_order_acquire)) {
      const cudaError_t e =
          cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::bytes_conv);
      if (e != cudaSuccess) return e;
      attr_done[dev].store(1, std::memory_order_release);
    }
    return launch_dependent(kernel, dim3(F::L + 1, b.count), dim3(threads), C::bytes_conv, st, b);
  };
  if constexpr (C::kConvSplit) return go(kb_cols_conv<LOGL>, 2 * F::T);
  else return go(kb_cols_conv_seq<LOGL>, F::T);
}

template <int LOGL>
cudaError_t launch_blk_impl(const RegBatch& b, int max_n, cudaStream_t st, cudaEvent_t* ev, bool dense) {
  using F = BlkFFT<LOGL>;
  using C = Cfg<LOGL>;
  static LaunchCache attr_done[kLauncherDevices];
  const int dev = device_slot();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (dense ? !C::kDense : !C::kGS) return cudaErrorInvalidValue;
  cudaError_t e;
  if (!attr_done[dev].load(std::memory_order_acquire)) {
    auto room = [](auto kernel, size_t bytes) {
      return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    if ((e = room(kb_rows_r2c<LOGL>, C::bytes))) return e;
    if constexpr (C::kDense)
      if ((e = room(kb_rows_solve<LOGL, true>, C::bytes))) return e;
    if constexpr (C::kGS)
      if ((e = room(kb_rows_solve<LOGL, false>, C::bytes)) || (e = room(kb_cols_solve<LOGL>, C::bytes))) return e;
    attr_done[dev].store(1, std::memory_order_release);
  }
  // every kernel of the step is a programmatic dependent of the one before
  // it; the row kernels run in clusters of V blocks
  auto launch = [&](auto kernel, dim3 grid, int threads, size_t smem) {
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    a[1].id = cudaLaunchAttributeClusterDimension;
    a[1].val.clusterDim.x = C::CL;
    a[1].val.clusterDim.y = 1;
    a[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = a;
    cfg.numAttrs = C::CL > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, b);
  };
  const dim3 rgrid((max_n + C::V - 1) / C::V * C::CL, b.count);
  if (ev) cudaEventRecord(ev[0], st);
  if ((e = launch(kb_rows_r2c<LOGL>, rgrid, C::R * F::T, C::bytes))) return e;
  if (ev) cudaEventRecord(ev[1], st);
  if ((e = launch_blk_conv<LOGL>(b, st))) return e;
  if (ev) cudaEventRecord(ev[2], st);
  if constexpr (C::kDense)
    if (dense) return launch(kb_rows_solve<LOGL, true>, rgrid, C::R * F::T, C::bytes);
  if constexpr (C::kGS) {
    const bool border = border::any(b);
    if (border && !C::kBorder) return cudaErrorInvalidValue;
    if ((e = launch(kb_rows_solve<LOGL, false>, rgrid, C::R * F::T, C::bytes))) return e;
    if constexpr (C::kBorder)
      if (border && (e = border::launch<0>(b, max_n, st))) return e;
    if (ev) cudaEventRecord(ev[3], st);
    if ((e = launch(kb_cols_solve<LOGL>, rgrid, C::R * F::T, C::bytes))) return e;
    if constexpr (C::kBorder)
      if (border && (e = border::launch<1>(b, max_n, st))) return e;
    if (ev) cudaEventRecord(ev[4], st);
  }
  return cudaSuccess;
}

}  // namespace blk
}  // namespace sadi
