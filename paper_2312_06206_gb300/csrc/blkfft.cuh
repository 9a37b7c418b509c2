// blkfft.cuh -- block-wide register FFT of length L = R1 R2 R3 (256 .. 2048).
//
// T = R2 R3 threads own a vector; thread t holds the elements t + T q in
// registers x[q], q < E = R1, before and after the transform (frequencies in
// the same places), so that every pointwise product and every global access
// of a row is coalesced with natural-order tables.  Three levels, one shared
// buffer of R1 rows of T + 1 elements:
//   1. R1-point DFT over q in registers -> k1; times exp(-2 pi i t k1 / L);
//      row k1, column t of the buffer
//   2. R2-point DFTs over q2 of t = t' + R3 q2 -> k2; times
//      exp(-2 pi i t' k2 / T); in place (a thread writes what it has read)
//   3. R3-point DFTs over t' -> k3; frequency k = k1 + R1 (k2 + R2 k3)
// so two shared-memory round trips and three barriers per transform, where a
// radix-8 engine with the vector in shared memory takes four round trips (and
// its index arithmetic) at L = 2048.  Half-warps (8-byte accesses) read and
// write 16 consecutive elements in levels 1 and 2 and a stride of T + 1 (odd)
// in level 3: no bank conflicts.
#pragma once

#include "regfft.cuh"

namespace sadi {
namespace bf {

using rf::cbrev;
using rf::clog2;
using rf::static_for;

// Complex sums as one packed instruction on the (re, im) register pair: the
// same lanes of the FP32 pipe, half the issue slots.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// N-point DFT in registers (exponent sign -), natural in, x[p] = X[brev(p)] out.
template <int N>
__device__ __forceinline__ void dft(float2* x) {
  constexpr int LG = clog2(N);
  static_for<0, LG>([&](auto lc) {
    constexpr int span = N >> decltype(lc)::value;
    constexpr int half = span >> 1;
    static_for<0, N / span>([&](auto gc) {
      constexpr int g = decltype(gc)::value * span;
      static_for<0, half>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const float2 a = x[g + j], b = x[g + j + half];
        x[g + j] = add2(a, b);
        x[g + j + half] = rf::rot<float, true, j, span>(sub2(a, b));
      });
    });
  });
}
// Its adjoint: x[p] = X[brev(p)] in, natural out (unnormalised, sign +).
template <int N>
__device__ __forceinline__ void idft(float2* x) {
  constexpr int LG = clog2(N);
  static_for<0, LG>([&](auto lc) {
    constexpr int span = 2 << decltype(lc)::value;
    constexpr int half = span >> 1;
    static_for<0, N / span>([&](auto gc) {
      constexpr int g = decltype(gc)::value * span;
      static_for<0, half>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        const float2 a = x[g + j];
        const float2 b = rf::rot<float, false, j, span>(x[g + j + half]);
        x[g + j] = add2(a, b);
        x[g + j + half] = sub2(a, b);
      });
    });
  });
}

// Radices by log2 L.  R1 >= R2, R3 (every thread gets whole DFTs of each
// level), T = R2 R3 a multiple of R1 and R3.
template <int LOGL>
struct Radix;
template <>
struct Radix<8> {
  static constexpr int R1 = 8, R2 = 4, R3 = 8;
};
template <>
struct Radix<9> {
  static constexpr int R1 = 8, R2 = 8, R3 = 8;
};
template <>
struct Radix<10> {
  static constexpr int R1 = 16, R2 = 8, R3 = 8;
};
template <>
struct Radix<11> {
  static constexpr int R1 = 16, R2 = 8, R3 = 16;
};

template <int LOGL>
struct BlkFFT {
  static constexpr int L = 1 << LOGL;
  static constexpr int R1 = Radix<LOGL>::R1, R2 = Radix<LOGL>::R2, R3 = Radix<LOGL>::R3;
  static constexpr int T = R2 * R3, E = R1;
  static constexpr int ROW = T + 1;
  static constexpr int BUF = R1 * ROW;   // float2 elements of the buffer
  static_assert(R1 * R2 * R3 == L && T % R1 == 0 && T % R3 == 0 && R1 % R2 == 0 && R1 % R3 == 0, "radices");

  // Forward transform X[k] = sum_j x_j exp(-2 pi i j (k + s) / L), s = 0, or 1/2
  // (odd): the transform of x_j exp(-i pi j / L), whose factor splits into a
  // constant per register, exp(-i pi q / E), and one per thread that tw1
  // carries: tw1[k1 T + t] = exp(-2 pi i t (k1 + s) / L) (global memory, read
  // through L1), tw2[k2 R3 + t'] as above.  odd must be uniform over each
  // warp.  Every thread of the vector calls it; sync() is their barrier.  The
  // buffer must be free on entry and is free on return.
  template <typename Sync>
  __device__ static __forceinline__ void fwd(float2* x, float2* sm, int t, const float2* __restrict__ tw1, bool odd,
                                             const float2* __restrict__ tw2, Sync sync) {
    if (odd) static_for<1, E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      x[q] = rf::rot<float, true, q, 2 * E>(x[q]);
    });
    dft<R1>(x);
    static_for<0, R1>([&](auto pc) {
      constexpr int p = decltype(pc)::value;
      constexpr int k1 = cbrev(p, clog2(R1));
      sm[k1 * ROW + t] = cmul(x[p], __ldg(&tw1[k1 * T + t]));
    });
    sync();
    const int tp = t % R3;
    float2* row = sm + (t / R3) * ROW + tp;
    static_for<0, R1 / R2>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      float2* y = x + j * R2;
      float2* base = row + j * R2 * ROW;
      static_for<0, R2>([&](auto qc) { y[decltype(qc)::value] = base[R3 * decltype(qc)::value]; });
      dft<R2>(y);
      static_for<0, R2>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        constexpr int k2 = cbrev(p, clog2(R2));
        base[R3 * k2] = k2 == 0 ? y[p] : cmul(y[p], __ldg(&tw2[k2 * R3 + tp]));
      });
    });
    sync();
    const float2* col = sm + (t % R1) * ROW + (t / R1) * R3;
    float2 z[E];
    static_for<0, R1 / R3>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      float2 y[R3];
      static_for<0, R3>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        y[s] = col[j * (T / R1) * R3 + s];
      });
      dft<R3>(y);
      static_for<0, R3>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        z[j + (R1 / R3) * cbrev(p, clog2(R3))] = y[p];
      });
    });
    static_for<0, E>([&](auto qc) { x[decltype(qc)::value] = z[decltype(qc)::value]; });
    sync();
  }

  // The adjoint (unnormalised inverse; with odd, times exp(+i pi j / L)): the
  // three levels backwards.
  template <typename Sync>
  __device__ static __forceinline__ void inv(float2* x, float2* sm, int t, const float2* __restrict__ tw1, bool odd,
                                             const float2* __restrict__ tw2, Sync sync) {
    float2* col = sm + (t % R1) * ROW + (t / R1) * R3;
    static_for<0, R1 / R3>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      float2 y[R3];
      static_for<0, R3>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        y[p] = x[j + (R1 / R3) * cbrev(p, clog2(R3))];
      });
      idft<R3>(y);
      static_for<0, R3>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        col[j * (T / R1) * R3 + s] = y[s];
      });
    });
    sync();
    const int tp = t % R3;
    float2* row = sm + (t / R3) * ROW + tp;
    static_for<0, R1 / R2>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      float2* y = x + j * R2;
      float2* base = row + j * R2 * ROW;
      static_for<0, R2>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        constexpr int k2 = cbrev(p, clog2(R2));
        y[p] = k2 == 0 ? base[0] : cmulc(base[R3 * k2], __ldg(&tw2[k2 * R3 + tp]));
      });
      idft<R2>(y);
      static_for<0, R2>([&](auto qc) { base[R3 * decltype(qc)::value] = y[decltype(qc)::value]; });
    });
    sync();
    static_for<0, R1>([&](auto pc) {
      constexpr int p = decltype(pc)::value;
      constexpr int k1 = cbrev(p, clog2(R1));
      x[p] = cmulc(sm[k1 * ROW + t], __ldg(&tw1[k1 * T + t]));
    });
    idft<R1>(x);
    if (odd) static_for<1, E>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      x[q] = rf::rot<float, false, q, 2 * E>(x[q]);
    });
    sync();
  }
};

}  // namespace bf
}  // namespace sadi
