// step_dir.cu -- small grids: the sweeps, and in FP64 the whole step, as dense
// products (direct path): no transform levels, no barriers inside a product.
//
// A small FFT is a chain of dependent levels: at N = 63 in FP64 one step was
// 11 transforms on 8 of 32 lanes of one warp per row, 64 cycles per FP64
// instruction, 80 us.  The products below have more operations (about 8 N^3
// multiply-adds per step) but no chain, and they spread over every SM:
//   k_dir_ab    (FP64) per y frequency k: Uhat = F u (cos and sin row of k),
//               then V = T_k Uhat, T_k the symmetric Toeplitz matrix along x
//               of L_h at that frequency
//   k_dir_mul   (FP64) conv = F^T V and B^n;  W = B H^-1;  uhat = H^-1 W and
//               the leapfrog
// F[2k + s][j] = cos / sin(pi k j / N), k = 0 .. N: the DFT of length 2N along
// y, which embeds the 2N - 1 diagonals of L_h's Toeplitz blocks.  H^-1 is the
// one the Gohberg-Semencul sweeps apply (Sec. 3), here as a matrix: as
// I + E while E is small (the identity is then exact), whole where E is of
// order one (B + B E would cancel).  The FP32 forms keep the FFT convolution:
// with these products and tables in FP32 a diffusion run at N = 255 was 3e-6
// from FP64 against 2e-7.
//
// Used where it measured faster than the transforms (dir_mode).
#include <cuda_runtime.h>

#include <type_traits>

#include "ddouble.cuh"
#include "sadi_internal.h"

namespace sadi {
namespace {

// Where a product lets its dependent be scheduled: from N = 65 on only once its
// own operands are read.  The FP64 products are bound by the FP64 pipes, and
// blocks that arrive earlier unbalance the blocks over the SMs (N = 127: 46 us
// a step, 56 with the dependent let in at the start of the work, 114 with it
// let in at the kernel's entry; N = 63: 19, 16, 22).
__device__ __forceinline__ void pdl_wait(bool early) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_late() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ double g_dir(const DirInst<double>& I, double u) {
  if (I.gkind == 1) return -u * u * u;
  if (I.gkind == 2) return -sin(u);
  if (I.gkind == 3) return (I.gc1 + I.gc3 * u * u) * u + I.gcs * sin(u);
  return 0.0;
}

// B^n of element (j, i) at `at` from the convolution there (rhs_at in
// step_kernels.cu, the plain form)
__device__ __forceinline__ double rhs_dir(const DirInst<double>& I, size_t at, double conv) {
  const double u = I.u[at];
  const double f = I.src ? I.fsc * I.src[at] : 0.0;
  if (I.eq == 0) {
    const double gg = I.tau2 * (g_dir(I, u) + f);
    return I.first ? I.tau * I.phi2[at] + 0.5 * (conv + gg) : conv + gg;
  }
  const double d = I.first ? 0.0 : u - I.aux[at];
  return conv + I.tau2 * (g_dir(I, u + 0.5 * d) + f) - d;
}

// u^{n+1} of one element: compensated (FP32, in place) or plain (FP64)
template <typename T>
__device__ __forceinline__ void leap_dir(const DirInst<T>& I, size_t at, T uh) {
  if constexpr (sizeof(T) == 4) {
    const float hi = I.u[at], lo = I.lo[at];
    const float d = I.first ? uh : I.aux[at] + uh;
    const float s = hi + d;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (d - bb);
    const float l2 = lo + err;
    const float h2 = s + l2;
    I.next[at] = h2;
    I.lo[at] = l2 - (h2 - s);
    I.aux[at] = d;
  } else {
    const T uc = I.u[at];
    I.next[at] = I.first ? uc + uh : (T(2) * uc - I.aux[at]) + uh;
  }
}

// ---------------------------------------------------------------------------
// FP64: block = one row of F (the FP64 rate is the limit: many blocks, a
// thread per column and K part, both products)
template <int NC>
__global__ void __launch_bounds__(256) k_dir_ab64(const __grid_constant__ DirBatch<double> B) {
  constexpr int KP = 256 / NC;
  __shared__ double sF[NC], sU[NC], sT[NC], red[256];
  const DirInst<double>& I = B.in[blockIdx.y];
  const int N = I.N, r = blockIdx.x, tid = threadIdx.x;
  if (r >= 2 * N + 2) return;
  const int c = tid % NC, ks = tid / NC;
  if (tid < N) {
    sF[tid] = I.F[(size_t)r * N + tid];
    sT[tid] = I.T_[(size_t)(r / 2) * N + tid];
  }
  __syncthreads();
  pdl_wait(N <= 64);
  double a = 0.0;
  if (c < N) {
    if (I.beta == 0.0) {
#pragma unroll 8
      for (int j = ks; j < N; j += KP) a += sF[j] * I.x[(size_t)j * I.ld + c];
    } else {
      // the extrapolated field u + beta (u - u^{n-1})
#pragma unroll 4
      for (int j = ks; j < N; j += KP) {
        const size_t at = (size_t)j * I.ld + c;
        const double v = I.x[at];
        a += sF[j] * (v + I.beta * (v - I.x2[at]));
      }
    }
  }
  red[tid] = a;
  __syncthreads();
  if (tid < NC) {
    double s = red[tid];
#pragma unroll
    for (int p = 1; p < KP; ++p) s += red[p * NC + tid];
    sU[tid] = s;
  }
  __syncthreads();
  a = 0.0;
  if (c < N) {
#pragma unroll 8
    for (int i = ks; i < N; i += KP) a += sT[i > c ? i - c : c - i] * sU[i];
  }
  pdl_late();
  red[tid] = a;
  __syncthreads();
  if (tid < N) {
    double s = red[tid];
#pragma unroll
    for (int p = 1; p < KP; ++p) s += red[p * NC + tid];
    I.V[(size_t)r * I.ld + tid] = s;
  }
}

// ---------------------------------------------------------------------------
// C[m][n] = sum_k A(k, m) X(k, n) and the epilogue of its place in the step.
// MODE 0 (FP64): A = F, X = V (K = 2N + 2): B^n to Bm.  MODE 1: A = Bm by rows,
// X = E: W = B H^-1 to Wm.  MODE 2: A = E, X = Wm: uhat = H^-1 W, leapfrog.
// One of the two operands is a table in every mode: it is staged in shared
// memory before the kernel waits for the one before it (programmatic
// dependent launch), under that kernel's tail.
template <int MODE, typename T>
__device__ __forceinline__ void finish(const DirInst<T>& I, int m, int n, T acc) {
  const size_t at = (size_t)m * I.ld + n;
  if constexpr (MODE == 0) I.Bm[at] = rhs_dir(I, at, acc);
  else if constexpr (MODE == 1) I.Wm[at] = I.ident ? I.Bm[at] + acc : acc;
  else leap_dir(I, at, I.ident ? I.Wm[at] + acc : acc);
}

// FP32: 32 x 32 tile per block; four groups of 64 threads share the K range,
// each stages its own part of both operands whole (16-byte cp.async, one
// memory latency for the whole part; N <= 512: at most 133 KB a block) and
// works through it without a barrier: 4 x 4 outputs a thread, two 16-byte
// shared loads per 16 multiply-adds.  The partial sums meet in shared memory.
constexpr int kTile32 = 32;
struct Mul32Shape {
  int kq;    // K range of a group, a multiple of 4
  int pa;    // row pitch of the A panel of MODE 1 (by rows): pa / 4 odd, so that
             // eight rows' 16-byte pieces fall into distinct banks
  int group; // floats per group
};
__host__ __device__ inline Mul32Shape mul32_shape(int n) {
  Mul32Shape s;
  s.kq = ((n + 3) / 4 + 3) / 4 * 4;
  s.pa = (s.kq / 4) % 2 ? s.kq : s.kq + 4;
  s.group = kTile32 * (s.kq + s.pa);
  if (s.group < kTile32 * (kTile32 + 4)) s.group = kTile32 * (kTile32 + 4);   // the partial sums
  return s;
}
__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
template <int MODE>
__global__ void __launch_bounds__(256) k_dir_mul32(const __grid_constant__ DirBatch<float> B) {
  static_assert(MODE == 1 || MODE == 2, "the FP32 form has the sweeps only");
  extern __shared__ __align__(16) float smem[];
  const DirInst<float>& I = B.in[blockIdx.z];
  const int N = I.N, ld = I.ld, m0 = blockIdx.y * kTile32, n0 = blockIdx.x * kTile32;
  if (m0 >= N || n0 >= N) return;
  const int tid = threadIdx.x, g = tid / 64, lt = tid % 64, tx = lt % 8, ty = lt / 8;
  const Mul32Shape sh = mul32_shape(N);
  const int kq = sh.kq, kb = g * kq;
  float* sA = smem + g * sh.group;         // MODE 1: [32][pa]; MODE 2: [kq][32]
  float* sX = sA + kTile32 * sh.pa;        // [kq][32]
  // rows kb .. of a K-major operand (pitch ld, columns c0 .. c0 + 31; the
  // padding up to ld is finite and only reaches outputs that are not stored)
  auto panel = [&](float* dst, const float* src, int c0) {
    for (int e = lt; e < kq * 8; e += 64) {
      const int k = kb + e / 8;
      const bool ok = k < N;
      cp16(dst + (e / 8) * kTile32 + 4 * (e % 8), src + (size_t)(ok ? k : 0) * ld + c0 + 4 * (e % 8), ok);
    }
  };
  if constexpr (MODE == 1) panel(sX, I.E, n0);
  else panel(sA, I.E, m0);
  pdl_wait(N <= 64);
  if constexpr (MODE == 1) {
    // rows m0 .. of B^n, columns kb .. kb + kq - 1 (zero from N on)
    const int q4 = kq / 4;
    for (int e = lt; e < kTile32 * q4; e += 64) {
      const int m = e / q4, k = kb + 4 * (e % q4);
      const bool ok = m0 + m < N && k < N;
      cp16(sA + m * sh.pa + 4 * (e % q4), I.Bm + (size_t)(ok ? m0 + m : 0) * ld + (ok ? k : 0), ok);
    }
  } else {
    panel(sX, I.Wm, n0);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  asm volatile("bar.sync %0, 64;" ::"r"(1 + g) : "memory");
  // MODE 1: rows ty + 8 i (B^n's columns from N on are row padding, which the
  // zero rows of the E panel meet); MODE 2: rows 4 ty + i
  float acc[4][4] = {};
#pragma unroll 2
  for (int k = 0; k < kq; k += 4) {
    float a[4][4], x[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = MODE == 1 ? *reinterpret_cast<const float4*>(sA + (ty + 8 * i) * sh.pa + k)
                                 : *reinterpret_cast<const float4*>(sA + (k + i) * kTile32 + 4 * ty);
      const float4 w = *reinterpret_cast<const float4*>(sX + (k + i) * kTile32 + 4 * tx);
      a[i][0] = v.x, a[i][1] = v.y, a[i][2] = v.z, a[i][3] = v.w;
      x[i][0] = w.x, x[i][1] = w.y, x[i][2] = w.z, x[i][3] = w.w;
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += (MODE == 1 ? a[i][kk] : a[kk][i]) * x[kk][j];
  }
  pdl_late();
  __syncthreads();
  constexpr int LD = kTile32 + 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4*>(sA + (MODE == 1 ? ty + 8 * i : 4 * ty + i) * LD + 4 * tx) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int m = tid / 32 + 8 * e, n = tid % 32, o = m * LD + n;
    if (m0 + m < N && n0 + n < N)
      finish<MODE>(I, m0 + m, n0 + n,
                   (smem[o] + smem[sh.group + o]) + (smem[2 * sh.group + o] + smem[3 * sh.group + o]));
  }
}

// FP64: 4 x 8 outputs per block, one per lane; four warps share the K range.
// The table's panel in shared memory, the other operand 16 loads at a time.
template <int MODE>
__global__ void __launch_bounds__(128) k_dir_mul64(const __grid_constant__ DirBatch<double> B) {
  constexpr int KMAX = MODE == 0 ? 2 * 128 + 2 : 128, TC = MODE == 1 ? 8 : 4;   // table columns of the tile
  __shared__ double part[4][32], tab[KMAX * TC];
  const DirInst<double>& I = B.in[blockIdx.z];
  const int N = I.N, lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int m0 = blockIdx.y * 4, n0 = blockIdx.x * 8;
  if (m0 >= N || n0 >= N) return;
  const int m = m0 + lane / 8, n = n0 + lane % 8;
  const int K = MODE == 0 ? 2 * N + 2 : N, kq = (K + 3) / 4, k0 = w * kq, k1 = min(K, k0 + kq);
  const double* table = MODE == 0 ? I.F : I.E;
  const int c0 = MODE == 1 ? n0 : m0;
  for (int e = threadIdx.x; e < K * TC; e += 128) {
    const int c = c0 + e % TC;
    tab[e] = c < N ? table[(size_t)(e / TC) * N + c] : 0.0;
  }
  __syncthreads();
  pdl_wait(N <= 64);
  const bool ok = m < N && n < N;
  const int mc = ok ? m : 0, nc = ok ? n : 0;
  auto dyn = [&](int k) {   // volatile: sixteen loads in flight before the first product
    const double* p = MODE == 1 ? I.Bm + (size_t)mc * I.ld + k : (MODE == 0 ? I.V : I.Wm) + (size_t)k * I.ld + nc;
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
  };
  const double* tc = tab + (MODE == 1 ? lane % 8 : lane / 8);
  double a0 = 0.0, a1 = 0.0;
  for (int k = k0; k < k1; k += 16) {
    double v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = dyn(min(k + q, k1 - 1));
#pragma unroll
    for (int q = 0; q < 16; q += 2) {
      if (k + q < k1) a0 += tc[(k + q) * TC] * v[q];
      if (k + q + 1 < k1) a1 += tc[(k + q + 1) * TC] * v[q + 1];
    }
  }
  pdl_late();
  part[w][lane] = a0 + a1;
  __syncthreads();
  if (w == 0 && ok) finish<MODE>(I, m, n, (part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]));
}

// ---- tables ---------------------------------------------------------------------
// They are applied in every step, so their rounding is an error of the operator
// that a long run adds up, not noise.  F is rounded from double-double; E is
// refined (run_dir_inverse).
__global__ void k_dir_F(double* F, int N) {
  const size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (idx >= (size_t)(2 * N + 2) * N) return;
  const int r = (int)(idx / N), j = (int)(idx % N), k = r / 2;
  const int m = k * j % (2 * N);
  // sin(pi m / N) = cos(pi (2 m - N) / 2 N)
  if (!(r & 1)) F[idx] = dd::cospi(m, N).hi;
  else F[idx] = (k == 0 || k == N) ? 0.0 : dd::cospi(2 * m < N ? N - 2 * m : 2 * m - N, 2 * N).hi;
}
// T[k][d] = scale w_k / 2N (a_d0 + 2 sum_e a_de cos(pi k e / N)), w_k = 1 at k = 0, N, else 2
//
// The eigenvalues of L_h at low frequencies are small differences of these
// numbers.  So the sums are double-double, and the rounding error of entry d
// is carried to entry d + 1 (halved from d = 0, which appears once in a row
// where the others appear twice): at low frequencies the errors cancel, at high
// ones they stay within the rounding of the eigenvalue itself.  Against 64-bit
// sums rounded one by one, and E as the recurrence leaves it, the field after 60
// steps at N = 128, alpha = 1.9 is 3.5e-15 from the scheme on the same weights
// instead of 1.4e-13 (the transforms: 2.1e-14), with the same products in the
// step; creating a context of N = 127 takes 2.07 instead of 1.98 ms.  One block
// per k, a thread per d.
__global__ void __launch_bounds__(128) k_dir_T(double* out, const double* __restrict__ a2d, int N, double scale) {
  __shared__ dd::D2 c[2 * 128], t[128];
  const int k = blockIdx.x;
  for (int m = threadIdx.x; m < 2 * N; m += blockDim.x) c[m] = dd::cospi(m, N);
  __syncthreads();
  for (int d = threadIdx.x; d < N; d += blockDim.x) {
    dd::D2 acc{a2d[(size_t)d * N], 0.0};
    for (int e = 1; e < N; ++e) acc = dd::add(acc, dd::mul(c[k * e % (2 * N)], 2.0 * a2d[(size_t)d * N + e]));
    t[d] = dd::div(dd::mul(acc, (k == 0 || k == N) ? scale : 2.0 * scale), 2.0 * N);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  dd::D2 carry{0.0, 0.0};
  for (int d = 0; d < N; ++d) {
    const dd::D2 w = dd::add(t[d], carry);   // w.hi: w rounded
    out[(size_t)k * N + d] = w.hi;
    carry = {d == 0 ? 0.5 * w.lo : w.lo, 0.0};
  }
}

template <typename K, typename Batch>
cudaError_t launch_pdl(K kernel, dim3 grid, int threads, cudaStream_t st, const Batch& b, size_t smem = 0) {
  cudaLaunchAttribute a[1];
  a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = a;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, b);
}

template <int MODE, typename T>
cudaError_t launch_mul(const DirBatch<T>& b, int n, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    static LaunchCache done[kLauncherDevices];
    const int dev = device_slot();
    if (dev < 0) return cudaErrorInvalidDevice;
    if (!done[dev].load(std::memory_order_acquire)) {
      const cudaError_t e = cudaFuncSetAttribute(k_dir_mul32<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 4 * mul32_shape(512).group * (int)sizeof(float));
      if (e != cudaSuccess) return e;
      done[dev].store(1, std::memory_order_release);
    }
    return launch_pdl(k_dir_mul32<MODE>, dim3((n + 31) / 32, (n + 31) / 32, b.count), 256, st, b,
                      4 * mul32_shape(n).group * sizeof(float));
  } else
    return launch_pdl(k_dir_mul64<MODE>, dim3((n + 7) / 8, (n + 3) / 4, b.count), 128, st, b);
}

}  // namespace

template <typename T>
cudaError_t launch_dir_sweeps(const DirBatch<T>& b, int max_n, cudaStream_t st, cudaEvent_t* ev) {
  cudaError_t e = launch_mul<1>(b, max_n, st);
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[3], st);
  e = launch_mul<2>(b, max_n, st);
  if (e == cudaSuccess && ev) cudaEventRecord(ev[4], st);
  return e;
}

cudaError_t launch_dir_step(const DirBatch<double>& b, int max_n, cudaStream_t st, cudaEvent_t* ev) {
  cudaError_t e;
  if (ev) cudaEventRecord(ev[0], st);
  const dim3 grid(2 * max_n + 2, b.count);
  if (max_n <= 64) e = launch_pdl(k_dir_ab64<64>, grid, 256, st, b);
  else if (max_n <= 128) e = launch_pdl(k_dir_ab64<128>, grid, 256, st, b);
  else e = cudaErrorInvalidValue;
  if (e != cudaSuccess) return e;
  if (ev) cudaEventRecord(ev[1], st);
  if ((e = launch_mul<0>(b, max_n, st))) return e;
  if (ev) cudaEventRecord(ev[2], st);
  return launch_dir_sweeps<double>(b, max_n, st, ev);
}

cudaError_t run_dir_tables(double* F, double* Tk, const double* a2d, int N, double scale, cudaStream_t st) {
  if (N > 128) return cudaErrorInvalidValue;
  const size_t nf = (size_t)(2 * N + 2) * N;
  k_dir_F<<<(unsigned)((nf + 255) / 256), 256, 0, st>>>(F, N);
  k_dir_T<<<(unsigned)(N + 1), 128, 0, st>>>(Tk, a2d, N, scale);
  return cudaGetLastError();
}

template cudaError_t launch_dir_sweeps<float>(const DirBatch<float>&, int, cudaStream_t, cudaEvent_t*);

}  // namespace sadi
