// border.cuh -- the border correction of a Gohberg-Semencul sweep as one tiled
// product: C[m][n] += sum_p P[p][m] Q[p][n], p < r = N' - N.
//
// A sweep on N points solves a bordered system of N' = 2^k unknowns and adds
// G ybot to each vector (ybot: its r bottom entries).  For small r the sweep
// kernels add it themselves, one column of G per bottom entry.  From
// r > kBorderInline on every vector would read the whole of G (N = 700: 0.9 MB
// per row), so the sweep kernels store ybot (r x N) instead and this kernel
// multiplies 64 x 64 tiles, each operand element read once per 64 outputs: bound
// by the FP32 multiply-adds (N = 700, r = 324: 0.16 G per sweep; the step 124
// us, 1485 with G read per vector).  Below the line the extra launch costs more
// than it saves.
#pragma once
#include <cuda_runtime.h>

#include "sadi_internal.h"

namespace sadi {
namespace border {

constexpr int kTile = 64, kK = 16, kThreads = 256;

// MODE 0: the x sweep by columns, W[k][row] += sum_p G[p][k] ybot[p][row].
// MODE 1: the y sweep, uhat[j][i] = U[j][i] + sum_p G[p][j] ybot[p][i], and the
// compensated leapfrog of its element (step_blk.cuh).
template <int MODE>
__global__ void __launch_bounds__(kThreads) k_border(const __grid_constant__ RegBatch B) {
  __shared__ __align__(16) float sp[2][kK][kTile], sq[2][kK][kTile];
  const RegInst& I = B.in[blockIdx.z];
  const int N = I.N, r = I.r;
  const int m0 = blockIdx.y * kTile, n0 = blockIdx.x * kTile;
  if (r <= kBorderInline || m0 >= N || n0 >= N) return;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  pdl_entry();
  const float *P = I.G, *Q = ybot_of(I, N + r);   // N' = N + r
  const int ldp = N, ldq = I.ld;
  float acc[4][4] = {};
  // thread -> element (p, column) of a K block: 4 of each operand
  float pv[4], qv[4];
  auto load = [&](int p0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + kThreads * e, p = p0 + idx / kTile, c = idx % kTile;
      pv[e] = (p < r && m0 + c < N) ? P[(size_t)p * ldp + m0 + c] : 0.f;
      qv[e] = (p < r && n0 + c < N) ? Q[(size_t)p * ldq + n0 + c] : 0.f;
    }
  };
  auto stage = [&](int b) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int idx = tid + kThreads * e;
      sp[b][idx / kTile][idx % kTile] = pv[e];
      sq[b][idx / kTile][idx % kTile] = qv[e];
    }
  };
  load(0);
  stage(0);
  __syncthreads();
  const int nk = (r + kK - 1) / kK;
  for (int kb = 0; kb < nk; ++kb) {
    if (kb + 1 < nk) load((kb + 1) * kK);
    const int b = kb & 1;
#pragma unroll
    for (int p = 0; p < kK; ++p) {
      const float4 a = *reinterpret_cast<const float4*>(&sp[b][p][4 * ty]);
      const float4 c = *reinterpret_cast<const float4*>(&sq[b][p][4 * tx]);
      const float av[4] = {a.x, a.y, a.z, a.w}, cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += av[i] * cv[j];
    }
    if (kb + 1 < nk) stage(b ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + 4 * ty + i;
    if (m >= N) break;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n >= N) break;
      const size_t at = (size_t)m * I.ld + n;
      if constexpr (MODE == 0) {
        I.W[at] += acc[i][j];
      } else {
        const float uh = reinterpret_cast<const float*>(I.S)[at] + acc[i][j];
        const float hi = I.u_hi[at], lo = I.u_lo[at];
        const float d = I.first ? uh : I.u_d[at] + uh;
        const float s = hi + d;
        const float bb = s - hi;
        const float err = (hi - (s - bb)) + (d - bb);
        const float l2 = lo + err;
        const float h2 = s + l2;
        I.u_hi[at] = h2;
        I.u_lo[at] = l2 - (h2 - s);
        I.u_d[at] = d;
      }
    }
  }
}

// whether a member of the batch needs the separate correction
inline bool any(const RegBatch& b) {
  for (int k = 0; k < b.count; ++k)
    if (b.in[k].r > kBorderInline) return true;
  return false;
}

// one launch for all members (a programmatic dependent of the kernel before it)
template <int MODE>
cudaError_t launch(const RegBatch& b, int max_n, cudaStream_t st) {
  cudaLaunchAttribute a[1];
  a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  const unsigned t = (unsigned)((max_n + kTile - 1) / kTile);
  cfg.gridDim = dim3(t, t, (unsigned)b.count);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cfg.attrs = a;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_border<MODE>, b);
}

}  // namespace border
}  // namespace sadi
