// Dense centre term of the multiscale butterfly factorization (§4.2, eq. f1):
//   forward  u[r][x]      (= or +=) sum_c K_C[c][x] g[r][idx[c]]
//   adjoint  g[r][idx[c]]   +=      sum_x conj(K_C[c][x]) u[r][x]
// K_C is stored centre-point-major ([c][x], complex64), so a warp reads consecutive x.
#include <cuda_runtime.h>

#include <cstdint>

#include "msbf.hpp"

namespace mbf {

namespace {

constexpr int kCThreads = 256;
constexpr int kCRhs = 8;      // RHS per CTA
constexpr int kCX = 64;       // outputs x of a CTA (forward)
constexpr int kCShares = kCThreads / kCX;   // shares of the centre points (forward)
constexpr int kCTile = 128;   // centre points staged per round
constexpr int kCBatch = 8;    // K_C entries in flight per thread
constexpr int kCPts = 4;      // centre points per CTA (adjoint)

// Forward: a CTA computes 64 outputs x for 8 RHS; its four shares of 64 threads take the
// centre points of a round in turn and their sums are added at the end, always in the
// same order.  One thread per x over all the centre points (an earlier form) left each
// thread a serial chain of loads and the chip at 14 warps an SM: 81 us for n = 128, 289
// points, 32 RHS, from a cold cache; now 52 us.
__global__ void __launch_bounds__(kCThreads) center_fwd_kernel(const float2* __restrict__ Kc,
                                                               const int32_t* __restrict__ idx, int n_c,
                                                               const float2* __restrict__ g, int64_t len_in,
                                                               float2* __restrict__ u, int64_t n_out, int nrhs,
                                                               int accumulate) {
  __shared__ __align__(16) float2 gs[kCTile][kCRhs];
  __shared__ float2 part[kCShares - 1][kCRhs][kCX];
  const int xl = threadIdx.x % kCX, share = threadIdx.x / kCX;
  const int64_t x = int64_t(blockIdx.x) * kCX + xl;
  const int r0 = blockIdx.y * kCRhs;
  const float2* kx = Kc + (x < n_out ? x : n_out - 1);
  float2 acc[kCRhs];
#pragma unroll
  for (int r = 0; r < kCRhs; ++r) acc[r] = make_float2(0.f, 0.f);
  for (int c0 = 0; c0 < n_c; c0 += kCTile) {
    const int nc = min(kCTile, n_c - c0);
    __syncthreads();
    for (int q = threadIdx.x; q < nc * kCRhs; q += kCThreads) {
      const int cc = q / kCRhs, r = q - cc * kCRhs;
      gs[cc][r] = r0 + r < nrhs ? __ldg(g + int64_t(r0 + r) * len_in + idx[c0 + cc]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int cc = share; cc < nc; cc += kCShares * kCBatch) {
      float2 k[kCBatch];
#pragma unroll
      for (int b = 0; b < kCBatch; ++b)
        if (cc + b * kCShares < nc) k[b] = __ldg(kx + int64_t(c0 + cc + b * kCShares) * n_out);
#pragma unroll
      for (int b = 0; b < kCBatch; ++b)
        if (cc + b * kCShares < nc) {
          const float4* gv = reinterpret_cast<const float4*>(gs[cc + b * kCShares]);
#pragma unroll
          for (int r2 = 0; r2 < kCRhs / 2; ++r2) {
            const float4 v = gv[r2];
            acc[2 * r2].x = fmaf(k[b].x, v.x, fmaf(-k[b].y, v.y, acc[2 * r2].x));
            acc[2 * r2].y = fmaf(k[b].x, v.y, fmaf(k[b].y, v.x, acc[2 * r2].y));
            acc[2 * r2 + 1].x = fmaf(k[b].x, v.z, fmaf(-k[b].y, v.w, acc[2 * r2 + 1].x));
            acc[2 * r2 + 1].y = fmaf(k[b].x, v.w, fmaf(k[b].y, v.z, acc[2 * r2 + 1].y));
          }
        }
    }
  }
  if (share > 0)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) part[share - 1][r][xl] = acc[r];
  __syncthreads();
  if (share == 0) {
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) {
#pragma unroll
      for (int s = 0; s < kCShares - 1; ++s) {
        acc[r].x += part[s][r][xl].x;
        acc[r].y += part[s][r][xl].y;
      }
      if (x < n_out && r0 + r < nrhs) {
        float2* o = u + int64_t(r0 + r) * n_out + x;
        float2 v = acc[r];
        if (accumulate) {
          const float2 w = *o;
          v.x += w.x;
          v.y += w.y;
        }
        *o = v;
      }
    }
  }
}

// Adjoint: one CTA per kCPts centre points and 8 RHS, a block reduction over x; each u
// value read serves all the CTA's centre points.
__global__ void __launch_bounds__(kCThreads) center_adj_kernel(const float2* __restrict__ Kc,
                                                               const int32_t* __restrict__ idx, int n_c,
                                                               const float2* __restrict__ u, int64_t n_out,
                                                               float2* __restrict__ g, int64_t len_in, int nrhs) {
  __shared__ float2 red[kCThreads / 32][kCPts][kCRhs];
  const int c0 = blockIdx.x * kCPts, r0 = blockIdx.y * kCRhs;
  float2 acc[kCPts][kCRhs];
#pragma unroll
  for (int p = 0; p < kCPts; ++p)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) acc[p][r] = make_float2(0.f, 0.f);
  for (int64_t x = threadIdx.x; x < n_out; x += kCThreads) {
    float2 k[kCPts], v[kCRhs];
#pragma unroll
    for (int p = 0; p < kCPts; ++p) k[p] = __ldg(Kc + int64_t(min(c0 + p, n_c - 1)) * n_out + x);   // use conj(k)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r)
      v[r] = r0 + r < nrhs ? __ldg(u + int64_t(r0 + r) * n_out + x) : make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < kCPts; ++p)
#pragma unroll
      for (int r = 0; r < kCRhs; ++r) {
        acc[p][r].x = fmaf(k[p].x, v[r].x, fmaf(k[p].y, v[r].y, acc[p][r].x));
        acc[p][r].y = fmaf(k[p].x, v[r].y, fmaf(-k[p].y, v[r].x, acc[p][r].y));
      }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int p = 0; p < kCPts; ++p)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) {
      float sx = acc[p][r].x, sy = acc[p][r].y;
      for (int off = 16; off > 0; off >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, off);
        sy += __shfl_xor_sync(0xffffffffu, sy, off);
      }
      if (lane == 0) red[warp][p][r] = make_float2(sx, sy);
    }
  __syncthreads();
  const int p = int(threadIdx.x) / kCRhs, r = int(threadIdx.x) % kCRhs;
  if (p < kCPts && c0 + p < n_c && r0 + r < nrhs) {
    float2 s = make_float2(0.f, 0.f);
    for (int w = 0; w < kCThreads / 32; ++w) {
      s.x += red[w][p][r].x;
      s.y += red[w][p][r].y;
    }
    float2* o = g + int64_t(r0 + r) * len_in + idx[c0 + p];
    const float2 w = *o;
    *o = make_float2(w.x + s.x, w.y + s.y);
  }
}

}  // namespace

cudaError_t launch_center_fwd(const float2* Kc, const int32_t* idx, int n_c, const float2* g, int64_t len_in,
                              float2* u, int64_t n_out, int nrhs, bool accumulate, cudaStream_t st) {
  if (n_c == 0) {
    if (accumulate) return cudaSuccess;
    return cudaMemsetAsync(u, 0, size_t(nrhs) * size_t(n_out) * sizeof(float2), st);
  }
  const dim3 grid(unsigned((n_out + kCX - 1) / kCX), unsigned((nrhs + kCRhs - 1) / kCRhs));
  center_fwd_kernel<<<grid, kCThreads, 0, st>>>(Kc, idx, n_c, g, len_in, u, n_out, nrhs, accumulate ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_center_adj(const float2* Kc, const int32_t* idx, int n_c, const float2* u, int64_t n_out,
                              float2* g, int64_t len_in, int nrhs, cudaStream_t st) {
  if (n_c == 0) return cudaSuccess;
  const dim3 grid(unsigned((n_c + kCPts - 1) / kCPts), unsigned((nrhs + kCRhs - 1) / kCRhs));
  center_adj_kernel<<<grid, kCThreads, 0, st>>>(Kc, idx, n_c, u, n_out, g, len_in, nrhs);
  return cudaGetLastError();
}

}  // namespace mbf
