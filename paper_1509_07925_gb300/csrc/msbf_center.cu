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
constexpr int kCLanes = 64;   // threads of a share (forward)
constexpr int kCXt = 4;       // outputs x per thread (forward), kCLanes apart
constexpr int kCX = kCLanes * kCXt;
constexpr int kCShares = kCThreads / kCLanes;   // shares of the centre points (forward)
constexpr int kCTile = 512;   // centre points staged per round (what the buffer holds)
constexpr int kCBatch = 2;    // centre points whose kernel entries are in flight per thread

// Forward, few CTAs: a CTA computes 256 outputs x for 8 RHS; its four shares of 64 threads
// take the centre points of a round in turn and their sums are added at the end, always in
// the same order.  Four outputs a thread, so that a shared load of g serves four of them.
// n = 128, 289 points, 32 RHS from a cold cache (16 us of multiply-adds): 88 us with one
// thread per x over all the centre points, 53 us so (58 us with 16 RHS a CTA).
__global__ void __launch_bounds__(kCThreads) center_fwd_kernel(const float2* __restrict__ Kc,
                                                               const int32_t* __restrict__ idx, int n_c,
                                                               const float2* __restrict__ g, int64_t len_in,
                                                               float2* __restrict__ u, int64_t n_out, int nrhs,
                                                               int accumulate) {
  // g of the round's centre points [point][RHS]; at the end sums [share][RHS][x]
  __shared__ __align__(16) float2 buf[2 * kCRhs * kCX];
  static_assert(kCTile <= 2 * kCX && kCShares == 4, "buf holds either");
  const int xl = threadIdx.x % kCLanes, share = threadIdx.x / kCLanes;
  const int64_t x0 = int64_t(blockIdx.x) * kCX + xl;
  const int r0 = blockIdx.y * kCRhs;
  int64_t xk[kCXt];             // (outputs beyond the last: the last one's entries, not stored)
#pragma unroll
  for (int i = 0; i < kCXt; ++i) xk[i] = x0 + i * kCLanes < n_out ? x0 + i * kCLanes : n_out - 1;
  float2 acc[kCXt][kCRhs];
#pragma unroll
  for (int i = 0; i < kCXt; ++i)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) acc[i][r] = make_float2(0.f, 0.f);
  for (int c0 = 0; c0 < n_c; c0 += kCTile) {
    const int nc = min(kCTile, n_c - c0);
    __syncthreads();
#pragma unroll 4
    for (int q = threadIdx.x; q < nc * kCRhs; q += kCThreads) {
      const int cc = q / kCRhs, r = q - cc * kCRhs;
      buf[q] = r0 + r < nrhs ? __ldg(g + int64_t(r0 + r) * len_in + __ldg(idx + c0 + cc)) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int cc = share; cc < nc; cc += kCShares * kCBatch) {
      float2 k[kCBatch][kCXt];
#pragma unroll
      for (int b = 0; b < kCBatch; ++b)
        if (cc + b * kCShares < nc)
#pragma unroll
          for (int i = 0; i < kCXt; ++i) k[b][i] = __ldg(Kc + int64_t(c0 + cc + b * kCShares) * n_out + xk[i]);
#pragma unroll
      for (int b = 0; b < kCBatch; ++b)
        if (cc + b * kCShares < nc) {
          const float4* gv = reinterpret_cast<const float4*>(buf + (cc + b * kCShares) * kCRhs);
#pragma unroll
          for (int r2 = 0; r2 < kCRhs / 2; ++r2) {
            const float4 v = gv[r2];
#pragma unroll
            for (int i = 0; i < kCXt; ++i) {
              float2 &s = acc[i][2 * r2], &t = acc[i][2 * r2 + 1];
              s.x = fmaf(k[b][i].x, v.x, fmaf(-k[b][i].y, v.y, s.x));
              s.y = fmaf(k[b][i].x, v.y, fmaf(k[b][i].y, v.x, s.y));
              t.x = fmaf(k[b][i].x, v.z, fmaf(-k[b][i].y, v.w, t.x));
              t.y = fmaf(k[b][i].x, v.w, fmaf(k[b][i].y, v.z, t.y));
            }
          }
        }
    }
  }
  // shares 2 and 3 to 0 and 1, then 1 to 0
  for (int n = 2; n > 0; n >>= 1) {
    __syncthreads();
    if (share >= n && share < 2 * n)
#pragma unroll
      for (int i = 0; i < kCXt; ++i)
#pragma unroll
        for (int r = 0; r < kCRhs; ++r) buf[((share - n) * kCRhs + r) * kCX + i * kCLanes + xl] = acc[i][r];
    __syncthreads();
    if (share < n)
#pragma unroll
      for (int i = 0; i < kCXt; ++i)
#pragma unroll
        for (int r = 0; r < kCRhs; ++r) {
          const float2 w = buf[(share * kCRhs + r) * kCX + i * kCLanes + xl];
          acc[i][r].x += w.x;
          acc[i][r].y += w.y;
        }
  }
  if (share == 0)
#pragma unroll
    for (int i = 0; i < kCXt; ++i)
#pragma unroll
      for (int r = 0; r < kCRhs; ++r)
        if (x0 + i * kCLanes < n_out && r0 + r < nrhs) {
          float2* o = u + int64_t(r0 + r) * n_out + x0 + i * kCLanes;
          float2 v = acc[i][r];
          if (accumulate) {
            const float2 w = *o;
            v.x += w.x;
            v.y += w.y;
          }
          *o = v;
        }
}

// Forward, many CTAs: one output a thread over all the centre points, so that six CTAs share
// an SM (42 registers; two of the kernel above) and hide one another's loads.
__global__ void __launch_bounds__(kCThreads) center_fwd_many_kernel(const float2* __restrict__ Kc,
                                                                    const int32_t* __restrict__ idx, int n_c,
                                                                    const float2* __restrict__ g, int64_t len_in,
                                                                    float2* __restrict__ u, int64_t n_out, int nrhs,
                                                                    int accumulate) {
  __shared__ float2 gs[kCTile][kCRhs];
  const int64_t x = int64_t(blockIdx.x) * kCX + threadIdx.x;
  const int r0 = blockIdx.y * kCRhs;
  static_assert(kCX == kCThreads, "one output a thread");
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
    if (x < n_out)
      for (int cc = 0; cc < nc; ++cc) {
        const float2 k = __ldg(Kc + int64_t(c0 + cc) * n_out + x);
#pragma unroll
        for (int r = 0; r < kCRhs; ++r) {
          const float2 v = gs[cc][r];
          acc[r].x = fmaf(k.x, v.x, fmaf(-k.y, v.y, acc[r].x));
          acc[r].y = fmaf(k.x, v.y, fmaf(k.y, v.x, acc[r].y));
        }
      }
  }
  if (x >= n_out) return;
#pragma unroll
  for (int r = 0; r < kCRhs; ++r) {
    if (r0 + r >= nrhs) break;
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

// Adjoint: one CTA per P centre points and 8 RHS, a block reduction over x; each u
// value read serves all the CTA's centre points.
template <int P>
__global__ void __launch_bounds__(kCThreads) center_adj_kernel(const float2* __restrict__ Kc,
                                                               const int32_t* __restrict__ idx, int n_c,
                                                               const float2* __restrict__ u, int64_t n_out,
                                                               float2* __restrict__ g, int64_t len_in, int nrhs) {
  __shared__ float2 red[kCThreads / 32][P][kCRhs];
  const int c0 = blockIdx.x * P, r0 = blockIdx.y * kCRhs;
  float2 acc[P][kCRhs];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r) acc[p][r] = make_float2(0.f, 0.f);
  for (int64_t x = threadIdx.x; x < n_out; x += kCThreads) {
    float2 k[P], v[kCRhs];
#pragma unroll
    for (int p = 0; p < P; ++p) k[p] = __ldg(Kc + int64_t(min(c0 + p, n_c - 1)) * n_out + x);   // use conj(k)
#pragma unroll
    for (int r = 0; r < kCRhs; ++r)
      v[r] = r0 + r < nrhs ? __ldg(u + int64_t(r0 + r) * n_out + x) : make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int r = 0; r < kCRhs; ++r) {
        acc[p][r].x = fmaf(k[p].x, v[r].x, fmaf(k[p].y, v[r].y, acc[p][r].x));
        acc[p][r].y = fmaf(k[p].x, v[r].y, fmaf(-k[p].y, v[r].x, acc[p][r].y));
      }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int p = 0; p < P; ++p)
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
  if (p < P && c0 + p < n_c && r0 + r < nrhs) {
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
                              float2* u, int64_t n_out, int nrhs, bool accumulate, int sms, cudaStream_t st) {
  if (n_c == 0) {
    if (accumulate) return cudaSuccess;
    return cudaMemsetAsync(u, 0, size_t(nrhs) * size_t(n_out) * sizeof(float2), st);
  }
  const dim3 grid(unsigned((n_out + kCX - 1) / kCX), unsigned((nrhs + kCRhs - 1) / kCRhs));
  // four shares a CTA up to the two CTAs to an SM that they leave room for; beyond those one
  // output a thread.  us of either with 256, 512 and 2048 CTAs: n = 128, 81 points 22 / 30,
  // 37 / 31; 289 points 53 / 88, 94 / 92; n = 256, 289 points 63 / 107, 113 / 109, 361 / 301.
  // (Between 768 and 1024 CTAs the shares are at times faster, 553 / 678 us at 1089 points.)
  const auto kern = int64_t(grid.x) * grid.y <= 2 * int64_t(sms) ? center_fwd_kernel : center_fwd_many_kernel;
  kern<<<grid, kCThreads, 0, st>>>(Kc, idx, n_c, g, len_in, u, n_out, nrhs, accumulate ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_center_adj(const float2* Kc, const int32_t* idx, int n_c, const float2* u, int64_t n_out,
                              float2* g, int64_t len_in, int nrhs, int sms, cudaStream_t st) {
  if (n_c == 0) return cudaSuccess;
  // four centre points a CTA, or two where that leaves fewer CTAs than SMs.  us with two and
  // with four: n = 128, 289 points, 8 RHS (73 CTAs of four) 53 and 57, 32 RHS (292) 108 and 59;
  // n = 64, 1 RHS 18 and 20; n = 256, 1089 points (273) 386 and 245 us.  (One point a CTA,
  // the RHS loop cut at nrhs: 117, 196, 18 and 418 us.)
  const int y = (nrhs + kCRhs - 1) / kCRhs;
  const bool few = int64_t((n_c + 3) / 4) * y < sms;
  const dim3 grid(unsigned(few ? (n_c + 1) / 2 : (n_c + 3) / 4), unsigned(y));
  const auto kern = few ? center_adj_kernel<2> : center_adj_kernel<4>;
  kern<<<grid, kCThreads, 0, st>>>(Kc, idx, n_c, u, n_out, g, len_in, nrhs);
  return cudaGetLastError();
}

}  // namespace mbf
