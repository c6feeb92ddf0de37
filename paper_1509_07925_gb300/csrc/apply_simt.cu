// Persistent SIMT apply of a butterfly factorization on sm_103a (FP32 arithmetic on
// complex64 factors; one pass of 1, 2, 4 or 8 right-hand sides per launch).
//
// A CTA walks every stage of eq. (gbf) -- (V^L)^*, (H^l)^*, M^h, G^l, U^L -- in order (or
// in reverse, conjugated, for K^*) and works as one on a group at a time; its warps have
// roles that run ahead of one another:
//   consumers (W)  multiply the group's block by its inputs, reduce, store;
//   gather (GA)    each takes every GA-th group, waits until the group's inputs are counted
//                  in and copies them (or the leaf points' values) into its shared-memory
//                  buffer, so that dependency waits and L2 round trips overlap the products;
//   producer       streams the factor chunks (cp.async.bulk) into a ring of 8 KB slots;
//                  factor data does not depend on the vectors, so the stream runs ahead
//                  across group and stage boundaries;
//   signal         makes finished groups' outputs visible and counts them in for their
//                  consumers, off the consumers' path.
// There is no grid-wide barrier: a group starts when its c inputs are counted in.
// Every wait gives up after a limit and sets the status word; all roles then leave,
// each after waiting for its own copies.
//
// What bounds it: the factor bytes from HBM (a pass reads each once), next to the chain
// per group (wait, block, reduction, stores: about 2 us on one CTA's warps, whose products
// take a fifth of it).  So two CTAs share an SM where each has a group (launch_n), and one
// group's chain hides the other's.  A group to a warp, as before, had 1/8 of the SM's
// bandwidth and a private ring of three slots for it: every stage ended in a wait for
// streams.  Polar FIO n = 256, L = 6, r = 24 (389 MB of factors), one RHS: 110.6 us with a
// group to a warp, 111 us with a group to a CTA of 8 warps and one CTA to an SM, 76 us
// with two CTAs of 4 (5.08 TB/s); adjoint 280 -> 117 us (16-byte loads, 16 totals reduced
// over the lanes in 16 exchanges instead of 5 each); n = 128 with 7 RHS 472 -> 144 us (one
// pass of 8 instead of 4 + 3); n = 64, L = 4 with 5 RHS 199 -> 36 us; 2-D DFT n = 64, L = 4,
// r = 16, one RHS 50 -> 20 us.  Many small blocks, where a group to a warp did best: 2-D DFT
// n = 64, L = 6 with 1 and 2 RHS, r = 4 44.5 / 46.5 -> 43.6 / 46.2 us, r = 8 46.7 / 50.6 ->
// 43.7 / 48.7; n = 256, L = 8, r = 4 654 / 776 -> 655 / 757 (the many lines side by side of such
// blocks are added in pairs; one after another they took r = 4 to 55.1 / 61.2 and 876 / 1002).
// The kernels of 4 and 8 RHS spill 40 to 120 bytes (128 registers a thread).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "apply.hpp"

namespace mbf {

constexpr int kMaxSlots = 24;

// ------------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Row of RHS `rhs` of the input / output: contiguous [nrhs][len], or the row table.
__device__ __forceinline__ const float2* in_row(const ApplyArgs& a, int rhs) {
  return a.use_rows ? a.rows.in[rhs] : a.in + int64_t(rhs) * a.in_len;
}
__device__ __forceinline__ float2* out_row(const ApplyArgs& a, int rhs) {
  return a.use_rows ? a.rows.out[rhs] : a.out + int64_t(rhs) * a.out_len;
}

__device__ __forceinline__ void set_status(int* status, volatile int* abort, int code) {
  atomicCAS(status, 0, code);
  *abort = 1;
}

// B, c^h and c are powers of two: the group and segment maps are shifts (a division each for
// the gather and signal warps cost 4 us of 48 over the 7 stages of n = 64, L = 6).
__device__ __forceinline__ int lg2(int x) { return 31 - __clz(x); }

// The group of stage `s` whose input pattern `pat` reads segment P (position P * R).
__device__ __forceinline__ int pat_group(int pat, int P, const Stage& s, int c) {
  const int lc = lg2(c), lb = lg2(s.B);
  if (pat == PAT_CONTIG) return P >> lc;
  if (pat == PAT_SPLIT) return (((P >> lb) >> lc) << lb) + (P & (s.B - 1));
  return ((P & (s.ch - 1)) << lb) + ((P >> lg2(s.ch)) >> lc);   // PAT_CORNER: P = (c b + t) ch + a, g = a B + b
}

__device__ __forceinline__ bool item_ok(const Item& it) {
  return it.len >= 1 && it.len <= kMaxLen && it.lpc >= 1 && it.lpc <= kMaxChunkLines &&
         it.nlines <= (it.kind == ITEM_MAIN ? kMaxLen : kMaxLeaf) &&
         chunk_bytes(it.lpc, it.len) <= kSlotBytes;
}

// Bounded wait on an mbarrier phase.  False on a timeout (which sets the status) or when
// the launch is being abandoned.  The clock is read every 64th try only: reading it costs
// more than a try.
__device__ __forceinline__ bool wait_bar(uint64_t* b, uint32_t ph, const ApplyArgs& a, volatile int* abort,
                                         uint64_t lim, int code) {
  if (mbar_try(b, ph)) return true;
  uint64_t t0 = 0;
  for (unsigned n = 1;; ++n) {
    if (mbar_try(b, ph)) return true;
    if ((n & 63u) == 0) {
      if (*abort) return false;
      const uint64_t t = gtimer();
      if (t0 == 0) t0 = t;
      if (t - t0 > lim) {
        set_status(a.status, abort, code);
        return false;
      }
    }
  }
}
// Non-blocking test of a phase (try_wait may suspend the whole warp).
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b, uint32_t count = 1) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
// Group counter in shared memory: written by one consumer after the CTA's barrier, read
// by the signal warp.
__device__ __forceinline__ void st_release_cta(volatile unsigned* p, unsigned v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_addr(const_cast<unsigned*>(p))), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_cta(const volatile unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];"
               : "=r"(v)
               : "r"(smem_addr(const_cast<const unsigned*>(p)))
               : "memory");
  return v;
}
template <int W>
__device__ __forceinline__ void cons_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(W * 32) : "memory");
}

// Segment t of a group starts at base + t * step in the coefficient vector.
struct SegMap {
  int base, step;        // entries (the coefficient vectors hold fewer than 2^31)
};
__device__ __forceinline__ SegMap seg_map(int pat, int g, const Stage& s, int R, int c) {
  if (pat == PAT_CONTIG) return {c * g * R, R};
  const int a = g >> lg2(s.B), b = g & (s.B - 1);
  if (pat == PAT_SPLIT) return {(c * a * s.B + b) * R, s.B * R};
  return {(c * b * s.ch + a) * R, s.ch * R};         // PAT_CORNER
}
// Segment of entry e of c segments of R entries (c = 4 or 8).
__device__ __forceinline__ int seg_of(int e, int R, int c) {
  int t = (e >= R ? 1 : 0) + (e >= 2 * R ? 1 : 0) + (e >= 3 * R ? 1 : 0);
  if (c > 4) t += (e >= 4 * R ? 1 : 0) + (e >= 5 * R ? 1 : 0) + (e >= 6 * R ? 1 : 0) + (e >= 7 * R ? 1 : 0);
  return t;
}

// Loads by shared-memory address (32-bit address arithmetic, and never a generic load).
__device__ __forceinline__ float lds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
// NR consecutive complex values (16-byte aligned for NR >= 2).
template <int NR>
__device__ __forceinline__ void lds_rhs(uint32_t a, float2 (&v)[NR]) {
  if constexpr (NR == 1) {
    v[0] = lds2(a);
  } else {
#pragma unroll
    for (int r = 0; r < NR; r += 2) {
      const float4 w = lds4(a + 8 * r);
      v[r] = make_float2(w.x, w.y);
      v[r + 1] = make_float2(w.z, w.w);
    }
  }
}

// What the gather warp of a group leaves beside its input values.
struct GroupMeta {
  Item it[2];            // items in execution order
  int nch[2];            // their chunks
  SegMap out;            // where the group's output segments go
  int p0, npts;          // leaf stages: tree-order points [p0, p0 + npts) of the group's leaves
  int lb[10];            // start of leaf t relative to p0 (t = 0 .. c)
  int nat[kMaxGroupPoints];   // natural index of each point
};

// Main block, forward: y[e] += sum_l T[l][e] x[l].  A lane owns four consecutive entries
// (one 16-byte load per plane; c R is a multiple of 4, so rows stay aligned) of every
// LPW-th line: with G = entries / 4 lanes to a line, LPW = 32 / G lines go side by side.
// re, im: the lane's entries of its first line; n: the lane's lines (row bytes times LPW
// apart), x its first input.
template <int NR, int B>
__device__ __forceinline__ void lines_vec4(uint32_t re, uint32_t im, uint32_t step, uint32_t x, uint32_t xstep, int n,
                                           float2 (&acc)[4][NR]) {
  float4 ar[B], ai[B];
  float2 xv[B][NR];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    ar[b] = ai[b] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < NR; ++r) xv[b][r] = make_float2(0.f, 0.f);
    if (b < n) {
      ar[b] = lds4(re + b * step);
      ai[b] = lds4(im + b * step);
      lds_rhs<NR>(x + b * xstep, xv[b]);
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const float tr[4] = {ar[b].x, ar[b].y, ar[b].z, ar[b].w}, ti[4] = {ai[b].x, ai[b].y, ai[b].z, ai[b].w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc[i][r].x = fmaf(tr[i], xv[b][r].x, fmaf(-ti[i], xv[b][r].y, acc[i][r].x));
        acc[i][r].y = fmaf(tr[i], xv[b][r].y, fmaf(ti[i], xv[b][r].x, acc[i][r].y));
      }
  }
}

// acc[j] += sum_l T[l][e + 32 j] x[l] over nl lines, lanes on consecutive entries (j < JE;
// the last exists for the lane only if tail_on): main blocks of 4 and 8 RHS, where every
// lane multiplies whatever the row length, (V^L)^* points and U^L columns.  The lane's
// inputs of line l are at x + l NR complex values.
template <int NR, int JE, int B>
__device__ __forceinline__ void lines_axpy(uint32_t re, uint32_t im, uint32_t row, bool tail_on, uint32_t x,
                                           float2 (&acc)[4][NR]) {
  float2 xv[B][NR];
  float ar[B][JE], ai[B][JE];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    lds_rhs<NR>(x + b * NR * 8, xv[b]);
#pragma unroll
    for (int j = 0; j < JE; ++j) {
      ar[b][j] = ai[b][j] = 0.f;
      if (j < JE - 1 || tail_on) {
        ar[b][j] = lds(re + b * row + 128 * j);
        ai[b][j] = lds(im + b * row + 128 * j);
      }
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b)
#pragma unroll
    for (int j = 0; j < JE; ++j)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        acc[j][r].x = fmaf(ar[b][j], xv[b][r].x, fmaf(-ai[b][j], xv[b][r].y, acc[j][r].x));
        acc[j][r].y = fmaf(ar[b][j], xv[b][r].y, fmaf(ai[b][j], xv[b][r].x, acc[j][r].y));
      }
}
template <int NR, int JE>
__device__ __forceinline__ void chunk_axpy(uint32_t re, uint32_t im, int nl, uint32_t row, bool tail_on, uint32_t x,
                                           float2 (&acc)[4][NR]) {
  constexpr int B = NR == 8 ? (JE > 2 ? 1 : 2) : NR == 4 ? 2 : 4;
  int l = 0;
  for (; l + B <= nl; l += B) {
    lines_axpy<NR, JE, B>(re, im, row, tail_on, x, acc);
    re += B * row;
    im += B * row;
    x += B * NR * 8;
  }
  for (; l < nl; ++l) {
    lines_axpy<NR, JE, 1>(re, im, row, tail_on, x, acc);
    re += row;
    im += row;
    x += NR * 8;
  }
}

// Sums over groups of W lanes (32 or 16) of V = 16 values per lane: afterwards lane L of a
// group holds the total of value L 16 / W (halving steps: 15 exchanges, then one per
// remaining lane bit, instead of 16 per bit).
template <int W>
__device__ __forceinline__ float transpose_reduce16(float (&v)[16], int lane) {
  int s = W / 2;
#pragma unroll
  for (int n = 8; n > 0; n >>= 1, s >>= 1) {
    const bool up = lane & s;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  if (W == 32) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  return v[0];
}

// The lane's four consecutive inputs (zero for a lane beyond the entries).
template <int NR>
__device__ __forceinline__ void load_x4(uint32_t x, bool on, float2 (&xr)[4][NR]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int r = 0; r < NR; ++r) xr[i][r] = make_float2(0.f, 0.f);
    if (on) lds_rhs<NR>(x + i * NR * 8, xr[i]);
  }
}

// Adjoint main block: out[line] = sum_e conj(T[line][e]) x[e] for nb lines, a group of W
// lanes to a line (W = 32, or 16 for lines of at most 64 entries: two sets of lines side by
// side), each lane on four consecutive entries.  BL = 8 / NR lines a group.  re, im: the
// lane's entries of its group's first line; len > 128: two halves, inputs read again.
template <int NR, int W>
__device__ __forceinline__ void adj_batch(uint32_t re, uint32_t im, uint32_t row, int nb, int len, int lane, bool on,
                                          float2 (&xr)[4][NR], uint32_t x, float* __restrict__ out) {
  constexpr int BL = 8 / NR;
  float v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = 0.f;
  for (int h0 = 0; h0 < len; h0 += 128) {
    const bool onh = len <= 128 ? on : h0 + 4 * lane < len;
    if (len > 128) load_x4<NR>(x + (h0 + 4 * lane) * NR * 8, onh, xr);
#pragma unroll
    for (int i = 0; i < BL; ++i) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (onh && i < nb) {
        a = lds4(re + i * row + h0 * 4);
        b = lds4(im + i * row + h0 * 4);
      }
      const float ar[4] = {a.x, a.y, a.z, a.w}, ai[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int r = 0; r < NR; ++r) {                 // (the four products added pairwise)
        float tx[4], ty[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          tx[q] = fmaf(ar[q], xr[q][r].x, ai[q] * xr[q][r].y);
          ty[q] = fmaf(ar[q], xr[q][r].y, -ai[q] * xr[q][r].x);
        }
        v[(i * NR + r) * 2] += (tx[0] + tx[1]) + (tx[2] + tx[3]);
        v[(i * NR + r) * 2 + 1] += (ty[0] + ty[1]) + (ty[2] + ty[3]);
      }
    }
  }
  const float t = transpose_reduce16<W>(v, lane);
  constexpr int kRep = W / 16;                       // lanes holding the same total
  const int idx = (lane & (W - 1)) / kRep, i = idx / (2 * NR);
  if ((lane & (kRep - 1)) == 0 && i < nb) out[idx] = t;
}

// sum_k conj(T[k]) x[k] over n entries from entry k0 on, cyclically (so that threads on
// different lines read different banks), in four interleaved sums; x: `xs` bytes apart.
__device__ __forceinline__ float2 conj_dot(uint32_t re, uint32_t im, uint32_t x, uint32_t xs, int n, int k0) {
  float2 s[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) s[u] = make_float2(0.f, 0.f);
  int k = k0;
  for (int i = 0; i < n; i += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u < n) {
        const float ar = lds(re + 4 * k), ai = lds(im + 4 * k);
        const float2 v = lds2(x + k * xs);
        s[u].x = fmaf(ar, v.x, fmaf(ai, v.y, s[u].x));
        s[u].y = fmaf(ar, v.y, fmaf(-ai, v.x, s[u].y));
        if (++k == n) k = 0;
      }
  }
  return make_float2((s[0].x + s[1].x) + (s[2].x + s[3].x), (s[0].y + s[1].y) + (s[2].y + s[3].y));
}

// Blocks of more than 128 entries are split in two parts among the warps (and the lines
// into half as many shares): a lane owns four entries at most.
__host__ __device__ constexpr int entry_parts(int len) { return len > 128 ? 2 : 1; }

// ---------------------------------------------------------------- kernel

// W consumer warps, GA gather warps (and input buffers), CPS CTAs to an SM.
template <int NRB, bool ADJ, int W, int GA, int CPS>
__global__ void __launch_bounds__((W + GA + 2) * 32, CPS) bf_apply_simt(const __grid_constant__ ApplyArgs a) {
  static_assert(W == 4 || W == 8, "consumer warps");
  static_assert(GA % 2 == 0, "the partial sums start 16-byte aligned for any xcap");
  constexpr int LW = W == 8 ? 3 : 2;
  constexpr int NR = NRB;
  const uint64_t dep_lim = a.wait_ns ? a.wait_ns : kTimeoutNs;
  const uint64_t lim = 2 * dep_lim;                  // waits inside the CTA outlast its dependency waits
  extern __shared__ __align__(1024) uint8_t smem[];
  const int D = a.n_slots;
  uint8_t* ring = smem;
  float2* xbuf = reinterpret_cast<float2*>(smem + size_t(D) * kSlotBytes);
  float2* red = xbuf + size_t(GA) * a.xcap * NRB;      // partial sums (forward), line results (adjoint)
  float2* ybuf = red + size_t(a.redcap) * NRB;               // main output before U^L; U^* output before the block
  GroupMeta* meta = reinterpret_cast<GroupMeta*>(ybuf + size_t(a.xcap) * NRB);
  uint64_t* full = reinterpret_cast<uint64_t*>(meta + GA);
  uint64_t* empty = full + kMaxSlots;
  uint64_t* xfull = empty + kMaxSlots;
  uint64_t* xempty = xfull + GA;
  volatile unsigned* done = reinterpret_cast<volatile unsigned*>(xempty + GA);   // groups stored by this CTA
  volatile int* abort = reinterpret_cast<volatile int*>(done + 1);
  uint32_t* latest = reinterpret_cast<uint32_t*>(const_cast<int*>(abort + 1));   // 1 + phase of each slot's latest copy

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < D; ++s) {
      latest[s] = 0;
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], W);
    }
    for (int s = 0; s < GA; ++s) {
      mbar_init(&xfull[s], 1);
      mbar_init(&xempty[s], 1);
    }
    *done = 0;
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  const Plan& plan = a.plan;
  const int S = plan.n_stages, c = plan.c;
  // This CTA's groups of stage e are first_group(e), + grid, ...: the CTAs that get one
  // group more than the others change from stage to stage.
  const int grid = int(gridDim.x);
  const auto first_group = [&](int e) { return int((blockIdx.x + unsigned(e) * unsigned(a.rot)) % unsigned(grid)); };
  const auto stage_of = [&](int e) -> const Stage& { return plan.st[ADJ ? S - 1 - e : e]; };
  const unsigned n_cnt = unsigned(S) * unsigned(plan.st[0].n_groups);   // (every stage has as many groups)

  if (warp == W + GA) {
    // ------------------------------------------------------------------ producer
    // The lanes take an item's chunks side by side, up to one ring of them at a time: each
    // tests its own slot and issues its copy as soon as that is free.  (A thread that waits
    // for slot after slot issues a copy every few hundred ns only, and lanes that wait
    // apart suspend one another.)
    uint32_t slot0 = 0, ph0 = 1;                     // slot and free-phase parity of the next chunk
    int e = 0, g = first_group(0), mi = 0;
    const auto fix = [&]() {                         // first existing item at or after (e, g, mi)
      while (e < S) {
        const Stage& st = stage_of(e);
        if (g < st.n_groups && mi < st.n_items) return true;
        mi = 0;
        if (g < st.n_groups) g += grid;
        else if (++e < S) g = first_group(e);
      }
      return false;
    };
    const auto load = [&]() {
      const Stage& st = stage_of(e);
      return a.items[st.item_base + int64_t(g) * st.n_items + (ADJ ? st.n_items - 1 - mi : mi)];
    };
    bool ok = true, have = fix();
    Item nx{};
    if (have) nx = load();
    while (have && ok) {
      const Item it = nx;                            // the following descriptor is in flight meanwhile
      ++mi;
      have = fix();
      if (have) nx = load();
      if (!item_ok(it)) {
        if (lane == 0) set_status(a.status, abort, ST_BAD_ITEM);
        break;
      }
      const int nch = (int(it.nlines) + it.lpc - 1) / it.lpc;
      const uint8_t* src = a.arena + uint64_t(it.off128) * 128u;
      const uint32_t cb = uint32_t(chunk_bytes(it.lpc, it.len));
      const int tail = int(it.nlines) - (nch - 1) * int(it.lpc);
      const uint32_t tb = uint32_t(chunk_bytes(tail, it.len));
      const int width = min(D, 32);                  // (D <= kMaxSlots)
      for (int c0 = 0; c0 < nch && ok; c0 += width) {
        const int n = min(width, nch - c0);
        uint32_t slot = slot0 + uint32_t(lane), ph = ph0;
        if (slot >= uint32_t(D)) {
          slot -= uint32_t(D);
          ph ^= 1u;
        }
        const int ci = c0 + lane;
        bool pend = lane < n;
        uint64_t t0 = 0;
        for (unsigned tries = 1;; ++tries) {
          if (pend && mbar_test(&empty[slot], ph)) {
            const uint32_t bytes = ci == nch - 1 ? tb : cb;
            mbar_expect_tx(&full[slot], bytes);
            bulk_g2s(ring + size_t(slot) * kSlotBytes, src + uint64_t(ci) * cb, bytes, &full[slot]);
            latest[slot] = (ph ^ 1u) + 1u;
            pend = false;
          }
          if (!__any_sync(0xffffffffu, pend)) break;
          __nanosleep(40);                           // (leaves the shared-memory pipe to the products)
          if ((tries & 63u) == 0) {
            bool stop = *abort != 0;
            const uint64_t t = gtimer();
            if (t0 == 0) t0 = t;
            if (t - t0 > lim) {
              if (lane == 0) set_status(a.status, abort, ST_EMPTY_TIMEOUT);
              stop = true;
            }
            if (__any_sync(0xffffffffu, stop)) {
              ok = false;
              break;
            }
          }
        }
        slot0 += uint32_t(n);
        if (slot0 >= uint32_t(D)) {
          slot0 -= uint32_t(D);
          ph0 ^= 1u;
        }
      }
    }
    // wait (bounded) for each slot's latest copy, so that none writes shared memory after
    // the CTA exits
    __syncwarp();
    if (lane < D && latest[lane]) {
      const uint64_t t1 = gtimer();
      while (!mbar_try(&full[lane], latest[lane] - 1) && gtimer() - t1 < kTimeoutNs) {
      }
    }
  } else if (warp == W + GA + 1) {
    // ------------------------------------------------------------------ signal
    // As soon as groups are stored, make their outputs visible GPU-wide and add one per
    // segment to the counters of the groups that read them; one fence covers every group
    // stored by then.
    unsigned j = 0, avail = 0;
    bool ok = true;
    unsigned* counters = counter_set(a.counters, a.ctl, n_cnt);
    for (int e = 0; e + 1 < S && ok; ++e) {
      const Stage& st = stage_of(e);
      const Stage& nst = stage_of(e + 1);
      const int out_pat = ADJ ? st.in_pat : st.out_pat, next_in = ADJ ? nst.out_pat : nst.in_pat;
      unsigned* cnt_out = counters + int64_t(e + 1) * nst.n_groups;
      for (int g = first_group(e); g < st.n_groups; g += grid, ++j) {
        if (j >= avail) {
          uint64_t t0 = 0;
          for (unsigned n = 1; (avail = ld_acquire_cta(done)) <= j; ++n) {
            __nanosleep(40);                         // (leaves the shared-memory pipe to the products)
            if ((n & 63u) == 0) {
              const uint64_t t = gtimer();
              if (t0 == 0) t0 = t;
              if (*abort) { ok = false; break; }
              if (t - t0 > lim) { set_status(a.status, abort, ST_FULL_TIMEOUT); ok = false; break; }
            }
          }
          if (__any_sync(0xffffffffu, !ok)) {
            ok = false;
            break;
          }
          avail = __reduce_min_sync(0xffffffffu, avail);   // what every lane has seen
          __threadfence();
        }
        if (lane < c) {
          const SegMap sm = seg_map(out_pat, g, st, 1, c);
          atomicAdd(cnt_out + pat_group(next_in, sm.base + lane * sm.step, nst, c), 1u);
        }
      }
    }
  } else if (warp >= W) {
    // ------------------------------------------------------------------ gather
    const int gw = warp - W;                // takes groups j = gw mod GA, buffer gw
    float2* xin = xbuf + size_t(gw) * a.xcap * NRB;
    GroupMeta& m = meta[gw];
    unsigned j = 0;
    bool ok = true;
    const unsigned* counters = counter_set(a.counters, a.ctl, n_cnt);
    for (int e = 0; e < S && ok; ++e) {
      const Stage& st = stage_of(e);
      const int in_pat = ADJ ? st.out_pat : st.in_pat, out_pat = ADJ ? st.in_pat : st.out_pat;
      const int Rin = ADJ ? st.R_out : st.R_in;      // execution-sense segment length
      const bool leaf_w = st.in_pat == PAT_LEAF, leaf_x = st.out_pat == PAT_LEAF;
      const int32_t* lperm = leaf_w ? a.w_perm : a.x_perm;
      const int32_t* loff = leaf_w ? a.w_off : a.x_off;
      const float2* src = a.bufs + (e > 0 ? e - 1 : 0) * a.buf_stride;
      const unsigned* cnt_in = counters + int64_t(e) * st.n_groups;
      for (int g = first_group(e); g < st.n_groups && ok; g += grid, ++j) {
        if (int(j % GA) != gw) continue;
        Item myit{};                                 // (in flight while the buffer is waited for)
        if (lane < st.n_items)
          myit = a.items[st.item_base + int64_t(g) * st.n_items + (ADJ ? st.n_items - 1 - lane : lane)];
        if (!__all_sync(0xffffffffu, wait_bar(&xempty[gw], ((j / GA) & 1u) ^ 1u, a, abort, lim, ST_EMPTY_TIMEOUT))) {
          ok = false;
          break;
        }
        if (__any_sync(0xffffffffu, lane < st.n_items && !item_ok(myit))) {
          if (lane == 0) set_status(a.status, abort, ST_BAD_ITEM);
          ok = false;
          break;
        }
        if (lane < st.n_items) {
          m.it[lane] = myit;
          m.nch[lane] = (int(myit.nlines) + myit.lpc - 1) / myit.lpc;
        }
        if (lane == 0 && out_pat != PAT_LEAF) m.out = seg_map(out_pat, g, st, ADJ ? st.R_in : st.R_out, c);
        if (leaf_w || leaf_x) {
          int v = 0;
          if (lane <= c) v = loff[c * g + lane];
          const int p0 = __shfl_sync(0xffffffffu, v, 0);
          const int npts = min(__shfl_sync(0xffffffffu, v, c) - p0, kMaxGroupPoints);
          if (lane <= c) m.lb[lane] = v - p0;
          if (lane == 0) {
            m.p0 = p0;
            m.npts = npts;
          }
          for (int pb = 0; pb < npts; pb += 32 * 8) {
            int idx[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int pt = pb + lane + 32 * u;
              idx[u] = pt < npts ? lperm[p0 + pt] : 0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int pt = pb + lane + 32 * u;
              if (pt < npts) m.nat[pt] = idx[u];
            }
            if (in_pat == PAT_LEAF) {                // the points' values: 8 loads in flight per RHS
#pragma unroll
              for (int r = 0; r < NRB; ++r) {
                const bool on = a.rhs0 + r < a.nrhs;
                const float2* row = on ? in_row(a, a.rhs0 + r) : nullptr;
                float2 v8[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int pt = pb + lane + 32 * u;
                  v8[u] = (on && pt < npts) ? __ldg(row + idx[u]) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int pt = pb + lane + 32 * u;
                  if (pt < npts) xin[pt * NRB + r] = v8[u];
                }
              }
            }
          }
        }
        if (in_pat != PAT_LEAF) {
          // the segments come from the previous stage's vector (L2), packed one after the other;
          // a compact stage's block holds only the first r_t lines of segment t (c = 4), so
          // only those are read.  Everything but the loads is worked out before the wait.
          const SegMap sm = seg_map(in_pat, g, st, Rin, c);
          int p1 = Rin, p2 = 2 * Rin, p3 = 3 * Rin, nlin = c * Rin;
          if (st.compact && !ADJ) {
            const int32_t rk = __shfl_sync(0xffffffffu, myit.base, st.main_idx);
            p1 = seg_lines(rk, 0);
            p2 = p1 + seg_lines(rk, 1);
            p3 = p2 + seg_lines(rk, 2);
            nlin = p3 + seg_lines(rk, 3);
          }
          const auto place = [&](int line) -> int {
            int t, kk;
            if (c == 4) {
              t = (line >= p1 ? 1 : 0) + (line >= p2 ? 1 : 0) + (line >= p3 ? 1 : 0);
              kk = line - (t == 0 ? 0 : t == 1 ? p1 : t == 2 ? p2 : p3);
            } else {
              t = seg_of(line, Rin, c);
              kk = line - t * Rin;
            }
            return sm.base + t * sm.step + kk;
          };
          // entries are moved as 16-byte pairs of RHS (one RHS: 8 bytes each)
          using V = std::conditional_t<NRB == 1, float2, float4>;
          constexpr int H = NRB == 1 ? 1 : NRB / 2, U = 8;
          const int nq = nlin * H;
          const V* sv = reinterpret_cast<const V*>(src);
          V* dv = reinterpret_cast<V*>(xin);
          const V* from[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            // (one RHS forward: not for batches that a small block does not fill; elsewhere the test
            // costs more than it saves, 8 RHS n = 128: 144 us without it, 156 with)
            if (ADJ || NRB > 1 || u == 0 || 32 * u < nq)
              from[u] = sv + int64_t(place(min(lane + 32 * u, max(nq, 1) - 1) / H)) * H + lane % H;
          // wait until the group's c input segments have been counted in
          bool got = true;
          const unsigned* cp = cnt_in + g;
          const unsigned need = unsigned(c) + (e + 1 == a.stall_stage1 && g == 0 ? 1u : 0u);
          uint64_t t0 = 0;
          for (unsigned n = 1; ld_acquire(cp) < need; ++n) {
            if ((n & 15u) == 0) {
              const uint64_t t = gtimer();
              if (t0 == 0) t0 = t;
              if (*abort || *reinterpret_cast<volatile int*>(a.status) != 0) {
                *abort = 1;
                got = false;
                break;
              }
              if (t - t0 > dep_lim) {
                set_status(a.status, abort, ST_DEP_TIMEOUT);
                got = false;
                break;
              }
            }
          }
          if (__any_sync(0xffffffffu, !got)) {
            ok = false;
            break;
          }
          {
            V v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (lane + 32 * u < nq) v[u] = __ldcg(from[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (lane + 32 * u < nq) dv[lane + 32 * u] = v[u];
          }
          for (int qb = 32 * U; qb < nq; qb += 32 * U) {
            V v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int q = qb + lane + 32 * u;
              if (q < nq) v[u] = __ldcg(sv + int64_t(place(q / H)) * H + q % H);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int q = qb + lane + 32 * u;
              if (q < nq) dv[q] = v[u];
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&xfull[gw]);
      }
    }
  } else {
    // ------------------------------------------------------------------ consumers
    constexpr bool kVec = NRB <= 2;                  // lane mapping of the main blocks (forward)
    const int tid = threadIdx.x;
    clear_other_set(a.counters, a.ctl, n_cnt, unsigned(tid), W * 32);
    const uint32_t ring_a = smem_addr(ring);
    uint32_t rslot = 0, rph = 0;                     // ring slot and phase of the next item's first chunk
    unsigned j = 0;
    bool dead = false;                               // a wait gave up: no more work, only the barriers
    for (int e = 0; e < S; ++e) {
      const Stage& st = stage_of(e);
      const int in_pat = ADJ ? st.out_pat : st.in_pat, out_pat = ADJ ? st.in_pat : st.out_pat;
      const int Rout = ADJ ? st.R_in : st.R_out;
      const bool last = e + 1 == S;
      float2* dst = a.bufs + int64_t(e) * a.buf_stride;
      // forward main block (all of the stage's have the same entries): this warp's part of
      // the entries and share of the lines; kVec: the lane's four entries and which of the
      // side-by-side lines, else its first entry
      const int tot = c * Rout, es = entry_parts(tot), lks = es == 1 ? LW : LW - 1;
      const int ks = warp & ((1 << lks) - 1), eh = warp >> lks;
      const int part = 4 * ((tot + 4 * es - 1) / (4 * es)), G = part / 4, LPW = 32 / G;
      const int s_line = lane / G, q4 = lane - s_line * G;
      const bool lane_on = s_line < LPW && eh * part + 4 * q4 < tot;
      const int ea = eh * part, je = (min(part, tot - ea) + 31) >> 5;
      const bool tail_main = ea + 32 * (je - 1) + lane < min(tot, ea + part);
      const int Gt = G * es;                           // float4 columns of a share's partial sums (kVec)
      const uint32_t inv_gt = (65535u + uint32_t(Gt)) / uint32_t(Gt);
      for (int g = first_group(e); g < st.n_groups; g += grid, ++j) {
        // The number of barriers below depends only on the stage, so the warps stay
        // together when a wait gives up (it skips the work, not the barriers).
        const int xb = int(j % GA);
        const float2* xin = xbuf + size_t(xb) * a.xcap * NRB;
        const uint32_t xin_a = smem_addr(xin);
        const GroupMeta& m = meta[xb];
        bool ok = !dead && wait_bar(&xfull[xb], (j / GA) & 1u, a, abort, lim, ST_FULL_TIMEOUT);
        ok = __all_sync(0xffffffffu, ok);
        // Wait for chunk ci of the current item: address of its first entry (0: gave up).
        const auto chunk_at = [&](int ci, uint32_t& slot) -> uint32_t {
          uint32_t ph = rph;
          slot = rslot + uint32_t(ci);
          while (slot >= uint32_t(D)) {
            slot -= uint32_t(D);
            ph ^= 1u;
          }
          ok = ok && wait_bar(&full[slot], ph, a, abort, lim, ST_FULL_TIMEOUT);
          ok = __all_sync(0xffffffffu, ok);
          return ring_a + slot * uint32_t(kSlotBytes);
        };
        const auto advance = [&](int nch) {
          rslot += uint32_t(nch);
          while (rslot >= uint32_t(D)) {
            rslot -= uint32_t(D);
            rph ^= 1u;
          }
        };
        // Every chunk of an item, for all warps: body(re, im, first line, lines).
        const auto each_chunk = [&](int mi, auto&& body) {
          if (!ok) return;
          const Item it = m.it[mi];
          const int nch = m.nch[mi], lpc = it.lpc;
          for (int ci = 0; ci < nch && ok; ++ci) {
            uint32_t slot;
            const uint32_t re = chunk_at(ci, slot);
            if (!ok) break;
            const int nl = min(lpc, int(it.nlines) - ci * lpc);
            body(re, re + 4u * uint32_t(pad4(int64_t(nl) * it.len)), ci * lpc, nl);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot]);
          }
          advance(nch);
        };
        // The chunks of an item dealt to 2^ls shares by their number in the CTA's stream: a
        // share's chunks use slots of one residue (the ring is a multiple of W slots), so a
        // warp never waits for a slot whose previous chunk it has not itself consumed, or seen
        // consumed at a barrier: a barrier's one-bit phase allows no more.  W arrivals a chunk.
        const auto my_chunks = [&](int mi, int k, int ls, auto&& body) {
          if (!ok) return;
          const Item it = m.it[mi];
          const int nch = m.nch[mi], lpc = it.lpc, len = it.len, n = 1 << ls;
          const uint32_t weight = uint32_t(n);
          for (int ci = int((uint32_t(k) - rslot) & uint32_t(n - 1)); ci < nch; ci += n) {
            uint32_t slot;
            const uint32_t re = chunk_at(ci, slot);
            if (!ok) break;
            const int nl = min(lpc, int(it.nlines) - ci * lpc);
            body(re, re + uint32_t(nl * len) * 4u, ci * lpc, nl);   // (planes of len % 4 == 0: no padding)
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot], weight);
          }
          advance(nch);
        };
        const auto emit_point = [&](int pt, int r, float2 v) {
          if (a.rhs0 + r < a.nrhs) {
            float2* o = out_row(a, a.rhs0 + r) + m.nat[pt];
            if (a.accumulate) {
              const float2 w = *o;
              v.x += w.x;
              v.y += w.y;
            }
            *o = v;
          }
        };
        // 32 entries of one RHS a warp at a time: body(entry, RHS) over n entries.
        const auto by_rhs = [&](int n, auto&& body) {
          for (int w = warp; w < NRB * ((n + 31) >> 5); w += W) {
            const int q = (w / NRB) * 32 + lane;
            if (q < n) body(q, w % NRB);
          }
        };
        if constexpr (!ADJ) {
          float2 acc[4][NR];
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < NR; ++r) acc[q][r] = make_float2(0.f, 0.f);
          if (in_pat == PAT_LEAF) {
            // (V^L)^*: lines are the group's points.  A warp takes one leaf t (two of 8 with four
            // warps), and one of KL shares of its points; partial sums red[share][RHS][t R + k].
            const int lc = c == 4 ? 2 : 3, NL = c > W ? c / W : 1, KL = c > W ? 1 : W >> lc;
            const int t0 = warp & (c - 1), kl = c > W ? 0 : warp >> lc;
            const int jl = (Rout + 31) >> 5;         // (1 for 8 leaves)
            const bool tail_on = lane + 32 * (jl - 1) < Rout;
            const uint32_t row = uint32_t(Rout) * 4u;
            int pa[2] = {0, 0}, pe[2] = {0, 0};
            if (ok)
#pragma unroll
              for (int i = 0; i < 2; ++i)
                if (i < NL) {
                  const int b0 = m.lb[t0 + i * W], n = m.lb[t0 + i * W + 1] - b0;
                  pa[i] = b0 + n * kl / KL;
                  pe[i] = b0 + n * (kl + 1) / KL;
                }
            float2 acc2[4][NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) acc2[0][r] = make_float2(0.f, 0.f);
            each_chunk(0, [&](uint32_t re, uint32_t im, int l0, int nl) {
              const int s0 = max(pa[0], l0), s1 = min(pe[0], l0 + nl);
              if (s0 < s1) {
                const uint32_t o = uint32_t(s0 - l0) * row + uint32_t(lane) * 4u;
                const uint32_t x = xin_a + uint32_t(s0 * NRB) * 8u;
                if (jl == 1) chunk_axpy<NR, 1>(re + o, im + o, s1 - s0, row, tail_on, x, acc);
                else chunk_axpy<NR, 2>(re + o, im + o, s1 - s0, row, tail_on, x, acc);
              }
              if (W == 4 && NL == 2) {
                const int u0 = max(pa[1], l0), u1 = min(pe[1], l0 + nl);
                const uint32_t o = uint32_t(u0 - l0) * row + uint32_t(lane) * 4u;
                if (u0 < u1)
                  chunk_axpy<NR, 1>(re + o, im + o, u1 - u0, row, tail_on, xin_a + uint32_t(u0 * NRB) * 8u, acc2);
              }
            });
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (q < jl && lane + 32 * q < Rout)
#pragma unroll
                for (int r = 0; r < NR; ++r) red[(kl * NRB + r) * tot + t0 * Rout + lane + 32 * q] = acc[q][r];
            if (W == 4 && NL == 2 && lane < Rout)
#pragma unroll
              for (int r = 0; r < NR; ++r) red[r * tot + (t0 + W) * Rout + lane] = acc2[0][r];
            cons_sync<W>();
            if (ok)
              by_rhs(tot, [&](int q, int r) {
                float2 v = red[r * tot + q];
                for (int k = 1; k < KL; ++k) {
                  const float2 w = red[(k * NRB + r) * tot + q];
                  v.x += w.x;
                  v.y += w.y;
                }
                dst[int64_t(m.out.base + q) * NRB + r] = v;
              });
          } else {
            my_chunks(0, ks, lks, [&](uint32_t re, uint32_t im, int l0, int nl) {
              const uint32_t row = uint32_t(tot) * 4u;
              if constexpr (kVec) {
                constexpr int B = NR == 1 ? 4 : 2;
                const uint32_t o = uint32_t(ea + 4 * q4) * 4u + uint32_t(s_line) * row;
                const uint32_t x = xin_a + uint32_t((l0 + s_line) * NRB) * 8u;
                for (int l = 0; l < nl; l += B * LPW) {
                  int left = 0;                      // the lane's lines of this step
#pragma unroll
                  for (int b = 0; b < B; ++b) left += lane_on && l + b * LPW + s_line < nl ? 1 : 0;
                  lines_vec4<NR, B>(re + o + uint32_t(l) * row, im + o + uint32_t(l) * row, uint32_t(LPW) * row,
                                    x + uint32_t(l * NRB) * 8u, uint32_t(LPW * NRB) * 8u, left, acc);
                }
              } else {
                const uint32_t o = uint32_t(ea + lane) * 4u, x = xin_a + uint32_t(l0 * NRB) * 8u;
                if (je == 1) chunk_axpy<NR, 1>(re + o, im + o, nl, row, tail_main, x, acc);
                else if (je == 2) chunk_axpy<NR, 2>(re + o, im + o, nl, row, tail_main, x, acc);
                else if (je == 3) chunk_axpy<NR, 3>(re + o, im + o, nl, row, tail_main, x, acc);
                else if (je == 4) chunk_axpy<NR, 4>(re + o, im + o, nl, row, tail_main, x, acc);
              }
            });
            if constexpr (kVec) {
              // add the side-by-side lines in pairs, then pairs of pairs ... (up to 32 lines of rows of
              // four entries), then the warp's sums go to its share of `red`: float4 units
              // [share][pair of values][column], a column a lane
              for (int t = 1; t < LPW; t *= 2) {
                const bool add = (s_line & (2 * t - 1)) == 0 && s_line + t < LPW;
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                  for (int r = 0; r < NR; ++r) {
                    const float px = __shfl_sync(0xffffffffu, acc[i][r].x, (lane + t * G) & 31);
                    const float py = __shfl_sync(0xffffffffu, acc[i][r].y, (lane + t * G) & 31);
                    if (add) {
                      acc[i][r].x += px;
                      acc[i][r].y += py;
                    }
                  }
              }
              float4* red4 = reinterpret_cast<float4*>(red);
              if (s_line == 0 && lane_on)
#pragma unroll
                for (int p = 0; p < 2 * NR; ++p) {
                  const float2 u = NR == 1 ? acc[(2 * p) & 3][0] : acc[p & 3][0];
                  const float2 w = NR == 1 ? acc[(2 * p + 1) & 3][0] : acc[p & 3][NR - 1];
                  red4[(ks * 2 * NR + p) * Gt + eh * G + q4] = make_float4(u.x, u.y, w.x, w.y);
                }
              cons_sync<W>();
              // sum the shares (always in the same order); a unit is two values: entries 2p and
              // 2p + 1 of the column (one RHS) or the two RHS of its entry p
              if (ok) {
                const int units = 2 * NR * Gt, KS = 1 << lks;
                for (int u = tid; u < units; u += (W * 32)) {
                  float4 v = red4[u];
#pragma unroll
                  for (int k = 1; k < W; ++k)
                    if (k < KS) {
                      const float4 w = red4[k * units + u];
                      v.x += w.x;
                      v.y += w.y;
                      v.z += w.z;
                      v.w += w.w;
                    }
                  const int p = int((uint32_t(u) * inv_gt) >> 16), qg = u - p * Gt;
                  const int ee = 4 * qg + (NR == 1 ? 2 * p : p);
                  if (ee >= tot) continue;
                  if (out_pat == PAT_LEAF) {
                    *reinterpret_cast<float4*>(ybuf + ee * NRB) = v;
                  } else if constexpr (NR == 1) {
                    const int t0 = seg_of(ee, Rout, c), t1 = seg_of(ee + 1, Rout, c);
                    dst[m.out.base + t0 * m.out.step + ee - t0 * Rout] = make_float2(v.x, v.y);
                    dst[m.out.base + t1 * m.out.step + ee + 1 - t1 * Rout] = make_float2(v.z, v.w);
                  } else {
                    const int t = seg_of(ee, Rout, c);
                    *reinterpret_cast<float4*>(dst + int64_t(m.out.base + t * m.out.step + ee - t * Rout) * NRB) = v;
                  }
                }
              }
            } else {
              // the warp's sums go to its share of `red`, [share][entry][RHS] in float4 units (two
              // RHS), unit u of entry e at u ^ swz(e): a quarter warp's writes (8 entries, one
              // unit) and its reads (consecutive units) both touch every bank once
              constexpr int U = NR / 2 > 0 ? NR / 2 : 1;
              const auto swz = [](int ee) { return NR == 8 ? (ee >> 1) & 3 : (ee >> 2) & 1; };
              float4* red4 = reinterpret_cast<float4*>(red);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int ee = ea + lane + 32 * q;
                if (q < je && ee < min(tot, ea + part))
#pragma unroll
                  for (int u = 0; u < U; ++u)
                    red4[(ks * tot + ee) * U + (u ^ swz(ee))] =
                        make_float4(acc[q][(2 * u) % NR].x, acc[q][(2 * u) % NR].y, acc[q][(2 * u + 1) % NR].x,
                                    acc[q][(2 * u + 1) % NR].y);
              }
              cons_sync<W>();
              if (ok)
                for (int q = tid; q < tot * U; q += W * 32) {
                  const int ee = q / U, u = q % U, at = ee * U + (u ^ swz(ee));
                  float4 v = red4[at];
#pragma unroll
                  for (int k = 1; k < W; ++k)
                    if (k < 1 << lks) {
                      const float4 w = red4[k * tot * U + at];
                      v.x += w.x;
                      v.y += w.y;
                      v.z += w.z;
                      v.w += w.w;
                    }
                  if (out_pat == PAT_LEAF) {
                    *reinterpret_cast<float4*>(ybuf + ee * NRB + 2 * u) = v;
                  } else {
                    const int t = seg_of(ee, Rout, c);
                    *reinterpret_cast<float4*>(dst + int64_t(m.out.base + t * m.out.step + ee - t * Rout) * NRB + 2 * u) = v;
                  }
                }
            }
            if (out_pat == PAT_LEAF) {
              // U^L of the block's outputs (ybuf): lines are the columns, entries the group's points,
              // each taking its own leaf's coefficient.  A warp takes 32 points and one of KU
              // shares of the columns; partial sums red[share][RHS][point].
              cons_sync<W>();
              const int npts = ok ? m.npts : 0;
              const int lnb = npts > 128 ? 3 : npts > 64 ? 2 : npts > 32 ? 1 : 0;   // blocks of 32 points
              const int lku = max(0, LW - lnb), NB = max(1, (1 << lnb) >> LW);      // shares; blocks a warp
              const int pb = lnb < LW ? warp & ((1 << lnb) - 1) : warp, ku = lnb < LW ? warp >> lnb : 0;
              const int ka = (Rout * ku) >> lku, kb = (Rout * (ku + 1)) >> lku;
              float2 sum[2][4][NR];
              uint32_t y[2];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int pt = (pb + i * W) * 32 + lane;
                int t = 0;
                if (pt < npts)
                  for (int u = 1; u < c; ++u) t += pt >= m.lb[u] ? 1 : 0;
                y[i] = smem_addr(ybuf) + uint32_t(t * Rout * NRB) * 8u;
#pragma unroll
                for (int r = 0; r < NR; ++r) sum[i][0][r] = make_float2(0.f, 0.f);
              }
              each_chunk(1, [&](uint32_t re, uint32_t im, int l0, int nl) {
                const int s0 = max(ka, l0), s1 = min(kb, l0 + nl);
                const uint32_t row = uint32_t(npts) * 4u;
                if (s0 < s1)
#pragma unroll
                  for (int i = 0; i < (W == 4 ? 2 : 1); ++i)
                    if (i < NB) {
                      const int pt = (pb + i * W) * 32 + lane;
                      const uint32_t o = uint32_t(s0 - l0) * row + uint32_t(pt) * 4u;
                      chunk_axpy<NR, 1>(re + o, im + o, s1 - s0, row, pt < npts, y[i] + uint32_t(s0 * NRB) * 8u, sum[i]);
                    }
              });
#pragma unroll
              for (int i = 0; i < (W == 4 ? 2 : 1); ++i) {
                const int pt = (pb + i * W) * 32 + lane;
                if (i < NB && pt < npts)
#pragma unroll
                  for (int r = 0; r < NR; ++r) red[(ku * NRB + r) * npts + pt] = sum[i][0][r];
              }
              cons_sync<W>();
              if (ok)
                by_rhs(npts, [&](int q, int r) {
                  float2 v = red[r * npts + q];
                  for (int k = 1; k < 1 << lku; ++k) {
                    const float2 w = red[(k * NRB + r) * npts + q];
                    v.x += w.x;
                    v.y += w.y;
                  }
                  emit_point(q, r, v);
                });
            }
          }
        } else {
          const float2* x = xin;                     // inputs of the block (or of the V^L products)
          if (in_pat == PAT_LEAF) {
            // U^*: ybuf[t][k] = sum over leaf t's points of conj(U[k][point]) u[point]; one thread
            // per (leaf, column, RHS), each starting at another point of the leaf so that the
            // lanes' reads spread over the banks
            const int R = st.R_out;
            if (ok && m.it[0].nlines == 0)
              for (int q = tid; q < c * R * NRB; q += (W * 32)) ybuf[q] = make_float2(0.f, 0.f);
            each_chunk(0, [&](uint32_t re, uint32_t im, int l0, int nl) {
              const int len = m.npts;
              for (int q = tid; q < c * nl * NRB; q += (W * 32)) {
                const int r = q % NRB, l = (q / NRB) % nl, t = q / (NRB * nl);
                const int b0 = m.lb[t], nt = m.lb[t + 1] - b0;
                const uint32_t o = uint32_t(l * len + b0) * 4u;
                ybuf[(t * R + l0 + l) * NRB + r] =
                    conj_dot(re + o, im + o, xin_a + uint32_t(b0 * NRB + r) * 8u, NRB * 8, nt, nt > 0 ? l % nt : 0);
              }
            });
            cons_sync<W>();
            x = ybuf;
          }
          if (out_pat != PAT_LEAF) {
            // block: a warp takes its share of the lines; results per line in `red`
            const int mi = st.n_items - 1, len = c * st.R_out;
            const uint32_t xa = smem_addr(x), row = uint32_t(len) * 4u;
            constexpr int BL = 8 / NR;
            const bool two = len <= 64;              // two groups of 16 lanes, each with its own lines
            const int l4 = two ? lane & 15 : lane;
            const bool on = 4 * l4 < len;
            float2 xr[4][NR];
            load_x4<NR>(xa + uint32_t(4 * l4 * NRB) * 8u, ok && on && len <= 128, xr);
            my_chunks(mi, warp, LW, [&](uint32_t re, uint32_t im, int l0, int nl) {
              const int grp = two ? lane >> 4 : 0, stride = two ? 2 * BL : BL;
              for (int l = 0; l < nl; l += stride) {
                const int mine = l + grp * BL;       // this group's first line
                const uint32_t o = uint32_t(mine) * row + uint32_t(4 * l4) * 4u;
                const int nb = max(0, min(BL, nl - mine));
                float* out = reinterpret_cast<float*>(red + size_t(l0 + mine) * NRB);
                if (two) adj_batch<NR, 16>(re + o, im + o, row, nb, len, lane, on, xr, xa, out);
                else adj_batch<NR, 32>(re + o, im + o, row, nb, len, lane, on, xr, xa, out);
              }
            });
            cons_sync<W>();
            // scatter to the next vector; in a compact stage `red` holds the first r_t entries
            // of each segment t, and the entries beyond r_t are zero
            if (ok) {
              const int rk = m.it[mi].base;
              for (int q = tid; q < tot * NRB; q += (W * 32)) {
                const int ee = q / NRB, r = q % NRB, t = seg_of(ee, Rout, c), kk = ee - t * Rout;
                float2 v;
                if (st.compact) {
                  int pre = 0;
                  for (int u = 0; u < t; ++u) pre += seg_lines(rk, u);
                  v = kk < seg_lines(rk, t) ? red[(pre + kk) * NRB + r] : make_float2(0.f, 0.f);
                } else {
                  v = red[q];
                }
                dst[int64_t(m.out.base + t * m.out.step + kk) * NRB + r] = v;
              }
            }
          } else {
            // V^L: a line is a point p of leaf t: out[p] = sum_k conj(W[p][k]) x[t][k]; one thread
            // per (point, RHS), each starting at another k
            const int len = st.R_out;
            each_chunk(0, [&](uint32_t re, uint32_t im, int l0, int nl) {
              for (int q = tid; q < nl * NRB; q += (W * 32)) {
                const int r = q / nl, l = q - r * nl, p = l0 + l;
                int t = 0;
                for (int u = 1; u < c; ++u) t += p >= m.lb[u] ? 1 : 0;
                const uint32_t xt = xin_a + uint32_t(t * len * NRB + r) * 8u;
                const uint32_t o = uint32_t(l * len) * 4u;
                emit_point(p, r, conj_dot(re + o, im + o, xt, NRB * 8, len, l % len));
              }
            });
          }
        }
        cons_sync<W>();
        dead = !ok;
        if (tid == 0 && ok) {
          mbar_arrive(&xempty[xb]);
          if (!last) st_release_cta(done, j + 1);
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) finish_counters(a.ctl);
}

// ---------------------------------------------------------------- host side

namespace {

// Entries (per RHS) of the partial-sum buffer for blocks and leaf groups of at most xcap:
// shares x entries of a main block, of a leaf group's sums and of its points; the adjoint
// keeps one result per line.
int red_entries(int warps, int xcap) {
  int most = xcap;
  for (int n = 1; n <= xcap; ++n) {
    const int parts = entry_parts(n), rounded = parts * 4 * ((n + 4 * parts - 1) / (4 * parts));
    const int blocks = n > 128 ? 8 : n > 64 ? 4 : n > 32 ? 2 : 1;
    most = std::max({most, warps / parts * rounded, std::max(1, warps / 4) * n, std::max(1, warps / blocks) * n});
  }
  return most;
}

size_t fixed_smem(int nrb, int xcap, int warps, int gathers) {
  return (size_t(gathers + 1) * xcap + size_t(red_entries(warps, xcap))) * size_t(nrb) * sizeof(float2) +
         size_t(gathers) * sizeof(GroupMeta) + (2 * kMaxSlots + 2 * gathers + 1) * 8 + kMaxSlots * 4;
}

// Ring slots (a multiple of the warps) that fit beside the rest; 0: not even one per warp.
int ring_slots(int nrb, int xcap, int warps, int gathers, size_t limit) {
  const size_t fixed = fixed_smem(nrb, xcap, warps, gathers);
  int d = kMaxSlots / warps * warps;
  while (d > 0 && fixed + size_t(d) * kSlotBytes > limit) d -= warps;
  return d;
}

template <int NRB, bool ADJ, int W, int GA, int CPS>
cudaError_t launch_t(ApplyArgs a, int grid, const SimtConfig& cfg_s, cudaStream_t stream) {
  auto kern = bf_apply_simt<NRB, ADJ, W, GA, CPS>;
  a.n_slots = cfg_s.slots;
  a.redcap = red_entries(W, a.xcap);
  a.rot = a.plan.st[0].n_groups % grid;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cfg_s.smem));
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3((W + GA + 2) * 32);
  cfg.dynamicSmemBytes = cfg_s.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

// The launch shapes: one CTA of 8 consumer warps to an SM, or two CTAs of 4.
constexpr int kWideWarps = 8, kWideGathers = 4, kPairWarps = 4, kPairGathers = 2;

template <int NRB, bool ADJ>
cudaError_t launch_n(const ApplyArgs& a, int sms, const SimtConfig cfg[2], cudaStream_t stream) {
  const SimtShape s = simt_shape(a.plan.st[0].n_groups, sms, cfg);   // (as many groups in every stage)
  if (s.pair) return launch_t<NRB, ADJ, kPairWarps, kPairGathers, 2>(a, s.grid, cfg[1], stream);
  return launch_t<NRB, ADJ, kWideWarps, kWideGathers, 1>(a, s.grid, cfg[0], stream);
}

}  // namespace

// Two CTAs to an SM where each gets at least a group per stage: a group's chain of waits,
// gathers and reductions on one overlaps the other's products.  Fewer groups than that are
// finished soonest by the most warps.
SimtShape simt_shape(int groups, int sms, const SimtConfig cfg[2]) {
  if (cfg[1].slots > 0 && groups >= 2 * sms)
    return {true, 2 * sms, (kPairWarps + kPairGathers + 2) * 32, cfg[1].smem};
  return {false, std::min(sms, groups), (kWideWarps + kWideGathers + 2) * 32, cfg[0].smem};
}

int simt_pass_rhs(int64_t rhs_left) { return rhs_left > 4 ? 8 : rhs_left > 2 ? 4 : rhs_left == 2 ? 2 : 1; }

// Ring slots and shared memory of both launch shapes (one and two CTAs to an SM) for passes
// of nrb RHS over blocks and leaf groups of at most xcap entries (<= 256).
cudaError_t simt_config(int nrb, int xcap, SimtConfig cfg[2]) {
  int dev = 0, optin = 0, per_sm = 0, reserved = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if ((err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return err;
  if ((err = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess)
    return err;
  if ((err = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev)) != cudaSuccess)
    return err;
  const int warps[2] = {kWideWarps, kPairWarps}, gathers[2] = {kWideGathers, kPairGathers};
  const size_t limit[2] = {size_t(optin), size_t(per_sm / 2 - reserved)};
  for (int k = 0; k < 2; ++k) {
    cfg[k].slots = ring_slots(nrb, xcap, warps[k], gathers[k], limit[k]);
    cfg[k].smem = fixed_smem(nrb, xcap, warps[k], gathers[k]) + size_t(cfg[k].slots) * kSlotBytes;
  }
  return cfg[0].slots > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

size_t counter_bytes(const Plan& plan) {
  size_t n = 0;
  for (int e = 0; e < plan.n_stages; ++e) n += size_t(plan.st[e].n_groups);
  return (n * sizeof(unsigned) + 255) & ~size_t(255);
}

// One pass: RHS a.rhs0 .. a.rhs0 + nrb - 1 (those below a.nrhs), on `sms` SMs.
cudaError_t launch_apply_simt(const ApplyArgs& a, int nrb, bool adj, int sms, const SimtConfig cfg[2],
                              cudaStream_t stream) {
  sms = std::max(1, sms);
  if (!a.ctl) {
    const cudaError_t err = cudaMemsetAsync(a.counters, 0, counter_bytes(a.plan), stream);
    if (err != cudaSuccess) return err;
  }
  switch (nrb * 2 + (adj ? 1 : 0)) {
    case 2: return launch_n<1, false>(a, sms, cfg, stream);
    case 3: return launch_n<1, true>(a, sms, cfg, stream);
    case 4: return launch_n<2, false>(a, sms, cfg, stream);
    case 5: return launch_n<2, true>(a, sms, cfg, stream);
    case 8: return launch_n<4, false>(a, sms, cfg, stream);
    case 9: return launch_n<4, true>(a, sms, cfg, stream);
    case 16: return launch_n<8, false>(a, sms, cfg, stream);
    case 17: return launch_n<8, true>(a, sms, cfg, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mbf
