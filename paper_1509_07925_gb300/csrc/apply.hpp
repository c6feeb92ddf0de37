// Host/device interface of the apply kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "layout.hpp"

namespace mbf {

// Per-RHS row addresses of an apply's input and output, for up to kRowTab RHS: a served
// batch applies its requests' rows where the callers put them, with no staging copies.
// in[r] (n_in entries) and out[r] (n_out entries) for RHS r < nrhs.
constexpr int kRowTab = 64;
struct RowTable {
  const float2* in[kRowTab];
  float2* out[kRowTab];
};

struct ApplyArgs {
  const uint8_t* arena;
  const Item* items;
  const int32_t* x_perm;
  const int32_t* x_off;
  const int32_t* w_perm;
  const int32_t* w_off;
  const float2* in;        // forward: g [nrhs][n_in]; adjoint: u [nrhs][n_out]
  float2* out;             // forward: u; adjoint: g
  int64_t in_len, out_len;
  float2* bufs;            // stage e < S - 1 writes bufs + e * buf_stride ([pos][NRB]); stage e+1 reads it
  int64_t buf_stride;
  // [stage][group]: input segments written so far.  With ctl, two sets of them: a launch
  // counts in set ctl[0] & 1 and clears the other one for the next launch, so that no
  // memset precedes it (the last CTA to finish, counted in ctl[1], flips ctl[0]; the state
  // lives on the device, so a captured launch may be replayed).  Without, one set, cleared by
  // launch_apply_simt.
  unsigned int* counters;
  unsigned int* ctl;
  int* status;             // 0 = ok; nonzero = a device wait ran out of time (sticky)
  int32_t nrhs, rhs0;      // this launch applies RHS rhs0 .. min(nrhs, rhs0 + NRB) - 1
  int32_t xcap;            // most entries of a block side or points of a leaf group (<= 256)
  // set by the launch: ring slots; partial-sum entries; shift of the CTAs' groups per stage
  int32_t n_slots, redcap, rot;
  int32_t accumulate;      // 1: out += result (the caller initialised out), 0: out = result
  // Failure-detection test hook (mbf_op_debug_stall); zero leaves the apply unchanged.
  // stall_stage1 = 1 + s: the dependency wait of group 0 of stage s (execution order)
  // waits for one more producer than exists, so that it can only end by running out of
  // time.  wait_ns > 0: a wait on a dependency counter gives up after wait_ns instead of
  // kTimeoutNs, the waits inside a CTA after twice as long.
  uint64_t wait_ns;
  int32_t stall_stage1, stall_pad_;
  int32_t use_rows, rows_pad_;   // 1: in / out rows from `rows` (nrhs <= kRowTab)
  RowTable rows;
  Plan plan;
};

// Words before a workspace's counters: ctl[0], ctl[1] and padding.
constexpr int kCtlWords = 64;
// Bytes of a workspace's counters for a kernel that counts in `set_bytes`.
MBF_HD size_t counters_alloc(size_t set_bytes) { return kCtlWords * sizeof(unsigned) + 2 * set_bytes; }

#if defined(__CUDACC__)
// The launch's counter set, of `words` counters.
__device__ __forceinline__ unsigned* counter_set(unsigned* counters, const unsigned* ctl, unsigned words) {
  return ctl && (__ldcg(ctl) & 1u) ? counters + words : counters;
}
// Clears this CTA's part of the other set (threads tid < nth of each CTA).
__device__ __forceinline__ void clear_other_set(unsigned* counters, const unsigned* ctl, unsigned words, unsigned tid,
                                                unsigned nth) {
  if (!ctl) return;
  unsigned* other = __ldcg(ctl) & 1u ? counters : counters + words;
  for (unsigned i = blockIdx.x * nth + tid; i < words; i += gridDim.x * nth) other[i] = 0;
}
// By one thread of each CTA when all the CTA's counting is done: the last one flips the sets.
__device__ __forceinline__ void finish_counters(unsigned* ctl) {
  if (!ctl) return;
  const unsigned epoch = __ldcg(ctl);
  __threadfence();
  if (atomicAdd(ctl + 1, 1u) == gridDim.x - 1) {
    ctl[1] = 0;
    ctl[0] = epoch ^ 1u;
  }
}
#endif

enum DeviceStatus : int {
  ST_OK = 0,
  ST_FULL_TIMEOUT = 1,
  ST_EMPTY_TIMEOUT = 2,
  ST_BAD_ITEM = 3,
  ST_DEP_TIMEOUT = 4
};


// Vectors between the tensor-core stages are "split blocks": block P of a level holds
// the R8 coefficients of one tree-node pair for the kTcNR right-hand sides of a panel
// as bf16 pairs hi = bf16(x), lo = bf16(x - hi), laid out as the MMA's K-major A
// operand with the real and imaginary parts of RHS n interleaved on M (rows
// m = 2 n + ri, ri = 0 real, 1 imaginary):
//   byte (hl, k, m) = hl R8 4 NR + (k / 8) 32 NR + (m / 8) 128 + (m % 8) 16 + (k % 8) 2
// with NR the panel's RHS.  A consumer copies each hi / lo half of a block into shared
// memory as it is.
constexpr int kTcNR = 64;        // RHS of a tensor-core panel (MMAs of M = 128) ...
// ... or half of them (M = 64): a panel of at most 32 RHS moves half the vector bytes, its
// buffers take half the shared memory (so the tile ring is deeper) and its leaf products
// are half as many.  n = 128, r = 16 with 20 RHS: 84 us with panels of 64, 77 with 32;
// multiscale n = 128 with 32 RHS: 324 and 280; 3-D n = 32, r = 32 with 32 RHS: 252 (two ring
// slots beside one panel buffer) and 173 (four).  On a few dozen groups it may be the slower
// one by a microsecond: n = 64, L = 4, r = 24 with 20 RHS 35.5 and 36.9, r = 64 76.7 and 60.1.
constexpr int kTcNRHalf = 32;
MBF_HD int64_t split_block_bytes(int R8, int nr = kTcNR) { return int64_t(R8) * nr * 8; }
// With TF32 operands the same block holds FP32 (TF32-rounded) values instead, byte
//   (k, m) = (k / 4) 32 NR + (m / 8) 128 + (m % 8) 16 + (k % 4) 4
// (the MMA's K-major A operand for 32-bit types): the same R8 x 8 NR bytes.

struct TCArgs {
  const uint8_t* arena;
  const uint8_t* x_in;     // input of main stage 0 (split blocks)
  uint8_t* bufs;           // output of main stage e < S - 1: bufs + e * buf_stride (split blocks)
  float* y_out;            // output of the last main stage: row block * R + k, [re NR | im NR] floats
  int64_t buf_stride;      // bytes
  unsigned* counters;      // [stage][group], two sets as in ApplyArgs
  unsigned* ctl;
  int* status;
  int32_t nsa, nxb;        // A ring slots; panel buffers (1 or 2)
  int32_t nsets, mt_max;   // accumulator sets (1 or 2, 2 mt_max TMEM columns each); largest M_t
  int32_t kpad_max, pad_;  // largest K_pad
  TCPlan plan;
};

struct LeafArgs {
  const uint8_t* arena;    // packed arena of the SIMT path (leaf items)
  const Item* items;
  int64_t item_base;       // item of group 0; group g's item is item_base + g * item_stride
  const int32_t* perm;     // U^L: tree -> natural x index; permute: natural -> tree Omega index
  const int32_t* off;      // leaf offsets (tree order)
  const float2* vec;       // (V^L)^*: panel in tree order [point][64]; permute: g [nrhs][len_vec]
  const float* wl;         // U^L: level-L coefficients, row block * R + k, [re NR | im NR] floats
  float2* outp;            // U^L: u [nrhs][len_out]; permute: panel in tree order
  uint8_t* outs;           // (V^L)^*: split blocks of the level-L vector (block c g + t)
  int64_t len_vec, len_out;
  int32_t nrhs, rhs0, c, R;
  int32_t R8, item_stride;
  int32_t accumulate;       // U^L: 1 adds into u
  int32_t pts_cap;          // (V^L)^*: points staged per round (leaf_pts_cap of the largest leaf)
  int32_t leaf_split;       // U^L side: 1 = one CTA per leaf (ragged trees, few groups), 0 = one per group
  int32_t small_leaves;     // U^L side, leaf_split: rounds of 16 points instead of 64
  int32_t gather;           // (V^L)^* side: 1 = vec is [nrhs][len_vec] in natural order, read through
                            // nat; 0 = the tree-ordered panel
  int32_t nat_stride;       // (V^L)^* gather: entries per leaf in nat
  const int32_t* nat;       // (V^L)^* gather: leaf j's natural indices at nat[j * nat_stride + b]
  int32_t use_rows, rows_pad_;   // 1: (V^L)^* gather reads rows.in[rhs], U^L writes rows.out[rhs]
  RowTable rows;
};

// FP32 SIMT path (apply_simt.cu): one launch per pass of 1, 2, 4 or 8 RHS.
// The launch of a pass over plans of `groups` groups on `sms` SMs: one CTA to an SM or two.
struct SimtShape {
  bool pair;
  int grid, threads;
  size_t smem;
};
SimtShape simt_shape(int groups, int sms, const SimtConfig cfg[2]);
int simt_pass_rhs(int64_t rhs_left);   // RHS of the next pass (the last one may be padded)
cudaError_t simt_config(int nrb, int xcap, SimtConfig cfg[2]);
cudaError_t launch_apply_simt(const ApplyArgs& a, int nrb, bool adj, int sms, const SimtConfig cfg[2],
                              cudaStream_t stream);
// Bytes of dependency counters for a plan (S stages x groups, rounded up to 256).
size_t counter_bytes(const Plan& plan);

// tensor-core path (apply_tc.cu)
size_t tc_smem_bytes(int nsa, int nxb, int nsets, int mt_max, int kpad_max, int nr = kTcNR);
size_t tc_counter_bytes(const TCPlan& plan);
// Dynamic shared memory of a leaf kernel; the (V^L)^* side stages pts_cap points a round.
size_t leaf_smem_bytes(int R, int c, bool u_side, int pts_cap = 64, int nr = kTcNR);
// Points per round of the (V^L)^* leaf kernel for leaves of at most max_leaf_points
// points: rounded up to 8, within [8, 64].
int leaf_pts_cap(int64_t max_leaf_points);
bool leaf_fits(int R8, int c);   // leaf kernels: R8 <= 64, c <= 8
// tf32: TF32 tiles and vectors (kind::tf32 MMAs), else split-BF16x3.
// nr: RHS of the panel (kTcNR or kTcNRHalf).
cudaError_t launch_apply_tc(const TCArgs& a, int grid, size_t smem, cudaStream_t stream, bool tf32, int nr);
// TF32 tiles (two FP32 planes per K16 chunk) converted from n_chunks split-BF16 chunks of M_t rows.
cudaError_t launch_tf32_tiles(const uint8_t* src, uint8_t* dst, int64_t n_chunks, int M_t, cudaStream_t stream);
// U^L side: one CTA per group of c leaves; (V^L)^* side: one CTA per leaf (c n_groups CTAs).
// xpose: the adjoint's leaf products (U^* from the U^L items, V from the (V^L)^* items).
cudaError_t launch_leaf(const LeafArgs& a, bool u_side, int n_groups, cudaStream_t stream, int nr, bool tf32 = false,
                        bool xpose = false);
// Adjoint (conjugate-transposed) split-BF16 tiles of one stage from its forward tiles.
cudaError_t launch_adjoint_tiles(const uint8_t* src, uint8_t* dst, int n_groups, int M_t, int K_t, cudaStream_t stream);
// vec = g [nrhs][len_vec], perm = inverse tree permutation (natural -> tree, -1 if absent),
// outp = panel in tree order [tree point][64]
cudaError_t launch_permute_in(const LeafArgs& a, cudaStream_t stream);

}  // namespace mbf
