// Autotuner for one operator (the paper has no counterpart): times the FP32 SIMT apply
// over RHS counts and the tensor-core panels of 64 and of 32 RHS over (panel buffers,
// A-ring depth) on the device, keeps each panel's fastest configuration, the present one
// where none is faster, and sets the RHS count from which MBF_PREC_AUTO switches to the
// tensor cores.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <utility>
#include <vector>

#include "apply.hpp"
#include "op_internal.hpp"

namespace {

using mbf::fail;

void cuda_ok(cudaError_t e, const char* what) {
  if (e != cudaSuccess) fail(MBF_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

struct DevBuf {
  void* p = nullptr;
  ~DevBuf() { cudaFree(p); }
};
struct Events {
  cudaEvent_t a = nullptr, b = nullptr;
  ~Events() {
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
  }
};

// Device time of one apply (median-free: best of `reps` after one warm-up).
double time_apply(mbf_op_s* op, const void* g, void* u, int64_t nrhs, int32_t prec, cudaStream_t st, Events& ev,
                  int reps) {
  mbf::apply_dev(op, g, u, nrhs, prec, st, false, 0);
  double best = 1e30;
  for (int r = 0; r < reps; ++r) {
    cuda_ok(cudaEventRecord(ev.a, st), "event");
    mbf::apply_dev(op, g, u, nrhs, prec, st, false, 0);
    cuda_ok(cudaEventRecord(ev.b, st), "event");
    cuda_ok(cudaEventSynchronize(ev.b), "event sync");
    float ms = 0.f;
    cuda_ok(cudaEventElapsedTime(&ms, ev.a, ev.b), "elapsed");
    best = std::min(best, double(ms));
  }
  return best;
}

// Configurations (ring slots, panel buffers) to time, 8 at most: the present one first, then
// with two and three buffers the deepest rings that fit beside them (deepest[b - 1] slots,
// 0: none).
std::vector<std::pair<int, int>> tune_candidates(int slots, int buffers, const int deepest[3]) {
  std::vector<std::pair<int, int>> c{{slots, buffers}};
  for (int b = 2; b <= 3; ++b) {
    const int quota = b == 2 ? 5 : 3, top = deepest[b - 1];
    for (int n = std::max(2, top - 2 * (quota - 1)); n <= top && c.size() < 8; n += 2)
      if (n != slots || b != buffers) c.push_back({n, b});
  }
  return c;
}

// Smallest measured RHS count whose SIMT apply takes longer than the panel it would fill (of
// 32 RHS at narrow_ms, else of 64 at full_ms); 65 if none does.
int tune_crossover(int n, const int32_t* rhs, const double* simt_ms, double narrow_ms, double full_ms) {
  for (int i = 0; i < n; ++i)
    if (simt_ms[i] > (rhs[i] <= mbf::kTcNRHalf ? narrow_ms : full_ms)) return rhs[i];
  return mbf::kTcNR + 1;
}

// Times a panel's configurations on `op` (nsa, nxb, smem: the operator's own) and leaves the
// fastest in place, the one found there where none is faster; record(slots, buffers, ms) each.
// Returns its time.  An exception leaves the operator as it was.
template <class F>
double tune_panel(mbf_op_s* op, int nr, int& nsa, int& nxb, size_t& smem, const void* g, void* u, cudaStream_t st,
                  Events& ev, F record) {
  int optin = 0;
  cuda_ok(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, op->device), "attr");
  const auto bytes = [&](int n, int b) {
    return mbf::tc_smem_bytes(n, b, op->tc_nsets, op->tc_mt_max, op->tc_kpad_max, nr);
  };
  int deepest[3] = {0, 0, 0};
  for (int b = 1; b <= 3; ++b)
    for (int n = 2; n <= 16; n += 2)
      if (bytes(n, b) <= size_t(optin)) deepest[b - 1] = n;
  const int nsa0 = nsa, nxb0 = nxb;
  const size_t smem0 = smem;
  int best_nsa = nsa, best_nxb = nxb;
  size_t best_smem = smem;
  double best = 1e30;
  try {
    for (const auto& [n, b] : tune_candidates(nsa0, nxb0, deepest)) {
      nsa = n;
      nxb = b;
      smem = std::max(bytes(n, b), size_t(optin) / 2 + 1024);
      const double ms = time_apply(op, g, u, nr, MBF_PREC_BF16X3, st, ev, 3);
      record(n, b, ms);
      if (ms < best) {
        best = ms;
        best_nsa = n;
        best_nxb = b;
        best_smem = smem;
      }
    }
  } catch (...) {
    nsa = nsa0;
    nxb = nxb0;
    smem = smem0;
    throw;
  }
  nsa = best_nsa;
  nxb = best_nxb;
  smem = best_smem;
  return best;
}

}  // namespace

extern "C" mbf_status mbf_op_tune(mbf_op_t op, void* stream, mbf_tune_result_t* out) {
  return mbf::abi_guard([&] {
    if (!op || !out) fail(MBF_ERR_INVALID, "NULL argument");
    *out = mbf_tune_result_t{};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    constexpr int kMaxRhs = 64;
    DevBuf g, u;
    cuda_ok(cudaMalloc(&g.p, size_t(kMaxRhs) * size_t(op->n_in) * sizeof(float2)), "cudaMalloc");
    cuda_ok(cudaMalloc(&u.p, size_t(kMaxRhs) * size_t(op->n_out) * sizeof(float2)), "cudaMalloc");
    // inputs: every float = 0x3c3c3c3c (about 0.0115), a finite nonzero pattern
    cuda_ok(cudaMemsetAsync(g.p, 0x3c, size_t(kMaxRhs) * size_t(op->n_in) * sizeof(float2), st), "memset");
    Events ev;
    cuda_ok(cudaEventCreate(&ev.a), "event");
    cuda_ok(cudaEventCreate(&ev.b), "event");
    const int rhs_list[] = {1, 2, 4, 8, 16, 32, 64};
    for (int R : rhs_list) {
      if (!op->simt_unavailable.empty()) break;   // tensor-only operator
      out->simt_rhs[out->n_simt] = R;
      out->simt_ms[out->n_simt] = time_apply(op, g.p, u.p, R, MBF_PREC_FP32_SIMT, st, ev, 3);
      ++out->n_simt;
    }
    if (op->tc_unavailable.empty()) {
      const double full = tune_panel(op, mbf::kTcNR, op->tc_nsa, op->tc_nxb, op->tc_smem, g.p, u.p, st, ev,
                                     [&](int n, int b, double ms) {
                                       out->slots[out->n_slots] = n;
                                       out->panel_buffers[out->n_slots] = b;
                                       out->tc_ms[out->n_slots] = ms;
                                       ++out->n_slots;
                                     });
      const double narrow = tune_panel(op, mbf::kTcNRHalf, op->tc_nsa32, op->tc_nxb32, op->tc_smem32, g.p, u.p, st, ev,
                                       [](int, int, double) {});
      out->tc_slots_chosen = op->tc_nsa;
      out->tc_buffers_chosen = op->tc_nxb;
      out->tc_min_rhs = op->simt_unavailable.empty()
                            ? tune_crossover(out->n_simt, out->simt_rhs, out->simt_ms, narrow, full)
                            : 1;
      op->tc_min_rhs = out->tc_min_rhs;
    } else {
      out->tc_min_rhs = 1 << 30;
    }
    cuda_ok(cudaStreamSynchronize(st), "sync");
    int dev_status = 0;
    cuda_ok(cudaMemcpy(&dev_status, op->ws.status, sizeof(int), cudaMemcpyDeviceToHost), "status");
    if (dev_status != 0) {
      cuda_ok(mbf::zero_now(op->ws.status, sizeof(int)), "clear status");
      fail(MBF_ERR_TIMEOUT, "a device wait gave up while tuning");
    }
  });
}

extern "C" mbf_status mbf_debug_tune_candidates(int32_t slots, int32_t buffers, const int32_t* deepest, int32_t* n,
                                                int32_t* slots_out, int32_t* buffers_out) {
  return mbf::abi_guard([&] {
    if (!deepest || !n || !slots_out || !buffers_out) fail(MBF_ERR_INVALID, "NULL argument");
    const int d[3] = {deepest[0], deepest[1], deepest[2]};
    const auto c = tune_candidates(slots, buffers, d);
    *n = int32_t(c.size());
    for (size_t k = 0; k < c.size(); ++k) {
      slots_out[k] = c[k].first;
      buffers_out[k] = c[k].second;
    }
  });
}

extern "C" mbf_status mbf_debug_tune_crossover(int32_t n, const int32_t* rhs, const double* simt_ms, double narrow_ms,
                                               double full_ms, int32_t* min_rhs) {
  return mbf::abi_guard([&] {
    if (n < 0 || (n > 0 && (!rhs || !simt_ms)) || !min_rhs) fail(MBF_ERR_INVALID, "NULL argument or negative count");
    *min_rhs = tune_crossover(n, rhs, simt_ms, narrow_ms, full_ms);
  });
}
